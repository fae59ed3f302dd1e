"""Entries of the factored blocks where a warp's last round is spread over idle
lanes (8, 4 and 2 lanes per entry for up to 4, 8 and 16 entries left over, one
above that), against the oracle's matrix: cluster sizes of 3 or 4, 7 or 8, 15 or
16, 31 or 32 and 62 or 63 panels, and everything above them that is admissible.

Each block within 10 eps of the oracle's in the Frobenius norm: the stopping test
takes the last cross's size for the remainder, which decays geometrically; a
wrong value in a pivot row or column would stay in the block at its own size."""
import numpy as np
import pytest

import meshgen

from hm_gpu_util import GpuH, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [4, 8, 16, 32, 63])
def test_blocks(orc, leaf):
    need_gpu()
    eps = 1e-5
    V, T = meshgen.bump_sphere(3, 1808)[:2]
    T = np.ascontiguousarray(T[:1003])
    g = GpuH(V, T, leaf=leaf, eta=1.5, eps=eps)
    try:
        perm, al, ex = g.perm(), g.leaves(False).reshape(-1, 4), g.export()
        A = orc.dense_matrix(V, T)[np.ix_(perm, perm)]
        assert al.shape[0] > 0
        for b, (rb, re, cb, ce) in enumerate(al):
            m, n, k = re - rb, ce - cb, int(ex["rank"][b])
            U = ex["uw"][ex["u_off"][b]:ex["u_off"][b] + m * k].reshape(k, m)
            W = ex["uw"][ex["w_off"][b]:ex["w_off"][b] + n * k].reshape(k, n)
            B = A[rb:re, cb:ce]
            assert np.linalg.norm(U.T @ W - B) <= 10 * eps * np.linalg.norm(B), (b, m, n, k)
    finally:
        g.close()


def test_squares_below_the_normal_float_range():
    # squared distances around 2^-126, where the estimate of the reciprocal square root needs its wide form (below
    # 2^-128 its square overflows); the products of the areas, and with them the regular entries, are 0 there
    need_gpu()
    V, T = meshgen.icosphere(2)
    g = GpuH(V * 2.0 ** -61.5, T, leaf=20, eta=1.5, eps=1e-6)
    try:
        ex = g.export()
        assert np.isfinite(ex["dense"]).all() and np.isfinite(ex["uw"]).all()
    finally:
        g.close()
