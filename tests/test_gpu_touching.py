"""Entries of touching panels (one warp per entry, eight entries per CTA) for
quadrature orders whose point counts are below, at and beyond a multiple of 32
and meshes whose number of touching pairs is not a multiple of eight, against
the oracle's matrix: within 1e-12 of each entry (points to 2^-47 of their largest
term, at most 8,192 positive weights times reciprocal distances summed in
double-float)."""
import numpy as np
import pytest

import meshgen
import oracle

from hm_gpu_util import GpuH, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2, 3, 8, 16])
@pytest.mark.parametrize("fp64", [0, 1])
def test_orders(orc, order, fp64):
    need_gpu()
    V, T = meshgen.bump_sphere(1, 1808)[:2]
    T = np.ascontiguousarray(T[:53])
    g = GpuH(V, T, leaf=9, eta=0.1, eps=1e-6, ss_order=order, nearfield_fp64=fp64)
    try:
        perm, ex = g.perm(), g.export()
        A = orc.dense_matrix(V, T, oracle.Quad(order))[np.ix_(perm, perm)]
        for b, (rb, re, cb, ce) in enumerate(g.leaves(True)):
            m, n = re - rb, ce - cb
            B = ex["dense"][ex["dense_off"][b]:ex["dense_off"][b] + m * n].reshape(m, n)
            assert (np.abs(B - A[rb:re, cb:ce]) <= 1e-12 * np.abs(A[rb:re, cb:ce])).all()
    finally:
        g.close()
