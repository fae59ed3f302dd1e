"""Regular entries in double-float arithmetic on both sides of the separation
at which the sums by orbits of the rule take over from the differences of the
49 point pairs, against the oracle's FP64 entries.

Bound per pair, with r the smallest distance of its quadrature points and c
the largest coordinate: 1e-13 for the double-float sums (as in
test_gpu_parity.py), plus the rounding of the points in the oracle itself,
three roundings of c per point and coordinate: 2 * 3 * 2^-53 c / r, taken as
8 * 2^-53 c / r.
"""
import numpy as np
import pytest

import meshgen

from hm_gpu_util import GpuH, need_gpu

pytestmark = pytest.mark.gpu


def _soup(n, spread, thin=1.0, seed=5):
    """n separate triangles of circumradius ~1 around random points of a cube of side `spread`."""
    rng = np.random.default_rng(seed)
    v = rng.standard_normal((n, 3, 3)) * [1.0, 1.0, thin]
    v -= v.mean(axis=1, keepdims=True)
    v /= np.linalg.norm(v, axis=2).max(axis=1)[:, None, None]
    v += rng.uniform(0.0, spread, (n, 1, 3))
    return np.ascontiguousarray(v.reshape(-1, 3)), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


def _case(name):
    V, T = meshgen.icosphere(2)
    return {
        "soup_near": lambda: _soup(200, 20.0),          # most distances between 1 and 20 circumradii
        "soup_thin": lambda: _soup(160, 40.0, 0.02),
        "soup_far": lambda: _soup(100, 3000.0),
        "one_pair": lambda: _soup(2, 4.0),
        "sphere": lambda: (V, T[:248]),
        "shifted": lambda: (V + [100.0, -50.0, 25.0], T[:248]),
        "tiny": lambda: (V * 1e-6, T[:248]),
        "huge": lambda: (V * 1e8, T[:248]),
    }[name]()


@pytest.mark.parametrize("name", ["soup_near", "soup_thin", "soup_far", "one_pair", "sphere", "shifted", "tiny", "huge"])
def test_regular_entries_vs_oracle(orc, name):
    need_gpu()
    V, T = _case(name)
    n = T.shape[0]
    g = GpuH(V, T, leaf=248, eta=1.5, eps=1e-6)  # one dense leaf
    try:
        perm, leaves, ex = g.perm(), g.leaves(True), g.export()
        assert len(leaves) == 1 and tuple(leaves[0]) == (0, n, 0, n)
        blk = ex["dense"][ex["dense_off"][0]:ex["dense_off"][0] + n * n].reshape(n, n)
    finally:
        g.close()
    ref = orc.dense_matrix(V, T)[np.ix_(perm, perm)]
    bary = orc.Quad().bary
    X = np.einsum("qk,nkd->nqd", bary, V[T])[perm]
    r = np.empty((n, n))
    for i in range(n):
        r[i] = np.sqrt(((X[i][None, :, None, :] - X[:, None, :, :]) ** 2).sum(-1)).min(axis=(1, 2))
    Tp = T[perm]
    touch = (Tp[:, None, :, None] == Tp[None, :, None, :]).any(axis=(2, 3))
    assert (~touch).any()
    tol = 1e-13 + 8 * 2.0 ** -53 * np.abs(V).max() / np.where(touch, 1.0, r)
    rel = np.abs(blk - ref) / np.abs(ref)
    worst = (rel / tol)[~touch].max()
    assert worst <= 1.0, (worst, rel[~touch].max())
