"""The product of the FP64 master with many right-hand sides at the edges of
its tiles (16 rows, five tiles per CTA, chunks of 32 columns, 8 or 16
right-hand sides, panels cut into several work items) and of its number range,
against the oracle applying the exported operator in FP64.

Bounds, as in test_gpu_df.py: each row within 2e-13 of the row sum of
|H||x|, and within 2e-14 of it in norm.  The digits keep 54 bits of every x on
the scale of the largest x_r of its column and of every entry on that of the
largest term of its row, products below 2^-56 of that are dropped, and the
float pairs that carry the sums round at 2^-48: 4e-15 of |H||x|, times the
ratio of the largest term to a right-hand side's own (at most ~50 here).
"""
import numpy as np
import pytest

import meshgen

from hm_gpu_util import GpuH, need_gpu
from test_gpu_df import abs_operator, oracle_apply

pytestmark = pytest.mark.gpu


def _product(g, X):
    torch = g.torch
    Xd = torch.from_numpy(np.ascontiguousarray(X)).cuda()
    Y = torch.empty_like(Xd)
    g.hm.hm_matvec_block(g.A, Xd, Y, prec=g.hm.HM_F64)
    torch.cuda.synchronize()
    return Y.cpu().numpy()


def _check(orc, g, X):
    ex = g.export()
    Y = _product(g, X)
    ref, mag = oracle_apply(orc, g, ex, X), oracle_apply(orc, g, abs_operator(ex), np.abs(X))
    assert np.isfinite(Y).all()
    assert (np.abs(Y - ref) <= 2e-13 * mag).all(), (np.abs(Y - ref) / mag).max()
    assert (np.linalg.norm(Y - ref, axis=1) <= 2e-14 * np.linalg.norm(mag, axis=1)).all()


# leaves of 1 to 248 rows: one row, one tile and one more, two CTAs of tiles and one more, sixteen tiles; right-hand
# sides: one, a fragment of 8 and one more, a pass of 16 and one more
@pytest.mark.parametrize("leaf,nrhs", [(1, 16), (16, 1), (17, 8), (33, 9), (80, 16), (81, 17), (248, 16)])
def test_tile_edges(orc, leaf, nrhs):
    need_gpu()
    V, T = meshgen.bump_sphere(3, 1808)[:2]
    g = GpuH(V, np.ascontiguousarray(T[:1003]), leaf=leaf, eta=1.5, eps=1e-6)
    try:
        _check(orc, g, np.random.default_rng(leaf).standard_normal((nrhs, g.n)))
    finally:
        g.close()


def test_ranges_and_non_finite_values(orc):
    need_gpu()
    V, T = meshgen.icosphere(3)
    g = GpuH(V, T, leaf=40, eta=1.5, eps=1e-6)
    try:
        rng = np.random.default_rng(3)
        # scales beyond FP32, positive vectors, entries over many decades, zeros
        X = rng.standard_normal((16, g.n)) * 10.0 ** np.linspace(-200, 200, 16)[:, None]
        X[3] = np.abs(X[3])
        X[7] *= 10.0 ** rng.uniform(-12, 0, g.n)
        X[9] = 0.0
        _check(orc, g, X)
        # a NaN or an infinity reaches every row of its own right-hand side and no other
        Y = _product(g, X)
        X[1, 5], X[14, 700] = np.nan, np.inf
        Z = _product(g, X)
        for r in range(16):
            if r in (1, 14):
                assert np.isnan(Z[r]).all()
            else:
                assert np.linalg.norm(Z[r] - Y[r]) <= 2e-13 * max(np.linalg.norm(Y[r]), 1e-300)
    finally:
        g.close()


def test_panels_cut_into_items(orc):
    # leaf clusters that the Morton order tears apart have near fields many times the mean width
    need_gpu()
    V, T = meshgen.icosphere(4)
    g = GpuH(V, T, leaf=20, eta=1.5, eps=1e-6)
    try:
        dl = g.leaves(True)
        width = np.bincount(dl[:, 0], weights=dl[:, 3] - dl[:, 2])
        assert width.max() > 24 * 32  # more than the fewest chunks an item may hold
        _check(orc, g, np.random.default_rng(1).uniform(0.5, 1.5, (16, g.n)))
    finally:
        g.close()
