"""The product of the FP64 master with many right-hand sides where the sizes
of what is summed lie far apart, against the oracle applying the exported
operator in FP64.

Bounds, as in test_gpu_df.py: each row within 2e-13 of its own right-hand
side's row sum of |H||x|, and within 2e-14 of it in norm, whatever the scale of
the mesh.
"""
import numpy as np
import pytest

import meshgen

from hm_gpu_util import GpuH, need_gpu
from test_gpu_fx import _check, _product

pytestmark = pytest.mark.gpu


# entries of H scale as the third power of the mesh: about 1e-25 and 1e-28 here, and the coefficients t of a mirrored
# block as they do, while its rows are multiplied by factors of size 1
@pytest.mark.parametrize("scale", [1e-7, 1e-8])
def test_small_meshes(orc, scale):
    need_gpu()
    V, T = meshgen.icosphere(4)
    g = GpuH(V * scale, T, leaf=64, eta=1.5, eps=1e-6)
    try:
        _check(orc, g, np.random.default_rng(4).standard_normal((16, g.n)))
    finally:
        g.close()


def _graded_sphere(level, power):
    """A sphere whose panels shrink towards a pole: polar angles pi (theta / pi)^power."""
    V, T = meshgen.icosphere(level)
    R = np.linalg.qr(np.random.default_rng(2).standard_normal((3, 3)))[0]  # no vertex on the pole's axis
    V = V @ R
    th, ph = np.arccos(np.clip(V[:, 2], -1, 1)), np.arctan2(V[:, 1], V[:, 0])
    th = np.pi * (th / np.pi) ** power
    return np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], axis=1), T


# each row has terms of some right-hand sides that are far below the others': beside its diagonal, of panels that are
# a million times smaller, and in columns where only one of the vectors is not zero; panels in one part and in several
@pytest.mark.parametrize("nrhs,leaf", [(16, 32), (7, 32), (16, 248)])
def test_unit_vectors_on_a_graded_mesh(orc, nrhs, leaf):
    need_gpu()
    V, T = _graded_sphere(4, 2.5)
    area = np.linalg.norm(np.cross(V[T[:, 1]] - V[T[:, 0]], V[T[:, 2]] - V[T[:, 0]]), axis=1)
    assert area.max() > 1e6 * area.min()
    g = GpuH(V, T, leaf=leaf, eta=1.5, eps=1e-6)
    try:
        order, X = np.argsort(area), np.zeros((nrhs, g.n))
        X[np.arange(nrhs), order[np.linspace(0, g.n - 1, nrhs).astype(int)]] = 1.0
        _check(orc, g, X)
        # and full vectors of sizes that cross between the small panels and the large ones
        X = np.random.default_rng(5).standard_normal((nrhs, g.n))
        X[::2, order[: g.n // 2]] *= 1e-8
        X[1::2, order[g.n // 2 :]] *= 1e-8
        _check(orc, g, X)
    finally:
        g.close()


# peaks on 20 of 5,120 panels in all right-hand sides but one: 256 leaves a few of the 256 clusters' rows unsure (only what they
# read is formed again), 16,384 all of them
@pytest.mark.parametrize("nrhs,peak", [(16, 2 ** 8), (7, 2 ** 8), (16, 2 ** 14)])
def test_peaks_beside_a_vector_without(orc, nrhs, peak):
    need_gpu()
    V, T = meshgen.icosphere(4)
    g = GpuH(V, T, leaf=20, eta=1.5, eps=1e-6)
    try:
        at = np.argsort(-(V[T].mean(1) @ np.array([0.3, 0.5, 0.8])))[:20]
        X = np.random.default_rng(9).standard_normal((nrhs, g.n))
        X[1:, at] *= peak
        _check(orc, g, X)
    finally:
        g.close()


def test_sizes_that_cross_within_one_cluster(orc):
    need_gpu()  # 80 panels, no far field
    V, T = meshgen.icosphere(1)
    g = GpuH(V, T, leaf=100, eta=1.5, eps=1e-6)
    try:
        X = np.random.default_rng(7).standard_normal((16, g.n)) * 10.0 ** np.linspace(-9, 0, 16)[:, None]
        X[:, ::2] = X[::-1, ::2]
        X[5] = 0.0
        _check(orc, g, X)
    finally:
        g.close()


def test_lowest_orders_of_the_digit_products(orc):
    # 1,280 panels against sums in extended precision.  Digits of 62 bits and the orders 0 to 7 of their products are
    # off by 2^-56 of the row's scale at most; what is left are the pairs of floats: up to ten additions per row, each off by
    # 2^-48 of the sum so far, for random vectors less than a fifth of the row sum of |H||x|, at random: sqrt(10) 2^-48 / 5
    # = 2.3e-15, twice (t and y) and in norm below 5e-15 / sqrt(16).  Without the orders 6 and 7 (products below 2^-48
    # of the scale, some thousands per row) it is above that.
    need_gpu()
    V, T = meshgen.icosphere(3)
    g = GpuH(V, T, leaf=64, eta=1.5, eps=1e-6)
    try:
        ex, perm = g.export(), g.perm()
        X = np.random.default_rng(8).standard_normal((16, g.n))
        x = X[:, perm].T.astype(np.longdouble)
        ref, mag = np.zeros_like(x), np.zeros_like(x)
        for i, (rb, re, cb, ce) in enumerate(g.leaves(True)):
            D = ex["dense"][ex["dense_off"][i]:][: (re - rb) * (ce - cb)].reshape(re - rb, ce - cb).astype(np.longdouble)
            ref[rb:re] += D @ x[cb:ce]
            mag[rb:re] += np.abs(D) @ np.abs(x[cb:ce])
        for i, (rb, re, cb, ce) in enumerate(g.leaves(False)):
            k = ex["rank"][i]
            U = ex["uw"][ex["u_off"][i]:][: (re - rb) * k].reshape(k, re - rb).T.astype(np.longdouble)
            W = ex["uw"][ex["w_off"][i]:][: (ce - cb) * k].reshape(k, ce - cb).astype(np.longdouble)
            ref[rb:re] += U @ (W @ x[cb:ce])
            mag[rb:re] += np.abs(U) @ (np.abs(W) @ np.abs(x[cb:ce]))
        Y = _product(g, X)[:, perm].T
        for r in (16, 8):
            err = np.abs(Y[:, :r] - ref[:, :r]) if r == 16 else np.abs(_product(g, X[:r])[:, perm].T - ref[:, :r])
            assert np.sqrt((err * err).sum()) <= 1.25e-15 * np.sqrt((mag[:, :r] * mag[:, :r]).sum())
    finally:
        g.close()


class _Forest(GpuH):
    """Several spheres in one operator."""

    def __init__(self, sizes, leaf, **kw):
        torch = need_gpu()
        import paper_1806_11558_gb300 as hm
        self.hm, self.torch = hm, torch
        Vs, Ts, self.off, nv = [], [], [0], 0
        for k, level in enumerate(sizes):
            V, T = meshgen.icosphere(level)
            Vs.append(V * (1.0 + 0.3 * k))
            Ts.append(T + nv)
            nv += V.shape[0]
            self.off.append(self.off[-1] + T.shape[0])
        self.n = self.off[-1]
        self.Vd = torch.from_numpy(np.concatenate(Vs)).cuda()
        self.Td = torch.from_numpy(np.concatenate(Ts).astype(np.int32)).cuda()
        self.tree = hm.hm_build_forest(self.Vd, self.Td, self.off, eta=1.5, leaf_size=leaf)
        self.A = hm.hm_assemble(self.tree, aca_eps=1e-8, aca_kmax=64, ss_order=8, **kw)


def test_right_hand_sides_whose_sizes_cross_between_geometries(orc):
    g = _Forest((3, 2), 32, factor_dtype=1, dense_dtype=1)
    try:
        torch, hm = g.torch, g.hm
        rng = np.random.default_rng(6)
        size = np.ones((16, g.n))
        size[::2, g.off[1]:] = 1e-8
        size[1::2, : g.off[1]] = 1e-8
        _check(orc, g, size * rng.standard_normal((16, g.n)))
        # every (geometry, right-hand side) is a system with its own stopping test
        b = torch.from_numpy(size[:6] * rng.uniform(0.5, 1.5, (6, g.n))).cuda()
        x = torch.zeros_like(b)
        info = hm.hm_solve(g.A, b, x, rel_tol=1e-12, restart=60, max_iter=3000, precond=1, batched=1, refine=1,
                           inner_dtype=hm.HM_F32, inner_tol=1e-4, max_refine=40, resid_df=1)
        assert info.status == 0 and info.rel_resid <= 1e-12
        y = torch.empty_like(x)
        hm.hm_matvec(g.A, x, y)
        for k in range(2):
            r, f = (b - y)[:, g.off[k]:g.off[k + 1]], b[:, g.off[k]:g.off[k + 1]]
            # the stopping test's 1e-12 and the float pairs' 1e-14 of |H||x|, some tens of |b|
            assert (torch.linalg.norm(r, dim=1) <= 2e-12 * torch.linalg.norm(f, dim=1)).all()
    finally:
        g.close()
