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


@pytest.mark.parametrize("leaf,count", [(20, 40), (40, 100)])
def test_blocks_shared_by_a_cta(orc, leaf, count):
    # with fewer blocks than warps a CTA works on one block, with many copies of the geometry a warp does:
    # the same ranks and factors, bit for bit
    torch = need_gpu()
    import paper_1806_11558_gb300 as hm
    V, T = meshgen.bump_sphere(3, 1808)[:2]
    g = GpuH(V, T, leaf=leaf, eta=1.5, eps=1e-6)
    n, nv = T.shape[0], V.shape[0]
    Vs = torch.from_numpy(np.tile(V, (count, 1))).cuda()
    Ts = torch.from_numpy(np.ascontiguousarray((T[None] + nv * np.arange(count)[:, None, None]).reshape(-1, 3)
                                               .astype(np.int32))).cuda()
    tree = hm.hm_build_forest(Vs, Ts, [n * k for k in range(count + 1)], eta=1.5, leaf_size=leaf)
    A = hm.hm_assemble(tree, aca_eps=1e-6)
    try:
        ti = hm.hm_tree_get_info(tree)
        one, all_ = g.export(), hm.hm_matrix_export(A, ti["n_dense"], ti["n_adm"])
        al = g.leaves(False).reshape(-1, 4)
        ak = {tuple(b): k for k, b in enumerate(hm.hm_tree_get_leaves(tree, False).cpu().numpy().reshape(-1, 4).tolist())}
        assert al.shape[0] > 0 and ti["n_adm"] == count * al.shape[0]
        for b, blk in enumerate(al.tolist()):
            c, k = ak[tuple(blk)], int(one["rank"][b])
            assert int(all_["rank"][c]) == k
            for off, size in (("u_off", blk[1] - blk[0]), ("w_off", blk[3] - blk[2])):
                x = one["uw"][one[off][b]:one[off][b] + size * k]
                assert np.array_equal(x, all_["uw"][all_[off][c]:all_[off][c] + size * k])
    finally:
        hm.hm_free(A)
        hm.hm_free(tree)
        g.close()
