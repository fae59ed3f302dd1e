"""Values of what test_gpu_aca_lanes.py and test_gpu_rows.py reach without looking
at them: the wide forms of the entries (squared distances from 2^-128 to 2^-126), and
the one-right-hand-side product of the BF16 copies at the edges of its blocks."""
import numpy as np
import pytest

import meshgen

from hm_gpu_util import GpuH, need_gpu

pytestmark = pytest.mark.gpu


def _dense(g):
    ex, H = g.export(), np.zeros((g.n, g.n))
    perm = g.perm()
    for off, (rb, re, cb, ce) in zip(ex["dense_off"], g.leaves(True)):
        H[np.ix_(perm[rb:re], perm[cb:ce])] = ex["dense"][off:off + (re - rb) * (ce - cb)].reshape(re - rb, ce - cb)
    return H


def test_touching_entries_of_a_tiny_mesh():
    # entries scale as the third power of the mesh.  Squares from 2^-128 on have 21 bits or more beside the smallest
    # float, their reciprocal roots half of that error: 2^-22 of each positive term
    need_gpu()
    V, T = meshgen.icosphere(2)
    scale, H = 2.0 ** -61.5, []
    for s in (1.0, scale):
        g = GpuH(V * s, T, leaf=20, eta=1.5, eps=1e-6)
        try:
            H.append(_dense(g) / s ** 3)
        finally:
            g.close()
    shared = (T[:, None, :, None] == T[None, :, None, :]).any(3).sum(2)
    for kind in (1, 2, 3):
        at = shared == kind
        assert (np.abs(H[1][at] - H[0][at]) <= 2.0 ** -21 * H[0][at]).all(), kind


def test_regular_entry_of_close_panels():
    # two panels one above the other at 2^-63.5: the seven terms of coinciding points are the whole entry but 1e-18 of it
    need_gpu()
    d = 2.0 ** -63.5
    V = np.array([[-1.0, -1, 0], [2, -1, 0], [-1, 2, 0]])
    V = np.concatenate([V, V + [0, 0, d]])
    g = GpuH(V, np.array([[0, 1, 2], [3, 4, 5]], dtype=np.int32), leaf=4, eta=1.5, eps=1e-6)
    try:
        H = _dense(g)
    finally:
        g.close()
    r = np.sqrt(15.0)
    w2 = (9 / 40) ** 2 + 3 * ((155 - r) / 1200) ** 2 + 3 * ((155 + r) / 1200) ** 2
    ref = 4.5 ** 2 / (4 * np.pi) * w2 / d
    assert np.abs(H[[0, 1], [1, 0]] - ref).max() <= 2.0 ** -20 * ref


@pytest.mark.parametrize("leaf", [1, 7, 9, 16, 100, 248])
def test_bf16_product_at_block_edges(orc, leaf):
    # against the oracle applying the operator with its factors rounded to BF16 (the near field is FP32): 2^-24 per entry
    # and addition, as for the FP32 copies
    torch = need_gpu()
    V, T = meshgen.bump_sphere(3, 1808)[:2]
    g = GpuH(V, np.ascontiguousarray(T[:1003]), leaf=leaf, eta=1.5, eps=1e-6, factor_dtype=2, dense_dtype=1)
    try:
        ex, perm, dl, al = g.export(), g.perm(), g.leaves(True), g.leaves(False)
        uw = torch.from_numpy(ex["uw"]).to(torch.bfloat16).to(torch.float64).numpy()
        x = np.random.default_rng(leaf).standard_normal(g.n)
        for trans in (0, 1):
            ref = np.empty(g.n)
            ref[perm] = orc.hmatvec_raw(g.n, dl, ex["dense_off"], ex["dense"], al, ex["rank"], ex["u_off"],
                                        ex["w_off"], uw, x[perm], trans=bool(trans))
            y = g.matvec(x, prec=2, trans=trans)
            assert np.linalg.norm(y - ref) <= 1e-5 * np.linalg.norm(ref)
    finally:
        g.close()
