"""The one-right-hand-side product at the edges of its blocks: eight rows per
CTA in the row pass, 128 threads' columns per CTA in the column pass.  Leaves
of 1, 7, 9, 16, 100 and 248 rows (less than, just above and a multiple of
eight rows; panels of one to many parts), an open surface with a ragged panel
count, both directions.  FP64: within 1e-12 of the oracle applying the exported
operator (sums of at most ~2,000 terms in another order); FP32 copies: within
1e-5 of the FP64 product (2^-24 per entry and addition)."""
import numpy as np
import pytest

import meshgen

from hm_gpu_util import GpuH, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [1, 7, 9, 16, 100, 248])
def test_product_at_block_edges(orc, leaf):
    need_gpu()
    V, T = meshgen.bump_sphere(3, 1808)[:2]
    g = GpuH(V, np.ascontiguousarray(T[:1003]), leaf=leaf, eta=1.5, eps=1e-6, factor_dtype=1, dense_dtype=1)
    try:
        ex, perm, dl, al = g.export(), g.perm(), g.leaves(True), g.leaves(False)
        x = np.random.default_rng(leaf).standard_normal(g.n)
        for trans in (0, 1):
            ref = np.empty(g.n)
            ref[perm] = orc.hmatvec_raw(g.n, dl, ex["dense_off"], ex["dense"], al, ex["rank"], ex["u_off"],
                                        ex["w_off"], ex["uw"], x[perm], trans=bool(trans))
            y = g.matvec(x, trans=trans)
            assert np.linalg.norm(y - ref) <= 1e-12 * np.linalg.norm(ref)
            y32 = g.matvec(x, prec=1, trans=trans)
            assert np.linalg.norm(y32 - y) <= 1e-5 * np.linalg.norm(y)
    finally:
        g.close()
