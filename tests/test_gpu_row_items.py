"""The row pass of the product of the reduced copies with many right-hand sides
at the edges of its work items: leaves of less than one tile of 16 rows, of
three and five tiles and one row more, of more than 80 rows (items of 64 rows
and a remainder), on a ragged open surface whose Morton order tears clusters
apart (panels of more than twice the mean width: one item per tile of rows).

Each row within 2^-14 of the row sum of |H||x| from the oracle applying the
exported operator: x and the FP32 entries are pairs of BF16 numbers (2^-17 of
each value, twice for t = W x), their low-low product (2^-16) is left out, and
the FP32 sums add less than 2^-16."""
import numpy as np
import pytest

import meshgen

from hm_gpu_util import GpuH, need_gpu
from test_gpu_df import abs_operator, oracle_apply

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [7, 48, 49, 80, 81, 130, 254])
def test_items(orc, leaf):
    need_gpu()
    V, T = meshgen.bump_sphere(4, 1808)[:2]
    g = GpuH(V, np.ascontiguousarray(T[:3011]), leaf=leaf, eta=1.5, eps=1e-6, factor_dtype=1, dense_dtype=1)
    try:
        torch, hm, ex = g.torch, g.hm, g.export()
        X = np.random.default_rng(leaf).standard_normal((17, g.n))
        ref, mag = oracle_apply(orc, g, ex, X), oracle_apply(orc, g, abs_operator(ex), np.abs(X))
        Xd = torch.from_numpy(X).cuda()
        Y = torch.full_like(Xd, float("nan"))
        hm.hm_matvec_block(g.A, Xd, Y, prec=hm.HM_F32)
        torch.cuda.synchronize()
        assert (np.abs(Y.cpu().numpy() - ref) <= 2.0 ** -14 * mag).all()
    finally:
        g.close()
