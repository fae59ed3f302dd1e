"""The set-up's sorts and scans at the edges of their tiles: 2,048 keys per sort
tile, up to 64 tiles whose counts every tile adds up itself and one more, 4,096
values per scan tile.  Random triangles: the order of the panels is the oracle's
Morton order, the block tree the oracle's, both exactly."""
import numpy as np
import pytest

from hm_gpu_util import GpuH, as_set, need_gpu, split_dense_rows

pytestmark = pytest.mark.gpu


def soup(n):
    rng = np.random.default_rng(n)
    V = rng.standard_normal((n + 2, 3))
    i = np.arange(n, dtype=np.int32)
    return V, np.ascontiguousarray(np.stack([i, i + 1, i + 2], axis=1))


@pytest.mark.parametrize("n", [2, 2047, 2048, 2049, 4097, 64 * 2048, 64 * 2048 + 1])
def test_panel_order(orc, n):
    need_gpu()
    V, T = soup(n)
    g = GpuH(V, T, leaf=120, eta=1.5, eps=None)
    try:
        ref = orc.morton_order(orc.morton_codes(orc.panel_geometry(V, T)[0]))
        assert np.array_equal(g.perm(), ref)
    finally:
        g.close()


@pytest.mark.parametrize("n,leaf", [(1200, 7), (4097, 60)])
def test_block_tree(orc, n, leaf):
    need_gpu()
    V, T = soup(n)
    tr = orc.Tree(V, T, leaf, 1.5)
    g = GpuH(V, T, leaf=leaf, eta=1.5, eps=None)
    try:
        assert as_set(g.leaves(False)) == as_set(tr.adm)
        assert as_set(g.leaves(True)) == as_set(split_dense_rows(tr.dense, leaf))
    finally:
        g.close()
