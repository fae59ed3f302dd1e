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
from test_gpu_fx import _check

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
