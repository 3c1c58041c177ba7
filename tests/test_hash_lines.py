"""Uploads on both sides of the sizes where the hash build changes hands: one cluster,
its bounding box alone by one cluster, many kernels.
"""
import numpy as np
import pytest

import oracle
from gpu_util import Lib, assert_idw
from synth import GridSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [98_304, 98_305, 262_144, 262_145])
@pytest.mark.parametrize("on_device", [True, False])
def test_hash_builds_at_their_lines(n, on_device):
    r = np.random.Generator(np.random.PCG64(n))
    x, y = (r.integers(0, 60_000, n).astype(np.int32) for _ in range(2))
    z = (3500 + r.normal(0, 5, n)).astype(np.float32)
    z[::97] = np.nan
    g = GridSpec(25_000, 1_000, 900, 13, 60)
    lib = Lib(x, y, z, g, on_device=on_device)
    try:
        d, nb = lib.idw(8, 2.0)
    finally:
        lib.close()
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    ref, ridx = oracle.idw(x, y, z, qx, qy, 8, 2.0, want_idx=True)
    assert np.array_equal(nb, ridx)
    assert_idw(d, ref)
