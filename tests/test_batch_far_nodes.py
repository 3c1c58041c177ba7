"""Batched tiles whose grids lie where the bound of a packed key ends: some nodes
are the packed search's, the rest the wide-key pass's, and every node is written
by one of them. Their grids must equal the per-grid calls bit for bit.
"""
import numpy as np
import pytest

import oracle
from gpu_util import Lib, assert_idw
from synth import GridSpec

pytestmark = pytest.mark.gpu

# 2^20 soundings (20 index bits) over 1 km: a squared distance fits a packed key
# up to 2^44 cm^2, 41.9 km; the grid's columns cross that line
N, SIDE = 1 << 20, 100_000
GRID = GridSpec(-(1 << 22) - 1_400, 48_000, 50, 64, 64)


@pytest.fixture(scope="module")
def soundings():
    r = np.random.Generator(np.random.PCG64(44))
    return (r.integers(0, SIDE, N).astype(np.int32), r.integers(0, SIDE, N).astype(np.int32),
            (3500 + r.normal(0, 5, N)).astype(np.float32))


@pytest.mark.parametrize("ppc", [1.0, 2.0])
@pytest.mark.parametrize("method,k", [(0, 1), (0, 5), (0, 9), (0, 12), (0, 16), (0, 20), (1, 3), (1, 12), (1, 20)])
def test_every_node_is_written(soundings, method, k, ppc):
    import torch

    import paper_2505_22675_gb300 as bg
    x, y, z = soundings
    lib = Lib(x, y, z, GRID)
    try:
        if method == 0:
            (d, nb), v = lib.idw(k, 2.0), None
        else:
            d, v, nb = lib.okrige(k, want_nbr=False)
        dev = [torch.from_numpy(a).cuda() for a in (x, y, z)]
        m = GRID.nx * GRID.ny
        bd, bv = torch.full((m,), -1.0, device="cuda"), torch.full((m,), -1.0, device="cuda")
        b = bg.batch_create(lib.ctx, [dict(
            x_cm=dev[0], y_cm=dev[1], z_m=dev[2], grid_spec=(GRID.x0_cm, GRID.y0_cm, GRID.cell_cm, GRID.nx, GRID.ny),
            method=method, k=k, power=2.0, vgm=bg.variogram(0, 0.25, 100.0, 50.0), depth_out=bd,
            var_out=bv if method == 1 else None)])
        bg.batch_set_cell_target(b, ppc)
        bg.batch_run(b)
        torch.cuda.synchronize()
        assert bg.batch_status(b) == 2  # the wide-key pass had nodes to take
        bg.batch_destroy(b)
        assert np.array_equal(bd.cpu().numpy().view(np.uint32), d.view(np.uint32))
        if method == 1:
            assert np.array_equal(bv.cpu().numpy().view(np.uint32), v.view(np.uint32))
    finally:
        lib.close()
    if method == 0:
        sel = np.random.default_rng(k).choice(m, 60, replace=False)
        qx, qy = oracle.grid_nodes(GRID.x0_cm, GRID.y0_cm, GRID.cell_cm, GRID.nx, GRID.ny)
        ref, ridx = oracle.idw(x, y, z, qx[sel], qy[sel], k, 2.0, want_idx=True)
        assert np.array_equal(nb[sel], ridx)
        assert_idw(d[sel], ref)
