"""Kriging on a device with room for the neighbour ids in rows, but not for them in
whole-patch slots: the rows are taken.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

K, NX, NY = 32, 15, 1 << 23  # 16 slots of a row of 15 nodes
ROWS, SLOTS = 4 * K * NX * NY, 4 * K * (NX + 1) * NY


def test_batch_of_one_tile():
    import torch

    import paper_2505_22675_gb300 as bg
    r = np.random.Generator(np.random.PCG64(5))
    x, y = (torch.from_numpy(r.integers(0, 4_000, 2_000).astype(np.int32)).cuda() for _ in range(2))
    z = torch.from_numpy((3500 + r.normal(0, 5, 2_000)).astype(np.float32)).cuda()
    d = torch.empty(NX * NY, device="cuda")
    ctx = bg.ctx_create(0)
    hog = None
    try:
        tile = dict(x_cm=x, y_cm=y, z_m=z, grid_spec=(0, 0, 2, NX, NY), method=1, k=K, depth_out=d)
        bg.batch_destroy(bg.batch_create(ctx, [dict(tile, grid_spec=(0, 0, 2, 8, 8))]))  # kernels loaded
        torch.cuda.synchronize()
        room = (ROWS + SLOTS) // 2
        hog = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
        b = bg.batch_create(ctx, [tile])
        assert ROWS <= bg.ctx_device_bytes(ctx) < SLOTS
        bg.batch_destroy(b)
    finally:
        del hog
        torch.cuda.empty_cache()
        bg.ctx_destroy(ctx)
