"""Device memory that a kriging call takes for its neighbour ids, 4 k bytes a node:
none beside the caller's nbr_out, and whole 8 x 4 patches of nodes only where a grid
fills them.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

K = 32
SHAPES = [(1, 1 << 20), (1 << 20, 1), (3, 1 << 18), (1 << 17, 9), (1024, 1024)]


def _soundings(torch):
    r = np.random.Generator(np.random.PCG64(3))
    n = 50_000
    return [torch.from_numpy(a).cuda() for a in (
        r.integers(0, 100_000, n).astype(np.int32), r.integers(0, 100_000, n).astype(np.int32),
        (3500 + r.normal(0, 5, n)).astype(np.float32))]


@pytest.mark.parametrize("lists", [False, True])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_ids_of_a_grid(nx, ny, lists):
    """Device memory that one call makes the context's pool take."""
    import torch

    import paper_2505_22675_gb300 as bg
    xyz = _soundings(torch)
    m = nx * ny
    d, v = torch.empty(m, device="cuda"), torch.empty(m, device="cuda")
    nb = torch.empty(m * K, dtype=torch.int32, device="cuda") if lists else None
    vgm = bg.variogram(0, 0.25, 100.0, 50.0)
    ctx = bg.ctx_create(0)
    try:
        s = bg.soundings_upload(ctx, *xyz)
        small = bg.grid_create(ctx, 0, 0, 2, 16, 16)
        bg.interp_okrige(s, small, K, vgm, d, v)  # the kernels are loaded
        grid = bg.grid_create(ctx, 0, 0, 2, nx, ny)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        bg.interp_okrige(s, grid, K, vgm, d, v, nb)
        torch.cuda.synchronize()
        taken = before - torch.cuda.mem_get_info()[0]
        for g in (small, grid):
            bg.grid_destroy(g)
        bg.soundings_destroy(s)
    finally:
        bg.ctx_destroy(ctx)
    assert taken <= (0 if lists else 1.1 * 4 * K * m) + (96 << 20)  # the pool maps whole blocks


@pytest.mark.parametrize("nx,ny", [(nx // 16 if nx > ny else nx, ny // 16 if ny >= nx else ny) for nx, ny in SHAPES])
def test_ids_of_a_batch(nx, ny):
    import torch

    import paper_2505_22675_gb300 as bg
    x, y, z = _soundings(torch)
    d, v = torch.empty(nx * ny, device="cuda"), torch.empty(nx * ny, device="cuda")
    ctx = bg.ctx_create(0)
    try:
        held = []
        for method in (0, 1):
            b = bg.batch_create(ctx, [dict(x_cm=x, y_cm=y, z_m=z, grid_spec=(0, 0, 2, nx, ny), method=method, k=K,
                                           depth_out=d, var_out=v)])
            held.append(bg.ctx_device_bytes(ctx))
            bg.batch_destroy(b)
    finally:
        bg.ctx_destroy(ctx)
    assert held[1] - held[0] <= 1.1 * 4 * K * nx * ny + 4096
