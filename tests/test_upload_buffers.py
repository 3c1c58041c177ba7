"""Device arrays passed to soundings_upload may be written again as soon as it
returns, from any stream: the handle keeps its own copy.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# one block, one cluster, and the many-kernel build (for its soundings or, at a small
# cell side, for its cells)
@pytest.mark.parametrize("n,hint", [(3_000, 0), (20_000, 0), (60_000, 60), (262_144, 0), (262_144, 100), (300_000, 0)])
def test_depths_overwritten_on_return(n, hint):
    import torch

    import paper_2505_22675_gb300 as bg
    r = np.random.Generator(np.random.PCG64(n))
    x, y = (torch.from_numpy(r.integers(0, 50_000, n).astype(np.int32)).cuda() for _ in range(2))
    z = torch.from_numpy((3500 + r.normal(0, 5, n)).astype(np.float32)).cuda()
    kept = z.clone()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    ctx = bg.ctx_create(0)
    try:
        grid = bg.grid_create(ctx, 0, 0, 400, 125, 125)
        out = [torch.empty(125 * 125, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        for turn in range(12):
            z.copy_(kept)
            torch.cuda.synchronize()
            s = bg.soundings_upload(ctx, x, y, z, cell_cm_hint=hint, stream=a)
            if turn > 0:
                with torch.cuda.stream(b):
                    z.fill_(9_000.0)
            bg.interp_idw(s, grid, 8, 2.0, out[1], stream=a)
            bg.interp_okrige(s, grid, 8, bg.variogram(0, 0.25, 100.0, 50.0), out[2], stream=a)
            torch.cuda.synchronize()
            bg.soundings_destroy(s)
            if turn == 0:
                ref = [t.clone() for t in out]
            assert torch.equal(out[1], ref[1]) and torch.equal(out[2], ref[2])
        bg.grid_destroy(grid)
    finally:
        bg.ctx_destroy(ctx)
