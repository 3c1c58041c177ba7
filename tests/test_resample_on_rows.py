"""Output grids whose nodes are nodes of the source (the same grid, and grids shifted by
whole cells, partly off it): the row kernel against the point entry point, value for
value (up to the sign of a zero) and code for code, with missing and infinite nodes.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", [0, 1])
@pytest.mark.parametrize("dx,dy,nx,ny", [(0, 0, 1_028, 37), (4, 3, 1_028, 37), (-8, -5, 64, 60), (1_020, 0, 32, 9),
                                         (0, 36, 1_028, 1), (0, 30, 512, 11)])
def test_nodes_on_nodes(method, dx, dy, nx, ny):
    import torch

    import paper_2505_22675_gb300 as bg
    spec = (300, -500, 200, 1_028, 37)
    r = np.random.Generator(np.random.PCG64(7))
    src = (3500 + r.normal(0, 5, 1_028 * 37)).astype(np.float32)
    src[r.random(src.size) < 0.1] = np.nan
    src[r.random(src.size) < 0.01] = np.inf
    src[r.random(src.size) < 0.01] = 0.0
    z = torch.from_numpy(src).cuda()
    out = (spec[0] + 200 * dx, spec[1] + 200 * dy, 200, nx, ny)
    qx, qy = oracle.grid_nodes(*out)
    m = nx * ny
    got, ref = torch.full((m,), -7.0, device="cuda"), torch.full((m,), -7.0, device="cuda")
    gh, rh = torch.full((m,), 9, dtype=torch.int8, device="cuda"), torch.full((m,), 9, dtype=torch.int8, device="cuda")
    bg.resample_grid(z, spec, method, out, got, gh)
    bg.resample_points(z, spec, method, torch.from_numpy(qx.astype(np.int32)).cuda(),
                       torch.from_numpy(qy.astype(np.int32)).cuda(), ref, rh)
    torch.cuda.synchronize()
    assert torch.equal(gh, rh)
    assert np.array_equal(got.cpu().numpy(), ref.cpu().numpy(), equal_nan=True)
