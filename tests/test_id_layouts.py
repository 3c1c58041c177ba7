"""The two layouts of the neighbour ids and the kernels that write and read them: the
same grids, bit for bit, whichever is taken, for both variogram models and every
system size, next to the lines where a search changes hands.
"""
import numpy as np
import pytest

import oracle
from gpu_util import Lib
from synth import GridSpec

pytestmark = pytest.mark.gpu


def _uniform(seed, n, w_cm, h_cm):
    r = np.random.Generator(np.random.PCG64(seed))
    return (r.integers(0, w_cm, n).astype(np.int32), r.integers(0, h_cm, n).astype(np.int32),
            (3500 + r.normal(0, 5, n)).astype(np.float32))


def _bits(t):
    return t.cpu().numpy().view(np.uint32)


def _run_tiles(bg, torch, ctx, xyz, specs):
    out = [[torch.full((nx * ny,), -1.0, device="cuda") for _ in range(2)] for _, _, (_, _, _, nx, ny) in specs]
    b = bg.batch_create(ctx, [dict(x_cm=xyz[0], y_cm=xyz[1], z_m=xyz[2], grid_spec=g, method=1, k=k,
                                   vgm=bg.variogram(model, 0.25, 100.0, 50.0), depth_out=d, var_out=v)
                              for (k, model, g), (d, v) in zip(specs, out)])
    held = bg.ctx_device_bytes(ctx)
    bg.batch_run(b)
    torch.cuda.synchronize()
    bg.batch_destroy(b)
    return out, held


def _direct(bg, torch, ctx, xyz, k, model, g):
    s, grid = bg.soundings_upload(ctx, *xyz), bg.grid_create(ctx, *g)
    d, v = (torch.empty(g[3] * g[4], device="cuda") for _ in range(2))
    bg.interp_okrige(s, grid, k, bg.variogram(model, 0.25, 100.0, 50.0), d, v)
    torch.cuda.synchronize()
    bg.soundings_destroy(s)
    bg.grid_destroy(grid)
    return d, v


def test_batch_of_both_models_and_every_size():
    import torch

    import paper_2505_22675_gb300 as bg
    xyz = [torch.from_numpy(a).cuda() for a in _uniform(31, 5_000, 8_000, 8_000)]
    specs = [(k, model, (0, 0, 200, nx, 37)) for k in (3, 8, 13, 16, 20, 32) for model, nx in ((0, 40), (1, 33), (1, 5))]
    ctx = bg.ctx_create(0)
    try:
        out, _ = _run_tiles(bg, torch, ctx, xyz, specs)
        for spec, got in zip(specs, out):
            for a, b in zip(got, _direct(bg, torch, ctx, xyz, *spec)):
                assert np.array_equal(_bits(a), _bits(b)), spec
    finally:
        bg.ctx_destroy(ctx)


def test_batch_under_a_budget_without_room_for_slots():
    import torch

    import paper_2505_22675_gb300 as bg
    xyz = [torch.from_numpy(a).cuda() for a in _uniform(32, 5_000, 8_000, 8_000)]
    specs = [(32, 0, (0, 0, 8, 15, 1_000)), (13, 1, (0, 0, 8, 15, 1_000))]  # 16 slots a row
    rows, slots = (sum(4 * k * w * 1_000 for k, _, _ in specs) for w in (15, 16))
    ctx = bg.ctx_create(0)
    try:
        ref, held = _run_tiles(bg, torch, ctx, xyz, specs)
    finally:
        bg.ctx_destroy(ctx)
    ctx = bg.ctx_create(0, held - (slots - rows) // 2)
    try:
        out, less = _run_tiles(bg, torch, ctx, xyz, specs)
    finally:
        bg.ctx_destroy(ctx)
    assert less == held - (slots - rows)
    for a, b in zip(out, ref):
        assert all(np.array_equal(_bits(p), _bits(q)) for p, q in zip(a, b))


# the longest lists of lanes of a warp each, and the next of a thread each
@pytest.mark.parametrize("k,m", [(5, 34_048), (5, 34_049), (12, 87_552), (12, 87_553), (32, 58_368), (32, 58_369)])
@pytest.mark.parametrize("model", [0, 1])
def test_points_with_and_without_lists(k, m, model):
    import torch

    import paper_2505_22675_gb300 as bg
    x, y, z = _uniform(33, 20_000, 30_000, 30_000)
    r = np.random.Generator(np.random.PCG64(m))
    q = [r.integers(-3_000, 33_000, m).astype(np.int32) for _ in range(2)]
    q[0][::1_009] = 1 << 30  # out of range
    lib = Lib(x, y, z, GridSpec(0, 0, 100, 4, 4))
    try:
        qx, qy = (torch.from_numpy(a).cuda() for a in q)
        vgm = bg.variogram(model, 0.25, 100.0, 50.0)
        d, v, d2, v2 = (torch.empty(m, device="cuda") for _ in range(4))
        nb = torch.empty(m * k, dtype=torch.int32, device="cuda")
        bg.interp_okrige_points(lib.s, qx, qy, k, vgm, d, v, nb)
        bg.interp_okrige_points(lib.s, qx, qy, k, vgm, d2, v2)
        torch.cuda.synchronize()
        assert np.array_equal(_bits(d), _bits(d2)) and np.array_equal(_bits(v), _bits(v2))
        nb = nb.cpu().numpy().reshape(m, k)
    finally:
        lib.close()
    assert np.isnan(d.cpu().numpy()[::1_009]).all() and (nb[::1_009] == -1).all()
    sel = np.setdiff1d(np.random.default_rng(k).choice(m, 300, replace=False), np.arange(0, m, 1_009))
    assert np.array_equal(nb[sel], oracle.idw(x, y, z, q[0][sel], q[1][sel], k, 2.0, want_idx=True)[1])


@pytest.mark.parametrize("k", [3, 12, 20, 32])
def test_far_nodes_in_slots(k):
    """A grid that lies across the line where the bound of a packed key ends (2^20
    soundings, 42 km): the wide-key pass writes its nodes into slots."""
    x, y, z = _uniform(44, 1 << 20, 100_000, 100_000)
    g = GridSpec(-(1 << 22) - 1_400, 48_000, 50, 64, 64)
    lib = Lib(x, y, z, g)
    try:
        d, v, nb = lib.okrige(k)
        d2, v2, _ = lib.okrige(k, want_nbr=False)
    finally:
        lib.close()
    assert np.array_equal(d.view(np.uint32), d2.view(np.uint32))
    assert np.array_equal(v.view(np.uint32), v2.view(np.uint32))
    sel = np.random.default_rng(k).choice(g.nx * g.ny, 60, replace=False)
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    assert np.array_equal(nb[sel], oracle.idw(x, y, z, qx[sel], qy[sel], k, 2.0, want_idx=True)[1])
