"""GPU parity of the patch search (one warp per 8 x 4 nodes) against the FP64
oracle, at the sizes where it changes course: patch remainders, equal distances
everywhere, more soundings than its list holds, gaps wider than its first
radius, distances beyond its keys, clusters at one position.

Neighbour lists are bit-exact, depths within the IDW tolerance of
tests/gpu_util.py.
"""
import numpy as np
import pytest

import oracle
from gpu_util import Lib, assert_idw
from synth import GridSpec

pytestmark = pytest.mark.gpu


def _uniform(seed, n, w_cm, h_cm):
    r = np.random.Generator(np.random.PCG64(seed))
    return (r.integers(0, w_cm, n).astype(np.int32), r.integers(0, h_cm, n).astype(np.int32),
            (3500 + r.normal(0, 5, n)).astype(np.float32))


def _lattice(nx, ny, step):
    x, y = np.meshgrid(np.arange(nx) * step, np.arange(ny) * step)
    z = 3500 + 0.01 * x + 0.02 * y
    return x.ravel().astype(np.int32), y.ravel().astype(np.int32), z.ravel().astype(np.float32)


def _gap(seed):
    """Two strips of soundings, 40 m deep and 130 m apart."""
    x, y, z = _uniform(seed, 12_000, 30_000, 8_000)
    return x, np.where(y < 4_000, y, y + 13_000).astype(np.int32), z


def _cluster(seed):
    """A scatter with 300 soundings at one position and 40 at another."""
    x, y, z = _uniform(seed, 4_000, 6_000, 6_000)
    x[:300], y[:300] = 3_000, 3_000
    x[300:340], y[300:340] = 1_111, 4_444
    return x, y, z


CASES = {
    "one_node": (lambda: _uniform(1, 3_000, 6_000, 6_000), GridSpec(2_000, 2_000, 100, 1, 1)),
    "whole_patch": (lambda: _uniform(2, 3_000, 6_000, 6_000), GridSpec(1_000, 1_000, 100, 8, 4)),
    "remainders": (lambda: _uniform(3, 3_000, 6_000, 6_000), GridSpec(500, 700, 150, 33, 17)),
    "past_the_edge": (lambda: _uniform(4, 3_000, 6_000, 6_000), GridSpec(-9_000, -3_000, 250, 70, 30)),
    "lattice": (lambda: _lattice(60, 60, 100), GridSpec(-50, -50, 100, 57, 59)),
    "half_lattice": (lambda: _lattice(60, 60, 100), GridSpec(0, 0, 100, 41, 23)),
    "many_per_node": (lambda: _uniform(5, 60_000, 4_000, 4_000), GridSpec(0, 0, 200, 20, 19)),
    "near_capacity": (lambda: _uniform(6, 12_000, 4_000, 4_000), GridSpec(0, 0, 100, 40, 39)),
    "gap": (lambda: _gap(7), GridSpec(0, 0, 200, 150, 105)),
    "sparse": (lambda: _uniform(8, 3_000, 200_000, 200_000), GridSpec(50_000, 50_000, 600, 45, 33)),
    "very_sparse": (lambda: _uniform(11, 2_000, 400_000, 400_000), GridSpec(100_000, 150_000, 1_300, 31, 27)),
    "cluster": (lambda: _cluster(9), GridSpec(0, 0, 150, 40, 40)),
    "few": (lambda: _uniform(10, 40, 6_000, 6_000), GridSpec(0, 0, 300, 20, 20)),
}


@pytest.mark.parametrize("k", [3, 8, 16, 32])
@pytest.mark.parametrize("name", CASES)
def test_idw_neighbours_and_depths(name, k):
    make, g = CASES[name]
    x, y, z = make()
    lib = Lib(x, y, z, g)
    try:
        d, nb = lib.idw(k, 2.0)
    finally:
        lib.close()
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    ref, ridx = oracle.idw(x, y, z, qx, qy, k, 2.0, want_idx=True)
    assert np.array_equal(nb, ridx)
    assert_idw(d, ref)


@pytest.mark.parametrize("model,nugget,k", [(0, 0.25, 32), (0, 0.25, 15), (0, 0.25, 7), (1, 0.25, 32), (1, 0.25, 13),
                                            (0, 0.25, 3)])
@pytest.mark.parametrize("name", ["one_node", "whole_patch", "remainders", "past_the_edge", "many_per_node", "gap",
                                  "sparse", "few"])
def test_kriging_systems_of_every_size(name, model, nugget, k):
    """Systems of k unknowns in tiles of 8 (whole and padded), by patches and by
    rows, with the neighbour lists and without (the two layouts of the ids)."""
    from gpu_util import assert_okrige
    make, g = CASES[name]
    x, y, z = make()
    lib = Lib(x, y, z, g)
    try:
        d, v, nb = lib.okrige(k, model, nugget, 100.0, 50.0)
        d2, v2, _ = lib.okrige(k, model, nugget, 100.0, 50.0, want_nbr=False)
    finally:
        lib.close()
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    rd, rv, ridx = oracle.okrige(x, y, z, qx, qy, k, model, nugget, 100.0, 50.0, want_idx=True)
    assert np.array_equal(nb, ridx)
    assert_okrige(d, v, rd, rv, nugget)
    assert np.array_equal(d, d2) and np.array_equal(v, v2)


@pytest.mark.parametrize("k", [3, 8, 13, 32])
@pytest.mark.parametrize("rows", [170, 171, 291, 292, 437, 438])
@pytest.mark.parametrize("name", ["uniform", "lattice", "gap"])
def test_queries_by_warps_and_by_threads(name, rows, k):
    """The largest grids of lanes of a warp each where patches do not serve (200 x
    170 nodes for k <= 8, x 437 up to 16, x 291 beyond) and the next of a thread each, as a grid of many soundings per node and as a list of points."""
    import torch
    make, cell = {"uniform": (lambda: _uniform(21, 400_000, 20_000, 29_200), 100),
                  "lattice": (lambda: _lattice(400, 600, 50), 100),
                  "gap": (lambda: _gap(22), 150)}[name]
    x, y, z = make()
    g = GridSpec(0, 0, cell, 200, rows)
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    lib = Lib(x, y, z, g)
    try:
        d, nb = lib.idw(k, 2.0)
        pd = torch.empty(qx.size, device="cuda")
        pn = torch.empty(qx.size * k, dtype=torch.int32, device="cuda")
        lib.bg.interp_idw_points(lib.s, torch.from_numpy(qx.astype(np.int32)).cuda(),
                                 torch.from_numpy(qy.astype(np.int32)).cuda(), k, 2.0, pd, pn)
        _, _, kn = lib.okrige(k, 0, 0.25, 100.0, 50.0)
        torch.cuda.synchronize()
    finally:
        lib.close()
    assert np.array_equal(d.view(np.uint32), pd.cpu().numpy().view(np.uint32))
    assert np.array_equal(nb, pn.cpu().numpy().reshape(-1, k)) and np.array_equal(nb, kn)
    sel = np.random.default_rng(k).choice(qx.size, 1_500, replace=False)
    ref, ridx = oracle.idw(x, y, z, qx[sel].astype(np.int32), qy[sel].astype(np.int32), k, 2.0, want_idx=True)
    assert np.array_equal(nb[sel], ridx)
    assert_idw(d[sel], ref)


@pytest.mark.parametrize("k", [12, 32])
@pytest.mark.parametrize("range_m", [0.05, 2.0, 30.0, 400.0])
def test_exponential_model_at_every_range(range_m, k):
    """Entries from h / a << 1 (where 1 - exp(-h / a) cancels) to h / a > 25
    (where it is 1)."""
    from gpu_util import assert_okrige
    x, y, z = _uniform(3, 3_000, 8_000, 8_000)
    g = GridSpec(0, 0, 200, 41, 37)
    lib = Lib(x, y, z, g)
    try:
        d, v, _ = lib.okrige(k, 1, 0.25, 100.0, range_m, want_nbr=False)
    finally:
        lib.close()
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    rd, rv = oracle.okrige(x, y, z, qx, qy, k, 1, 0.25, 100.0, range_m)[:2]
    assert_okrige(d, v, rd, rv, 0.25)


@pytest.mark.parametrize("n,w,h,hint", [(4_096, 8_000, 8_000, 0), (4_097, 8_000, 8_000, 0), (9_000, 900_000, 40, 0),
                                        (9_000, 40, 900_000, 0), (30_000, 20_000, 20_000, 87), (30_000, 20_000, 20_000, 80),
                                        (262_144, 60_000, 60_000, 400), (262_145, 60_000, 60_000, 400),
                                        (5_000, 3, 3, 0)])
def test_hash_builds_of_every_size(n, w, h, hint):
    """One block, one cluster and the multi-kernel build: sizes on both sides of
    their limits (soundings, cells), one row or column of cells, a single cell."""
    x, y, z = _uniform(n, n, w, h)
    z[::97] = np.nan
    g = GridSpec(w // 3, h // 3, 2 * max(1, max(w, h) // 400), 9, 5)
    lib = Lib(x, y, z, g, cell_hint=hint)
    try:
        d, nb = lib.idw(8, 2.0)
    finally:
        lib.close()
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    ref, ridx = oracle.idw(x, y, z, qx, qy, 8, 2.0, want_idx=True)
    assert np.array_equal(nb, ridx)
    assert_idw(d, ref)
