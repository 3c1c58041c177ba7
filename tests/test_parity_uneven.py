"""GPU parity of the searches where the soundings lie unevenly: to one side, in clusters,
along lines, or nowhere near the grid. The patch search then takes its
radii from a node in the middle or leaves lanes to their own searches, and the search
by lanes widens its bound in steps.

Neighbour lists are bit-exact, depths within the IDW tolerance of tests/gpu_util.py.
"""
import numpy as np
import pytest

import oracle
from gpu_util import Lib, assert_idw
from synth import GridSpec

pytestmark = pytest.mark.gpu


def _gen(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _with_depths(r, x, y):
    return x.astype(np.int32), y.astype(np.int32), (3500 + r.normal(0, 5, x.size)).astype(np.float32)


def _one_side(n, w):
    """All but one of the soundings in the left half of a square."""
    r = _gen(n)
    return _with_depths(r, np.append(r.integers(0, w // 2, n), w), np.append(r.integers(0, w, n), w))


def _clusters(n, w, sd):
    r = _gen(n + 1)
    c, k = r.integers(0, w, (12, 2)), r.integers(0, 12, n)
    return _with_depths(r, *(np.clip(c[k, i] + r.normal(0, sd, n), 0, w - 1) for i in (0, 1)))


def _lines(per, w):
    """Four lines 250 m apart."""
    r = _gen(per)
    return _with_depths(r, r.integers(0, w, 4 * per), np.repeat(np.arange(4), per) * 25_000 + r.integers(-30, 31, 4 * per))


CASES = {
    "one_side": (lambda: _one_side(8_000, 30_000), GridSpec(0, 0, 500, 61, 59)),
    "one_side_dense": (lambda: _one_side(60_000, 30_000), GridSpec(9_000, 0, 300, 45, 37)),
    "clusters": (lambda: _clusters(12_000, 40_000, 700), GridSpec(0, 0, 600, 67, 66)),
    "sharp_clusters": (lambda: _clusters(12_000, 40_000, 90), GridSpec(0, 0, 500, 50, 41)),
    "lines": (lambda: _lines(2_500, 100_000), GridSpec(20_000, -4_000, 700, 45, 120)),
    "dense_lines": (lambda: _lines(20_000, 60_000), GridSpec(20_000, -4_000, 500, 45, 150)),
    "off_the_data": (lambda: _clusters(5_000, 20_000, 4_000), GridSpec(-31_000, -12_000, 400, 43, 50)),
    "far_off": (lambda: _clusters(5_000, 20_000, 4_000), GridSpec(700_000, 300_000, 400, 33, 30)),
    "partly_off": (lambda: _clusters(5_000, 20_000, 4_000), GridSpec(-90_000, -20_000, 2_000, 60, 40)),
}


@pytest.mark.parametrize("k", [3, 8, 13, 16, 32])
@pytest.mark.parametrize("name", CASES)
def test_neighbours_and_depths(name, k):
    import torch
    make, g = CASES[name]
    x, y, z = make()
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    lib = Lib(x, y, z, g)
    try:
        d, nb = lib.idw(k, 2.0)
        _, _, kn = lib.okrige(k)
        pd = torch.empty(qx.size, device="cuda")  # (by lanes of a warp each)
        pn = torch.empty(qx.size * k, dtype=torch.int32, device="cuda")
        lib.bg.interp_idw_points(lib.s, torch.from_numpy(qx.astype(np.int32)).cuda(),
                                 torch.from_numpy(qy.astype(np.int32)).cuda(), k, 2.0, pd, pn)
        torch.cuda.synchronize()
    finally:
        lib.close()
    ref, ridx = oracle.idw(x, y, z, qx, qy, k, 2.0, want_idx=True)
    assert np.array_equal(nb, ridx) and np.array_equal(kn, ridx)
    assert np.array_equal(pn.cpu().numpy().reshape(-1, k), ridx)
    assert_idw(d, ref)
    assert np.array_equal(d.view(np.uint32), pd.cpu().numpy().view(np.uint32))


@pytest.mark.parametrize("k", [8, 16, 32])
def test_strips_of_patches(k):
    """A grid large enough for strips of several patches, over lines: the radius of the
    patch before misses or holds too much."""
    x, y, z = _lines(6_000, 150_000)
    g = GridSpec(0, -5_000, 100, 1_500, 900)
    lib = Lib(x, y, z, g)
    try:
        d, nb = lib.idw(k, 2.0)
    finally:
        lib.close()
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    sel = _gen(k).choice(qx.size, 4_000, replace=False)
    ref, ridx = oracle.idw(x, y, z, qx[sel], qy[sel], k, 2.0, want_idx=True)
    assert np.array_equal(nb[sel], ridx)
    assert_idw(d[sel], ref)
