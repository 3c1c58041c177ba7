"""GPU parity of the patch search where many soundings are at the same distance from a
node: lattices (fine ones, and coarse ones whose distances a key holds only in part) and
positions that hold several soundings. Neighbour lists are bit-exact: equal distances in
the order of upload.
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


def _lattice(nx, ny, step):
    """In shuffled order: the order of upload is not that of the cells."""
    r = _gen(step)
    x, y = np.meshgrid(np.arange(nx) * step, np.arange(ny) * step)
    p = r.permutation(x.size)
    return _with_depths(r, x.ravel()[p], y.ravel()[p])


def _doubled(n, w, m):
    """m soundings at every position."""
    r = _gen(m)
    x, y, p = np.repeat(r.integers(0, w, n // m), m), np.repeat(r.integers(0, w, n // m), m), r.permutation(n // m * m)
    return _with_depths(r, x[p], y[p])


CASES = {
    "lattice": (lambda: _lattice(70, 66, 200), GridSpec(-100, -100, 200, 69, 67)),
    "between": (lambda: _lattice(70, 66, 200), GridSpec(0, 0, 200, 69, 67)),
    "quarters": (lambda: _lattice(70, 66, 200), GridSpec(2_000, 2_000, 100, 61, 59)),
    "coarse": (lambda: _lattice(40, 40, 2_000), GridSpec(8_000, 8_000, 1_000, 57, 45)),
    "coarser": (lambda: _lattice(30, 30, 6_000), GridSpec(30_000, 30_000, 1_200, 50, 43)),
    "doubled": (lambda: _doubled(8_000, 20_000, 8), GridSpec(0, 0, 400, 47, 46)),
    "in_pairs": (lambda: _doubled(8_000, 20_000, 2), GridSpec(0, 0, 400, 47, 46)),
    "in_heaps": (lambda: _doubled(8_000, 20_000, 100), GridSpec(0, 0, 400, 47, 46)),
}


@pytest.mark.parametrize("k", [1, 3, 8, 13, 16, 32])
@pytest.mark.parametrize("name", CASES)
def test_neighbours_in_order(name, k):
    make, g = CASES[name]
    x, y, z = make()
    lib = Lib(x, y, z, g)
    try:
        d, nb = lib.idw(k, 2.0)
        _, _, kn = lib.okrige(k)
    finally:
        lib.close()
    qx, qy = oracle.grid_nodes(g.x0_cm, g.y0_cm, g.cell_cm, g.nx, g.ny)
    ref, ridx = oracle.idw(x, y, z, qx, qy, k, 2.0, want_idx=True)
    assert np.array_equal(nb, ridx) and np.array_equal(kn, ridx)
    assert_idw(d, ref)
