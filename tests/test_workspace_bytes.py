"""Device workspace of grids of few planes, of small capacities and of ordinary
ones (host only): no more than these grids have needed before, so that a
caller's buffer keeps its size; and the wall columns of a pipe stay within the
capacity of their tables."""
import numpy as np
import pytest

# (nx, ny, nz, storage, capacity of links, markers and sites, lattice): bytes
CEILINGS = {
    (16, 16, 4, 0, 1, 19): 1656576,
    (64, 64, 4, 1, 1, 19): 4786944,
    (64, 64, 4, 2, 5000, 19): 5768192,
    (148, 148, 1, 1, 0, 19): 27560448,
    (148, 148, 1, 2, 1, 19): 4569088,
    (148, 148, 4, 0, 1, 27): 53761280,
    (148, 148, 4, 1, 0, 19): 47111424,
    (148, 148, 16, 1, 1, 27): 100360704,
    (148, 148, 438, 1, 0, 19): 2875652608,
    (300, 300, 4, 2, 0, 19): 91451392,
    (1000, 1000, 4, 1, 1, 19): 819764224,
    (64, 64, 64, 0, 1, 19): 94679296,
    (256, 256, 256, 1, 0, 19): 4861509376,
}


@pytest.fixture(scope="module")
def lbm():
    from paper_1906_05448_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


@pytest.mark.parametrize("key", CEILINGS)
def test_no_more_than_before(lbm, key):
    nx, ny, nz, storage, cap, lattice = key
    g = lbm.make_grid(nx, ny, nz, storage=storage, max_links=cap, max_markers=cap, max_sites=cap, lattice=lattice)
    assert 0 < lbm.workspace_bytes(g) <= CEILINGS[key]


def test_wall_columns_fit_their_tables():
    rng = np.random.default_rng(0)
    for nx in [*range(4, 48), 80, 101, 148, 256]:
        for ny in {nx, nx + 1, 2 * nx}:
            x, y = np.arange(nx) - 0.5 * (nx - 1), np.arange(ny) - 0.5 * (ny - 1)
            top = 0.5 * min(nx, ny)
            for R in [1.001, top, top - 0.5, *rng.uniform(1.0, top, 8)]:
                if not 1.0 < R <= top:
                    continue
                solid = x[None, :] ** 2 + y[:, None] ** 2 >= R * R
                near = np.zeros_like(solid)
                for a in (-1, 0, 1):
                    for b in (-1, 0, 1):
                        near |= np.roll(solid, (a, b), (0, 1))
                assert np.count_nonzero(~solid & near) <= min(nx * ny, 2 * (nx + ny))
