"""Spheres at the edges of their kernels. IBM forcing: one block per particle
with the box of its markers in shared memory, up to the radius where two such
boxes fit an SM, and the kernels that walk marker by marker beyond it; the
support flags by box rows of up to 32 cells and beyond; boxes that wrap
around the grid's faces or are as wide as the grid; odd extents; several
radii together.

Interpolated bounce-back: the box passes and the momentum-exchange sums over
boxes of less and more than one round, and blocks of both sizes (one particle
or a few, and more than an SM count of them).

Tolerances are those of the other IBM comparisons with the oracle (sums in
another order, differences of nearly equal sums): FP64 1e-10 of the field,
1e-8 of the force; FP32 1e-5 of the field, 1e-5 of 2 max|u| for the force.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_05448_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


# (nz, ny, nx), centres (x, y, z), radii
CASES = {
    "smallest": ((6, 7, 9), [[8.7, 0.2, 5.9]], [0.6]),
    "grid_wide_box": ((13, 14, 17), [[0.1, 6.5, 12.9]], [4.0]),
    "wider_than_the_grid": ((13, 13, 13), [[6.3, 12.8, 0.4]], [4.05]),
    "corner_and_mixed_radii": ((22, 19, 27), [[26.9, 18.8, 21.7], [13.2, 9.1, 10.6]], [2.3, 4.5]),
    "largest_box_of_a_block": ((21, 18, 23), [[3.3, 17.5, 8.0]], [5.0]),
    "marker_by_marker": ((21, 19, 23), [[3.3, 17.5, 8.0]], [6.7]),
    "rows_of_32": ((32, 33, 31), [[30.2, 3.5, 17.75]], [13.4]),
    "rows_beyond_32": ((34, 35, 36), [[30.2, 3.5, 17.75]], [14.5]),
}


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("case", CASES)
def test_ibm_spheres_edges(lbm, case, storage):
    shape, X, R = CASES[case]
    nz, ny, nx = shape
    X, R = np.array(X), np.array(R)
    n = len(R)
    g = lbm.Lattice(nx, ny, nz, 0.62, storage=lbm.STORAGE[storage], rates=oracle.RATES_DHUMIERES, max_particles=n,
                    max_sites=nx * ny * nz, max_markers=int(sum(13 * r * r + 40 for r in R)))
    o = oracle.Sim(nx, ny, nz, 0.62, rates=oracle.RATES_DHUMIERES)
    u = workloads.noise_velocity(shape, 0.02, seed=5)
    U, W = np.full((n, 3), 0.01), np.full((n, 3), -0.002)
    for s in (g, o):
        s.init_velocity(u)
        s.add_spheres(X, R, density_ratio=5.0, U=U, W=W)
    g.step(3, lbm.BC_IBM_B)
    o.step(3, oracle.BC_IBM_B)
    uo = o.macro()[1]
    field, force, part = (1e-10, 1e-8 * np.max(np.abs(o.ibm_force())), 1e-10) if storage == "f64" else \
        (1e-5, 1e-5 * 2 * np.max(np.abs(uo)), 1e-5)
    assert np.max(np.abs(g.macro()[1] - uo)) < field * np.max(np.abs(uo))
    assert np.max(np.abs(g.ibm_force() - o.ibm_force())) < force
    Pg, Po = g.particles(), o.particles()
    for k in ("X", "U", "W"):
        assert np.max(np.abs(Pg[k] - Po[k])) < part * max(1.0, np.max(np.abs(Po[k]))), k


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("case", [*CASES, "many"])
def test_ibb_spheres_edges(lbm, case, storage):
    if case == "many":  # more particles than SMs
        shape = (40, 40, 40)
        X, R = workloads.place_spheres(shape, 160, 1.6, 1.2, seed=4), np.full(160, 1.6)
    else:
        shape, X, R = CASES[case]
        X, R = np.array(X), np.array(R)
    nz, ny, nx = shape
    n = len(R)
    g = lbm.Lattice(nx, ny, nz, 0.62, storage=lbm.STORAGE[storage], rates=oracle.RATES_DHUMIERES, max_particles=n,
                    max_links=19 * nx * ny * nz, max_sites=nx * ny * nz)
    o = oracle.Sim(nx, ny, nz, 0.62, rates=oracle.RATES_DHUMIERES)
    u = workloads.noise_velocity(shape, 0.02, seed=5)
    U, W = np.full((n, 3), 0.01), np.full((n, 3), -0.002)
    for s in (g, o):
        s.init_velocity(u)
        s.add_spheres(X, R, density_ratio=5.0, U=U, W=W)
    g.step(3, lbm.BC_IBB)
    o.step(3, oracle.BC_IBB)
    tol = 1e-10 if storage == "f64" else 1e-5
    uo = o.macro()[1]
    fluid = o.solid()[0] == 0
    assert np.max(np.abs((g.macro()[1] - uo)[:, fluid])) < tol * np.max(np.abs(uo))
    Pg, Po = g.particles(), o.particles()
    for k in ("X", "U", "W"):
        assert np.max(np.abs(Pg[k] - Po[k])) < tol * max(1.0, np.max(np.abs(Po[k]))), k
    assert np.max(np.abs(Pg["F"] - Po["F"])) < (1e-10 if storage == "f64" else 1e-5) * np.max(np.abs(Po["F"]))
