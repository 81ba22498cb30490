"""The routes of the IBM forcing of spheres, told by the launches of the group
"ibm_passes" (two per pass where one block forms a sphere's whole pass, three
else): the largest radius that a block holds and the ones beyond it, boxes as
wide as the grid and wider, in both precisions, against the oracle. Bars of the
other IBM comparisons: FP64 1e-10 of the field and 1e-8 of the force, FP32 1e-5
of the field and 1e-5 of 2 max|u| for the force."""
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


# storage, bc, (nz, ny, nx), centre (x, y, z), radius, launches per step
CASES = [
    ("f32", "IBM_B", (21, 19, 23), [3.3, 17.5, 8.0], 6.7, 6),  # the largest box of a block, one block per SM
    ("f32", "IBM_B", (21, 22, 23), [3.3, 17.5, 8.0], 8.0, 9),  # force box in shared memory, wider than the grid
    ("f32", "IBM_B", (33, 31, 34), [30.2, 3.5, 17.75], 8.7, 9),  # the same inside the grid, across two faces
    ("f32", "IBM_U", (13, 13, 13), [6.3, 12.8, 0.4], 4.05, 9),  # a small box, wider than the grid
    ("f64", "IBM_U", (13, 13, 13), [6.3, 12.8, 0.4], 4.05, 9),
    ("f32", "IBM_B", (34, 35, 36), [30.2, 3.5, 17.75], 14.5, 9),  # global atomics
    ("f64", "IBM_B", (21, 19, 23), [3.3, 17.5, 8.0], 4.3, 6),
]


@pytest.mark.parametrize("storage,bc,shape,X,R,launches", CASES)
def test_route_and_result(lbm, storage, bc, shape, X, R, launches):
    nz, ny, nx = shape
    g = lbm.Lattice(nx, ny, nz, 0.62, storage=storage, rates=oracle.RATES_DHUMIERES, max_particles=1,
                    max_sites=nx * ny * nz, max_markers=int(13 * R * R + 40))
    o = oracle.Sim(nx, ny, nz, 0.62, rates=oracle.RATES_DHUMIERES)
    u = workloads.noise_velocity(shape, 0.02, seed=5)
    for s in (g, o):
        s.init_velocity(u)
        s.add_spheres(np.array([X]), np.array([R]), density_ratio=5.0, U=np.full((1, 3), 0.01), W=np.full((1, 3), -0.002))
    g.step(1, getattr(lbm, "BC_" + bc))
    g.profile_enable()
    g.step(2, getattr(lbm, "BC_" + bc))
    assert g.profile(0)["launches"]["ibm_passes"] == 2 * launches
    o.step(3, getattr(oracle, "BC_" + bc))
    uo = o.macro()[1]
    field, force, part = (1e-10, 1e-8 * np.max(np.abs(o.ibm_force())), 1e-10) if storage == "f64" else \
        (1e-5, 1e-5 * 2 * np.max(np.abs(uo)), 1e-5)
    assert np.max(np.abs(g.macro()[1] - uo)) < field * np.max(np.abs(uo))
    assert np.max(np.abs(g.ibm_force() - o.ibm_force())) < force
    Pg, Po = g.particles(), o.particles()
    for k in ("X", "U", "W"):
        assert np.max(np.abs(Pg[k] - Po[k])) < part * max(1.0, np.max(np.abs(Po[k]))), k
    g.close()
