"""The pipe sweep on the column layout (z fastest) against the oracle: plane
counts around the 32-cell chunk and the column pitch, odd sections, walls
that touch the box faces, single-node links, every storage type and both
collisions; populations in and out of the layout."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5, "f16s": 2e-3, "bf16s": 3e-2}


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_05448_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


def rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


def pair(lbm, nx, ny, nz, R, storage, rates, seed=3):
    u = workloads.pipe_velocity(nx, ny, nz, R, 0.03, perturbation=0.1, seed=seed)
    g = lbm.Lattice(nx, ny, nz, 0.57, force=(1e-6, 0, 4e-6), storage=storage, rates=rates)
    o = oracle.Sim(nx, ny, nz, 0.57, force=(1e-6, 0, 4e-6), rates=rates)
    for s in (g, o):
        s.init_velocity(u)
        s.set_pipe(R)
    return g, o


@pytest.mark.parametrize("nx,ny,nz,R", [
    (24, 24, 4, 10.3),     # fewer planes than a pitch group
    (27, 26, 31, 11.7),    # one chunk, one lane idle
    (27, 26, 32, 11.7),    # one whole chunk
    (27, 29, 33, 12.1),    # a second chunk of one cell
    (31, 30, 65, 13.6),
    (16, 16, 20, 8.0),     # the wall touches the box faces: pulls wrap in x and y
    (16, 16, 9, 6.4),      # single-node links
])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16s", "bf16s"])
def test_steps_match_the_oracle(lbm, nx, ny, nz, R, storage):
    for rates in (oracle.RATES_SRT, oracle.RATES_DHUMIERES):
        g, o = pair(lbm, nx, ny, nz, R, storage, rates)
        g.step(20, lbm.BC_IBB)
        o.step(20, oracle.BC_IBB)
        fluid = o.solid()[0] == 0
        rg, ug = g.macro()
        ro, uo = o.macro()
        assert rel(ug[:, fluid], uo[:, fluid]) < TOL[storage]
        assert rel(rg[fluid], ro[fluid]) < TOL[storage]
        assert not np.any(ug[:, ~fluid]) and not np.any(rg[~fluid])
        if storage == "f64":
            assert rel(g.populations()[:, fluid], o.populations()[:, fluid]) < TOL[storage]
        g.close()
        o.close()


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_populations_set_between_steps(lbm, storage):
    """Populations taken out of the layout and put into another context that
    is already stepping continue the same run."""
    g, _ = pair(lbm, 27, 26, 33, 11.7, storage, oracle.RATES_SRT)
    h, _ = pair(lbm, 27, 26, 33, 11.7, storage, oracle.RATES_SRT, seed=8)
    g.step(3, lbm.BC_IBB)
    h.step(1, lbm.BC_IBB)
    f = g.populations()
    h.set_populations(f)
    assert rel(h.populations(), f) < 1e-7
    g.step(4, lbm.BC_IBB)
    h.step(4, lbm.BC_IBB)
    fluid = (g.flags() & 1) == 0
    # FP32: f = g + w read out in FP64 loses nothing, put back it rounds to the same g
    assert np.array_equal(g.populations()[:, fluid], h.populations()[:, fluid]) if storage == "f32" else \
        rel(h.populations()[:, fluid], g.populations()[:, fluid]) < 1e-14
    g.close()
    h.close()


@pytest.mark.parametrize("nz", [4, 32, 33])
@pytest.mark.parametrize("nx,ny,R", [(27, 24, 10.3), (16, 16, 8.0)])  # the second wraps in x and y
def test_d3q27_plane_counts(lbm, nx, ny, R, nz):
    from oracle import d3q27 as q27
    tau, F = 0.62, (1e-6, 0.0, 3e-6)
    u = workloads.pipe_velocity(nx, ny, nz, R, 0.02, perturbation=0.1, seed=5)
    g = lbm.Lattice(nx, ny, nz, tau, force=F, storage="f64", lattice=27)
    g.init_velocity(u)
    g.set_pipe(R)
    solid = q27.pipe_solid(nx, ny, nz, R)
    links = q27.pipe_links(solid, R)
    o = q27.feq(np.ones((nz, ny, nx)), u)
    fl = ~solid.reshape(-1)
    g.step(3, lbm.BC_IBB)
    for _ in range(3):
        o = q27.step_pipe(o, solid, links, tau, F)
    assert rel(g.populations()[:, fl], o.reshape(27, -1)[:, fl]) < 1e-12
    rg, ug = g.macro()
    ro, uo = q27.macro(o, F)
    assert rel(ug[:, fl], uo.reshape(3, -1)[:, fl]) < 1e-12 and rel(rg[fl], ro.reshape(-1)[fl]) < 1e-12
    g.close()


@pytest.mark.parametrize("nx,ny,nz,R,nbins", [
    (27, 26, 33, 11.7, 1), (27, 26, 33, 11.7, 7), (27, 26, 33, 11.7, 60), (25, 25, 4, 11.2, 1),
    (25, 25, 4, 11.2, 7), (40, 33, 64, 15.9, 60),  # small sections refuse more bins (LBM_ENOMEM)
])
def test_pipe_statistics_of_a_snapshot(lbm, nx, ny, nz, R, nbins):
    """Profiles and budget of the library's own fields against their numpy
    statements: odd sections (a column on the axis: in the profiles, not in
    the budget), runs of planes with a remainder, one bin to more bins than
    columns along the radius. Bars of the full-field tests of each."""
    from oracle import profiles, tke_budget as tb
    g, _ = pair(lbm, nx, ny, nz, R, "f64", oracle.RATES_SRT)
    g.step(5, lbm.BC_IBB)
    rho, u = g.macro()
    solid = g.flags() & 1
    args = (u, rho, solid, nx, ny, nz, 0.5 * (nx - 1), 0.5 * (ny - 1), R, 0.07 / 3, nbins)
    for got, ref, tol in ((g.pipe_profiles(nbins), profiles.pipe_profiles(*args), 1e-10),
                          (g.tke_budget(nbins), tb.tke_budget(*args), 1e-7)):
        assert np.array_equal(got[:, 0], ref[:, 0])
        for k in range(1, ref.shape[1]):
            scale = max(np.max(np.abs(ref[:, k])), 1e-300)
            if k in (1, 2) and ref.shape[1] == 12:  # u_r, u_theta: means that nearly vanish, on the velocity's scale
                scale = np.max(np.abs(u))
            assert np.max(np.abs(got[:, k] - ref[:, k])) <= tol * scale, k
    g.close()


@pytest.mark.parametrize("nx,ny,nz,R", [
    (27, 26, 1, 11.7), (27, 26, 7, 11.7), (27, 26, 28, 11.7),  # cells across the ends of the columns
    (27, 26, 29, 11.7), (27, 26, 61, 11.7), (27, 26, 95, 11.7),  # warps per column, the last with idle lanes
    (16, 16, 31, 8.0), (16, 15, 64, 6.4),  # the same with wraps in x and y, and with single-node links
    (16, 15, 33, 7.4), (16, 16, 5, 6.4),  # both walked cell by cell
])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16s"])
def test_both_walks_over_the_columns(lbm, nx, ny, nz, R, storage):
    """Plane counts on both sides of the rule that picks the walk
    (column_flat), every wall treatment, against the oracle."""
    for bc in ("IBB", "IBM_B"):
        g, o = pair(lbm, nx, ny, nz, R if bc == "IBB" else min(R, nx / 2 - 4.4), storage, oracle.RATES_SRT)
        g.step(5, getattr(lbm, "BC_" + bc))
        o.step(5, getattr(oracle, "BC_" + bc))
        keep = o.solid()[0] == 0 if bc == "IBB" else slice(None)
        rg, ug = g.macro()
        ro, uo = o.macro()
        # the diffuse wall's sums run in another order: as in the other IBM comparisons
        tol = TOL[storage] if bc == "IBB" or storage != "f64" else 1e-10
        assert rel(ug[:, keep], uo[:, keep]) < tol
        assert rel(rg[keep], ro[keep]) < tol
        g.close()
        o.close()
