"""lbm_stats against its numpy statement on the library's own fields: FP64 and
FP32 fields (sums of float pairs), spheres of one and of several radii across
the box faces, odd boxes, plane counts around the 64-plane run, masked and raw
solid cells."""
import numpy as np
import pytest

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


def expected(u, rho, flags, P, R, shape, nu):
    """Energies, dissipation and radial bins of the masked velocity."""
    nz, ny, nx = shape
    n = np.array([nx, ny, nz])
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    pos = np.stack([x, y, z], -1).reshape(-1, 3).astype(float)
    solid = (flags & 1).astype(bool)
    s = np.full(len(pos), np.inf)
    near = np.zeros(len(pos), dtype=int)
    for p in range(len(R)):
        d = pos - P["X"][p]
        d -= n * np.rint(d / n)
        sp = np.sqrt((d * d).sum(1)) - R[p]
        m = sp < s
        s[m], near[m] = sp[m], p
    d = pos - P["X"][near]
    d -= n * np.rint(d / n)
    rigid = P["U"][near] + np.cross(P["W"][near], d)
    v = np.where(solid[:, None], rigid, u.T).T.reshape(3, nz, ny, nx)
    G = [[0.5 * (np.roll(v[a], -1, k) - np.roll(v[a], 1, k)) for k in (2, 1, 0)] for a in range(3)]
    eps = (2 * nu * sum((0.5 * (G[a][b] + G[b][a])) ** 2 for a in range(3) for b in range(3))).reshape(-1)
    ke = 0.5 * (v ** 2).sum(0).reshape(-1)
    fl = ~solid
    b = np.floor((s / R[near]) / 0.05).astype(int)
    ok = fl & (s > 0) & (b < 40)  # a cell on the surface to the last bit has no bin
    cnt = np.bincount(b[ok], minlength=40)[:40]
    per = [np.bincount(b[ok], weights=q[ok], minlength=40)[:40] / np.maximum(cnt, 1) for q in (ke, eps)]
    return dict(mass=rho.sum(), momentum=(u * rho).sum(1), kinetic_energy=ke.mean(), dissipation=eps.mean(),
                kinetic_energy_fluid=ke[fl].mean(), dissipation_fluid=eps[fl].mean(), nfluid=int(fl.sum()),
                bin_count=cnt, bin_tke=per[0] / ke[fl].mean(), bin_eps=per[1] / eps[fl].mean())


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("shape,R", [((33, 37, 41), [4.0, 4.0, 4.0]), ((65, 30, 33), [3.0, 4.5, 2.2])])
def test_stats_of_a_snapshot(lbm, storage, shape, R):
    nz, ny, nx = shape
    R = np.array(R)
    X = np.array([[1.3, 2.1, 0.7], [nx / 2 + 0.2, ny / 2, 12.4], [nx - 9.5, 9.1, nz - 9.6]])
    rng = np.random.default_rng(3)
    U, W = rng.normal(0, 0.01, (3, 3)), rng.normal(0, 0.002, (3, 3))
    g = lbm.Lattice(nx, ny, nz, 0.56, storage=storage, max_particles=3)
    g.init_velocity(workloads.noise_velocity(shape, 0.02, seed=4) + 0.01)
    g.add_spheres(X, R, U=U, W=W)
    got = g.stats(lbm.STATS_BINS)
    rho, u = g.macro()
    ref = expected(u, rho, g.flags(), g.particles(), R, shape, 0.06 / 3)
    assert got["nfluid"] == ref["nfluid"]
    assert np.array_equal(got["bin_count"], ref["bin_count"])
    # sums of N terms in FP64, or as pairs of 48 bits: far below 1e-12 of the result
    for k in ("mass", "kinetic_energy", "dissipation", "kinetic_energy_fluid", "dissipation_fluid"):
        assert got[k] == pytest.approx(ref[k], rel=1e-12), k
    for k in ("momentum", "bin_tke", "bin_eps"):
        assert np.allclose(got[k], ref[k], rtol=1e-11, atol=0), k
    g.step(2, lbm.BC_IBM_B)  # raw statistics count the fluid inside the particles
    raw = g.stats(lbm.STATS_UNMASK)
    rho, u = g.macro()
    ke = 0.5 * (u ** 2).sum(0)
    assert raw["kinetic_energy"] == pytest.approx(ke.mean(), rel=1e-12)
    assert np.allclose(raw["momentum"], (u * rho).sum(1), rtol=1e-11, atol=0)
    g.close()


@pytest.mark.parametrize("wall", ["pipe", "spheres"])
@pytest.mark.parametrize("storage", ["f32", "f16s"])
def test_statistics_leave_the_populations_alone(lbm, wall, storage, tmp_path):
    """lbm_stats names no population buffer as its scratch: a run that takes
    them (and, with a pipe, writes a checkpoint) between steps holds the same
    populations in every cell, solid ones included, as one that does not."""
    shape = (18, 21, 23)
    nz, ny, nx = shape
    u = workloads.noise_velocity(shape, 0.02, seed=4)
    runs = []
    for taken in (False, True):
        g = lbm.Lattice(nx, ny, nz, 0.6, storage=storage, max_particles=1)
        g.init_velocity(u)
        if wall == "pipe":
            g.set_pipe(9.3)
        else:
            g.add_spheres(np.array([[11.2, 9.7, 8.1]]), 4.0, U=np.full((1, 3), 0.01), W=np.zeros((1, 3)), fixed=True)
        for _ in range(3):
            g.step(1, lbm.BC_IBB)
            if taken:
                g.stats(lbm.STATS_BINS)
                if wall == "pipe":
                    g.checkpoint(str(tmp_path / "c.bin"))
        runs.append(g.populations())
        g.close()
    assert np.array_equal(*runs)


def test_bins_of_a_small_sphere_beside_a_large_one(lbm):
    """Spheres of radius 0.6 beside one of 64: the distances of the small ones
    are formed in the coarse coordinates of the large one's reach. The centres
    put one cell of each within that error of a bin edge."""
    n, r, R = 134, 0.6, 64.0
    frac = [[0.6503087487684525, 0.2039073800978315, 0.353350778146563],
            [0.5836530203021653, 0.6346187417687474, 0.040459510349080574],
            [0.30313713100829887, 0.18944387380685157, 0.8637899145128074],
            [0.576195652467419, 0.878151356172026, 0.39333355485314314],
            [0.3109796451597333, 0.4064864649216986, 0.45511893301826944],
            [0.29087156922514623, 0.4230262586893332, 0.9846860944370519],
            [0.2924158302428168, 0.9461288070160094, 0.6216942062295914],
            [0.37036860357278556, 0.42926034510139743, 0.22518122567558407]]
    corner = [[x, y, z] for x in (4, 124) for y in (4, 124) for z in (4, 124)]
    X = np.concatenate([np.array(corner) + np.array(frac), [[66.5, 66.5, 66.5]]])
    radii = np.array([r] * 8 + [R])
    g = lbm.Lattice(n, n, n, 0.6, storage="f32", max_particles=9)
    g.add_spheres(X, radii, U=np.zeros((9, 3)), W=np.zeros((9, 3)))
    got = g.stats(lbm.STATS_BINS)
    z, y, x = np.meshgrid(*[np.arange(n)] * 3, indexing="ij", sparse=True)
    near, who = np.full((n, n, n), np.inf), np.zeros((n, n, n), dtype=int)
    for p in range(9):
        d2 = 0.0
        for a, c in ((x, 0), (y, 1), (z, 2)):
            d = a - X[p, c]
            d2 = d2 + (d - n * np.rint(d / n)) ** 2
        s = np.sqrt(d2) - radii[p]
        m = s < near
        near[m], who[m] = s[m], p
    b = np.floor(near / radii[who] / 0.05).astype(int)
    ok = (near > 0) & (b < 40)
    assert np.array_equal(got["bin_count"], np.bincount(b[ok], minlength=40))
    g.close()


@pytest.mark.parametrize("storage", ["f32", "f16s"])
@pytest.mark.parametrize("u_scale,p_scale", [(1e-18, 1e-18), (1e-30, 1e-30), (1e-18, 1.0), (1.0, 0.0)])
def test_stats_of_tiny_velocities(lbm, storage, u_scale, p_scale):
    """Squares far below FP32's range, of the whole field or of the fluid
    beside particles that move at an ordinary speed: the sums are those of
    FP64. (FP16 storage rounds the small fields to rest: zeros.)"""
    shape = (17, 19, 21)
    nz, ny, nx = shape
    R = np.array([3.0, 2.5])
    X = np.array([[1.31, 2.12, 0.73], [12.23, 11.07, 9.41]])  # no cell on a bin edge to the last bit
    rng = np.random.default_rng(3)
    U, W = p_scale * rng.normal(0, 0.01, (2, 3)), p_scale * rng.normal(0, 0.002, (2, 3))
    g = lbm.Lattice(nx, ny, nz, 0.56, storage=storage, max_particles=2)
    g.init_velocity(u_scale * (workloads.noise_velocity(shape, 0.02, seed=4) + 0.01))
    g.add_spheres(X, R, U=U, W=W)
    got = g.stats(lbm.STATS_BINS)
    rho, u = g.macro()
    with np.errstate(invalid="ignore", divide="ignore"):
        ref = expected(u, rho, g.flags(), g.particles(), R, shape, 0.06 / 3)
    assert np.array_equal(got["bin_count"], ref["bin_count"])
    # sums of N terms in FP64, or as pairs of 48 bits
    for k in ("kinetic_energy", "dissipation", "kinetic_energy_fluid", "dissipation_fluid"):
        assert got[k] == pytest.approx(ref[k], rel=1e-12, abs=0), k
    if np.any(u):
        assert got["kinetic_energy_fluid"] > 0
        for k in ("bin_tke", "bin_eps"):
            assert np.allclose(got[k], ref[k], rtol=1e-11, atol=0), k
    g.close()
