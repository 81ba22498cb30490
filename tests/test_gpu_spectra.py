"""3D spectra on the GPU (hand-written FP32 FFT) against the numpy oracle
of oracle/spectra.py on the oracle's own velocity field, bin by bin.

Tolerance per shell: |gpu - oracle| <= 1e-5 max(oracle) + 1e-4 |oracle|,
from the FP32 transform (relative rounding ~1e-7 per stage, 3 log2 n
stages) against FP64 numpy."""
import numpy as np
import pytest

import oracle
import workloads
from oracle import spectra

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


def close(g, o):
    tol = 1e-5 * np.max(np.abs(o)) + 1e-4 * np.abs(o)
    return bool(np.all(np.abs(g - o) <= tol)), float(np.max(np.abs(g - o) / (np.max(np.abs(o)))))


def test_periodic_hit_spectrum_matches_oracle(lbm):
    n, tau, nb = 32, 0.6, 30
    u = workloads.hit_velocity(n, seed=2, k_peak=4.0, u_rms=0.03)
    g = lbm.Lattice(n, n, n, tau, storage=lbm.F64)
    o = oracle.Sim(n, n, n, tau)
    for s in (g, o):
        s.init_velocity(u)
    g.step(20)
    o.step(20)
    Eg, Dg = g.spectrum(nb)
    Eo, Do = spectra.spectra(o.masked_velocity(), n, (tau - 0.5) / 3, nb)
    okE, eE = close(Eg, Eo)
    okD, eD = close(Dg, Do)
    assert okE and okD, (eE, eD)
    # the two sums: mean kinetic energy and the spectral dissipation
    assert Eg.sum() == pytest.approx(o.stats()["kinetic_energy"], rel=1e-5)


def test_masked_sphere_spectrum_matches_oracle(lbm):
    p = workloads.SPHERE_32
    n = p["n"]
    u = workloads.noise_velocity((n, n, n), 1e-3, seed=1)
    g = lbm.Lattice(n, n, n, p["tau"], force=p["force"], storage=lbm.F64, max_particles=1)
    o = oracle.Sim(n, n, n, p["tau"], force=p["force"])
    X = np.array([p["centre"]])
    for s in (g, o):
        s.init_velocity(u)
        s.add_spheres(X, p["radius"], U=np.array([[0.01, 0.0, 0.0]]), W=np.zeros((1, 3)), fixed=True)
    g.step(10, lbm.BC_IBB)
    o.step(10, oracle.BC_IBB)
    Eg, Dg = g.spectrum(28)
    Eo, Do = spectra.spectra(o.masked_velocity(), n, (p["tau"] - 0.5) / 3, 28)
    okE, eE = close(Eg, Eo)
    okD, eD = close(Dg, Do)
    assert okE and okD, (eE, eD)


@pytest.mark.parametrize("n,m", [(16, 3), (64, 7)])
def test_single_mode_lands_in_its_shell(lbm, n, m):
    A = 0.02
    z, y, x = np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij")
    u = np.zeros((3, n, n, n))
    u[2] = A * np.sin(2 * np.pi * m * x / n)
    g = lbm.Lattice(n, n, n, 0.6, storage=lbm.F32)
    g.init_velocity(u)
    E, D = g.spectrum(n)
    assert E[m] == pytest.approx(A * A / 4, rel=1e-5)
    assert np.sum(np.delete(E, m)) < 1e-9 * E[m]
    nu = 0.1 / 3
    assert D[m] == pytest.approx(2 * nu * (2 * np.pi * m / n) ** 2 * A * A / 4, rel=1e-5)
    g.close()


def test_non_cube_is_rejected(lbm):
    g = lbm.Lattice(32, 32, 16, 0.6, storage=lbm.F32)
    g.init_velocity(np.zeros((3, 16, 32, 32)))
    with pytest.raises(lbm.LbmError):
        g.spectrum(8)
    g.close()


@pytest.mark.parametrize("n", [8, 16, 32, 128, 256])
def test_every_transform_length_on_noise(lbm, n):
    """White noise fills every shell: the last pass of the transform is of
    radix 8, 2 or 4 in turn, the smallest cubes take fewer lines per block;
    the bars of the other spectra tests."""
    u = workloads.noise_velocity((n, n, n), 0.02, seed=n)
    g = lbm.Lattice(n, n, n, 0.6, storage=lbm.F32)
    g.init_velocity(u)
    nb = 7 if n == 8 else n  # 8^3: the scratch limit
    Eg, Dg = g.spectrum(nb)
    Eo, Do = spectra.spectra(u, n, 0.1 / 3, nb)
    okE, eE = close(Eg, Eo)
    okD, eD = close(Dg, Do)
    assert okE and okD, (eE, eD)
    g.close()


@pytest.mark.parametrize("storage", ["f16s", "bf16s"])
def test_most_bins_of_a_small_cube_stay_in_the_scratch(lbm, storage):
    """64^3 in 16-bit storage with the most bins the call accepts and no slack
    behind the populations: the sums match the oracle, and neither the flags
    nor the next steps notice that the statistics were taken."""
    n, nb = 64, 1616
    u = workloads.noise_velocity((n, n, n), 0.02, seed=6)
    pair = [lbm.Lattice(n, n, n, 0.6, storage=storage, max_sites=1, max_links=1, max_markers=1) for _ in range(2)]
    for g in pair:
        g.init_velocity(u)
    E, D = pair[0].spectrum(nb)
    Eo, Do = spectra.spectra(pair[1].macro()[1], n, 0.1 / 3, nb)
    okE, eE = close(E, Eo)
    okD, eD = close(D, Do)
    assert okE and okD, (eE, eD)
    for g in pair:
        assert not g.flags().any()
        g.step(3)
    assert np.array_equal(pair[0].populations(), pair[1].populations())
    with pytest.raises(lbm.LbmError):
        pair[0].spectrum(nb + 1)
    for g in pair:
        g.close()


@pytest.mark.parametrize("scale", [1e-18, 1e-24, 1e-33])
def test_tiny_velocities_keep_their_spectrum(lbm, scale):
    """Squares below FP32's range: the shells are those of the same field at
    an ordinary size, on the bars of the other tests (a fluid coming to rest)."""
    n = 32
    u = workloads.noise_velocity((n, n, n), 0.02, seed=n) * scale
    g = lbm.Lattice(n, n, n, 0.6, storage=lbm.F64)
    g.init_velocity(u)
    Eg, Dg = g.spectrum(n)
    Eo, Do = spectra.spectra(g.macro()[1] / scale, n, 0.1 / 3, n)
    okE, eE = close(Eg / scale ** 2, Eo)
    okD, eD = close(Dg / scale ** 2, Do)
    assert okE and okD, (eE, eD)
    g.close()
