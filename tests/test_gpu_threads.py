"""Contexts of several host threads, each on a stream of its own, whose calls
need different amounts of shared memory from the same kernel: every call
succeeds and gives what it gives alone."""
import threading

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


def together(work):
    """Run the callables in threads; their results, or the first error."""
    out, errors = [None] * len(work), []

    def run(k):
        try:
            out[k] = work[k]()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]
    return out


def test_ibm_spheres_of_different_radii(lbm):
    import torch
    n = 24
    u = workloads.noise_velocity((n, n, n), 0.02, seed=5)

    def run(R):
        def go():
            g = lbm.Lattice(n, n, n, 0.62, storage="f32", max_particles=1, stream=torch.cuda.Stream())
            g.init_velocity(u)
            g.add_spheres(np.array([[11.3, 12.1, 10.7]]), R, density_ratio=5.0)
            for _ in range(600):
                g.step(1, lbm.BC_IBM_B)
            X = g.particles()["X"]
            g.close()
            return X
        return go

    radii = (1.2, 5.9, 2.7, 4.4)
    alone = [run(R)() for R in radii]
    for a, b in zip(alone, together([run(R) for R in radii])):
        assert np.array_equal(a, b)


def test_spectra_of_different_bins(lbm):
    import torch
    n = 64
    u = workloads.noise_velocity((n, n, n), 0.02, seed=6)

    def run(nb):
        def go():
            g = lbm.Lattice(n, n, n, 0.6, storage="f32", stream=torch.cuda.Stream())
            g.init_velocity(u)
            for _ in range(300):
                E, _ = g.spectrum(nb)
            g.close()
            return E[:20]
        return go

    bins = (20, 2048, 64, 1000)
    ref = run(57)()
    for E in together([run(nb) for nb in bins]):
        assert np.allclose(E, ref, rtol=1e-9, atol=0)  # other numbers of blocks: FP64 sums in another order
