"""Timing cases: the work a user of the library has it do, through its public
entry points, over the range of sizes, wall treatments and storage types it
runs in earnest.

A case is a plain dict; `listed()` holds the fixed ones and `draw(rng)` gives
further ones of the same ranges. `prepare` builds what a program has in hand
before the call (a lattice with its initial field and geometry, or samples
and weights on the GPU), `run` makes one pass, `work` counts what that pass
cannot do without, and `exact` states the same result in 64 bits with torch
alone.

Outputs are handed on in the precision the fluid state is stored in: the C
ABI widens an FP32 lattice's fields to doubles, whose further digits carry
nothing. Statistics that the library sums in FP64 stay in FP64.
"""
import math

import numpy as np
import torch

import workloads
from paper_1906_05448_gb300 import lbm

DEV = "cuda"
F64 = torch.float64
NU = 0.0032           # pipe viscosity
U_BULK = 0.08         # pipe bulk velocity of the initial profile
TAU_BOX = 0.51        # relaxation time of the turbulent boxes
U_SCALE, G_SCALE = 0.03, 4.0 / 0.03  # scales of the learned closure
STORAGE_BYTES = {"f64": 8, "f32": 4, "f16s": 2, "bf16s": 2}
OUT_TYPE = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16, "bf16s": torch.bfloat16}
MLP_SIZES = (85, 64, 64, 64, 9)


def listed():
    return [
        # the smallest call: one fixed sphere in a small box, double precision,
        # a hundred steps and a snapshot (validation runs, drag curves)
        dict(name="sphere32_fixed_f64", kind="sphere", n=32, radius=4.0, storage="f64", steps=100),
        # turbulence without walls on an odd, non-cubic box (spin-up of an
        # initial field before particles are released)
        dict(name="box_250x131x97_mrt_f32", kind="box", nx=250, ny=131, nz=97, storage="f32", steps=200),
        # the benchmark: turbulent pipe, interpolated bounce-back, FP32,
        # advanced between two saved snapshots
        dict(name="pipe148_ibb_f32", kind="pipe", nx=148, nz=438, radius=73.0, storage="f32", wall="ibb",
             lattice=19, steps=500),
        # the same pipe on 16-bit populations (longer pipes on one GPU)
        dict(name="pipe148_ibb_f16s", kind="pipe", nx=148, nz=438, radius=73.0, storage="f16s", wall="ibb",
             lattice=19, steps=500),
        # the same pipe with the immersed boundary wall
        dict(name="pipe148_ibm_b_f32", kind="pipe", nx=148, nz=438, radius=73.0, storage="f32", wall="ibm_b",
             lattice=19, steps=200),
        # the same pipe on the 27-velocity lattice
        dict(name="pipe148_q27_f32", kind="pipe", nx=148, nz=438, radius=73.0, storage="f32", wall="ibb",
             lattice=27, steps=200),
        # decaying turbulence laden with 2000 moving spheres, bounce-back walls
        dict(name="hit256_2000p_ibb_f32", kind="suspension", n=256, np=2000, storage="f32", wall="ibb", steps=100),
        # the same with the immersed boundary
        dict(name="hit256_2000p_ibm_b_f32", kind="suspension", n=256, np=2000, storage="f32", wall="ibm_b", steps=50),
        # snapshot statistics of the laden box: energies, dissipation, radial
        # bins around the particles, near-surface gradients from the closure
        dict(name="stats_hit256_closure", kind="stats", n=256, np=2000, closure=True),
        # energy and dissipation spectra of a 256^3 snapshot
        dict(name="spectrum_hit256", kind="spectrum", n=256, nbins=222),
        # radial profiles and the energy budget of a pipe snapshot
        dict(name="budget_pipe148", kind="budget", nx=148, nz=438, radius=73.0, nbins=64),
        # training of the closure on new samples, then its evaluation on
        # held-out ones
        dict(name="closure_train_131k", kind="closure", n=131149, held=250003, batch=4096, epochs=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sphere", "box", "pipe", "pipe", "pipe", "suspension", "suspension", "stats", "spectrum",
                       "budget", "closure"])
    if kind == "sphere":
        n = _log_int(rng, 24, 96)
        return dict(kind=kind, n=n, radius=round(rng.uniform(3.0, n / 7.0), 2),
                    storage=rng.choice(["f64", "f32"]), steps=_log_int(rng, 20, 200))
    if kind == "box":
        return dict(kind=kind, nx=_log_int(rng, 32, 256), ny=_log_int(rng, 32, 256), nz=_log_int(rng, 32, 256),
                    storage=rng.choice(["f32", "f32", "f64", "f16s", "bf16s"]), steps=_log_int(rng, 10, 100))
    if kind == "pipe":
        nx = _log_int(rng, 40, 148)
        lattice = rng.choice([19, 19, 19, 27])
        wall = "ibb" if lattice == 27 else rng.choice(["ibb", "ibb", "ibm_u", "ibm_b"])
        storage = rng.choice(["f32", "f64"] if lattice == 27 or wall != "ibb" else ["f32", "f16s", "bf16s", "f64"])
        # the diffuse wall keeps its four-point stencil inside the box
        radius = nx / 2 - (4.3 if wall != "ibb" else rng.uniform(0.7, 2.5))
        return dict(kind=kind, nx=nx, nz=_log_int(rng, 24, 400), radius=round(radius, 3), storage=storage, wall=wall,
                    lattice=lattice, steps=_log_int(rng, 20, 100))
    if kind == "suspension":
        n = _log_int(rng, 48, 224)
        return dict(kind=kind, n=n, np=max(1, int(n ** 3 * rng.uniform(0.4, 1.0) * 1.2e-4)),
                    storage=rng.choice(["f32", "f32", "f64", "f16s"]), wall=rng.choice(["ibb", "ibm_b", "ibm_u"]),
                    steps=_log_int(rng, 10, 30))
    if kind == "stats":
        n = _log_int(rng, 48, 240)
        return dict(kind=kind, n=n, np=max(1, int(n ** 3 * rng.uniform(0.4, 1.0) * 1.2e-4)),
                    closure=rng.random() < 0.5)
    if kind == "spectrum":
        n = rng.choice([32, 64, 128, 256])
        return dict(kind=kind, n=n, nbins=rng.randint(n // 2, int(0.87 * n)))
    if kind == "budget":
        nx = _log_int(rng, 40, 148)
        return dict(kind=kind, nx=nx, nz=_log_int(rng, 24, 400), radius=round(nx / 2 - rng.uniform(0.7, 2.5), 3),
                    nbins=rng.randint(16, 128))
    return dict(kind="closure", n=_log_int(rng, 3000, 300000), held=_log_int(rng, 300, 1500000),
                batch=rng.choice([1000, 2048, 4096, 8192]), epochs=rng.randint(1, 2))


# ----------------------------------------------------------------- inputs --
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _turbulence(nx, ny, nz, seed, u_rms, k_peak):
    """Random solenoidal periodic field, (3, nz, ny, nx) doubles on the GPU:
    amplitudes of a k^4 exp(-2 (k / k_peak)^2) spectrum, k in waves per 256
    cells, projected to be divergence-free, on top of a mean drift."""
    g = _gen(seed)
    kz = torch.fft.fftfreq(nz, dtype=F64, device=DEV)[:, None, None]
    ky = torch.fft.fftfreq(ny, dtype=F64, device=DEV)[None, :, None]
    kx = torch.fft.rfftfreq(nx, dtype=F64, device=DEV)[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    k = 256.0 * torch.sqrt(k2)
    amp = k * torch.exp(-((k / k_peak) ** 2)) * (kx.abs() < 0.5) * (ky.abs() < 0.5) * (kz.abs() < 0.5)
    a = torch.randn((3,) + tuple(k2.shape), generator=g, dtype=torch.complex128, device=DEV) * amp
    dot = (kx * a[0] + ky * a[1] + kz * a[2]) / torch.where(k2 > 0, k2, 1.0)
    for c, kc in enumerate((kx, ky, kz)):
        a[c] -= kc * dot
    u = torch.fft.irfftn(a, s=(nz, ny, nx), dim=(1, 2, 3))
    u *= u_rms / torch.sqrt((u * u).sum() / (3.0 * nx * ny * nz))
    u += torch.tensor([0.004, -0.003, 0.002], dtype=F64, device=DEV)[:, None, None, None]
    return u


def _pipe_radius2(nx, dtype=F64):
    x = torch.arange(nx, dtype=dtype, device=DEV) - 0.5 * (nx - 1)
    return x[None, :] ** 2 + x[:, None] ** 2


def _pipe_field(nx, nz, radius, seed):
    """Laminar profile plus a 5 % perturbation that vanishes at the wall."""
    r2 = _pipe_radius2(nx) / radius ** 2
    inside = (r2 < 1.0).to(F64)
    u = _turbulence(nx, nx, nz, seed, 1.0, 30.0) * (0.05 * U_BULK) * (inside * (1.0 - r2) ** 2)
    u[2] += inside * (2.0 * U_BULK * (1.0 - r2))
    return u


def _pipe_force(radius):
    """Body force: the benchmark's friction velocity for the large pipes; the
    balance of the laminar profile for small ones, which would relaminarise
    and speed up without end under the former."""
    u_tau = 180.0 * NU / 73.0
    return 2.0 * u_tau ** 2 / radius if radius > 60.0 else 8.0 * NU * U_BULK / radius ** 2


def _weights(seed):
    """He-normal weights of the closure's perceptron, small biases (FP32)."""
    g = _gen(seed + 7)
    parts = []
    for a, b in zip(MLP_SIZES[:-1], MLP_SIZES[1:]):
        parts.append(torch.randn(a * b, generator=g, device=DEV) * math.sqrt(2.0 / a))
        parts.append(torch.randn(b, generator=g, device=DEV) * 0.05)
    return torch.cat(parts)


def _samples(n, seed):
    """Feature rows and gradients with the spread of real ones: correlated
    relative velocities, a distance in (0, 2], targets that depend on them."""
    g = _gen(seed)
    base = torch.randn((n, 3), generator=g, device=DEV)
    X = torch.randn((n, 85), generator=g, device=DEV) * 0.3
    X[:, :81] += base.repeat(1, 27)
    X[:, 81] = 2.0 * (1.0 - torch.rand(n, generator=g, device=DEV))
    X[:, 82:] = X[:, 39:42]
    mix = torch.randn((85, 9), generator=_gen(12345), device=DEV) * 0.12
    T = torch.tanh(X @ mix) + 0.1 * torch.randn((n, 9), generator=g, device=DEV)
    return X, T


def _spheres(case, seed):
    n, k = case["n"], case["np"]
    X = workloads.place_spheres((n, n, n), k, 4.0, 1.0, seed=seed)
    rng = np.random.default_rng(seed + 1)
    return X, rng.normal(0.004, 0.02, (k, 3)), rng.normal(0.0, 0.003, (k, 3))


def _host(u):
    return u.cpu().numpy()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "closure":
        X, T = _samples(case["n"], seed)
        Xh, _ = _samples(case["held"], seed + 1)
        return dict(case=case, mlp=lbm.MLP(), X=X, T=T, Xh=Xh, w=_weights(seed))
    if kind == "sphere":
        n = case["n"]
        L = lbm.Lattice(n, n, n, 0.6, force=(1e-6, 0.0, 0.0), storage=case["storage"], max_particles=1)
        L.init_velocity(_host(_turbulence(n, n, n, seed, 0.01, 512.0 / n)))
        L.add_spheres([[0.5 * n - 0.5] * 3], case["radius"], U=np.zeros((1, 3)), W=np.zeros((1, 3)), fixed=True)
    elif kind == "box":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        L = lbm.Lattice(nx, ny, nz, TAU_BOX, storage=case["storage"], rates=lbm.RATES_DHUMIERES)
        L.init_velocity(_host(_turbulence(nx, ny, nz, seed, 0.03, 8.0)))
    elif kind in ("pipe", "budget"):
        nx, nz, R = case["nx"], case["nz"], case["radius"]
        L = lbm.Lattice(nx, nx, nz, 3.0 * NU + 0.5, force=(0.0, 0.0, _pipe_force(R)),
                        storage=case.get("storage", "f32"), lattice=case.get("lattice", 19))
        L.init_velocity(_host(_pipe_field(nx, nz, R, seed)))
        L.set_pipe(R)
        if kind == "budget":  # a snapshot of a run in progress
            L.step(20, lbm.BC_IBB)
    elif kind == "spectrum":
        n = case["n"]
        L = lbm.Lattice(n, n, n, TAU_BOX, rates=lbm.RATES_DHUMIERES)
        L.init_velocity(_host(_turbulence(n, n, n, seed, 0.03, 8.0 * 256.0 / n)))
    else:  # suspension, stats
        n = case["n"]
        X, U, W = _spheres(case, seed)
        L = lbm.Lattice(n, n, n, TAU_BOX, storage=case.get("storage", "f32"), rates=lbm.RATES_DHUMIERES,
                        max_particles=case["np"])
        L.init_velocity(_host(_turbulence(n, n, n, seed, 0.03, 8.0)))
        if kind == "suspension":  # released with the fluid's velocity
            L.add_spheres(X, 4.0, density_ratio=5.0)
        else:
            L.add_spheres(X, 4.0, density_ratio=5.0, U=U, W=W)
            if case["closure"]:
                L.closure_set_weights(_host(_weights(seed)), U_SCALE, G_SCALE)
    return dict(case=case, L=L)


# -------------------------------------------------------------------- run --
def _fields(L, storage):
    rho, u = L.macro()
    # a density near 1 has nothing left to show in 16 bits
    rt = torch.float64 if storage == "f64" else torch.float32
    return dict(rho=torch.from_numpy(rho).to(rt), u=torch.from_numpy(u).to(OUT_TYPE[storage]))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "closure":
        w, loss = state["mlp"].train(state["X"], state["T"], state["w"], case["epochs"], batch=case["batch"])
        return dict(w=w, loss=np.float32(loss), Y=state["mlp"].forward(state["Xh"], w))
    L = state["L"]
    if kind == "stats":
        s = L.stats(lbm.STATS_BINS | (lbm.STATS_CLOSURE if case["closure"] else 0))
        return {k: np.asarray(v) for k, v in s.items()}
    if kind == "spectrum":  # the library's transform is in FP32
        E, D = L.spectrum(case["nbins"])
        return dict(E=E.astype(np.float32), D=D.astype(np.float32))
    if kind == "budget":
        P, B = L.pipe_profiles(case["nbins"]), L.tke_budget(case["nbins"])
        return dict(count=P[:, 0].astype(np.int64), profiles=P[:, 1:], budget_count=B[:, 0].astype(np.int64),
                    budget=B[:, 1:])
    L.step(case["steps"], case.get("wall", "ibb" if kind == "sphere" else "none"))
    out = _fields(L, case["storage"])
    if kind in ("sphere", "suspension"):
        t = torch.float64 if case["storage"] == "f64" else torch.float32
        out.update({k: torch.from_numpy(v).to(t) for k, v in L.particles().items()})
    return out


# ------------------------------------------------------------------- work --
def _fluid_per_plane(nx, radius):
    x = np.arange(nx) - 0.5 * (nx - 1)
    return int(np.count_nonzero(x[None, :] ** 2 + x[:, None] ** 2 < radius * radius))


def work(case):
    """Each step reads and writes the populations of the cells it advances
    once; the fields come out once."""
    kind = case["kind"]
    if kind == "closure":
        per = 2.0 * sum(a * b for a, b in zip(MLP_SIZES[:-1], MLP_SIZES[1:]))
        n, held = case["n"], case["held"]
        return dict(bytes=4.0 * (94.0 * n * case["epochs"] + 94.0 * held), flops=per * (3.0 * n * case["epochs"] + held))
    if kind in ("stats", "spectrum"):
        n3 = float(case["n"]) ** 3
        flops = n3 * (60.0 if kind == "stats" else 3 * 2.5 * 3 * math.log2(case["n"]))
        if kind == "stats" and case["closure"]:
            flops += 600.0 * case["np"] * 28416.0
        return dict(bytes=76.0 * n3, flops=flops)
    if kind == "budget":
        cells = float(_fluid_per_plane(case["nx"], case["radius"])) * case["nz"]
        return dict(bytes=76.0 * cells, flops=300.0 * cells)
    sb = STORAGE_BYTES[case["storage"]]
    q = case.get("lattice", 19)
    if kind == "pipe":
        N = float(case["nx"]) ** 2 * case["nz"]
        cells = float(_fluid_per_plane(case["nx"], case["radius"])) * case["nz"] if case["wall"] == "ibb" else N
    elif kind == "box":
        N = cells = float(case["nx"]) * case["ny"] * case["nz"]
    else:
        N = float(case["n"]) ** 3
        k, R = case.get("np", 1), case.get("radius", 4.0)
        cells = N - (k * 4.0 / 3.0 * math.pi * R ** 3 if case.get("wall", "ibb") == "ibb" else 0.0)
    per_cell = 250.0 if kind in ("pipe", "sphere") else 500.0
    return dict(bytes=case["steps"] * cells * 2.0 * q * sb + 4.0 * N * sb, flops=case["steps"] * cells * per_cell)


# ------------------------------------------------- the same in 64 bits ----
def _velocities(q):
    c = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1) if q == 27 or abs(x) + abs(y) + abs(z) < 3]
    w19, w27 = (1 / 3, 1 / 18, 1 / 36), (8 / 27, 2 / 27, 1 / 54, 1 / 216)
    w = [(w27 if q == 27 else w19)[sum(map(abs, v))] for v in c]
    return c, w, [c.index((-x, -y, -z)) for x, y, z in c]


def _mrt_matrix(c, tau):
    """M^-1 S M of the 19-velocity collision, each row of M a polynomial in
    the velocity components with its relaxation rate."""
    rows, rates = [], []
    om = 1.0 / tau
    v = np.array(c, dtype=float)
    x, y, z = v[:, 0], v[:, 1], v[:, 2]
    s = x * x + y * y + z * z
    for poly, rate in ((0 * x + 1, 0), (19 * s - 30, 1.19), (10.5 * s * s - 26.5 * s + 12, 1.4),
                       (x, 0), (y, 0), (z, 0), ((5 * s - 9) * x, 1.2), ((5 * s - 9) * y, 1.2), ((5 * s - 9) * z, 1.2),
                       (3 * x * x - s, om), ((3 * s - 5) * (3 * x * x - s), 1.4),
                       (y * y - z * z, om), ((3 * s - 5) * (y * y - z * z), 1.4),
                       (x * y, om), (y * z, om), (x * z, om),
                       ((y * y - z * z) * x, 1.98), ((z * z - x * x) * y, 1.98), ((x * x - y * y) * z, 1.98)):
        rows.append(poly)
        rates.append(rate)
    M = np.array(rows)
    return torch.tensor(np.linalg.inv(M) @ np.diag(rates) @ M, dtype=F64, device=DEV)


def _equilibrium(rho, u, c, w):
    uu = 1.0 - 1.5 * (u * u).sum(0)
    f = torch.empty((len(c),) + tuple(rho.shape), dtype=F64, device=DEV)
    for i, v in enumerate(c):
        cu = v[0] * u[0] + v[1] * u[1] + v[2] * u[2]
        f[i] = w[i] * rho * (uu + cu * (3.0 + 4.5 * cu))
    return f


def _moments(f, c):
    cv = torch.tensor(c, dtype=F64, device=DEV)
    return f.sum(0), (cv.T @ f.reshape(len(c), -1)).reshape((3,) + tuple(f.shape[1:]))


def _collide(f, F, tau, c, w, mrt=None):
    """In place: BGK with the Guo force F (3 fields or None), or the MRT
    matrix without a force."""
    rho, m = _moments(f, c)
    if mrt is not None:
        d = _equilibrium(rho, m / rho, c, w) - f
        f += (mrt @ d.reshape(len(c), -1)).reshape(f.shape)
        return
    u = (m + 0.5 * F) / rho
    uu = 1.0 - 1.5 * (u * u).sum(0)
    uF = (u * F).sum(0)
    k = 1.0 - 0.5 / tau
    for i, v in enumerate(c):
        cu = v[0] * u[0] + v[1] * u[1] + v[2] * u[2]
        cF = v[0] * F[0] + v[1] * F[1] + v[2] * F[2]
        f[i] += (w[i] * rho * (uu + cu * (3.0 + 4.5 * cu)) - f[i]) / tau + (w[i] * k) * (3.0 * (cF - uF) + 9.0 * cu * cF)


def _stream(f, c):
    return torch.stack([torch.roll(f[i], shifts=(v[2], v[1], v[0]), dims=(0, 1, 2)) for i, v in enumerate(c)])


def _pipe_links(nx, radius, c):
    """Per velocity: the columns of fluid cells whose neighbour lies outside,
    and the wall fraction; None when a link would need another scheme."""
    x = torch.arange(nx, dtype=F64, device=DEV) - 0.5 * (nx - 1)
    X, Y = x[None, :].expand(nx, nx), x[:, None].expand(nx, nx)
    out = X * X + Y * Y >= radius * radius
    links = []
    for v in c:
        a = float(v[0] ** 2 + v[1] ** 2)
        m = ~out & torch.roll(out, shifts=(-v[1], -v[0]), dims=(0, 1))
        if a == 0 or not bool(m.any()):
            links.append(None)
            continue
        b = (X * v[0] + Y * v[1])[m]
        q = ((-b + torch.sqrt(b * b + a * (radius * radius - (X * X + Y * Y)[m]))) / a).clamp(0.0, 1.0)
        if bool((torch.roll(out, shifts=(v[1], v[0]), dims=(0, 1))[m] & (q < 0.5)).any()):
            return None, None
        links.append((m, q))
    return out, links


def _peskin(r):
    a = np.abs(r)
    with np.errstate(invalid="ignore"):
        near = (3.0 - 2.0 * a + np.sqrt(1.0 + 4.0 * a - 4.0 * a * a)) / 8.0
        far = (5.0 - 2.0 * a - np.sqrt(np.maximum(0.0, -7.0 + 12.0 * a - 4.0 * a * a))) / 8.0
    return np.where(a <= 1.0, near, np.where(a <= 2.0, far, 0.0))


def _pipe_markers(nx, radius):
    """Ring markers of one plane as a sparse (markers, nx*nx) weight matrix,
    and the marker volume."""
    n = int(math.floor(2.0 * math.pi * radius + 0.5))
    th = 2.0 * math.pi * np.arange(n) / n
    mx, my = 0.5 * (nx - 1) + radius * np.cos(th), 0.5 * (nx - 1) + radius * np.sin(th)
    row, col, val = [], [], []
    for ky in range(-1, 3):
        for kx in range(-1, 3):
            gx, gy = np.floor(mx) + kx, np.floor(my) + ky
            row.append(np.arange(n))
            col.append(gx.astype(int) % nx + nx * (gy.astype(int) % nx))
            val.append(_peskin(gx - mx) * _peskin(gy - my))
    A = torch.sparse_coo_tensor(np.stack([np.concatenate(row), np.concatenate(col)]), np.concatenate(val),
                                (n, nx * nx), dtype=F64).coalesce().to(DEV)
    return A, A.t().coalesce(), 2.0 * math.pi * radius / n


def _z_smooth(a):
    """The four-point kernel on integer planes: 1/4, 1/2, 1/4 along dim 0."""
    return 0.5 * a + 0.25 * (torch.roll(a, 1, 0) + torch.roll(a, -1, 0))


def _pipe_state(case, seed, steps):
    """Populations of the pipe after `steps` steps, the force of the last
    collision, and the outside mask of a plane."""
    nx, nz, R = case["nx"], case["nz"], case["radius"]
    wall, q = case.get("wall", "ibb"), case.get("lattice", 19)
    c, w, opp = _velocities(q)
    tau = 3.0 * NU + 0.5
    out, links = _pipe_links(nx, R, c)
    if wall == "ibb" and links is None:
        return None
    if out is None:
        out = _pipe_radius2(nx) >= R * R
    body = torch.zeros((3, nz, nx, nx), dtype=F64, device=DEV)
    body[2] = _pipe_force(R) * (~out).to(F64)
    if wall != "ibb":
        A, At, dV = _pipe_markers(nx, R + (0.4 if wall == "ibm_b" else 0.0))
    u = _pipe_field(nx, nz, R, seed)
    f = _equilibrium(torch.ones_like(u[0]), u, c, w)
    F = body
    for _ in range(steps):
        g = _stream(f, c)
        if wall == "ibb":
            for i, l in enumerate(links):
                if l is None:
                    continue
                m, qq = l
                low = (2.0 * qq) * f[i][:, m] + (1.0 - 2.0 * qq) * g[i][:, m]
                high = (f[i][:, m] + (2.0 * qq - 1.0) * f[opp[i]][:, m]) / (2.0 * qq)
                low = torch.where(qq < 0.5, low, high)
                links[i] = (m, qq, low)
            for i, l in enumerate(links):
                if l is not None:
                    g[opp[i]][:, l[0]] = l[2]
                    links[i] = l[:2]
        else:
            rho, mom = _moments(g, c)
            us = (mom + 0.5 * body) / rho
            total = torch.zeros_like(body)
            flat = rho.reshape(nz, -1)
            rl = _z_smooth(torch.sparse.mm(A, flat.T.contiguous()).T)
            for _ in range(3):
                for d in range(3):
                    ul = _z_smooth(torch.sparse.mm(A, us[d].reshape(nz, -1).T.contiguous()).T)
                    fl = _z_smooth(-2.0 * rl * ul * dV)
                    fx = torch.sparse.mm(At, fl.T.contiguous()).T.reshape(nz, nx, nx)
                    us[d] += fx / (2.0 * rho)
                    total[d] += fx
            F = body + total
        _collide(g, F, tau, c, w)
        f = g
    return f, F, out, c


def _macro(f, F, c):
    rho, m = _moments(f, c)
    return rho, (m if F is None else m - 0.5 * F) / rho


def _exact_pipe(case, seed):
    s = _pipe_state(case, seed, case["steps"])
    if s is None:
        return None
    f, F, out, c = s
    rho, u = _macro(f, F, c)
    if case["wall"] == "ibb":  # cells outside the pipe report no velocity, and no density or that at rest
        rho, u = torch.where(out, 1.0 if case["lattice"] == 27 else 0.0, rho), u * ~out
    return dict(rho=rho.reshape(-1), u=u.reshape(3, -1))


def _exact_box(case, seed):
    c, w, _ = _velocities(19)
    K = _mrt_matrix(c, TAU_BOX)
    u = _turbulence(case["nx"], case["ny"], case["nz"], seed, 0.03, 8.0)
    f = _equilibrium(torch.ones_like(u[0]), u, c, w)
    for _ in range(case["steps"]):
        f = _stream(f, c)
        _collide(f, None, TAU_BOX, c, w, K)
    rho, u = _macro(f, None, c)
    return dict(rho=rho.reshape(-1), u=u.reshape(3, -1))


def _exact_sphere(case, seed):
    """One fixed sphere, quadratic interpolated bounce-back, momentum exchange."""
    n, R, tau = case["n"], case["radius"], 0.6
    c, w, opp = _velocities(19)
    x = torch.arange(n, dtype=F64, device=DEV) - (0.5 * n - 0.5)
    Z, Y, X = torch.meshgrid(x, x, x, indexing="ij")
    solid = X * X + Y * Y + Z * Z <= R * R
    links = []
    for v in c:
        s = lambda k: torch.roll(solid, shifts=(-k * v[2], -k * v[1], -k * v[0]), dims=(0, 1, 2))  # noqa: E731
        m = ~solid & s(1) if any(v) else torch.zeros_like(solid)
        if bool((s(-1)[m] | s(-2)[m]).any()):
            return None  # another scheme
        b, a = (X * v[0] + Y * v[1] + Z * v[2])[m], float(sum(t * t for t in v))
        q = (-b - torch.sqrt(b * b - a * ((X * X + Y * Y + Z * Z)[m] - R * R))) / max(a, 1.0)
        arm = torch.stack([X[m] + 0.5 * v[0], Y[m] + 0.5 * v[1], Z[m] + 0.5 * v[2]], 1)
        links.append((m, q, arm))
    F = torch.zeros((3, n, n, n), dtype=F64, device=DEV)
    F[0] = 1e-6 * (~solid).to(F64)
    u = _turbulence(n, n, n, seed, 0.01, 512.0 / n)
    f = _equilibrium(torch.ones_like(u[0]), u, c, w)
    for _ in range(case["steps"]):
        g = _stream(f, c)
        up2 = _stream(g, c)
        force, torque = torch.zeros(3, dtype=F64, device=DEV), torch.zeros(3, dtype=F64, device=DEV)
        vals = []
        for i, v in enumerate(c):
            m, q, arm = links[i]
            o, f0, f1, f2 = opp[i], f[i][m], g[i][m], up2[i][m]
            low = q * (1 + 2 * q) * f0 + (1 - 4 * q * q) * f1 - q * (1 - 2 * q) * f2
            # f_o at x - c_i: the value that streams against c_o
            fo1 = torch.roll(f[o], shifts=(v[2], v[1], v[0]), dims=(0, 1, 2))[m]
            high = f0 / (q * (2 * q + 1)) + (2 * q - 1) / q * f[o][m] - (2 * q - 1) / (2 * q + 1) * fo1
            val = torch.where(q < 0.5, low, high)
            vals.append(val)
            dP = (f0 + val)[:, None] * torch.tensor(v, dtype=F64, device=DEV)
            force += dP.sum(0)
            torque += torch.linalg.cross(arm, dP).sum(0)
        for i in range(len(c)):
            g[opp[i]][links[i][0]] = vals[i]
        _collide(g, F, tau, c, w)
        f = g
    rho, u = _macro(f, F, c)
    fl = (~solid).to(F64)
    centre = torch.full((1, 3), 0.5 * n - 0.5, dtype=F64)
    zero = torch.zeros((1, 3), dtype=F64)
    return dict(rho=(rho * fl).reshape(-1), u=(u * fl).reshape(3, -1), X=centre, U=zero, W=zero, F=force[None],
                T=torque[None])


def _gradients(u):
    """G[a][b] = du_a/dx_b, central differences on the periodic box."""
    d = lambda a, k: 0.5 * (torch.roll(a, -1, k) - torch.roll(a, 1, k))  # noqa: E731
    return [[d(u[a], 2), d(u[a], 1), d(u[a], 0)] for a in range(3)]


def _dissipation(G, nu):
    s = 0.0
    for a in range(3):
        for b in range(3):
            s = s + (0.5 * (G[a][b] + G[b][a])) ** 2
    return 2.0 * nu * s


def _network(w, X):
    o = 0
    for k, (a, b) in enumerate(zip(MLP_SIZES[:-1], MLP_SIZES[1:])):
        X = X @ w[o:o + a * b].reshape(a, b) + w[o + a * b:o + a * b + b]
        o += a * b + b
        X = torch.relu(X) if k < 3 else X
    return X


def _exact_closure(case, seed):
    X, T = _samples(case["n"], seed)
    Xh, _ = _samples(case["held"], seed + 1)
    X, T, Xh = X.to(F64), T.to(F64), Xh.to(F64)
    w = _weights(seed).to(F64)
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    step, loss = 0, 0.0
    for _ in range(case["epochs"]):
        loss = 0.0
        for s in range(0, case["n"], case["batch"]):
            p = w.clone().requires_grad_(True)
            d = _network(p, X[s:s + case["batch"]]) - T[s:s + case["batch"]]
            L = (d * d).mean()
            (g,) = torch.autograd.grad(L, p)
            loss = loss + L.detach() * d.numel()
            step += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            w = w - 1e-3 * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    return dict(w=w, loss=float(loss) / (case["n"] * 9), Y=_network(w, Xh))


def _exact_stats(case, seed):
    n, k, R = case["n"], case["np"], 4.0
    nu = (TAU_BOX - 0.5) / 3.0
    u = _turbulence(n, n, n, seed, 0.03, 8.0)
    Xh, Uh, Wh = _spheres(case, seed)
    X, U, W = (torch.tensor(a, dtype=F64, device=DEV) for a in (Xh, Uh, Wh))
    # every cell of a box around each particle: offset from its centre
    h = int(math.ceil(3.0 * R)) + 2
    o = torch.arange(-h, h + 1, device=DEV)
    oz, oy, ox = torch.meshgrid(o, o, o, indexing="ij")
    off = torch.stack([ox, oy, oz], -1).reshape(-1, 3)
    inf = 1e30
    dist = torch.full((n ** 3,), inf, dtype=F64, device=DEV)
    near = torch.zeros(n ** 3, dtype=torch.int64, device=DEV)
    for turn in (0, 1):  # the smallest distance, then whose it is
        for p0 in range(0, k, 256):
            base = torch.floor(X[p0:p0 + 256]).to(torch.int64)
            cell = base[:, None, :] + off[None]
            d = cell.to(F64) - X[p0:p0 + 256][:, None, :]
            r = torch.sqrt((d * d).sum(-1)).reshape(-1)
            cc = cell % n
            idx = (cc[..., 0] + n * (cc[..., 1] + n * cc[..., 2])).reshape(-1)
            if turn == 0:
                dist.scatter_reduce_(0, idx, r, "amin")
            else:
                own = r == dist[idx]
                pid = torch.arange(p0, min(p0 + 256, k), device=DEV)[:, None].expand(-1, off.shape[0]).reshape(-1)
                near[idx[own]] = pid[own]
    z, y, x = torch.meshgrid(*[torch.arange(n, device=DEV, dtype=F64)] * 3, indexing="ij")
    rel = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1) - X[near]
    rel -= n * torch.round(rel / n)
    rigid = U[near] + torch.linalg.cross(W[near], rel)
    solid = dist <= R
    fl = ~solid
    raw = u.reshape(3, -1)
    um = torch.where(solid, rigid.T, raw)
    eps = _dissipation(_gradients(um.reshape(3, n, n, n)), nu).reshape(-1)
    if case["closure"]:
        take = torch.nonzero(fl & (dist - R > 0) & (dist - R <= 2.0)).reshape(-1)
        w = _weights(seed).to(F64)
        for s in range(0, take.numel(), 1 << 18):
            t = take[s:s + (1 << 18)]
            tx, ty, tz = t % n, (t // n) % n, t // (n * n)
            feats = []
            for dz in (-1, 0, 1):
                for dy in (-1, 0, 1):
                    for dx in (-1, 0, 1):
                        q = (tx + dx) % n + n * ((ty + dy) % n + n * ((tz + dz) % n))
                        at = rel[t] + torch.tensor([dx, dy, dz], dtype=F64, device=DEV)
                        feats.append((raw[:, q].T - U[near[t]] - torch.linalg.cross(W[near[t]], at)) / U_SCALE)
            f = torch.cat(feats + [(dist[t] - R)[:, None], feats[13]], 1)
            G = (_network(w, f) / G_SCALE).T
            eps[t] = _dissipation([[G[3 * a + b] for b in range(3)] for a in range(3)], nu)
    ke = 0.5 * (um * um).sum(0)
    kf, ef = ke[fl].mean(), eps[fl].mean()
    b = torch.floor((dist / R - 1.0) / 0.05)
    ok = fl & (b >= 0) & (b < 40)
    bi = b[ok].to(torch.int64)
    cnt = torch.bincount(bi, minlength=40).to(F64)
    per = lambda q: torch.bincount(bi, weights=q[ok], minlength=40) / cnt.clamp(min=1.0)  # noqa: E731
    m = 5.0 * 4.0 / 3.0 * math.pi * R ** 3
    return dict(mass=float(n ** 3), momentum=raw.sum(1), kinetic_energy=float(ke.mean()), dissipation=float(eps.mean()),
                kinetic_energy_fluid=float(kf), dissipation_fluid=float(ef),
                particle_ke=float(0.5 * m * (U * U).sum()), particle_ake=float(0.2 * m * R * R * (W * W).sum()),
                force=None, torque=None, bulk_velocity=None, nbins=None,
                bin_r=1.0 + 0.05 * (torch.arange(40, dtype=F64) + 0.5), bin_tke=per(ke) / kf, bin_eps=per(eps) / ef,
                bin_count=None, nfluid=None, nlinks=None, nmarkers=None, step=None)


def _exact_spectrum(case, seed):
    n, nb = case["n"], case["nbins"]
    u = _turbulence(n, n, n, seed, 0.03, 8.0 * 256.0 / n)
    k = torch.fft.fftfreq(n, 1.0 / n, dtype=F64, device=DEV)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
    shell = torch.round(torch.sqrt(k2)).to(torch.int64).reshape(-1)
    e = sum(0.5 * (torch.fft.fftn(u[c]).abs() / n ** 3) ** 2 for c in range(3)).reshape(-1)
    d = 2.0 * (TAU_BOX - 0.5) / 3.0 * (2.0 * math.pi / n) ** 2 * k2.reshape(-1) * e
    return dict(E=torch.bincount(shell, weights=e, minlength=nb)[:nb], D=torch.bincount(shell, weights=d, minlength=nb)[:nb])


def _exact_budget(case, seed):
    """Bin means of the pipe's cylindrical velocity, and the production,
    transport, pressure, diffusion and dissipation terms of the fluctuations."""
    nx, nz, R, nb = case["nx"], case["nz"], case["radius"], case["nbins"]
    s = _pipe_state(dict(case, wall="ibb", lattice=19), seed, 20)
    if s is None:
        return None
    f, F, out, c = s
    nu = NU
    rho, u = _macro(f, F, c)
    u = u * ~out
    x = torch.arange(nx, dtype=F64, device=DEV) - 0.5 * (nx - 1)
    dx, dy = x[None, None, :].expand(nz, nx, nx), x[None, :, None].expand(nz, nx, nx)
    r = torch.sqrt(dx * dx + dy * dy)
    bins = torch.floor(r * nb / R).to(torch.int64)
    G = _gradients(u)
    eps = _dissipation(G, nu)

    def means(keep):
        b = bins[keep]
        cnt = torch.bincount(b, minlength=nb).to(F64)
        return b, lambda q: torch.bincount(b, weights=q, minlength=nb) / cnt.clamp(min=1.0)

    keep = (~out)[None].expand(nz, nx, nx) & (bins < nb)
    on_axis = r == 0
    sr = torch.where(on_axis, 1.0, r)
    ex, ey = torch.where(on_axis, 1.0, dx / sr), dy / sr
    ur, ut, uz = u[0] * ex + u[1] * ey, u[1] * ex - u[0] * ey, u[2]
    _, mean = means(keep)
    prof = torch.stack([mean(q[keep]) for q in (ur, ut, uz, ur * ur, ut * ut, uz * uz, ur * uz, ur * ut, ut * uz, rho,
                                                eps)], 1)
    keep = keep & ~on_axis
    b, mean = means(keep)
    E = [torch.stack([ex, ey, 0 * ex])[:, keep], torch.stack([-ey, ex, 0 * ex])[:, keep]]
    E.append(torch.stack([0 * E[0][0], 0 * E[0][0], 1 + 0 * E[0][0]]))
    Gk = [[G[a][k][keep] for k in range(3)] for a in range(3)]
    T = [[sum(E[i][a] * Gk[a][k] * E[j][k] for a in range(3) for k in range(3)) for j in range(3)] for i in range(3)]
    S = [[0.5 * (T[i][j] + T[j][i]) for j in range(3)] for i in range(3)]
    rk, v = r[keep], [ur[keep], ut[keep], uz[keep]]
    dth = [T[0][1] + v[1] / rk, T[1][1] - v[0] / rk, T[2][1]]
    p = rho[keep] / 3.0

    def avg(*qs):
        prod = 1.0
        for q in qs:
            prod = prod * (q - mean(q)[b])
        return mean(prod)

    h = R / nb
    rb = (torch.arange(nb, dtype=F64, device=DEV) + 0.5) * h
    ddr = lambda q: torch.gradient(q, spacing=h)[0]  # noqa: E731
    div = lambda q: ddr(rb * q) / rb  # noqa: E731
    diss = lambda i: -2.0 * nu * (avg(S[i][0], T[i][0]) + avg(S[i][1], dth[i]) + avg(S[i][2], T[i][2]))  # noqa: E731
    terms = [-avg(v[2], v[0]) * ddr(mean(v[2])), -div(0.5 * avg(v[2], v[2], v[0])), avg(p, T[2][2]),
             2 * nu * div(avg(v[2], S[2][0])), diss(2),
             -div(0.5 * avg(v[0], v[0], v[0])), -ddr(avg(v[0], p)) + avg(p, T[0][0]), 2 * nu * div(avg(v[0], S[0][0])),
             diss(0),
             -div(0.5 * avg(v[1], v[1], v[0])), avg(p, dth[1]), 2 * nu * div(avg(v[1], S[1][0])), diss(1)]
    has = torch.bincount(b, minlength=nb) > 0
    return dict(count=None, profiles=prof, budget_count=None, budget=torch.stack(terms, 1) * has[:, None])


def exact(case, seed):
    """The result of `run` on a new state in 64 bits. None for the moving
    suspensions: their particle dynamics has no statement short of a second
    implementation of the method; and for the rare wall that needs another
    interpolation than the usual one."""
    kind = case["kind"]
    if kind == "suspension":
        return None
    return dict(sphere=_exact_sphere, box=_exact_box, pipe=_exact_pipe, stats=_exact_stats, spectrum=_exact_spectrum,
                budget=_exact_budget, closure=_exact_closure)[kind](case, seed)
