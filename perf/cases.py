"""The work this solver is used for, as cases that can be timed and checked.

Each case is one pass through the public entry points of
``paper_2512_23116_gb300``: time steps of a forced large-eddy simulation, the
statistics a run takes at its cadence, a batch of runs, a snapshot of the
state, and the structure functions of a velocity field that a program already
holds.  ``exact`` restates the same pass in FP64 with torch alone.
"""
import math

import numpy as np
import torch

import paper_2512_23116_gb300 as lbm

DEV = "cuda"
U0, CF, RE = 0.043, 0.2, 2.0e4        # characteristic velocity, forcing amplitude, Re of the 100^3 LES
SPIN = 4                              # steps taken before a pass: the state has left its initial equilibrium
SEPARATIONS = (1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64)
STORAGE = {"fp32": lbm.LBM_FP32, "fp16": lbm.LBM_FP16_SHIFTED, "bf16": lbm.LBM_BF16_SHIFTED}
# slot order of a cell row in the row-interleaved array (include/lbm.h, lbm_device_ptr)
GPOS = (0, 1, 15, 4, 11, 8, 16, 5, 6, 17, 18, 3, 14, 7, 12, 9, 10, 13, 2)
FLOPS_PER_CELL = 230                  # collision of one cell


def _box(kind, name, nx, ny, nz, steps, storage="fp32", cs=0.13, nu0=0.0, strain=0, **more):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "steps": steps, "storage": storage, "cs": cs,
         "nu0": nu0 or U0 * nx / RE, "strain": strain, **more}
    return {"name": name, **c} if name else c


def listed():
    return [
        # a small box stepped in one call: launches and latency (the parity tests' and the smoke run's size)
        _box("step", "tgv32_100_steps", 32, 32, 32, 100, cs=0.1, nu0=0.01, init="tgv"),
        # a small LES whose program looks at it every 10 steps
        _box("step", "les64_10_steps", 64, 64, 64, 10),
        # the LES of the paper, between two statistics
        _box("step", "les100_100_steps", 100, 100, 100, 100),
        # the same with its statistics time series: spectrum, structure functions, theta slice
        _box("stats", "les100_series", 100, 100, 100, 50),
        # energy balance of an LES with the self-consistent strain: statistics fused into every 10th step
        _box("fused", "les128_balance", 128, 128, 128, 40, strain=1, every=10),
        # an uneven box, x-lines that end inside a 16-byte vector, bfloat16 storage
        _box("step", "ragged_bf16", 250, 190, 131, 10, storage="bf16"),
        # a large LES in half-precision storage
        _box("step", "les512_fp16", 512, 512, 512, 4, storage="fp16"),
        # the DNS-shape run
        _box("step", "dns800_fp32", 800, 800, 800, 2, cs=0.0),
        # statistics of a larger LES
        _box("stats", "stats400_fp16", 400, 400, 400, 2, storage="fp16"),
        # an ensemble of uneven boxes advanced together
        {"name": "batch12", "kind": "batch", "sizes": "64 96 100 128", "copies": 3, "steps": 20,
         "storage": "fp32", "cs": 0.13},
        # structure functions of a velocity field in a framework's own memory
        {"name": "increments160", "kind": "increments", "nx": 160, "ny": 160, "nz": 160, "separations": 12},
        # checkpoint and field output of a run, and its resumption, through host arrays
        _box("snapshot", "snapshot100", 100, 100, 100, 0),
    ]


def _extents(rng, lo, hi):
    """An uneven box of lo to hi cells (logarithmically spread), extents at least 12."""
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    n = cells ** (1.0 / 3.0)
    a, b = rng.uniform(0.75, 1.33), rng.uniform(0.75, 1.33)
    nx, ny = max(12, round(n * a)), max(12, round(n * b))
    if rng.random() < 0.4:  # sizes with many small factors are common
        nx, ny = max(12, nx // 4 * 4), max(12, ny // 4 * 4)
    return nx, ny, max(12, round(cells / (nx * ny)))


def _steps(rng, cells, most):
    top = max(2, min(128, int(most / cells)))
    return max(2, int(math.exp(rng.uniform(math.log(2), math.log(top)))) // 2 * 2)


def draw(rng):
    kind = rng.choices(["step", "stats", "fused", "batch", "increments", "snapshot"], [10, 4, 2, 2, 2, 1])[0]
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    strain = 1 if rng.random() < 0.2 else 0
    if kind == "step":
        nx, ny, nz = _extents(rng, 2e4, 4e8)
        cells = nx * ny * nz
        dns = cells > 2e7 and rng.random() < 0.4
        return _box(kind, None, nx, ny, nz, _steps(rng, cells, 8e8), storage, 0.0 if dns else round(rng.uniform(0.1, 0.16), 3),
                    nu0=max(U0 * nx / RE, 2e-4), strain=strain)
    if kind == "stats":
        nx, ny, nz = _extents(rng, 2e5, 1e8)
        return _box(kind, None, nx, ny, nz, _steps(rng, nx * ny * nz, 5e7), storage, nu0=max(U0 * nx / RE, 2e-4), strain=strain)
    if kind == "fused":
        nx, ny, nz = _extents(rng, 1e5, 2e7)
        return _box(kind, None, nx, ny, nz, 40, storage, nu0=max(U0 * nx / RE, 2e-4), strain=strain, every=rng.choice([5, 10, 20]))
    if kind == "batch":
        sizes = sorted(rng.choice([32, 48, 50, 64, 80, 96, 100, 112, 128]) for _ in range(rng.randint(2, 4)))
        return {"kind": kind, "sizes": " ".join(map(str, sizes)), "copies": rng.randint(1, 3), "steps": 2 * rng.randint(5, 20),
                "storage": storage, "cs": 0.13}
    if kind == "increments":
        nx, ny, nz = _extents(rng, 1e5, 1e7)
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "separations": rng.randint(3, len(SEPARATIONS))}
    nx, ny, nz = _extents(rng, 5e4, 1.5e6)
    return _box(kind, None, nx, ny, nz, 0, storage, nu0=max(U0 * nx / RE, 2e-4))


# ---- inputs ------------------------------------------------------------------------


def _boxes(case):
    """(nx, ny, nz, nu0) of every instance of a case."""
    if case["kind"] != "batch":
        return [(case["nx"], case["ny"], case["nz"], case["nu0"])]
    return [(n, n, n, U0 * n / RE) for n in map(int, case["sizes"].split()) for _ in range(case["copies"])]


def _wavenumbers(n, half=False):
    k = torch.fft.rfftfreq(n, device=DEV) if half else torch.fft.fftfreq(n, device=DEV)
    return k * n


def _random_velocity(nx, ny, nz, seed, urms):
    """A random solenoidal field [3][nz][ny][nx] in FP32, energy spectrum s^4 exp(-2 (s/4)^2)."""
    gen = torch.Generator(DEV).manual_seed(seed)
    kx, ky, kz = _wavenumbers(nx, True), _wavenumbers(ny)[:, None], _wavenumbers(nz)[:, None, None]
    s = torch.sqrt(kx * kx + ky * ky + kz * kz)
    cut = min(24, min(nx, ny, nz) // 2 - 1)
    amp = torch.where((s > 0) & (s <= cut), s * torch.exp(-(s / 4.0) ** 2), torch.zeros_like(s))
    spec = [torch.fft.rfftn(torch.randn(nz, ny, nx, generator=gen, device=DEV)) * amp for _ in range(3)]
    q = (kx / nx, ky / ny, kz / nz)  # the box may be uneven: solenoidal in lattice units
    q2 = q[0] ** 2 + q[1] ** 2 + q[2] ** 2
    q2[0, 0, 0] = 1.0
    along = (q[0] * spec[0] + q[1] * spec[1] + q[2] * spec[2]) / q2
    u = torch.empty(3, nz, ny, nx, device=DEV)
    for d in range(3):
        u[d] = torch.fft.irfftn(spec[d] - q[d] * along, s=(nz, ny, nx))
        spec[d] = None
    u *= urms / math.sqrt(sum(float(u[d].square().mean()) for d in range(3)) / 3.0)
    return u


def _urms(case):
    return 0.05 if case["cs"] > 0 else 0.0289  # C = 0: sqrt(<u.u>) = 0.05, from which the scheme stays stable


def _tgv_amplitude(seed):
    return 0.04 + 0.02 * ((seed * 0.6180339887498949) % 1.0)


class _DeviceArray:
    """__cuda_array_interface__ of memory that a lattice owns."""

    def __init__(self, lattice, ptr, shape, typestr):
        self.lattice = lattice
        self.__cuda_array_interface__ = {"shape": shape, "typestr": typestr, "data": (ptr, False), "version": 3,
                                         "strides": None}


def _populations_in_place(lat, inst, storage, whole=False):
    """The population array of an instance as torch sees it, without a copy (at
    an even time slot a of a cell holds its f'_a): a list of 19 [nz][ny][nx], or
    whole as [19][nz][ny][nx] where the handle keeps the population-major order."""
    ptr, _, nxp = lbm.lbm_device_ptr(lat.h, inst)
    nz, ny, nx = lat.shapes[inst]
    rows = lat.config()["layout"] == 2
    shape = (nz, ny, 19, nxp) if rows else (19, nz, ny, nxp)
    a = torch.as_tensor(_DeviceArray(lat, ptr, shape, {"fp32": "<f4", "fp16": "<f2", "bf16": "<i2"}[storage]), device=DEV)
    if storage == "bf16":
        a = a.view(torch.bfloat16)
    if whole:
        return a[:, :, :, :nx]
    return [a[:, :, GPOS[k], :nx] if rows else a[k, :, :, :nx] for k in range(19)]


def prepare(case, seed):
    if case["kind"] == "increments":
        r = list(SEPARATIONS[:case["separations"]])
        return {"case": case, "u": _random_velocity(case["nx"], case["ny"], case["nz"], seed, 0.05), "r": r,
                "sp": torch.empty(len(r), 6, dtype=torch.float64, device=DEV), "stream": torch.cuda.current_stream()}
    batch = case["kind"] == "batch"
    params = [lbm.make_params(nx, ny, nz, precision=STORAGE[case["storage"]], nu0=nu0, cs=case["cs"], f0=CF * U0 * U0 / nx,
                              force_mode=lbm.LBM_FORCE_PAPER_SIN, strain_mode=case.get("strain", 0),
                              stats_every=case.get("every", 0), layout=1 if batch else 0)
              for nx, ny, nz, nu0 in _boxes(case)]
    lat = lbm.Lattice(params)
    for i, (nx, ny, nz, _) in enumerate(_boxes(case)):
        if case.get("init") == "tgv":
            lat.init(lbm.LBM_INIT_TGV3D, amplitude=_tgv_amplitude(seed), inst=i)
        else:
            u = _random_velocity(nx, ny, nz, seed + 1000 * i, _urms(case))
            lat.init(lbm.LBM_INIT_VELOCITY, u=u, inst=i)
            lat.sync()  # the kernel has read u
            del u
    torch.cuda.empty_cache()  # the lattice's memory is the library's own
    lat.step(SPIN)
    if case["kind"] == "fused":
        lat.series()  # the records of the steps above
    lat.sync()
    f = [_populations_in_place(lat, i, case["storage"], whole=batch) for i in range(len(params))]
    return {"case": case, "lat": lat, "f": f if batch else f[0]}


# ---- one pass ------------------------------------------------------------------------


def _max_shell(nx, ny, nz):
    return math.floor(math.sqrt((nx // 2) ** 2 + (ny // 2) ** 2 + (nz // 2) ** 2) + 0.5)


def _statistics(st, spectrum, theta):
    """What a series keeps of a state.  The sums run over FP32 values of the
    cells in an order that depends on the kernel configuration the handle has
    picked, so they are kept in FP32; mass and momentum, which are conserved and
    hold rounding alone, are not kept."""
    f32 = np.float32
    return {"energy": f32([st["E_k"], st["inj"], st["eps0"], st["eps_sgs"]]), "uu": f32(st["uu"]),
            "theta": f32([st["theta_mean"], st["theta_min"], st["theta_max"]]), "theta_var": f32(st["theta_var"]),
            "theta_percentiles": f32([st[k] for k in ("theta_p05", "theta_p50", "theta_p95", "theta_p99")]),
            "scales": [f32(st[k]) for k in ("L", "eps_spec", "eta", "lambda", "u_rms", "Re_lambda")],
            "S12": f32(st["Sp"][:, 0:2]), "S34": f32(st["Sp"][:, 2:4]), "S56": f32(st["Sp"][:, 4:6]), "F4": f32(st["F4"]),
            "r": np.array(st["r"], dtype=np.int64), "spectrum": f32(spectrum), "theta_slice": f32(theta)}


def _records(rec):
    f32 = np.float32
    return {"step": np.array([r["step"] for r in rec], dtype=np.int64),
            "energy": f32([[r["E_k"], r["inj"], r["eps0"], r["eps_sgs"]] for r in rec]),
            "theta": f32([[r["theta_mean"], r["theta_min"], r["theta_max"]] for r in rec]),
            "theta_var": f32([r["theta_var"] for r in rec])}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "increments":
        lbm.lbm_structure_functions_noalloc(state["u"], state["r"], state["sp"], stream=state["stream"])
        return state["sp"]
    lat = state["lat"]
    if kind == "snapshot":
        f = lat.populations()
        fields = lat.fields()
        lat.set_populations(f)
        return {"populations": f, "fields": fields, "f": state["f"]}
    lat.step(case["steps"])
    if kind == "stats":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        st = lat.stats(what=lbm.LBM_STATS_SPECTRUM | lbm.LBM_STATS_STRUCTURE)
        out = _statistics(st, lat.spectrum(_max_shell(nx, ny, nz)), lat.theta_slice(2, nz // 2))
        return {"f": state["f"], **out}
    if kind == "fused":
        return {"f": state["f"], **_records(lat.series())}
    return {"f": state["f"]}


def work(case):
    """One pass reads its state once and writes it once, however many steps it
    takes; the flops are those of its collisions, of the transforms and of the
    increments."""
    kind = case["kind"]
    size = 4 if case.get("storage", "fp32") == "fp32" else 2
    if kind == "increments":
        cells = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 12 * cells, "flops": cells * 3 * 12 * case["separations"]}
    cells = sum(nx * ny * nz for nx, ny, nz, _ in _boxes(case))
    if kind == "snapshot":  # populations read and written; the host arrays written and read
        return {"bytes": cells * (3 * 19 * size + 2 * 19 * 8 + 6 * 8), "flops": cells * FLOPS_PER_CELL}
    w = {"bytes": 2 * 19 * size * cells, "flops": case["steps"] * cells * FLOPS_PER_CELL}
    if kind == "stats":
        seps = len(_separations(min(case["nx"], case["ny"], case["nz"])))
        w["flops"] += cells * (FLOPS_PER_CELL + 3 * 2.5 * math.log2(cells) + 3 * 12 * seps)
    return w


# ---- the same in FP64 ------------------------------------------------------------------

_C = np.array([[1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 0], [-1, -1, 0], [1, -1, 0],
               [-1, 1, 0], [0, 1, 1], [0, -1, -1], [0, 1, -1], [0, -1, 1], [1, 0, 1], [-1, 0, -1], [1, 0, -1], [-1, 0, 1],
               [0, 0, 0]])


def _moment_matrix():
    x, y, z = (_C[:, k].astype(float) for k in range(3))
    c2 = x * x + y * y + z * z
    return torch.tensor(np.array([
        1 + 0 * c2, 19 * c2 - 30, (21 * c2 * c2 - 53 * c2 + 24) / 2, x, (5 * c2 - 9) * x, y, (5 * c2 - 9) * y, z, (5 * c2 - 9) * z,
        3 * x * x - c2, (3 * c2 - 5) * (3 * x * x - c2), y * y - z * z, (3 * c2 - 5) * (y * y - z * z), x * y, y * z, x * z,
        (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z]), dtype=torch.float64, device=DEV)


def _equilibrium_moments(drho, u):
    """m^eq of density 1 + drho and velocity u (App. B)."""
    rho = 1 + drho
    ux, uy, uz = u
    uu = ux * ux + uy * uy + uz * uz
    zero = torch.zeros_like(ux)
    return torch.stack([drho, -11 * drho + 19 * rho * uu, -475 / 63 * rho * uu, rho * ux, -2 / 3 * rho * ux, rho * uy,
                        -2 / 3 * rho * uy, rho * uz, -2 / 3 * rho * uz, rho * (2 * ux * ux - uy * uy - uz * uz), zero,
                        rho * (uy * uy - uz * uz), zero, rho * ux * uy, rho * uy * uz, rho * ux * uz, zero, zero, zero])


class _Reference:
    """One box in FP64: pre-collision weight-shifted populations f [19][nz][ny][nx]."""

    def __init__(self, nx, ny, nz, nu0, cs, strain, u):
        self.shape, self.nu0, self.cs, self.strain = (nz, ny, nx), nu0, cs, strain
        f0 = CF * U0 * U0 / nx
        wave = lambda n: f0 * torch.sin(2 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n)  # noqa: E731
        self.fx, self.fy, self.fz = wave(ny)[None, :, None], wave(nz)[:, None, None], wave(nx)[None, None, :]
        self.M = _moment_matrix()
        self.inv = self.M.T / (self.M * self.M).sum(1)
        self.f = torch.empty(19, nz, ny, nx, dtype=torch.float64, device=DEV)
        for z in self.planes():
            v = [u[d][z].double() for d in range(3)]
            self.f[:, z] = torch.tensordot(self.inv, _equilibrium_moments(torch.zeros_like(v[0]), v), 1)

    def planes(self):
        nz, ny, nx = self.shape
        n = max(1, (8 << 20) // (ny * nx))
        return [slice(z, min(z + n, nz)) for z in range(0, nz, n)]

    def cells(self, z):
        """Moments, force and fields of the planes z."""
        m = torch.tensordot(self.M, self.f[:, z], 1)
        like = torch.zeros_like(m[0])
        F = [self.fx + like, self.fy[z] + like, self.fz + like]
        rho = 1 + m[0]
        u = [(m[k] + 0.5 * F[d]) / rho for d, k in enumerate((3, 5, 7))]
        eq = _equilibrium_moments(m[0], u)
        n = m - eq
        trace = 1.19 / 38 * n[1]
        txx, tyy, tzz = -0.5 * n[9], 0.25 * (n[9] - 3 * n[11]), 0.25 * (n[9] + 3 * n[11])
        tt = txx ** 2 + tyy ** 2 + tzz ** 2 + 4.5 * (n[13] ** 2 + n[14] ** 2 + n[15] ** 2)
        b = 0.5 + 3 * self.nu0
        s = torch.sqrt(2 * (tt / b ** 2 + 3 * trace ** 2))
        if self.strain:  # |S| with the shear rate it gives itself: bisection between 0 and the bare one's
            lo, hi = torch.zeros_like(s), s.clone()
            for _ in range(60):
                mid = 0.5 * (lo + hi)
                low = mid * mid < 2 * (tt / (b + 3 * self.cs * mid) ** 2 + 3 * trace ** 2)
                lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
            s = 0.5 * (lo + hi)
        return m, F, u, n, s, 3 * (self.nu0 + self.cs * s)

    def step(self):
        for z in self.planes():
            m, F, u, n, s, theta = self.cells(z)
            rate = 1 / (0.5 + theta)
            one = torch.ones_like(rate)
            rates = [one, 1.19, 1.4, one, 1.2, one, 1.2, one, 1.2, rate, 1.4, rate, 1.4, rate, rate, rate, 1.98, 1.98, 1.98]
            uf = sum(u[d] * F[d] for d in range(3))
            t, w = 3 * u[0] * F[0] - uf, u[1] * F[1] - u[2] * F[2]
            force = [0, 38 * uf, -11 * uf, F[0], -2 / 3 * F[0], F[1], -2 / 3 * F[1], F[2], -2 / 3 * F[2], 2 * t, -t, 2 * w, -w,
                     u[1] * F[0] + u[0] * F[1], u[2] * F[1] + u[1] * F[2], u[2] * F[0] + u[0] * F[2], 0, 0, 0]
            for k in range(19):
                m[k] += (1 - 0.5 * rates[k]) * force[k] - rates[k] * n[k]
            self.f[:, z] = torch.tensordot(self.inv, m, 1)
        for a in range(18):
            x, y, z = (int(v) for v in _C[a])
            self.f[a] = torch.roll(self.f[a], (z, y, x), (0, 1, 2))

    def fields(self):
        out = {"drho": [], "u": [], "snorm": [], "theta": []}
        for z in self.planes():
            m, _, u, _, s, theta = self.cells(z)
            for k, v in (("drho", m[0]), ("u", torch.stack(u)), ("snorm", s), ("theta", theta)):
                out[k].append(v.clone())
        return {k: torch.cat(v, 1 if k == "u" else 0) for k, v in out.items()}

    def energy(self, g):
        u, s = g["u"], g["snorm"]
        inj = (self.fx * u[0]).mean() + (self.fy * u[1]).mean() + (self.fz * u[2]).mean()
        return [float(v) for v in (0.5 * sum(u[d].square().mean() for d in range(3)), inj, self.nu0 * s.square().mean(),
                                   self.cs * (s ** 3).mean())]

    @staticmethod
    def theta(g):
        return [float(g["theta"].mean()), float(g["theta"].min()), float(g["theta"].max())]


def _separations(n):
    r = set()
    k = 1
    while k <= n // 2:
        r.add(k)
        if k >= 2 and 3 * k // 2 <= n // 2:
            r.add(3 * k // 2)
        k *= 2
    return sorted(r)[:24]


def _structure(u, r):
    sp = torch.empty(len(r), 6, dtype=torch.float64, device=DEV)
    for i, k in enumerate(r):
        tot = [0.0] * 6
        for a, dim in enumerate((2, 1, 0)):
            d = torch.roll(u[a].double(), -k, dim) - u[a].double()
            p = d.clone()
            for q in range(6):
                tot[q] = tot[q] + p.sum()
                p *= d
        sp[i] = torch.stack(tot) / (3.0 * u[0].numel())
    return sp


def _spectrum(u, shells):
    _, nz, ny, nx = u.shape
    kx, ky, kz = (_wavenumbers(n, h).double().round() for n, h in ((nx, True), (ny, False), (nz, False)))
    kx, ky, kz = kx.abs(), ky.abs()[:, None], kz.abs()[:, None, None]
    shell = torch.floor(torch.sqrt(kx * kx + ky * ky + kz * kz) + 0.5).long().reshape(-1)
    twice = torch.full((nx // 2 + 1,), 2.0, dtype=torch.float64, device=DEV)
    twice[0] = 1.0
    if nx % 2 == 0:
        twice[-1] = 1.0
    E = torch.zeros(shells + 1, dtype=torch.float64, device=DEV)
    for d in range(3):
        e = torch.fft.rfftn(u[d]).abs().square_() * twice
        E.index_add_(0, shell, (0.5 / float(nx * ny * nz) ** 2 * e).reshape(-1))
    return E


def _exact_statistics(ref, case):
    g = ref.fields()
    u, theta = g["u"], g["theta"]
    nx, ny, nz, nu0 = case["nx"], case["ny"], case["nz"], case["nu0"]
    E = _spectrum(u, _max_shell(nx, ny, nz))
    k = 2 * math.pi * torch.arange(1, E.numel(), device=DEV, dtype=torch.float64) / nx
    urms = math.sqrt(sum(float(u[d].square().mean()) for d in range(3)) / 3)
    eps = 2 * nu0 * float((k * k * E[1:]).sum())
    lam = math.sqrt(15 * nu0 * urms * urms / eps)
    r = _separations(min(nx, ny, nz))
    sp = _structure(u, r)
    pairs = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
    arr = np.array
    return {"energy": arr(ref.energy(g)), "uu": arr([float((u[i] * u[j]).mean()) for i, j in pairs]), "theta": arr(ref.theta(g)),
            "theta_var": arr(float(theta.var(unbiased=False))), "theta_percentiles": None,
            "scales": [arr(v) for v in (0.75 * math.pi * float((E[1:] / k).sum() / E[1:].sum()), eps, (nu0 ** 3 / eps) ** 0.25, lam, urms,
                                        urms * lam / nu0)],
            "S12": sp[:, 0:2], "S34": sp[:, 2:4], "S56": sp[:, 4:6], "F4": sp[:, 3] / sp[:, 1] ** 2,
            "r": arr(r), "spectrum": E, "theta_slice": theta[nz // 2].clone()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "increments":
        u = _random_velocity(case["nx"], case["ny"], case["nz"], seed, 0.05)
        return _structure(u, SEPARATIONS[:case["separations"]])
    out = []
    for i, (nx, ny, nz, nu0) in enumerate(_boxes(case)):
        if case.get("init") == "tgv":
            X, Y, Z = (2 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n for n in (nx, ny, nz))
            Y, Z, A = Y[:, None], Z[:, None, None], _tgv_amplitude(seed)
            u = [A * torch.sin(X) * torch.cos(Y) * torch.cos(Z), -A * torch.cos(X) * torch.sin(Y) * torch.cos(Z), 0 * (X + Y + Z)]
        else:
            u = _random_velocity(nx, ny, nz, seed + 1000 * i, _urms(case))
        ref = _Reference(nx, ny, nz, nu0, case["cs"], case.get("strain", 0), u)
        del u
        recs = []
        for t in range(SPIN + case["steps"]):
            if kind == "fused" and t >= SPIN and t % case["every"] == 0:
                g = ref.fields()
                recs.append((t, ref.energy(g), ref.theta(g), float(g["theta"].var(unbiased=False))))
            ref.step()
        out.append(ref)
    if kind == "batch":
        return {"f": [r.f for r in out]}
    f = [ref.f[a] for a in range(19)]
    if kind == "stats":
        return {"f": f, **_exact_statistics(ref, case)}
    if kind == "fused":
        t, e, th, var = (np.array(v) for v in zip(*recs))
        return {"f": f, "step": t, "energy": e, "theta": th, "theta_var": var}
    if kind == "snapshot":
        return {"populations": ref.f, "fields": ref.fields(), "f": f}
    return {"f": f}
