"""Performance cases of the batched 1D-TDSE engine: what its users run, through its public calls.

listed() names twelve cases, draw() gives more of the same ranges; prepare() makes a case's inputs and
the handle a program keeps, run() is one pass, work() what a pass cannot do without, exact() the same
result in plain torch, in 64 bits.  Sizes are the library's own workloads (inputs.py, bench.py, tests)
or scaled from them: a chunk of steps near the pulse's peak stands for a chunked propagation.
"""
import math
import random
from fractions import Fraction

import numpy as np
import torch

from paper_2507_04115_gb300 import inputs, tdse

MASK = (20.0, 0.125)          # the workloads' absorber: outer 20 a.u., cos^(1/8)
SOFT = 1.19                   # argon-like soft-core parameter
GS = dict(dtau=0.1, max_iter=400, tol=0.0)   # a fixed number of iterations, as the tests use
HARTREE_TIME_S = 2.4188843265857e-17
C_M_S = 299792458.0
MU0 = 1.25663706212e-6
UNEVEN_N = (1024, 2048, 4096, 8192)


def listed():
    return [
        # one atom, the smallest call: latency of the serial sweeps
        dict(name="single_atom_fp64", kind="propagate", n=1, N=2000, dx=0.2, dt=0.05, steps=512, ragged=False,
             scheme="full_cn", precision="fp64"),
        # a line of radii on an odd grid with pulses of different lengths, single-precision states
        dict(name="radial_line_odd_mixed", kind="propagate", n=333, N=1537, dx=0.2, dt=0.05, steps=301, ragged=True,
             scheme="full_cn", precision="mixed"),
        # the macroscopic volume (64 radii x 128 planes), a chunk of a propagation: the main workload,
        # in both precisions and with the paper's own scheme
        dict(name="volume_fp64", kind="propagate", n=8192, N=4096, dx=0.15, dt=0.02, steps=160, ragged=False,
             scheme="full_cn", precision="fp64"),
        dict(name="volume_mixed", kind="propagate", n=8192, N=4096, dx=0.15, dt=0.02, steps=160, ragged=False,
             scheme="full_cn", precision="mixed"),
        dict(name="volume_numerov_fp64", kind="propagate", n=8192, N=4096, dx=0.15, dt=0.02, steps=160, ragged=False,
             scheme="numerov", precision="fp64"),
        # a parameter scan: mixed grids, spacings and pulse lengths in one batch
        dict(name="uneven_scan_fp64", kind="uneven", n=1024, steps=300, dt=0.02, precision="fp64"),
        # field shaping: forward and backward through the propagation (torch.autograd)
        dict(name="adjoint_volume_fp64", kind="adjoint", n=1024, N=2048, dx=0.15, dt=0.02, steps=96, ckpt=32),
        # initial states of the scan's grids
        dict(name="ground_states", kind="ground", grids=8, N=8192, iters=600, scheme="full_cn"),
        # coarse fields of a beam propagation brought onto the time grid of the volume batch
        dict(name="field_resampling", kind="resample", rows=256, M=2400, dt_c=0.5, dt_f=0.02, n_fine=55160),
        # harmonic spectra up to harmonic 40 of a 10-cycle pulse, plain DFT of every row
        dict(name="harmonic_spectra", kind="spectrum", rows=512, L=55160, k0=0, k1=400, ragged=False),
        # the far field of a volume: source spectrum of every row, then the direct Hankel integration
        dict(name="far_field", kind="far", n_r=32, n_z=32, L=27580, n_w=340, n_obs=256),
        # electron energy distribution and populations of a batch's states
        dict(name="energy_distribution", kind="energy", n=1024, N=4096, dx=0.15, dt=0.02, n_E=128, eps=0.02,
             scheme="full_cn", precision="fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["propagate"] * 5 + ["uneven", "adjoint", "ground", "resample", "spectrum", "far", "energy"])
    dx, dt = rng.choice([(0.15, 0.02), (0.2, 0.05), (0.2, 0.02)])
    if kind == "propagate":
        N, n = _log(rng, 500, 8192), _log(rng, 1, 8192)
        steps = max(16, min(_log(rng, 60, 400), int(4.0e9 / (N * n))))
        scheme = rng.choice(["full_cn", "full_cn", "numerov"])
        if scheme == "numerov":
            N -= N % 2       # the grids of the workloads with this scheme are even
        return dict(kind=kind, n=n, N=N, dx=dx, dt=dt, steps=steps, ragged=rng.random() < 0.3,
                    scheme=scheme, precision=rng.choice(["fp64", "fp64", "mixed"]))
    if kind == "uneven":
        return dict(kind=kind, n=_log(rng, 64, 2048), steps=rng.randint(100, 300), dt=0.02,
                    precision=rng.choice(["fp64", "mixed"]))
    if kind == "adjoint":
        n, N = _log(rng, 8, 1024), _log(rng, 700, 2048)
        return dict(kind=kind, n=n, N=N, dx=dx, dt=dt, steps=rng.randint(40, 96), ckpt=rng.choice([16, 32, 64]))
    if kind == "ground":
        return dict(kind=kind, grids=rng.randint(1, 8), N=_log(rng, 500, 8192), iters=rng.randint(200, 600),
                    scheme=rng.choice(["full_cn", "numerov"]))
    if kind == "resample":
        M = _log(rng, 100, 4000)
        dt_c = rng.choice([0.25, 0.5, 1.0])
        dt_f = rng.choice([0.02, 0.05])
        return dict(kind=kind, rows=_log(rng, 4, 200), M=M, dt_c=dt_c, dt_f=dt_f,
                    n_fine=min(55160, max(64, int(0.9 * M * dt_c / dt_f))))
    if kind == "spectrum":
        L = _log(rng, 2000, 55160)
        k1 = min(L, _log(rng, 60, 400))
        return dict(kind=kind, rows=_log(rng, 1, 512), L=L, k0=rng.choice([0, k1 // 3]), k1=k1,
                    ragged=rng.random() < 0.3)
    if kind == "far":
        return dict(kind=kind, n_r=rng.randint(8, 32), n_z=rng.randint(1, 32), L=_log(rng, 2000, 27580),
                    n_w=_log(rng, 30, 340), n_obs=_log(rng, 30, 256))
    return dict(kind="energy", n=_log(rng, 8, 512), N=_log(rng, 500, 4096), dx=dx, dt=dt, n_E=_log(rng, 16, 128),
                eps=rng.choice([0.01, 0.02, 0.05]), scheme=rng.choice(["full_cn", "numerov"]),
                precision=rng.choice(["fp64", "mixed"]))


# ------------------------------------------------------------------------------------------- inputs

def _dev():
    return torch.device("cuda", 0)


def _case_seed(seed):
    return np.random.default_rng(int(seed) + 12345)


def _pulse_rows(rng, nts, dt):
    """Rows E(t0 + n dt), n = 0..nt, of 800 nm pulses near their envelope's peak: intensities of a
    focused beam (5e13 to 2e14 W/cm^2), carrier phases over the beam.  Returns the flat rows, offsets."""
    n = len(nts)
    w = inputs.omega_from_wavelength_nm(800.0)
    E0 = inputs.field_from_intensity(np.exp(rng.uniform(math.log(5e13), math.log(2e14), n)))
    phi = rng.uniform(0.0, 2.0 * math.pi, n)
    offs = np.concatenate([[0], np.cumsum(np.asarray(nts, dtype=np.int64) + 1)])
    dev = _dev()
    nmax = int(max(nts))
    t = torch.arange(nmax + 1, dtype=torch.float64, device=dev) * dt
    env = torch.cos((t - 0.5 * nmax * dt) * w / 20.0) ** 2       # the centre of a 10-cycle sin^2 envelope
    full = torch.from_numpy(E0).to(dev)[:, None] * env[None, :] * torch.cos(w * t[None, :] + torch.from_numpy(phi).to(dev)[:, None])
    if all(int(k) == nmax for k in nts):
        return full.reshape(-1).contiguous(), offs
    keep = torch.arange(nmax + 1, device=dev)[None, :] <= torch.from_numpy(np.asarray(nts, dtype=np.int64)).to(dev)[:, None]
    return full[keep].contiguous(), offs


def _geometry(case):
    """Per-instance (N, dx, nt) of a propagation case, the same for every seed."""
    n = case["n"]
    rng = np.random.default_rng(2)
    if case["kind"] == "uneven":
        N = rng.choice(np.array(UNEVEN_N), n)
        dx = rng.choice(np.array([0.15, 0.2]), n)
        cyc = rng.integers(4, 17, n)
        lam = rng.choice(np.array([800.0, 1030.0, 1800.0]), n)
        nt = np.maximum(16, np.rint(case["steps"] * (cyc / 16.0) * (lam / 1800.0))).astype(np.int64)
        return N, dx, nt
    nt = np.full(n, case["steps"], dtype=np.int64)
    if case.get("ragged"):
        nt = rng.integers(max(16, case["steps"] // 3), case["steps"] + 1, n)
        nt[0] = case["steps"]
    return np.full(n, case["N"]), np.full(n, case["dx"]), nt


def _scheme(case):
    return tdse.TDSE_NUMEROV_SPLIT if case.get("scheme") == "numerov" else tdse.TDSE_FULL_CN


def _precision(case):
    return tdse.TDSE_MIXED if case.get("precision") == "mixed" else tdse.TDSE_FP64


def _a_rows(rng, offs, dt):
    """Dipole-acceleration rows: odd harmonics of 800 nm falling off over a plateau, under a sin^2 envelope."""
    dev = _dev()
    n = len(offs) - 1
    L = int(max(offs[1:] - offs[:-1]))
    w = inputs.omega_from_wavelength_nm(800.0)
    t = torch.arange(L, dtype=torch.float64, device=dev) * dt
    out = torch.zeros((n, L), dtype=torch.float64, device=dev)
    for q in range(1, 30, 4):
        amp = torch.from_numpy(rng.uniform(0.5, 1.5, n) * 10.0 ** (-0.1 * q)).to(dev)
        ph = torch.from_numpy(rng.uniform(0.0, 2.0 * math.pi, n)).to(dev)
        out += amp[:, None] * torch.cos(q * w * t[None, :] + ph[:, None])
    out *= (torch.sin(math.pi * torch.arange(L, dtype=torch.float64, device=dev) / L) ** 2)[None, :]
    lens = torch.from_numpy(np.asarray(offs[1:] - offs[:-1])).to(dev)
    keep = torch.arange(L, device=dev)[None, :] < lens[:, None]
    return out[keep].contiguous()


def _far_grids(case):
    k = np.arange(1, case["n_w"] + 1)
    om = 2.0 * math.pi * k / (27580 * 0.02)
    return dict(om=om, k=om / HARTREE_TIME_S / C_M_S, rho=np.linspace(0.0, 50e-6, case["n_r"]),
                z=np.linspace(-5e-3, 5e-3, case["n_z"]) if case["n_z"] > 1 else np.array([0.0]),
                ro=np.linspace(0.0, 5e-3, case["n_obs"]), z_obs=0.5)


def _packets(rng, n, N, dx):
    """States after ionisation: a bound part at the nucleus and wave packets running out, norm 1 (n x N)."""
    dev = _dev()
    x = (torch.arange(N, dtype=torch.float64, device=dev) - 0.5 * (N - 1)) * dx

    def col(v):
        return torch.from_numpy(v).to(dev)[:, None]

    half = 0.3 * N * dx
    psi = col(rng.uniform(0.8, 1.0, n)) * torch.exp(-torch.sqrt(x * x + 1.0))[None, :].to(torch.complex128)
    for amp in (0.3, 0.1, 0.03):
        x0, p0 = col(rng.uniform(-half, half, n)), col(rng.uniform(-1.8, 1.8, n))
        s = col(rng.uniform(4.0, 15.0, n))
        psi = psi + amp * torch.exp(-((x[None, :] - x0) / s) ** 2) * torch.exp(1j * p0 * x[None, :]) / torch.sqrt(s)
    return psi / torch.sqrt((psi.abs() ** 2).sum(1, keepdim=True) * dx)


# ------------------------------------------------------------------------------------------ prepare

def prepare(case, seed):
    rng = _case_seed(seed)
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("propagate", "uneven"):
        N, dx, nt = _geometry(case)
        st["E"], offs = _pulse_rows(rng, nt, case["dt"])
        b = tdse.Batch(N, dx, SOFT, nt, case["dt"], row_offsets=offs, absorber=MASK, precision=_precision(case),
                       scheme=_scheme(case))
        b.ground_state(**GS)
        st.update(b=b, psi0=b.save_state(), d=torch.zeros_like(st["E"]), a=torch.zeros_like(st["E"]))
    elif kind == "adjoint":
        nt = np.full(case["n"], case["steps"], dtype=np.int64)
        E, offs = _pulse_rows(rng, nt, case["dt"])
        b = tdse.Batch(np.full(case["n"], case["N"]), case["dx"], SOFT, nt, case["dt"], row_offsets=offs, absorber=MASK)
        b.ground_state(**GS)
        gd, ga = (torch.from_numpy(rng.standard_normal(E.numel())).to(_dev()) for _ in range(2))
        st.update(b=b, E=E.requires_grad_(True), gd=gd, ga=ga)
    elif kind == "ground":
        N, dx, a = _ground_classes(case, rng)
        b = tdse.Batch(N, dx, a, 1, 0.02, absorber=MASK, scheme=_scheme(case))
        st.update(b=b)
    elif kind == "resample":
        st["coarse"] = torch.from_numpy(_coarse(case, rng)).to(_dev())
        st["out"] = torch.zeros((case["rows"], case["n_fine"]), dtype=torch.float64, device=_dev())
    elif kind == "spectrum":
        offs = _row_offsets(case)
        st.update(offs=offs, a=_a_rows(rng, offs, 0.02))
    elif kind == "far":
        n = case["n_r"] * case["n_z"]
        offs = np.arange(n + 1, dtype=np.int64) * case["L"]
        st.update(offs=offs, a=_a_rows(rng, offs, 0.02), g=_far_grids(case),
                  dens=torch.from_numpy(rng.uniform(0.5, 1.0, n)).to(_dev()))
    elif kind == "energy":
        n, N = case["n"], case["N"]
        b = tdse.Batch(np.full(n, N), case["dx"], SOFT, 1, case["dt"], absorber=MASK, precision=_precision(case),
                       scheme=_scheme(case))
        b.ground_state(**GS)
        psi = _packets(rng, n, N, case["dx"])
        for i in range(n):
            b.set_psi(i, psi[i])
        st.update(b=b, grid=np.linspace(-0.7, 2.5, case["n_E"]))
    else:
        raise ValueError(kind)
    return st


def _ground_classes(case, rng):
    g = case["grids"]
    N = np.array([max(300, case["N"] // (1 << (i % 4))) for i in range(g)])
    return N, np.array([0.15 if i % 2 else 0.2 for i in range(g)]), rng.uniform(1.0, 1.4, g)


def _row_offsets(case):
    rng = np.random.default_rng(3)
    lens = np.full(case["rows"], case["L"], dtype=np.int64)
    if case.get("ragged"):
        lens = rng.integers(max(2, case["L"] // 2), case["L"] + 1, case["rows"])
        lens[0] = case["L"]
    return np.concatenate([[0], np.cumsum(lens)])


def _coarse(case, rng):
    """Coarse 800 nm fields with a third harmonic and a little broadband noise, zero towards the window's end."""
    M, R = case["M"], case["rows"]
    t = np.arange(M) * case["dt_c"]
    w = inputs.omega_from_wavelength_nm(800.0)
    env = np.sin(math.pi * np.minimum(t / (0.9 * M * case["dt_c"]), 1.0)) ** 2
    f = np.cos(w * t[None, :] + rng.uniform(0, 6.28, R)[:, None]) + 0.05 * np.cos(3 * w * t[None, :] + rng.uniform(0, 6.28, R)[:, None])
    f = f + 1e-3 * rng.standard_normal((R, M))
    return np.ascontiguousarray(0.06 * rng.uniform(0.5, 1.0, R)[:, None] * env[None, :] * f)


# --------------------------------------------------------------------------------------------- run

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind in ("propagate", "uneven"):
        b = st["b"]
        b.load_state(st["psi0"])
        b.propagate(st["E"], st["d"], st["a"])
        if case["n"] == 1:
            psi = b.get_psi(0)
        else:
            psi = b.save_state()
            if case["precision"] == "mixed":
                psi = psi.view(torch.float32)
        return {"d": st["d"], "a": st["a"], "psi": psi}
    if kind == "adjoint":
        d, a = tdse.tdse_propagate_autograd(st["E"], st["b"], case["ckpt"])
        (gE,) = torch.autograd.grad((d, a), st["E"], (st["gd"], st["ga"]))
        return {"d": d.detach(), "a": a.detach(), "gE": gE}
    if kind == "ground":
        e, it = st["b"].ground_state(dtau=GS["dtau"], max_iter=case["iters"], tol=0.0)
        return {"energy": e, "iterations": it, "psi": torch.cat([st["b"].get_psi(i) for i in range(case["grids"])])}
    if kind == "resample":
        return tdse.resample_field(st["coarse"], case["dt_c"], case["dt_f"], case["n_fine"], out=st["out"])
    if kind == "spectrum":
        return tdse.spectrum(st["a"], st["offs"], 0.02, case["k0"], case["k1"])
    if kind == "far":
        g = st["g"]
        S = tdse.dipole_spectrum(st["a"], st["offs"], 0.02, g["om"], weight=st["dens"])
        E = tdse.hankel(S.view(case["n_r"], case["n_z"], case["n_w"]), g["rho"], g["z"], g["k"], g["z_obs"], g["ro"])
        return {"S": S, "E": E}
    P = st["b"].energy_distribution(st["grid"], case["eps"])
    return {"P": P, "populations": st["b"].populations(2.0)}


def work(case):
    """Inputs read once, outputs written once; operations of the methods as the paper states them:
    48 per point and step of a Crank-Nicolson step (its tridiagonal solve, update and observables),
    about 60 for the Numerov scheme's three substeps, a sweep back and one recomputation for the
    gradient, 22 per point of a resolvent solve, 8 per term of a Bessel-weighted sum besides the
    Bessel value itself; transforms by the fast algorithm (5 L log2 L)."""
    kind = case["kind"]
    if kind in ("propagate", "uneven"):
        N, _, nt = _geometry(case)
        pts, cx = float((N * nt).sum()), 8 if case["precision"] == "mixed" else 16
        return dict(bytes=24.0 * float((nt + 1).sum()) + 2.0 * cx * float(N.sum()),
                    flops=pts * (60.0 if case.get("scheme") == "numerov" else 48.0))
    if kind == "adjoint":
        pts = float(case["n"]) * case["N"] * case["steps"]
        return dict(bytes=48.0 * case["n"] * (case["steps"] + 1) + 16.0 * case["n"] * case["N"], flops=3.0 * 48.0 * pts)
    if kind == "ground":
        N, _, _ = _ground_classes(case, _case_seed(0))
        return dict(bytes=16.0 * float(N.sum()), flops=20.0 * float(N.sum()) * case["iters"])
    if kind == "resample":
        R, M, n = case["rows"], case["M"], case["n_fine"]
        return dict(bytes=8.0 * R * (M + n), flops=R * (5.0 * M * math.log2(M) + 5.0 * n * math.log2(n)))
    if kind == "spectrum":
        L, nb = case["L"], case["k1"] - case["k0"]
        return dict(bytes=8.0 * case["rows"] * (L + nb), flops=case["rows"] * min(4.0 * L * nb, 2.5 * L * math.log2(L)))
    if kind == "far":
        n, w = case["n_r"] * case["n_z"], case["n_w"]
        return dict(bytes=8.0 * n * case["L"] + 32.0 * n * w + 16.0 * w * case["n_obs"],
                    flops=n * min(4.0 * case["L"] * w, 2.5 * case["L"] * math.log2(case["L"])) + 8.0 * n * w * case["n_obs"])
    cx = 8 if case["precision"] == "mixed" else 16
    return dict(bytes=cx * float(case["n"]) * case["N"] + 8.0 * case["n"] * (case["n_E"] + 2),
                flops=22.0 * case["n"] * case["N"] * case["n_E"])


# -------------------------------------------------------------------------------------------- exact

def _shift(v, s):
    """v[..., j - s], zero outside the grid (s > 0: the neighbour on the left)."""
    out = torch.zeros_like(v)
    if abs(s) >= v.shape[-1]:
        return out
    if s > 0:
        out[..., s:] = v[..., :-s]
    else:
        out[..., :s] = v[..., -s:]
    return out


class _Tridiagonal:
    """Parallel cyclic reduction of diagonally dominant tridiagonal systems along the last axis: the
    matrix (lo, di, up) is reduced once, solve() applies it to right-hand sides."""

    def __init__(self, lo, di, up):
        self.levels = []
        s, N = 1, di.shape[-1]
        while s < N and max(float(lo.abs().max()), float(up.abs().max())) > 1e-25:
            r = 1.0 / di
            al, ga = -lo * _shift(r, s), -up * _shift(r, -s)
            di = di + al * _shift(up, s) + ga * _shift(lo, -s)
            lo, up = al * _shift(lo, s), ga * _shift(up, -s)
            self.levels.append((s, al, ga))
            s *= 2
        self.inv = 1.0 / di

    def solve(self, d):
        for s, al, ga in self.levels:
            d = d + al * _shift(d, s) + ga * _shift(d, -s)
        return d * self.inv


def _cn_solve(beta, di, d):
    """(tridiag(-i beta, di, -i beta))^{-1} d; symmetric, so one off-diagonal is carried."""
    N = di.shape[-1]
    lo = torch.full_like(di, -1j * beta)
    lo[..., 0] = 0
    s = 1
    while s < N and float(lo.abs().max()) > 1e-25:
        r = 1.0 / di
        up = _shift(lo, -s)
        al, ga = lo * _shift(r, s), up * _shift(r, -s)
        d = d - al * _shift(d, s) - ga * _shift(d, -s)
        di = di - al * lo - ga * up
        lo = -al * _shift(lo, s)
        s *= 2
    return d / di


class _Grid:
    """x, V, dV/dx and the mask of one grid, and the field-free matrices of both schemes."""

    def __init__(self, N, dx, soft, scheme):
        dev = _dev()
        self.N, self.dx, self.scheme = N, dx, scheme
        self.x = (torch.arange(N, dtype=torch.float64, device=dev) - 0.5 * (N - 1)) * dx
        r2 = self.x * self.x + soft * soft
        self.V = -1.0 / torch.sqrt(r2)
        self.dV = self.x / (r2 * torch.sqrt(r2))
        ax = self.x.abs() - (0.5 * N * dx - MASK[0])
        self.m = torch.where(ax > 0, torch.clamp(torch.cos(0.5 * math.pi * ax / MASK[0]), min=0.0) ** MASK[1],
                             torch.ones_like(ax))

    def mat(self, c):
        """Rows (lo, di, up) of M + c K (M = 1 and the three-point H0, or the Numerov pencil)."""
        i2 = 1.0 / (self.dx * self.dx)
        if self.scheme == "numerov":
            lo = 1.0 / 12.0 + c * (-0.5 * i2 + _shift(self.V, 1) / 12.0)
            up = 1.0 / 12.0 + c * (-0.5 * i2 + _shift(self.V, -1) / 12.0)
            di = 10.0 / 12.0 + c * (i2 + (10.0 / 12.0) * self.V)
        else:
            lo = c * (-0.5 * i2) * torch.ones_like(self.V)
            up, di = lo.clone(), 1.0 + c * (i2 + self.V)
        lo[0] = 0
        up[-1] = 0
        return lo, di, up

    def M(self, v):
        if self.scheme != "numerov":
            return v
        return (10.0 * v + _shift(v, 1) + _shift(v, -1)) / 12.0

    def ground(self, iters):
        T = _Tridiagonal(*self.mat(0.5 * GS["dtau"]))
        psi = torch.exp(-self.x * self.x)
        for _ in range(iters):
            psi = 2.0 * T.solve(self.M(psi)) - psi
            psi = psi / torch.sqrt((psi * psi).sum() * self.dx)
        psi = psi if float(psi[self.N // 2]) >= 0 else -psi
        y = -0.5 * (_shift(psi, 1) - 2.0 * psi + _shift(psi, -1)) / (self.dx * self.dx)
        if self.scheme == "numerov":
            one = torch.ones_like(psi)
            lo, up = one / 12.0, one / 12.0
            lo[0] = 0
            up[-1] = 0
            y = _Tridiagonal(lo, one * (10.0 / 12.0), up).solve(y)
        return psi, float((psi * (y + self.V * psi)).sum() * self.dx)


def _propagate_exact(g, E, dt, keep=False):
    """Rows E (n x (nt + 1)) on one grid: d, a, the final states, and with `keep` the pre-mask states."""
    n, nt = E.shape[0], E.shape[1] - 1
    psi0, _ = g.ground(GS["max_iter"])
    psi = psi0.to(torch.complex128)[None, :].repeat(n, 1)
    d, a = torch.zeros_like(E), torch.zeros_like(E)
    h, i2 = 0.5 * dt, 1.0 / (g.dx * g.dx)
    T = None
    if g.scheme == "numerov":
        T = _Tridiagonal(*(v for v in g.mat(torch.tensor(1j * h, dtype=torch.complex128, device=_dev()))))
    states = [psi]

    def obs(k):
        rho = psi.real ** 2 + psi.imag ** 2
        d[:, k] = rho @ g.x * g.dx
        a[:, k] = (rho @ g.dV + E[:, k] * rho.sum(1)) * g.dx

    obs(0)
    for k in range(nt):
        if T is not None:
            t = (2.0 * T.solve(g.M(psi)) - psi) * torch.exp(-1j * dt * E[:, k][:, None] * g.x[None, :])
        else:
            Eb = 0.5 * (E[:, k] + E[:, k + 1])
            di = torch.complex(torch.ones_like(g.x)[None, :].expand(n, -1), h * (i2 + g.V[None, :] + g.x[None, :] * Eb[:, None]))
            t = 2.0 * _cn_solve(0.25 * dt * i2, di, psi) - psi
        psi = t * g.m[None, :]
        if keep:
            states += [t, psi]
        obs(k + 1)
    return d, a, psi, states


def _adjoint_exact(g, E, dt, gd, ga):
    d, a, psi, states = _propagate_exact(g, E, dt, keep=True)
    nt = E.shape[1] - 1
    h, i2 = 0.5 * dt, 1.0 / (g.dx * g.dx)
    gE = torch.zeros_like(E)

    def local(k, psi):
        rho = psi.real ** 2 + psi.imag ** 2
        gE[:, k] += ga[:, k] * g.dx * rho.sum(1)
        return 2.0 * g.dx * (gd[:, k][:, None] * g.x + ga[:, k][:, None] * (g.dV + E[:, k][:, None])) * psi

    lam = local(nt, psi)
    for k in range(nt - 1, -1, -1):
        prev, tilde = states[2 * k], states[2 * k + 1]
        v = lam * g.m[None, :]
        Eb = 0.5 * (E[:, k] + E[:, k + 1])
        di = torch.complex(torch.ones_like(prev.real), h * (i2 + g.V[None, :] + g.x[None, :] * Eb[:, None]))
        mu = _cn_solve(0.25 * dt * i2, di, v.conj().resolve_conj()).conj().resolve_conj()
        gb = h * ((mu.conj() * (prev + tilde)).imag @ g.x)
        gE[:, k] += 0.5 * gb
        gE[:, k + 1] += 0.5 * gb
        lam = 2.0 * mu - v + local(k, prev)
    return d, a, gE


def _bessel_j0(x):
    """J0 as the mean of cos(x sin t) over a quarter period, by the midpoint rule: its error is 2 J_4m(x)."""
    m = int(0.25 * float(x.max())) + 24
    out = torch.zeros_like(x)
    for j in range(m):
        out += torch.cos(x * math.sin(0.5 * math.pi * (j + 0.5) / m))
    return out / m


def _phase_matrix(M, dt_c, dt_f, n0, n1, K):
    """cos and sin of 2 pi k n dt_f / (M dt_c) for k = 0..K and n0 <= n < n1: the phase in turns as a
    64-bit binary fraction, exact to k 2^-64."""
    r = Fraction(dt_f) / Fraction(M * dt_c)
    p, q = r.numerator, r.denominator
    U = np.array([((n * p % q) << 64) // q for n in range(n0, n1)], dtype=np.uint64).view(np.int64)
    k = torch.arange(K + 1, dtype=torch.int64, device=_dev())
    ph = (k[:, None] * torch.from_numpy(U).to(_dev())[None, :]).double() * (2.0 * math.pi / 2.0 ** 64)
    return torch.cos(ph), torch.sin(ph)


def exact(case, seed):
    rng = _case_seed(seed)
    kind = case["kind"]
    if kind in ("propagate", "uneven"):
        N, dx, nt = _geometry(case)
        E, offs = _pulse_rows(rng, nt, case["dt"])
        d, a, psi = torch.zeros_like(E), torch.zeros_like(E), None
        L = int(nt.max())                                # shorter rows are padded to the longest
        for Nc, dxc in sorted(set(zip(N.tolist(), dx.tolist()))):
            idx = np.nonzero((N == Nc) & (dx == dxc))[0]
            g = _Grid(int(Nc), float(dxc), SOFT, case.get("scheme", "full_cn"))
            for i0 in range(0, len(idx), 2048):
                part = idx[i0: i0 + 2048]
                rows = torch.zeros((len(part), L + 1), dtype=torch.float64, device=_dev())
                for r, i in enumerate(part):
                    rows[r, : nt[i] + 1] = E[offs[i]: offs[i + 1]]
                dd, aa, ps, _ = _propagate_exact(g, rows, case["dt"])
                for r, i in enumerate(part):
                    d[offs[i]: offs[i + 1]] = dd[r, : nt[i] + 1]
                    a[offs[i]: offs[i + 1]] = aa[r, : nt[i] + 1]
                psi = ps
        return {"d": d, "a": a, "psi": psi[0] if case["n"] == 1 else None}
    if kind == "adjoint":
        nt = np.full(case["n"], case["steps"], dtype=np.int64)
        E, _ = _pulse_rows(rng, nt, case["dt"])
        gd, ga = (torch.from_numpy(rng.standard_normal(E.numel())).to(_dev()) for _ in range(2))
        g = _Grid(case["N"], case["dx"], SOFT, "full_cn")
        shape = (case["n"], case["steps"] + 1)
        d, a, gE = _adjoint_exact(g, E.view(shape), case["dt"], gd.view(shape), ga.view(shape))
        return {"d": d.reshape(-1), "a": a.reshape(-1), "gE": gE.reshape(-1)}
    if kind == "ground":
        N, dx, a = _ground_classes(case, rng)
        out = [_Grid(int(N[i]), float(dx[i]), float(a[i]), case["scheme"]).ground(case["iters"]) for i in range(case["grids"])]
        return {"energy": np.array([e for _, e in out]), "iterations": None,
                "psi": torch.cat([p for p, _ in out]).to(torch.complex128)}
    if kind == "resample":
        c = torch.from_numpy(_coarse(case, rng)).to(_dev())
        M, n = case["M"], case["n_fine"]
        K = M // 2
        F = torch.fft.rfft(c, dim=1) / M
        F[:, 1:] *= 2.0
        if M % 2 == 0:
            F[:, K] *= 0.5
        out = torch.empty((case["rows"], n), dtype=torch.float64, device=_dev())
        for n0 in range(0, n, 8192):
            n1 = min(n, n0 + 8192)
            co, si = _phase_matrix(M, case["dt_c"], case["dt_f"], n0, n1, K)
            out[:, n0:n1] = F.real @ co - F.imag @ si
        return out
    if kind == "spectrum":
        offs = _row_offsets(case)
        a = _a_rows(rng, offs, 0.02)
        k = torch.arange(case["k0"], case["k1"], device=_dev())
        out = []
        for r in range(case["rows"]):
            F = torch.fft.fft(a[offs[r]: offs[r + 1]].to(torch.complex128))
            out.append(0.02 ** 2 * F[k % F.numel()].abs() ** 2)
        return torch.stack(out)
    if kind == "far":
        n, L = case["n_r"] * case["n_z"], case["L"]
        a = _a_rows(rng, np.arange(n + 1, dtype=np.int64) * L, 0.02).view(n, L)
        dens = torch.from_numpy(rng.uniform(0.5, 1.0, n)).to(_dev())
        g = {k: torch.as_tensor(v, dtype=torch.float64, device=_dev()) for k, v in _far_grids(case).items()}
        t = torch.arange(L, dtype=torch.float64, device=_dev()) * 0.02
        S = torch.empty((n, case["n_w"]), dtype=torch.complex128, device=_dev())
        for w0 in range(0, case["n_w"], 64):
            ph = t[:, None] * g["om"][None, w0: w0 + 64]
            S[:, w0: w0 + 64] = torch.complex(a @ torch.cos(ph), a @ torch.sin(ph))
        S *= dens[:, None] * 0.02 / math.sqrt(2.0 * math.pi)
        S3 = S.view(case["n_r"], case["n_z"], case["n_w"])

        def trap(x):
            if x.numel() == 1:
                return torch.ones_like(x)
            w = torch.zeros_like(x)
            w[1:] += 0.5 * (x[1:] - x[:-1])
            w[:-1] += 0.5 * (x[1:] - x[:-1])
            return w

        wr, wz = trap(g["rho"]), trap(g["z"])
        E = torch.zeros((case["n_w"], case["n_obs"]), dtype=torch.complex128, device=_dev())
        for i in range(case["n_z"]):
            D = g["z_obs"] - g["z"][i]
            k = g["k"][:, None]
            src = (S3[:, i, :].T * wr[None, :] * g["rho"][None, :] * wz[i] / D
                   * torch.exp(1j * k * (g["rho"][None, :] ** 2 / (2.0 * D) - g["z"][i])))
            J = _bessel_j0((k * g["ro"][None, :] / D)[:, :, None] * g["rho"][None, None, :])
            E += torch.exp(1j * k * g["ro"][None, :] ** 2 / (2.0 * D)) * torch.einsum("woj,wj->wo", J.to(torch.complex128), src)
        E *= -MU0 / (4.0 * math.pi) * torch.exp(1j * g["k"] * g["z_obs"])[:, None]
        return {"S": S, "E": E}
    return _energy_exact(case, rng)


def _energy_exact(case, rng):
    """Resolvent solves by elimination from the left, all states and energies side by side."""
    n, N, dx, eps = case["n"], case["N"], case["dx"], case["eps"]
    psi = _packets(rng, n, N, dx)
    if case["precision"] == "mixed":
        psi = psi.to(torch.complex64).to(torch.complex128)
    g = _Grid(N, dx, SOFT, case["scheme"])
    Ek = torch.from_numpy(np.linspace(-0.7, 2.5, case["n_E"])).to(_dev())
    z = Ek.to(torch.complex128) - 1j * eps
    mlo, mdi, mup = (v.real if v.is_complex() else v for v in g.mat(0.0))
    if case["scheme"] != "numerov":
        mlo, mup = torch.zeros_like(mlo), torch.zeros_like(mup)
    klo, kdi, kup = (p - m for p, m in zip(g.mat(1.0), (mlo, mdi, mup)))
    rhs = g.M(psi).T.contiguous()                       # N x n
    P = torch.empty((n, case["n_E"]), dtype=torch.float64, device=_dev())
    for e0 in range(0, case["n_E"], 32):
        ze = z[e0: e0 + 32]
        fwd = torch.empty((N, n, ze.numel()), dtype=torch.complex128, device=_dev())
        cp = torch.empty((N, ze.numel()), dtype=torch.complex128, device=_dev())
        prev, cprev = None, torch.zeros_like(ze)
        for j in range(N):
            lo = ze * mlo[j] - klo[j]
            inv = 1.0 / (ze * mdi[j] - kdi[j] - lo * cprev)
            cprev = (ze * mup[j] - kup[j]) * inv
            cp[j] = cprev
            r = rhs[j][:, None]
            prev = r * inv if prev is None else (r - lo * prev) * inv
            fwd[j] = prev
        y, s = fwd[N - 1], torch.zeros((n, ze.numel()), dtype=torch.float64, device=_dev())
        for j in range(N - 1, -1, -1):
            if j < N - 1:
                y = fwd[j] - cp[j] * y
            s += y.real ** 2 + y.imag ** 2
        P[:, e0: e0 + 32] = s * dx * eps / math.pi
        del fwd
    psi0, _ = g.ground(GS["max_iter"])
    ov = (psi @ psi0.to(torch.complex128)) * dx
    core = (psi.abs() ** 2)[:, g.x.abs() < 2.0].sum(1) * dx
    return {"P": P, "populations": torch.stack([ov.abs() ** 2, core], dim=1)}


if __name__ == "__main__":
    for c in listed() + [draw(random.Random(i)) for i in range(12)]:
        print(c, work(c))
