"""What a program that uses this library has it do, as cases to time and to compare.

A case is one call sequence through the public entry points (paper_2001_01609_gb300.rbc) on
states that live on the GPU:

  step       rbc_step_batch(_ra): B states of one grid by nsteps steps (the fine batches, the
             serial coarse sweeps, the serving engine's mixed batches)
  sampled    rbc_step_batch_sampled: the same with the averages of Sec. 2.2 along the run
  parareal   a whole Parareal run from native-grid values to native-grid values
  tick       what a serving tick does between propagations: restriction, correction (Eq. 20)
             and the defect norms of B slices

Initial states are convection rolls with thermal boundary layers and the paper's small grid
noise (all modes filled), formed here from the seed; time steps follow the stability rule of
the serving engine, so repeated passes go on along the trajectory.
"""
import math

import numpy as np
import torch

from paper_2001_01609_gb300 import rbc

LX, PR = 2.0, 1.0
STAGES = {0: 4, 1: 2, 2: 1}


# --------------------------------------------------------------------------
# The cases.
# --------------------------------------------------------------------------
def _step(name, Nx, Nz, Ra, dt, B, nsteps, precision, scheme=0, bc=0, uneven=False):
    return dict(name=name, kind="step", Nx=Nx, Nz=Nz, Ra=Ra, dt=dt, B=B, nsteps=nsteps, precision=precision,
                scheme=scheme, bc=bc, uneven=uneven)


def listed():
    return [
        # one slice of the serial coarse sweep of the 32-slice Ra 1e6 workload: latency counts
        _step("coarse_128x32_fp64", 128, 32, 1e6, 1.5625e-5, 1, 40, 0),
        # the same sweep in mixed precision with the lower-order coarse scheme of Sec. 3.6
        _step("coarse_128x32_mixed_rk222", 128, 32, 1e6, 1.5625e-5, 1, 40, 1, scheme=1),
        # the serial all-FP64 fine propagator, the baseline of every time-to-tolerance run
        _step("serial_256x64_fp64", 256, 64, 1e6, 1.25e-5, 1, 10, 0),
        # the fine sweep of all 32 slices in one batch, FP64
        _step("fine_256x64_fp64_b32", 256, 64, 1e6, 1.25e-5, 32, 2, 0),
        # a fine group of the overlapped Parareal schedule, mixed precision (TF32 operands)
        _step("group_256x64_mixed_b8", 256, 64, 1e6, 1.25e-5, 8, 8, 1),
        # the 64-slice Ra 1e7 workload, BF16 operands
        _step("fine_512x128_bf16_b64", 512, 128, 1e7, 7.8125e-7, 64, 2, 2),
        # the Ra 1e8 workload's grid, a quarter of its 128 slices (the largest case)
        _step("fine_1024x256_mixed_b32", 1024, 256, 1e8, 7.8125e-8, 32, 2, 1),
        # a serving batch: requests of different Ra at different points of their slices, fixed flux
        _step("serving_64x32_fp64_b23", 64, 32, 1e5, 1e-4, 23, 9, 0, bc=1, uneven=True),
        # an FP64 request on a fine grid, alone in its class
        _step("serving_512x128_fp64_b3", 512, 128, 1e6, 7.8125e-7, 3, 2, 0),
        # the plain Ra 1e4 workload end to end: grid values in, Parareal, grid values out
        dict(name="parareal_64x32_fp64", kind="parareal", Nx=64, Nz=32, Nxc=32, Nzc=16, Ra=1e4, dt=1e-3, nf=20,
             nc=5, slices=4, iters=2, precision=0, scheme=0),
        # statistics along a fine sweep (Re, Nu, energy balance, T_rms), sampled every few steps
        dict(name="sampled_256x64_fp64_b8", kind="sampled", Nx=256, Nz=64, Ra=1e6, dt=1.25e-5, B=8, nsteps=4, every=2,
             precision=0, scheme=0, bc=0),
        # the serving engine between two propagations of a class
        dict(name="tick_256x64_b16", kind="tick", Nx=256, Nz=64, Nxc=128, Nzc=32, Ra=1e6, dt=1.25e-5, B=16),
    ]


def _dt(Nz, Ra):
    """Largest 1e-3 2^-j under the stability rule 20 / (Nz^2 sqrt(Ra))."""
    lim, dt = 20.0 / (Nz * Nz * math.sqrt(Ra)), 1e-3
    while dt > lim:
        dt *= 0.5
    return dt


# nothing drawn costs more than the largest listed case: DOF-steps, FP64 transforms weighed by four
_COST = 1024 * 256 * 32 * 2


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    Nx = 1 << rng.randint(4, 10)
    Nz = 2 * max(5, min(128, int(round(Nx / 8 * math.exp(rng.uniform(-0.7, 0.7))))))
    Ra = float("%.3g" % math.exp(rng.uniform(math.log(1e4), math.log(1e4 * max(2.0, (Nz / 16.0) ** 3)))))
    kind = rng.choice(["step"] * 6 + ["sampled", "parareal", "tick"])
    precision = rng.choice([0, 1, 2])
    dt = _dt(Nz, Ra)
    room = _COST / (Nx * Nz * (4 if precision == 0 else 1) * (2 if Nz > 64 else 1))
    B = max(1, min(logint(1, 128), int(room / 2)))
    nsteps = max(1, min(logint(1, 40), int(room / B)))
    if kind == "step":
        return dict(kind=kind, Nx=Nx, Nz=Nz, Ra=Ra, dt=dt, B=B, nsteps=nsteps, precision=precision,
                    scheme=rng.choice([0, 0, 1, 2]), bc=rng.choice([0, 0, 1]) if Nz <= 64 else 0,
                    uneven=rng.random() < 0.3)
    B = min(B, 24)
    if kind == "sampled":
        return dict(kind=kind, Nx=Nx, Nz=Nz, Ra=Ra, dt=dt, B=B, nsteps=min(nsteps, 8), every=rng.randint(1, 4),
                    precision=precision, scheme=rng.choice([0, 1]), bc=0)
    Nxc, Nzc = Nx // 2, max(8, 2 * ((Nz + 2) // 4))
    if kind == "parareal":
        nc = rng.randint(2, 6)
        slices = max(2, min(rng.randint(2, 8), int(room / (8 * nc))))
        return dict(kind=kind, Nx=Nx, Nz=Nz, Nxc=Nxc, Nzc=Nzc, Ra=Ra, dt=dt, nf=2 * nc, nc=nc, slices=slices,
                    iters=rng.randint(1, 2), precision=precision, scheme=rng.choice([0, 1]))
    return dict(kind=kind, Nx=Nx, Nz=Nz, Nxc=Nxc, Nzc=Nzc, Ra=Ra, dt=dt, B=B)


# --------------------------------------------------------------------------
# Inputs.
# --------------------------------------------------------------------------
def _interp(Nz):
    """Values at s_j = -cos(pi j / (Nz - 1)) -> Chebyshev coefficients (FP64, GPU)."""
    th = np.pi * (Nz - 1 - np.arange(Nz)) / (Nz - 1)
    c = np.ones(Nz)
    c[0] = c[-1] = 2.0
    W = 2.0 / (Nz - 1) * np.cos(np.outer(np.arange(Nz), th)) / np.outer(c, c)
    return torch.from_numpy(W).cuda()


def _states(case, B, seed):
    """B states (B, 2, Nz, Nx/2, 2): rolls, boundary layers and noise, made from the seed."""
    Nx, Nz, Ra, nm = case["Nx"], case["Nz"], case["Ra"], case["Nx"] // 2
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) % (1 << 62))

    def normal(*shape):
        return torch.randn(shape, generator=g, dtype=torch.float64, device="cuda")

    z = torch.from_numpy(-0.5 * np.cos(np.pi * np.arange(Nz) / (Nz - 1))).cuda()
    env = (z + 0.5) * (0.5 - z)
    k = 2.0 * math.pi / LX * torch.arange(nm, dtype=torch.float64, device="cuda")
    flux = case.get("bc", 0) == 1
    K, L = min(6, nm - 1), 4
    amp = torch.zeros(nm, dtype=torch.float64, device="cuda")
    amp[1:K + 1] = 0.5 ** torch.arange(K, dtype=torch.float64, device="cuda")
    zl = torch.stack([torch.cos(l * torch.acos((2.0 * z).clamp(-1, 1))) * 0.5 ** l for l in range(L)], 1)
    X = torch.zeros((B, 2, Nz, nm, 2), dtype=torch.float64, device="cuda")
    W = _interp(Nz)
    # temperature: conduction, a mean boundary-layer shape, rolls, grid noise (amplitude 1e-3)
    te = env * env if flux else env
    T = (0.6 * amp * te[:, None]).expand(B, Nz, nm).unsqueeze(-1) * torch.einsum("zl,blmc->bzmc", zl, normal(B, L, nm, 2))
    T = T + 1e-3 / math.sqrt(2.0 * Nx) * te[None, :, None, None] * normal(B, Nz, nm, 2)
    T[:, :, 0, 1] = 0.0
    T[:, :, 0, 0] += 0.5 - z - 0.3 * te * z
    # streamfunction of free-fall size (psi = psi' = 0 at the walls), mean flow a tenth of it
    e2 = 16.0 * env * env
    P = 0.01 * math.sqrt(Ra * PR) * (amp * e2[:, None]).expand(B, Nz, nm).unsqueeze(-1) \
        * torch.einsum("zl,blmc->bzmc", zl, normal(B, L, nm, 2))
    P = P + 1e-3 / math.sqrt(2.0 * Nx) * e2[None, :, None, None] * normal(B, Nz, nm, 2)
    P[:, :, 0, :] = 0.0
    P[:, :, 0, 0] = 0.01 * math.sqrt(Ra * PR) * 4.0 * env * normal(B, 1)
    X[:, 0] = torch.einsum("nz,bzmc->bnmc", W, T)
    X[:, 1] = torch.einsum("nz,bzmc->bnmc", W, P)
    return X


def _uneven(case, seed):
    """Step counts and Rayleigh numbers per state: requests at different points of their slices."""
    r = np.random.default_rng(int(seed) + 99)
    ns = r.integers(0, case["nsteps"] + 1, case["B"])
    ns[0] = case["nsteps"]
    return [int(v) for v in ns], [float(v) for v in case["Ra"] * np.exp(r.uniform(-2.0, 0.0, case["B"]))]


def _grid(case, seed):
    """Native-grid T, u, w of one state (Nz, Nx), host arrays."""
    Nx, Nz, nm = case["Nx"], case["Nz"], case["Nx"] // 2
    X = _states(case, 1, seed)[0].cpu().numpy()
    th = np.pi * (Nz - 1 - np.arange(Nz)) / (Nz - 1)
    V = np.cos(np.outer(th, np.arange(Nz)))
    D = np.zeros((Nz, Nz))
    for n in range(1, Nz):
        for q in range(n - 1, -1, -2):
            D[q, n] = 2.0 * n * (0.5 if q == 0 else 1.0)
    Tm = V @ (X[0, :, :, 0] + 1j * X[0, :, :, 1])
    P = X[1, :, :, 0] + 1j * X[1, :, :, 1]
    um = 2.0 * (V @ D @ P)
    um[:, 0] = V @ P[:, 0]
    wm = -1j * (2.0 * np.pi / LX * np.arange(nm)) * (V @ P)
    wm[:, 0] = 0.0

    def values(c):
        full = np.zeros((Nz, nm + 1), dtype=complex)
        full[:, :nm] = c
        return np.ascontiguousarray(np.fft.irfft(full, n=Nx, axis=1) * Nx)

    return values(Tm), values(um), values(wm)


def _handle(case, coarse=False):
    if coarse:
        return rbc.Propagator(case["Ra"], PR, LX, case["Nxc"], case["Nzc"], case["dt"] * case.get("nf", 2) / case.get("nc", 1),
                              case.get("precision", 0), scheme=case.get("scheme", 0))
    # in a Parareal run the lower-order scheme is the coarse propagator's only
    scheme = 0 if case["kind"] == "parareal" else case.get("scheme", 0)
    return rbc.Propagator(case["Ra"], PR, LX, case["Nx"], case["Nz"], case["dt"], case.get("precision", 0),
                          bc=case.get("bc", 0), scheme=scheme)


def prepare(case, seed):
    s = dict(case=case, F=_handle(case))
    kind = case["kind"]
    if kind in ("step", "sampled"):
        s["X"] = _states(case, case["B"], seed)
        s["nu"] = torch.zeros(case["B"], dtype=torch.float64, device="cuda")
        s["ns"], s["ra"] = _uneven(case, seed) if case.get("uneven") else (case["nsteps"], None)
        s["F"].reserve(case["B"])
    elif kind == "parareal":
        s["G"] = _handle(case, coarse=True)
        s["grid"] = _grid(case, seed)
        s["U0"] = s["F"].new_states(1)
        s["U"] = s["F"].new_states(case["slices"] + 1)
        s["P"] = rbc.Parareal(s["F"], s["G"], 0.0, case["slices"] * case["nf"] * case["dt"], case["slices"])
    else:
        s["G"] = _handle(case, coarse=True)
        B = case["B"]
        X = _states(case, 2 * B, seed)
        s["Ff"], s["old"] = X[:B].clone(), X[B:].clone()
        small = _states(dict(case, Nx=case["Nxc"], Nz=case["Nzc"]), 2 * B, int(seed) + 1)
        s["Gnew"], s["Gold"] = small[:B].clone(), small[B:].clone()
        s["U"] = torch.empty_like(s["Ff"])
        s["C"] = torch.empty_like(s["Gnew"])
        s["d2"] = torch.empty(B, dtype=torch.float64, device="cuda")
        s["u2"] = torch.empty(B, dtype=torch.float64, device="cuda")
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "step":
        s["F"].step_batch(s["X"], s["ns"], s["nu"], ra=s["ra"])
        return s["X"], s["nu"]
    if kind == "sampled":
        stat = s["F"].step_batch_sampled(s["X"], case["nsteps"], case["every"], nu=s["nu"])
        return s["X"], s["nu"], stat
    if kind == "parareal":
        T, u, w = s["grid"]
        s["F"].set_state(s["U0"][0], T, u, w)
        _, k, defects, nus = s["P"].iterate(s["U0"][0], s["U"], case["iters"])
        T1, u1, w1 = s["F"].get_state(s["U"][-1])
        return s["U"], defects, nus, T1, u1, w1, k
    rbc.parareal_correct(s["F"], s["G"], s["Ff"], s["Gnew"], s["Gold"], s["U"])
    rbc.restrict(s["F"], s["G"], s["U"], s["C"])
    rbc.l2_diff(s["F"], s["U"], s["old"], s["d2"])
    rbc.l2_diff(s["F"], s["U"], None, s["u2"])
    return s["U"], s["C"], s["d2"], s["u2"]


# --------------------------------------------------------------------------
# Work that a pass cannot do without.
# --------------------------------------------------------------------------
def _stage_work(Nx, Nz):
    """Bytes and flops of one implicit-explicit stage of one state: the state and the explicit
    terms that the stage sums carry on read once and written once; split-parity z transforms of
    six operators and two products, six complex FFTs per padded row, products, banded solves."""
    nm, Mx, Mz = Nx // 2, 3 * Nx // 2, 3 * Nz // 2
    S = 16.0 * Nx * Nz
    flops = 24.0 * (Mz / 2) * nm * Nz + Mz * (6 * 5.0 * Mx * math.log2(Mx) + 14.0 * Mx) + 8.0 * (Mz / 2) * nm * Nz \
        + 120.0 * nm * Nz
    return 4.0 * S, flops


def _run_work(Nx, Nz, scheme, steps):
    by, fl = _stage_work(Nx, Nz)
    return steps * STAGES[scheme] * by, steps * STAGES[scheme] * fl


def work(case):
    Nx, Nz, kind = case["Nx"], case["Nz"], case["kind"]
    S = 16.0 * Nx * Nz
    if kind in ("step", "sampled"):
        steps = case["B"] * case["nsteps"] * (0.5 if case.get("uneven") else 1.0)
        by, fl = _run_work(Nx, Nz, case["scheme"], steps)
        if kind == "sampled":
            n = case["B"] * (1 + -(-case["nsteps"] // case["every"]))
            by, fl = by + n * S, fl + n * 24.0 * (3 * Nz // 4) * (Nx // 2) * Nz
        return {"bytes": by, "flops": fl}
    if kind == "parareal":
        N, it = case["slices"], case["iters"]
        bf, ff = _run_work(Nx, Nz, 0, case["nf"] * sum(N - i for i in range(it)))
        bc, fc = _run_work(case["Nxc"], case["Nzc"], case["scheme"], case["nc"] * (N + sum(N - 1 - i for i in range(it))))
        return {"bytes": bf + bc + N * it * 4 * S, "flops": ff + fc}
    Sc = 16.0 * case["Nxc"] * case["Nzc"]
    return {"bytes": case["B"] * (3 * S + 3 * Sc), "flops": case["B"] * (2 * S / 8 + 2 * 2.0 * Nx * Nz * Nz / 2)}


# --------------------------------------------------------------------------
# Tolerances: about four times the largest relative difference seen between the library and
# exact() below, over the listed and several drawn cases: FP64 1.1e-12 (defects of a Parareal
# run; states 8e-14), FP32 products 2.2e-6 (Nu integrals; states 1.1e-6), norms 4e-16.
# --------------------------------------------------------------------------
def tolerance(case):
    if case["kind"] == "tick":
        return {"rel": 2e-15, "max": 8e-14}
    if case.get("precision", 0) == 0:
        return {"rel": 5e-12, "max": 2e-10}
    return {"rel": 1e-5, "max": 4e-4}


# --------------------------------------------------------------------------
# The same in plain torch, 64 bits.
# --------------------------------------------------------------------------
_AE = {0: [[0.5], [11 / 18, 1 / 18], [5 / 6, -5 / 6, 1 / 2], [1 / 4, 7 / 4, 3 / 4, -7 / 4]],
       2: [[1.0]]}
_AI = {0: [[0.5], [1 / 6, 1 / 2], [-1 / 2, 1 / 2, 1 / 2], [3 / 2, -3 / 2, 1 / 2, 1 / 2]],
       2: [[1.0]]}
_G = 1.0 - 1.0 / math.sqrt(2.0)
_D = 1.0 - 1.0 / (2.0 * _G)
_AE[1], _AI[1] = [[_G], [_D, 1.0 - _D]], [[_G], [1.0 - _G, _G]]


class _Plain:
    """The propagator of Secs. 2.1 and 3.2 (ultraspherical tau, 3/2-padded advective products) on
    batches (B, Nz, nm) of complex coefficients, with pivoted dense LU per Fourier mode."""

    def __init__(self, Ra, Nx, Nz, dt, scheme=0, bc=0):
        self.Ra, self.Nx, self.Nz, self.dt, self.bc = Ra, Nx, Nz, dt, bc
        self.AE, self.AI = _AE[scheme], _AI[scheme]
        self.nm, self.Mx, self.Mz = Nx // 2, 3 * Nx // 2, 3 * Nz // 2
        nm, Mz = self.nm, self.Mz
        k = 2.0 * np.pi / LX * np.arange(nm)
        D = np.zeros((Nz, Nz))
        for n in range(1, Nz):
            D[n - 1::-2, n] = 2.0 * n
        D[0] *= 0.5

        def conv(l):        # C^(l) -> C^(l+1), l = 0: T -> C^(1)
            S = np.zeros((Nz, Nz))
            for n in range(Nz):
                S[n, n] = (1.0 if n == 0 else 0.5) if l == 0 else l / (n + l)
                if n >= 2:
                    S[n - 2, n] = -0.5 if l == 0 else -l / (n + l)
            return S

        def der(l):         # T -> C^(l), d^l/ds^l
            M = np.zeros((Nz, Nz))
            for n in range(l, Nz):
                M[n - l, n] = 2.0 ** (l - 1) * math.factorial(l - 1) * n
            return M

        S2 = conv(1) @ conv(0)
        C32 = conv(3) @ conv(2)
        S4, S4D2, D2, D4 = C32 @ S2, C32 @ der(2), der(2), der(4)
        n = np.arange(Nz)
        lo, hi = (-1.0) ** n, np.ones(Nz)
        slo, shi = -((-1.0) ** n) * n ** 2.0, n ** 2.0
        h = self.AI[0][0] * dt
        kk = k[:, None, None]
        MT, LT = S2[:-2], 4.0 * D2[:-2] - kk * kk * S2[:-2]
        MP = 4.0 * S4D2[:-4] - kk * kk * S4[:-4]
        LP = PR * (16.0 * D4[:-4] - 8.0 * kk * kk * S4D2[:-4] + kk ** 4 * S4[:-4])
        LU = 4.0 * PR * D2[:-2]
        rows = np.stack([slo, shi] if bc else [lo, hi])
        AT = np.concatenate([MT - h * LT, np.broadcast_to(rows, (nm, 2, Nz))], 1)
        AP = np.concatenate([MP - h * LP, np.broadcast_to(np.stack([lo, hi, slo, shi]), (nm, 4, Nz))], 1)
        AP[0] = np.concatenate([MT - h * LU, lo[None], hi[None]], 0)      # m = 0: the mean flow
        up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
        self.k, self.D2z = up(k), up(2.0 * D)
        self.S2, self.S4, self.LU, self.LT, self.MP, self.LP = up(S2[:-2]), up(S4[:-4]), up(LU), up(LT), up(MP), up(LP)

        def factor(A):
            scale = 1.0 / np.abs(A).max(axis=2)                            # rows of equal size
            return up(scale), torch.linalg.lu_factor(up(A * scale[:, :, None]))

        (self.sT, self.fT), (self.sP, self.fP) = factor(AT), factor(AP)
        th = np.pi * np.arange(Mz) / (Mz - 1)
        self.V = up(np.cos(np.outer(th, n)))
        c = np.ones(Mz)
        c[0] = c[-1] = 2.0
        Wf = 2.0 / (Mz - 1) * np.cos(np.outer(np.arange(Mz), th)) / np.outer(c, c)
        self.W = up(Wf[:Nz])
        ev = np.arange(0, Mz, 2)
        self.cc = up((Wf[ev] * (2.0 / (1.0 - ev ** 2.0))[:, None]).sum(0))
        self.bval = (-0.5, -0.5) if bc else (1.0, 0.0)

    def mm(self, A, c):
        """A (r, Nz) applied along z to complex (B, Nz, nm); A may have a mode axis first."""
        A = A.to(torch.complex128)
        return torch.einsum("rn,bnm->brm", A, c) if A.dim() == 2 else torch.einsum("mrn,bnm->brm", A, c)

    def values(self, c):
        full = torch.zeros(c.shape[0], self.Mz, self.Mx // 2 + 1, dtype=torch.complex128, device=c.device)
        full[:, :, :self.nm] = self.mm(self.V, c)
        return torch.fft.irfft(full, n=self.Mx, dim=2) * self.Mx

    def coefs(self, g):
        return self.mm(self.W, torch.fft.rfft(g, dim=2)[:, :, :self.nm] / self.Mx)

    def fields(self, T, P):
        ik = 1j * self.k
        U = P[:, :, 0].clone()
        u = self.mm(self.D2z, P)
        u[:, :, 0] = U
        w = -ik * P
        w[:, :, 0] = 0.0
        om = ik * w - self.mm(self.D2z, u)
        return u, w, om

    def explicit(self, T, P):
        ik = 1j * self.k
        u, w, om = self.fields(T, P)
        ug, wg = self.values(u), self.values(w)
        NT = self.coefs(ug * self.values(ik * T) + wg * self.values(self.mm(self.D2z, T)))
        NO = self.coefs(ug * self.values(ik * om) + wg * self.values(self.mm(self.D2z, om)))
        NU = self.coefs(ug * self.values(ik * u) + wg * self.values(self.mm(self.D2z, u)))[:, :, 0]
        NO[:, :, 0] = NU.real
        wT = (wg * self.values(T)).mean(2)
        return NT, NO, wT

    def solve(self, rT, rP, ra):
        """(M - h L) X = r with the boundary rows; the buoyancy of the new T on the right of psi."""
        B, Nz, nm = rT.shape[0], self.Nz, self.nm
        h = self.AI[0][0] * self.dt

        def lu(f, s, b):      # complex right-hand sides (B, Nz, nm) with real matrices
            b = b * s.T
            x = torch.linalg.lu_solve(f[0], f[1], torch.cat([b.real, b.imag]).permute(2, 1, 0).contiguous())
            x = x.permute(2, 1, 0)
            return torch.complex(x[:B], x[B:])

        bT = torch.zeros(B, Nz, nm, dtype=torch.complex128, device="cuda")
        bT[:, :-2] = rT
        bT[:, -2, 0], bT[:, -1, 0] = self.bval
        T = lu(self.fT, self.sT, bT)
        bP = torch.zeros_like(bT)
        bP[:, :-4, 1:] = (rP[:, :-2] - h * 1j * self.k * PR * ra[:, None, None] * self.mm(self.S4, T))[:, :, 1:]
        bP[:, :-2, 0] = rP[:, :, 0]
        return T, lu(self.fP, self.sP, bP)

    @staticmethod
    def pad(x):               # Nz - 4 tau rows of psi kept beside the mean flow's Nz - 2
        return torch.nn.functional.pad(x, (0, 0, 0, 2))

    def rows(self, T, P, NT, NO, ra):
        """Tau rows of M X, F(X) and L X: T and (psi, m >= 1; mean flow, m = 0)."""
        def mixed(a, b):      # b (Nz - 4 rows) with its m = 0 column from a (Nz - 2 rows)
            out = self.pad(b)
            out[:, :, 0] = a[:, :, 0]
            return out

        MT = self.mm(self.S2, T)
        MP = mixed(self.mm(self.S2, P[:, :, :1]), self.mm(self.MP, P))
        FT = -self.mm(self.S2, NT)
        FP = mixed(-self.mm(self.S2, NO[:, :, :1]), self.mm(self.S4, NO))
        LT = self.mm(self.LT, T)
        LP = self.mm(self.LP, P) - 1j * self.k * PR * ra[:, None, None] * self.mm(self.S4, T)
        return MT, MP, FT, FP, LT, mixed(self.mm(self.LU, P[:, :, :1]), LP)

    def nuv(self, T, wT):
        return -2.0 * T[:, 1::2, 0].real.sum(1) + 0.5 * (wT * self.cc).sum(1)

    def run(self, T, P, nsteps, ra):
        """nsteps steps; the trapezoid integral of Nu_V."""
        nu = torch.zeros(T.shape[0], dtype=torch.float64, device="cuda")
        for i in range(nsteps):
            F, L = [], []
            MT = MP = None
            Tn, Pn = T, P
            for st in range(len(self.AE) + 1):
                NT, NO, wT = self.explicit(Tn, Pn) if st < len(self.AE) else (None, None, None)
                if st == 0:
                    nu += (0.5 if i == 0 else 1.0) * self.dt * self.nuv(T, wT)
                    MT, MP, FT, FP, _, _ = self.rows(T, P, NT, NO, ra)
                    F.append((FT, FP))
                    L.append(None)
                elif st < len(self.AE):
                    _, _, FT, FP, LT, LP = self.rows(Tn, Pn, NT, NO, ra)
                    F.append((FT, FP))
                    L.append((LT, LP))
                else:
                    break
                rT, rP = MT.clone(), MP.clone()
                for j, a in enumerate(self.AE[st]):
                    rT += self.dt * a * F[j][0]
                    rP += self.dt * a * F[j][1]
                for j, a in enumerate(self.AI[st][:-1]):
                    rT += self.dt * a * L[j + 1][0]
                    rP += self.dt * a * L[j + 1][1]
                Tn, Pn = self.solve(rT, rP, ra)
            T, P = Tn, Pn
        if nsteps:
            nu += 0.5 * self.dt * self.nuv(T, self.explicit(T, P)[2])
        return T, P, nu

    def diagnostics(self, T, P):
        u, w, om = self.fields(T, P)
        ik = 1j * self.k
        ug, wg, Tg = self.values(u), self.values(w), self.values(T)
        vol = lambda f: 0.5 * (f.mean(2) * self.cc).sum(1)   # noqa: E731
        lapdot = -ug * self.values(self.mm(self.D2z, om)) + wg * self.values(ik * om)
        Tm = Tg.mean(2)
        n2 = torch.arange(self.Nz, dtype=torch.float64, device="cuda") ** 2
        sg = (-1.0) ** torch.arange(self.Nz, dtype=torch.float64, device="cuda")
        a = T[:, :, 0].real
        head = torch.stack([torch.sqrt(vol(ug * ug + wg * wg)), vol(lapdot), vol(wg * Tg), self.nuv(T, (wg * Tg).mean(2)),
                            2.0 * (a * n2 * sg).sum(1), -2.0 * (a * n2).sum(1)], 1)
        return torch.cat([head, Tm, (Tg * Tg).mean(2)], 1)


def _split(X):
    return torch.view_as_complex(X[:, 0].contiguous()), torch.view_as_complex(X[:, 1].contiguous())


def _join(T, P):
    X = torch.stack([torch.view_as_real(T.resolve_conj()), torch.view_as_real(P.resolve_conj())], 1)
    X[:, :, :, 0, 1] = 0.0
    return X


def _l2(X, gram):
    w = torch.full((X.shape[3],), 2.0, dtype=torch.float64, device="cuda")
    w[0] = 1.0
    return 0.5 * LX * torch.einsum("bimc,ij,bjmc,m->b", X[:, 0], gram, X[:, 0], w)


def _gram(Nz):
    a, b = np.meshgrid(np.arange(Nz), np.arange(Nz), indexing="ij")
    g = np.where((a + b) % 2 == 0, 1.0, 0.0)
    s, d = 1.0 - (a + b) ** 2.0, 1.0 - (a - b) ** 2.0
    return torch.from_numpy(g * (1.0 / np.where(s == 0, 1.0, s) + 1.0 / np.where(d == 0, 1.0, d))).cuda()


def exact(case, seed):
    kind = case["kind"]
    full = lambda B: torch.full((B,), float(case["Ra"]), dtype=torch.float64, device="cuda")   # noqa: E731
    if kind in ("step", "sampled"):
        X = _states(case, case["B"], seed)
        p = _Plain(case["Ra"], case["Nx"], case["Nz"], case["dt"], case["scheme"], case["bc"])
        out, nu = X.clone(), torch.zeros(case["B"], dtype=torch.float64, device="cuda")
        if kind == "sampled":
            (T, P), stat, done = _split(X), 0.0, 0
            prev = p.diagnostics(T, P)
            while done < case["nsteps"]:
                c = min(case["every"], case["nsteps"] - done)
                T, P, nc = p.run(T, P, c, full(case["B"]))
                cur = p.diagnostics(T, P)
                stat = stat + 0.5 * (c * case["dt"]) * (prev + cur)
                prev, nu, done = cur, nu + nc, done + c
            return _join(T, P), nu, stat
        ns, ra = _uneven(case, seed) if case["uneven"] else ([case["nsteps"]] * case["B"], [case["Ra"]] * case["B"])
        ra = torch.tensor(ra, dtype=torch.float64, device="cuda")
        size = max(1, (1 << 21) // (case["Nx"] * case["Nz"]))
        for n in sorted(set(ns)):
            at = [b for b in range(case["B"]) if ns[b] == n and n > 0]
            for i in range(0, len(at), size):
                part = at[i:i + size]
                T, P, nb = p.run(*_split(X[part]), n, ra[part])
                out[part], nu[part] = _join(T, P), nb
        return out, nu
    if kind == "tick":
        s = prepare(case, seed)
        Nzc, nmc = case["Nzc"], case["Nxc"] // 2
        U = s["Ff"].clone()
        U[:, :, :Nzc, :nmc] += s["Gnew"] - s["Gold"]
        g = _gram(case["Nz"])
        return U, U[:, :, :Nzc, :nmc].contiguous(), _l2(U - s["old"], g), _l2(U, g)
    return _exact_parareal(case, seed)


def _exact_parareal(case, seed):
    Nx, Nz, N, nm = case["Nx"], case["Nz"], case["slices"], case["Nx"] // 2
    Nzc, nmc = case["Nzc"], case["Nxc"] // 2
    F = _Plain(case["Ra"], Nx, Nz, case["dt"], 0)
    G = _Plain(case["Ra"], case["Nxc"], Nzc, case["dt"] * case["nf"] / case["nc"], case["scheme"])
    ra = torch.full((N,), float(case["Ra"]), dtype=torch.float64, device="cuda")
    T, u, w = _grid(case, seed)
    to_modes = lambda g: torch.fft.rfft(torch.from_numpy(g).cuda(), dim=1)[:, :nm] / Nx   # noqa: E731
    W = _interp(Nz).to(torch.complex128)
    ik = 1j * F.k
    P = torch.zeros(Nz, nm, dtype=torch.complex128, device="cuda")
    P[:, 1:] = (W @ to_modes(w))[:, 1:] / -ik[1:]
    P[:, 0] = (W @ to_modes(u))[:, 0].real
    T0 = W @ to_modes(T)
    T0[:, 0] = T0[:, 0].real.clone()
    U0 = _join(T0[None], P[None])[0]

    def coarse(x):
        a, b, _ = G.run(*_split(x[None, :, :Nzc, :nmc].contiguous()), case["nc"], ra[:1])
        out = torch.zeros_like(x)
        out[:, :Nzc, :nmc] = _join(a, b)[0]
        return out

    U = torch.zeros((N + 1,) + tuple(U0.shape), dtype=torch.float64, device="cuda")
    U[0] = U0
    old = []
    for n in range(N):
        old.append(coarse(U[n]))
        U[n + 1] = old[n]
    gram, defects, nus, nui = _gram(Nz), [], [], torch.zeros(N, dtype=torch.float64, device="cuda")
    k = 0
    for k in range(1, min(case["iters"], N) + 1):
        a, b, nu = F.run(*_split(U[k - 1:N].contiguous()), case["nf"], ra[:N - k + 1])
        fine, new = _join(a, b), U.clone()
        nui[k - 1:] = nu
        for n in range(k - 1, N):
            g = old[n] if n == k - 1 else coarse(new[n])
            new[n + 1] = fine[n - k + 1] + (g - old[n])
            old[n] = g
        d2, u2 = _l2(new - U, gram)[k:], _l2(new, gram)[k:]
        defects.append(float(torch.sqrt(d2 / u2).max()))
        nus.append(float(nui[N // 2:].sum()) / (case["nf"] * case["dt"] * (N - N // 2)))
        U = new
    end = torch.view_as_complex(U[-1].contiguous())
    V = torch.from_numpy(np.cos(np.outer(np.pi * (Nz - 1 - np.arange(Nz)) / (Nz - 1), np.arange(Nz)))).cuda().to(torch.complex128)
    um = V @ (F.D2z.to(torch.complex128) @ end[1])
    um[:, 0] = V @ end[1][:, 0]
    wm = -ik * (V @ end[1])

    def values(c):
        f = torch.zeros(Nz, nm + 1, dtype=torch.complex128, device="cuda")
        f[:, :nm] = c
        return (torch.fft.irfft(f, n=Nx, dim=1) * Nx).cpu().numpy()

    return U, np.array(defects), np.array(nus), values(V @ end[0]), values(um), values(wm), k
