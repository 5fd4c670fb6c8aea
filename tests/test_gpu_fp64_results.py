"""What the FP64 mode's own arithmetic has to give: rows with a broad spectrum, and
results that ill-conditioned outputs of a run depend on to the last bits."""
import os

import numpy as np
import pytest

from layout import from_abi, to_abi
from oracle.rbc import RBC, State
from paper_2001_01609_gb300.inputs import initial_temperature

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::DeprecationWarning")]

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fp64_parareal_defects.txt")


@pytest.fixture(scope="module")
def rbc():
    from paper_2001_01609_gb300 import build
    build.build()
    from paper_2001_01609_gb300 import rbc as r
    r.load()
    return r


@pytest.mark.parametrize("decay", [np.inf, 40.0, 3.0])
@pytest.mark.parametrize("Nx", [256, 1024])
def test_mean_flow_of_rows_with_a_broad_spectrum(rbc, Nx, decay):
    """White and decaying modes, one forward-backward Euler step from rest in the mean: U is the x-mean of the products
    alone.  Three FFTs of log2(Mx) passes and the sum over Mx points, 2^-53 relative to the rms each: 4e-15; 1e-14."""
    Nz, dt, nm = 10, 1e-6, Nx // 2
    o = RBC(1e4, 1.0, 2.0, Nx, Nz, dt, scheme="RK111")
    g = np.random.default_rng(Nx)
    amp = np.exp(-np.arange(nm) / decay)[:, None] * 0.7 ** np.arange(Nz)
    T, psi = ((g.standard_normal((nm, Nz)) + 1j * g.standard_normal((nm, Nz))) * amp for _ in range(2))
    T[0] = T[0].real
    psi[0] = 0.0
    X = State(T, 1e6 * psi, np.zeros(Nz))
    F = rbc.Propagator(1e4, 1.0, 2.0, Nx, Nz, dt, rbc.RBC_FP64, scheme=rbc.RBC_RK111)
    st = F.new_states(1)
    st[0].copy_(torch.from_numpy(to_abi(X)))
    F.step_batch(st, 1)
    U, ref = from_abi(st[0].cpu().numpy()).U, o.run(X, 1)[0].U
    assert np.linalg.norm(U - ref) <= 1e-14 * np.linalg.norm(ref)


RUNS = [(64, 32, 32, 16, 1e4, 1e-3, 20, 5, 4), (256, 34, 128, 18, 18800.0, 1.25e-4, 12, 6, 2),
        (128, 64, 64, 32, 1e5, 1.5625e-5, 8, 4, 3)]


def parareal_defects(rbc, Nx, Nz, Nxc, Nzc, Ra, dt, nf, nc, slices):
    F = rbc.Propagator(Ra, 1.0, 2.0, Nx, Nz, dt)
    G = rbc.Propagator(Ra, 1.0, 2.0, Nxc, Nzc, dt * nf / nc)
    U0, U = F.new_states(1), F.new_states(slices + 1)
    x, z = 2.0 * np.pi * np.arange(Nx) / Nx, -0.5 * np.cos(np.pi * np.arange(Nz) / (Nz - 1))
    w = 0.2 * np.outer((0.25 - z * z) ** 2, np.cos(x) + 0.3 * np.sin(3.0 * x))
    F.set_state(U0[0], initial_temperature(Nx, Nz, seed=5, amplitude=1e-3, Lx=2.0), 0.0 * w, w)
    return rbc.Parareal(F, G, 0.0, slices * nf * dt, slices).iterate(U0[0], U, 2)[2]


@pytest.mark.parametrize("i", range(len(RUNS)))
def test_parareal_defects_are_the_recorded_ones(rbc, i):
    """A defect of 1e-6 or less is a difference of nearly equal states: it moves by 1e-10 when any rounding of the FP64
    arithmetic changes (an FFT's radices, the order of a sum or of a recurrence).  Recorded on GB300, CUDA 13.0; 5e-12."""
    with open(GOLDEN) as f:
        rows = [[float.fromhex(v) for v in s.split()] for s in f if not s.startswith("#")]
    for d, ref in zip(parareal_defects(rbc, *RUNS[i]), rows[i]):
        assert abs(d - ref) <= 5e-12 * ref
