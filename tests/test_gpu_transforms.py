"""The transform kernels at the edges of their sizes, against the FP64 oracle.

One step of every row length (Nx = 4 .. 1024: odd and even numbers of radix-4
steps, rows in shared memory together and in turn) and batch size (a cluster or
a block per row, several rows per block, a ragged last block), and of column
lengths up to the largest, around the dense solve's limit, the chunks of the
recurrences and the tensor-core tiles, alone and in batches of other tilings.
Tolerances: FP64 1e-12 relative to the largest coefficient (the
implementations' roundings differ by up to 2e-15 in one step of the tall grids);
FP32 products 1e-5, the bound of the mixed mode's parity tests.
"""
import numpy as np
import pytest

from layout import from_abi, max_rel_diff, to_abi
from oracle.rbc import RBC
from paper_2001_01609_gb300.inputs import initial_temperature

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::DeprecationWarning")]


@pytest.fixture(scope="module")
def rbc():
    from paper_2001_01609_gb300 import build
    build.build()
    from paper_2001_01609_gb300 import rbc as r
    r.load()
    return r


def nonlinear_state(o, seed):
    X = o.from_grid(initial_temperature(o.Nx, o.Nz, seed=seed, amplitude=0.3, Lx=o.Lx))
    X, _ = o.step(X)
    return X


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
@pytest.mark.parametrize("Nx", [4, 8, 16, 32, 64, 128, 256, 512, 1024])
def test_every_row_length_matches_oracle(rbc, Nx, precision, tol):
    Nz, Ra, dt = 10, 1e5, 1e-4
    o = RBC(Ra, 1.0, 2.0, Nx, Nz, dt)
    F = rbc.Propagator(Ra, 1.0, 2.0, Nx, Nz, dt, precision)
    Xs = [nonlinear_state(o, s) for s in range(3)]
    st = F.new_states(3)
    for b, X in enumerate(Xs):
        st[b].copy_(torch.from_numpy(to_abi(X)))
    nu = torch.zeros(3, dtype=torch.float64, device="cuda")
    F.step_batch(st, [2, 0, 1], nu)
    assert F.check_diverged() == rbc.RBC_OK
    for b, n in enumerate([2, 0, 1]):
        ref, integ = o.run(Xs[b], n)
        assert max_rel_diff(from_abi(st[b].cpu().numpy()), ref) < tol
        assert abs(nu[b].item() - integ) <= tol * max(abs(integ), 1e-30)


@pytest.mark.parametrize("Nz", [8, 16, 18, 32, 34, 36, 64, 66, 128, 130, 258, 384, 510, 512])
def test_column_lengths_match_oracle_and_batches_agree(rbc, Nz, Nx=8):
    Ra, dt = 1e4, 1e-5
    o = RBC(Ra, 1.0, 2.0, Nx, Nz, dt)
    F = rbc.Propagator(Ra, 1.0, 2.0, Nx, Nz, dt, 0)
    X0 = nonlinear_state(o, 7)
    alone = F.new_states(1)
    alone[0].copy_(torch.from_numpy(to_abi(X0)))
    states = {B: alone[:1].repeat(B, 1, 1, 1, 1) for B in (3, 40, 100)}
    nu = torch.zeros(100, dtype=torch.float64, device="cuda")
    F.step_batch(alone, 1, nu[:1])
    ref, integ = o.run(X0, 1)
    assert max_rel_diff(from_abi(alone[0].cpu().numpy()), ref) < 1e-12
    assert abs(nu[0].item() - integ) <= 1e-12 * abs(integ)
    for B, st in states.items():
        nub = torch.zeros(B, dtype=torch.float64, device="cuda")
        F.step_batch(st, 1, nub)
        assert torch.equal(st, alone.expand_as(st)) and torch.equal(nub, nu[:1].expand(B)), B
    assert F.check_diverged() == rbc.RBC_OK


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("Nx", [4, 8, 16, 32, 64, 128, 256, 512, 1024])
def test_rows_alone_and_in_batches_agree(rbc, Nx, precision, Nz=10):
    """15 rows (FP64: a cluster each; mixed: one per block, the last inverse pass spread), 345 and 2250 rows (FP64: a
    block each; mixed: several per block, a ragged last one)."""
    F = rbc.Propagator(1e5, 1.0, 2.0, Nx, Nz, 1e-4, precision)
    o = RBC(1e5, 1.0, 2.0, Nx, Nz, 1e-4)
    alone = F.new_states(1)
    alone[0].copy_(torch.from_numpy(to_abi(nonlinear_state(o, 5))))
    states = [alone[:1].repeat(B, 1, 1, 1, 1) for B in (23, 150)]
    nu = torch.zeros(1, dtype=torch.float64, device="cuda")
    F.step_batch(alone, 2, nu)
    for st in states:
        nub = torch.zeros(st.shape[0], dtype=torch.float64, device="cuda")
        F.step_batch(st, 2, nub)
        assert torch.equal(st, alone.expand_as(st)) and torch.equal(nub, nu.expand_as(nub))
    assert F.check_diverged() == rbc.RBC_OK


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("Nz", [34, 62, 64, 66, 96, 128, 130, 256, 258, 384, 510, 512])
def test_mixed_column_lengths_match_oracle_and_batches_agree(rbc, Nz, precision, Nx=16):
    """K-chunks and row tiles of the tensor-core transforms (one per CTA alone, all of a field's in batches), rows per
    thread and chunks of the stage solve; the FP32 CUDA-core transforms where TF32 operands do not fit (Nz = 384: the
    inverse, 510 and 512: both)."""
    Ra, dt = 1e4, 1e-5
    o = RBC(Ra, 1.0, 2.0, Nx, Nz, dt)
    F = rbc.Propagator(Ra, 1.0, 2.0, Nx, Nz, dt, precision)
    X0 = nonlinear_state(o, 3)
    alone = F.new_states(1)
    alone[0].copy_(torch.from_numpy(to_abi(X0)))
    states = [alone[:1].repeat(B, 1, 1, 1, 1) for B in (5, 60, 170)]
    nu = torch.zeros(1, dtype=torch.float64, device="cuda")
    F.step_batch(alone, 1, nu)
    ref, integ = o.run(X0, 1)
    assert max_rel_diff(from_abi(alone[0].cpu().numpy()), ref) < 1e-5
    for st in states:
        nub = torch.zeros(st.shape[0], dtype=torch.float64, device="cuda")
        F.step_batch(st, 1, nub)
        assert torch.equal(st, alone.expand_as(st)) and torch.equal(nub, nu.expand_as(nub))
    assert F.check_diverged() == rbc.RBC_OK
