"""GMRES solves longer than the 100 vectors of a cycle. A torus of magnetic
material (mu_r = 100; the condition number of Q_0 is 2.7e3) takes some 110
iterations without a preconditioner to gain six digits, so every solve below
restarts. The first step has no history and shows the solve alone, against the
FP64 oracle's Q_0 solved directly; the bounds are the residual asked for
times that condition number."""
import numpy as np
import pytest

from oracle import mot as O
from oracle import product as P
from paper_2510_07989_gb300.inputs import meshes as MS
from paper_2510_07989_gb300.inputs.assemble import assemble

pytestmark = pytest.mark.gpu
COND = 2.7e3


@pytest.fixture(scope="module")
def M():
    from paper_2510_07989_gb300.build import build
    build()
    from paper_2510_07989_gb300 import mot
    return mot


@pytest.fixture(scope="module")
def torus():
    ops = assemble(MS.torus(1.0, 0.3, 10, 5), 2.0, 100.0, 1.0)
    exc = MS.fibonacci_batch(8, ops.dt, w_steps=20, t0_steps=4, r_obj=1.3)
    S = P.ProductSystem(ops)
    Q = np.array([S.q0(c) for c in np.eye(2 * ops.ne)]).T
    ref = np.array([np.linalg.solve(Q, S.left(*O.rhs_parts(ops, exc, b, 1))) for b in range(8)])
    return ops, exc, ref


def first_step(M, s, ops, exc, B):
    out = np.zeros((B, 2, ops.ne))
    assert M.mot_step(s.h, M.mot_waves(exc), B, out) == M.MOT_OK
    assert s.info()["last_gmres_iters"] > 100
    return out.reshape(B, -1)


def err(w, ref):
    return (np.linalg.norm(w - ref, axis=1) / np.linalg.norm(ref, axis=1)).max()


@pytest.mark.parametrize("emu", [False, True], ids=["fp32", "slices"])
def test_refinement_through_a_restart(M, torus, emu):
    """The solve with the reduced-precision Q_0 leaves a residual of 2e-6 (its
    tolerance and that Q_0's rounding), the correction gains six digits on it; a
    correction that takes up that Q_0's own solution ends at 1e-6 instead."""
    ops, exc, ref = torus
    flags = M.MOT_MIX_HIST32 | M.MOT_MIX_Q032 | M.MOT_MIX_REFINE | M.MOT_MIX_TC | (M.MOT_MIX_EMU64 if emu else 0)
    s = M.Solver(ops, precision=M.MOT_PREC_MIXED, mixed_flags=flags, gmres_maxit=400)
    assert err(first_step(M, s, ops, exc, 8), ref) < COND * 2e-12


@pytest.mark.parametrize("B", [1, 8])
def test_fp64_solve_through_a_restart(M, torus, B):
    ops, exc, ref = torus
    s = M.Solver(ops, gmres_maxit=800)
    assert err(first_step(M, s, ops, exc, B), ref[:B]) < COND * 2e-13


def test_correction_gains_six_digits_whatever_the_tolerance(M):
    """gmres_tol says when a step's residual needs no (further) correction; a
    correction that is made goes six digits below its residual. Without the
    preconditioner the first solve ends between 1e-7 and 1e-6, so the step is within
    4e-12 (the correction, and the emulated products of the two right-hand sides)
    times the condition number of Q_0, here 250."""
    ops = assemble(MS.torus(1.0, 0.3, 9, 5), 4.0, 1.0, 0.3)
    exc = MS.fibonacci_batch(8, ops.dt, w_steps=20, t0_steps=4, r_obj=1.3)
    S = P.ProductSystem(ops)
    Q = np.array([S.q0(c) for c in np.eye(2 * ops.ne)]).T
    ref = np.array([np.linalg.solve(Q, S.left(*O.rhs_parts(ops, exc, b, 1))) for b in range(8)])
    flags = M.MOT_MIX_DEFAULT & ~M.MOT_MIX_PRECOND
    s = M.Solver(ops, precision=M.MOT_PREC_MIXED, mixed_flags=flags, gmres_tol=1e-7)
    out = np.zeros((8, 2, ops.ne))
    assert M.mot_step(s.h, M.mot_waves(exc), 8, out) == M.MOT_OK
    assert s.info()["last_gmres_resid"] > 1e-7
    assert err(out.reshape(8, -1), ref) < 250 * 4e-12


@pytest.mark.parametrize("B", [3, 7, 33, 64])
def test_long_iterations_over_batches(M, B):
    """Solves of 100 vectors and more, whose iterations change from one launch to
    several on the way (here at 32 vectors): batches that fill the threads of a row
    stride or leave some over."""
    ops = assemble(MS.torus(1.0, 0.3, 10, 5), 2.0, 100.0, 1.0)
    exc = MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=4, r_obj=1.3)
    S = P.ProductSystem(ops)
    Q = np.array([S.q0(c) for c in np.eye(2 * ops.ne)]).T
    ref = np.linalg.solve(Q, np.array([S.left(*O.rhs_parts(ops, exc, b, 1)) for b in range(B)]).T).T
    s = M.Solver(ops, gmres_maxit=800)
    assert err(first_step(M, s, ops, exc, B), ref) < COND * 2e-13
