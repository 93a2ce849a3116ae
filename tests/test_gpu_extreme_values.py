"""Values at the ends of the range. Waves of subnormal amplitude (2^-1030), as a march decayed that far has them:
every path scales its columns by powers of two, so the first step (no history:
the mixed path's bf16 panels hold nothing this small) and the FP64 march are the
unit-amplitude ones up to the quantum of the values themselves, 4.9e-324 or
5.7e-14 of the amplitude. Bound: a step's right-hand side is 3e-2 of the amplitude
and some five sums deep, 1e-11 of it is quantum, and the condition number of Q_0
(250) makes 3e-9 of that at worst: 1e-8."""
import numpy as np
import pytest

from paper_2510_07989_gb300.inputs import meshes as MS
from paper_2510_07989_gb300.inputs.assemble import assemble

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_2510_07989_gb300.build import build
    build()
    from paper_2510_07989_gb300 import mot
    return mot


@pytest.fixture(scope="module")
def ops():
    return assemble(MS.torus(1.0, 0.3, 9, 5), 4.0, 1.0, 0.3)


PATHS = [({}, 1), ({}, 9), ({"fp64_precond": 1}, 3), ({"fp64_direct": 1}, 3), ({"precision": 1}, 3),
         ({"precision": 1}, 8)]


@pytest.mark.parametrize("kw,B", PATHS, ids=lambda v: str(v) if isinstance(v, int) else "-".join(v) or "plain")
def test_subnormal_amplitude(M, ops, kw, B):
    n = 1 if "precision" in kw else 12
    exc = MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=4, r_obj=1.3)
    one = M.Solver(ops, **kw).run(exc, n)
    exc.A[:] = 2.0 ** -1030
    s = M.Solver(ops, **kw)
    tiny = s.run(exc, n)
    assert s.noconv == 0 and np.isfinite(tiny).all()
    assert np.abs(tiny * 2.0 ** 1000 * 2.0 ** 30 - one).max() < 1e-8 * np.abs(one).max()


def test_a_column_that_is_no_number(M, ops):
    """A NaN in one wave's history: the step says that a solve did not converge,
    and the waves whose columns share a cluster with it are the undisturbed ones
    (1e-12: the sweeps of a solve stop together)."""
    B = 5
    exc = MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=4, r_obj=1.3)
    waves, out, ref = M.mot_waves(exc), np.zeros((B, 2, ops.ne)), np.zeros((B, 2, ops.ne))
    s = M.Solver(ops)
    s.run(exc, 4, keep=False)
    blob = bytearray(M.mot_save_state(s.h))
    assert M.mot_step(s.h, waves, B, ref) == M.MOT_OK
    npad = (ops.ne + 31) // 32 * 32
    # after the header and the waves: [slot][part][variant][row][2B]; row 5, u of wave 1 of step 3
    ring = np.frombuffer(blob, dtype=np.float64, offset=40 + 80 * B)[:4 * 6 * npad * 2 * B]
    assert ring.any()
    ring = ring.reshape(4, 6, npad, 2 * B)
    ring[3, :2, 5, 1] = np.nan
    t = M.Solver(ops)
    M.mot_load_state(t.h, bytes(blob))
    assert M.mot_step(t.h, waves, B, out) == M.MOT_ENOCONV
    keep = [0, 2, 3, 4]
    assert np.abs(out[keep] - ref[keep]).max() < 1e-12 * np.abs(ref).max()
