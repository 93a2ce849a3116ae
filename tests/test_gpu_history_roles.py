"""Role layouts of the tensor-core history kernel that other tests do not end
early: with hist_stall_test the first CTA of every launch withholds one stage's
copies -- four epilogue warps (gather workers that also copy the tiles) with
one task per stage, eight (a warp of its own for the tiles) with two -- and
mot_step returns MOT_ECUDA with the context usable, a fresh handle marching to
the oracle's result."""
import numpy as np
import pytest

from oracle import product as P
from paper_2510_07989_gb300.inputs import meshes as MS
from paper_2510_07989_gb300.inputs.assemble import assemble

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", [(5, 1, 4), (2, 2, 8), (3, 2, 8)])
def test_stalled_stage_ends_in_error_status(cfg):
    from paper_2510_07989_gb300.build import build
    build()
    from paper_2510_07989_gb300 import mot as M
    ops = assemble(MS.torus(1.0, 0.3, 9, 5), 4.0, 1.0, 0.2)
    exc = MS.fibonacci_batch(16, ops.dt, w_steps=20, t0_steps=20, r_obj=1.3)
    waves = M.mot_waves(exc)
    s = M.Solver(ops, precision=M.MOT_PREC_MIXED, hist_stall_test=3)
    M.mot_step(s.h, waves, 16)
    M.mot_set_tc_config(s.h, 512, 0.4, *cfg)
    with pytest.raises(M.MotError) as e:
        for _ in range(ops.kmax + 8):
            M.mot_step(s.h, waves, 16)
    assert e.value.code == M.MOT_ECUDA and "ran out of time" in str(e.value)
    del s
    n = 40
    s = M.Solver(ops, precision=M.MOT_PREC_MIXED)
    out = np.zeros((16, 2, ops.ne))
    W = np.zeros((n, 2 * ops.ne))
    for i in range(n):
        M.mot_step(s.h, waves, 16, out)
        if i == 0:
            M.mot_set_tc_config(s.h, 512, 0.4, *cfg)
        W[i] = out[7].reshape(-1)
    ref = P.ProductSystem(ops).march(exc, n, b=7)
    assert np.abs(W - ref).max() < 1e-6 * np.abs(ref).max()
