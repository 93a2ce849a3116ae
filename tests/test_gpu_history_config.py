"""A refused configuration of the tensor-core history leaves a handle that steps
on: the chunking is replaced all the same, and one task per chunk is many times
the chunks that the handle's buffer of partial sums was sized for. Against the
product-form oracle within the mixed path's 1e-6."""
import numpy as np
import pytest

from oracle import product as P
from paper_2510_07989_gb300.inputs import meshes as MS
from paper_2510_07989_gb300.inputs.assemble import assemble

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at", [1, 30])
def test_march_after_a_refused_configuration(at):
    from paper_2510_07989_gb300.build import build
    build()
    from paper_2510_07989_gb300 import mot as M
    ops = assemble(MS.torus(1.0, 0.3, 9, 5), 4.0, 1.0, 0.2)
    B, n = 16, 40
    exc = MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=20, r_obj=1.3)
    waves = M.mot_waves(exc)
    s = M.Solver(ops, precision=M.MOT_PREC_MIXED)
    out, W = np.zeros((B, 2, ops.ne)), np.zeros((n, 2 * ops.ne))
    for i in range(n):
        M.mot_step(s.h, waves, B, out)
        W[i] = out[7].reshape(-1)
        if i + 1 == at:
            with pytest.raises(M.MotError) as e:
                M.mot_set_tc_config(s.h, 1, 0.4, 5, 2, 8)  # no pipeline of five two-task stages
            assert e.value.code == M.MOT_EINVAL
    assert s.info()["tc_chunk_cap"] == 1
    ref = P.ProductSystem(ops).march(exc, n, b=7)
    assert np.abs(W - ref).max() < 1e-6 * np.abs(ref).max()
