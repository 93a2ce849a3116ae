"""Frequencies of the running Fourier sums: a refused list changes nothing."""
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


@pytest.mark.parametrize("bad", [[-1.0], [0.5, np.nan]])
def test_refused_list(M, ops, bad):
    exc = MS.fibonacci_batch(3, ops.dt, w_steps=20, t0_steps=4, r_obj=1.3)
    dirs = np.array([[0.0, 0.6, 0.8]])
    s, t = M.Solver(ops), M.Solver(ops)
    for u in (s, t):
        M.mot_set_frequencies(u.h, np.array([0.7]))
    with pytest.raises(M.MotError) as e:
        M.mot_set_frequencies(s.h, np.array(bad))
    assert e.value.code == M.MOT_EINVAL
    E = []
    for u in (s, t):
        u.run(exc, 5, keep=False)
        E.append(M.mot_fields(u.h, M.mot_waves(exc), dirs, 1, 3))
    assert np.array_equal(*E) and np.abs(E[0]).max() > 0
