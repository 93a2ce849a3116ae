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


@pytest.mark.parametrize("B,n_dir,F", [(1, 1, 40), (1, 1, 90), (1, 1, 160), (3, 2, 80), (64, 1, 20), (64, 1, 1), (10, 2, 3), (5, 33, 1), (64, 9, 17)])
def test_far_field_of_many_frequencies(M, ops, B, n_dir, F):
    """Shapes that the far field cuts differently: more frequencies than its point
    currents hold (17 at this size and 64 waves), waves over several clusters, ragged
    wave and direction tiles, one direction. Against the oracle's radiation integrals
    of the same steps' currents, the 1e-9 of the far field's other parity tests."""
    from oracle import farfield as FF
    from oracle import product as P
    S = P.ProductSystem(ops)
    exc = MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=20, r_obj=1.3)
    n, omegas = 30, np.linspace(0.0, 1.1, F)
    s = M.Solver(ops, fp64_precond=1)
    M.mot_set_frequencies(s.h, omegas)
    W = s.run(exc, n)
    t = np.linspace(0.1, 3.0, n_dir)
    dirs = np.stack([np.sin(t) * np.cos(2 * t), np.sin(t) * np.sin(2 * t), np.cos(t)], axis=1)
    E = M.mot_fields(s.h, M.mot_waves(exc), dirs, F, B)
    for b in sorted({0, B // 2, B - 1}):
        parts = [S.split(w) for w in W[:, b].reshape(n, -1)]
        ell = np.array([p[0] for p in parts])
        sg = np.array([p[1] for p in parts])
        cur = ell + ops.tmax / ops.dt * np.diff(sg, axis=0, prepend=np.zeros((1, sg.shape[1])))
        for f in sorted({0, F // 2, F - 1}):
            X = cur.T @ FF.dft_weights(omegas[f], ops.dt, n)
            ref = FF.far_field(ops.rwg, X[:ops.ne], X[ops.ne:], omegas[f], 1.0, dirs)
            ref = ref / FF.pulse_spectrum(exc, b, omegas[f])
            assert np.abs(E[b, f] - ref).max() <= 1e-9 * np.abs(ref).max()
