"""FP64 march over the batch sizes at which its dense products and its history
contraction change form: skinny products (B columns of Q_0, 2B and 4B columns
of the left factor) by rows, in 16- and in 32-column tiles, whole and split,
ragged last tiles; the history with whole tiles (B < 4) and by nonzero masks
(warps inside one row, and across two). Against the product-form FP64 oracle
within the 1e-10 of the FP64 path's other parity tests (the dense oracle's
pseudo-inverse of Lambda^T Lambda keeps a rounding-sized singular value of this
45-vertex mesh: its projector misses P^2 = P by 1e-4)."""
import numpy as np
import pytest

from oracle import product as P
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
def torus():
    ops = assemble(MS.torus(1.0, 0.3, 9, 5), 4.0, 1.0, 0.3)  # 135 edges: ragged last row block
    return ops, P.ProductSystem(ops)


CASES = [({}, B) for B in (1, 2, 3, 5, 7, 8, 9, 15, 16, 17, 24, 33, 64)]
CASES += [({k: 1}, B) for k in ("fp64_precond", "fp64_direct") for B in (3, 9, 33)]


@pytest.mark.parametrize("kw,B", CASES, ids=lambda v: str(v) if isinstance(v, int) else "-".join(v) or "plain")
def test_fp64_march_over_batches(M, torus, kw, B):
    ops, S = torus
    exc = MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=20, r_obj=1.3)
    n = 35
    s = M.Solver(ops, **kw)
    W = s.run(exc, n)
    assert s.noconv == 0
    for b in sorted({0, B - 1}):
        ref = S.march(exc, n, b=b)
        assert np.abs(W[:, b].reshape(n, -1) - ref).max() < 1e-10 * np.abs(ref).max()


def test_preconditioned_solve_past_the_kept_vectors(M, torus):
    """A preconditioned solve longer than the Krylov vectors M V_j it keeps
    (12): 14 iterations forced by a tolerance that 14 do not reach (each gains some
    14 digits). The status
    says so, and the iterate kept is the solution to the same 1e-10."""
    ops, S = torus
    exc = MS.fibonacci_batch(2, ops.dt, w_steps=20, t0_steps=20, r_obj=1.3)
    n = 35
    s = M.Solver(ops, fp64_precond=1, gmres_tol=1e-300, gmres_maxit=14)
    W = s.run(exc, n)
    assert s.noconv > 0 and s.info()["last_gmres_iters"] == 14
    ref = S.march(exc, n, b=1)
    assert np.abs(W[:, 1].reshape(n, -1) - ref).max() < 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("B,n_dir", [(1, 1), (1, 17), (9, 9), (48, 6), (64, 3)])
def test_far_field_over_batches(M, torus, B, n_dir):
    """The far field for batches and direction counts that fill a CTA's threads
    (direction, wave, share of the points) in different ways, ragged last
    direction tiles among them: against the oracle's radiation integrals of the
    currents recovered from the same steps, the 1e-9 of the parity test."""
    from oracle import farfield as FF
    ops, S = torus
    exc = MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=20, r_obj=1.3)
    n, omegas = 30, np.array([0.0, 0.7])
    s = M.Solver(ops, fp64_precond=1)
    M.mot_set_frequencies(s.h, omegas)
    W = s.run(exc, n)
    t = np.linspace(0.1, 3.0, n_dir)
    dirs = np.stack([np.sin(t) * np.cos(2 * t), np.sin(t) * np.sin(2 * t), np.cos(t)], axis=1)
    E = M.mot_fields(s.h, M.mot_waves(exc), dirs, 2, B)
    for b in sorted({0, B - 1}):
        parts = [S.split(w) for w in W[:, b].reshape(n, -1)]
        ell = np.array([p[0] for p in parts])
        sg = np.array([p[1] for p in parts])
        cur = ell + ops.tmax / ops.dt * np.diff(sg, axis=0, prepend=np.zeros((1, sg.shape[1])))
        for f, w in enumerate(omegas):
            X = cur.T @ FF.dft_weights(w, ops.dt, n)
            ref = FF.far_field(ops.rwg, X[:ops.ne], X[ops.ne:], w, 1.0, dirs) / FF.pulse_spectrum(exc, b, w)
            assert np.abs(E[b, f] - ref).max() <= 1e-9 * np.abs(ref).max()


@pytest.mark.parametrize("kw,B,tol", [({}, 2, 1e-10), ({"fp64_precond": 1}, 5, 1e-10), ({"precision": 1}, 8, 1e-6)],
                         ids=["plain", "precond", "mixed"])
def test_two_separate_spheres(M, kw, B, tol):
    """One mesh of two components: its graph Laplacians have a null space larger
    than the constants, so the dense inverses behind the projector solves do not
    serve and plain CG takes their place. Against the product-form oracle,
    within the paths' usual bounds."""
    a = MS.icosphere(1)
    m = MS.build_edges(MS.Mesh(np.concatenate([a.verts * 0.5 - [0.8, 0, 0], a.verts * 0.5 + [0.8, 0, 0]]),
                               np.concatenate([a.tris, a.tris + a.nv]).astype(np.int32), name="two spheres"))
    ops = assemble(m, 2.0, 1.0, 0.3)
    exc = MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=20, r_obj=1.4)
    n = 40
    s = M.Solver(ops, **kw)
    W = s.run(exc, n)
    assert s.noconv == 0
    ref = P.ProductSystem(ops).march(exc, n, b=B - 1)
    assert np.abs(W[:, B - 1].reshape(n, -1) - ref).max() < tol * np.abs(ref).max()
