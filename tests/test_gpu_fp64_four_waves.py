"""Four waves on the FP64 path: the widest of the history kernels that keep their
sums in registers (2B = 8 columns). Against the product-form oracle, 1e-10."""
import numpy as np
import pytest

from oracle import product as P
from paper_2510_07989_gb300.inputs import meshes as MS
from paper_2510_07989_gb300.inputs.assemble import assemble

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [{}, {"fp64_precond": 1}], ids=["plain", "precond"])
def test_fp64_march_of_four_waves(kw):
    from paper_2510_07989_gb300.build import build
    build()
    from paper_2510_07989_gb300 import mot as M
    ops = assemble(MS.torus(1.0, 0.3, 9, 5), 4.0, 1.0, 0.3)
    exc, n = MS.fibonacci_batch(4, ops.dt, w_steps=20, t0_steps=20, r_obj=1.3), 35
    s = M.Solver(ops, **kw)
    W = s.run(exc, n)
    assert s.noconv == 0
    S = P.ProductSystem(ops)
    for b in range(4):
        ref = S.march(exc, n, b=b)
        assert np.abs(W[:, b].reshape(n, -1) - ref).max() < 1e-10 * np.abs(ref).max()
