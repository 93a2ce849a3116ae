"""Device memory of a handle: what mot_get_info reports is what the handle
holds -- the march state goes with mot_reset, and marching again after it
takes the same memory as before, on every path."""
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


PATHS = [{}, {"fp64_precond": 1}, {"fp64_direct": 1}, {"precision": 1}]


@pytest.mark.parametrize("kw", PATHS, ids=lambda k: "-".join(k) or "plain")
def test_device_bytes_over_resets(M, ops, kw):
    s = M.Solver(ops, **kw)
    M.mot_set_frequencies(s.h, np.array([0.5]))
    loaded, seen = s.info()["device_bytes"], []
    for B in (16, 3, 16, 3):
        s.run(MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=20, r_obj=1.3), 3, keep=False)
        seen.append(s.info()["device_bytes"])
        M.mot_reset(s.h)
        assert s.info()["device_bytes"] >= loaded
        seen.append(s.info()["device_bytes"])
    # from the first reset on only buffers that outlive a march stay; none grows in the second pair
    assert seen[4:] == [seen[4], seen[3], seen[6], seen[3]]
    assert seen[4] > seen[6] > seen[3]
