"""Device memory of a handle: what mot_get_info reports is what the handle
holds -- the march state goes with mot_reset, and marching again after it
takes the same memory as before, on every path."""
from contextlib import contextmanager, nullcontext

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


@contextmanager
def only(free):
    """Device memory taken meanwhile so that about `free` bytes are left."""
    import torch
    held = torch.empty(max(0, torch.cuda.mem_get_info()[0] - int(free)), dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del held
        torch.cuda.empty_cache()


@pytest.mark.parametrize("kw", [{}, {"precision": 1}], ids=["fp64", "mixed"])
def test_march_after_a_refused_state(M, ops, kw):
    """A step that finds no memory for its state (half of it is there) says so and
    leaves a handle that marches once there is: the same steps as any other."""
    exc = MS.fibonacci_batch(64, ops.dt, w_steps=20, t0_steps=20, r_obj=1.3)
    s = M.Solver(ops, **kw)
    loaded = s.info()["device_bytes"]
    ref = s.run(exc, 3)
    state = s.info()["device_bytes"] - loaded
    M.mot_reset(s.h)
    t = M.Solver(ops, **kw)
    with only(state / 2):
        for _ in range(2):
            with pytest.raises(M.MotError) as e:
                t.run(exc, 1)
            assert e.value.code == M.MOT_EOOM
    assert np.array_equal(t.run(exc, 3), ref)


@pytest.fixture(scope="module")
def larger():
    return assemble(MS.torus(1.0, 0.3, 36, 12), 4.0, 1.0, 0.3)  # 1296 edges: dense Q_0 of 55 MB


@pytest.mark.parametrize("kw,when", [({}, "load"), ({}, "state"), ({"fp64_precond": 1}, "state")],
                         ids=["plain-load", "plain-state", "precond-state"])
def test_march_where_the_dense_operators_do_not_fit(M, larger, kw, when):
    """A march that fits without the operators it can do without runs without
    them: not formed at the load, or given back at its first step. Two ways to the
    same solution, to the 1e-10 of the FP64 path."""
    ops, B, n = larger, 16, 3
    exc = MS.fibonacci_batch(B, ops.dt, w_steps=20, t0_steps=4, r_obj=1.3)
    s = M.Solver(ops, **kw)
    loaded = s.info()["device_bytes"]
    ref = s.run(exc, n)
    state = s.info()["device_bytes"] - loaded
    M.mot_destroy(s.h)
    q0 = 8 * (2 * ((ops.ne + 31) // 32 * 32)) ** 2
    with only(loaded - 0.5 * q0) if when == "load" else nullcontext():
        t = M.Solver(ops, **kw)
    assert (t.info()["device_bytes"] < loaded - q0) == (when == "load")
    with only(state - 0.3 * q0) if when == "state" else nullcontext():
        W = t.run(exc, n)
    assert t.info()["device_bytes"] < loaded + state - q0
    assert t.noconv == 0
    assert np.abs(W - ref).max() < 1e-10 * np.abs(ref).max()


def test_mixed_handle_holds_what_its_march_reads(M, larger):
    """The FP32 history without tensor cores or preconditioner: dense Q_0 and
    [M1 | M2] in both precisions, T_0, tiles, column orders and the face inverse, and
    beside them the split workspace (64 x 32 tiles of doubles, four CTAs per SM), 32
    bytes a tile for the task lists and a megabyte of tables: no Gram inverse (7.2 MB),
    which only the load needs."""
    import torch
    ops = larger
    s = M.Solver(ops, precision=M.MOT_PREC_MIXED, mixed_flags=M.MOT_MIX_HIST32 | M.MOT_MIX_Q032)
    q = s.info()
    n, f = (ops.ne + 31) // 32 * 32, (ops.mesh.nf + 63) // 64 * 64
    dense = 12 * (2 * n) ** 2 + 12 * n * 2 * n + 2 * 8 * n ** 2 + 4 * f ** 2
    tiles = (4 * 1024 + 32) * q["tile_count"] + 4 * n * (n // 32)
    split = 4 * torch.cuda.get_device_properties(0).multi_processor_count * 64 * 32 * 8
    assert dense < q["device_bytes"] < dense + tiles + split + (1 << 20)
