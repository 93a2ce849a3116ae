"""Workloads of the MOT library as a user's program runs them: single time steps
of a march (the unit of all work), a whole short march, several scatterers
marched together, and the far field of a finished march. Sizes are those of
this repository's benchmark, tests and configurations, or lie between them.

A state is a loaded handle in the middle of its march: enough steps have been
taken that every lag of the history is live, with the pulse's response spread
over the stored lags. One pass of a step case is the next step of that march;
the scatterer is lit by a train of Gaussian pulses, so the march goes on for
as many passes as are asked for. Seeds choose the waves' polarisations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_07989_gb300 import mot as M
from paper_2510_07989_gb300.inputs import meshes as MS
from paper_2510_07989_gb300.inputs.assemble import assemble

QUADRATURE = dict(nq=3, ntheta=3, nrad=3, far_plain=6)  # the benchmark's operator assembly
TUNED = (512, 0.4, 3, 2, 4)  # the history configuration a program stores for a large batch (bench record)


def listed():
    return [
        # the smallest call: one plane wave on the 120-edge sphere, FP64, plain GMRES (latency and launches)
        dict(name="sphere_l1_fp64", mesh="sphere", a=1, b=0, eps=2.0, cdt=0.2, B=1, path="fp64", call="step"),
        # a sphere experiment of the method's paper: 1920 edges, one wave, FP64, plain GMRES on the product form
        dict(name="sphere_l3_fp64", mesh="sphere", a=3, b=0, eps=2.0, cdt=0.5, B=1, path="fp64", call="step"),
        # a non-smooth scatterer with an odd edge count (270) and an odd batch, FP64 with the direct solves
        dict(name="pyramid_fp64_direct", mesh="pyramid", a=3, b=0, eps=5.0, cdt=0.4, B=5, path="fp64_direct",
             call="step"),
        # the FP64 arm of the benchmark (64 waves, Q_0^-1 preconditioner) at a size with the same 53 lags
        dict(name="torus_fp64_batch", mesh="torus", a=18, b=8, eps=4.0, cdt=0.1, B=64, path="fp64_precond",
             call="step"),
        # mixed precision, a batch that is no multiple of 8 (FP32 history on the CUDA cores)
        dict(name="sphere_l2_mixed_b3", mesh="sphere", a=2, b=0, eps=3.0, cdt=0.3, B=3, path="mixed", call="step"),
        # mixed precision, the smallest tensor-core batch, 216 edges (ragged row block), 53 lags
        dict(name="torus_mixed_b8", mesh="torus", a=12, b=6, eps=4.0, cdt=0.1, B=8, path="mixed", call="step"),
        # the non-smooth cube at its configuration's batch of 32, 35 lags
        dict(name="cube_mixed_b32", mesh="cube", a=6, b=0, eps=6.0, cdt=0.25, B=32, path="mixed", call="step"),
        # the benchmark's batched mixed step on a smaller torus (924 edges), the library's default configuration
        dict(name="torus_mixed_b64", mesh="torus", a=28, b=11, eps=4.0, cdt=0.1, B=64, path="mixed", call="step"),
        # the same, the largest scatterer here (1512 edges), with a stored history configuration
        dict(name="torus_large_mixed_b64", mesh="torus", a=36, b=14, eps=4.0, cdt=0.1, B=64, path="mixed_set",
             call="step"),
        # a whole march from rest with every step kept on the device: partial histories and the restart
        dict(name="sphere_l2_mixed_march", mesh="sphere", a=2, b=0, eps=3.0, cdt=0.3, B=16, path="mixed",
             call="march"),
        # scatterers of uneven size marched together, four steps a call
        dict(name="uneven_mixed_many", mesh="uneven", a=5, b=0, eps=0.0, cdt=0.2, B=16, path="mixed", call="many"),
        # the results of a march: recovered currents and the bistatic far field at three frequencies
        dict(name="sphere_l2_fields", mesh="sphere", a=2, b=0, eps=3.0, cdt=0.3, B=8, path="fp64_precond", call="fields"),
    ]


def draw(rng):
    path = rng.choice(["fp64", "fp64_precond", "fp64_direct", "mixed", "mixed", "mixed", "mixed_set"])
    call = rng.choice(["step", "step", "step", "step", "march" if path == "mixed" else "fields"])
    kind = rng.choice(["torus", "torus", "cube", "sphere", "ellipsoid", "pyramid"])
    if path == "mixed_set":
        call = "step"
    if call == "fields":
        path = "fp64_precond"
    lo, hi = (120, 480) if path.startswith("fp64") else (216, 1000 if call == "step" else 600)
    edges = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    a, b = 0, 0
    if kind == "torus":
        b = rng.randint(5, 12)
        a = max(6, round(edges / (3 * b)))
        eps, cdt = 4.0, round(rng.uniform(0.1, 0.3), 3)
    elif kind == "cube":
        a = max(3, round(math.sqrt(edges / 18)))
        eps, cdt = 6.0, round(rng.uniform(0.25, 0.6), 3)
    elif kind == "sphere":
        a = 1 if edges < 240 else 2
        eps, cdt = round(rng.uniform(1.5, 4.0), 3), round(rng.uniform(0.2, 0.6), 3)
    elif kind == "ellipsoid":
        a, b = max(3, round(math.sqrt(edges / 30))), rng.randrange(1000)
        eps, cdt = round(rng.uniform(1.5, 8.0), 3), round(rng.uniform(0.2, 0.5), 3)
    else:
        a = max(2, round(math.sqrt(edges / 30)))
        eps, cdt = 5.0, round(rng.uniform(0.2, 0.4), 3)
    if path in ("fp64", "fp64_direct"):
        cdt = round(3.0 * cdt, 3)  # the plain FP64 experiments take few lags
    if path == "mixed":
        B = rng.choice([1, 3, 5, 8, 16, 24, 32, 48, 64])
    elif path == "mixed_set":
        B = rng.choice([16, 32, 40, 64])
    else:
        B = round(math.exp(rng.uniform(0.0, math.log(16))))
    return dict(mesh=kind, a=a, b=b, eps=eps, cdt=cdt, B=B, path=path, call=call)


# ---------------------------------------------------------------------------------------------
# what a program has in hand
# ---------------------------------------------------------------------------------------------

_OPS = {}  # operators of the scatterers met so far (host): they do not depend on the seed


def _mesh(kind, a, b):
    if kind == "sphere":
        return MS.icosphere(a)
    if kind == "torus":
        return MS.torus(1.0, 0.3, a, b)
    if kind == "cube":
        return MS.cube(2.0, a)
    if kind == "pyramid":
        return MS.star_pyramid(m=a)
    g = np.random.default_rng(b)
    axes = g.uniform(0.5, 1.5, size=3)
    q, r = np.linalg.qr(g.standard_normal((3, 3)))
    q = q * np.sign(np.diag(r))[None, :]
    if np.linalg.det(q) < 0:
        q[:, 0] = -q[:, 0]
    return MS.ellipsoid(a, axes, q)


def _operators(case):
    """One Operators object per scatterer of the case."""
    key = (case["mesh"], case["a"], case["b"], case["eps"], case["cdt"])
    if key not in _OPS:
        if case["mesh"] == "uneven":
            # the smaller members of the benchmark's uneven batch
            specs = sorted(MS.uneven_batch(24), key=lambda s: s[0].ne)[:case["a"]]
        else:
            specs = [(_mesh(case["mesh"], case["a"], case["b"]), case["eps"])]
        _OPS[key] = [assemble(m, e, 1.0, case["cdt"], **QUADRATURE) for m, e in specs]
    return _OPS[key]


def _span(ops):
    """Steps the pulse's response is spread over: the stored lags, at least 8."""
    return max(ops.kmax + 1, 8)


def _excitation(ops, case, seed, i):
    n = _span(ops)
    r = float(np.linalg.norm(ops.mesh.verts, axis=1).max())
    return MS.fibonacci_batch(case["B"], case["cdt"], seed=seed + 1000 * i, w_steps=float(n), t0_steps=0.6 * n, r_obj=r)


def _options(case):
    return {"fp64": dict(precision=M.MOT_PREC_FP64), "fp64_direct": dict(precision=M.MOT_PREC_FP64, fp64_direct=1),
            "fp64_precond": dict(precision=M.MOT_PREC_FP64, fp64_precond=1),
            "mixed": dict(precision=M.MOT_PREC_MIXED), "mixed_set": dict(precision=M.MOT_PREC_MIXED)}[case["path"]]


FREQUENCIES = (0.5, 1.0, 1.5)  # angular, of the far-field case
DIRECTIONS = 181
MANY_STEPS = 4


def _directions():
    """A bistatic cut, every two degrees of a full circle in the x-z plane."""
    t = np.linspace(0.0, 2 * np.pi, DIRECTIONS)
    return np.stack([np.sin(t), np.zeros_like(t), np.cos(t)], axis=1)


class _Scatterer:
    """A handle with its waves; next_pulse() lights it again once a pulse has passed."""

    def __init__(self, ops, case, seed, i):
        self.ops, self.B = ops, case["B"]
        self.solver = M.Solver(ops, **_options(case))
        self.h = self.solver.h
        self.waves = M.mot_waves(_excitation(ops, case, seed, i))
        self.period = 3 * _span(ops)
        self.step, self.pulse_end = 0, self.period
        if case["call"] == "fields":
            M.mot_set_frequencies(self.h, FREQUENCIES)

    def advance(self, n):
        """n more steps are being taken: later ones may belong to the next pulse of the train."""
        self.step += n
        if self.step > self.pulse_end:
            for w in self.waves:
                w.t0 += self.period * self.ops.dt
                w.t_trunc += self.period * self.ops.dt
            self.pulse_end += self.period

    def out(self, *lead):
        return torch.empty(*lead, self.B, 2, self.ops.ne, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    ops = _operators(case)
    s = dict(case=case, sc=[_Scatterer(o, case, seed, i) for i, o in enumerate(ops)])
    one = s["sc"][0]
    mixed = case["path"].startswith("mixed")
    s["narrow"] = mixed
    if case["call"] == "march":
        s["n"] = 2 * _span(one.ops)
        s["out"] = one.out(s["n"])
    elif case["call"] == "many":
        n = max(_span(x.ops) for x in s["sc"]) + 2
        M.mot_run_many([x.h for x in s["sc"]], n, [x.waves for x in s["sc"]], [x.B for x in s["sc"]])
        for x in s["sc"]:
            x.advance(n)
        s["out"] = [x.out(MANY_STEPS) for x in s["sc"]]
    else:
        n = _span(one.ops) + 2
        M.mot_run(one.h, n, one.waves, one.B)
        one.advance(n)
        s["out"] = one.out()
        if case["path"] == "mixed_set":
            M.mot_set_tc_config(one.h, *TUNED)
        if case["call"] == "fields":
            s["out"] = torch.empty(one.B, 4, one.ops.ne, dtype=torch.float64, device="cuda")
            s["dirs"] = _directions()
    return s


def _kept(s, w):
    """The record of a step that the program keeps: the mixed path resolves w_i to
    single precision (1e-6 of the march's peak), so it is stored as that."""
    return w.float() if s["narrow"] else w


def run(s):
    call, one = s["case"]["call"], s["sc"][0]
    if call == "step":
        one.advance(1)
        M.mot_step(one.h, one.waves, one.B, s["out"])
        return _kept(s, s["out"])
    if call == "march":
        M.mot_reset(one.h)
        M.mot_run(one.h, s["n"], one.waves, one.B, s["out"])
        return _kept(s, s["out"])
    if call == "many":
        for x in s["sc"]:
            x.advance(MANY_STEPS)
        M.mot_run_many([x.h for x in s["sc"]], MANY_STEPS, [x.waves for x in s["sc"]], [x.B for x in s["sc"]], s["out"])
        return [_kept(s, w) for w in s["out"]]
    M.mot_get_currents(one.h, s["out"])
    E = M.mot_fields(one.h, one.waves, s["dirs"], len(FREQUENCIES), one.B)
    return {"currents": s["out"], "far_field": E}


# ---------------------------------------------------------------------------------------------
# work of a pass: operators, coefficients and results once each
# ---------------------------------------------------------------------------------------------


def work(case):
    total = dict(bytes=0.0, flops=0.0)
    for ops in _operators(case):
        ne, B, K = ops.ne, case["B"], ops.kmax + 1
        if case["call"] == "fields":
            # currents (read, written), Fourier sums, quadrature points; one phase and 24 multiply-adds per sample
            nq, nf = ops.rwg.x.shape[1], len(FREQUENCIES)
            total["bytes"] += 8.0 * (2 * 4 * ne * B + 8 * nf * ne * B + 6 * nq * ne + 6 * B * nf * DIRECTIONS)
            total["flops"] += 2.0 * 12 * ne * nq * nf * DIRECTIONS * B
            continue
        v = 4.0 if case["path"].startswith("mixed") else 8.0
        nnz = uses = 0
        for name, m in ops.mats.items():
            n = int(np.minimum(m.cnt, np.maximum(m.k0 + m.cnt - 1, 0)).sum())  # stored values at lags >= 1
            if m.ta is not None:
                n += int(((m.ta >= 1) & (m.ta <= ops.kmax - 1) & (m.tc != 0)).sum())
            nnz += n
            uses += n * (2 if name[0] == "A" else 1)
        # history operators and coefficients, the static dense operators, w_i; then the lag sum and the two dense products
        step_bytes = v * (nnz + 4.0 * ne * B * K + 2.0 * ne * ne) + 8.0 * 2 * ne * B
        step_flops = 2.0 * uses * 2 * B + 2.0 * 2 * ne * ne * 2 * B
        n, depth = 1, 1.0
        if case["call"] == "many":
            n = MANY_STEPS
        elif case["call"] == "march":
            n = 2 * _span(ops)
            depth = 1.0 - 0.5 * K / n  # the first K steps see a growing history
        total["bytes"] += n * depth * step_bytes
        total["flops"] += n * depth * step_flops
    return total


# ---------------------------------------------------------------------------------------------
# the same outputs in 64 bits, from the definition, with torch's dense algebra
# ---------------------------------------------------------------------------------------------


class _Dense:
    """Q_0 w_i = r_i - sum_k Q_k w_{i-k} in product form with dense FP64 matrices on the GPU."""

    def __init__(self, ops):
        self.ops, ne, mesh = ops, ops.ne, ops.mesh
        self.ne = ne
        f = dict(dtype=torch.float64, device="cuda")
        eye = torch.eye(ne, **f)

        def incidence(plus, minus, n):
            D = torch.zeros(ne, n, **f)
            r = torch.arange(ne, device="cuda")
            D[r, torch.as_tensor(np.asarray(plus, dtype=np.int64), device="cuda")] += 1.0
            D[r, torch.as_tensor(np.asarray(minus, dtype=np.int64), device="cuda")] -= 1.0
            # projector onto the range of D: D (D^T D)^+ D^T, the null space of D^T D being the constants
            J = torch.full((n, n), 1.0 / n, **f)
            return D @ torch.linalg.solve(D.T @ D + J, D.T)

        self.PS = incidence(mesh.ef[:, 0], mesh.ef[:, 1], mesh.nf)
        PL = incidence(mesh.ev[:, 1], mesh.ev[:, 0], mesh.nv)
        G = torch.as_tensor(ops.G.toarray(), **f)
        Ginv = torch.linalg.inv(G)
        PSH = eye - PL
        self.M1 = PSH @ torch.as_tensor(ops.T0s, **f) @ PSH @ Ginv
        self.M2 = PL @ torch.as_tensor(ops.T0h, **f) @ PL @ Ginv @ (eye - self.PS)
        self.lim = {"A": ops.kmax, "H": ops.kmax + 1, "T": ops.kmax - 1}
        self.Z = {fam: self._family(fam) for fam in self.lim}
        Q0 = torch.empty(2 * ne, 2 * ne, **f)
        for c in range(0, 2 * ne, 512):
            w = torch.zeros(2, ne, min(512, 2 * ne - c), **f)
            w.view(2 * ne, -1)[torch.arange(c, c + w.shape[2], device="cuda"), torch.arange(w.shape[2], device="cuda")] = 1
            Q0[:, c:c + w.shape[2]] = self.left(*self.sums([self.split(w)], 0)).reshape(2 * ne, -1)
        self.lu = torch.linalg.lu_factor(Q0)

    def _family(self, fam):
        """Per lag (eta T + eta' T', T/eta + T'/eta', K + K')."""
        o, ne, lim = self.ops, self.ne, self.lim[fam]
        Z = torch.zeros(3, lim + 1, ne * ne, dtype=torch.float64, device="cuda")
        for name, uses in ((fam + "T", ((0, o.eta), (1, 1 / o.eta))), (fam + "Tp", ((0, o.etap), (1, 1 / o.etap))),
                           (fam + "K", ((2, 1.0),)), (fam + "Kp", ((2, 1.0),))):
            m = o.mats[name]
            t = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
            rows = torch.repeat_interleave(torch.arange(ne, device="cuda"), t(np.diff(m.rowptr)))
            place = rows * ne + t(m.col).long()
            k0, cnt, voff, val = t(m.k0).long(), t(m.cnt).long(), t(m.voff), t(m.val)
            for k in range(lim + 1):
                e = torch.nonzero((k0 <= k) & (k < k0 + cnt)).reshape(-1)
                for j, c in uses:
                    Z[j, k].index_add_(0, place[e], c * val[voff[e] + k - k0[e]])
                if m.ta is not None and k <= o.kmax - 1:
                    e = torch.nonzero((t(m.ta) <= k) & ~((k0 <= k) & (k < k0 + cnt))).reshape(-1)
                    for j, c in uses:
                        Z[j, k].index_add_(0, place[e], c * t(m.tc)[e])
        return Z.view(3, lim + 1, ne, ne)

    def split(self, w):
        sg = torch.matmul(self.PS, w)
        return w - sg, sg

    def sums(self, past, first):
        """s1 = sum A_k l + A^_k s, s2 = sum A~_k l + A_k s over past[j] = (l, s) of lag first + j."""
        s1 = torch.zeros_like(past[0][0]) if past else None
        s2 = torch.zeros_like(s1) if past else None
        for j, (l, sg) in enumerate(past):
            k = first + j
            for fam, x, s in (("A", l, s1), ("H", sg, s1), ("T", l, s2), ("A", sg, s2)):
                if k <= self.lim[fam]:
                    Zu, Zv, Zk = self.Z[fam][:, k]
                    s[0] += Zu @ x[0] - Zk @ x[1]
                    s[1] += Zk @ x[0] + Zv @ x[1]
        return s1, s2

    def left(self, y1, y2):
        return torch.matmul(self.M1, y1) + torch.matmul(self.M2, y2)

    def rhs(self, exc, i):
        o = self.ops
        f = dict(dtype=torch.float64, device="cuda")
        t = lambda a: torch.as_tensor(a, **f)  # noqa: E731
        x, wf = t(o.rwg.x), t(o.rwg.wf)
        A, p, k, w, t0 = t(exc.A), t(exc.p), t(exc.k), t(exc.w), t(exc.t0)
        g = lambda ti: A / (2 * o.c) * (1 + torch.erf(4 / w * (o.c * (ti - t0) - x @ k.T)))  # noqa: E731  [ne, nq, B]
        now, before = g(i * o.dt), g((i - 1) * o.dt)

        def test(s):
            F = torch.einsum("eqd,eqb->ebd", wf, s)
            return -torch.stack([(F * p).sum(-1), (F * (torch.linalg.cross(k, p) / o.eta)).sum(-1)])

        on = (i * o.dt <= t(exc.t_trunc)).double()
        return test(now - before) / o.dt, test(now) / o.tmax * on

    def march(self, exc, n):
        """w_1 .. w_n, each [2][ne][B], and their loop and star parts."""
        W, parts = [], []
        for i in range(1, n + 1):
            y1, y2 = self.rhs(exc, i)
            past = parts[::-1][:self.ops.kmax + 1]
            if past:
                s1, s2 = self.sums(past, 1)
                y1, y2 = y1 - s1, y2 - s2
            b = self.left(y1, y2)
            w = torch.linalg.lu_solve(*self.lu, b.reshape(2 * self.ne, -1)).reshape(b.shape)
            W.append(w)
            parts.append(self.split(w))
        return W, parts


def _fields(d, exc, parts):
    """Recovered currents of the last step and the far field of the whole march."""
    o, ne = d.ops, d.ne
    f = dict(dtype=torch.float64, device="cuda")
    w = torch.as_tensor(FREQUENCIES, **f)
    c = o.tmax / o.dt
    zero = torch.zeros_like(parts[0][1])
    sums = torch.zeros(len(FREQUENCIES), 2, ne, exc.B, dtype=torch.complex128, device="cuda")
    for i, (l, sg) in enumerate(parts, 1):
        before = parts[i - 2][1] if i > 1 else zero
        cur = (l, c * (sg - before))
        weight = torch.exp(-1j * w * i * o.dt) * (torch.exp(1j * w * o.dt) - 1) / (1j * w)
        sums += weight[:, None, None, None] * (cur[0] + cur[1])
    currents = torch.stack([cur[0][0], cur[1][0], cur[0][1], cur[1][1]]).permute(2, 0, 1)
    x, wf = torch.as_tensor(o.rwg.x, **f), torch.as_tensor(o.rwg.wf, **f)
    dirs = torch.as_tensor(_directions(), **f)
    E = torch.empty(exc.B, len(FREQUENCIES), DIRECTIONS, 3, dtype=torch.complex128, device="cuda")
    for q, om in enumerate(FREQUENCIES):
        k = om / o.c
        ph = torch.einsum("eqd,eqr->red", wf.to(torch.complex128), torch.exp(1j * k * (x @ dirs.T)))
        N = torch.einsum("red,eb->brd", ph, sums[q, 0])
        L = torch.einsum("red,eb->brd", ph, sums[q, 1])
        r = dirs.to(torch.complex128)[None].expand_as(N)
        far = o.eta * torch.linalg.cross(r, torch.linalg.cross(r, N)) + torch.linalg.cross(r, L)
        A, wp, t0 = (torch.as_tensor(a, **f) for a in (exc.A, exc.w, exc.t0))
        spec = A / o.c * torch.exp(-1j * om * t0) * torch.exp(-(om * wp / (8 * o.c)) ** 2)
        E[:, q] = 1j * k / (4 * math.pi) * far / spec[:, None, None]
    return {"currents": currents.contiguous(), "far_field": E.cpu().numpy()}


def exact(case, seed):
    outs = []
    every = _operators(case)
    if sum((o.kmax + 2.0) ** 2 * o.ne ** 2 * case["B"] for o in every) > 6e11:
        return None  # over 20 seconds
    for i, o in enumerate(every):
        d, exc = _Dense(o), _excitation(o, case, seed, i)
        if case["call"] == "many":
            n, keep = max(_span(x) for x in every) + 2 + MANY_STEPS, MANY_STEPS
        elif case["call"] == "march":
            n = keep = 2 * _span(o)
        else:
            n, keep = _span(o) + 3 - (case["call"] == "fields"), 1
        W, parts = d.march(exc, n)
        if case["call"] == "fields":
            return _fields(d, exc, parts)
        outs.append(torch.stack([w.permute(2, 0, 1) for w in W[-keep:]]))
        del d, W, parts
    return outs if case["call"] == "many" else outs[0] if case["call"] == "march" else outs[0][0]
