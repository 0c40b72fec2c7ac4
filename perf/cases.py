"""Timed cases of the projection library: what its users call, over the sizes they call it with.

A planner on a constraint manifold spends its time in the calls below: batches
of configurations projected and collision-checked, uneven interpolation
segments, whole ParallelConstrainedExtend steps, the adjoint of the projection
for gradient-based optimisation, path shortening, and the check alone.  Robots,
constraints and obstacles are those of ``paper_2604_13323_gb300.workloads``;
the batches are drawn on the GPU from a seed with the distributions of those
workloads.  The launch shape is left at its default (autotuning is optional).

``exact`` repeats each computation in 64 bits in plain torch: forward
kinematics, residuals, Jacobians and the damped Newton iteration are written
out here a second time, independently of the library.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2604_13323_gb300 import mcproj, shorten
from paper_2604_13323_gb300 import workloads as W

DEV = "cuda"

# Newton steps per start (means over the workloads) and flops of one step, of
# one residual evaluation and of one collision check, multiplications by
# structural zeros not counted (sin / cos not counted either).
STEPS = {"humanoid": 4.7, "humanoid_hull": 4.7, "arm": 4.3, "tray": 4.0, "peg": 4.0, "tsr": 4.0, "dual": 5.5,
         "rod": 3.5, "sphere": 1.5}
STEP_FLOPS = {"humanoid": 13301, "humanoid_hull": 13301, "arm": 253, "tray": 400, "peg": 500, "tsr": 1100, "dual": 2545,
              "rod": 1100, "sphere": 20}
EVAL_FLOPS = {"humanoid": 1426, "humanoid_hull": 1426, "arm": 122, "tray": 190, "peg": 200, "tsr": 250, "dual": 421,
              "rod": 400, "sphere": 8}
CHECK_FLOPS = {"humanoid": 13700, "humanoid_hull": 13700, "arm": 1523, "tray": 1523, "peg": 1523, "tsr": 1523,
               "dual": 3500, "rod": 3500, "sphere": 80}
DOF = {"humanoid": 36, "humanoid_hull": 36, "arm": 7, "tray": 7, "peg": 7, "tsr": 7, "dual": 14, "rod": 14, "sphere": 3}
SEGMENT_LENGTHS = (2, 200)   # points of one interpolation segment


def listed():
    return [
        # the whole-body planner's bulk work: a million sampled stances projected and checked
        {"name": "humanoid_1048576", "call": "project_check", "problem": "humanoid", "n": 1048576},
        # one planning iteration of the humanoid: the frontier's samples, a ragged batch
        {"name": "humanoid_4099", "call": "project_check", "problem": "humanoid", "n": 4099},
        # the smallest humanoid call: the points of one edge, inside a control loop
        {"name": "humanoid_32", "call": "project", "problem": "humanoid", "n": 32},
        # a manipulator's sampled batch, end effector kept upright
        {"name": "arm_65536", "call": "project_check", "problem": "arm", "n": 65536},
        # one tree extension of a manipulator's planner: latency and launches
        {"name": "arm_257", "call": "project_check", "problem": "arm", "n": 257},
        # a bounded task-space region: inequality constraints switch rows on and off
        {"name": "tsr_8195", "call": "project_check", "problem": "tsr", "n": 8195},
        # the bimanual planner's interpolated edges, lengths 2 to 200 in one call
        {"name": "dual_segments_262144", "call": "segments", "problem": "dual", "n": 262144},
        # whole constrained extensions (steer, particles, interpolation, bisection, collision)
        {"name": "dual_extend_16384", "call": "extend", "problem": "dual", "n": 16384, "particles": 8},
        # the backward direction: adjoints of the projection at points on the manifold
        {"name": "dual_vjp_65536", "call": "vjp", "problem": "dual", "n": 65536},
        # one descent step of path shortening: projection, length, backward, waypoint step
        {"name": "dual_shorten_4096x64", "call": "shorten", "problem": "dual", "n": 4096, "way": 64},
        # the FP64 path: geodesics on the unit sphere in double precision
        {"name": "sphere_fp64_28672", "call": "segments", "problem": "sphere", "n": 28672},
        # validation of already projected configurations: the collision check alone
        {"name": "humanoid_check_262147", "call": "check", "problem": "humanoid", "n": 262147},
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi], half of them odd."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, n if rng.random() < 0.5 else n | 1))


def draw(rng):
    pick = rng.random()
    if pick < 0.30:
        return {"call": rng.choice(["project_check", "project"]), "problem": rng.choice(["humanoid", "humanoid", "humanoid_hull"]),
                "n": _size(rng, 32, 524288)}
    if pick < 0.50:
        return {"call": rng.choice(["project_check", "project"]), "problem": rng.choice(["arm", "tray", "peg", "tsr"]),
                "n": _size(rng, 64, 262144)}
    if pick < 0.58:
        return {"call": "project_check", "problem": rng.choice(["dual", "rod"]), "n": _size(rng, 64, 262144),
                "cyclic": rng.random() < 0.25}
    if pick < 0.68:
        return {"call": "segments", "problem": "dual", "n": _size(rng, 1024, 262144)}
    if pick < 0.76:
        return {"call": "extend", "problem": "dual", "n": _size(rng, 64, 16384), "particles": rng.choice([4, 8, 8, 16])}
    if pick < 0.83:
        return {"call": "vjp", "problem": rng.choice(["dual", "arm"]), "n": _size(rng, 256, 262144)}
    if pick < 0.89:
        return {"call": "shorten", "problem": "dual", "n": _size(rng, 16, 4096), "way": rng.randint(16, 64)}
    if pick < 0.95:
        return {"call": "check", "problem": rng.choice(["humanoid", "arm", "dual"]), "n": _size(rng, 256, 524288)}
    return {"call": "project", "problem": rng.choice(["arm", "dual", "humanoid"]), "n": _size(rng, 64, 32768), "fp64": True}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _workload(case):
    p = case["problem"]
    if p in ("humanoid", "humanoid_hull"):
        wl = W.humanoid_workload(n=1, hull=p == "humanoid_hull")
    elif p == "arm":
        wl = W.arm_workload(n=1)
    elif p in ("tray", "peg", "tsr"):
        wl = W.arm_task_workload(p, n=1)
    elif p == "rod":
        wl = W.dual_rod_workload(n=1)
    elif p == "sphere":
        wl = W.sphere_workload(n_pairs=1)
    elif case["call"] == "extend":
        wl = W.extend_workload(n_ext=1, n=case["particles"])
    else:
        wl = W.dual_arm_workload(total=10)
    if case.get("fp64"):
        wl.params = dataclasses.replace(wl.params, precision=W.PREC_FP64)
    if case.get("cyclic"):
        wl.params = dataclasses.replace(wl.params, cyclic=True)
    return wl


class _Rand:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=torch.float64)

    def uniform(self, lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, generator=self.g, device=DEV, dtype=torch.float64)


def _starts(case, wl, n, rnd):
    """[d, n] start configurations with the workload's distribution."""
    p = case["problem"]
    if p in ("humanoid", "humanoid_hull"):
        sigma = torch.tensor(np.where(wl.robot.type == W.PRISMATIC, 0.05, 0.3), device=DEV)
        return torch.tensor(wl.extra["q_nom"], device=DEV)[:, None] + sigma[:, None] * rnd.normal(36, n)
    if p == "arm":
        return rnd.uniform(-2.8, 2.8, 7, n)
    q_ref = torch.tensor(wl.extra["q_ref"], device=DEV)
    return q_ref[:, None] + 0.3 * rnd.normal(DOF[p], n)


def _inputs(case, seed):
    """The user's arrays (and the workload that goes with them)."""
    wl = _workload(case)
    rnd = _Rand(seed)
    call, n = case["call"], case["n"]
    f = torch.float64 if wl.params.precision == W.PREC_FP64 else torch.float32
    x = {}
    if call in ("project", "project_check"):
        x["q"] = _starts(case, wl, n, rnd).to(f)
    elif call == "check":   # what gets checked are projected configurations: near the manifold, not uniform
        q = _starts(case, wl, n, rnd)
        x["q"] = _reference(wl).project(q, steps=2)[0].to(f)
    elif call == "vjp":
        x["q"] = _reference(wl).project(_starts(case, wl, n, rnd))[0].to(f)
        x["g"] = rnd.normal(wl.dof, n).to(f)
    elif call == "segments":
        lens = np.random.default_rng(seed)
        if case["problem"] == "sphere":
            # geodesics between random points, spaced at most 0.05 apart; about 28 points each
            m = n // 16 + 8
            a, b = (torch.nn.functional.normalize(rnd.normal(3, m), dim=0) for _ in range(2))
            length = torch.ceil((b - a).norm(dim=0) / 0.05).to(torch.int32) + 1
            x["delta"] = ((b - a) / (length - 1).clamp(min=1)).to(f)
            m = int((length.cumsum(0) < n).sum()) + 1   # the last one ends after n points in all
            length[m - 1] -= int(length[:m].sum()) - n
            x["start"], x["delta"], x["length"] = a[:, :m].to(f).contiguous(), x["delta"][:, :m].contiguous(), length[:m].contiguous()
            x["total"] = n
        else:
            length, acc = [], 0
            while acc < n:   # the last one ends after n points in all
                length.append(min(int(lens.integers(SEGMENT_LENGTHS[0], SEGMENT_LENGTHS[1] + 1)), n - acc))
                acc += length[-1]
            m = len(length)
            raw = torch.tensor(wl.extra["q_ref"], device=DEV)[:, None] + 0.2 * rnd.normal(wl.dof, m)
            x["start"] = _reference(wl).project(raw)[0].to(f)
            x["delta"] = (0.05 * torch.nn.functional.normalize(rnd.normal(wl.dof, m), dim=0)).to(f)
            x["length"] = torch.tensor(length, dtype=torch.int32, device=DEV)
            x["total"] = acc
    elif call == "extend":
        q_ref = torch.tensor(wl.extra["q_ref"], device=DEV)[:, None]
        x["q_s"] = _reference(wl).project(q_ref + 0.2 * rnd.normal(wl.dof, n))[0].to(f)
        x["q_t"] = (q_ref + rnd.uniform(-1.0, 1.0, wl.dof, n)).to(f)
        x["eps"] = (0.05 * rnd.normal(case["particles"], n)).to(f)
    elif call == "shorten":
        q_ref = torch.tensor(wl.extra["q_ref"], device=DEV)[:, None]
        ref = _reference(wl)
        a, b = (ref.project(q_ref + 0.3 * rnd.normal(wl.dof, n))[0] for _ in range(2))
        t = torch.linspace(0.0, 1.0, case["way"], device=DEV, dtype=torch.float64)
        noise = 0.05 * rnd.normal(wl.dof, n, case["way"])
        noise[:, :, 0] = noise[:, :, -1] = 0.0
        Q = a[:, :, None] + (b - a)[:, :, None] * t + noise
        x["Q"] = Q.reshape(wl.dof, -1).to(f).contiguous()
    return wl, x


def prepare(case, seed):
    wl, x = _inputs(case, seed)
    x["case"], x["params"], x["workload"] = case, wl.params, wl
    x["P"] = mcproj.Projector(wl.robot, wl.constraints, wl.obstacles)
    return x


def run(s):
    P, p, call = s["P"], s["params"], s["case"]["call"]
    if call == "project_check":
        return P.project_check(s["q"], p)
    if call == "project":
        return P.project(s["q"], p)
    if call == "check":
        return P.check(s["q"])
    if call == "vjp":
        return P.vjp(s["q"], s["g"])
    if call == "segments":
        return P.project_segments(s["start"], s["delta"], s["length"], p, total=s["total"])
    if call == "extend":
        e = s["workload"].extra
        return P.extend(s["q_s"], s["q_t"], s["eps"], p, e["r"], e["delta"])
    n, way = s["case"]["n"], s["case"]["way"]
    Qv = s["Q"].detach().requires_grad_(True)
    Qs = shorten.ProjectFn.apply(Qv, P, p)
    L = shorten.PathLengthFn.apply(Qs, P, n, way)
    L.sum().backward()
    Q = Qs.detach().clone()
    P.path_step(Q, Qv.grad, n, way, 0.1, 0.05)
    return {"Q": Q, "length": L.detach(), "grad": Qv.grad}


def work(case):
    p, n, d, call = case["problem"], case["n"], DOF[case["problem"]], case["call"]
    w = 8 if case.get("fp64") or p == "sphere" else 4
    proj = STEPS[p] * STEP_FLOPS[p] + 2 * EVAL_FLOPS[p]
    if call in ("project", "project_check"):
        check = call == "project_check"
        return {"bytes": n * (2 * d * w + 10 + check), "flops": n * (proj + check * CHECK_FLOPS[p])}
    if call == "segments":
        return {"bytes": n * (d * w + 10), "flops": n * proj}
    if call == "check":
        return {"bytes": n * (d * w + 1), "flops": n * CHECK_FLOPS[p]}
    if call == "vjp":
        return {"bytes": n * (3 * d * w + 1), "flops": n * STEP_FLOPS[p]}
    if call == "extend":   # the particles, and about ten validated points per extension
        points = case["particles"] + 10
        return {"bytes": n * (3 * d * w + case["particles"] * w + 9), "flops": n * (points * proj + 10 * CHECK_FLOPS[p])}
    m = n * case["way"]    # shortening: projection, adjoint, length gradient and step
    return {"bytes": m * 3 * d * w, "flops": m * (proj + STEP_FLOPS[p] + 8 * d)}


# ---------------------------------------------------------------------------
# The same computations in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _se3(x):
    m = torch.as_tensor(np.asarray(x, dtype=np.float64).reshape(3, 4), device=DEV)
    return m[:, :3], m[:, 3]


def _inv(T):
    return T[0].T, -(T[0].T @ T[1])


def _mv(R, v):
    return (R @ v[..., None])[..., 0]


def _log(R):
    """log of rotations [n, 3, 3]: (phi, theta)."""
    w = 0.5 * torch.stack([R[:, 2, 1] - R[:, 1, 2], R[:, 0, 2] - R[:, 2, 0], R[:, 1, 0] - R[:, 0, 1]], 1)
    s, c = w.norm(dim=1), 0.5 * (R[:, 0, 0] + R[:, 1, 1] + R[:, 2, 2] - 1.0)
    th = torch.atan2(s, c)
    f = torch.where(th < 1e-4, 1.0 + th * th / 6.0, th / s.clamp(min=1e-300))
    phi = f[:, None] * w
    far = th > 0.75 * math.pi   # near pi the axis comes from the symmetric part
    if far.any():
        S = 0.5 * (R[far] + R[far].transpose(1, 2)) - c[far, None, None] * torch.eye(3, device=DEV, dtype=R.dtype)
        col = torch.diagonal(S, dim1=1, dim2=2).argmax(1)
        a = torch.nn.functional.normalize(S[torch.arange(S.shape[0], device=DEV), :, col], dim=1)
        a = torch.where(((a * w[far]).sum(1) < 0)[:, None], -a, a)
        phi[far] = th[far, None] * a
    return phi, th


def _jl_inv(phi, th, v):
    """Inverse left Jacobian of SO(3) applied to v [n, d, 3]."""
    th = th.clamp(min=1e-300)
    beta = torch.where(th < 1e-2, 1.0 / 12.0 + th ** 2 / 720.0 + th ** 4 / 30240.0,
                       1.0 / th ** 2 - torch.sin(th) / (2.0 * th * (1.0 - torch.cos(th)).clamp(min=1e-300)))
    ph = phi[:, None, :].expand_as(v)
    a = torch.linalg.cross(ph, v)
    return v - 0.5 * a + beta[:, None, None] * torch.linalg.cross(ph, a)


class _Ref:
    """One robot under one constraint stack, batched over [n, d] configurations in 64 bits."""

    def __init__(self, wl):
        self.rb, self.p = wl.robot, wl.params
        self.d = wl.robot.n_joints
        self.X = [_se3(x) for x in wl.robot.X]
        self.fX = [_se3(x) for x in wl.robot.frame_X]
        self.parent = [int(v) for v in wl.robot.parent]
        self.mass = torch.tensor(wl.robot.mass, device=DEV)
        self.com = torch.tensor(np.asarray(wl.robot.com, dtype=np.float64).reshape(-1, 3), device=DEV)
        anc = np.zeros((self.d, self.d), bool)   # anc[j, l]: joint j moves link l
        for l in range(self.d):
            j = l
            while j >= 0:
                anc[j, l] = True
                j = self.parent[j]
        self.anc = torch.tensor(anc, device=DEV, dtype=torch.float64)
        self.link = [int(v) for v in wl.robot.frame_link]
        self.cons = [self._resolve(c) for c in wl.constraints]

    def fk(self, q):
        R, p, n = [], [], q.shape[0]
        for j in range(self.d):
            XR, Xp = self.X[j]
            pa = self.parent[j]
            if pa < 0:
                Rj, pj = XR.expand(n, 3, 3), Xp.expand(n, 3)
            else:
                Rj, pj = R[pa] @ XR, p[pa] + R[pa] @ Xp
            if int(self.rb.type[j]) == W.PRISMATIC:
                pj = pj + q[:, j, None] * Rj[:, :, 2]
            else:
                s, c = torch.sin(q[:, j])[:, None], torch.cos(q[:, j])[:, None]
                Rj = torch.stack([c * Rj[:, :, 0] + s * Rj[:, :, 1], c * Rj[:, :, 1] - s * Rj[:, :, 0], Rj[:, :, 2]], 2)
            R.append(Rj)
            p.append(pj)
        fr = [(R[l] @ self.fX[f][0], p[l] + R[l] @ self.fX[f][1]) for f, l in enumerate(self.link)]
        return R, p, fr

    def _resolve(self, c):
        P, Q, t, B = _se3(c.P), _se3(c.Q), [float(v) for v in c.target], c.B
        if c.q_ref is not None:
            _, _, fr = self.fk(torch.tensor(np.asarray(c.q_ref, dtype=np.float64), device=DEV)[None])
            fr = [(R[0], p[0]) for R, p in fr]
            a, b = fr[c.frame_a] if c.frame_a >= 0 else None, fr[c.frame_b] if c.frame_b >= 0 else None
            if c.kind in (W.C_POSE, W.C_POSE_BOUNDED):
                Qi = _inv(Q)
                P = (a[0] @ Qi[0], a[0] @ Qi[1] + a[1])
            elif c.kind == W.C_REL_POSE:
                P = (a[0].T @ b[0], a[0].T @ (b[1] - a[1]))
            elif c.kind in (W.C_PLANE, W.C_LINE):
                P = (P[0], a[1])
            elif c.kind == W.C_DIST:
                t[0] = float((b[1] - a[1]).norm())
            elif c.kind == W.C_COM_XY:
                t[:2] = [float(v) for v in 0.5 * (a[1] + b[1])[:2]]
        return c.kind, c.frame_a, c.frame_b, P, Q, t, B

    def residual_jacobian(self, q):
        n = q.shape[0]
        R, p, fr = self.fk(q)
        z = torch.stack([r[:, :, 2] for r in R], 1)          # [n, d, 3]
        o = torch.stack([v.expand(n, 3) for v in p], 1)
        rev = torch.tensor(np.asarray(self.rb.type) != W.PRISMATIC, device=DEV)[None, :, None]

        def velocity(x):   # of the point x [n, 3] when joint j moves
            return torch.where(rev, torch.linalg.cross(z, x[:, None, :] - o), z)

        F, J = [], []
        for kind, fa, fb, P, Q, t, B in self.cons:
            if kind == W.C_SPHERE:
                r = q.norm(dim=1, keepdim=True)
                F.append(r - t[0])
                J.append((q / r)[:, None, :])
            elif kind == W.C_AXIS_ALIGN:
                za = fr[fa][0][:, :, 2]
                on = self.anc[:, self.link[fa]][None, :, None] * rev
                v = torch.linalg.cross(z, za[:, None, :].expand_as(z)) * on
                F.append(za[:, :2])
                J.append(v[:, :, :2].transpose(1, 2))
            elif kind in (W.C_POSE, W.C_POSE_BOUNDED, W.C_REL_POSE):
                Pi = _inv(P)
                if kind == W.C_REL_POSE:
                    (Ra, pa), (Rb, pb) = fr[fa], fr[fb]
                    G = Pi[0] @ Ra.transpose(1, 2)
                    E, x, base = G @ Rb, pb, pb - pa
                    sgn = self.anc[:, self.link[fb]] - self.anc[:, self.link[fa]]
                else:
                    Qi = _inv(Q)
                    G = Pi[0].expand(n, 3, 3)
                    E = G @ fr[fa][0] @ Qi[0]
                    x = fr[fa][1] + _mv(fr[fa][0], Qi[1].expand(n, 3))
                    base, sgn = x, self.anc[:, self.link[fa]]
                phi, th = _log(E)
                e = torch.cat([_mv(G, base) + Pi[1], phi], 1)
                lin = velocity(x) @ G.transpose(1, 2)
                ang = _jl_inv(phi, th, (z * rev) @ G.transpose(1, 2))
                Jc = torch.cat([lin, ang], 2).transpose(1, 2) * sgn[None, None, :]
                if kind == W.C_POSE_BOUNDED:
                    lo, hi = (torch.tensor(np.asarray(B[i:i + 6], dtype=np.float64), device=DEV) for i in (0, 6))
                    f = e - torch.minimum(torch.maximum(e, lo), hi)
                    Jc = Jc * (f != 0)[:, :, None]
                    e = f
                F.append(e)
                J.append(Jc)
            elif kind in (W.C_PLANE, W.C_LINE):
                Pi = _inv(P)
                rows = [2] if kind == W.C_PLANE else [0, 1]
                on = self.anc[:, self.link[fa]][None, :, None]
                F.append((_mv(Pi[0].expand(n, 3, 3), fr[fa][1]) + Pi[1])[:, rows])
                J.append(((velocity(fr[fa][1]) * on) @ Pi[0].T)[:, :, rows].transpose(1, 2))
            elif kind == W.C_DIST:
                dv = fr[fb][1] - fr[fa][1]
                r = dv.norm(dim=1, keepdim=True)
                on = [self.anc[:, self.link[f]][None, :, None] for f in (fa, fb)]
                v = velocity(fr[fb][1]) * on[1] - velocity(fr[fa][1]) * on[0]
                F.append(r - t[0])
                J.append((v @ (dv / r)[:, :, None]).transpose(1, 2))
            else:   # centre of mass at a point
                cm = torch.stack([p[j] + _mv(R[j], self.com[j].expand(n, 3)) for j in range(self.d)], 1)
                M = self.mass.sum()
                C = self.anc @ (self.mass[:, None] * cm)     # subtree moments
                Mj = (self.anc @ self.mass)[None, :, None]
                v = torch.where(rev, torch.linalg.cross(z, C - Mj * o), Mj * z) / M
                F.append(((self.mass[:, None] * cm).sum(1) / M)[:, :2] - torch.tensor(t[:2], device=DEV, dtype=q.dtype))
                J.append(v[:, :, :2].transpose(1, 2))
        return torch.cat(F, 1), torch.cat(J, 1)

    def project(self, q, steps=None, chunk=262144):
        """Damped Newton on [d, n] starts until the residual is below tol, the
        cap (or `steps`) is reached, or a step exceeds max_step.  Returns
        ([d, n], converged, steps taken, left by max_step)."""
        cap = self.p.max_iters if steps is None else steps
        n = q.shape[1]
        conv = torch.zeros(n, dtype=torch.bool, device=DEV)
        div = torch.zeros(n, dtype=torch.bool, device=DEV)
        count = torch.zeros(n, dtype=torch.int32, device=DEV)
        out = q.double().t().contiguous()
        for c0 in range(0, n, chunk):
            idx = torch.arange(c0, min(n, c0 + chunk), device=DEV)
            for it in range(cap + 1):
                F, J = self.residual_jacobian(out[idx])
                done = F.norm(dim=1) < self.p.tol
                conv[idx[done]] = True
                if it == cap or bool(done.all()):
                    break
                idx, F, J = idx[~done], F[~done], J[~done]
                dq = self._pinv(J, F, self.p.lam)
                if self.p.max_step > 0:
                    far = dq.norm(dim=1) > self.p.max_step
                    div[idx[far]] = True
                    idx, dq = idx[~far], dq[~far]
                out[idx] -= dq
                count[idx] += 1
                if idx.numel() == 0:
                    break
        return out.t().contiguous(), conv, count, div

    @staticmethod
    def _pinv(J, F, lam):
        A = J @ J.transpose(1, 2) + lam * torch.eye(J.shape[1], device=DEV, dtype=J.dtype)
        L = torch.linalg.cholesky_ex(A)[0]
        y = torch.linalg.solve_triangular(L, F[:, :, None], upper=False)
        y = torch.linalg.solve_triangular(L.transpose(1, 2), y, upper=True)
        return (J.transpose(1, 2) @ y)[:, :, 0]

    def vjp(self, q, g):
        _, J = self.residual_jacobian(q.double().t())
        g = g.double().t()
        return (g - self._pinv(J, (J @ g[:, :, None])[:, :, 0], 0.0)).t().contiguous()


def _reference(wl):
    return _Ref(wl)


def exact(case, seed):
    call = case["call"]
    if case["problem"] == "humanoid_hull" or case.get("cyclic") or call == "check":
        return None
    if case["problem"] in ("arm", "tray", "peg", "tsr") and call != "vjp":
        # starts drawn from the whole joint box: where a few of them end is
        # decided by rounding (a step near a singular J goes many turns away,
        # or the cap is reached far from the manifold)
        return None
    wl, x = _inputs(case, seed)
    ref = _Ref(wl)
    if call in ("project", "project_check"):
        return [ref.project(x["q"])[0]] + [None] * (4 if call == "project_check" else 3)
    if call == "vjp":
        return [ref.vjp(x["q"], x["g"]), None]
    if call == "segments":
        length = x["length"].long()
        seg = torch.repeat_interleave(torch.arange(length.numel(), device=DEV), length)
        t = torch.arange(x["total"], device=DEV) - torch.repeat_interleave(length.cumsum(0) - length, length)
        q = x["start"].double()[:, seg] + t[None, :] * x["delta"].double()[:, seg]
        return [ref.project(q)[0], None, None, None]
    if call == "extend":
        # the particle that converges after the fewest steps, unless one left earlier by max_step
        qs, qt, eps = (x[k].double() for k in ("q_s", "q_t", "eps"))
        n, k = qs.shape[1], eps.shape[0]
        length = (qt - qs).norm(dim=0)
        v = (qt - qs) / length
        q0 = qs[:, None, :] + (length.clamp(max=wl.extra["r"]) + eps)[None] * v[:, None, :]
        q, conv, count, div = ref.project(q0.reshape(wl.dof, k * n))
        big = torch.full((k, n), 1 << 20, dtype=torch.int32, device=DEV)
        c = torch.where(conv.reshape(k, n), count.reshape(k, n), big)
        left = torch.where(div.reshape(k, n), count.reshape(k, n), big).min(0)[0]
        best = c.min(0)[0]
        win = (c == best).to(torch.int32).argmax(0)
        q = q.reshape(wl.dof, k, n)[:, win, torch.arange(n, device=DEV)]
        return [torch.where(((best >= 1 << 20) | (left < best))[None], qs, q), None, None, None]
    n, way = case["n"], case["way"]
    q = ref.project(x["Q"])[0]
    e = q.reshape(wl.dof, n, way).diff(dim=2)
    ln = e.norm(dim=0)
    u = e / ln.clamp(min=1e-300)
    g = torch.zeros_like(q).reshape(wl.dof, n, way)
    g[:, :, 1:] += u
    g[:, :, :-1] -= u
    grad = ref.vjp(q, g.reshape(wl.dof, n * way))
    step = 0.1 * grad
    step = step * (0.05 / step.abs().amax(0).clamp(min=1e-300)).clamp(max=1.0)
    inner = torch.ones(way, device=DEV, dtype=q.dtype)
    inner[0] = inner[-1] = 0.0
    return {"Q": q - step * inner.repeat(n), "length": ln.sum(1), "grad": grad}
