"""The framework's work, as cases that can be timed and compared.

Each case is one pass through a public entry point: a step, a rollout (plain,
with outputs for logging, with the environment layer, streamed from the
host), a gradient (through torch.autograd as the policy-gradient demo takes
it, or through the reverse pass with the caller's own workspace) or a
heterogeneous batch.  Sizes follow the repository's own workloads (one
environment up to 65,536, one step up to the 1,000-step rollout), with odd
ones among them.  Inputs are made on the GPU from the seed alone: default
poses by forward kinematics in FP64, joint angles spread by N(0, 0.1^2), the
root lowered onto the ground where a pass is too short to fall there, so that
contacts are part of every case, and actions U[-1, 1].

`exact` states the same step (Algorithm 1: kinematic integrator; spring
joints, actuators and contacts on the same state; potential and collision
integrators) in plain torch FP64 without this repository's code, with
gradients by torch.autograd.  It answers for rollouts short enough that FP32
still follows FP64, and for scenes without capsule-box contacts.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2106_13281_gb300 import autograd as G
from paper_2106_13281_gb300 import scenes as S
from paper_2106_13281_gb300.system import BraxBatch, BraxSystem

# Algorithmic flops of one environment step and of its reverse pass, counted
# over sampled rollouts (contact responses only where contacts are active).
FLOPS = {"quadruped": (42995, 142500), "biped": (181615, 630057), "pendulum": (11200, 36630), "arm_box": (57082, 161783)}
# How far a scene's root is lowered so that it starts within 5 cm above (or
# slightly in) the ground; the other scenes already stand on it or hang.
DROP = {"quadruped": 0.36}
BATCH = ("pendulum", "quadruped", "biped", "arm_box")


def listed():
    return [
        # one environment stepped once: closed-loop evaluation of a policy, all latency
        {"name": "step_one", "kind": "step", "scene": "quadruped", "n": 1},
        # one control step of a training batch
        {"name": "step_batch", "kind": "step", "scene": "quadruped", "n": 4096},
        # experience collection of an RL learner: 2,048 environments, an unroll of 20 steps with auto reset
        {"name": "env_unroll", "kind": "env", "scene": "quadruped", "n": 2048, "T": 20},
        # an odd-sized rollout that logs the torso path and the contact counts
        {"name": "rollout_ragged", "kind": "rollout", "scene": "quadruped", "n": 3001, "T": 50, "logs": True},
        # the headline workload: 65,536 environments for 1,000 steps
        {"name": "rollout_large", "kind": "rollout", "scene": "quadruped", "n": 65536, "T": 1000, "logs": False},
        # the humanoid workload: 3-DOF joints and 120 self-collision pairs
        {"name": "biped_rollout", "kind": "rollout", "scene": "biped", "n": 16384, "T": 50, "logs": False},
        {"name": "biped_small", "kind": "rollout", "scene": "biped", "n": 500, "T": 10, "logs": True},
        # host-resident inputs streamed through the GPU, the state read back
        {"name": "streamed", "kind": "streamed", "scene": "quadruped", "n": 16384, "T": 100},
        # one step of an analytic policy gradient: forward and reverse of a single step
        {"name": "apg_step", "kind": "grad", "scene": "quadruped", "n": 1024, "T": 1, "K": 1},
        # gradients of a short horizon through torch.autograd with its default checkpoint interval
        {"name": "grad_horizon", "kind": "grad", "scene": "quadruped", "n": 4096, "T": 20, "K": 10},
        # the reverse pass at the headline's width, a checkpoint at every step, the caller's own workspace
        {"name": "grad_large", "kind": "grad_ws", "scene": "quadruped", "n": 65536, "T": 20, "K": 1},
        # systems of different sizes stepped and differentiated together
        {"name": "batch_grad", "kind": "batch", "n": 8192, "T": 8, "K": 4},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "env", "rollout", "rollout", "streamed", "grad", "grad", "grad_ws", "batch"])
    if kind == "batch":
        n = _log_int(rng, 64, 8192)
        return {"kind": kind, "n": n, "T": rng.randint(1, 10), "K": rng.choice([1, 2, 5])}
    if kind in ("step", "rollout"):
        scene = rng.choice(["quadruped", "quadruped", "pendulum", "biped", "arm_box"])
    elif kind == "env":
        scene = rng.choice(["quadruped", "quadruped", "biped"])
    elif kind == "streamed":
        scene = rng.choice(["quadruped", "pendulum"])
    else:
        scene = rng.choice(["quadruped", "quadruped", "quadruped", "pendulum", "arm_box"])
    wide = scene in ("quadruped", "pendulum")
    n = _log_int(rng, 1 if kind != "streamed" else 1024, 65536 if wide else 16384)
    if rng.random() < 0.5:  # multiples of a warp as often as odd sizes
        n = max(32, n // 32 * 32)
    case = {"kind": kind, "scene": scene, "n": n}
    if kind == "rollout":
        most = 1000 if wide else 50
        case |= {"T": _log_int(rng, 1, most), "logs": rng.random() < 0.5}
    elif kind == "streamed":
        case |= {"T": _log_int(rng, 20, 200)}
    elif kind == "env":
        case |= {"T": _log_int(rng, 1, 50)}
    elif kind in ("grad", "grad_ws"):
        most = 20 if wide else 3
        case |= {"T": _log_int(rng, 1, most), "K": rng.choice([1, 1, 2, 5, 10])}
    return case


# ------------------------------------------------------------------ inputs (torch, FP64, then FP32)
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _quat_mul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1)


def _rot(q):
    """Rotation matrices [..., 3, 3] of unit quaternions (w, x, y, z)."""
    w, x, y, z = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).unflatten(-1, (3, 3))


def _poses(desc, n, gen, drop):
    """States [n, B, 13]: the rest pose with spread joint angles and root
    heights, the bodies placed by forward kinematics, at rest."""
    dev = gen.device
    t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=dev)
    B, D = len(desc["mass"]), S.n_dof(desc)
    ang = t(S.joint_angle_centres(desc)) + 0.1 * torch.randn((n, D), generator=gen, device=dev, dtype=torch.float64)
    lift = 0.05 * torch.rand((n,), generator=gen, device=dev, dtype=torch.float64) - drop
    x = t(desc["rest_pos"]).repeat(n, 1, 1)
    q = t(desc["rest_rot"]).repeat(n, 1, 1)
    x[:, 0, 2] += lift
    todo, placed, first = list(range(len(desc["parent"]))), set(range(B)) - {int(c) for c in desc["child"]}, []
    at = 0
    for d in desc["dof"]:
        first.append(at)
        at += int(d)
    while todo:
        j = next(k for k in todo if int(desc["parent"][k]) in placed)
        todo.remove(j)
        p, c = int(desc["parent"][j]), int(desc["child"][j])
        rel = torch.zeros((n, 4), device=dev, dtype=torch.float64)
        rel[:, 0] = 1
        for a in range(int(desc["dof"][j])):
            half = torch.zeros((n, 4), device=dev, dtype=torch.float64)
            half[:, 0], half[:, 1 + a] = torch.cos(0.5 * ang[:, first[j] + a]), torch.sin(0.5 * ang[:, first[j] + a])
            rel = _quat_mul(rel, half)
        fp, fc = t(desc["parent_frame"][j]), t(desc["child_frame"][j]) * t([1, -1, -1, -1])
        q[:, c] = _quat_mul(_quat_mul(_quat_mul(q[:, p], fp.expand(n, 4)), rel), fc.expand(n, 4))
        q[:, c] /= q[:, c].norm(dim=-1, keepdim=True)
        x[:, c] = x[:, p] + _rot(q[:, p]) @ t(desc["parent_offset"][j]) - _rot(q[:, c]) @ t(desc["child_offset"][j])
        placed.add(c)
    return torch.cat([x, q, torch.zeros((n, B, 6), device=dev, dtype=torch.float64)], -1).float().contiguous()


def _inputs(case, seed, dev=None):
    """What a program has in hand: per system (name, descriptor, n), the start
    states, the actions and, for gradients, the cotangents of the final state
    and of the torso path (a learnt value's gradient and a progress reward)."""
    gen = torch.Generator(device=dev or _device())
    gen.manual_seed(1_000_003 * int(seed) + 17)
    rand = lambda *s: 2 * torch.rand(s, generator=gen, device=gen.device) - 1
    if case["kind"] == "batch":
        n = case["n"]
        parts = [("pendulum", n), ("quadruped", max(1, n // 2)), ("biped", max(1, n // 4)), ("arm_box", max(1, n // 4))]
    else:
        parts = [(case["scene"], case["n"])]
    T = case.get("T", 1)
    low = case["kind"] != "env" and T < 200  # an environment starts from its reset pose, a long rollout falls
    got = []
    for name, n in parts:
        d = S.SCENES[name]()
        st = _poses(d, n, gen, DROP.get(name, 0.0) if low else 0.0)
        one = {"scene": name, "desc": d, "n": n, "state0": st, "actions": rand(T, n, len(d["gear"]))}
        if case["kind"] in ("grad", "grad_ws", "batch"):
            one["g_state"] = rand(n, len(d["mass"]), 13)
            one["g_torso"] = rand(T, n, 3) / T
        got.append(one)
    return got


def prepare(case, seed):
    parts = _inputs(case, seed)
    s = {"case": case, "sys": [BraxSystem(p["desc"]) for p in parts]}
    if case["kind"] == "batch":
        T, K = case["T"], case["K"]
        flat = lambda k: torch.cat([p[k].reshape(-1) for p in parts])
        s |= {"batch": BraxBatch(s["sys"], [p["n"] for p in parts]), "state0": flat("state0"), "actions": flat("actions"),
              "g_state": flat("g_state"), "g_torso": flat("g_torso")}
        s["ws"] = torch.empty((s["batch"].workspace_size(T, K),), device="cuda", dtype=torch.uint8)
        s["shapes"] = [(tuple(p["state0"].shape), tuple(p["actions"].shape)) for p in parts]
        return s
    p, sysm = parts[0], s["sys"][0]
    s |= {k: p[k] for k in ("state0", "actions", "g_state", "g_torso") if k in p}
    if case["kind"] == "streamed":
        host = lambda t: t.cpu().pin_memory()
        s["h_state"], s["h_actions"], s["h_out"], s["bufs"] = host(s.pop("state0")), host(s.pop("actions")), None, {}
        s["h_out"] = torch.empty_like(s["h_state"]).pin_memory()
    elif case["kind"] == "grad":
        s["state0"].requires_grad_(True)
        s["actions"].requires_grad_(True)
    elif case["kind"] == "grad_ws":
        s["ws"] = torch.empty((sysm.workspace_size(case["n"], case["T"], case["K"]),), device="cuda", dtype=torch.uint8)
    return s


def run(s):
    case, sysm = s["case"], s["sys"][0]
    kind = case["kind"]
    if kind == "step":
        return {"state": sysm.step(s["state0"], s["actions"][0])}
    if kind == "rollout":
        return sysm.rollout(s["state0"], s["actions"], torso=case["logs"], contact_count=case["logs"])
    if kind == "env":
        return sysm.env_rollout(s["state0"], s["actions"])
    if kind == "streamed":
        sysm.rollout_streamed(s["h_state"], s["h_actions"], s["h_out"], chunk_steps=50, bufs=s["bufs"])
        torch.cuda.current_stream().synchronize()  # the state is read on the host next
        return {"state_T": s["h_out"]}
    if kind == "grad":
        state_T, torso = G.rollout(sysm, s["state0"], s["actions"], case["K"])
        g0, ga = torch.autograd.grad((state_T, torso), (s["state0"], s["actions"]), (s["g_state"], s["g_torso"]))
        return {"state_T": state_T, "torso": torso, "g_state0": g0, "g_actions": ga}
    if kind == "grad_ws":
        o = sysm.rollout(s["state0"], s["actions"], K=case["K"], checkpoints=True)
        ga, g0 = sysm.rollout_backward(s["state0"], s["actions"], o["checkpoints"], s["g_state"], s["g_torso"],
                                       K=case["K"], workspace=s["ws"])
        return {"state_T": o["state_T"], "checkpoints": o["checkpoints"], "g_state0": g0, "g_actions": ga}
    T, K = case["T"], case["K"]
    o = s["batch"].rollout(s["state0"], s["actions"], T, K=K, checkpoints=True)
    ga, g0 = s["batch"].rollout_backward(s["state0"], s["actions"], o["checkpoints"], s["g_state"], T, K=K,
                                         g_torso=s["g_torso"], workspace=s["ws"])
    out, i, j = [], 0, 0
    for ss, aa in s["shapes"]:  # each system's own share of the batch's arrays
        ns, na = math.prod(ss), math.prod(aa)
        out.append({"state_T": o["state_T"][i:i + ns].view(ss), "g_state0": g0[i:i + ns].view(ss),
                    "g_actions": ga[j:j + na].view(aa)})
        i, j = i + ns, j + na
    return out


def work(case):
    T = case.get("T", 1)
    if case["kind"] == "batch":
        n = case["n"]
        parts = [("pendulum", n), ("quadruped", max(1, n // 2)), ("biped", max(1, n // 4)), ("arm_box", max(1, n // 4))]
    else:
        parts = [(case["scene"], case["n"])]
    by = fl = 0
    for name, n in parts:
        d = S.SCENES[name]()
        state, act = len(d["mass"]) * 52 * n, len(d["gear"]) * 4 * n * T
        fwd, rev = FLOPS[name]
        by += 2 * state + act
        fl += fwd * n * T
        if case["kind"] == "env":
            by += T * n * ((11 + 2 * S.n_dof(d)) * 4 + 5)
        if case.get("logs"):
            by += T * n * 12 + 4 * n
        if case["kind"] in ("grad", "grad_ws", "batch"):  # checkpoints out and in, cotangents in, gradients out
            by += 2 * state * -(-T // case["K"]) + 2 * state + act + T * n * 12
            fl += (fwd + rev) * n * T  # the reverse pass recomputes the forward once
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ the step in FP64
def _cross(a, b):
    return torch.linalg.cross(a, b)


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


class _Step64:
    """Algorithm 1 on states (x, q, v, w) of shapes [N, B, .], vectorised over
    environments, joints, contact points and pairs."""

    def __init__(self, d, dev):
        t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=dev)
        ix = lambda a: torch.as_tensor(np.asarray(a, dtype=np.int64), device=dev)
        self.B, self.J, self.sub = len(d["mass"]), len(d["parent"]), int(d["substeps"])
        self.dt, self.h = float(d["dt"]), float(d["dt"]) / int(d["substeps"])
        self.g, self.beta, self.eps = t(d["gravity"]), float(d["baumgarte"]), float(d["contact_eps"])
        self.inv_m, self.inv_I = 1 / t(d["mass"])[:, None], 1 / t(d["inertia"])
        self.mp, self.mr = 1 - t(d["frozen_pos"]), 1 - t(d["frozen_rot"])
        self.par, self.chi, self.dof = ix(d["parent"]), ix(d["child"]), [int(k) for k in d["dof"]]
        self.hinge = (ix(self.dof) == 1).double()[:, None]
        self.off_p, self.off_c = t(d["parent_offset"]), t(d["child_offset"])
        unit = lambda q: t(q) / t(q).norm(dim=-1, keepdim=True)
        self.fp, self.fc = _rot(unit(d["parent_frame"])), _rot(unit(d["child_frame"]))  # columns: joint axes
        col = lambda k: t(d[k])[:, None]
        self.k, self.c, self.ka, self.ca = col("stiffness"), col("spring_damping"), col("angular_stiffness"), col("angular_damping")
        self.kl, self.lo, self.hi = col("limit_stiffness"), t(np.deg2rad(d["limit_lo"])), t(np.deg2rad(d["limit_hi"]))
        self.has = t([[a < k for a in range(3)] for k in self.dof]).reshape(-1, 3)
        self.gear, self.act_at = t(d["gear"]), ix(3 * np.asarray(d["act_joint"]) + np.asarray(d["act_axis"]))
        # plane-contact points (sphere centres in the body frame) and capsule pairs
        rc = _rot(unit(d["col_rot"]))
        pt, pairs, self.boxes = [], [], False
        for a, b in zip(d["pair_a"], d["pair_b"]):
            a, b = (int(b), int(a)) if d["col_body"][a] < 0 else (int(a), int(b))
            mu, e = d["friction"][a] * d["friction"][b], d["elasticity"][a] * d["elasticity"][b]
            body, kind = int(d["col_body"][a]), int(d["col_type"][a])
            half = max(0.5 * float(d["length"][a]) - float(d["radius"][a]), 0.0)
            pos = t(d["col_pos"][a])
            if int(d["col_body"][b]) < 0:
                if kind == S.CAPSULE:
                    at = [pos + s * half * rc[a][:, 2] for s in ((-1, 1) if half else (0,))]
                    r = float(d["radius"][a])
                else:
                    at = [pos + rc[a] @ (t(d["half_extents"][a]) * t([i, j, k])) for i in (-1, 1) for j in (-1, 1) for k in (-1, 1)]
                    r = 0.0
                pt += [(body, o, r, rc[b][:, 2], t(d["col_pos"][b]), mu, e) for o in at]
            elif kind == S.CAPSULE and int(d["col_type"][b]) == S.CAPSULE:
                hb = max(0.5 * float(d["length"][b]) - float(d["radius"][b]), 0.0)
                ends = [t(d["col_pos"][i]) + s * h_ * rc[i][:, 2] for i, h_ in ((a, half), (b, hb)) for s in (-1, 1)]
                pairs.append((body, int(d["col_body"][b]), *ends, float(d["radius"][a]), float(d["radius"][b]), mu, e))
            else:
                self.boxes = True
        z = lambda rows, k: t([r[k] for r in rows])[:, None]
        st = lambda rows, k: torch.stack([r[k] for r in rows])
        self.pt = pt and (ix([r[0] for r in pt]), st(pt, 1), z(pt, 2), st(pt, 3), st(pt, 4), z(pt, 5), z(pt, 6))
        self.pr = pairs and (ix([r[0] for r in pairs]), ix([r[1] for r in pairs]), *(st(pairs, k) for k in (2, 3, 4, 5)),
                             *(z(pairs, k) for k in (6, 7, 8, 9)))

    def angles(self, R):
        """Joint angles [N, J, 3], the parent's joint axes and the child's, [N, J, 3, 3] (columns)."""
        P, C = R[:, self.par] @ self.fp, R[:, self.chi] @ self.fc
        M = P.transpose(-1, -2) @ C
        one = torch.atan2(M[..., 2, 1], M[..., 1, 1])
        sq = (M[..., 0, 0] ** 2 + M[..., 0, 1] ** 2).clamp_min(1e-30).sqrt()
        three = torch.stack([torch.atan2(-M[..., 1, 2], M[..., 2, 2]), torch.atan2(M[..., 0, 2], sq),
                             torch.atan2(-M[..., 0, 1], M[..., 0, 0])], -1)
        hinge = torch.stack([one, torch.zeros_like(one), torch.zeros_like(one)], -1)
        return torch.where(self.hinge > 0, hinge, three) * self.has, P, C

    def respond(self, sides, n, depth, mu, e, live, acc):
        """One set of contacts: sides = (body index, sign, lever arm); adds the velocity changes to acc = (dv, dw, count)."""
        v, w, Ii = self._v, self._w, self._Ii
        u = sum(s * (v[:, b] + _cross(w[:, b], l)) for b, s, l in sides)

        def mass(dirn):
            k = 0
            for b, _, l in sides:
                ld = _cross(l, dirn)
                k = k + _dot(self.mp[b] * dirn, dirn) * self.inv_m[b] + _dot(self.mr[b] * (Ii[:, b] @ ld[..., None])[..., 0], ld)
            return k

        kn = mass(n)
        live = live & (kn > 0)
        un = _dot(u, n)
        jn = ((torch.maximum(self.beta / self.h * depth, -e * un) - un) / torch.where(live, kn, 1.0)).clamp_min(0)
        ut = u - un * n
        ut2 = _dot(ut, ut)
        slip = ut2 > self.eps ** 2
        utn = torch.where(slip, ut2, 1.0).sqrt()
        tang = ut / utn
        jt = torch.minimum(utn / torch.where(slip & live, mass(tang), 1.0), mu * jn)
        J = jn * n - torch.where(slip, jt, 0.0) * tang
        for b, s, l in sides:
            dv = self.mp[b] * self.inv_m[b] * s * J
            dw = self.mr[b] * (Ii[:, b] @ _cross(l, s * J)[..., None])[..., 0]
            acc = [acc[0].index_add(1, b, torch.where(live, dv, 0.0)), acc[1].index_add(1, b, torch.where(live, dw, 0.0)),
                   acc[2].index_add(1, b, live.double())]
        return acc

    def plane_contacts(self, x, R, acc):
        b, o, r, n, p0, mu, e = self.pt
        ro = (R[:, b] @ o[..., None])[..., 0]
        depth = r - _dot(x[:, b] + ro - p0, n)
        return self.respond([(b, 1.0, ro - r * n)], n.expand_as(ro), depth, mu, e, depth > 0, acc)

    def pair_contacts(self, x, R, acc):
        a, b, a0, a1, b0, b1, ra, rb, mu, e = self.pr
        at = lambda i, o: x[:, i] + (R[:, i] @ o[..., None])[..., 0]
        P, Q = at(a, a0), at(b, b0)
        d1, d2 = at(a, a1) - P, at(b, b1) - Q
        r = P - Q
        aa, ee, f, c, bb = _dot(d1, d1), _dot(d2, d2), _dot(d2, r), _dot(d1, r), _dot(d1, d2)
        den = aa * ee - bb * bb
        skew = den > 1e-5 * aa * ee
        s = torch.where(skew, ((bb * f - c * ee) / torch.where(skew, den, 1.0)).clamp(0, 1), 0.0)
        t = (bb * s + f) / ee
        s = torch.where(t < 0, (-c / aa).clamp(0, 1), torch.where(t > 1, ((bb - c) / aa).clamp(0, 1), s))
        t = t.clamp(0, 1)
        c1, c2 = P + s * d1, Q + t * d2
        df = c1 - c2
        d2_ = _dot(df, df)
        far = d2_ >= self.eps ** 2
        dl = torch.where(far, d2_, 1.0).sqrt()
        depth = ra + rb - dl
        n = df / dl
        p = 0.5 * ((c1 - ra * n) + (c2 + rb * n))
        return self.respond([(a, 1.0, p - x[:, a]), (b, -1.0, p - x[:, b])], n, depth, mu, e, far & (depth > 0), acc)

    def substep(self, x, q, v, w, act):
        h = self.h
        v, w = self.mp * v, self.mr * w
        x = x + h * v
        q = q + 0.5 * h * _quat_mul(torch.cat([torch.zeros_like(w[..., :1]), w], -1), q)
        q = q / q.norm(dim=-1, keepdim=True)
        R = _rot(q)
        self._v, self._w, self._Ii = v, w, (R * self.inv_I[:, None, :]) @ R.transpose(-1, -2)
        F, tau = torch.zeros_like(v), torch.zeros_like(w)
        if self.J:
            p, c = self.par, self.chi
            rp, rc = (R[:, p] @ self.off_p[..., None])[..., 0], (R[:, c] @ self.off_c[..., None])[..., 0]
            f = self.k * (x[:, p] + rp - x[:, c] - rc) - self.c * (v[:, c] + _cross(w[:, c], rc) - v[:, p] - _cross(w[:, p], rp))
            th, P, C = self.angles(R)
            L = self.kl * torch.where(th < self.lo, self.lo - th, torch.where(th > self.hi, self.hi - th, 0.0)) * self.has + act
            wr, P0 = w[:, c] - w[:, p], P[..., 0]
            tj = (P @ L[..., None])[..., 0] - self.ca * torch.where(self.hinge > 0, _dot(wr, P0) * P0, wr)
            tj = tj + self.hinge * self.ka * _cross(C[..., 0], P0)
            F = F.index_add(1, c, f).index_add(1, p, -f)
            tau = tau.index_add(1, c, _cross(rc, f) + tj).index_add(1, p, -_cross(rp, f) - tj)
        acc = [torch.zeros_like(v), torch.zeros_like(w), torch.zeros_like(v[..., :1])]
        acc = self.plane_contacts(x, R, acc) if len(self.pt) else acc
        acc = self.pair_contacts(x, R, acc) if len(self.pr) else acc
        many = acc[2].clamp_min(1)
        v = self.mp * (v + h * (self.inv_m * F + self.g)) + acc[0] / many
        w = self.mr * (w + h * (self._Ii @ tau[..., None])[..., 0]) + acc[1] / many
        return (x, q, v, w), acc[2].sum((1, 2))

    def step(self, s, a):
        act = torch.zeros((a.shape[0], 3 * self.J), dtype=a.dtype, device=a.device)
        act = act.index_add(1, self.act_at, self.gear * a.clamp(-1, 1)).unflatten(1, (self.J, 3))
        for _ in range(self.sub):
            s, _n = self.substep(*s, act)
        return s


def _split(st):
    return st[..., :3], st[..., 3:7], st[..., 7:10], st[..., 10:]


def _env64(f, st, a):
    dof = [(j, k) for j, d in enumerate(f.dof) for k in range(d)]
    s, first, obs, rew, done = _split(st), _split(st), [], [], []
    for t in range(a.shape[0]):
        was = s[0][:, 0, 0]
        s = f.step(s, a[t])
        x, q, v, w = s
        th, P, _ = f.angles(_rot(q))
        rate = (P.transpose(-1, -2) @ (w[:, f.chi] - w[:, f.par])[..., None])[..., 0]
        pick = lambda y: torch.stack([y[:, j, k] for j, k in dof], -1)
        obs.append(torch.cat([x[:, 0, 2:], q[:, 0], v[:, 0], w[:, 0], pick(th), pick(rate)], -1))
        d = (x[:, 0, 2] < 0.2) | (x[:, 0, 2] > 1.0)
        rew.append((x[:, 0, 0] - was) / f.dt + (~d).double() - 0.5 * (a[t].clamp(-1, 1) ** 2).sum(-1))
        done.append(d)
        s = tuple(torch.where(d[:, None, None], r, y) for r, y in zip(first, s))
    return {"state_T": torch.cat(s, -1), "obs": torch.stack(obs), "reward": torch.stack(rew), "done": torch.stack(done)}


def _exact_part(p, T, want_grad, logs):
    f = _Step64(p["desc"], p["state0"].device)
    if f.boxes or (f.pr and T > 5):  # self-collisions part FP32 from FP64 within a few steps
        return None
    out = []
    for i in range(0, p["n"], 8192):  # environments are independent
        st = p["state0"][i:i + 8192].double().requires_grad_(want_grad)
        a = p["actions"][:, i:i + 8192].double().requires_grad_(want_grad)
        s, torso, ck = _split(st), [], []
        for t in range(T):
            ck.append(torch.cat(s, -1).detach())
            s = f.step(s, a[t])
            torso.append(s[0][:, 0])
        s, torso = torch.cat(s, -1), torch.stack(torso)
        g = [None, None]
        if want_grad:
            g = torch.autograd.grad((s, torso), (st, a), (p["g_state"][i:i + 8192].double(), p["g_torso"][:, i:i + 8192].double()))
        out.append((s.detach(), torso.detach(), g[0], g[1], torch.stack(ck)))
    cat = lambda k, dim: None if out[0][k] is None else torch.cat([o[k] for o in out], dim)
    return {"state_T": cat(0, 0), "torso": cat(1, 1), "g_state0": cat(2, 0), "g_actions": cat(3, 1), "checkpoints": cat(4, 1)}


def exact(case, seed):
    kind, T = case["kind"], case.get("T", 1)
    grad = kind in ("grad", "grad_ws", "batch")
    # longer rollouts leave what FP32 follows; larger gradients take too long
    if T > 20 or (grad and case["n"] * T > 100_000):
        return None
    parts = _inputs(case, seed)
    if kind == "env":
        p = parts[0]
        o = _env64(_Step64(p["desc"], p["state0"].device), p["state0"].double(), p["actions"].double())
        return dict(o, done=None)
    got = [_exact_part(p, T, grad, case.get("logs", False)) for p in parts]
    if kind == "batch":
        return [{k: g[k] for k in ("g_actions", "g_state0", "state_T")} if g else
                {k: None for k in ("g_actions", "g_state0", "state_T")} for g in got]
    g = got[0]
    if g is None:
        return None
    if kind == "step":
        return {"state": g["state_T"]}
    if kind == "rollout":
        return {"state_T": g["state_T"], "torso": g["torso"], "contact_count": None} if case["logs"] else {"state_T": g["state_T"]}
    if kind == "streamed":
        return {"state_T": g["state_T"]}
    if kind == "grad":
        return {k: g[k] for k in ("state_T", "torso", "g_state0", "g_actions")}
    return {"state_T": g["state_T"], "checkpoints": g["checkpoints"][::case["K"]], "g_state0": g["g_state0"], "g_actions": g["g_actions"]}
