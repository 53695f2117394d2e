"""Performance cases: the calls that users of the whole-body evaluation make, over the range of robots and batches they make them with.

The robots have the shapes of the paper's (a 7-DoF arm, a 23-DoF tree, a 48-DoF humanoid with 15,392 masked sphere pairs); the joint
states, upstream gradients and control points follow the distributions of the benchmark's workloads.  Every call runs with the library's
default launch choices, as a program that has not tuned anything makes it.
"""
import functools
import math
import types

import numpy as np
import torch

from paper_2603_05493_gb300 import wbe

# ---------------------------------------------------------------------------
# robots (descriptor arrays only)
# ---------------------------------------------------------------------------


def _limbs(spine, neck, arm, leg, fingers, finger):
    """Parents of a fixed-base humanoid: pelvis, spine, neck, two arms (each with fingers on its last link), two legs from the pelvis."""
    parent = [-1]

    def chain(p, length):
        for _ in range(length):
            parent.append(p)
            p = len(parent) - 1
        return p

    top = chain(0, spine)
    chain(top, neck)
    for _ in range(2):
        hand = chain(top, arm)
        for _ in range(fingers):
            chain(hand, finger)
    for _ in range(2):
        chain(0, leg)
    return parent


# name: parents, joint of link 0, base spheres, sphere radii, least tree distance of a masked-in pair, seed
_SHAPES = {
    "arm7": (list(range(-1, 6)), 1, 0, (0.03, 0.08), 2, 7),
    "tree23": (_limbs(1, 0, 5, 6, 0, 0), 0, 8, (0.02, 0.10), 2, 23),
    "humanoid48": (_limbs(2, 2, 7, 6, 3, 3), 0, 8, (0.02, 0.10), 5, 48),
}


def _unit(rng):
    v = rng.normal(size=3)
    return v / np.linalg.norm(v)


def _apart(parent):
    """Edges between every two links of the tree."""
    n = len(parent)
    d = np.zeros((n, n), np.int64)
    for k in range(1, n):
        d[k, :k] = d[parent[k], :k] + 1
        d[:k, k] = d[k, :k]
    return d


@functools.lru_cache(maxsize=None)
def describe(name):
    """The descriptor of a robot; "humanoid48+3kg" carries a 3 kg point payload on each hand."""
    base = name.split("+")[0]
    parent, joint0, base_spheres, radii, least, seed = _SHAPES[base]
    rng = np.random.default_rng(seed)
    n = len(parent)
    jtype = np.array([joint0] + [1] * (n - 1), np.int32)
    jidx = np.cumsum(jtype > 0).astype(np.int32) - 1
    jidx[jtype == 0] = -1
    axis, fixed = np.zeros((n, 3)), np.zeros((n, 12))
    fixed[:, 0] = fixed[:, 4] = fixed[:, 8] = 1.0
    for k in range(n):
        if jtype[k]:
            axis[k] = _unit(rng)
            fixed[k, 9:] = rng.uniform(0.05, 0.4) * _unit(rng)
    first_child = {}
    for k in range(n):
        first_child.setdefault(parent[k], k)
    out = np.array([fixed[first_child[k], 9:] if k in first_child else rng.uniform(0.05, 0.4) * _unit(rng) for k in range(n)])
    link, centre, radius = [], [], []
    for k in range(n):
        for s in range(4 if jtype[k] else base_spheres):
            link.append(k)
            centre.append((s + 0.5) / 4 * out[k] + rng.uniform(-0.01, 0.01, 3) if jtype[k] else rng.uniform(-0.1, 0.1, 3))
            radius.append(rng.uniform(*radii))
    link = np.array(link, np.int32)
    i, j = np.triu_indices(len(link), 1)
    keep = _apart(parent)[link[i], link[j]] >= least
    mass, inertia = rng.uniform(0.5, 3.0, n), np.zeros((n, 6))
    for k in range(n):
        side = rng.uniform(0.05, 0.3, 3) ** 2
        turn = np.linalg.qr(rng.normal(size=(3, 3)))[0]
        box = turn @ np.diag(mass[k] / 12 * (side.sum() - side)) @ turn.T
        inertia[k] = box[0, 0], box[1, 1], box[2, 2], box[0, 1], box[0, 2], box[1, 2]
    f32 = lambda x: np.asarray(x, np.float32).astype(np.float64)  # noqa: E731
    hands = [k for k in range(n) if parent.count(k) >= 3 and k > 2] if "+" in name else []
    return types.SimpleNamespace(
        n=n, dof=int(jidx.max()) + 1, S=len(link), P=int(keep.sum()), moving=int((jtype > 0).sum()),
        parent=np.array(parent, np.int32), jtype=jtype, axis=f32(axis), T_fixed=f32(fixed), jidx=jidx, mimic_mult=np.ones(n),
        mimic_off=np.zeros(n), gravity=np.array([0.0, 0.0, -9.81]), sph_link=link, sph_c=f32(centre), sph_r=f32(radius),
        pairs=np.stack([i[keep], j[keep]], 1).astype(np.int32), mass=f32(mass), com=f32(rng.uniform(-0.05, 0.05, (n, 3)) + 0.5 * out),
        Icom=f32(inertia), pm_link=np.array(hands, np.int32), pm_mass=np.full(len(hands), 3.0),
        pm_pos=np.tile(f32([0.0, 0.0, 0.05]), (len(hands), 1)))


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------


def listed():
    return [
        # A controller's tick on a single arm: the smallest call, all launches and latency.
        {"name": "arm_tick", "kind": "forward", "robot": "arm7", "B": 64, "bits": False},
        # Sampling for an arm: 4096 seeds x 32 timesteps of feasibility checks, forward only.
        {"name": "arm_seeds", "kind": "forward", "robot": "arm7", "B": 131072, "bits": False},
        # A few seeds of a humanoid with the colliding-pair mask wanted (a planner's edge check).
        {"name": "humanoid_check", "kind": "forward", "robot": "humanoid48", "B": 1501, "bits": True},
        # One humanoid trajectory through torch's autograd: an online optimiser's step.
        {"name": "humanoid_tick", "kind": "gradient", "robot": "humanoid48", "B": 37},
        # A ragged medium batch on a legged robot with arms.
        {"name": "tree_step", "kind": "gradient", "robot": "tree23", "B": 3001},
        # The headline: 1024 seeds x 32 timesteps of the humanoid, forward and adjoint through torch's autograd.
        {"name": "humanoid_step", "kind": "gradient", "robot": "humanoid48", "B": 32768},
        # The same with as many seeds as an offline planner uses.
        {"name": "humanoid_many", "kind": "gradient", "robot": "humanoid48", "B": 99999},
        # Trajectory optimisation: control points to cost and control-point gradient, worst pair and motion terms, payload on the hands.
        {"name": "trajopt", "kind": "trajopt", "robot": "humanoid48+3kg", "seeds": 512, "T": 64, "K": 16, "hinge": False},
        # The same with every close pair in the cost, fewer seeds, an odd number of timesteps.
        {"name": "trajopt_hinge", "kind": "trajopt", "robot": "humanoid48+3kg", "seeds": 150, "T": 61, "K": 14, "hinge": True},
        # An arm's replanning from its measured state to a goal at rest: boundary conditions, states in arrays.
        {"name": "replan", "kind": "replan", "robot": "arm7", "seeds": 100, "T": 33, "K": 9},
        # Different robots with different horizons in one batch, forward and backward.
        {"name": "uneven", "kind": "uneven", "each": 256, "lo": 16, "hi": 64},
        # Whole-body control's matrices: poses, four links' Jacobians, centre of mass and its Jacobian.
        {"name": "jacobians", "kind": "kinematics", "robot": "humanoid48+3kg", "B": 20011, "targets": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "gradient", "gradient", "trajopt", "replan", "uneven", "kinematics"])
    robot = rng.choice(["arm7", "tree23", "humanoid48", "humanoid48+3kg"])
    if kind == "forward":
        return {"kind": kind, "robot": robot, "B": _log(rng, 1, 131072), "bits": rng.random() < 0.3}
    if kind == "gradient":
        return {"kind": kind, "robot": robot, "B": _log(rng, 1, 99999)}
    if kind == "trajopt":
        T = rng.randint(16, 96)
        return {"kind": kind, "robot": robot, "seeds": _log(rng, 1, 48000 // T), "T": T, "K": rng.randint(6, 20), "hinge": rng.random() < 0.4}
    if kind == "replan":
        T = rng.randint(16, 96)
        return {"kind": kind, "robot": robot, "seeds": _log(rng, 1, 48000 // T), "T": T, "K": rng.randint(4, 20)}
    if kind == "uneven":
        lo = rng.randint(1, 32)
        return {"kind": kind, "each": _log(rng, 1, 256), "lo": lo, "hi": rng.randint(lo, 64)}
    return {"kind": kind, "robot": robot, "B": _log(rng, 1, 60000), "targets": rng.randint(1, 6)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
DT = 0.25  # knot interval of the trajectories
ETA = 0.02  # activation distance of the summed hinge
LIMIT = {"arm7": 150.0, "tree23": 300.0, "humanoid48": 300.0}  # torque limits, exceeded by few samples
WEIGHTS = {"w_coll": 1.0, "smooth": 0.01, "length": 1.0, "energy": 0.01}


def _maker(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    uniform = lambda r, *shape: (torch.rand(shape, generator=g, device="cuda") * 2 - 1) * r  # noqa: E731
    normal = lambda *shape: torch.randn(shape, generator=g, device="cuda")  # noqa: E731
    return uniform, normal


def _states(d, B, uniform):
    return [uniform(r, d.dof, B) for r in (math.pi, 2.0, 5.0)]


def _upstream(d, B, normal):
    return [normal(B, d.n, 12), normal(B, d.S, 3), normal(B), normal(d.dof, B)]


def _problems(case, seed):
    """(robot, horizon) of each problem of an uneven batch; the mix is part of the case, the states are the seed's."""
    rng = np.random.default_rng(case["each"] * 10007 + case["lo"] * 101 + case["hi"])
    robot = np.repeat(np.arange(3), case["each"])
    rng.shuffle(robot)
    return [(int(r), int(h)) for r, h in zip(robot, rng.integers(case["lo"], case["hi"] + 1, len(robot)))]


UNEVEN = ("arm7", "tree23", "humanoid48")


def _targets(d, count):
    """Links whose Jacobians are wanted: the last links of the limbs first."""
    leaves = [k for k in range(d.n) if k not in set(d.parent.tolist())]
    return sorted((leaves + [k for k in range(d.n - 1, -1, -1) if k not in leaves])[:count])


def _dt_cost(case):
    return DT * (case["K"] - 3) / (case["T"] - 1)


def _inputs(case, seed):
    """The tensors of a case from its seed, in the library's layouts."""
    uniform, normal = _maker(seed)
    s = dict(case)
    if case["kind"] == "uneven":
        s["problems"] = _problems(case, seed)
        descs = [describe(UNEVEN[r]) for r, _ in s["problems"]]
        total = [sum(f(d) * h for d, (_, h) in zip(descs, s["problems"]))
                 for f in (lambda d: d.dof, lambda d: 12 * d.n, lambda d: 3 * d.S, lambda d: 1)]
        s["q"], s["qd"], s["qdd"] = (uniform(r, total[0]) for r in (math.pi, 2.0, 5.0))
        s["g_pose"], s["g_sphere"], s["g_dmin"], s["g_tau"] = normal(total[1]), normal(total[2]), normal(total[3]), normal(total[0])
        return s
    d = describe(case["robot"])
    if case["kind"] in ("forward", "gradient", "kinematics"):
        s["q"], s["qd"], s["qdd"] = _states(d, case["B"], uniform)
        if case["kind"] == "gradient":
            s["up"] = _upstream(d, case["B"], normal)
        return s
    s["U"] = uniform(math.pi / 2, case["seeds"], d.dof, case["K"])
    limit = LIMIT[case["robot"].split("+")[0]]
    s["lo"], s["hi"] = (torch.full((d.dof,), v, device="cuda") for v in (-limit, limit))
    if case["kind"] == "replan":
        start = torch.stack([uniform(r, case["seeds"], d.dof) for r in (math.pi / 2, 1.0, 1.0)], -1)
        s["start"] = start.contiguous()
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "uneven":
        s["robots"] = [wbe.Robot(describe(r)) for r in UNEVEN]
        s["batch"] = b = wbe.Batch(s["robots"], s["problems"])
        s["out"] = {"pose": b.empty("pose"), "sphere": b.empty("sphere"), "dmin": b.empty("config"),
                    "worst": b.empty("config", torch.int32), "tau": b.empty("joint")}
        s["grads"] = [b.empty("joint") for _ in range(3)]
        return s
    s["rob"] = wbe.Robot(describe(case["robot"]))
    if kind == "gradient":
        for k in ("q", "qd", "qdd"):
            s[k].requires_grad_(True)
    if kind == "kinematics":
        s["links"] = _targets(describe(case["robot"]), case["targets"])
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------


def _run_forward(s):
    o = s["rob"].eval(s["q"], s["qd"], s["qdd"], bits=s["bits"])
    return {k: v for k, v in o.items() if v is not None}


def _run_gradient(s):
    pose, sphere, dmin, tau, worst = wbe.whole_body_eval(s["rob"], s["q"], s["qd"], s["qdd"])
    gq, gqd, gqdd = torch.autograd.grad((pose, sphere, dmin, tau), (s["q"], s["qd"], s["qdd"]), s["up"])
    return {"pose": pose, "sphere": sphere, "dmin": dmin, "tau": tau, "worst": worst, "gq": gq, "gqd": gqd, "gqdd": gqdd}


def _run_trajopt(s):
    rob, U, T, dt = s["rob"], s["U"], s["T"], DT
    o = rob.eval_spline(U, T, dt, sphere=False, dmin=False)
    w = dict(WEIGHTS, dt_cost=_dt_cost(s))
    r = {"tau": o["tau"]}
    if s["hinge"]:
        r["hinge"], g_sphere = rob.self_collision_hinge(o["pose"], ETA)
        near = {"g_sphere": g_sphere}
    else:
        c = rob.self_collision(o["pose"], sphere=False, diff=True)
        r["dmin"], r["worst"] = c["dmin"], c["worst"]
        near = {"d_min": c["dmin"], "worst": c["worst"], "worst_diff": c["diff"]}
    gq, gqd, gqdd, r["cost"] = rob.eval_backward_spline_cost(U, T, dt, o["tau"], s["lo"], s["hi"], **w, **near)
    r["gU"] = wbe.bspline_backward(gq, gqd, gqdd, s["seeds"], s["K"], T, dt)
    return r


def _run_replan(s):
    rob, U, T, K, dt = s["rob"], s["U"], s["T"], s["K"], DT
    q, qd, qdd = wbe.bspline_eval(U, T, dt, start=s["start"], end_static=True)
    o = rob.eval(q, qd, qdd, sphere=False)
    gq, gqd, gqdd, cost = rob.eval_backward_cost(q, qd, qdd, o["tau"], s["lo"], s["hi"], **WEIGHTS, dt=_dt_cost(s), d_min=o["dmin"],
                                                 worst=o["worst"])
    gU, _ = wbe.bspline_backward_bc(gq, gqd, gqdd, s["seeds"], K, T, dt, has_start=True, end_static=True, want_start=False)
    return {"q": q, "tau": o["tau"], "dmin": o["dmin"], "worst": o["worst"], "cost": cost, "gU": gU}


def _run_uneven(s):
    o, g = s["out"], s["grads"]
    s["batch"].eval(s["q"], s["qd"], s["qdd"], o["pose"], o["sphere"], o["dmin"], o["worst"], o["tau"])
    s["batch"].eval_backward(s["q"], s["qd"], s["qdd"], o["worst"], s["g_pose"], s["g_sphere"], s["g_dmin"], s["g_tau"], *g)
    return dict(o, gq=g[0], gqd=g[1], gqdd=g[2])


def _run_kinematics(s):
    o = s["rob"].eval(s["q"], sphere=False, dmin=False, tau=False)
    jac, com, jac_com = s["rob"].kinematics(o["pose"], s["links"])
    return {"pose": o["pose"], "jac": jac, "com": com, "jac_com": jac_com}


_RUN = {"forward": _run_forward, "gradient": _run_gradient, "trajopt": _run_trajopt, "replan": _run_replan, "uneven": _run_uneven,
        "kinematics": _run_kinematics}


def run(state):
    return _RUN[state["kind"]](state)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------


def _one(d, forward=True, backward=False, pose=True, sphere=True, pairs=True, tau=True):
    """Bytes and operations of one configuration: joint states in, outputs out, and with `backward` the upstream gradients in and the
    joint gradients out.  The pair stage counts its spheres and one distance a sphere: how many more it needs depends on the values."""
    byte = flop = 0
    if forward:
        byte += 4 * ((3 if tau else 1) * d.dof + 12 * d.n * pose + 3 * d.S * sphere + 2 * pairs + d.dof * tau)
        flop += 150 * d.moving + (330 * d.n if tau else 0) + (29 * d.S if pairs or sphere else 0)
    if backward:
        byte += 4 * (12 * d.n + 3 * d.S + 1 + 4 * d.dof)
        flop += 1050 * d.n + 15 * d.S
    return np.array([byte, flop], np.float64)


def work(case):
    kind = case["kind"]
    if kind == "uneven":
        total = sum(_one(describe(UNEVEN[r]), backward=True) * h for r, h in _problems(case, 0))
    else:
        d = describe(case["robot"])
        if kind == "forward":
            total = (_one(d) + [4 * ((d.P + 31) // 32) * case["bits"], 0]) * case["B"]
        elif kind == "gradient":
            total = _one(d, backward=True) * case["B"]
        elif kind == "kinematics":
            total = (_one(d, sphere=False, pairs=False, tau=False) + [4 * (6 * d.dof * case["targets"] + 3 + 3 * d.dof), 60 * d.dof]) * case["B"]
        else:  # control points in, cost, torques and control-point gradient out; the poses in between need not leave the chip
            samples, knots = case["seeds"] * case["T"], case["seeds"] * d.dof * case["K"]
            flops = _one(d, pose=False, backward=True)[1] + 100 * d.dof
            total = np.array([4 * (2 * knots + samples * (d.dof * (2 if kind == "replan" else 1) + 3)), flops * samples], np.float64)
    return {"bytes": float(total[0]), "flops": float(total[1])}


# ---------------------------------------------------------------------------
# the same in 64 bits, with plain torch
# ---------------------------------------------------------------------------


def _f64(x):
    return torch.as_tensor(np.asarray(x), dtype=torch.float64, device="cuda")


def _mat(v):
    """[b][3] -> the matrix of its cross product."""
    z = torch.zeros_like(v[..., 0])
    return torch.stack([z, -v[..., 2], v[..., 1], v[..., 2], z, -v[..., 0], -v[..., 1], v[..., 0], z], -1).reshape(*v.shape[:-1], 3, 3)


def _times(R, x):
    return (R @ x.unsqueeze(-1)).squeeze(-1)


def _body(d, q, qd=None, qdd=None):
    """World rotations [b][n][3][3], origins [b][n][3] and joint torques [dof][b] of revolute trees (Newton-Euler in the world frame)."""
    b = q.shape[1]
    R, p, w, al, acc, F, N = ([None] * d.n for _ in range(7))
    axis, off, com = _f64(d.axis), _f64(d.T_fixed[:, 9:]), _f64(d.com)
    eye = torch.eye(3, dtype=torch.float64, device="cuda")
    cross = torch.linalg.cross
    zero = torch.zeros(b, 3, dtype=torch.float64, device="cuda")
    masses = [[(float(d.mass[k]), com[k], _f64(d.Icom[k][[0, 3, 4, 3, 1, 5, 4, 5, 2]].reshape(3, 3)))]
              + [(float(m), _f64(x), None) for l, m, x in zip(d.pm_link, d.pm_mass, d.pm_pos) if l == k] for k in range(d.n)]
    for k in range(d.n):
        pa, j = int(d.parent[k]), int(d.jidx[k])
        Rp, pp = (R[pa], p[pa]) if pa >= 0 else (eye.expand(b, 3, 3), zero)
        r = _times(Rp, off[k].expand(b, 3))
        p[k] = pp + r
        if j >= 0:
            K = _mat(axis[k])
            R[k] = Rp @ (eye + torch.sin(q[j])[:, None, None] * K + (1 - torch.cos(q[j]))[:, None, None] * (K @ K))
        else:
            R[k] = Rp
        if qd is None:
            continue
        wp, ap, cp = (w[pa], al[pa], acc[pa]) if pa >= 0 else (zero, zero, zero - _f64(d.gravity))
        acc[k] = cp + cross(ap, r) + cross(wp, cross(wp, r))
        if j >= 0:
            s = _times(R[k], axis[k].expand(b, 3))
            w[k] = wp + s * qd[j][:, None]
            al[k] = ap + s * qdd[j][:, None] + cross(wp, s * qd[j][:, None])
        else:
            w[k], al[k] = wp, ap
        F[k], N[k] = zero, zero
        for m, c, I in masses[k]:
            c = _times(R[k], c.expand(b, 3))
            f = m * (acc[k] + cross(al[k], c) + cross(w[k], cross(w[k], c)))
            F[k], N[k] = F[k] + f, N[k] + cross(c, f)
            if I is not None:
                Iw = R[k] @ I @ R[k].transpose(1, 2)
                N[k] = N[k] + _times(Iw, al[k]) + cross(w[k], _times(Iw, w[k]))
    tau = [None] * d.dof
    if qd is not None:
        for k in range(d.n - 1, -1, -1):
            pa, j = int(d.parent[k]), int(d.jidx[k])
            if j >= 0:
                tau[j] = (_times(R[k], axis[k].expand(b, 3)) * N[k]).sum(-1)
            if pa >= 0:
                F[pa], N[pa] = F[pa] + F[k], N[pa] + N[k] + cross(p[k] - p[pa], F[k])
    return torch.stack(R, 1), torch.stack(p, 1), torch.stack(tau) if qd is not None else None


def _centres(d, R, p):
    link = torch.as_tensor(d.sph_link, device="cuda", dtype=torch.long)
    return (R[:, link] @ _f64(d.sph_c)[None, :, :, None]).squeeze(-1) + p[:, link]


@functools.lru_cache(maxsize=None)
def _mask(name):
    d = describe(name)
    m = torch.zeros(d.S, d.S, dtype=torch.bool, device="cuda")
    ij = torch.as_tensor(d.pairs, device="cuda", dtype=torch.long)
    m[ij[:, 0], ij[:, 1]] = True
    return m


def _distances(name, c):
    """Signed distances of the masked pairs as a matrix [b][S][S], infinite elsewhere."""
    d, r = describe(name), _f64(describe(name).sph_r)
    d2 = sum((c[:, :, None, k] - c[:, None, :, k]) ** 2 for k in range(3))
    m = _mask(name)
    return torch.where(m, torch.where(m, d2, 1.0).sqrt() - r[:, None] - r[None, :], math.inf)


def _worst(name, c):
    """Least signed distance, differentiable through the pair that has it."""
    d = describe(name)
    with torch.no_grad():
        at = _distances(name, c).flatten(1).argmin(1)
    i, j = at // d.S, at % d.S
    row = torch.arange(len(c), device="cuda")
    r = _f64(d.sph_r)
    return (c[row, i] - c[row, j]).norm(dim=-1) - r[i] - r[j]


def _pose12(R, p):
    return torch.cat([R.flatten(2), p], -1)


def _spline_rows(K, T, dt):
    """The matrices [T][K] that take control points to positions, velocities and accelerations."""
    t = np.arange(T) * (K - 3)
    seg = np.minimum(t // (T - 1), K - 4)
    a = (t - seg * (T - 1)) / (T - 1)
    C = np.array([[-1, 3, -3, 1], [3, -6, 3, 0], [-3, 0, 3, 0], [1, 4, 1, 0]]) / 6.0
    one, none = np.ones(T), np.zeros(T)
    rows = [np.stack(x, 1) @ C for x in ([a ** 3, a ** 2, a, one], [3 * a ** 2 / dt, 2 * a / dt, one / dt, none],
                                         [6 * a / dt ** 2, 2 * one / dt ** 2, none, none])]
    out = np.zeros((3, T, K))
    for l in range(4):
        out[:, np.arange(T), seg + l] = np.stack([x[:, l] for x in rows])
    return _f64(out)


def _cost(d, case, q, qd, qdd, tau):
    limit, w = LIMIT[case["robot"].split("+")[0]], WEIGHTS
    c = (tau - limit).clamp(min=0).sum(0) + (-limit - tau).clamp(min=0).sum(0)
    return c + w["smooth"] * (qdd ** 2).sum(0) + w["length"] * (qd ** 2).sum(0) + w["energy"] * ((qd * tau * _dt_cost(case)) ** 2).sum(0)


def _exact_rows(name, q, qd, qdd, up):
    """Outputs and gradients of a block of configurations."""
    d = describe(name)
    leaf = [x.double().requires_grad_(up is not None) for x in (q, qd, qdd)]
    R, p, tau = _body(d, *leaf)
    c = _centres(d, R, p)
    o = {"pose": _pose12(R, p), "sphere": c, "dmin": _worst(name, c), "tau": tau}
    if up is not None:
        o["gq"], o["gqd"], o["gqdd"] = torch.autograd.grad([o["pose"], o["sphere"], o["dmin"], o["tau"]], leaf, [u.double() for u in up])
    return {k: v.detach() for k, v in o.items()}


def _joined(parts, joint):
    return {k: torch.cat([x[k] for x in parts], 1 if k in joint else 0) for k in parts[0]}


JOINT = ("tau", "q", "gq", "gqd", "gqdd")


def _exact_states(case, s):
    up, parts = s.get("up"), []
    step = 8192 if case["robot"] == "arm7" else 2048
    for b in range(0, case["B"], step):
        e = slice(b, b + step)
        parts.append(_exact_rows(case["robot"], s["q"][:, e], s["qd"][:, e], s["qdd"][:, e],
                                 up and [up[0][e], up[1][e], up[2][e], up[3][:, e]]))
    o = dict(_joined(parts, JOINT), worst=None)
    return dict(o, bits=None) if case.get("bits") else o


def _exact_spline(case, s):
    """Trajectory cases: gradients of the summed cost through the spline."""
    name, T, K, replan = case["robot"], case["T"], case["K"], case["kind"] == "replan"
    d = describe(name)
    rows = _spline_rows(K + 6 * replan, T, DT)
    each = max(1, (512 if case.get("hinge") else 2048) // T)
    parts = []
    for t in range(0, case["seeds"], each):
        U = s["U"][t:t + each].double().requires_grad_(True)
        X = U
        if replan:  # the knots of the start state before, the goal repeated after
            th, v, a = (s["start"][t:t + each].double()[..., k:k + 1] for k in range(3))
            X = torch.cat([th - a * DT ** 2 / 6, th + v * DT + a * DT ** 2 / 3, th + 2 * v * DT + 11 * a * DT ** 2 / 6, U]
                          + [U[..., -1:]] * 3, -1)
        q, qd, qdd = (torch.einsum("tk,sdk->dst", r, X).flatten(1) for r in rows)
        R, p, tau = _body(d, q, qd, qdd)
        c = _centres(d, R, p)
        cost = _cost(d, case, q, qd, qdd, tau)
        o = {"tau": tau}
        if case.get("hinge"):
            o["hinge"] = (ETA - _distances(name, c)).clamp(min=0).flatten(1).sum(1)
            total = (cost + o["hinge"]).sum()
        else:
            o["dmin"] = _worst(name, c)
            cost = cost + WEIGHTS["w_coll"] * (-o["dmin"]).clamp(min=0)
            total = cost.sum()
        o["cost"] = cost
        if replan:
            o["q"] = q
        o["gU"], = torch.autograd.grad(total, U)
        parts.append({k: v.detach() for k, v in o.items()})
    o = _joined(parts, JOINT)
    return o if case.get("hinge") else dict(o, worst=None)


def _exact_uneven(case, s):
    """All horizons of one robot at a time, then back to the packed order."""
    at, place = [0, 0, 0, 0], []  # offsets of joints, poses, spheres, configurations
    for r, h in s["problems"]:
        d = describe(UNEVEN[r])
        place.append((r, h, list(at)))
        at = [a + n for a, n in zip(at, (d.dof * h, 12 * d.n * h, 3 * d.S * h, h))]
    new = lambda k: torch.zeros(at[k], dtype=torch.float64, device="cuda")  # noqa: E731
    which = {"pose": 1, "sphere": 2, "dmin": 3, "tau": 0, "gq": 0, "gqd": 0, "gqdd": 0}
    out = {k: new(i) for k, i in which.items()}
    for r, name in enumerate(UNEVEN):
        d, mine, n = describe(name), [(h, o) for i, h, o in place if i == r], 0
        cut = lambda x, k, size: x[k:k + size]  # noqa: E731
        joint = {k: torch.cat([cut(s[k], o[0], d.dof * h).reshape(d.dof, h) for h, o in mine], 1) for k in ("q", "qd", "qdd", "g_tau")}
        gp, gs, gd = (torch.cat([cut(s[k], o[i], w * h).reshape((h,) + shape) for h, o in mine])
                      for k, i, w, shape in (("g_pose", 1, 12 * d.n, (d.n, 12)), ("g_sphere", 2, 3 * d.S, (d.S, 3)), ("g_dmin", 3, 1, ())))
        e = _exact_states({"robot": name, "B": joint["q"].shape[1]}, dict(joint, up=[gp, gs, gd, joint["g_tau"]]))
        for h, o in mine:
            for k, i in which.items():
                x = (e[k][:, n:n + h] if k in JOINT else e[k][n:n + h]).reshape(-1)
                out[k][o[i]:o[i] + x.numel()] = x
            n += h
    return dict(out, worst=None)


def _exact_kinematics(case, s):
    name = case["robot"]
    d, links = describe(name), _targets(describe(name), case["targets"])
    parent, below = d.parent.tolist(), np.eye(d.n, dtype=bool)  # below[k][l]: link l is link k or hangs from it
    for l in range(d.n):
        a = parent[l]
        while a >= 0:
            below[a, l] = True
            a = parent[a]
    m = _f64(d.mass)
    for l, x in zip(d.pm_link, d.pm_mass):
        m[l] += float(x)
    moment = _f64(d.mass)[:, None] * _f64(d.com)
    for l, x, y in zip(d.pm_link, d.pm_mass, d.pm_pos):
        moment[l] += float(x) * _f64(y)
    moving = [int(np.nonzero(d.jidx == j)[0][0]) for j in range(d.dof)]
    tree = _f64(below)[moving]
    parts = []
    for b in range(0, case["B"], 4096):
        R, p, _ = _body(d, s["q"][:, b:b + 4096].double())
        ax = (R @ _f64(d.axis)[None, :, :, None]).squeeze(-1)[:, moving]
        mx = m[None, :, None] * p + (R @ moment[None, :, :, None]).squeeze(-1)
        jac = torch.zeros(len(p), len(links), 6, d.dof, dtype=torch.float64, device="cuda")
        for t, e in enumerate(links):
            on = _f64(below[moving, e])[None, :, None]
            jac[:, t, :3] = (torch.linalg.cross(ax, p[:, e:e + 1] - p[:, moving]) * on).transpose(1, 2)
            jac[:, t, 3:] = (ax * on).transpose(1, 2)
        sums = torch.einsum("jk,bkc->bjc", tree, mx) - (tree @ m)[None, :, None] * p[:, moving]
        parts.append({"pose": _pose12(R, p), "jac": jac, "com": mx.sum(1) / m.sum(),
                      "jac_com": (torch.linalg.cross(ax, sums) / m.sum()).transpose(1, 2)})
    return _joined(parts, ())


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradient") and case["B"] > 140000:
        return None
    s = _inputs(case, seed)
    if kind == "uneven":
        return _exact_uneven(case, s)
    if kind == "kinematics":
        return _exact_kinematics(case, s)
    return _exact_states(case, s) if kind in ("forward", "gradient") else _exact_spline(case, s)
