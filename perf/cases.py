"""The work this framework is used for, as cases with inputs, one pass and its outputs.

A case is a planning query (Planner, kpx_plan_static), many of them at once
(BatchPlanner, serve.Server), or the refinement post-pass (refine.evaluate,
refine.validate), in the sizes of the repository's own configurations, and
around them.

The planner grows a tree by comparing FP32 costs, so what it returns is a
sequence of decisions and has no 64-bit value of its own; the refinement's
objective, gradient and edge costs do (``exact``).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2602_02846_gb300 as kpx
from paper_2602_02846_gb300 import refine, scenes, serve

# counters of kpx_iter_stats that are results (its clock stamps are not, and
# total_box_tests counts work that depends on the obstacle grid's resolution)
STATS = ("status", "iter", "n_nodes", "n_active", "n_inactive", "n_terminal", "lam", "first_solution_iter",
         "candidates", "winners", "total_candidates", "total_winners")
# with KPX_FLAG_EARLY_REJECT these depend on the order in which rollouts end
STATS_EVERY_ROLLOUT = ("valid", "total_valid", "total_steps")

# arithmetic of one integration step (dynamics, integrator, bounds; FMA = 2,
# sine or cosine = 1) per system and scheme
STEP_FLOPS = {(scenes.DI6, scenes.EULER): 22, (scenes.DI6, scenes.RK4): 60, (scenes.DUBINS6, scenes.EULER): 24,
              (scenes.DUBINS6, scenes.RK4): 96, (scenes.QUAD12, scenes.EULER): 80, (scenes.QUAD12, scenes.RK4): 270}


def listed():
    return [
        # the smallest call: a control loop that may not allocate replans a
        # point mass among 20 boxes in the library's static memory
        dict(name="static_di", kind="static", system="di", boxes=20, walls=False, cap=16384, lam=16, grid=12, sub=2,
             iters=24, integ=scenes.EULER, cost=scenes.COST_PATH_LENGTH, early=False, aniso=False, active=1000),
        # a new query from host arrays (create, iterate, read the solution,
        # destroy) for a quadcopter in a room of 120 boxes, as a server
        # without batching answers it; the tree fills its capacity
        dict(name="query_quad_room", kind="query", system="quad", boxes=120, walls=False, cap=1 << 16, lam=32,
             grid=16, sub=4, iters=64, integ=scenes.RK4, cost=scenes.COST_EFFORT_DURATION, early=False, aniso=False,
             active=900),
        # replanning with a kept planner: the double integrator on the grid
        # it is solved on
        dict(name="plan_di_room", kind="plan", system="di", boxes=20, walls=False, cap=32768, lam=16, grid=16, sub=2,
             iters=200, integ=scenes.EULER, cost=scenes.COST_PATH_LENGTH, early=False, aniso=False, active=160),
        # the airplane in the 300-column forest: a tree of about a hundred
        # nodes, an iteration's latency
        dict(name="plan_dubins_forest", kind="plan", system="dubins", boxes=300, walls=False, cap=1 << 20, lam=64,
             grid=16, sub=4, iters=200, integ=scenes.RK4, cost=scenes.COST_DURATION, early=False, aniso=False,
             active=46),
        # the airplane among 30 columns: the tree covers the workspace
        dict(name="plan_dubins_open", kind="plan", system="dubins", boxes=30, walls=False, cap=1 << 20, lam=64,
             grid=16, sub=4, iters=100, integ=scenes.RK4, cost=scenes.COST_DURATION, early=False, aniso=False,
             active=1300),
        # the quadcopter in the 1,000-box building (the benchmark's workload)
        dict(name="plan_quad_building", kind="plan", system="quad", boxes=964, walls=True, cap=1 << 22, lam=128,
             grid=16, sub=4, iters=200, integ=scenes.RK4, cost=scenes.COST_EFFORT_DURATION, early=False, aniso=False,
             active=12000),
        # the same among 1,000 boxes without walls: a tree of millions of nodes
        dict(name="plan_quad_clutter", kind="plan", system="quad", boxes=1000, walls=False, cap=1 << 22, lam=128,
             grid=16, sub=4, iters=120, integ=scenes.RK4, cost=scenes.COST_EFFORT_DURATION, early=False, aniso=False,
             active=160000),
        # many problems of uneven size planned together
        dict(name="batch_mixed", kind="batch", problems=48, iters=100),
        # queries through the request loop's slots, a backlog served at once
        dict(name="serve_backlog", kind="serve", problems=24, iters=64, slots=4),
        # refinement of trajectories of the length the planner returns:
        # objective and gradient
        dict(name="refine_returned", kind="refine", count=256, seg_lo=8, seg_hi=40, k_lo=10, k_hi=60, boxes=1000),
        # refinement of long horizons (the refinement benchmark's batch)
        dict(name="refine_long", kind="refine", count=4096, seg_lo=64, seg_hi=512, k_lo=10, k_hi=60, boxes=1000),
        # scoring candidate controls: objective without gradient, and
        # re-validation with the planner's stepper
        dict(name="score_candidates", kind="score", count=512, seg_lo=16, seg_hi=96, k_lo=10, k_hi=30, boxes=1000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: mostly single plans, every system,
    scheme, edge cost and option among them."""
    kind = rng.choice(["plan", "plan", "plan", "query", "static", "batch", "serve", "refine", "refine", "score"])
    if kind in ("plan", "query", "static"):
        system = rng.choice(["di", "dubins", "quad"]) if kind != "static" else "di"
        lam = rng.choice([0, 8, 16, 16, 31, 32, 64, 64, 100, 128])
        c = dict(kind=kind, system=system, walls=False, integ=scenes.EULER if system == "di" else scenes.RK4,
                 early=rng.random() < 0.2, aniso=False, boxes=rng.choice([0, _log_int(rng, 4, 600)]), lam=lam,
                 iters=_log_int(rng, 10, 200), grid=rng.randint(8, 20), sub=rng.randint(2, 5),
                 cap=_log_int(rng, 1 << 13, 1 << 20))
        if system == "di":
            c["cost"] = rng.choice([scenes.COST_PATH_LENGTH, scenes.COST_DURATION])
            c["sub"] = rng.randint(2, 3)
        elif system == "dubins":
            c["cost"] = rng.choice([scenes.COST_DURATION, scenes.COST_PATH_LENGTH])
        else:
            c["cost"] = rng.choice([scenes.COST_EFFORT_DURATION, scenes.COST_DURATION, scenes.COST_PATH_LENGTH])
            c["walls"] = rng.random() < 0.4
            c["aniso"] = rng.random() < 0.3
            c["iters"] = _log_int(rng, 10, 120)
            c["sub"] = rng.randint(2, 4)
        if rng.random() < 0.15:  # the scheme that is not the system's usual one
            c["integ"] = scenes.RK4 if c["integ"] == scenes.EULER else scenes.EULER
        if kind == "static":  # what the static memory holds
            c["cap"] = _log_int(rng, 1 << 14, 1 << 15)
            c["lam"] = rng.choice([0, 16, 23, 32])
            c["grid"], c["sub"], c["boxes"] = rng.randint(12, 15), 2, rng.choice([0, 7, 20, 33])
            c["iters"], c["early"] = _log_int(rng, 24, 64), False
        regions = c["grid"] ** 3 * (c["sub"] if system == "dubins" else c["sub"] ** 3)
        c["active"] = max(1, min(regions, c["cap"]) // 20)
        return c
    if kind == "batch":
        return dict(kind=kind, problems=rng.randint(2, 48), iters=_log_int(rng, 10, 100))
    if kind == "serve":
        return dict(kind=kind, problems=rng.randint(3, 24), iters=_log_int(rng, 8, 64), slots=rng.randint(1, 6))
    seg_hi = _log_int(rng, 2, 512)
    count = _log_int(rng, 1, 4096) if seg_hi < 200 else _log_int(rng, 1, 1500)
    if kind == "score":
        seg_hi, count = min(seg_hi, 96), min(count, 1024)
    k_lo = rng.randint(1, 10)
    return dict(kind=kind, count=count, seg_lo=rng.randint(1, seg_hi), seg_hi=seg_hi, k_lo=k_lo,
                k_hi=rng.randint(k_lo, 60), boxes=rng.choice([0, _log_int(rng, 3, 1000), 1000]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _problem(case, seed):
    s = case["system"]
    kw = dict(tree_cap=case["cap"], lam=case["lam"], iterations=case["iters"])
    if s == "di":
        p = scenes.di_scene(seed, n_obstacles=case["boxes"], grid_pos=case["grid"], grid_vel=case["sub"], **kw)
    elif s == "dubins":
        p = scenes.dubins_scene(seed, n_obstacles=case["boxes"], grid_pos=case["grid"], grid_yaw=case["sub"], **kw)
    else:
        p = scenes.quad_scene(seed, clutter=case["boxes"], grid_pos=case["grid"], grid_vel=case["sub"],
                              certify=False, walls=case["walls"], **kw)
        if case["aniso"]:
            par = list(p.param)
            par[3], par[4] = scenes.f32(1.25 * par[2]), scenes.f32(1.75 * par[2])
            p = p.replace(param=par)
    return p.replace(integ=case["integ"], cost_kind=case["cost"])


def _controls(case, seed):
    """Control sequences from the quadcopter's start: odd rows drift off with
    random thrusts and torques (the optimiser's far iterates), even rows keep
    station (groups of four segments that cancel), as trajectories that stay
    valid do."""
    prob = scenes.quad_scene(seed, clutter=max(0, case["boxes"] - 36), certify=False)
    prob = prob.replace(goal_c=[float(v) for v in prob.start[:3]])
    rng = np.random.default_rng([0xCA5E, seed])
    B, S = case["count"], case["seg_hi"]
    n_seg = rng.integers(case["seg_lo"], S + 1, B).astype(np.int32)
    steps = rng.integers(case["k_lo"], case["k_hi"] + 1, (B, S)).astype(np.int32)
    mg = float(np.float32(scenes.QUAD_MASS * scenes.QUAD_G))
    dev = rng.uniform(-0.5, 0.5, (B, S))
    tau = rng.uniform(-0.001, 0.001, (B, S, 3))
    sign = np.array([1.0, -1.0, -1.0, 1.0])[np.arange(S) % 4]
    lead = np.arange(S) // 4 * 4
    even = np.arange(B) % 2 == 0
    dev[even] = 0.4 * dev[even][:, lead] * sign
    tau[even] = 0.05 * tau[even][:, lead] * sign[None, :, None]
    steps[even] = np.minimum(steps[even][:, lead], 30)
    u = np.concatenate([(mg + dev)[:, :, None], tau], axis=2).astype(np.float32)
    live = np.arange(S)[None, :] < n_seg[:, None]
    u *= live[:, :, None]
    steps *= live
    x0 = np.tile(np.asarray(prob.start, np.float32), (B, 1))
    obs = np.asarray(prob.obstacles, np.float32)[:case["boxes"]]
    return prob, x0, u, steps, n_seg, obs


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, case=case)
    if kind in ("plan", "query", "static"):
        prob = st["prob"] = _problem(case, seed)
        st["flags"] = kpx.KPX_FLAG_EARLY_REJECT if case["early"] else 0
        st["stats"] = STATS if case["early"] else STATS + STATS_EVERY_ROLLOUT
        if kind != "static":  # the program's own device buffer, cleared once: rows past the tree stay zero
            size = kpx.kpx_workspace_size(prob, st["flags"])
            st["workspace"] = torch.zeros(size + 256, dtype=torch.uint8, device="cuda")
        if kind == "plan":
            st["planner"] = kpx.Planner(prob, flags=st["flags"], workspace=st["workspace"])
    elif kind == "batch":
        st["batch"] = kpx.BatchPlanner(scenes.mixed_batch(case["problems"], seed, case["iters"]))
    elif kind == "serve":
        st["server"] = serve.Server.create(4 << 30, slots_per_class=case["slots"])
        st["problems"] = scenes.mixed_batch(case["problems"], seed, case["iters"])
    else:
        prob, x0, u, steps, n_seg, obs = _controls(case, seed)
        st["spec"] = refine.default_cost(prob)
        st["batch"] = refine.Batch(prob, x0, u, steps, n_seg, obstacles=obs)
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _solutions(trajs, iters):
    """Trajectories as arrays of one size (an iteration adds one segment to a
    path at most), zero past their ends; length -1 and cost inf: no solution."""
    P = len(trajs)
    out = dict(length=np.full(P, -1, np.int32), cost=np.full(P, np.inf, np.float32),
               states=np.zeros((P, iters + 1, 12), np.float32), controls=np.zeros((P, iters, 4), np.float32),
               steps=np.zeros((P, iters), np.int32))
    for i, tr in enumerate(trajs):
        if tr is not None:
            k = len(tr["steps"])
            out["length"][i], out["cost"][i] = k, tr["cost"]
            out["states"][i, :k + 1, :tr["states"].shape[1]] = tr["states"]
            out["controls"][i, :k, :tr["controls"].shape[1]] = tr["controls"]
            out["steps"][i, :k] = tr["steps"]
    return out


def _tree(pl):
    """The tree as views of the workspace (kpx_layout)."""
    lay = pl.layout()
    base = pl.workspace.data_ptr()

    def view(ptr, count, dtype):
        off = int(ptr) - base
        return pl.workspace[off:off + count * dtype.itemsize].view(dtype)
    N = lay.N
    return dict(x=view(lay.x, lay.n * N, torch.float32), u=view(lay.u, lay.m * N, torch.float32),
                K=view(lay.K, N, torch.int16), parent=view(lay.parent, N, torch.int32),
                key=view(lay.key, N, torch.int64), region=view(lay.region, N, torch.int32),
                set=view(lay.set, N, torch.uint8), icount=view(lay.icount, N, torch.uint8),
                region_key=view(lay.region_key, lay.R, torch.int64))


def run(state):
    kind, case = state["kind"], state["case"]
    if kind in ("plan", "query"):
        if kind == "plan":
            pl = state["planner"]
            pl.reset()
        else:
            pl = kpx.Planner(state["prob"], flags=state["flags"], workspace=state["workspace"])
        st = pl.iterate(case["iters"], stats=True)
        out = _solutions([pl.best_trajectory()], case["iters"])
        out["stats"] = np.array([st[k] for k in state["stats"]], np.int64)
        out["best_cost"] = np.float32(st["best_cost"])
        out.update(_tree(pl))
        if kind == "query":
            pl.close()
        return out
    if kind == "static":
        status, tr = kpx.kpx_plan_static(state["prob"], case["iters"], stream=torch.cuda.current_stream(),
                                         flags=state["flags"])
        return dict(_solutions([tr], case["iters"]), status=status)
    if kind == "batch":
        b = state["batch"]
        b.reset()
        b.iterate(case["iters"])
        slots = b.poll()
        out = _solutions([b.member(i).best_trajectory() if s["goal_cost"] is not None else None
                          for i, s in enumerate(slots)], case["iters"])
        out["slots"] = np.array([[s["status"], s["iter"], s["n_nodes"], s["first_solution_iter"]] for s in slots])
        return out
    if kind == "serve":
        reqs = [serve.Request(i, p, 0.0, case["iters"]) for i, p in enumerate(state["problems"])]
        done = state["server"].serve(reqs, realtime=False)
        out = _solutions([o.trajectory for o in done], case["iters"])
        out["served"] = np.array([[o.status == "tree_full", o.status == "done", o.iterations, o.n_nodes,
                                   o.total_valid, o.first_solution_iter] for o in done])
        return out
    if kind == "refine":
        J, g = refine.evaluate(state["batch"], state["spec"], grad=True)
        return dict(J=J, grad=g)
    J = refine.evaluate(state["batch"], state["spec"])
    valid, cost, x_end = refine.validate(state["batch"])
    return dict(J=J, valid=valid, cost=cost, x_end=x_end)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Planning: the rollouts' arithmetic (|V_A| lambda rollouts an iteration,
    half of the mean step count each: an invalid point ends a rollout), and
    the tree rows written once.  ``active`` is about the mean |V_A| of the
    configuration.  Refinement: every step integrated once, with a gradient
    three times that for its reverse; inputs and outputs once."""
    kind = case["kind"]
    if kind in ("plan", "query", "static"):
        system = {"di": scenes.DI6, "dubins": scenes.DUBINS6, "quad": scenes.QUAD12}[case["system"]]
        n, m = scenes.STATE_DIM[system], scenes.CONTROL_DIM[system]
        mean_k = {"di": 17.5, "dubins": 15.0, "quad": 35.0}[case["system"]]
        rollouts = case["iters"] * (case["active"] * case["lam"] if case["lam"] else case["cap"])
        rows = min(case["cap"], case["iters"] * case["active"] // 4 + 1)
        return dict(bytes=24 * case["boxes"] + rows * (4 * n + 4 * m + 28),
                    flops=rollouts * mean_k / 2 * STEP_FLOPS[(system, case["integ"])])
    if kind in ("batch", "serve"):  # a third of the problems each system, capacities 2^14..2^20
        rollouts = case["problems"] * case["iters"] * 25000
        return dict(bytes=case["problems"] * (24 * 500 + 3000 * 80), flops=rollouts * (22 * 9 + 96 * 7 + 270 * 17) / 3)
    B, S = case["count"], case["seg_hi"]
    segs = B * (case["seg_lo"] + S) / 2
    steps = segs * (case["k_lo"] + case["k_hi"]) / 2
    inputs = segs * 20 + B * 52 + case["boxes"] * 24
    if kind == "refine":
        return dict(bytes=inputs + segs * 16 + B * 4, flops=steps * 4 * 328)
    return dict(bytes=inputs + B * 64, flops=steps * (328 + 270))


# ---------------------------------------------------------------------------
# 64-bit values of the refinement's outputs
# ---------------------------------------------------------------------------
def _deriv(x, u, mass, g, J):
    """x' = f(x, u) of the quadcopter, columns (p, roll, pitch, yaw, v, body rates)."""
    phi, th, psi = x[:, 3], x[:, 4], x[:, 5]
    p, q, r = x[:, 9], x[:, 10], x[:, 11]
    sp, cp, st, ct, ss, cs = phi.sin(), phi.cos(), th.sin(), th.cos(), psi.sin(), psi.cos()
    w = sp * q + cp * r
    a = u[:, 0] / mass
    return torch.stack([x[:, 6], x[:, 7], x[:, 8], p + st / ct * w, cp * q - sp * r, w / ct,
                        a * (cs * st * cp + ss * sp), a * (ss * st * cp - cs * sp), a * ct * cp - g,
                        (u[:, 1] - (J[2] - J[1]) * q * r) / J[0], (u[:, 2] - (J[0] - J[2]) * r * p) / J[1],
                        (u[:, 3] - (J[1] - J[0]) * p * q) / J[2]], dim=1)


def _penalty(pos, boxes, beta, margin):
    """Sum over boxes of softplus(margin - signed distance), per point."""
    total = torch.zeros(pos.shape[0], dtype=pos.dtype, device=pos.device)
    for b in boxes.split(64):
        lo, hi = b[None, :, :3], b[None, :, 3:]
        p = pos[:, None, :]
        off = torch.maximum(torch.maximum(lo - p, p - hi), torch.zeros((), dtype=pos.dtype, device=pos.device))
        d2 = (off * off).sum(-1)
        outside = d2 > 0
        depth = torch.minimum(p - lo, hi - p).amin(-1)
        d = torch.where(outside, torch.where(outside, d2, torch.ones_like(d2)).sqrt(), -depth)
        total = total + torch.nn.functional.softplus(beta * (margin - d), threshold=50.0).sum(1) / beta
    return total


def exact(case, seed):
    if case["kind"] not in ("refine", "score"):
        return None  # decisions on FP32 costs: no 64-bit value
    grad = case["kind"] == "refine"
    longest = case["seg_hi"] * case["k_hi"]
    if longest > 3000 or case["count"] * longest > 1 << 21:
        return None  # minutes of sequential 64-bit steps
    prob, x0, u, steps, n_seg, obs = _controls(case, seed)
    spec = refine.default_cost(prob)
    dev = torch.device("cuda")
    f64 = dict(dtype=torch.float64, device=dev)
    B, S = u.shape[:2]
    mass, g, J = prob.param[0], prob.param[1], prob.param[2:5]
    h = float(prob.h)
    uu = torch.as_tensor(u, **f64)
    uu.requires_grad_(grad)
    K = torch.as_tensor(steps.astype(np.int64), device=dev)
    boxes = torch.as_tensor(obs, **f64).reshape(-1, 6)
    live = torch.arange(S, device=dev)[None, :] < torch.as_tensor(n_seg, device=dev)[:, None]
    mg = float(np.float32(np.float32(mass) * np.float32(g)))
    tau_max = prob.param[5]
    effort = ((uu[:, :, 0] - mg) / mg) ** 2 + (uu[:, :, 1:] ** 2).sum(-1) / tau_max ** 2
    dur = K.to(torch.float64) * h
    edge = torch.where(live, dur * (1.0 + spec["w_effort"] * effort), torch.zeros((), **f64)).sum(1)
    # every trajectory's segment at every step; a finished one keeps its state
    ends = torch.cumsum(K, 1)
    total = ends[:, -1]
    n_steps = int(total.max())
    seg = torch.searchsorted(ends, torch.arange(n_steps, device=dev).repeat(B, 1), right=True).clamp(max=S - 1)
    x = torch.as_tensor(x0, **f64)
    rows = torch.arange(B, device=dev)
    points, owner = [], []
    with torch.set_grad_enabled(grad):
        for k in range(n_steps):
            uk = uu[rows, seg[:, k]]
            k1 = _deriv(x, uk, mass, g, J)
            k2 = _deriv(x + 0.5 * h * k1, uk, mass, g, J)
            k3 = _deriv(x + 0.5 * h * k2, uk, mass, g, J)
            k4 = _deriv(x + h * k3, uk, mass, g, J)
            xn = x + h / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
            run_k = k < total
            x = torch.where(run_k[:, None], xn, x)
            points.append(x[run_k, :3])
            owner.append(rows[run_k])
        pos, own = torch.cat(points) if points else x[:0, :3], torch.cat(owner) if owner else rows[:0]
        goal = torch.as_tensor(spec["goal"], **f64)
        pull = spec["w_goal"] * ((x[:, :3] - goal) ** 2).sum(1)
        # the penalty in chunks: its gradient at the points, then one reverse
        # pass through the rollout
        leaf = pos.detach()
        pen = torch.zeros(leaf.shape[0], **f64)
        gpos = torch.zeros_like(leaf)
        for i in range(0, leaf.shape[0], 1 << 16):
            q = leaf[i:i + (1 << 16)].clone().requires_grad_(grad)
            v = _penalty(q, boxes, spec["beta"], spec["margin"]) if len(boxes) else q[:, 0] * 0.0
            pen[i:i + (1 << 16)] = v.detach()
            if grad:
                gpos[i:i + (1 << 16)], = torch.autograd.grad(v.sum(), q)
        pen_sum = torch.zeros(B, **f64).index_add_(0, own, pen)
        Jv = (edge + pull).detach() + spec["w_obs"] * pen_sum
        if grad:
            ((edge + pull).sum() + spec["w_obs"] * (pos * gpos).sum()).backward()
            return dict(J=Jv, grad=uu.grad)
    # the re-validation's costs use the FP64 product of the FP32 mass and gravity
    mg64 = float(np.float32(mass)) * float(np.float32(g))
    e64 = ((uu[:, :, 0] - mg64) / mg64) ** 2 + (uu[:, :, 1:] ** 2).sum(-1) / tau_max ** 2
    cost = torch.where(live, dur * (1.0 + prob.w_effort * e64), torch.zeros((), **f64)).sum(1)
    return dict(J=Jv, valid=None, cost=cost, x_end=None)
