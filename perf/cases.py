"""Performance cases of the path optimiser: what a program that plans crane motions has the
library do, through its public entry points.

Each case is a dict of plain values; `prepare` makes what the program holds before the call
(scene, end points, candidates, and the planner, batch or solver it keeps), `run` is one pass,
`work` the bytes and operations a pass cannot do without, and `exact` the outputs in 64 bits
from plain torch where they have such a value. Scenes and sizes are those of the repository's
workloads (the 20-tree query, the 500-tree query, the dense forest, the differentiable form,
the batch of uneven queries, the grasp batch and the trajectory batch) and sizes between them.
"""
import math

import numpy as np
import torch

from paper_2503_14160_gb300 import autograd, workloads
from paper_2503_14160_gb300 import craneplan as cp

DEV = "cuda"
DENSITY = 1.66          # trees per m^2 of the larger scenes
W_C, W_L, LAMBDA_C = 100.0, 100.0, 1.0
SPREAD = (0.3, 0.15, 0.2, 0.25)   # candidate spread about the straight line, per joint
_stream = None


def listed():
    return [
        # The smallest call: a planner kept by a crane controller plans out to the log and back
        # among 20 trees (two new end-point pairs per pass): launches and latency count.
        dict(name="plan_small", kind="plan", N=256, K=8, S=32, T=50, trees=20, boxes=0, grid=0.0,
             sampler="factor", rule="paper", trips=2),
        # The single large query: 500 trees, polar index, factor-free tensor-core sampler.
        dict(name="plan_large", kind="plan", N=4096, K=16, S=64, T=100, trees=500, boxes=0, grid=0.5,
             sampler="elites", rule="paper", trips=2),
        # The dense forest, the largest call: 5000 spaced trees and 50 boxes (20 iterations of it).
        dict(name="plan_forest", kind="plan", N=65536, K=32, S=128, T=20, trees=5000, boxes=50, grid=0.5,
             sampler="factor", rule="paper", trips=1),
        # The CMA-ES update rule with the index-free evaluation, at an odd, middling size.
        dict(name="plan_cmaes", kind="plan", N=1001, K=11, S=50, T=40, trees=150, boxes=3, grid=0.0,
             sampler="factor", rule="cmaes", trips=2),
        # The serving form: uneven queries in one graph launch.
        dict(name="batch", kind="batch", queries=16, N_lo=1024, N_hi=16384, K_lo=8, K_hi=32, trees_lo=50,
             trees_hi=3000, S=64, T=20, mix=0),
        # A user's own candidates scored with every output (flags, terms, per-checkpoint depths),
        # ragged sizes, no index.
        dict(name="evaluate_outputs", kind="evaluate", N=3001, K=13, S=50, trees=300, boxes=10, grid=0.0,
             collision="spheres", outputs=True),
        # The convex-hull collision model on the single large query's population size.
        dict(name="evaluate_hulls", kind="evaluate", N=4096, K=16, S=64, trees=500, boxes=0, grid=0.0,
             collision="hulls", outputs=False),
        # Ranking, distribution update, factor and next sample for a program that scores the
        # dense forest's candidates itself.
        dict(name="update_sample", kind="update", N=65536, K=32),
        # The differentiable form through autograd: forward and backward over a population.
        dict(name="smooth_grad", kind="smooth", N=16384, K=32, S=64, trees=1000, boxes=0),
        # Gradient polish of the 64 best, nearly free of contact, before the hand-over to the
        # trajectory step (few candidates, ten steps of a length that descends in contact too).
        dict(name="polish", kind="polish", N=64, K=32, S=64, trees=20, boxes=0, steps=10, alpha=1e-6),
        # Goal configurations for a batch of grasp poses.
        dict(name="ik", kind="ik", N=16384, trees=20, restarts=8, iters=50),
        # The planned paths turned into trajectories (targets, starting point, solve).
        dict(name="trajectories", kind="traj", N=64, K=8, intervals=100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plan", "plan", "plan", "batch", "evaluate", "evaluate", "update", "smooth", "polish", "ik",
                       "traj"])
    K, S = rng.randint(8, 32), rng.randint(24, 128)
    if kind == "plan":
        N = _log(rng, 200, 65536)
        trees = _log(rng, 20, 3000)
        rule = rng.choice(["paper", "paper", "cmaes"])
        elites = rule == "paper" and N * (N // 2) * 4 * K <= 2 ** 31 and rng.random() < 0.5
        T = max(4, min(100, int(1.5e9 / (N * (K + 3) * S))))
        return dict(kind="plan", N=N, K=K, S=S, T=T, trees=trees, boxes=rng.choice([0, 0, 5, 40]),
                    grid=0.5 if trees > 250 else rng.choice([0.0, 0.5]), sampler="elites" if elites else "factor",
                    rule=rule, trips=rng.choice([1, 2]))
    if kind == "batch":
        return dict(kind="batch", queries=rng.randint(4, 16), N_lo=rng.randint(512, 1024), N_hi=_log(rng, 2048, 16384),
                    K_lo=8, K_hi=rng.randint(12, 32), trees_lo=rng.randint(20, 50), trees_hi=_log(rng, 300, 3000),
                    S=rng.randint(32, 64), T=rng.randint(10, 20), mix=rng.randint(1, 1000))
    if kind == "evaluate":
        hulls = rng.random() < 0.3
        trees = _log(rng, 20, 500 if hulls else 1500)
        N = _log(rng, 100, 4096 if hulls else 16384)
        return dict(kind="evaluate", N=N, K=K, S=min(S, 64), trees=trees, boxes=rng.choice([0, 10]),
                    grid=0.0 if hulls else rng.choice([0.0, 0.5]), collision="hulls" if hulls else "spheres",
                    outputs=rng.random() < 0.5)
    if kind == "update":
        return dict(kind="update", N=_log(rng, 600, 65536), K=K)
    if kind in ("smooth", "polish"):
        N = _log(rng, 256, 16384) if kind == "smooth" else rng.randint(16, 128)
        smooth = kind == "smooth"
        c = dict(kind=kind, N=N, K=K, S=min(S, 64), trees=_log(rng, 50, 1000) if smooth else _log(rng, 10, 40),
                 boxes=rng.choice([0, 10]) if smooth else 0)
        if kind == "polish":
            c["steps"], c["alpha"] = rng.randint(5, 20), 1e-6
        return c
    if kind == "ik":
        return dict(kind="ik", N=_log(rng, 100, 16384), trees=_log(rng, 5, 40), restarts=rng.choice([1, 4, 8, 13]),
                    iters=rng.randint(20, 50))
    return dict(kind="traj", N=rng.randint(4, 64), K=rng.randint(8, 16), intervals=rng.randint(40, 100))


# ---------------------------------------------------------------------------- inputs

def _side_stream():
    """The stream the program keeps for its planners (cp_plan records graphs only off the
    legacy default stream)."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def _scene(trees, boxes, seed):
    g = workloads.rng(seed, workloads.STREAM_SCENE, trees, boxes)
    if trees >= 4000:      # the dense forest: spaced trunks over a 50 m disc
        cyl = workloads.poisson_disc_cylinders(g, trees, 2.0, 50.0, 0.1, 0.5, 0.8)
        r_out = 12.0
    else:
        r_out = 8.0 if trees <= 80 else math.sqrt(4.0 + trees / (DENSITY * math.pi))
        cyl = workloads.annulus_cylinders(g, trees, 2.0, r_out, 0.1, 0.4)
    box = workloads.annulus_boxes(g, boxes, 2.0, max(r_out, 6.0), 0.5, 2.0) if boxes else np.zeros((0, 6))
    return workloads.Scene(cyl, box)


def _free_ends(crane, scene, seed, query=0):
    """Start and goal by the workloads' rule, with plain torch distances in 32 bits."""
    def dist(q):
        return _distance(crane, scene, torch.from_numpy(q).to(DEV, torch.float32)).cpu().numpy()

    q0, qd, _, _ = workloads.select_endpoints(crane, dist, seed=seed, query=query, batch=8192, max_draws=131072)
    return q0, qd


def _rule(case):
    return cp.CP_UPDATE_CMAES if case["rule"] == "cmaes" else cp.CP_UPDATE_PAPER


def _layer_inputs(case, seed):
    crane = workloads.forestry_crane()
    scene = _scene(case["trees"], case["boxes"], seed)
    q0, qd = _free_ends(crane, scene, seed)
    if case["kind"] != "polish":
        return crane, scene, q0, qd, workloads.random_candidates(q0, qd, case["K"], case["N"], seed, SPREAD)
    # the candidates with the least penetration, seen at 32 points of each path
    xi = workloads.random_candidates(q0, qd, case["K"], 4096, seed, tuple(0.3 * v for v in SPREAD))
    B = _basis(case["K"], case["S"])
    P = _control(q0, qd, torch.from_numpy(xi).to(DEV, torch.float64))
    q = torch.matmul(B[torch.linspace(0, B.shape[0] - 1, 32, device=DEV).long()], P).float().reshape(-1, 4)
    depth = (0.15 - _distance(crane, scene, q)).clamp_min(0).reshape(4096, 32).sum(1)
    return crane, scene, q0, qd, xi[torch.argsort(depth, stable=True)[:case["N"]].cpu().numpy()]


def _population(case, seed):
    """A population and its costs as a program that scores candidates itself hands them over."""
    g = workloads.rng(seed, workloads.STREAM_TEST, 5)
    crane = workloads.forestry_crane()
    q0, qd = workloads.uniform_configurations(crane, g, 2)
    xi = workloads.random_candidates(q0, qd, case["K"], case["N"], seed, SPREAD)
    return crane, q0, qd, xi, workloads.random_costs(case["N"], seed)


def _grasps(crane, scene, n, seed):
    """Grasp poses (x, y, z, yaw) of collision-free configurations near the ground."""
    def accept(q):
        t = torch.from_numpy(q).to(DEV, torch.float32)
        zg = _tip(crane, t)[:, 2] - 1.0
        ok = (zg > workloads.GRASP_Z[0]) & (zg < workloads.GRASP_Z[1])
        ok &= _distance(crane, scene, t) > workloads.GRASP_CLEARANCE
        return ok.cpu().numpy()

    q = workloads.grasp_configurations(crane, accept, n, seed=seed)
    tip = _tip(crane, torch.from_numpy(q).to(DEV)).cpu().numpy()
    return np.column_stack([tip[:, 0], tip[:, 1], tip[:, 2] - 1.0, q[:, 0]]).astype(np.float32)


def _paths(crane, n, K, seed):
    """Control points of n planned paths [n][K + 8][4]: a line with a smooth detour, the shape
    the path step hands over."""
    g = workloads.rng(seed, workloads.STREAM_TEST, 6)
    lo, hi = np.asarray(crane.q_min), np.asarray(crane.q_max)
    a = lo + (hi - lo) * (0.15 + 0.7 * g.random((n, 4)))
    b = lo + (hi - lo) * (0.15 + 0.7 * g.random((n, 4)))
    f = (np.arange(1, K + 1) / (K + 1.0))[None, :, None]
    mid = a[:, None] + f * (b - a)[:, None] + np.sin(math.pi * f) * (0.1 * (hi - lo) * g.uniform(-1, 1, (n, 4)))[:, None]
    return np.concatenate([np.repeat(a[:, None], 4, 1), mid, np.repeat(b[:, None], 4, 1)], axis=1)


def prepare(case, seed):
    seed = int(seed)
    kind = case["kind"]
    st = _side_stream()
    s = {"case": case, "stream": st}
    if kind == "plan":
        crane, scene = workloads.forestry_crane(), _scene(case["trees"], case["boxes"], seed)
        a, b = _free_ends(crane, scene, seed)
        s["trips"] = [(a, b), (b, a)][:case["trips"]]
        s["planner"] = cp.Planner(crane, scene, cp.make_params(
            case["N"], case["K"], case["S"], seed=seed, grid_cell=case["grid"], update_rule=_rule(case),
            sampler=cp.CP_SAMPLE_ELITES if case["sampler"] == "elites" else cp.CP_SAMPLE_FACTOR), st)
        D = 4 * case["K"]
        s["mu"] = torch.empty(case["trips"], D, dtype=torch.float64, device=DEV)
        s["C"] = torch.empty(case["trips"], D, D, dtype=torch.float64, device=DEV)
    elif kind == "batch":
        crane = workloads.forestry_crane()
        qs = workloads.batch_queries(case["queries"], case["mix"], case["N_lo"], case["N_hi"], case["K_lo"], case["K_hi"],
                                     case["trees_lo"], case["trees_hi"])
        scenes, params, q0s, qds = [], [], [], []
        for i, q in enumerate(qs):
            scene = workloads.batch_scene(q, seed, i)
            q0, qd = _free_ends(crane, scene, seed, i)
            scenes.append(cp.HostScene.from_scene(scene))
            params.append(cp.make_params(q.n_candidates, q.n_waypoints, case["S"], seed=seed, query=i, grid_cell=0.5))
            q0s.append(q0)
            qds.append(qd)
        s["Ks"], s["n"], s["ends"] = [q.n_waypoints for q in qs], len(qs), list(zip(q0s, qds))
        s["batch"] = _Batch(cp.cp_batch_init(cp.make_model(crane), scenes, params, q0s, qds, case["T"]), scenes)
    elif kind == "evaluate":
        crane, scene, q0, qd, xi = _layer_inputs(case, seed)
        hulls = case["collision"] == "hulls"
        s["planner"] = cp.Planner(crane, scene, cp.make_params(
            case["N"], case["K"], case["S"], grid_cell=case["grid"],
            collision_model=cp.CP_COLLISION_HULLS if hulls else cp.CP_COLLISION_SPHERES), st)
        cp.cp_set_endpoints(s["planner"].handle, q0, qd)
        n, n_s = case["N"], s["planner"].n_s
        s["xi"] = torch.from_numpy(xi).to(DEV)
        s["out"] = {"J": torch.empty(n, dtype=torch.float64, device=DEV),
                    "flag": torch.empty(n, dtype=torch.uint8, device=DEV),
                    "terms": torch.empty(n, 5, dtype=torch.float64, device=DEV)}
        if case["outputs"]:
            s["out"]["words"] = torch.empty(n, (n_s + 31) // 32, dtype=torch.int32, device=DEV)
            s["out"]["pen"] = torch.empty(n, n_s, dtype=torch.float32, device=DEV)
    elif kind == "update":
        crane, q0, qd, xi, J = _population(case, seed)
        D = 4 * case["K"]
        s["planner"] = cp.Planner(crane, _scene(20, 0, seed), cp.make_params(case["N"], case["K"], 4, seed=seed), st)
        cp.cp_set_endpoints(s["planner"].handle, q0, qd)
        s["xi"], s["J"] = torch.from_numpy(xi).to(DEV), torch.from_numpy(J).to(DEV)
        s["out"] = {"mu": torch.empty(D, dtype=torch.float64, device=DEV),
                    "C": torch.empty(D, D, dtype=torch.float64, device=DEV),
                    "L": torch.empty(D, D, dtype=torch.float64, device=DEV),
                    "elites": torch.empty(s["planner"].nu, dtype=torch.int32, device=DEV),
                    "next": torch.empty(case["N"], case["K"], 4, device=DEV)}
    elif kind in ("smooth", "polish"):
        crane, scene, q0, qd, xi = _layer_inputs(case, seed)
        s["planner"] = cp.Planner(crane, scene, cp.make_params(case["N"], case["K"], case["S"]), st)
        cp.cp_set_endpoints(s["planner"].handle, q0, qd)
        s["xi"] = torch.from_numpy(xi).to(DEV)
        if kind == "smooth":
            s["xi"].requires_grad_(True)
            s["g"] = torch.from_numpy(_upstream(case, seed)).to(DEV)
        else:
            s["work"] = torch.empty_like(s["xi"])
    elif kind == "ik":
        crane, scene = workloads.forestry_crane(), _scene(case["trees"], 0, seed)
        n = case["N"]
        s["planner"] = cp.Planner(crane, scene, cp.make_params(64, 2, 2), st)
        s["targets"] = torch.from_numpy(_grasps(crane, scene, n, seed)).to(DEV)
        s["ik"] = cp.make_ik_params(seed=seed, restarts=case["restarts"], iters=case["iters"])
        s["out"] = {"q": torch.empty(n, 4, device=DEV), "f": torch.empty(n, device=DEV),
                    "restart": torch.empty(n, dtype=torch.int32, device=DEV), "r": torch.empty(n, 5, device=DEV)}
    else:
        crane, n, N = workloads.forestry_crane(), case["N"], case["intervals"]
        s["solver"] = _Solver(cp.cp_traj_init(cp.make_model(crane), cp.make_traj_params(N=N), n, st))
        s["ctrl"] = torch.from_numpy(_paths(crane, n, case["K"], seed)).to(DEV)
        s["q"] = torch.empty(n, N + 1, 4, dtype=torch.float64, device=DEV)
        s["out"] = {"z": torch.empty(n, 1 + 16 * (N + 1), dtype=torch.float64, device=DEV),
                    "stats": torch.empty(n, 4, dtype=torch.float64, device=DEV)}
    torch.cuda.synchronize()   # the planners' stream does not wait for the default stream
    return s


class _Batch:
    """A batch handle and the host scenes it was made from."""

    def __init__(self, handle, scenes):
        self.handle, self.scenes = handle, scenes

    def __del__(self):
        cp.cp_batch_destroy(self.handle)


class _Solver:
    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        cp.cp_traj_destroy(self.handle)


# ---------------------------------------------------------------------------- one pass

def run(s):
    case = s["case"]
    kind = case["kind"]
    with torch.cuda.stream(s["stream"]):
        if kind == "plan":
            h, ctrls, stats = s["planner"].handle, [], []
            for t, (q0, qd) in enumerate(s["trips"]):
                cp.cp_set_endpoints(h, q0, qd)
                ctrl, st = cp.cp_plan(h, case["T"], K=case["K"])
                # the factor-free sampler keeps no covariance
                cp.cp_get_distribution(h, s["mu"][t], None if case["sampler"] == "elites" else s["C"][t])
                ctrls.append(ctrl)
                stats.append(st)
            out = _plan_outputs(ctrls, stats)
            out["mu"] = s["mu"]
            if case["sampler"] != "elites":
                out["C"] = s["C"]
            return out
        if kind == "batch":
            for i, (q0, qd) in enumerate(s["ends"]):
                cp.cp_batch_set_endpoints(s["batch"].handle, i, q0, qd)
            res = cp.cp_batch_run(s["batch"].handle, s["n"], s["Ks"])
            return _plan_outputs([r[0] for r in res], [r[1] for r in res])
        if kind == "evaluate":
            o = s["out"]
            cp.cp_evaluate(s["planner"].handle, s["xi"], case["N"], o["J"], o["flag"], o["terms"], o.get("words"),
                           o.get("pen"))
            return o
        if kind == "update":
            h, o = s["planner"].handle, s["out"]
            cp.cp_update(h, s["J"], s["xi"])
            cp.cp_sample(h, 1, o["next"])
            cp.cp_get_distribution(h, o["mu"], o["C"])
            cp.cp_get_factor(h, o["L"])
            cp.cp_get_elites(h, o["elites"])
            return o
        if kind == "smooth":
            J = autograd.path_cost(s["xi"], s["planner"])
            (dxi,) = torch.autograd.grad(J, s["xi"], s["g"])
            return {"J": J.detach(), "dxi": dxi}
        if kind == "polish":
            s["work"].copy_(s["xi"])
            cp.cp_polish(s["planner"].handle, s["work"], case["N"], case["steps"], case["alpha"])
            return {"xi": s["work"]}
        if kind == "ik":
            o = s["out"]
            cp.cp_ik(s["planner"].handle, s["targets"], case["N"], s["ik"], o["q"], o["f"], restart=o["restart"],
                     r=o["r"])
            return o
        h, o = s["solver"].handle, s["out"]
        cp.cp_traj_targets(h, s["ctrl"], case["K"], case["N"], s["q"])
        cp.cp_traj_initial_guess(h, s["q"], case["N"], o["z"])
        cp.cp_traj_solve(h, s["q"], case["N"], o["z"], o["stats"])
        return {"targets": s["q"], "z": o["z"], "stats": o["stats"]}


def _plan_outputs(ctrls, stats):
    return {"ctrl": np.concatenate(ctrls),
            "costs": np.array([[st[k] for k in ("J", "Jp", "Jc", "Jl", "length", "best_J")] for st in stats]),
            "counts": np.array([[st[k] for k in ("flag", "n_flagged", "iterations", "iteration")] for st in stats])}


# ---------------------------------------------------------------------------- the work of a pass

def work(case):
    """Bytes: inputs read and outputs written once. Operations: what one pass of the method
    takes with every obstacle far from a checkpoint left out for free (212 per checkpoint for
    spline, kinematics, sums and the reach test, 120 for the obstacles in reach)."""
    kind, N = case["kind"], case["N"] if "N" in case else 0
    if kind == "plan":
        D, n_s = 4 * case["K"], (case["K"] + 3) * case["S"]
        per = N * (n_s * 332.0 + 40.0 * D + D * D) + (N // 2) * D * D
        return {"flops": case["trips"] * case["T"] * per,
                "bytes": case["trips"] * (40.0 * case["trees"] + 8.0 * D * D + 64.0 * case["K"])}
    if kind == "batch":
        nq, N, K = case["queries"], 0.5 * (case["N_lo"] + case["N_hi"]), 0.5 * (case["K_lo"] + case["K_hi"])
        D, trees = 4 * K, 0.5 * (case["trees_lo"] + case["trees_hi"])
        per = N * ((K + 3) * case["S"] * 332.0 + 40.0 * D + D * D) + 0.5 * N * D * D
        return {"flops": nq * case["T"] * per, "bytes": nq * (40.0 * trees + 32.0 * K)}
    if kind == "update":
        D = 4 * case["K"]
        return {"flops": (N // 2) * D * (D + 3.0) + D ** 3 / 3.0 + N * (D * D + 40.0 * D),
                "bytes": 8.0 * N + 4.0 * (N // 2) * D + 4.0 * N * D + 16.0 * D * D + 2.0 * N}
    if kind == "ik":
        evals = N * case["restarts"] * (case["iters"] + 1.0)
        return {"flops": evals * (350.0 + 4.0 * case["trees"]), "bytes": N * (16.0 + 16.0 + 4.0 + 4.0 + 20.0)}
    if kind == "traj":
        # 120 steps; per grid point 16 derivative passes (200 each), assembly and a block
        # factorisation of 16 x 16 blocks
        n, pts = N, case["intervals"] + 1.0
        return {"flops": n * 120.0 * pts * (16 * 200.0 + 6 * 16.0 ** 3),
                "bytes": n * (pts * (32.0 + 128.0 + 32.0) + 32.0 * (case["K"] + 8))}
    n_s = (case["K"] + 3) * case["S"]
    xi = 16.0 * N * case["K"]
    if kind == "evaluate":
        out = 49.0 * N + (N * n_s * 4.125 if case["outputs"] else 0.0)
        return {"flops": N * n_s * (212.0 + (120.0 if case["collision"] == "spheres" else 1200.0)),
                "bytes": xi + out + 40.0 * case["trees"] + 48.0 * case["boxes"]}
    if kind == "smooth":
        return {"flops": N * n_s * (212.0 + 2 * 900.0 + 400.0), "bytes": 2 * xi + 16.0 * N + 40.0 * case["trees"]}
    return {"flops": case["steps"] * N * n_s * (212.0 + 900.0 + 400.0), "bytes": 2 * xi + 40.0 * case["trees"]}


# ---------------------------------------------------------------------------- 64-bit values

def exact(case, seed):
    seed = int(seed)
    kind = case["kind"]
    if kind == "evaluate":
        return _exact_evaluate(case, seed)
    if kind == "update":
        return _exact_update(case, seed)
    if kind in ("smooth", "polish"):
        # about 20 seconds of 64-bit pairs
        if case["N"] * (case["K"] + 3) * case["S"] * case.get("steps", 1) > 1.2e7:
            return None
        crane, scene, q0, qd, xi = _layer_inputs(case, seed)
        xi = torch.from_numpy(xi).to(DEV, torch.float64)
        if kind == "smooth":
            J, g = _smooth(crane, scene, q0, qd, case["S"], xi)
            return {"J": J, "dxi": g * torch.from_numpy(_upstream(case, seed)).to(DEV)[:, None, None]}
        for _ in range(case["steps"]):
            xi = xi - case["alpha"] * _smooth(crane, scene, q0, qd, case["S"], xi)[1]
        return {"xi": xi}
    return None   # searches and iterated solvers: where they end is no single value


def _upstream(case, seed):
    return workloads.rng(seed, workloads.STREAM_TEST, 8).uniform(0.1, 1.0, case["N"])


def _basis(K, S):
    """The cubic B-spline's weights at s_0 .. s_{n_s}: float64 [n_s + 1][K + 8]."""
    n_s = (K + 3) * S
    k = np.arange(1, n_s + 1)
    span = (k - 1) // S
    u = (k - span * S) / S
    b = np.stack([(1 - u) ** 3, 3 * u ** 3 - 6 * u ** 2 + 4, -3 * u ** 3 + 3 * u ** 2 + 3 * u + 1, u ** 3], 1) / 6.0
    B = np.zeros((n_s + 1, K + 8))
    B[0, 1:4] = np.array([1.0, 4.0, 1.0]) / 6.0
    for i in range(4):
        B[k, span + 1 + i] = b[:, i]
    return torch.from_numpy(B).to(DEV)


def _control(q0, qd, xi):
    n = xi.shape[0]
    a = torch.as_tensor(q0, dtype=torch.float64, device=DEV).expand(n, 4, 4)
    b = torch.as_tensor(qd, dtype=torch.float64, device=DEV).expand(n, 4, 4)
    return torch.cat([a, xi, b], 1)


def _excess(crane, q):
    lo = torch.tensor(crane.q_min, dtype=q.dtype, device=q.device)
    hi = torch.tensor(crane.q_max, dtype=q.dtype, device=q.device)
    return ((q - hi).clamp_min(0) ** 2 + (lo - q).clamp_min(0) ** 2).sum(-1)


def _chain(crane, q):
    """cos, sin of the slew, and the boom's and jib's in-plane directions."""
    a = q[..., 1] + q[..., 2]
    return torch.cos(q[..., 0]), torch.sin(q[..., 0]), torch.cos(q[..., 1]), torch.sin(q[..., 1]), torch.cos(a), \
        torch.sin(a)


def _tip(crane, q):
    c1, s1, c2, s2, c3, s3 = _chain(crane, q)
    L = crane.jib_len + q[..., 3]
    h = crane.boom_len * c2 + L * c3
    return torch.stack([h * c1, h * s1, crane.base_z + crane.boom_len * s2 + L * s3], -1)


def _centres(crane, q):
    """Link-sphere centres [..., spheres, 3]."""
    c1, s1, c2, s2, c3, s3 = _chain(crane, q)
    out = []
    for sp in crane.spheres:
        t, Lb, Lj = sp.offset, crane.boom_len, crane.jib_len
        if sp.link == 0:
            h, z = t * c2, t * s2
        elif sp.link == 1:
            h, z = Lb * c2 + t * c3, Lb * s2 + t * s3
        elif sp.link == 2:
            r = Lj + t * q[..., 3]
            h, z = Lb * c2 + r * c3, Lb * s2 + r * s3
        else:
            r = Lj + q[..., 3]
            h, z = Lb * c2 + r * c3, Lb * s2 + r * s3 - t
        out.append(torch.stack([h * c1, h * s1, z + crane.base_z], -1))
    return torch.stack(out, -2)


def _norm(*parts):
    return torch.sqrt(sum(p * p for p in parts))


def _sd_cyl(p, c):
    a = _norm(p[..., 0] - c[..., 0], p[..., 1] - c[..., 1]) - c[..., 2]
    b = torch.maximum(c[..., 3] - p[..., 2], p[..., 2] - c[..., 4])
    return torch.maximum(a, b).clamp_max(0) + _norm(a.clamp_min(0), b.clamp_min(0))


def _sd_box(p, b):
    d = (p - 0.5 * (b[..., :3] + b[..., 3:])).abs() - 0.5 * (b[..., 3:] - b[..., :3])
    m = d.clamp_min(0)
    return d.max(-1).values.clamp_max(0) + _norm(m[..., 0], m[..., 1], m[..., 2])


def _distance(crane, scene, q):
    """Signed distance d(q) of configurations q[n][4], in q's type."""
    r = torch.tensor([sp.radius for sp in crane.spheres], dtype=q.dtype, device=q.device)
    cyl = torch.from_numpy(scene.cylinders).to(q)
    box = torch.from_numpy(scene.boxes).to(q)
    d = torch.full((q.shape[0],), math.inf, dtype=q.dtype, device=q.device)
    step = max(1, (1 << 26) // (12 * max(1, scene.n_cyl, 3 * scene.n_box)))
    for i in range(0, q.shape[0], step):
        p = _centres(crane, q[i:i + step])
        v = d[i:i + step]
        if scene.n_cyl:
            v = torch.minimum(v, (_sd_cyl(p[:, :, None], cyl).min(-1).values - r).min(-1).values)
        if scene.n_box:
            v = torch.minimum(v, (_sd_box(p[:, :, None], box).min(-1).values - r).min(-1).values)
        d[i:i + step] = v
    return d


def _exact_evaluate(case, seed):
    K, S, N = case["K"], case["S"], case["N"]
    n_s = (K + 3) * S
    hulls = case["collision"] == "hulls"
    if N * n_s * 12.0 * (case["trees"] + 3 * case["boxes"]) > (4e10 if hulls else 6e10):
        return None
    crane, scene, q0, qd, xi = _layer_inputs(case, seed)
    B, P = _basis(K, S), _control(q0, qd, torch.from_numpy(xi).to(DEV, torch.float64))
    pen = torch.empty(N, n_s, dtype=torch.float64, device=DEV)
    terms = torch.empty(N, 5, dtype=torch.float64, device=DEV)
    step = max(1, 400000 // n_s)
    for i in range(0, N, step):
        q = torch.matmul(B, P[i:i + step])
        qk = q[:, 1:]
        dq2 = ((q[:, 1:] - q[:, :-1]) ** 2).sum(-1)
        flat = qk.reshape(-1, 4)
        depth = _hull_depth(crane, scene, flat) if hulls else (-_distance(crane, scene, flat)).clamp_min(0)
        pen[i:i + step] = depth.reshape(qk.shape[0], n_s)
        terms[i:i + step, 0] = dq2.sum(-1)
        terms[i:i + step, 2] = _excess(crane, qk).sum(-1)
        terms[i:i + step, 3] = dq2.sqrt().sum(-1)
    terms[:, 1] = LAMBDA_C * pen.sum(-1)
    terms[:, 4] = (pen > 0).sum(-1)
    out = {"J": terms[:, 0] + W_C * terms[:, 1] + W_L * terms[:, 2], "flag": None, "terms": terms}
    if case["outputs"]:
        out["words"], out["pen"] = None, pen
    return out


def _links(crane, q):
    """The four link boxes of the hull model: centres [n][4][3], axes [n][4][3][3], half
    extents [n][4][3] (half extents 0.2, 0.2, 0.15 m, pad 0.2 m, grapple 0.25 x 1.0 m)."""
    c1, s1, c2, s2, c3, s3 = _chain(crane, q)
    zero = torch.zeros_like(c1)
    one = torch.ones_like(c1)
    eb, ej = torch.stack([c2 * c1, c2 * s1, s2], -1), torch.stack([c3 * c1, c3 * s1, s3], -1)
    n, eg = torch.stack([-s1, c1, zero], -1), torch.stack([c1, s1, zero], -1)
    O = torch.tensor([0.0, 0.0, crane.base_z], dtype=q.dtype, device=q.device)
    J = O + crane.boom_len * eb
    q4p = q[:, 3].clamp_min(0)
    cen = [O + 0.5 * crane.boom_len * eb, J + 0.5 * crane.jib_len * ej, J + (crane.jib_len + 0.5 * q4p)[:, None] * ej,
           _tip(crane, q) - torch.tensor([0.0, 0.0, 0.5], dtype=q.dtype, device=q.device)]
    half = [torch.stack([(0.5 * crane.boom_len + 0.2) * one, 0.2 * one, 0.2 * one], -1),
            torch.stack([(0.5 * crane.jib_len + 0.2) * one, 0.2 * one, 0.2 * one], -1),
            torch.stack([0.5 * q4p + 0.2, 0.15 * one, 0.15 * one], -1),
            torch.stack([0.25 * one, 0.25 * one, 0.5 * one], -1)]
    axes = [torch.stack([e, n, torch.linalg.cross(e, n)], -2) for e in (eb, ej, ej)]
    axes.append(torch.stack([eg, n, torch.stack([zero, zero, one], -1)], -2))
    return torch.stack(cen, 1), torch.stack(axes, 1), torch.stack(half, 1)


def _hull_depth(crane, scene, q):
    """The largest separating-axis depth of the link boxes against the octagonal prisms of the
    trees and against the boxes, 0 where every pair is apart."""
    cen, axes, half = _links(crane, q)
    n = q.shape[0]
    cen, axes, half = cen.reshape(-1, 3), axes.reshape(-1, 3, 3), half.reshape(-1, 3)
    depth = torch.zeros(4 * n, dtype=q.dtype, device=q.device)
    flat = axes[:, :, 2].abs().mul(half).sum(-1)              # vertical half extent of each link box
    e = 0.5 * math.sqrt(2.0)
    octagon = torch.tensor([[1.0, 0, 0], [e, e, 0], [0, 1.0, 0], [-e, e, 0]], dtype=q.dtype, device=q.device)
    up = torch.tensor([[0.0, 0, 1.0]], dtype=q.dtype, device=q.device)
    for prism in (True, False):
        obs = torch.from_numpy(scene.cylinders if prism else scene.boxes).to(q)
        if not obs.shape[0]:
            continue
        if prism:
            oc = torch.stack([obs[:, 0], obs[:, 1], 0.5 * (obs[:, 3] + obs[:, 4])], -1)
            oh = torch.stack([obs[:, 2] / math.cos(math.pi / 8), 0.5 * (obs[:, 4] - obs[:, 3])], -1)
            reach, tall, dirs = oh[:, 0], oh[:, 1], torch.cat([up, octagon])
        else:
            oc, oh = 0.5 * (obs[:, :3] + obs[:, 3:]), 0.5 * (obs[:, 3:] - obs[:, :3])
            reach, tall, dirs = oh[:, :2].norm(dim=-1), oh[:, 2], torch.eye(3, dtype=q.dtype, device=q.device)
        wide = half.norm(dim=-1)
        step = max(1, (1 << 26) // obs.shape[0])
        for i in range(0, 4 * n, step):
            j = slice(i, i + step)
            near = (_norm(cen[j, None, 0] - oc[:, 0], cen[j, None, 1] - oc[:, 1]) < wide[j, None] + reach) & \
                ((cen[j, None, 2] - oc[:, 2]).abs() < flat[j, None] + tall)
            a, o = near.nonzero(as_tuple=True)
            for k in range(0, a.numel(), 1 << 20):
                u, v = a[k:k + (1 << 20)] + i, o[k:k + (1 << 20)]
                A, h, d = axes[u], half[u], oc[v] - cen[u]
                cross = torch.linalg.cross(A[:, :, None, :].expand(-1, 3, dirs.shape[0], 3),
                                           dirs.expand(A.shape[0], 3, -1, 3), dim=-1).reshape(A.shape[0], -1, 3)
                L = torch.cat([dirs.expand(A.shape[0], -1, 3), A, cross], 1)
                norm = L.norm(dim=-1, keepdim=True)
                L = L / norm.clamp_min(1e-9)
                ra = (torch.matmul(L, A.transpose(1, 2)).abs() * h[:, None]).sum(-1)
                if prism:
                    t = math.pi / 8
                    rb = torch.stack([(math.cos(w) * L[..., 0] + math.sin(w) * L[..., 1]).abs()
                                      for w in (t, 3 * t, 5 * t, 7 * t)]).max(0).values
                    rb = rb * oh[v, None, 0] + L[..., 2].abs() * oh[v, None, 1]
                else:
                    rb = (L.abs() * oh[v, None]).sum(-1)
                over = ra + rb - (L * d[:, None]).sum(-1).abs()
                over = torch.where(norm[..., 0] > 1e-9, over, math.inf).min(-1).values.clamp_min(0)
                depth.scatter_reduce_(0, u, over, "amax")
    return depth.reshape(n, 4).max(-1).values


def _smooth(crane, scene, q0, qd, S, xi):
    """The smooth cost (softplus penalty, margin 0.05 m, width 0.01 m) and its gradient."""
    n, K = xi.shape[0], xi.shape[1]
    B = _basis(K, S)
    J = torch.empty(n, dtype=torch.float64, device=DEV)
    grad = torch.empty_like(xi)
    cyl, box = torch.from_numpy(scene.cylinders).to(xi), torch.from_numpy(scene.boxes).to(xi)
    r = torch.tensor([sp.radius for sp in crane.spheres], dtype=torch.float64, device=DEV)
    m, beta = 0.05, 0.01
    far = m + 40 * beta + float(r.max())      # pairs beyond add less than e^-40 of a width
    step = max(1, 60000 // B.shape[0])
    for i in range(0, n, step):
        with torch.enable_grad():
            x = xi[i:i + step].detach().clone().requires_grad_(True)
            q = torch.matmul(B, _control(q0, qd, x))
            c = ((q[:, 1:] - q[:, :-1]) ** 2).sum((-1, -2)) + W_L * _excess(crane, q[:, 1:]).sum(-1)
            p = _centres(crane, q[:, 1:]).reshape(-1, 3)
            per = p.shape[0] // x.shape[0]
            for obs, sd in ((cyl, _sd_cyl), (box, _sd_box)):
                if not obs.shape[0]:
                    continue
                with torch.no_grad():
                    if sd is _sd_cyl:
                        xy, reach = obs[:, :2], obs[:, 2]
                        zlo, zhi = obs[:, 3], obs[:, 4]
                    else:
                        xy, reach = 0.5 * (obs[:, :2] + obs[:, 3:5]), 0.5 * (obs[:, 3:5] - obs[:, :2]).norm(dim=-1)
                        zlo, zhi = obs[:, 2], obs[:, 5]
                    live = ((p[:, 2] > zlo.min() - far) & (p[:, 2] < zhi.max() + far)).nonzero()[:, 0]
                    a, o = (torch.cdist(p[live, :2], xy, compute_mode="donot_use_mm_for_euclid_dist")
                            < reach + far).nonzero(as_tuple=True)
                    a = live[a]
                z = (m - (sd(p[a], obs[o]) - r[a % 12])) / beta
                c = c.index_add(0, a // per, W_C * LAMBDA_C * beta * torch.nn.functional.softplus(z, threshold=1e9))
            (g,) = torch.autograd.grad(c.sum(), x)
        J[i:i + step], grad[i:i + step] = c.detach(), g
    return J, grad


def _philox(c, seed):
    """Philox4x32-10 of counters c (four int64 tensors of 32-bit words) under a 64-bit key."""
    low = 0xFFFFFFFF
    k0, k1 = seed & low, (seed >> 32) & low
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((b >> 32) & low) ^ c[1] ^ k0, b & low, ((a >> 32) & low) ^ c[3] ^ k1, a & low]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return c


def _exact_update(case, seed):
    N, D = case["N"], 4 * case["K"]
    nu = N // 2
    _, _, _, xi, J = _population(case, seed)
    x = torch.from_numpy(xi).to(DEV, torch.float64).reshape(N, D)
    order = torch.sort(torch.from_numpy(J).to(DEV), stable=True).indices[:nu]
    w = math.log(nu + 0.5) - torch.log(torch.arange(1, nu + 1, dtype=torch.float64, device=DEV))
    w = w / w.sum()
    e = x[order]
    mu = (w[:, None] * e).sum(0)
    y = e - mu
    C = y.T @ (w[:, None] * y) + 1e-8 * torch.eye(D, dtype=torch.float64, device=DEV)
    L = torch.linalg.cholesky(C)
    j = torch.arange(D // 4, device=DEV).expand(N, -1).contiguous()
    i = torch.arange(N, device=DEV)[:, None].expand(-1, D // 4).contiguous()
    words = _philox([j, i, torch.ones_like(j), torch.zeros_like(j)], seed)
    z = torch.empty(N, D // 4, 4, dtype=torch.float64, device=DEV)
    for k in (0, 2):
        u1, u2 = ((words[k] >> 8) + 1).double() * 2.0 ** -24, (words[k + 1] >> 8).double() * 2.0 ** -24
        rad = torch.sqrt(-2.0 * torch.log(u1))
        z[..., k], z[..., k + 1] = rad * torch.cos(2 * math.pi * u2), rad * torch.sin(2 * math.pi * u2)
    return {"mu": mu, "C": C, "L": L, "elites": None, "next": (mu + z.reshape(N, D) @ L.T).reshape(N, -1, 4)}
