"""The largest scenes that the shared-memory forms of the evaluation accept, and what a failed call
leaves behind."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LIMIT = 232448   # shared memory of an opt-in block


@pytest.fixture(scope="module")
def lib():
    from paper_2503_14160_gb300 import build, craneplan
    build.build()
    craneplan.load()
    return craneplan


Q0, QD = np.array([-0.4, 0.4, -1.2, 0.5]), np.array([0.4, 0.6, -1.8, 1.5])


def _bytes(n_cyl, n_box, S):
    """Two records per obstacle, a group record per eight cylinders, the spline table, and eight
    warps' control points."""
    return 16 * (2 * n_cyl + 2 * n_box + (n_cyl + 7) // 8 + 2 * S + 8 * 40)


def _spheres(crane, sixteen):
    import dataclasses
    return dataclasses.replace(crane, spheres=(crane.spheres * 2)[:16]) if sixteen else crane


@pytest.mark.parametrize("sixteen", [False, True])
@pytest.mark.parametrize("short", [0, 16, 160, 320, 336, 704])
def test_scene_at_the_shared_memory_limit(lib, crane, short, sixteen):
    """Scenes `short` bytes below the limit: planned by the default and the exhaustive form and by
    cp_evaluate_static, with the results of the index form."""
    import torch
    from paper_2503_14160_gb300 import workloads
    crane = _spheres(crane, sixteen)
    K, S, n = 4, 3, 40
    left = (LIMIT - short) // 16 - 2 * S - 8 * 40
    n_cyl = next(c for c in range(left // 2, 0, -1)
                 if left - 2 * c - (c + 7) // 8 >= 0 and (left - 2 * c - (c + 7) // 8) % 2 == 0)
    n_box = (left - 2 * n_cyl - (n_cyl + 7) // 8) // 2
    assert _bytes(n_cyl, n_box, S) == LIMIT - short
    g = np.random.default_rng(short)
    cyl = workloads.annulus_cylinders(g, n_cyl, 2.0, 60.0, 0.05, 0.15)
    lo = np.stack([g.uniform(-9, 9, n_box), g.uniform(-9, 9, n_box), np.zeros(n_box)], 1)
    scene = workloads.Scene(cyl, np.concatenate([lo, lo + 0.3], 1))
    xi = workloads.random_candidates(Q0, QD, K, n, seed=1)
    out = []
    for kw in ({"grid_cell": 0.5}, {}, {"eval_exhaustive": 1}):
        with lib.Planner(crane, scene, lib.make_params(n, K, S, **kw)) as pl:
            lib.cp_set_endpoints(pl.handle, Q0, QD)
            x = torch.from_numpy(xi).cuda()
            J = torch.zeros(n, dtype=torch.float64, device="cuda")
            flag = torch.zeros(n, dtype=torch.uint8, device="cuda")
            terms = torch.zeros(n, 5, dtype=torch.float64, device="cuda")
            lib.cp_evaluate(pl.handle, x, n, J, flag, terms)
            lib.cp_synchronize(pl.handle)
            out.append([t.cpu().numpy() for t in (J, flag, terms)])
    J, flag, terms = (torch.zeros_like(t) for t in (J, flag, terms))
    lib.cp_evaluate_static(lib.make_model(crane), torch.from_numpy(cyl).cuda(), n_cyl,
                           torch.from_numpy(scene.boxes).cuda(), n_box, K, S, 100.0, 100.0, 1.0, Q0, QD, x, n, J,
                           flag, terms)
    torch.cuda.synchronize()
    out.append([t.cpu().numpy() for t in (J, flag, terms)])
    assert out[0][1].any()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            np.testing.assert_array_equal(a, b)
    one_more = workloads.Scene(np.concatenate([cyl] + [cyl[:1]] * (short // 32 + 1)), scene.boxes)
    with pytest.raises(lib.CranePlanError) as e:
        lib.Planner(crane, one_more, lib.make_params(n, K, S))
    assert e.value.status == -1 and "shared memory" in str(e.value)


@pytest.mark.parametrize("form", ["polar", "broad", "exhaustive", "hulls"])
@pytest.mark.parametrize("stream", [False, True])
def test_calls_after_a_failed_evaluation(lib, crane, form, stream):
    """An evaluation that fails between its main kernel and its sums (on the host: cp_evaluate, and
    an iteration of a plan, recorded on a stream of its own) leaves nothing that a later call takes
    for its own: the next evaluations and plans are right without new end points."""
    import torch
    from paper_2503_14160_gb300 import workloads
    kw = {"polar": {"grid_cell": 0.5}, "exhaustive": {"eval_exhaustive": 1},
          "hulls": {"collision_model": lib.CP_COLLISION_HULLS}}.get(form, {})
    scene = workloads.make_scene(workloads.WORKLOADS["single_small"])
    n, K, S = 300, 5, 9
    st = torch.cuda.Stream() if stream else None
    x = [torch.from_numpy(workloads.random_candidates(Q0, QD, K, n, seed=seed)).cuda() for seed in (1, 2)]
    torch.cuda.synchronize()

    def evaluate(pl, i):
        J = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        lib.cp_evaluate(pl.handle, x[i], n, J)
        lib.cp_synchronize(pl.handle)
        return J.cpu().numpy()

    with lib.Planner(crane, scene, lib.make_params(n, K, S, **kw), st) as fresh:
        lib.cp_set_endpoints(fresh.handle, Q0, QD)
        want = [evaluate(fresh, 0), evaluate(fresh, 1)]
        lib.cp_set_endpoints(fresh.handle, Q0, QD)
        want_plan = lib.cp_plan(fresh.handle, 3, K=K)
    with lib.Planner(crane, scene, lib.make_params(n, K, S, **kw), st) as pl:
        lib.cp_set_endpoints(pl.handle, Q0, QD)
        try:
            lib.cp_debug_fail_evaluations(1)
            with pytest.raises(lib.CranePlanError) as e:
                evaluate(pl, 0)
            assert e.value.status == -2
            assert np.array_equal(evaluate(pl, 1), want[1])
            lib.cp_debug_fail_evaluations(2)
            for _ in range(2):
                with pytest.raises(lib.CranePlanError):
                    lib.cp_plan(pl.handle, 3, K=K)
        finally:
            lib.cp_debug_fail_evaluations(0)
        assert np.array_equal(evaluate(pl, 0), want[0])
        assert np.array_equal(evaluate(pl, 1), want[1])
        if stream:   # its recording failed, so no iteration has run: the plan from the start
            ctrl, stats = lib.cp_plan(pl.handle, 3, K=K)
            assert np.array_equal(ctrl, want_plan[0]) and stats == want_plan[1]
        lib.cp_set_endpoints(pl.handle, Q0, QD)
        ctrl, stats = lib.cp_plan(pl.handle, 3, K=K)
        assert np.array_equal(ctrl, want_plan[0]) and stats == want_plan[1]


@pytest.mark.parametrize("K", [5, 8, 32])
def test_factor_whose_message_is_missing(lib, crane, K):
    """One message between the factor's blocks withheld: their wait ends by its limit, the call after
    reports it, and the next factor is right."""
    import torch
    from paper_2503_14160_gb300 import workloads
    D = 4 * K
    g = np.random.default_rng(K)
    A = g.normal(size=(D, D + 3))
    mu, C = torch.zeros(D, dtype=torch.float64, device="cuda"), torch.from_numpy(A @ A.T).cuda()
    L = [torch.empty(D, D, dtype=torch.float64, device="cuda") for _ in range(2)]
    with lib.Planner(crane, workloads.empty_scene(), lib.make_params(64, K, 2)) as pl:
        lib.cp_set_endpoints(pl.handle, Q0, QD)
        lib.cp_set_distribution(pl.handle, mu, C, 1)
        lib.cp_get_factor(pl.handle, L[0])
        lib.cp_synchronize(pl.handle)
        lib.cp_debug_withhold_factor(True)
        try:
            lib.cp_set_distribution(pl.handle, mu, C, 1)
        finally:
            lib.cp_debug_withhold_factor(False)
        with pytest.raises(lib.CranePlanError) as e:
            lib.cp_synchronize(pl.handle)
        assert e.value.status == -3
        lib.cp_set_distribution(pl.handle, mu, C, 1)
        lib.cp_get_factor(pl.handle, L[1])
        lib.cp_synchronize(pl.handle)
        assert torch.equal(L[0], L[1])
