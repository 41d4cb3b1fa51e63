"""Launch forms that must not change results: a recorded plan replayed for new end points, and
the trajectory solver's cluster sizes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2503_14160_gb300 import build, craneplan
    build.build()
    craneplan.load()
    return craneplan


@pytest.fixture(scope="module")
def crane():
    from paper_2503_14160_gb300 import workloads
    return workloads.forestry_crane()


ENDS = [(np.array([0.3, 0.4, -1.2, 0.5]), np.array([-2.0, 0.6, -1.8, 1.5])),
        (np.array([-1.1, 0.1, -0.7, 2.0]), np.array([1.4, 0.9, -2.1, 0.2]))]


@pytest.mark.parametrize("form", ["broad", "polar", "exhaustive", "hulls", "elites", "cmaes"])
def test_recorded_plan_takes_new_end_points(lib, crane, form):
    """The same planner planning A, B, A equals fresh planners bit for bit."""
    import torch
    from paper_2503_14160_gb300 import workloads
    kw = {"polar": {"grid_cell": 0.5}, "exhaustive": {"eval_exhaustive": 1},
          "hulls": {"collision_model": lib.CP_COLLISION_HULLS}, "elites": {"sampler": lib.CP_SAMPLE_ELITES},
          "cmaes": {"update_rule": lib.CP_UPDATE_CMAES}}.get(form, {})
    scene = workloads.make_scene(workloads.WORKLOADS["single_small"])
    st = torch.cuda.Stream()

    def plan(pl, ends):
        lib.cp_set_endpoints(pl.handle, *ends)
        return lib.cp_plan(pl.handle, 6, K=pl.K)

    with lib.Planner(crane, scene, lib.make_params(130, 5, 9, **kw), st) as kept:
        got = [plan(kept, ENDS[i]) for i in (0, 1, 0)]
    for i, (ctrl, stats) in zip((0, 1, 0), got):
        with lib.Planner(crane, scene, lib.make_params(130, 5, 9, **kw), st) as fresh:
            want_ctrl, want = plan(fresh, ENDS[i])
        assert np.array_equal(ctrl, want_ctrl)
        assert stats == want
    assert not np.array_equal(got[0][0], got[1][0])


@pytest.mark.parametrize("N", [2, 17, 100])
def test_trajectories_do_not_depend_on_the_cluster_size(lib, crane, N):
    """45 trajectories at once (two CTAs each) against the same in smaller calls (8 and 4)."""
    import torch
    n, K = 45, 8
    g = np.random.default_rng(5)
    lo, hi = np.asarray(crane.q_min), np.asarray(crane.q_max)
    a = lo + (hi - lo) * (0.2 + 0.6 * g.random((n, 1, 4)))
    b = lo + (hi - lo) * (0.2 + 0.6 * g.random((n, 1, 4)))
    f = (np.arange(1, K + 1) / (K + 1))[None, :, None]
    ctrl = torch.from_numpy(np.concatenate([np.repeat(a, 4, 1), a + f * (b - a), np.repeat(b, 4, 1)], 1)).cuda()
    h = lib.cp_traj_init(lib.make_model(crane), lib.make_traj_params(N=N, outer=3, inner=4), n)
    try:
        def solve(c):
            m = c.shape[0]
            q = torch.empty(m, N + 1, 4, dtype=torch.float64, device="cuda")
            z = torch.empty(m, 1 + 16 * (N + 1), dtype=torch.float64, device="cuda")
            s = torch.empty(m, 4, dtype=torch.float64, device="cuda")
            lib.cp_traj_targets(h, c, K, m, q)
            lib.cp_traj_initial_guess(h, q, m, z)
            lib.cp_traj_solve(h, q, m, z, s)
            return z.cpu().numpy(), s.cpu().numpy()

        z, s = solve(ctrl)
        for at, m in ((0, 3), (3, 24)):
            zs, ss = solve(ctrl[at:at + m].contiguous())
            assert np.array_equal(zs, z[at:at + m]) and np.array_equal(ss, s[at:at + m])
        assert np.isfinite(z).all()
    finally:
        lib.cp_traj_destroy(h)


@pytest.mark.parametrize("K", [1, 2, 4, 5, 8, 9, 16, 21, 31, 32])
def test_factor_against_fp64(lib, crane, K):
    """The cluster factor at every edge of its 16-row blocks: backward error of a few D units of
    rounding per entry, relative to the geometric mean of the two variances."""
    import torch
    from paper_2503_14160_gb300 import workloads
    D = 4 * K
    g = np.random.default_rng(K)
    A = g.normal(size=(D, D + 3)) * np.exp(g.normal(size=(D, 1)))
    C = A @ A.T
    sigma = 0.7
    with lib.Planner(crane, workloads.empty_scene(), lib.make_params(64, K, 2, sigma=sigma)) as pl:
        lib.cp_set_endpoints(pl.handle, *ENDS[0])
        mu = torch.zeros(D, dtype=torch.float64, device="cuda")
        lib.cp_set_distribution(pl.handle, mu, torch.from_numpy(C).cuda(), 1)
        L = torch.empty(D, D, dtype=torch.float64, device="cuda")
        lib.cp_get_factor(pl.handle, L)
        lib.cp_synchronize(pl.handle)
        L = L.cpu().numpy()
        assert np.all(np.triu(L, 1) == 0.0)
        scale = sigma ** 2 * np.sqrt(np.outer(np.diag(C), np.diag(C)))
        assert np.max(np.abs(L @ L.T - sigma ** 2 * C) / scale) < 4 * (D + 4) * 2.0 ** -53
        # a lost pivot in the last block is reported
        C[D - 1, D - 1] = -1.0
        lib.cp_set_distribution(pl.handle, mu, torch.from_numpy(C).cuda(), 1)
        with pytest.raises(lib.CranePlanError) as e:
            lib.cp_synchronize(pl.handle)
        assert e.value.status == -6
