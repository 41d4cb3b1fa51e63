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


def _moments_reference(x, w):
    """mu, C (without eps) and the second moments about x_1, in long double."""
    x, w = x.astype(np.longdouble), w.astype(np.longdouble)
    y = x - x[0]
    s1 = (w[:, None] * y).sum(0)
    s2 = (w[:, None] * y).T @ y
    return x[0] + s1, s2 - np.outer(s1, s1), s2, s1


@pytest.mark.parametrize("N,K,shape", [(16384, 8, "plain"), (16442, 8, "plain"), (1024, 32, "plain"),
                                       (2050, 23, "offset"), (4099, 17, "outlier"), (9001, 16, "plain"),
                                       (3001, 32, "still"), (65536, 32, "plain")])
def test_integer_moments(lib, crane, N, K, shape):
    """The tensor-core moments (nu D^2 >= 2^23) against long double. Bound per entry: the two
    factors' rounding to 2^-55 of the column's bound (at most 4 times the largest deviation times
    the largest root weight), by Cauchy-Schwarz over the elites, and 16 units of FP64 rounding of
    the two terms of C."""
    import torch
    from paper_2503_14160_gb300 import workloads
    g = np.random.default_rng(N + K)
    D, nu = 4 * K, N // 2
    assert nu * D * D >= 2 ** 23
    xi = (g.normal(size=(N, D)) * np.exp(g.normal(size=D) * 2)).astype(np.float32)
    if shape == "offset":
        xi += np.float32(1000.0)
    if shape == "outlier":
        xi[g.integers(0, N, 3)] *= np.float32(2e4)
    if shape == "still":
        xi[:, 5] = np.float32(0.3)
    J = workloads.random_costs(N, seed=N)
    order = np.argsort(J, kind="stable")[:nu]
    w = np.log(nu + 0.5) - np.log(np.arange(1, nu + 1))
    w = w / w.sum()
    x = xi[order].astype(np.float64)
    mu_ref, C_ref, s2, s1 = _moments_reference(x, w)
    with lib.Planner(crane, workloads.empty_scene(), lib.make_params(N, K, 2, eps=0.0)) as pl:
        lib.cp_set_endpoints(pl.handle, *ENDS[0])
        lib.cp_update(pl.handle, torch.from_numpy(J).cuda(), torch.from_numpy(xi).cuda())
        mu = torch.empty(D, dtype=torch.float64, device="cuda")
        C = torch.empty(D, D, dtype=torch.float64, device="cuda")
        lib.cp_get_distribution(pl.handle, mu, C)
        torch.cuda.synchronize()
    mu, C = mu.cpu().numpy(), C.cpu().numpy()
    y = np.abs(x - x[0]).max(0)
    z = 4.0 * y * np.sqrt(w[0]) * 2.0 ** -55            # rounding of one factor
    root = np.sqrt(nu * np.diag(s2).astype(np.float64))  # sum_j |z_j| at most
    u = 2.0 ** -53
    bound = np.outer(z, root) + np.outer(root, z) + 16 * u * (np.abs(s2) + np.abs(np.outer(s1, s1))
                                                               + np.sqrt(np.outer(np.diag(s2), np.diag(s2))))
    assert np.all(np.abs(C - C_ref) <= bound.astype(np.float64) + 1e-300)
    assert np.all(np.abs(mu - mu_ref) <= 4 * y * w[0] * nu * 2.0 ** -55 + 16 * u * (np.abs(mu_ref) + np.abs(s1)) + 1e-300)
    # no less exact than a plain FP64 sum, over all entries
    scale = np.sqrt(np.outer(np.diag(s2), np.diag(s2))).astype(np.float64) + 1e-300
    y64 = x - x[0]
    plain = (w[:, None] * y64).T @ y64 - np.outer(w @ y64, w @ y64)
    err = np.linalg.norm(((C - C_ref) / scale).astype(np.float64))
    assert err <= 1.5 * np.linalg.norm(((plain - C_ref) / scale).astype(np.float64)) + D * u


@pytest.mark.parametrize("bad", [np.inf, np.nan, 3e38])
def test_integer_moments_carry_non_finite_elites(lib, crane, bad):
    """An elite outside the fixed-point range: its column as FP64 arithmetic gives it, the other
    columns as without it."""
    import torch
    from paper_2503_14160_gb300 import workloads
    N, K = 4096, 16
    D, nu = 4 * K, N // 2
    g = np.random.default_rng(3)
    xi = g.normal(size=(N, D)).astype(np.float32)
    J = np.arange(N, dtype=np.float64)
    out = []
    for value in (np.float32(bad), xi[7, 9]):
        x = xi.copy()
        x[7, 9] = value
        if bad == 3e38:
            x[0, 9] = -value
        with lib.Planner(crane, workloads.empty_scene(), lib.make_params(N, K, 2)) as pl:
            lib.cp_set_endpoints(pl.handle, *ENDS[0])
            lib.cp_update(pl.handle, torch.from_numpy(J).cuda(), torch.from_numpy(x).cuda())
            mu = torch.empty(D, dtype=torch.float64, device="cuda")
            C = torch.empty(D, D, dtype=torch.float64, device="cuda")
            lib.cp_get_distribution(pl.handle, mu, C)
            torch.cuda.synchronize()
        out.append((mu.cpu().numpy(), C.cpu().numpy()))
    others = np.arange(D) != 9
    assert np.array_equal(out[0][0][others], out[1][0][others])
    assert np.array_equal(out[0][1][np.ix_(others, others)], out[1][1][np.ix_(others, others)])
    if bad == 3e38:
        w = np.log(nu + 0.5) - np.log(np.arange(1, nu + 1))
        w = w / w.sum()
        x = xi[:nu].astype(np.float64)
        x[7, 9], x[0, 9] = np.float32(bad), -np.float32(bad)
        want = (w[:, None] * x).sum(0)[9]
        assert abs(out[0][0][9] - want) <= 1e-10 * 3e38
        assert np.isfinite(out[0][1][:, 9]).all()
    else:
        assert not np.isfinite(out[0][0][9]) and not np.isfinite(out[0][1][9, 9])


@pytest.mark.parametrize("N", [8193, 9215, 9216, 9217, 65537, 262144, 262145])
def test_ranking_passes(lib, crane, N):
    """The one-launch radix passes at tile edges and at the last size that takes them, against a
    stable sort; ties, NaN, infinities and both zeros among the costs."""
    import torch
    from paper_2503_14160_gb300 import workloads
    g = np.random.default_rng(N)
    J = g.normal(size=N) * np.exp(g.normal(size=N) * 20)
    for value in (np.nan, np.inf, -np.inf, 0.0, -0.0, 1.5):
        J[g.integers(0, N, N // 50)] = value
    want = np.argsort(np.where(np.isnan(J), np.inf, J), kind="stable")
    xi = torch.zeros(N, 1, 4, device="cuda")
    with lib.Planner(crane, workloads.empty_scene(), lib.make_params(N, 1, 1, n_elites=N)) as pl:
        lib.cp_set_endpoints(pl.handle, *ENDS[0])
        lib.cp_update(pl.handle, torch.from_numpy(J).cuda(), xi)
        el = torch.empty(N, dtype=torch.int32, device="cuda")
        lib.cp_get_elites(pl.handle, el)
        torch.cuda.synchronize()
    assert np.array_equal(el.cpu().numpy(), want)


@pytest.mark.parametrize("K", [2, 8, 12, 20, 24, 28, 32])
def test_batch_factor_cluster_sizes(lib, crane, K):
    """Every number of 16-row blocks of the largest factor of a batch: the batch can be set up, and
    its plans are those of its planners alone."""
    from paper_2503_14160_gb300 import workloads
    Ks = [K, 3]
    scenes = [lib.HostScene.from_scene(workloads.empty_scene()) for _ in Ks]
    params = [lib.make_params(80, k, 4, seed=q, query=q, grid_cell=0.5) for q, k in enumerate(Ks)]
    b = lib.cp_batch_init(lib.make_model(crane), scenes, params, [e[0] for e in ENDS], [e[1] for e in ENDS], 2)
    try:
        res = lib.cp_batch_run(b, len(Ks), K=Ks)
        for q, k in enumerate(Ks):
            p = lib.cp_batch_planner(b, q)
            lib.cp_set_endpoints(p, *ENDS[q])
            ctrl, _ = lib.cp_plan(p, 2, K=k)
            assert np.array_equal(res[q][0], ctrl)
    finally:
        lib.cp_batch_destroy(b)


@pytest.mark.parametrize("K", [1, 7, 32])
def test_sample_adds_the_mean_in_fp64(lib, crane, K):
    """xi = float(mu + acc) with the sum in FP64, for means of all sizes, on ties of the rounding to
    FP32 and beside draws too small to leave them: acc is the draw about a zero mean."""
    import torch
    from paper_2503_14160_gb300 import workloads
    g = np.random.default_rng(K)
    D, N = 4 * K, 3001
    mu = g.normal(size=D) * 10.0 ** g.uniform(-42, 6, D)
    mu[0::4] = g.normal(size=K).astype(np.float32) * (1.0 + 2.0 ** -24)
    mu[1::4] = 1.0 + 2.0 ** -24
    std = np.where(np.arange(D) % 4 == 1, 1e-13, 10.0 ** g.uniform(-3, 1, D))
    C = torch.from_numpy(np.diag(std ** 2)).cuda()
    out = []
    with lib.Planner(crane, workloads.empty_scene(), lib.make_params(N, K, 2, sigma=1.0)) as pl:
        lib.cp_set_endpoints(pl.handle, *ENDS[0])
        for m in (np.zeros(D), mu):
            lib.cp_set_distribution(pl.handle, torch.from_numpy(m).cuda(), C, 1)
            xi = torch.zeros(N, K, 4, device="cuda")
            lib.cp_sample(pl.handle, 1, xi)
            lib.cp_synchronize(pl.handle)
            out.append(xi.cpu().numpy().reshape(N, D))
    assert np.array_equal(out[1], (mu + out[0].astype(np.float64)).astype(np.float32))


@pytest.mark.parametrize("K", [1, 4, 7, 12, 17, 20, 25, 32])
def test_sample_forms(lib, crane, K):
    """The sampler's row blocks (2, 4, 6 or 8 of 16 rows, ragged) and candidates per warp (4, 8 and
    16, by N): a candidate's draw is the same in every form, and is mu + L z to the sampler's bound."""
    import torch
    import oracle
    from helpers import factor_sample_bound
    from paper_2503_14160_gb300 import workloads
    g = np.random.default_rng(40 + K)
    D = 4 * K
    A, mu = g.normal(size=(D, D)), g.normal(size=D)
    C = A @ A.T / D + 0.1 * np.eye(D)
    out = []
    for N in (61, 7001, 20003):
        with lib.Planner(crane, workloads.empty_scene(), lib.make_params(N, K, 2, sigma=0.7, seed=11, query=3)) as pl:
            lib.cp_set_endpoints(pl.handle, *ENDS[0])
            lib.cp_set_distribution(pl.handle, torch.from_numpy(mu).cuda(), torch.from_numpy(C).cuda(), 5)
            xi = torch.full((N, K, 4), np.nan, device="cuda")
            lib.cp_sample(pl.handle, 5, xi)
            lib.cp_synchronize(pl.handle)
            out.append(xi.cpu().numpy().reshape(N, D))
    assert np.array_equal(out[0], out[1][:61]) and np.array_equal(out[1], out[2][:7001])
    assert np.all(np.isfinite(out[2]))
    L = oracle.factor(C, 0.7)
    want = oracle.sample(mu, L, 11, 5, 3, 61, K).reshape(61, D)
    assert np.all(np.abs(out[0] - want) <= factor_sample_bound(want, oracle.normals(11, 5, 3, 61, K), L))


@pytest.mark.parametrize("N,K", [(2, 1), (37, 3), (130, 8), (600, 8), (4000, 8), (4400, 8), (600, 32), (1000, 5),
                                 (2200, 4)])
def test_moment_forms(lib, crane, N, K):
    """Deviations formed in the partial sums' blocks or by a launch before, first moments summed in the
    combine's blocks or by a launch before: mean and covariance of one update against long double,
    each sum within nu + 16 FP64 roundings of its absolute terms."""
    import torch
    from paper_2503_14160_gb300 import workloads
    g = np.random.default_rng(N * K)
    D = 4 * K
    xi = g.normal(size=(N, D)).astype(np.float32)
    J = workloads.random_costs(N, seed=N)
    with lib.Planner(crane, workloads.empty_scene(), lib.make_params(N, K, 2, eps=0.125)) as pl:
        nu = pl.nu
        lib.cp_set_endpoints(pl.handle, *ENDS[0])
        lib.cp_update(pl.handle, torch.from_numpy(J).cuda(), torch.from_numpy(xi).cuda())
        mu = torch.empty(D, dtype=torch.float64, device="cuda")
        C = torch.empty(D, D, dtype=torch.float64, device="cuda")
        lib.cp_get_distribution(pl.handle, mu, C)
        torch.cuda.synchronize()
    w = np.log(nu + 0.5) - np.log(np.arange(1, nu + 1))
    w = w / w.sum()
    x = xi[np.argsort(J, kind="stable")[:nu]].astype(np.float64)
    mu_ref, C_ref, s2, s1 = _moments_reference(x, w)
    y = np.abs(x - x[0])
    a1, a2 = (w[:, None] * y).sum(0), (w[:, None] * y).T @ y
    u = (nu + 16) * 2.0 ** -53
    assert np.all(np.abs(mu.cpu().numpy() - mu_ref) <= u * (a1 + np.abs(x[0])))
    C_ref = C_ref + 0.125 * np.eye(D)
    assert np.all(np.abs(C.cpu().numpy() - C_ref) <= u * (a2 + 3 * np.outer(a1, a1) + 0.125 * np.eye(D)))
