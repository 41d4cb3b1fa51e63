"""An iteration driven by hand (cp_sample, cp_evaluate, cp_update) is an iteration of cp_plan, at
every size, and the update's sums are as exact as FP64 additions."""
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


ENDS = (np.array([0.3, 0.4, -1.2, 0.5]), np.array([-2.0, 0.6, -1.8, 1.5]))


def _distribution(lib, pl):
    import torch
    mu = torch.empty(pl.D, dtype=torch.float64, device="cuda")
    C = torch.empty(pl.D, pl.D, dtype=torch.float64, device="cuda")
    lib.cp_get_distribution(pl.handle, mu, C)
    lib.cp_synchronize(pl.handle)
    return mu.cpu().numpy(), C.cpu().numpy()


@pytest.mark.parametrize("N,K,kw", [(256, 8, {}), (1000, 32, {}), (1024, 32, {}), (9001, 16, {}), (16385, 8, {}),
                                    (512, 16, {"sampler": 1}), (512, 16, {"update_rule": 1}),
                                    (4096, 32, {"update_rule": 1})])
def test_steps_by_hand_are_the_plan(lib, crane, N, K, kw):
    """Five iterations either way, bit for bit: mean, covariance and costs. Sizes on both sides of
    the forms that the update and the ranking choose by size."""
    import torch
    from paper_2503_14160_gb300 import workloads
    scene = workloads.make_scene(workloads.WORKLOADS["single_small"])
    params = lib.make_params(N, K, 9, seed=3, **kw)
    with lib.Planner(crane, scene, params, torch.cuda.Stream()) as pl:
        lib.cp_set_endpoints(pl.handle, *ENDS)
        lib.cp_plan(pl.handle, 5)
        want = _distribution(lib, pl)
        J_plan = torch.empty(N, dtype=torch.float64, device="cuda")
        lib.cp_get_population(pl.handle, None, J_plan)
        lib.cp_synchronize(pl.handle)
    with lib.Planner(crane, scene, params) as pl:
        lib.cp_set_endpoints(pl.handle, *ENDS)
        xi = torch.zeros(N, K, 4, device="cuda")
        J = torch.zeros(N, dtype=torch.float64, device="cuda")
        for t in range(5):
            lib.cp_sample(pl.handle, t, xi)
            lib.cp_evaluate(pl.handle, xi, N, J)
            lib.cp_update(pl.handle, J, xi)
        got = _distribution(lib, pl)
    assert np.array_equal(J.cpu().numpy(), J_plan.cpu().numpy())
    assert np.array_equal(got[0], want[0])
    assert np.array_equal(got[1], want[1])


@pytest.mark.parametrize("N,K", [(1024, 32), (9001, 16), (65536, 32)])
@pytest.mark.parametrize("shape", ["plain", "outlier"])
def test_mean_is_as_exact_as_fp64_sums(lib, crane, N, K, shape):
    """mu = x_(1) + sum_j w_j (x_(j) - x_(1)) against long double. A sum runs through at most 256
    elites of a chunk, then its 32 interleaved sums of up to 512 chunks (16 each) and five
    pairings; with the product, the weight and the final addition that is at most 284 roundings of
    what the terms add up to in magnitude."""
    import torch
    from paper_2503_14160_gb300 import workloads
    g = np.random.default_rng(N + K)
    D, nu = 4 * K, N // 2
    xi = g.normal(size=(N, D)).astype(np.float32)
    if shape == "outlier":
        xi[g.integers(0, N, 3)] *= np.float32(2e4)
    J = workloads.random_costs(N, seed=N)
    with lib.Planner(crane, workloads.empty_scene(), lib.make_params(N, K, 2)) as pl:
        lib.cp_set_endpoints(pl.handle, *ENDS)
        lib.cp_update(pl.handle, torch.from_numpy(J).cuda(), torch.from_numpy(xi).cuda())
        mu, _ = _distribution(lib, pl)
    w = np.log(np.longdouble(nu) + np.longdouble(0.5)) - np.log(np.arange(1, nu + 1).astype(np.longdouble))
    w = w / w.sum()
    x = xi[np.argsort(J, kind="stable")[:nu]].astype(np.longdouble)
    y = x - x[0]
    want = x[0] + (w[:, None] * y).sum(0)
    # the weights themselves: a difference of logarithms and a quotient, a few roundings of ln(nu)
    w_err = 8 * np.log(nu) / float(np.sum(np.log(nu + 0.5) - np.log(np.arange(1, nu + 1)))) * np.abs(y).sum(0)
    u = 2.0 ** -53
    bound = u * (284 * (w[:, None] * np.abs(y)).sum(0) + 2 * np.abs(want) + w_err)
    assert np.all(np.abs(mu - want) <= bound.astype(np.float64))
