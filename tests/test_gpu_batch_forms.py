"""The forms that a batch chooses by its size, against its planners alone (which rank and factor
query by query): one-launch radix passes over more than 16384 candidates, two passes over the query
for more than 256 queries, and one CTA per factor for more queries than two waves of clusters."""
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


def _check(lib, crane, sizes, iters, S, alone, scene=None):
    """Runs the batch of (N, K) and plans the queries `alone` by themselves: same control points,
    costs and elites."""
    import torch
    from paper_2503_14160_gb300 import workloads
    nq = len(sizes)
    g = np.random.default_rng(nq)
    lo, hi = np.asarray(crane.q_min), np.asarray(crane.q_max)
    ends = lo + (hi - lo) * (0.25 + 0.5 * g.random((nq, 2, 4)))
    scene = scene or workloads.empty_scene()
    scenes = [lib.HostScene.from_scene(scene) for _ in sizes]
    params = [lib.make_params(N, K, S, seed=q, query=q, grid_cell=0.5) for q, (N, K) in enumerate(sizes)]
    b = lib.cp_batch_init(lib.make_model(crane), scenes, params, list(ends[:, 0]), list(ends[:, 1]), iters)
    try:
        res = lib.cp_batch_run(b, nq, K=[K for _, K in sizes])
        for q in alone:
            N, K = sizes[q]
            p = lib.cp_batch_planner(b, q)
            el = torch.zeros(2, N // 2, dtype=torch.int32, device="cuda")
            lib.cp_get_elites(p, el[0])
            lib.cp_synchronize(p)
            lib.cp_set_endpoints(p, ends[q, 0], ends[q, 1])
            ctrl, st = lib.cp_plan(p, iters, K=K)
            lib.cp_get_elites(p, el[1])
            lib.cp_synchronize(p)
            np.testing.assert_array_equal(res[q][0], ctrl)
            assert res[q][1]["J"] == st["J"] and res[q][1]["best_J"] == st["best_J"]
            el = el.cpu().numpy()
            np.testing.assert_array_equal(el[0], el[1])
    finally:
        lib.cp_batch_destroy(b)


@pytest.mark.parametrize("Ns", [[16383, 2], [8193, 8192], [5000, 1025, 9999, 1, 513],
                                [20000], [1023] * 17 + [7]])
def test_batches_of_more_than_16384_candidates(lib, crane, Ns):
    """Ragged queries whose boundaries lie inside the sort's tiles of 1024 (and a total of 16385).
    With few substeps and an empty scene, cost ties and near ties are common."""
    Ns = [max(n, 2) for n in Ns]
    _check(lib, crane, [(n, 2 + q % 3) for q, n in enumerate(Ns)], 3, 2, range(len(Ns)))


def test_equal_costs_across_queries(lib, crane):
    """An initial spread of zero makes every candidate of a query the same: all ties, kept in index
    order in every query."""
    import torch
    from paper_2503_14160_gb300 import workloads
    Ns = [6000, 7001, 5003]
    ends = (np.array([0.3, 0.4, -1.2, 0.5]), np.array([-1.0, 0.6, -1.8, 1.5]))
    params = [lib.make_params(n, 2, 2, seed=1, query=q, grid_cell=0.5, init_std_frac=1e-30, eps=1e-60)
              for q, n in enumerate(Ns)]
    scenes = [lib.HostScene.from_scene(workloads.empty_scene()) for _ in Ns]
    b = lib.cp_batch_init(lib.make_model(crane), scenes, params, [ends[0]] * 3, [ends[1]] * 3, 1)
    try:
        lib.cp_batch_run(b, 3)
        for q, n in enumerate(Ns):
            el = torch.zeros(n // 2, dtype=torch.int32, device="cuda")
            lib.cp_get_elites(lib.cp_batch_planner(b, q), el)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(el.cpu().numpy(), np.arange(n // 2))
    finally:
        lib.cp_batch_destroy(b)


@pytest.mark.parametrize("nq,N", [(257, 65), (300, 33)])
def test_batches_of_more_than_256_queries(lib, crane, nq, N):
    """257 queries of 65 candidates and more in all than 16384 (one-launch passes), 300 of 33 (three
    launches per pass): both take two passes over the query."""
    _check(lib, crane, [(N + q % 2, 1 + q % 3) for q in range(nq)], 2, 2, (0, 1, 127, 255, 256, nq - 1))


@pytest.mark.parametrize("K", [4, 17, 32])
def test_batch_factors_by_one_cta_each(lib, crane, K):
    """700 queries, more than two waves of clusters of any size: their factors come from one CTA
    per query, and the plans are those of the planners, whose factors come from a cluster."""
    _check(lib, crane, [(8, K)] * 700, 3, 1, (0, 1, 350, 699))
