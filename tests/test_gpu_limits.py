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
