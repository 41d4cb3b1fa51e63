"""Candidates and configurations with NaN or infinite entries: they are reported where they are, and
change nothing else."""
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


Q0, QD = np.array([-0.4, 0.4, -1.2, 0.5]), np.array([0.4, 0.6, -1.8, 1.5])


def _beside(boxes):
    """One obstacle in the crane's reach ahead of it: a trunk or a box."""
    from paper_2503_14160_gb300 import workloads
    if boxes:
        return workloads.Scene(np.zeros((0, 5)), np.array([[3.0, -2.0, 0.0, 6.0, 2.0, 15.0]]))
    return workloads.Scene(np.array([[4.0, 0.0, 0.5, 0.0, 15.0]]), np.zeros((0, 6)))


@pytest.mark.parametrize("boxes", [False, True])
@pytest.mark.parametrize("joint,value", [(2, np.nan), (3, np.nan)])
def test_hulls_report_a_nan_configuration(lib, crane, boxes, joint, value):
    """Hulls without a place beside an obstacle in the reach of the others have no separating axis:
    the depth is infinite, not 0."""
    import torch
    q = np.array([[0.0, 0.4, -1.0, 0.5], [0.0, 0.4, -1.0, 0.5]], np.float32)
    q[1, joint] = value
    with lib.Planner(crane, _beside(boxes), lib.make_params(4, 2, 2)) as pl:
        pen = torch.full((2,), -1.0, device="cuda")
        lib.cp_hull_penetration(pl.handle, torch.from_numpy(q).cuda(), 2, pen)
        torch.cuda.synchronize()
        pen = pen.cpu().numpy()
    assert np.isfinite(pen[0]) and pen[0] > 0.0
    assert pen[1] == np.inf


@pytest.mark.parametrize("boxes", [False, True])
def test_hull_paths_report_nan_checkpoints(lib, crane, boxes):
    import torch
    K, S = 8, 8
    f = (np.arange(1, K + 1) / (K + 1))[:, None]
    xi = np.repeat((Q0 + f * (QD - Q0))[None], 2, 0).astype(np.float32)
    xi[1, 3, 3] = np.nan
    with lib.Planner(crane, _beside(boxes), lib.make_params(2, K, S, collision_model=lib.CP_COLLISION_HULLS)) as pl:
        lib.cp_set_endpoints(pl.handle, Q0, QD)
        J = torch.zeros(2, dtype=torch.float64, device="cuda")
        flag = torch.zeros(2, dtype=torch.uint8, device="cuda")
        pen = torch.zeros(2, pl.n_s, device="cuda")
        lib.cp_evaluate(pl.handle, torch.from_numpy(xi).cuda(), 2, J, flag, None, None, pen)
        lib.cp_synchronize(pl.handle)
        J, flag, pen = J.cpu().numpy(), flag.cpu().numpy(), pen.cpu().numpy()
    # control point 3 (the seventh in all) acts on spans 3 .. 6 of the path
    near = pen[0, 3 * S:7 * S] > 0.0
    assert near.any() and np.isfinite(J[0])
    assert np.all(pen[1, 3 * S:7 * S][near] == np.inf)
    assert np.array_equal(pen[1, :3 * S], pen[0, :3 * S]) and np.array_equal(pen[1, 7 * S:], pen[0, 7 * S:])
    assert flag[1] == 1 and not np.isfinite(J[1])


@pytest.mark.parametrize("S", [2, 8, 24, 64])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_smooth_gradient_keeps_a_bad_entry_to_its_own_control_points(lib, crane, S, bad):
    """Control point 13 acts on four spans, and these on control points 10 .. 16: the others'
    gradients are those of the candidate without it, bit for bit. With 8 and 24 substeps a
    32-checkpoint chunk holds a bad span and a good one."""
    import torch
    from paper_2503_14160_gb300 import workloads
    K, n = 24, 2
    g = np.random.default_rng(S)
    f = (np.arange(1, K + 1) / (K + 1))[:, None]
    xi = ((Q0 + f * (QD - Q0))[None] + 0.02 * g.normal(size=(n, K, 4))).astype(np.float32)
    scene = workloads.make_scene(workloads.WORKLOADS["single_small"])
    out = []
    with lib.Planner(crane, scene, lib.make_params(n, K, S)) as pl:
        lib.cp_set_endpoints(pl.handle, Q0, QD)
        for value in (xi[1, 13, 1], bad):
            x = xi.copy()
            x[1, 13, 1] = value
            J = torch.zeros(n, dtype=torch.float64, device="cuda")
            d = torch.zeros(n, K, 4, device="cuda")
            lib.cp_smooth_cost_grad(pl.handle, torch.from_numpy(x).cuda(), n, None, J, d)
            lib.cp_synchronize(pl.handle)
            out.append((J.cpu().numpy(), d.cpu().numpy()))
    (J0, d0), (J1, d1) = out
    assert np.isfinite(d0).all() and np.isfinite(J0).all()
    far = np.r_[0:10, 17:K]
    np.testing.assert_array_equal(d1[0], d0[0])
    np.testing.assert_array_equal(d1[1, far], d0[1, far])
    assert J1[0] == J0[0] and not np.isfinite(J1[1]) and not np.isfinite(d1[1, 13]).all()


@pytest.mark.parametrize("joint,value", [(1, np.nan), (3, np.nan), (3, np.inf), (2, 1e30)])
def test_broad_phase_equals_exhaustive_beside_a_box(lib, crane, joint, value):
    """The default form and the exhaustive one give the same flags, penalties and costs for a
    candidate with such an entry, whose checkpoints the box is close to."""
    import torch
    K, S, n = 8, 8, 3
    f = (np.arange(1, K + 1) / (K + 1))[:, None]
    xi = np.repeat((Q0 + f * (QD - Q0))[None], n, 0).astype(np.float32)
    xi[1, 3, joint] = value
    out = []
    for exhaustive in (0, 1):
        with lib.Planner(crane, _beside(True), lib.make_params(n, K, S, eval_exhaustive=exhaustive)) as pl:
            lib.cp_set_endpoints(pl.handle, Q0, QD)
            J = torch.zeros(n, dtype=torch.float64, device="cuda")
            flag = torch.zeros(n, dtype=torch.uint8, device="cuda")
            terms = torch.zeros(n, 5, dtype=torch.float64, device="cuda")
            words = torch.zeros(n, (pl.n_s + 31) // 32, dtype=torch.int32, device="cuda")
            pen = torch.zeros(n, pl.n_s, device="cuda")
            lib.cp_evaluate(pl.handle, torch.from_numpy(xi).cuda(), n, J, flag, terms, words, pen)
            lib.cp_synchronize(pl.handle)
            out.append([t.cpu().numpy() for t in (J, flag, terms, words, pen)])
    assert out[0][1][0] == 1
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
