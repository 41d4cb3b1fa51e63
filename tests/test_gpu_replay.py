"""A recorded plan is replayed only for the scene it was recorded for: what its launches hold by
value is compared, not only the obstacles' addresses and number."""
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
        (np.array([0.7, 0.5, -0.9, 1.0]), np.array([1.4, 0.6, -1.1, 1.5]))]


@pytest.mark.parametrize("form", ["hulls", "broad", "polar"])
@pytest.mark.parametrize("second", [0, 1])
def test_recorded_plan_takes_a_new_scene(lib, crane, form, second):
    """One trunk replaced by another of the same height, thick enough that the prism around it
    reaches metres beyond the circle; then the first scene again. With the same end points and with
    others."""
    import torch
    from paper_2503_14160_gb300 import workloads
    kw = {"hulls": {"collision_model": lib.CP_COLLISION_HULLS}, "polar": {"grid_cell": 0.5}}.get(form, {})
    thin = workloads.Scene(np.array([[6.0, 3.0, 0.3, 0.0, 15.0]]), np.zeros((0, 6)))
    thick = workloads.Scene(np.array([[34.0, 0.0, 30.0, 0.0, 15.0]]), np.zeros((0, 6)))
    K = 5
    params = lib.make_params(200, K, 9, **kw, max_grid_items=4096 if form == "polar" else 0)
    st = torch.cuda.Stream()
    plans = [(thin, 0), (thick, second), (thin, 0)]
    got = []
    with lib.Planner(crane, thin, params, st) as kept:
        for scene, e in plans:
            lib.cp_set_scene(kept.handle, lib.HostScene.from_scene(scene))
            lib.cp_set_endpoints(kept.handle, *ENDS[e])
            got.append(lib.cp_plan(kept.handle, 4, K=K))
    for (scene, e), (ctrl, stats) in zip(plans, got):
        with lib.Planner(crane, scene, params, st) as fresh:
            lib.cp_set_endpoints(fresh.handle, *ENDS[e])
            want_ctrl, want = lib.cp_plan(fresh.handle, 4, K=K)
        assert np.array_equal(ctrl, want_ctrl)
        assert stats == want
