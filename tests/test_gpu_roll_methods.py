"""A rolling update gives the values of a full bake at the new place by the method of
the cascade's last bake (rt_cascade_recenter): the squared distances of
RT_BAKE_BRUTE, and of RT_BAKE_AUTO at these sizes, are summed in another order than
RT_BAKE_BVH's, and a moved level must not mix the two."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["BAKE_AUTO", "BAKE_BRUTE", "BAKE_BVH"])
@pytest.mark.parametrize("tris", [200, 3000])
@pytest.mark.parametrize("n,move", [(17, (1, 0, 0)), (17, (3, -2, 1)), (33, (-9, 5, 16)), (17, (40, 0, 0))])
def test_rolled_levels_equal_fresh_ones(method, tris, n, move):
    import paper_2305_07253_gb300 as rq

    rng = np.random.default_rng(7)
    V = (rng.uniform(0, 4, (tris, 1, 3)) + rng.normal(size=(tris, 3, 3)) * rng.uniform(0.02, 0.4, (tris, 1, 1)))
    F = np.arange(3 * tris, dtype=np.int32).reshape(tris, 3)
    scene = rq.rt_scene_build(torch.from_numpy(V.astype(np.float32).reshape(-1, 3)).cuda(), torch.from_numpy(F).cuda())
    method = getattr(rq, method)
    c0 = np.array([2.05, 2.05, 2.05])
    g = torch.empty((3, n, n, n), dtype=torch.float32, device="cuda")
    sdf = rq.rt_cascade_create(g, 0.1, c0)
    rq.rt_sdf_bake(scene, sdf, method)
    for c in (c0 + 0.1 * np.array(move), c0 - 0.1 * np.array(move)):
        rq.rt_cascade_recenter(scene, sdf, c)
        fresh = torch.empty_like(g)
        rq.rt_sdf_bake(scene, rq.rt_cascade_create(fresh, 0.1, c), method)
        assert torch.equal(g, fresh)
