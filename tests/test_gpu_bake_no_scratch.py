"""An exact bake of a cascade whose scratch cannot be had (the sites of two levels)
still runs, by the search that needs none, with the same values."""
import pytest

from synth import scene as S
from tests.test_gpu_prepare_failure import MB, _leave_free

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["BAKE_BVH", "BAKE_AUTO"])
def test_bake_without_scratch(method):
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("medium")
    scene = rq.rt_scene_build(torch.from_numpy(s.verts).cuda(), torch.from_numpy(s.tris).cuda())
    assert scene.info().n_tris > 1024
    g = torch.empty((2, 256, 256, 256), dtype=torch.float32, device="cuda")
    sdf = rq.rt_cascade_create(g, 0.02, s.camera.eye)
    rq.rt_sdf_bake(scene, sdf, getattr(rq, method))
    want = g.clone()
    g.zero_()
    torch.cuda.synchronize()
    held = _leave_free(64 * MB)  # the sites of two levels are 128 MB
    try:
        assert torch.cuda.mem_get_info()[0] < 120 * MB
        rq.rt_sdf_bake(scene, sdf, getattr(rq, method))
        assert torch.equal(g, want)
    finally:
        held.clear()
        torch.cuda.empty_cache()
