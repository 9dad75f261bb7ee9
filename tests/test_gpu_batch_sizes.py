"""rt_trace_batches around the sizes where the default tuning goes over from one
thread per query to the stage kernels: the records equal the stage kernels'."""
import pytest

from synth import rays as R
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROGRAMS = [dict(mode=1, m_near=2.0), dict(mode=2, m_near=2.0, m_far=2.0, any_hit=True), dict(mode=0), dict(mode=3)]


@pytest.fixture(scope="module")
def world():
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("medium")
    scene = rq.rt_scene_build(torch.from_numpy(s.verts).cuda(), torch.from_numpy(s.tris).cuda())
    sdf = rq.rt_sdf_create(torch.empty((40, 33, 41), dtype=torch.float32, device="cuda"), s.lo, s.hi)
    cas = rq.rt_cascade_create(torch.empty((3, 20, 20, 20), dtype=torch.float32, device="cuda"), 0.2, s.camera.eye)
    for f in (sdf, cas):
        rq.rt_sdf_bake(scene, f, rq.BAKE_BVH)
    return rq, scene, (sdf, cas), torch.from_numpy(R.gi_rays(s, 140000, 3, s.diagonal)).cuda()


@pytest.mark.parametrize("total", [131072, 131073, 524287, 524288, 524289])
@pytest.mark.parametrize("programs", [(0, 1, 2, 3), (2, 2, 2, 2)])
@pytest.mark.parametrize("field", [0, 1])
def test_records_equal_the_stage_kernels(world, total, programs, field):
    rq, scene, fields, rays = world
    sizes = [total // 4, total // 4, total // 4, total - 3 * (total // 4)]
    batches = [(rays[k:k + n], rq.split_params(**{"m_near": 0.0, "m_far": 0.0, **PROGRAMS[q]}))
               for k, (n, q) in enumerate(zip(sizes, programs))]
    prev, out = rq.rt_get_tuning(), []
    try:
        for kernel in (rq.KERNEL_AUTO, rq.KERNEL_WAVEFRONT):
            rq.rt_set_tuning(prev, kernel=kernel)
            out.append(rq.rt_trace_batches(scene, fields[field], batches))
    finally:
        rq.rt_set_tuning(prev)
    for (_, p), a, b in zip(batches, *out):
        if p.any_hit:  # the same outcome; which triangle is any of those hit
            a, b = a[:, 4], b[:, 4]
        assert torch.equal(a, b)
