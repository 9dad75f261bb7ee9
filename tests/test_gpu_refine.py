"""Refined field hits (refine_root) and the adjoint that reads their roots
(rt_trace.cu, rt_backward.cu).  The one-thread-per-query kernel refines where it
marches; the stage kernels mark their hits and refine them afterwards: the
records must be the same for every program that has a field stage.  The adjoint
of a record without a root (refine_root off in the call that made it) marches
the ray again: its gradient must equal that of the refined record."""
import numpy as np
import pytest

from synth import rays as R
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def world():
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("medium")
    scene = rq.rt_scene_build(torch.from_numpy(s.verts).cuda(), torch.from_numpy(s.tris).cuda())
    g = torch.empty((40, 33, 41), dtype=torch.float32, device="cuda")
    sdf = rq.rt_sdf_create(g, s.lo, s.hi)
    rq.rt_sdf_bake(scene, sdf, rq.BAKE_BVH)
    rays = R.gi_rays(s, 5000, 3, s.diagonal)
    rays[::97, 0] = np.nan      # invalid queries
    rays[5::101, 3] = 2.0       # marches that start along the ray
    rays[7::103, 0:3] = 0.01    # and beside a corner of the grid
    return rq, scene, sdf, torch.from_numpy(rays).cuda()


@pytest.mark.parametrize("layout", [0, 1, 2])
@pytest.mark.parametrize("mode,any_hit,m_near,m_far", [(3, False, 0, 0), (1, False, 2, 0), (1, True, 2, 0), (2, False, 1, 2),
                                                       (2, True, 2, 2), (1, False, 0, 0), (2, False, 0, 1)])
def test_stage_kernels_refine_as_one_thread_does(world, layout, mode, any_hit, m_near, m_far):
    rq, scene, sdf, rays = world
    p = rq.split_params(mode=mode, any_hit=any_hit, m_near=m_near, m_far=m_far, refine_root=True)
    prev = rq.rt_get_tuning()
    out = []
    try:
        for kernel in (rq.KERNEL_SIMPLE, rq.KERNEL_WAVEFRONT):
            rq.rt_set_tuning(prev, kernel=kernel, grid_layout=layout)
            for n in (rays.shape[0], 129, 1):
                hits = torch.full((n, 6), 0x102, dtype=torch.int32, device="cuda")  # stale records
                rq.rt_trace_combined(scene, sdf, rays[:n].contiguous(), p, hits=hits)
                out.append(hits.cpu().numpy())
    finally:
        rq.rt_set_tuning(prev)
    for a, b in zip(out[:3], out[3:]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("mode", [3, 1])
def test_adjoint_of_records_with_and_without_roots(world, mode):
    rq, scene, sdf, rays = world
    refined = rq.split_params(mode=mode, m_near=2.0, refine_root=True)
    raw = rq.split_params(mode=mode, m_near=2.0)
    gt = torch.rand(rays.shape[0], device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    grads = []
    for p in (refined, raw):
        hits = rq.rt_trace_combined(scene, sdf, rays, p)
        g = torch.zeros_like(sdf.grid)
        grads.append(rq.rt_trace_combined_backward(scene, sdf, rays, refined, hits, gt, g).double().cpu().numpy())
    # the same roots scattered in another order: single precision sums
    scale = np.abs(grads[0]).max()
    assert scale > 0 and np.abs(grads[0] - grads[1]).max() <= 1e-5 * scale
