"""The adjoint after the grid has changed between the forward call and it
(rt_trace_combined_backward): a new surface in front of the old one makes the old
record's t a root that is no longer the first, and the gradient must be that of
the grid as it is now.  Only records of the very copies that the adjoint reads
(rt_sdf_version) are taken without marching."""
import pytest

from synth import rays as R
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture()
def world():
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("medium")
    scene = rq.rt_scene_build(torch.from_numpy(s.verts).cuda(), torch.from_numpy(s.tris).cuda())
    g = torch.empty((40, 33, 41), dtype=torch.float32, device="cuda")
    sdf = rq.rt_sdf_create(g, s.lo, s.hi)
    rq.rt_sdf_bake(scene, sdf, rq.BAKE_BVH)
    return rq, scene, sdf, torch.from_numpy(R.gi_rays(s, 6000, 3, s.diagonal)).cuda()


def _new_surface(sdf):
    """A slab across the middle of the room, about a voxel and a half thick."""
    n = sdf.grid.shape[2]
    x = torch.arange(n, device="cuda", dtype=torch.float32)
    h = (float(sdf.hi[0]) - float(sdf.lo[0])) / (n - 1)
    return torch.minimum(sdf.grid.detach(), ((x - 0.52 * n).abs() - 1.5)[None, None, :] * h)


def _equal(a, b):
    a, b = a.double(), b.double()  # the same roots scattered in another order: single precision sums
    assert float(a.abs().max()) > 0 and float((a - b).abs().max()) <= 1e-5 * float(a.abs().max())


@pytest.mark.parametrize("mode", [3, 1])
def test_adjoint_of_old_records_is_the_new_grids(world, mode):
    rq, scene, sdf, rays = world
    p = rq.split_params(mode=mode, m_near=2.0, refine_root=True)
    old = rq.rt_trace_combined(scene, sdf, rays, p)
    sdf.grid.copy_(_new_surface(sdf))
    rq.rt_sdf_prepare(sdf)
    new = rq.rt_trace_combined(scene, sdf, rays, p)
    both = (old[:, 4] == rq.TRACER_SDF) & (new[:, 4] == rq.TRACER_SDF)
    moved = both & (rq.hit_fields(new)["t"] < 0.9 * rq.hit_fields(old)["t"])
    assert int(moved.sum()) > 300
    gt = torch.rand(rays.shape[0], device="cuda", generator=torch.Generator("cuda").manual_seed(1)) * both
    grads = [rq.rt_trace_combined_backward(scene, sdf, rays, p, h, gt, torch.zeros_like(sdf.grid)) for h in (old, new)]
    _equal(*grads)


def test_autograd_after_a_change(world):
    rq, scene, sdf, rays = world
    p = rq.split_params(mode=rq.MODE_SDF)
    gt = torch.rand(rays.shape[0], device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    sdf.grid.requires_grad_(True)
    t0, h0 = rq.SdfHitDistance.apply(sdf.grid, rays, None, sdf, p)
    with torch.no_grad():
        sdf.grid.copy_(_new_surface(sdf))
    t1, h1 = rq.SdfHitDistance.apply(sdf.grid, rays, None, sdf, p)  # prepares the new values
    both = (h0[:, 4] == rq.TRACER_SDF) & (h1[:, 4] == rq.TRACER_SDF)
    _equal(*(torch.autograd.grad(t, sdf.grid, grad_outputs=gt * both)[0] for t in (t0, t1)))


def test_version_of_the_copies(world):
    rq, scene, sdf, rays = world
    fresh = rq.rt_sdf_create(sdf.grid, sdf.lo, sdf.hi)
    assert rq.rt_sdf_version(fresh) == 0
    rq.rt_sdf_prepare(fresh)
    v = rq.rt_sdf_version(fresh)
    assert v > 0
    rq.rt_sdf_bake(scene, fresh, rq.BAKE_BVH)
    assert rq.rt_sdf_version(fresh) > v
    p = rq.split_params(mode=rq.MODE_SDF, refine_root=True)
    v, hits = rq.rt_sdf_version(fresh), rq.rt_trace_combined(None, fresh, rays, p)
    gt = torch.ones(rays.shape[0], device="cuda")
    _equal(*(rq.rt_trace_combined_backward(None, fresh, rays, p, hits, gt, torch.zeros_like(fresh.grid), version=k)
             for k in (0, v)))
    # a captured prepare may be replayed at any time
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s), torch.cuda.graph(g, stream=s):
        rq.rt_sdf_prepare(fresh, stream=s)
    torch.cuda.current_stream().wait_stream(s)
    assert rq.rt_sdf_version(fresh) == 0
    fresh.grid.copy_(_new_surface(fresh))
    g.replay()
    new = rq.rt_trace_combined(None, fresh, rays, p)
    both = ((hits[:, 4] == rq.TRACER_SDF) & (new[:, 4] == rq.TRACER_SDF)).float()
    _equal(*(rq.rt_trace_combined_backward(None, fresh, rays, p, h, both, torch.zeros_like(fresh.grid), version=v)
             for h in (hits, new)))
