"""Small calls run one thread per query in one launch (RT_KERNEL_AUTO), single
calls and mixed batches: their records must equal the stage kernels', for every
program, grid layout and tree, around the sizes where the choice changes, and
the call can be captured in a CUDA graph."""
import numpy as np
import pytest

from synth import rays as R
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

INF = float("inf")
PROGRAMS = [dict(mode=0), dict(mode=0, any_hit=True), dict(mode=1, m_near=2.0), dict(mode=1, m_near=INF), dict(mode=1, m_near=0.0),
            dict(mode=1, m_near=1.0, any_hit=True), dict(mode=2, m_near=2.0, m_far=1.0), dict(mode=2, m_near=2.0, m_far=2.0, any_hit=True),
            dict(mode=3)]


@pytest.fixture(scope="module")
def world():
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("medium")
    scene = rq.rt_scene_build(torch.from_numpy(s.verts).cuda(), torch.from_numpy(s.tris).cuda())
    fields = []
    for dtype in (torch.float32, torch.float16):
        g = torch.empty((40, 33, 41), dtype=dtype, device="cuda")
        fields.append(rq.rt_sdf_create(g, s.lo, s.hi))
        c = torch.empty((3, 20, 20, 20), dtype=dtype, device="cuda")
        fields.append(rq.rt_cascade_create(c, 0.2, s.camera.eye))
    for f in fields:
        rq.rt_sdf_bake(scene, f, rq.BAKE_BVH)
    rays = np.concatenate([R.gi_rays(s, 66000, 3, s.diagonal), R.primary_rays(s, 300, 220)])
    rays[::997, 4] = np.nan
    rays[3::991, 3] = 1e3  # t_min > t_max
    return rq, scene, fields, torch.from_numpy(rays).cuda()


def _both(rq, call):
    prev = rq.rt_get_tuning()
    out = []
    try:
        for kernel in (rq.KERNEL_AUTO, rq.KERNEL_WAVEFRONT):
            rq.rt_set_tuning(prev, kernel=kernel)
            out.append(call())
    finally:
        rq.rt_set_tuning(prev)
    return out


@pytest.mark.parametrize("n", [1, 33, 1000, 65537, 131072, 131073])
@pytest.mark.parametrize("program", range(len(PROGRAMS)))
@pytest.mark.parametrize("field", range(4))
def test_single_calls(world, n, program, field):
    rq, scene, fields, rays = world
    p = rq.split_params(**{"m_far": 0.0, **PROGRAMS[program]})
    a, b = _both(rq, lambda: rq.rt_trace_combined(scene, fields[field], rays[:n], p,
                                                  hits=torch.full((n, 6), 7, dtype=torch.int32, device="cuda")))
    assert torch.equal(a, b)


@pytest.mark.parametrize("layout,width", [(1, 2), (2, 2), (0, 8)])
def test_layouts_and_trees(world, layout, width):
    rq, scene, fields, rays = world
    prev = rq.rt_set_tuning(grid_layout=layout, bvh_width=width)
    try:
        for pr in PROGRAMS:
            p = rq.split_params(**{"m_far": 0.0, **pr})
            a, b = _both(rq, lambda: rq.rt_trace_combined(scene, fields[0], rays[:3000], p))
            assert torch.equal(a, b)
    finally:
        rq.rt_set_tuning(prev)


@pytest.mark.parametrize("sizes", [(5, 0, 700, 33), (40000, 60000, 1, 31071), (40000, 60000, 1, 31072)])
@pytest.mark.parametrize("field", range(4))
def test_batches(world, sizes, field):
    rq, scene, fields, rays = world
    for first in (0, 5):
        ps = [rq.split_params(**{"m_far": 0.0, **PROGRAMS[(first + k) % len(PROGRAMS)]}) for k in range(len(sizes))]
        a, b = _both(rq, lambda: rq.rt_trace_batches(scene, fields[field], [(rays[:n], p) for n, p in zip(sizes, ps)]))
        for x, y in zip(a, b):
            assert torch.equal(x, y)


def test_capture(world):
    rq, scene, fields, rays = world
    p = rq.split_params(mode=1, m_near=2.0)
    want = rq.rt_trace_combined(scene, fields[0], rays[:1000], p)
    hits, other = torch.zeros_like(want), torch.zeros_like(want)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        rq.rt_trace_combined(scene, fields[0], rays[:1000], p, hits=hits)
        rq.rt_trace_batches(scene, fields[0], [(rays[:1000], p, other)])
    hits.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(hits, want) and torch.equal(other, want)


@pytest.mark.parametrize("block", [32, 1024])
def test_any_block_of_the_tuning(world, block):
    """A block that only the stage kernels can hold still serves small calls."""
    rq, scene, fields, rays = world
    p = rq.split_params(mode=1, m_near=2.0)
    want = rq.rt_trace_combined(scene, fields[0], rays[:777], p)
    prev = rq.rt_set_tuning(block=block)
    try:
        got = rq.rt_trace_combined(scene, fields[0], rays[:777], p)
        batch = rq.rt_trace_batches(scene, fields[0], [(rays[:777], p)])[0]
    finally:
        rq.rt_set_tuning(prev)
    assert torch.equal(got, want) and torch.equal(batch, want)
