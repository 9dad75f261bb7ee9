"""The stage kernels and the concurrent programs where the default tuning would take
one thread per query: pieces of rt_trace_combined_host on their own streams, mixed
batches in the pipeline (with and without near sub-intervals, in any query order),
and both under graph capture."""
import itertools

import numpy as np
import pytest

from synth import rays as R
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROGRAMS = [dict(mode=1, m_near=2.0), dict(mode=1, m_near=2.0, refine_root=True), dict(mode=1, m_near=2.0, any_hit=True),
            dict(mode=2, m_near=2.0, m_far=2.0), dict(mode=2, m_near=1.0, m_far=2.0, any_hit=True), dict(mode=0), dict(mode=3)]


@pytest.fixture(scope="module")
def world():
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("medium")
    scene = rq.rt_scene_build(torch.from_numpy(s.verts).cuda(), torch.from_numpy(s.tris).cuda())
    sdf = rq.rt_sdf_create(torch.empty((40, 33, 41), dtype=torch.float32, device="cuda"), s.lo, s.hi)
    cas = rq.rt_cascade_create(torch.empty((3, 20, 20, 20), dtype=torch.float32, device="cuda"), 0.2, s.camera.eye)
    for f in (sdf, cas):
        rq.rt_sdf_bake(scene, f, rq.BAKE_BVH)
    return rq, scene, (sdf, cas), R.gi_rays(s, 20000, 3, s.diagonal)


@pytest.fixture(params=["KERNEL_WAVEFRONT"])
def stages(world, request):
    rq = world[0]
    prev = rq.rt_get_tuning()
    rq.rt_set_tuning(prev, kernel=getattr(rq, request.param))
    yield rq
    rq.rt_set_tuning(prev)


def _params(rq, program):
    return rq.split_params(**{"m_near": 0.0, "m_far": 0.0, **program})


def _same(rq, p, a, b):
    if p.any_hit:  # the same outcome; which triangle is any of those hit
        a, b = a[:, 4], b[:, 4]
    return torch.equal(a.cpu(), b.cpu())


def _host_call(rq, scene, sdf, rays, p, chunks, stream=None):
    n = rays.shape[0]
    rays_h = torch.from_numpy(rays).pin_memory()
    hits_h = torch.full((n, 6), 7, dtype=torch.int32).pin_memory()
    rays_d, hits_d = torch.empty((n, 8), device="cuda"), torch.empty((n, 6), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    rq.trace_combined_from_host(scene, sdf, rays_h, p, hits_h, rays_d, hits_d, chunks=chunks, stream=stream)
    return hits_h, (rays_h, rays_d, hits_d)


@pytest.mark.parametrize("program", range(len(PROGRAMS)))
@pytest.mark.parametrize("chunks", [0, 3, 7, 64])
@pytest.mark.parametrize("field", [0, 1])
def test_host_pieces(world, stages, program, chunks, field):
    rq, scene, fields, rays = world
    p = _params(rq, PROGRAMS[program])
    want = rq.rt_trace_combined(scene, fields[field], torch.from_numpy(rays).cuda(), p)
    got, _ = _host_call(rq, scene, fields[field], rays, p, chunks)
    torch.cuda.synchronize()
    assert _same(rq, p, got, want)


def test_large_host_pieces_on_two_streams(world):
    """Pieces of more than 131,072 queries take the stage kernels by themselves; calls
    on different streams share the library's, one after another."""
    rq, scene, fields, rays = world
    many = np.concatenate([rays] * 55)  # six pieces of 110,000 to 220,000
    p = _params(rq, PROGRAMS[0])
    calls = []
    for k, field in itertools.product(range(2), range(2)):
        r = np.roll(many, 1000 * k, axis=0)
        calls.append((r, field, _host_call(rq, scene, fields[field], r, p, 0, torch.cuda.Stream())))
    torch.cuda.synchronize()
    for r, field, (got, _) in calls:
        assert torch.equal(got, rq.rt_trace_combined(scene, fields[field], torch.from_numpy(r).cuda(), p).cpu())


@pytest.mark.parametrize("programs", [range(len(PROGRAMS)), (2, 4, 5, 6), (5,), (5, 0, 1)])
@pytest.mark.parametrize("field", [0, 1])
def test_batches(world, stages, programs, field):
    """programs (2, 4, 5, 6) and (5,) have no closest-hit near sub-interval: the launches
    run in sequence; the others run the concurrent program."""
    rq, scene, fields, rays = world
    refine = 1 in programs  # one value for all batches of a call
    ps = [_params(rq, {**PROGRAMS[k], "refine_root": refine}) for k in programs]
    batches = [(torch.from_numpy(rays[977 * k: 977 * k + 2900 + 31 * k]).cuda(), p) for k, p in enumerate(ps)]
    want = [rq.rt_trace_combined(scene, fields[field], r, p) for r, p in batches]
    prev = rq.rt_get_tuning()
    for bits in (0, 1, 3, 5):
        rq.rt_set_tuning(prev, order_bits=bits)
        for (_, p), got, w in zip(batches, rq.rt_trace_batches(scene, fields[field], batches), want):
            assert _same(rq, p, got, w), (bits, p.mode)
    # and replayed from a graph
    rq.rt_set_tuning(prev)
    hits = [torch.full_like(w, -1) for w in want]
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s), torch.cuda.graph(g, stream=s):
        rq.rt_trace_batches(scene, fields[field], [(r, p, h) for (r, p), h in zip(batches, hits)], stream=s)
    torch.cuda.current_stream().wait_stream(s)
    for _ in range(2):
        for h in hits:
            h.fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        assert all(_same(rq, p, h, w) for (_, p), h, w in zip(batches, hits, want))


@pytest.mark.parametrize("program", range(len(PROGRAMS)))
def test_captured_call(world, stages, program):
    rq, scene, fields, rays = world
    p, r = _params(rq, PROGRAMS[program]), torch.from_numpy(rays).cuda()
    want = rq.rt_trace_combined(scene, fields[0], r, p)
    hits = torch.full_like(want, -1)
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s), torch.cuda.graph(g, stream=s):
        rq.rt_trace_combined(scene, fields[0], r, p, hits=hits, stream=s)
    torch.cuda.current_stream().wait_stream(s)
    g.replay()
    torch.cuda.synchronize()
    assert _same(rq, p, hits, want)
