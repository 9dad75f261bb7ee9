"""Builds and bakes on many streams at once need scratch for all of them; once they
are done the library keeps at most 128 MB of it (rt_scratch_alloc)."""
import pytest

from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


def test_scratch_of_many_streams_is_given_back():
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("tiny")
    scene = rq.rt_scene_build(torch.from_numpy(s.verts).cuda(), torch.from_numpy(s.tris).cuda())
    sdf = rq.rt_sdf_create(torch.empty((128, 128, 128), device="cuda"), s.lo, s.hi)  # about 36 MB of scratch a call
    want = rq.rt_sdf_sites(scene, sdf, 3)
    streams = [torch.cuda.Stream() for _ in range(16)]
    out = [torch.empty_like(want) for _ in streams]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for st, o in zip(streams, out):
        st.wait_stream(torch.cuda.current_stream())
        rq.rt_sdf_sites(scene, sdf, 3, out=o, stream=st)
    for st in streams:
        st.synchronize()
    torch.cuda.synchronize()
    assert all(torch.equal(o, want) for o in out)
    assert free - torch.cuda.mem_get_info()[0] <= 160 * MB  # (allocated in steps of 32 MB)
