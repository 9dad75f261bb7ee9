"""A prepare that cannot have the memory for its copies (rt_sdf_prepare) returns
RT_ERR_OOM and leaves the handle as it was: traces read the plain grid, the copy
that was there is read on, and a later prepare succeeds."""
import pytest

from synth import rays as R
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


def _leave_free(nbytes):
    """Hold all device memory but nbytes to nbytes + 32 MB.  First everything, so that
    what idle memory pools keep (an allocation that fails empties them) is held too."""
    torch.cuda.empty_cache()
    held = [torch.empty(max(torch.cuda.mem_get_info()[0] - 4096 * MB, 32 * MB), dtype=torch.uint8, device="cuda")]
    try:
        while True:
            held.append(torch.empty(32 * MB, dtype=torch.uint8, device="cuda"))
    except torch.cuda.OutOfMemoryError:
        pass
    while torch.cuda.mem_get_info()[0] < nbytes:
        held.pop()
        torch.cuda.empty_cache()
    return held


@pytest.mark.parametrize("dtype,n", [("float32", (256, 256, 256)), ("float16", (320, 255, 301))])
def test_failed_prepare_changes_no_record(dtype, n):
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("tiny")
    gen = torch.Generator(device="cuda").manual_seed(5)
    grid = (torch.rand((n[2], n[1], n[0]), generator=gen, device="cuda") * 0.3 + 0.02).to(getattr(torch, dtype))
    rays = torch.from_numpy(R.gi_rays(s, 20000, 3, s.diagonal)).cuda()
    p = rq.split_params(mode=rq.MODE_SDF)
    hits = torch.empty((rays.shape[0], 6), dtype=torch.int32, device="cuda")
    want = rq.rt_trace_combined(None, rq.rt_sdf_create(grid, s.lo, s.hi), rays, p)  # the plain grid
    sdf = rq.rt_sdf_create(grid, s.lo, s.hi)
    esz = grid.element_size()
    cells, pairs = 4 * esz * n[0] * (n[1] - 1) * (n[2] - 1), 2 * esz * (n[0] - 1) * n[1] * n[2]
    held = _leave_free(cells + pairs // 2)  # room for the larger copy, not for both
    free = torch.cuda.mem_get_info()[0]
    assert cells + 4 * MB < free < cells + pairs - 4 * MB
    try:
        with pytest.raises(rq.RtError):
            rq.rt_sdf_prepare(sdf)
        assert abs(torch.cuda.mem_get_info()[0] - free) <= 4 * MB  # nothing kept
        assert torch.equal(rq.rt_trace_combined(None, sdf, rays, p, hits=hits), want)
    finally:
        held.clear()
        torch.cuda.empty_cache()
    rq.rt_sdf_prepare(sdf)
    assert torch.equal(rq.rt_trace_combined(None, sdf, rays, p, hits=hits), want)
