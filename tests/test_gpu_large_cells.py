"""The cell copy of a float32 grid of 2^26 entries or more holds both faces of every
cell, a smaller one each face once: the marches must read the same values from
either as from the caller's plain grid."""
import pytest

from synth import rays as R
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# (nx, ny, nz): nx (ny-1) (nz-1) just below 2^26, at it, and above with odd extents
@pytest.mark.parametrize("n", [(512, 513, 256), (512, 513, 257), (257, 513, 514), (2051, 260, 131), (3, 4736, 4737)])
@pytest.mark.parametrize("dtype", ["float32", "float16"])
def test_equal_to_plain_grid(n, dtype):
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("tiny")
    scene = rq.rt_scene_build(torch.from_numpy(s.verts).cuda(), torch.from_numpy(s.tris).cuda())
    gen = torch.Generator(device="cuda").manual_seed(5)
    grid = (torch.rand((n[2], n[1], n[0]), generator=gen, device="cuda") * 0.3 + 0.02).to(getattr(torch, dtype))
    sdf = rq.rt_sdf_create(grid, s.lo, s.hi)
    rq.rt_sdf_prepare(sdf)
    rays = torch.from_numpy(R.gi_rays(s, 140000, 3, s.diagonal)).cuda()
    p = rq.split_params(mode=rq.MODE_SPLIT1, m_near=2.0)
    prev, out = rq.rt_get_tuning(), []
    try:
        for layout in (rq.LAYOUT_CELLS, rq.LAYOUT_PLAIN):
            rq.rt_set_tuning(prev, grid_layout=layout)
            out.append([rq.rt_trace_combined(scene, sdf, rays[:k], p) for k in (2000, 140000)])
    finally:
        rq.rt_set_tuning(prev)
    for a, b in zip(*out):
        assert torch.equal(a, b)
