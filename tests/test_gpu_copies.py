"""The copies of the grid (rt_sdf_prepare) for rows shorter and longer than a block:
the marches read the same values from them as from the caller's plain grid."""
import pytest

from synth import rays as R
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [2, 3, 5, 8, 17, 32, 33, 64, 65, 96, 97, 128, 129, 193, 300, 1025])
@pytest.mark.parametrize("ny,nz", [(9, 10), (2, 2), (33, 3)])
@pytest.mark.parametrize("dtype", ["float32", "float16"])
def test_equal_to_plain_grid(nx, ny, nz, dtype):
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("tiny")
    gen = torch.Generator(device="cuda").manual_seed(5)
    grid = (torch.rand((nz, ny, nx), generator=gen, device="cuda") * 0.3 + 0.02).to(getattr(torch, dtype))
    sdf = rq.rt_sdf_create(grid, s.lo, s.hi)
    rq.rt_sdf_prepare(sdf)
    rays = torch.from_numpy(R.gi_rays(s, 20000, 3, s.diagonal)).cuda()
    prev, out = rq.rt_get_tuning(), []
    try:
        for layout in (rq.LAYOUT_PLAIN, rq.LAYOUT_CELLS, rq.LAYOUT_PAIRS):
            rq.rt_set_tuning(prev, grid_layout=layout)
            out.append(rq.rt_trace_combined(None, sdf, rays, rq.split_params(mode=rq.MODE_SDF)))
    finally:
        rq.rt_set_tuning(prev)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
