"""The field build's sites at the edges of its kernels (rt_dfgen.cu): lines shorter
and longer than a warp, at and past the longest line swept in shared memory,
thin grids, a single triangle and triangles far larger than a voxel, against the
CPU checker, equal after every step."""
import numpy as np
import pytest

import oracle as O
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("n", [(33, 20, 31), (2, 65, 2), (64, 32, 3), (1024, 2, 3), (1025, 3, 2), (2, 2, 2)])
@pytest.mark.parametrize("keep", ["all", 1, 13])
def test_sites_equal_the_checker(n, keep):
    import paper_2305_07253_gb300 as rq

    s = S.make_scene("tiny")
    tris = s.tris if keep == "all" else np.ascontiguousarray(s.tris[:keep])
    scene, bvh = rq.rt_scene_build(_cuda(s.verts), _cuda(tris)), O.BVH(s.verts, tris)
    g = torch.empty((n[2], n[1], n[0]), dtype=torch.float32, device="cuda")
    sdf = rq.rt_sdf_create(g, s.lo, s.hi)
    for stage in (1, 2, 3):
        got = rq.rt_sdf_sites(scene, sdf, stage).cpu().numpy().reshape(-1)
        want = O.df_sites(bvh, O.Grid(s.lo, s.hi, list(n), values=np.zeros(n[0] * n[1] * n[2])), stage=stage)
        assert np.array_equal(got, want), stage
