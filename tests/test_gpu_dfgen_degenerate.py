"""The field build on meshes with triangles of two or three equal vertices
(rt_dfgen.cu).  The squared distance to such a triangle is not a number at many
positions; the steps must treat it as the CPU checker does, so that the sites are
equal after every step."""
import numpy as np
import pytest

import oracle as O
from synth import scene as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("kind", ["ab", "bc", "ca", "point", "line", "mixed"])
@pytest.mark.parametrize("share", [1.0, 0.3])
@pytest.mark.parametrize("n", [(33, 20, 31), (64, 32, 3), (1025, 3, 2)])
def test_sites_equal_the_checker(kind, share, n):
    import paper_2305_07253_gb300 as rq

    rng = np.random.default_rng(11)
    s = S.make_scene("tiny")
    tris = s.tris[:: max(1, len(s.tris) // 300)].copy()
    verts = np.concatenate([s.verts, s.verts])
    for k in np.nonzero(rng.uniform(size=len(tris)) < share)[0]:
        a, b, c = tris[k]
        how = kind if kind != "mixed" else ("ab", "bc", "ca", "point", "line")[rng.integers(5)]
        if how == "line":  # three points on a line, exactly
            verts[len(s.verts) + c] = 0.5 * (verts[a] + verts[b])
        tris[k] = {"ab": (a, a, c), "bc": (a, b, b), "ca": (a, b, a), "point": (a, a, a),
                   "line": (a, b, len(s.verts) + c)}[how]
    tris = np.ascontiguousarray(tris)
    scene, bvh = rq.rt_scene_build(_cuda(verts), _cuda(tris)), O.BVH(verts, tris)
    sdf = rq.rt_sdf_create(torch.empty((n[2], n[1], n[0]), dtype=torch.float32, device="cuda"), s.lo, s.hi)
    for stage in (1, 2, 3):
        got = rq.rt_sdf_sites(scene, sdf, stage).cpu().numpy().reshape(-1)
        want = O.df_sites(bvh, O.Grid(s.lo, s.hi, list(n), values=np.zeros(n[0] * n[1] * n[2])), stage=stage)
        assert np.array_equal(got, want), (stage, int((got != want).sum()))
