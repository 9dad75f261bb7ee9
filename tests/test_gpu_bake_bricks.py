"""The brick search of the exact bake (rt_bake.cu) against the brute force
kernel, at the edges of its brick sizes, on badly shaped triangles and far from
the origin.  RT_BAKE_AUTO promises the brute force kernel's values at these
sizes, so the distances are compared bit for bit; the sign where it is decided
by more than rounding."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _mesh(kind, n, seed):
    rng = np.random.default_rng(seed)
    c = rng.uniform(0, 4, (n, 1, 3))
    if kind == "slivers":  # nearly parallel edges, and some triangles of no area
        e = rng.normal(size=(n, 1, 3)) * np.array([0.0, 0.5, 1.0])[None, :, None]
        V = c + e + rng.normal(size=(n, 3, 3)) * rng.choice([0.0, 1e-6, 1e-3], (n, 1, 1))
    elif kind == "shell":  # a round object around the middle: samples almost equidistant from all triangles
        d = rng.normal(size=(n, 1, 3))
        d /= np.linalg.norm(d, axis=2, keepdims=True)
        t = rng.normal(size=(n, 3, 3)) * 0.05
        V = 2 + d * 1.5 + t - (t * d).sum(2, keepdims=True) * d
    else:
        V = c + rng.normal(size=(n, 3, 3)) * rng.uniform(0.02, 0.4, (n, 1, 1))
    if kind == "far":
        V = V + np.array([700.0, -900.0, 500.0])
    return V.astype(np.float32).reshape(-1, 3), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


def _equal(a, b):
    assert np.array_equal(np.abs(a), np.abs(b))
    sure = np.abs(b) > 1e-3
    assert np.mean((a == b)[sure]) > 0.999  # a sign turns only where the pseudonormal is perpendicular


@pytest.mark.parametrize("kind", ["plain", "slivers", "shell", "far"])
@pytest.mark.parametrize("shape,f16", [((2, 2, 2), False), ((3, 97, 2), False), ((32, 32, 32), True),
                                       ((33, 31, 33), False), ((80, 81, 82), False)])
def test_auto_equals_brute(kind, shape, f16):
    import paper_2305_07253_gb300 as rq

    V, F = _mesh(kind, 700, 3)
    scene = rq.rt_scene_build(torch.from_numpy(V).cuda(), torch.from_numpy(F).cuda())
    lo, hi = V.min(0) - 0.3, V.max(0) + 0.2
    out = []
    for method in (rq.BAKE_AUTO, rq.BAKE_BRUTE):
        g = torch.empty(shape, dtype=torch.float16 if f16 else torch.float32, device="cuda")
        rq.rt_sdf_bake(scene, rq.rt_sdf_create(g, lo, hi), method)
        out.append(g.float().cpu().numpy())
    _equal(*out)


@pytest.mark.parametrize("levels,n", [(1, 33), (3, 17), (2, 40)])
def test_cascade_auto_equals_brute(levels, n):
    import paper_2305_07253_gb300 as rq

    V, F = _mesh("shell", 900, 5)
    scene = rq.rt_scene_build(torch.from_numpy(V).cuda(), torch.from_numpy(F).cuda())
    out = []
    for method in (rq.BAKE_AUTO, rq.BAKE_BRUTE):
        g = torch.empty((levels, n, n, n), dtype=torch.float32, device="cuda")
        rq.rt_sdf_bake(scene, rq.rt_cascade_create(g, 0.1, (2.0, 2.1, 1.9)), method)
        out.append(g.cpu().numpy())
    _equal(*out)


@pytest.mark.parametrize("move", [(1, 0, 0), (0, -1, 0), (0, 0, 2), (3, -2, 1), (-16, 5, 16), (40, 0, 0)])
def test_rolled_levels_equal_fresh_ones(move):
    import paper_2305_07253_gb300 as rq

    V, F = _mesh("plain", 400, 7)
    scene = rq.rt_scene_build(torch.from_numpy(V).cuda(), torch.from_numpy(F).cuda())
    c0 = np.array([2.05, 2.05, 2.05])
    c1 = c0 + 0.1 * np.array(move)
    g = torch.empty((2, 17, 17, 17), dtype=torch.float32, device="cuda")
    sdf = rq.rt_cascade_create(g, 0.1, c0)
    rq.rt_sdf_bake(scene, sdf, rq.BAKE_BVH)
    rq.rt_cascade_recenter(scene, sdf, c1)
    fresh = torch.empty_like(g)
    rq.rt_sdf_bake(scene, rq.rt_cascade_create(fresh, 0.1, c1), rq.BAKE_BVH)
    assert torch.equal(g, fresh)
