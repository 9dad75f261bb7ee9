"""The searches that the exact bake chooses by the number of triangles and samples
(rt_bake.cu: a thread a sample, bricks of one, eight and 32 samples) find the same
values.  Triangles far away, which are nearest to no sample, take the same mesh
from one search to the next."""
import numpy as np
import pytest

from tests.test_gpu_bake_bricks import _mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _scene(rq, kind, n, far):
    V, F = _mesh(kind, n, 3)
    rng = np.random.default_rng(4)
    W = np.array([900.0, 800.0, 700.0]) + rng.uniform(0, 50, (far, 1, 3)) + rng.normal(size=(far, 3, 3)) * 0.3
    V = np.concatenate([V, W.astype(np.float32).reshape(-1, 3)])
    F = np.arange(V.shape[0], dtype=np.int32).reshape(-1, 3)
    return rq.rt_scene_build(torch.from_numpy(V).cuda(), torch.from_numpy(F).cuda())


@pytest.mark.parametrize("kind", ["plain", "slivers", "shell"])
@pytest.mark.parametrize("n", [1, 2, 300, 512])
@pytest.mark.parametrize("method", ["BAKE_BVH", "BAKE_AUTO"])
@pytest.mark.parametrize("shape,f16", [((2, 2, 2), False), ((33, 31, 33), True), ((24, 16, 16), False), ((82, 80, 81), False)])
def test_grid(kind, n, method, shape, f16):
    import paper_2305_07253_gb300 as rq

    out = []
    for far in (0, 600, 17000):
        g = torch.empty(shape, dtype=torch.float16 if f16 else torch.float32, device="cuda")
        rq.rt_sdf_bake(_scene(rq, kind, n, far), rq.rt_sdf_create(g, (-0.3, -0.3, -0.3), (4.2, 4.2, 4.2)), getattr(rq, method))
        out.append(g)
    if method == "BAKE_AUTO" and n <= 256:
        out = [g.abs() for g in out]  # the brute force kernel's signs are rounded by its own sums
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])


@pytest.mark.parametrize("kind", ["plain", "shell"])
@pytest.mark.parametrize("n", [2, 1000])
@pytest.mark.parametrize("levels,cn", [(1, 9), (3, 17), (2, 54)])
def test_moving_cascade(kind, n, levels, cn):
    import paper_2305_07253_gb300 as rq

    out = []
    for far in (0, 600 + 424 * (n == 1000), 17000):
        sc = _scene(rq, kind, n, far)
        g = torch.empty((levels, cn, cn, cn), dtype=torch.float32, device="cuda")
        sdf = rq.rt_cascade_create(g, 0.07, (2.0, 2.1, 1.9))
        rq.rt_sdf_bake(sc, sdf, rq.BAKE_BVH)
        got = [g.clone()]
        for c in ((2.07, 2.1, 1.9), (1.8, 2.4, 1.9), (1.8, 2.4, 1.9 + 0.07 * (cn - 1)), (2.0, 2.1, 1.9)):
            rq.rt_cascade_recenter(sc, sdf, c)
            got.append(g.clone())
        out.append(got)
    for other in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(out[0], other))
