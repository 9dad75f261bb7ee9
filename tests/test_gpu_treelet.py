"""Treelet restructuring (rt_treelet.cu): a scene of at most seven triangles is
one treelet, so its tree must reach the least surface-area cost of all binary
trees over its triangles; larger ones must hold every triangle once."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

C_NODE, C_TRI = 1.2, 1.0


def _half_area(lo, hi):
    d = hi - lo
    return d[0] * d[1] + d[1] * d[2] + d[2] * d[0]


def _optimum(lo, hi):
    """Least cost over all binary trees on the boxes, by dynamic programming over subsets (float64)."""
    n = lo.shape[0]
    cost = {}
    for S in sorted(range(1, 1 << n), key=lambda s: bin(s).count("1")):
        idx = [i for i in range(n) if S >> i & 1]
        a = _half_area(lo[idx].min(0), hi[idx].max(0))
        if len(idx) == 1:
            cost[S] = C_TRI * a
            continue
        best, sub = np.inf, (S - 1) & S
        while sub:
            best = min(best, cost[sub] + cost[S ^ sub])
            sub = (sub - 1) & S
        cost[S] = C_NODE * a + best
    return cost[(1 << n) - 1]


def _tree(nodes, tris, ref):
    """(cost, lo, hi, input indices) of the exported subtree, from the triangles themselves."""
    if ref < 0:
        v = tris[~ref].reshape(3, 4)[:, :3].astype(np.float64)
        lo, hi = v.min(0), v.max(0)
        return C_TRI * _half_area(lo, hi), lo, hi, [int(tris[~ref].view(np.int32)[3])]
    c = nodes[ref].view(np.int32)[12:14]
    a, b = _tree(nodes, tris, int(c[0])), _tree(nodes, tris, int(c[1]))
    lo, hi = np.minimum(a[1], b[1]), np.maximum(a[2], b[2])
    return C_NODE * _half_area(lo, hi) + a[0] + b[0], lo, hi, a[3] + b[3]


@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("n", [3, 4, 5, 6, 7, 8, 31, 33, 257])
def test_treelets_reach_the_least_cost(n, seed):
    import paper_2305_07253_gb300 as rq

    rng = np.random.default_rng(100 * n + seed)
    centre = rng.uniform(0, 4, (n, 1, 3))
    V = (centre + rng.uniform(-1, 1, (n, 3, 3)) * rng.uniform(0.05, 1.0, (n, 1, 1))).astype(np.float32).reshape(-1, 3)
    F = np.arange(3 * n, dtype=np.int32).reshape(n, 3)
    scene = rq.rt_scene_build(torch.from_numpy(V).cuda(), torch.from_numpy(F).cuda())
    nodes, tris = (x.cpu().numpy() for x in rq.rt_scene_export(scene))
    cost, _, _, prims = _tree(nodes, tris, 0)
    assert sorted(prims) == list(range(n))
    if n <= 7:
        v = V.reshape(n, 3, 3).astype(np.float64)
        # single precision sums of at most 13 terms, and the 1e-6 a rewiring has to gain
        assert cost <= _optimum(v.min(1), v.max(1)) * (1 + 1e-5)
