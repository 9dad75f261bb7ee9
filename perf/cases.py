"""Performance cases of the combined ray query library.

Each case is one pass of work that a program using this library has it do:
trace a batch of queries, rebuild a scene, build or move a distance field, take
a fitting step.  Scenes are rooms filled with icospheres and boxes (the shape
and the sizes of the repository's own workloads), made here on the GPU from the
seed alone; ray batches are the paper's kinds: primary, ambient occlusion, GI
and shadow rays, in 8 x 8 screen tiles.

  listed()            the cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) what the program holds before the call
  run(state)          one pass through the public entry points
  work(case)          bytes and operations that the pass cannot do without
  exact(case, seed)   the same outputs in 64 bits, where that is computable
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2305_07253_gb300 as rq

# Rooms of the repository's workloads: edge lengths in metres, icospheres and
# their subdivision, boxes, smallest and largest object scale.
MEDIUM = dict(rx=8.0, ry=4.0, rz=8.0, spheres=20, subdiv=3, boxes=10, s_lo=0.3, s_hi=1.5)
FRAME = dict(rx=20.0, ry=6.0, rz=20.0, spheres=400, subdiv=4, boxes=200, s_lo=0.2, s_hi=2.0)
FIT = dict(rx=10.0, ry=4.0, rz=10.0, spheres=20, subdiv=4, boxes=10, s_lo=0.2, s_hi=2.0)

N_1080P = 1920 * 1080


def listed():
    f256 = dict(nx=256, ny=256, nz=256, f16=False)
    return [
        # one 32 x 32 tile of GI rays in a small scene: latency and launches
        dict(name="gi_tile_small", kind="trace", **MEDIUM, nx=64, ny=64, nz=64, f16=False, own_field=True, rays="gi",
             n=1000, t_max=12.0, mode=1, any_hit=False, m_near=2.0, m_far=0.0),
        # the headline: one GI ray per pixel of a 1080p frame, one split
        dict(name="gi_1080p", kind="trace", **FRAME, **f256, own_field=False, rays="gi", n=N_1080P, t_max=30.0,
             mode=1, any_hit=False, m_near=2.0, m_far=0.0),
        # shadow rays of a frame: two splits, any hit, a ragged count
        dict(name="shadow_1080p", kind="trace", **FRAME, **f256, own_field=False, rays="shadow", n=1683745, t_max=0.0,
             mode=2, any_hit=True, m_near=2.0, m_far=2.0),
        # field-only queries on a half-precision grid of odd sizes that the program fills itself
        dict(name="field_f16_ragged", kind="trace", **MEDIUM, nx=201, ny=63, nz=203, f16=True, own_field=True,
             rays="gi", n=777777, t_max=12.0, mode=3, any_hit=False, m_near=0.0, m_far=0.0),
        # GI rays through the paper's camera-centred cascade, 5 x 64^3 at 0.1 m
        dict(name="gi_cascade", kind="trace", **FRAME, levels=5, cn=64, h0=0.1, f16=False, rays="gi", n=N_1080P,
             t_max=30.0, mode=1, any_hit=False, m_near=2.0, m_far=0.0),
        # GI rays that live in pinned host memory, records back to the host
        dict(name="gi_host", kind="host", **FRAME, **f256, own_field=False, rays="gi", n=N_1080P, t_max=30.0, mode=1,
             any_hit=False, m_near=2.0, m_far=0.0),
        # the four ray kinds of one 1080p frame in one pipeline
        dict(name="mixed_frame", kind="batches", **FRAME, **f256, own_field=False, n=N_1080P, ao_spp=2.5,
             n_shadow=1283745, m_near=2.0),
        # a frame of a scene whose geometry changed: rebuild the tree, trace the primary rays
        dict(name="rebuild_primary", kind="rebuild", **FRAME, n=N_1080P),
        # the field of a new scene: the exact bake
        dict(name="bake_exact_256", kind="bake", **FRAME, **f256),
        # the paper's field build, once per frame of a scene that changes
        dict(name="build_cascade", kind="build", **FRAME, levels=5, cn=64, h0=0.1, f16=False),
        # a camera walk of one voxel at a time: the cascade's rolling updates
        dict(name="roll_cascade", kind="roll", **FRAME, levels=5, cn=64, h0=0.1, f16=False, step=1),
        # one step of fitting the grid: forward and adjoint
        dict(name="fit_step", kind="fit", **FIT, nx=128, ny=128, nz=128, f16=False, own_field=True, rays="gi",
             n=1024 * 1024, t_max=15.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(_log(rng, lo, hi)))))


def draw(rng):
    kind = rng.choice(["trace", "trace", "trace", "host", "batches", "rebuild", "bake", "build", "roll", "fit"])
    spheres = _log_int(rng, 8, 400)
    room = (6.0 + 14.0 * spheres / 400.0) * rng.uniform(0.9, 1.0)
    c = dict(kind=kind, rx=room, ry=room * rng.uniform(0.3, 0.5), rz=room * rng.uniform(0.8, 1.0), spheres=spheres,
             subdiv=rng.choice([2, 3, 4]), boxes=_log_int(rng, 4, 200), s_lo=0.2, s_hi=rng.uniform(0.8, 2.0))
    cascade = dict(levels=rng.choice([3, 4, 5]), cn=rng.choice([32, 41, 48, 64]), h0=rng.uniform(0.06, 0.12))
    dense = dict(nx=_log_int(rng, 33, 256), ny=_log_int(rng, 33, 200), nz=_log_int(rng, 33, 256))
    f16 = rng.random() < 0.3
    m = rng.choice([0.5, 1.0, 2.0, 2.0, 4.0])
    if kind == "rebuild":
        return dict(c, n=_log_int(rng, 5000, N_1080P))
    if kind == "bake":
        return dict(c, **dense, f16=f16)
    if kind == "build":
        return dict(c, **(cascade if rng.random() < 0.6 else
                          dict(nx=_log_int(rng, 33, 128), ny=_log_int(rng, 33, 100), nz=_log_int(rng, 33, 128))), f16=f16)
    if kind == "roll":
        return dict(c, **cascade, f16=f16, step=rng.choice([1, 1, 2, 3]))
    if kind == "fit":
        g = dict(nx=_log_int(rng, 33, 128), ny=_log_int(rng, 33, 128), nz=_log_int(rng, 33, 128))
        return dict(c, spheres=min(spheres, 40), boxes=min(c["boxes"], 20), **g, f16=False, own_field=True, rays="gi",
                    n=_log_int(rng, 10000, 1024 * 1024), t_max=1.5 * room)
    if kind == "batches":
        n = _log_int(rng, 20000, N_1080P)
        return dict(c, **dense, f16=f16, own_field=False, n=n, ao_spp=rng.uniform(1.0, 2.5),
                    n_shadow=int(n * rng.uniform(0.25, 0.6)), m_near=m)
    rays = rng.choice(["gi", "gi", "ao", "shadow", "primary"])
    c = dict(c, rays=rays, n=_log_int(rng, 700, N_1080P), any_hit=rays == "shadow",
             t_max={"ao": rng.uniform(0.5, 5.0), "shadow": 0.0}.get(rays, 1.6 * room))
    c["mode"] = 2 if rays == "shadow" else rng.choice([0, 1, 1, 1, 3]) if kind == "trace" else 1
    c["m_near"] = m if c["mode"] in (1, 2) else 0.0
    c["m_far"] = m if c["mode"] == 2 else 0.0
    if kind == "trace" and rng.random() < 0.25:
        return dict(c, **cascade, f16=f16)
    own = spheres <= 40 and c["boxes"] <= 20 and rng.random() < 0.5
    return dict(c, **dense, f16=f16, own_field=own)


# ---------------------------------------------------------------------------
# scenes (the seed alone; no code of the library)
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _icosphere(subdiv):
    """Unit icosphere: vertices (nv, 3) float64 and outward triangles (nt, 3)."""
    p = (1.0 + math.sqrt(5.0)) / 2.0
    v = np.array([(-1, p, 0), (1, p, 0), (-1, -p, 0), (1, -p, 0), (0, -1, p), (0, 1, p), (0, -1, -p), (0, 1, -p),
                  (p, 0, -1), (p, 0, 1), (-p, 0, -1), (-p, 0, 1)], dtype=np.float64)
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    # the faces are the triples of mutually nearest vertices
    near = (np.linalg.norm(v[:, None] - v[None], axis=2) < 1.1) & ~np.eye(12, dtype=bool)
    f = np.array([(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
                  if near[a, b] and near[b, c] and near[a, c]])
    for _ in range(subdiv):
        e = np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]), axis=1)
        u, inv = np.unique(e, axis=0, return_inverse=True)
        mid = v[u[:, 0]] + v[u[:, 1]]
        mid /= np.linalg.norm(mid, axis=1, keepdims=True)
        ab, bc, ca = (inv.reshape(-1).reshape(3, -1) + len(v))
        v = np.concatenate([v, mid])
        a, b, c = f.T
        f = np.concatenate([np.stack(t, axis=1) for t in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
    out = np.einsum("ij,ij->i", v[f[:, 0]], np.cross(v[f[:, 1]], v[f[:, 2]])) > 0
    f[~out] = f[~out][:, [0, 2, 1]]
    return v, f


@functools.lru_cache(maxsize=None)
def _box():
    """Cube [-0.5, 0.5]^3: 8 vertices and 12 outward triangles."""
    v = np.array([[x, y, z] for z in (-0.5, 0.5) for y in (-0.5, 0.5) for x in (-0.5, 0.5)])
    f = np.array([t for a, b, c, d in ((0, 2, 3, 1), (4, 5, 7, 6), (0, 1, 5, 4), (2, 6, 7, 3), (0, 4, 6, 2), (1, 3, 7, 5))
                  for t in ((a, b, c), (a, c, d))])
    return v, f


class World:
    """Placed objects of one scene: room, spheres (centre, radius, rotation), boxes (centre, edges, rotation)."""

    def __init__(self, case, seed):
        g = np.random.default_rng([seed, 1])
        room = np.array([case["rx"], case["ry"], case["rz"]])
        ns, nb = case["spheres"], case["boxes"]
        scale = np.exp(g.uniform(math.log(case["s_lo"]), math.log(case["s_hi"]), ns + nb))
        edges = scale[:, None] * np.where(np.arange(ns + nb)[:, None] < ns, 1.0, g.uniform(0.5, 1.0, (ns + nb, 3)))
        bound = np.where(np.arange(ns + nb) < ns, 0.5 * scale, 0.5 * np.linalg.norm(edges, axis=1))
        q = g.normal(size=(ns + nb, 4))
        self.room = room
        self.eye = np.array([0.5, 0.55, 0.06]) * room
        # larger objects first, each at the first free of its candidate places
        centre = np.full((ns + nb, 3), np.nan)
        pc, pr, gap = np.zeros((0, 3)), np.zeros(0), 0.02 * room.min()
        for j in np.argsort(-bound):
            span = room - 2 * (bound[j] + gap)
            if (span <= 0).any():
                continue
            cand = bound[j] + gap + g.uniform(size=(60, 3)) * span
            free = np.linalg.norm(cand - self.eye, axis=1) > bound[j] + 0.3
            if len(pr):
                free &= (np.linalg.norm(cand[:, None] - pc[None], axis=2) > pr + bound[j] + gap).all(axis=1)
            if free.any():
                centre[j] = cand[np.argmax(free)]
                pc, pr = np.vstack([pc, centre[j]]), np.append(pr, bound[j])
        ok = ~np.isnan(centre[:, 0])
        ball = np.arange(ns + nb) < ns
        q /= np.linalg.norm(q, axis=1, keepdims=True)
        w, x, y, z = q.T
        rot = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w), 2 * (x * y + z * w),
                        1 - 2 * (x * x + z * z), 2 * (y * z - x * w), 2 * (x * z - y * w), 2 * (y * z + x * w),
                        1 - 2 * (x * x + y * y)], axis=1).reshape(-1, 3, 3)
        self.sc, self.sr, self.srot = centre[ok & ball], 0.5 * scale[ok & ball], rot[ok & ball]
        self.bc, self.be, self.brot = centre[ok & ~ball], edges[ok & ~ball], rot[ok & ~ball]
        self.bound_c, self.bound_r = centre[ok], bound[ok]

    def mesh(self, subdiv):
        """Vertices float32 (nv, 3), triangles int32 (nt, 3) on the GPU, and per sphere / box / room the first triangle."""
        t = functools.partial(torch.as_tensor, device="cuda")
        bv, bf = _box()
        sv, sf = _icosphere(subdiv)
        rv = t((bv + 0.5) * self.room)[None]
        parts = [(rv, t(bf[:, [0, 2, 1]].copy()))]
        if len(self.sr):
            parts.append((torch.einsum("vj,oij->ovi", t(sv), t(self.srot)) * t(self.sr)[:, None, None] + t(self.sc)[:, None], t(sf)))
        if len(self.be):
            parts.append((torch.einsum("ovj,oij->ovi", t(bv)[None] * t(self.be)[:, None], t(self.brot)) + t(self.bc)[:, None], t(bf)))
        V, F, nv = [], [], 0
        for v, f in parts:
            V.append(v.reshape(-1, 3))
            F.append((f[None] + (nv + v.shape[1] * torch.arange(v.shape[0], device="cuda"))[:, None, None]).reshape(-1, 3))
            nv += v.shape[0] * v.shape[1]
        return torch.cat(V).float().contiguous(), torch.cat(F).int().contiguous()

    def field(self, nx, ny, nz, f16):
        """Signed distance to the ideal shapes at the samples of a dense grid over the room, (nz, ny, nx)."""
        ax = [torch.arange(k, device="cuda", dtype=torch.float32) * (float(e) / (k - 1)) for k, e in zip((nx, ny, nz), self.room)]
        z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
        W, H, D = (float(e) for e in self.room)
        phi = torch.stack([x, W - x, y, H - y, z, D - z]).amin(0)
        for c, r in zip(self.sc, self.sr):
            phi = torch.minimum(phi, torch.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2) - float(r))
        for c, e, R in zip(self.bc, self.be, self.brot):
            dx, dy, dz = x - c[0], y - c[1], z - c[2]
            q = [(dx * R[0, k] + dy * R[1, k] + dz * R[2, k]).abs() - 0.5 * e[k] for k in range(3)]
            out = torch.sqrt(sum(torch.clamp(v, min=0) ** 2 for v in q))
            phi = torch.minimum(phi, out + torch.clamp(torch.maximum(q[0], torch.maximum(q[1], q[2])), max=0))
        return (phi.half() if f16 else phi).contiguous()


# ---------------------------------------------------------------------------
# rays (the seed alone), float32 (n, 8) = o, t_min, d, t_max
# ---------------------------------------------------------------------------
def _camera(world):
    fwd = np.array([0.5, 0.35, 0.75]) * world.room - world.eye
    fwd /= np.linalg.norm(fwd)
    right = np.cross(fwd, [0.0, 1.0, 0.0])
    right /= np.linalg.norm(right)
    return fwd, right, np.cross(right, fwd), math.tan(math.radians(30.0)), 16.0 / 9.0


def _frame_size(n):
    h = max(1, math.ceil(math.sqrt(n * 9.0 / 16.0)))
    return -(-n // h), h


def _tile_key(px, py, w):
    return ((py // 8) * ((w + 7) // 8) + px // 8) * 64 + (py % 8) * 8 + px % 8


def _pack(o, t0, d, t1):
    r = torch.empty((d.shape[0], 8), device="cuda", dtype=torch.float32)
    r[:, 0:3], r[:, 3], r[:, 4:7], r[:, 7] = o, t0, d / d.norm(dim=1, keepdim=True), t1
    return r


def primary_rays(world, n):
    w, h = _frame_size(n)
    fwd, right, up, tan, aspect = (torch.as_tensor(v, device="cuda") if isinstance(v, np.ndarray) else v for v in _camera(world))
    i = torch.arange(w * h, device="cuda")
    i = i[torch.argsort(_tile_key(i % w, i // w, w), stable=True)][:n]
    x = (2 * (i % w + 0.5) / w - 1).double() * tan * aspect
    y = (1 - 2 * (i // w + 0.5) / h).double() * tan
    d = fwd + x[:, None] * right + y[:, None] * up
    return _pack(torch.as_tensor(world.eye, device="cuda"), 0.0, d, 1.01 * float(np.linalg.norm(world.room)))


def surface_points(world, V, F, subdiv, n, seed):
    """n points and unit normals on camera-facing surfaces inside the frustum, by area, in screen-tile order."""
    gen = torch.Generator("cuda").manual_seed(seed)
    per = 20 * 4 ** subdiv
    # patches of equal-area triangles: each sphere, each face of a box or the room
    tri = lambda f: 0.5 * np.linalg.norm(np.cross(f[..., 1, :] - f[..., 0, :], f[..., 2, :] - f[..., 0, :]), axis=-1)  # noqa: E731
    bv, bf = _box()
    first = [np.arange(12)] + ([12 + per * np.arange(len(world.sr))] if len(world.sr) else [])
    count = [np.ones(12, int)] + ([np.full(len(world.sr), per)] if len(world.sr) else [])
    area = [tri((bv * world.room)[bf])] + ([4 * math.pi * world.sr ** 2] if len(world.sr) else [])
    if len(world.be):
        first.append(12 + per * len(world.sr) + np.arange(12 * len(world.be)))
        count.append(np.ones(12 * len(world.be), int))
        area.append(tri((bv[None] * world.be[:, None])[:, bf]).reshape(-1))
    cdf = np.cumsum(np.concatenate(area))
    t = functools.partial(torch.as_tensor, device="cuda")
    cdf, first, count = t(cdf / cdf[-1]), t(np.concatenate(first)), t(np.concatenate(count))
    fwd, right, up, tan, aspect = (t(v).float() if isinstance(v, np.ndarray) else v for v in _camera(world))
    eye = t(world.eye).float()
    w, h = _frame_size(n)
    got, have = [], 0
    while have < n:
        m = max(5 * (n - have), 4096)
        u = torch.rand((4, m), device="cuda", generator=gen)
        patch = torch.searchsorted(cdf, u[0].double()).clamp(max=cdf.numel() - 1)
        k = first[patch] + torch.minimum((torch.rand(m, device="cuda", generator=gen) * count[patch]).long(), count[patch] - 1)
        A, B, C = (V[F[k, j].long()] for j in range(3))
        s = torch.sqrt(u[1])[:, None]
        p = A + (B - A) * (s * (1 - u[2][:, None])) + (C - A) * (s * u[2][:, None])
        nn = torch.linalg.cross(B - A, C - A)
        nn = nn / nn.norm(dim=1, keepdim=True)
        q = p - eye
        z = (q * fwd).sum(1)
        x = (q * right).sum(1) / (z.clamp(min=1e-9) * tan * aspect)
        y = (q * up).sum(1) / (z.clamp(min=1e-9) * tan)
        keep = torch.nonzero(((nn * q).sum(1) < 0) & (z > 0.05) & (x.abs() < 1) & (y.abs() < 1))[: n - have, 0]
        px = ((x[keep] + 1) * 0.5 * w).long().clamp(max=w - 1)
        py = ((1 - y[keep]) * 0.5 * h).long().clamp(max=h - 1)
        got.append((p[keep], nn[keep], _tile_key(px, py, w)))
        have += keep.numel()
    p, nn, key = (torch.cat([g[j] for g in got]) for j in range(3))
    order = torch.argsort(key, stable=True)
    return p[order], nn[order]


def cosine_rays(world, p, nn, t_max, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    u = torch.rand((2, p.shape[0]), device="cuda", generator=gen)
    r, phi = torch.sqrt(u[0]), 2 * math.pi * u[1]
    sign = torch.where(nn[:, 2] >= 0, 1.0, -1.0)
    a = -1.0 / (sign + nn[:, 2])
    b = nn[:, 0] * nn[:, 1] * a
    b1 = torch.stack([1 + sign * nn[:, 0] ** 2 * a, sign * b, -sign * nn[:, 0]], 1)
    b2 = torch.stack([b, sign + nn[:, 1] ** 2 * a, -nn[:, 1]], 1)
    d = (r * torch.cos(phi))[:, None] * b1 + (r * torch.sin(phi))[:, None] * b2 + torch.sqrt(1 - u[0])[:, None] * nn
    return _pack(p + 1e-3 * float(np.linalg.norm(world.room)) * nn, 0.0, d, t_max)


def shadow_rays(world, p, nn, seed):
    """From each point toward one of four lights in free space under the ceiling."""
    g = np.random.default_rng([seed, 2])
    cand = np.stack([g.uniform(0.1, 0.9, 400) * world.room[0], np.full(400, 0.93 * world.room[1]), g.uniform(0.1, 0.9, 400) * world.room[2]], 1)
    room_left = (np.linalg.norm(cand[:, None] - world.bound_c[None], axis=2) - world.bound_r).min(1) if len(world.bound_r) else np.ones(400)
    lights = torch.as_tensor(cand[np.argsort(-room_left)[:4]], device="cuda").float()
    gen = torch.Generator("cuda").manual_seed(seed)
    pick = torch.randint(0, 4, (p.shape[0],), device="cuda", generator=gen)
    bias = 1e-3 * float(np.linalg.norm(world.room))
    o = p + bias * nn
    v = lights[pick] - o
    return _pack(o, 0.0, v, (v.norm(dim=1) - bias).clamp(min=0.0))


def _rays(case, world, V, F, seed):
    n = case["n"]
    if case["rays"] == "primary":
        return primary_rays(world, n)
    per = 4 if case["rays"] == "ao" else 1
    p, nn = surface_points(world, V, F, case["subdiv"], -(-n // per), seed)
    p, nn = p.repeat_interleave(per, 0)[:n], nn.repeat_interleave(per, 0)[:n]
    return shadow_rays(world, p, nn, seed) if case["rays"] == "shadow" else cosine_rays(world, p, nn, case["t_max"], seed + 1)


def _inputs(case, seed):
    """World, mesh, rays and the program's own field values (where it has some), without the library."""
    world = World(case, seed)
    V, F = world.mesh(case["subdiv"])
    rays = _rays(case, world, V, F, seed) if "rays" in case else None
    grid = world.field(case["nx"], case["ny"], case["nz"], case["f16"]) if case.get("own_field") else None
    if case["kind"] == "fit":  # the grid to be fitted is a noisy one
        gen = torch.Generator("cuda").manual_seed(seed + 3)
        h = min(float(e) / (k - 1) for k, e in zip((case["nx"], case["ny"], case["nz"]), world.room))
        grid = (grid + 0.05 * h * torch.randn(grid.shape, device="cuda", generator=gen)).contiguous()
    return world, V, F, rays, grid


def _ideal_hits(world, rays):
    """Closed-form distance of each ray to the ideal shapes (float64)."""
    o, d = rays[:, 0:3].double(), rays[:, 4:7].double()
    room = torch.as_tensor(world.room, device="cuda")
    safe = torch.where(d.abs() < 1e-12, torch.full_like(d, 1e-12), d)
    t = torch.where(d > 0, (room - o) / safe, -o / safe).amin(1)
    for c, r in zip(world.sc, world.sr):
        oc = o - torch.as_tensor(c, device="cuda")
        b = (oc * d).sum(1)
        disc = b * b - ((oc * oc).sum(1) - float(r) ** 2)
        s = -b - torch.sqrt(disc.clamp(min=0))
        t = torch.where((disc > 0) & (s > 0) & (s < t), s, t)
    for c, e, R in zip(world.bc, world.be, world.brot):
        R = torch.as_tensor(R, device="cuda")
        ol, dl = (o - torch.as_tensor(c, device="cuda")) @ R, d @ R
        dl = torch.where(dl.abs() < 1e-12, torch.full_like(dl, 1e-12), dl)
        half = 0.5 * torch.as_tensor(e, device="cuda")
        a, b = (-half - ol) / dl, (half - ol) / dl
        s, u = torch.minimum(a, b).amax(1), torch.maximum(a, b).amin(1)
        t = torch.where((s <= u) & (s > 0) & (s < t), s, t)
    return torch.where(t <= rays[:, 7], t, torch.full_like(t, math.inf))


# ---------------------------------------------------------------------------
# the program's side: handles, buffers, one pass
# ---------------------------------------------------------------------------
def _cascade(case, world, scene, method):
    grid = torch.empty((case["levels"],) + (case["cn"],) * 3, device="cuda", dtype=torch.float16 if case["f16"] else torch.float32)
    sdf = rq.rt_cascade_create(grid, case["h0"], [float(v) for v in world.eye])
    if method is not None:
        rq.rt_sdf_bake(scene, sdf, method)
    return sdf


def _dense(case, world, scene, grid):
    baked = grid is None and scene is not None
    if grid is None:
        grid = torch.empty((case["nz"], case["ny"], case["nx"]), device="cuda", dtype=torch.float16 if case["f16"] else torch.float32)
    sdf = rq.rt_sdf_create(grid, [0.0, 0.0, 0.0], [float(v) for v in world.room])
    if baked:
        rq.rt_sdf_bake(scene, sdf)
    else:
        rq.rt_sdf_prepare(sdf)
    return sdf


def prepare(case, seed):
    world, V, F, rays, grid = _inputs(case, seed)
    kind = case["kind"]
    s = {"kind": kind, "mode": case.get("mode"), "verts": V, "tris": F}
    if kind == "rebuild":
        s.update(rays=primary_rays(world, case["n"]), scene=None)
        s["hits"] = torch.zeros((case["n"], 6), dtype=torch.int32, device="cuda")
    elif kind == "fit":
        # the grid tensor is a parameter of the program's optimiser
        sdf = _dense(case, world, None, grid)
        sdf.grid.requires_grad_(True)
        s.update(sdf=sdf, rays=rays, t_ref=_ideal_hits(world, rays).float(), params=rq.split_params(mode=rq.MODE_SDF))
        return s
    else:
        s["scene"] = rq.rt_scene_build(V, F)
    if kind == "bake":
        g = torch.empty((case["nz"], case["ny"], case["nx"]), device="cuda", dtype=torch.float16 if case["f16"] else torch.float32)
        s["sdf"] = rq.rt_sdf_create(g, [0.0, 0.0, 0.0], [float(v) for v in world.room])
    elif kind == "build":
        s["sdf"] = _cascade(case, world, s["scene"], None) if "levels" in case else _dense(case, world, None, None)
    elif kind == "roll":
        s["sdf"] = _cascade(case, world, s["scene"], rq.BAKE_AUTO)
        e, d = [float(v) for v in world.eye], case["step"] * case["h0"]
        # a walk to the right, forward, up and back again, one move per frame
        s["walk"] = [(e[0] + a * d, e[1] + b * d, e[2] + c * d) for a, b, c in
                     ((1, 0, 0), (1, 0, 1), (1, 1, 1), (2, 1, 2), (1, 0, 1), (0, 0, 0))]
    elif kind in ("trace", "host"):
        s["params"] = rq.split_params(mode=case["mode"], any_hit=case["any_hit"], m_near=case["m_near"], m_far=case["m_far"])
        s["sdf"] = _cascade(case, world, s["scene"], rq.BAKE_AUTO) if "levels" in case else _dense(case, world, s["scene"], grid)
        s["rays"] = rays
        s["hits"] = torch.zeros((case["n"], 6), dtype=torch.int32, device="cuda")
        if kind == "host":
            s["rays_host"] = rays.cpu().pin_memory()
            s["hits_host"] = torch.zeros((case["n"], 6), dtype=torch.int32).pin_memory()
    elif kind == "batches":
        s["sdf"] = _dense(case, world, s["scene"], None)
        n, m = case["n"], case["m_near"]
        p, nn = surface_points(world, V, F, case["subdiv"], n, seed)
        # ambient occlusion rays: ao_spp a pixel on average, a different number at each
        pick = torch.randint(0, n, (int(n * case["ao_spp"]),), device="cuda", generator=torch.Generator("cuda").manual_seed(seed + 4)).sort()[0]
        pa, na = p[pick], nn[pick]
        every = [(primary_rays(world, n), rq.split_params(mode=rq.MODE_BVH)),
                 (cosine_rays(world, pa, na, 0.5, seed + 5), rq.split_params(mode=1, m_near=m)),
                 (cosine_rays(world, p, nn, 30.0, seed + 6), rq.split_params(mode=1, m_near=m)),
                 (shadow_rays(world, p[: case["n_shadow"]], nn[: case["n_shadow"]], seed + 7),
                  rq.split_params(mode=2, any_hit=True, m_near=m, m_far=m))]
        s["batches"] = [(r, q, torch.zeros((r.shape[0], 6), dtype=torch.int32, device="cuda")) for r, q in every]
        s["out"] = [rq.hit_fields(b[2]) for b in s["batches"]]
    if "hits" in s:
        # the record buffer is kept from frame to frame, and so are its columns
        s["out"] = rq.hit_fields(s["hits_host"] if kind == "host" else s["hits"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "trace":
        if s["mode"] == rq.MODE_BVH:
            rq.rt_trace_bvh(s["scene"], s["rays"], hits=s["hits"])
        elif s["mode"] == rq.MODE_SDF:
            rq.rt_trace_sdf(s["sdf"], s["rays"], s["params"], hits=s["hits"])
        else:
            rq.rt_trace_combined(s["scene"], s["sdf"], s["rays"], s["params"], hits=s["hits"])
        return s["out"]
    if kind == "host":
        rq.trace_combined_from_host(s["scene"], s["sdf"], s["rays_host"], s["params"], s["hits_host"], s["rays"], s["hits"])
        return s["out"]
    if kind == "batches":
        rq.rt_trace_batches(s["scene"], s["sdf"], s["batches"])
        return s["out"]
    if kind == "rebuild":
        s["scene"] = rq.rt_scene_build(s["verts"], s["tris"])
        rq.rt_trace_bvh(s["scene"], s["rays"], hits=s["hits"])
        return s["out"]
    if kind == "bake":
        rq.rt_sdf_bake(s["scene"], s["sdf"])
        return s["sdf"].grid
    if kind == "build":
        rq.rt_sdf_bake(s["scene"], s["sdf"], rq.BAKE_JFA)
        return s["sdf"].grid
    if kind == "roll":
        for c in s["walk"]:
            rq.rt_cascade_recenter(s["scene"], s["sdf"], c)
        return s["sdf"].grid
    grid = s["sdf"].grid
    t, hits = rq.SdfHitDistance.apply(grid, s["rays"], None, s["sdf"], s["params"])
    both = torch.isfinite(t) & torch.isfinite(s["t_ref"])
    diff = torch.where(both, t - s["t_ref"], torch.zeros_like(t))
    loss = diff.pow(2).sum() / t.shape[0]
    (g,) = torch.autograd.grad(loss, grid)
    return {"t": t.detach(), "grad": g, "loss": loss.detach(), "tracer": hits[:, 4]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    esz = 2 if case.get("f16") else 4
    tris = 12 + case["spheres"] * 20 * 4 ** case["subdiv"] + 12 * case["boxes"]
    verts = 8 + case["spheres"] * (2 + 10 * 4 ** case["subdiv"]) + 8 * case["boxes"]
    if "levels" in case:
        samples = case["levels"] * case["cn"] ** 3
    else:
        samples = case.get("nx", 0) * case.get("ny", 0) * case.get("nz", 0)
    if kind == "rebuild":
        # vertices and indices in; nodes (64 B), triangles (48 B) and pseudonormals (112 B) out; rays and records
        return {"bytes": 12 * verts + 12 * tris + 224 * tris + 56 * case["n"], "flops": 400 * tris + 600 * case["n"]}
    if kind in ("bake", "build"):
        # triangles in, samples and the copy of every cell's eight corners out
        return {"bytes": 48 * tris + samples * esz * 9, "flops": 60 * 8 * samples}
    if kind == "roll":
        # the slabs that enter each level: six moves, about two levels each; a level moved within its memory
        slab = case["cn"] ** 2 * case["step"]
        return {"bytes": 6 * 2 * (2 * samples / case["levels"] * esz), "flops": 6 * 2 * slab * 60 * 8}
    if kind == "fit":
        # rays, reference and records; the grid read and its cell copy, the gradient
        return {"bytes": case["n"] * (32 + 24 + 8) + samples * esz * 10, "flops": case["n"] * 45 * (25 + 24)}
    n = case["n"]
    if kind == "batches":
        n = int(n * (2 + case["ao_spp"])) + case["n_shadow"]
    # each ray in, each record out; the grid and the triangles that the rays can touch, once
    touched = min(samples * esz, 20 * 32 * n) * (case.get("mode") != 0) + min(112 * tris, 15 * 64 * n) * (case.get("mode") != 3)
    return {"bytes": 56 * n + touched, "flops": n * (20 * 45 + 15 * 30)}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------
def _exact_field(grid, room):
    """phi(p) of a (nz, ny, nx) grid over [0, room], its cell and fractions, in float64."""
    nz, ny, nx = grid.shape
    n = torch.tensor([nx, ny, nz], device="cuda")
    h = torch.as_tensor(room, device="cuda").float() / (n - 1).float()  # the handle's spacing is in single precision
    h = h.double()
    g = grid.double().reshape(-1)

    def locate(p):
        u = torch.minimum(torch.clamp(p / h, min=0.0), (n - 1).double())
        i0 = torch.minimum(u.floor().long(), n - 2)
        return i0, u - i0

    def corners(i0):
        b = i0[:, 0] + nx * (i0[:, 1] + ny * i0[:, 2])
        return torch.stack([b + dx + nx * (dy + ny * dz) for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)], 1)

    def weights(f):
        return torch.stack([(f[:, 0] if dx else 1 - f[:, 0]) * (f[:, 1] if dy else 1 - f[:, 1]) * (f[:, 2] if dz else 1 - f[:, 2])
                            for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)], 1)

    def phi(p):
        i0, f = locate(p)
        return (g[corners(i0)] * weights(f)).sum(1)

    return phi, locate, corners, weights, g, h


def _exact_march(grid, room, rays, ta, tb, max_steps=256):
    """Sphere tracing by the documented step rule on [ta, tb]: (hit, t, t_prev)."""
    phi, _, _, _, _, h = _exact_field(grid, room)
    eps = 0.01 * float(h.min())
    o, d = rays[:, 0:3].double(), rays[:, 4:7].double()
    hi = torch.as_tensor(room, device="cuda")
    safe = torch.where(d.abs() < 1e-30, torch.full_like(d, 1e-30), d)
    a, b = -o / safe, (hi - o) / safe
    ta = torch.maximum(ta, torch.minimum(a, b).amax(1))
    tb = torch.minimum(tb, torch.maximum(a, b).amin(1))
    hit = torch.zeros_like(ta, dtype=torch.bool)
    t, prev = ta.clone(), torch.full_like(ta, math.nan)
    live = torch.nonzero(ta <= tb)[:, 0]
    for _ in range(max_steps):
        if live.numel() == 0:
            break
        v = phi(o[live] + t[live, None] * d[live])
        got = v < eps
        hit[live[got]] = True
        on = live[~got]
        prev[on] = t[on]
        t[on] = t[on] + torch.clamp(v[~got], min=eps)
        live = on[t[on] <= tb[on]]
    return hit, t, prev, eps


def _exact_triangles(V, F, rays, ta, tb):
    """Closest hit of each ray among all triangles in [ta, tb]: (t, u, v)."""
    A, B, C = (V[F[:, k].long()].double() for k in range(3))
    e1, e2 = B - A, C - A
    T, U, W = [], [], []
    for r, a, b in zip(*(x.split(max(1, 20_000_000 // F.shape[0])) for x in (rays, ta, tb))):
        o, d = r[:, None, 0:3].double(), r[:, None, 4:7].double().expand(-1, F.shape[0], -1)
        p = torch.linalg.cross(d, e2.expand_as(d))
        det = (p * e1).sum(2)
        s = o - A
        u = (s * p).sum(2) / det
        q = torch.linalg.cross(s, e1.expand_as(s))
        v = (d * q).sum(2) / det
        t = (q * e2).sum(2) / det
        t = torch.where((det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t >= a[:, None]) & (t <= b[:, None]), t, torch.full_like(t, math.inf))
        best, k = t.min(1)
        miss = torch.isinf(best)
        T.append(best)
        U.append(torch.where(miss, 0.0, u.gather(1, k[:, None])[:, 0]))
        W.append(torch.where(miss, 0.0, v.gather(1, k[:, None])[:, 0]))
    return torch.cat(T), torch.cat(U), torch.cat(W)


def _exact_bake(V, F, pos):
    """Unsigned distance of each position to the nearest triangle."""
    A, B, C = (V[F[:, k].long()].double() for k in range(3))

    def segment(p, a, b):
        ab, ap = b - a, p - a
        s = ((ap * ab).sum(-1) / (ab * ab).sum(-1).clamp(min=1e-300)).clamp(0, 1)
        r = ap - s[..., None] * ab
        return (r * r).sum(-1)

    out = []
    n = torch.linalg.cross(B - A, C - A)
    nn = (n * n).sum(-1)
    for p in pos.split(max(1, 12_000_000 // F.shape[0])):
        p = p[:, None]
        d2 = torch.minimum(segment(p, A, B), torch.minimum(segment(p, B, C), segment(p, C, A)))
        inside = torch.ones_like(d2, dtype=torch.bool)
        for a, b in ((A, B), (B, C), (C, A)):
            inside &= (torch.linalg.cross(n, b - a) * (p - a)).sum(-1) >= 0
        h = ((p - A) * n).sum(-1)
        out.append(torch.where(inside, torch.minimum(d2, h * h / nn), d2).amin(1).sqrt())
    return torch.cat(out)


def exact(case, seed):
    kind, tris = case["kind"], 12 + case["spheres"] * 20 * 4 ** case["subdiv"] + 12 * case["boxes"]
    if kind == "bake":
        if case["nx"] * case["ny"] * case["nz"] * tris > 6e9:
            return None
        world, V, F, _, _ = _inputs(case, seed)
        # lattice coordinates as the handle has them, in single precision
        ax = [torch.arange(k, device="cuda", dtype=torch.float32) * (torch.tensor(float(e), device="cuda") / (k - 1))
              for k, e in zip((case["nx"], case["ny"], case["nz"]), world.room)]
        z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
        pos = torch.stack([x, y, z], -1).reshape(-1, 3).double()
        d = _exact_bake(V, F, pos)
        # inside an object: the ideal box, or behind every face of the (convex) icosphere
        phi = world.field(case["nx"], case["ny"], case["nz"], False).reshape(-1)
        neg = phi < 0
        per = 20 * 4 ** case["subdiv"]
        for k, (c, r) in enumerate(zip(world.sc, world.sr)):
            near = torch.nonzero((pos - torch.as_tensor(c, device="cuda")).norm(dim=1) < float(r) * 1.0001)[:, 0]
            f = F[12 + per * k:12 + per * (k + 1)].long()
            A, B, C = (V[f[:, j]].double() for j in range(3))
            nn = torch.linalg.cross(B - A, C - A)
            for i in near.split(20000):
                neg[i] = (pos[i] @ nn.T - (A * nn).sum(1)).amax(1) < 0
        return torch.where(neg, -d, d).reshape(case["nz"], case["ny"], case["nx"])
    if kind == "fit":
        world, _, _, rays, grid = _inputs(case, seed)
        t0, t1 = rays[:, 3].double(), rays[:, 7].double()
        hit, t, prev, eps = _exact_march(grid, world.room, rays, t0, t1)
        phi, locate, corners, weights, g, h = _exact_field(grid, world.room)
        o, d = rays[:, 0:3].double(), rays[:, 4:7].double()
        root = hit & ~torch.isnan(prev)
        lo, hi = torch.where(root, prev, t), t.clone()
        for _ in range(50):
            mid = 0.5 * (lo + hi)
            below = phi(o + mid[:, None] * d) < eps
            hi, lo = torch.where(below, mid, hi), torch.where(below, lo, mid)
        t = torch.where(hit, torch.where(root, hi, t), torch.full_like(t, math.inf))
        ref = _ideal_hits(world, rays).float().double()
        both = torch.isfinite(t) & torch.isfinite(ref)
        diff = torch.where(both, t - ref, torch.zeros_like(t))
        # dt/dtheta = -w / (grad phi . d) at the root, scattered to the eight corners
        i0, f = locate(o + torch.where(root, t, torch.zeros_like(t))[:, None] * d)
        at = corners(i0)
        w, v = weights(f), g[at]
        gd = torch.zeros_like(t)
        for ax in range(3):
            one = f.clone()
            one[:, ax] = 1.0
            w1 = weights(one)
            one[:, ax] = 0.0
            gd = gd + (v * (w1 - weights(one))).sum(1) / h[ax] * d[:, ax]
        up = 2.0 * diff / t.shape[0]
        s = torch.where(root & both & (gd <= -1e-6), -up / torch.where(gd <= -1e-6, gd, torch.full_like(gd, -1.0)), torch.zeros_like(gd))
        grad = torch.zeros_like(g).index_add_(0, at.reshape(-1), (s[:, None] * w).reshape(-1)).reshape(grid.shape)
        return {"t": t, "grad": grad, "loss": diff.pow(2).sum() / t.shape[0], "tracer": None}
    if kind not in ("trace", "host") or case["any_hit"] or not case.get("own_field"):
        return None
    if case["mode"] != 3 and case["n"] * tris > 4e8:
        return None
    world, V, F, rays, grid = _inputs(case, seed)
    t0, t1 = rays[:, 3].double(), rays[:, 7].double()
    none = torch.full_like(t0, math.inf)
    t, u, v = none, torch.zeros_like(t0), torch.zeros_like(t0)
    split = t0
    if case["mode"] != 3:
        h = max(float(e) / (k - 1) for k, e in zip((case["nx"], case["ny"], case["nz"]), world.room))
        split = t1 if case["mode"] == 0 else torch.minimum(t0 + case["m_near"] * h, t1)
        t, u, v = _exact_triangles(V, F, rays, t0, split)
    if case["mode"] != 0:
        hit, tf, _, _ = _exact_march(grid, world.room, rays, split, t1)
        t = torch.where(torch.isinf(t) & hit & ((split < t1) | (case["mode"] == 3)), tf, t)
    return {"t": t, "prim": None, "u": u, "v": v, "tracer": None, "flags": None}
