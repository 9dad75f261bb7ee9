// The paper's distance-field build (Section 3, "Distance Field Generation"):
// the triangles are voxelised, the voxelisation is turned into a distance
// field by jump flooding, and fast sweeping refines it.  The paper names the
// three steps only; the steps taken here:
//
//   1. Conservative voxelisation.  Sample s owns the voxel box of side
//      h (1 + 2^-8) centred on it.  Every triangle is tested (separating axes,
//      Akenine-Moller, JGT 2001) against the voxels its bounds can reach: one
//      thread per triangle when they are few, one block per triangle when they
//      are many; an overlapping triangle is a candidate site of the sample.
//      The best candidate wins through a 64-bit atomicMin on (squared
//      distance bits, triangle index).  On a cascade level below the
//      coarsest, the site of the nearest sample of the next coarser level is a
//      candidate too.
//   2. Jump flooding (Rong & Tan, I3D 2006): steps k = 2^(ceil(log2 n)-1) ...
//      1; each sample takes the best of the sites of itself and its 26
//      neighbours at offsets in {-k, 0, k}^3, from the previous step.
//   3. Fast sweeping as axis sweeps, +x, -x, +y, -y, +z, -z: the best site is
//      carried along each grid line, by a warp (by a thread on lines too long for
//      its shared memory).
//   4. The field value is the signed distance to the site triangle (the
//      exact bake's closest point and pseudonormal sign).
//
// "Best" is the smallest (squared distance from the sample to the site's
// triangle, triangle index).  Every operation of steps 1-3 is rounded once
// (explicit intrinsics), so the sites are those of the CPU checker's single
// precision build, bit for bit.
#include "rt_bake_dev.cuh"
#include "rt_trace_dev.cuh"

namespace {

constexpr int kBlock = 256;

// ---------------------------------------------------------------------------
// single precision geometry, each operation rounded once
// ---------------------------------------------------------------------------
__device__ __forceinline__ float dot3r(const float* a, const float* b)
{
    return __fadd_rn(__fadd_rn(__fmul_rn(a[0], b[0]), __fmul_rn(a[1], b[1])), __fmul_rn(a[2], b[2]));
}

// Squared distance from p to triangle abc (Ericson's Voronoi regions).  Lanes
// mostly fall in different regions, so there are no branches: the region picks
// the operands of one division and of q = (base + s1 dir1) + s2 dir2.  A vertex
// has s1 = s2 = 0 and an edge s2 = 0, which leave base + s1 dir1 as it is.
// Infinite where it is not a number: a triangle with two equal vertices divides by
// the length of their edge at half of all positions.  A distance that compares with
// every other is what makes the best site independent of the order in which the
// steps meet the candidates.
__device__ __forceinline__ float tri_d2_rn(const float* p, const float* a, const float* b, const float* c)
{
    float ab[3], ac[3], ap[3], bp[3], cp[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        ab[k] = __fsub_rn(b[k], a[k]);
        ac[k] = __fsub_rn(c[k], a[k]);
        ap[k] = __fsub_rn(p[k], a[k]);
        bp[k] = __fsub_rn(p[k], b[k]);
        cp[k] = __fsub_rn(p[k], c[k]);
    }
    const float d1 = dot3r(ab, ap), d2 = dot3r(ac, ap), d3 = dot3r(ab, bp), d4 = dot3r(ac, bp);
    const float d5 = dot3r(ab, cp), d6 = dot3r(ac, cp);
    const float vc = __fsub_rn(__fmul_rn(d1, d4), __fmul_rn(d3, d2));
    const float vb = __fsub_rn(__fmul_rn(d5, d2), __fmul_rn(d1, d6));
    const float va = __fsub_rn(__fmul_rn(d3, d6), __fmul_rn(d5, d4));
    const float e43 = __fsub_rn(d4, d3), e56 = __fsub_rn(d5, d6);
    // the regions in the order they are tested; the first that holds
    const bool at_a = d1 <= 0.f && d2 <= 0.f;
    const bool at_b = !at_a && d3 >= 0.f && d4 <= d3;
    const bool on_ab = !at_a && !at_b && vc <= 0.f && d1 >= 0.f && d3 <= 0.f;
    const bool past_ab = !at_a && !at_b && !on_ab;
    const bool at_c = past_ab && d6 >= 0.f && d5 <= d6;
    const bool on_ac = past_ab && !at_c && vb <= 0.f && d2 >= 0.f && d6 <= 0.f;
    const bool on_bc = past_ab && !at_c && !on_ac && va <= 0.f && e43 >= 0.f && e56 >= 0.f;
    const bool vertex = at_a || at_b || at_c, face = past_ab && !at_c && !on_ac && !on_bc;
    const float num = vertex ? 0.f : (on_ab ? d1 : (on_ac ? d2 : (on_bc ? e43 : 1.f)));
    const float den = vertex ? 1.f
                             : (on_ab ? __fsub_rn(d1, d3)
                                      : (on_ac ? __fsub_rn(d2, d6)
                                               : (on_bc ? __fadd_rn(e43, e56) : __fadd_rn(__fadd_rn(va, vb), vc))));
    const float r = __fdiv_rn(num, den);
    const float s1 = face ? __fmul_rn(vb, r) : r, s2 = face ? __fmul_rn(vc, r) : 0.f;
    const bool from_b = at_b || on_bc;
    float pq[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float base = from_b ? b[k] : (at_c ? c[k] : a[k]);
        const float dir = on_ac ? ac[k] : (on_bc ? __fsub_rn(c[k], b[k]) : ab[k]);
        const float q = __fadd_rn(__fadd_rn(base, __fmul_rn(s1, dir)), __fmul_rn(s2, ac[k]));
        pq[k] = __fsub_rn(p[k], q);
    }
    return fminf(dot3r(pq, pq), __int_as_float(0x7f800000));  // (the minimum of a NaN and a number is the number)
}

// Separation along an axis on which the triangle's vertices lie at p0, p1, p2 and
// the box reaches r to either side of the origin
__device__ __forceinline__ bool separated(float p0, float p1, float p2, float r)
{
    return rtdev::min3f(p0, p1, p2) > r || rtdev::max3f(p0, p1, p2) < -r;
}

// Triangle / box overlap by separating axes (touching counts).  Components of an
// axis that are zero are left out: adding their products changes nothing.
__device__ bool tri_box(const float* c, const float* hs, const float* A, const float* B, const float* C)
{
    float v[3][3], e[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[0][k] = __fsub_rn(A[k], c[k]);
        v[1][k] = __fsub_rn(B[k], c[k]);
        v[2][k] = __fsub_rn(C[k], c[k]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (separated(v[0][k], v[1][k], v[2][k], hs[k])) return false;
        e[0][k] = __fsub_rn(v[1][k], v[0][k]);
        e[1][k] = __fsub_rn(v[2][k], v[1][k]);
        e[2][k] = __fsub_rn(v[0][k], v[2][k]);
    }
    const float n[3] = {__fsub_rn(__fmul_rn(e[0][1], e[1][2]), __fmul_rn(e[0][2], e[1][1])),
                        __fsub_rn(__fmul_rn(e[0][2], e[1][0]), __fmul_rn(e[0][0], e[1][2])),
                        __fsub_rn(__fmul_rn(e[0][0], e[1][1]), __fmul_rn(e[0][1], e[1][0]))};
    const float an[3] = {fabsf(n[0]), fabsf(n[1]), fabsf(n[2])};
    if (separated(dot3r(n, v[0]), dot3r(n, v[1]), dot3r(n, v[2]), dot3r(hs, an))) return false;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            // unit axis k x edge j: (0, -e2, e1), (e2, 0, -e0), (-e1, e0, 0), its two
            // components in the order of the coordinates
            const int s = k == 0 ? 1 : 0, t = k == 2 ? 1 : 2;
            const float es = k == 1 ? e[j][t] : -e[j][t], et = k == 1 ? -e[j][s] : e[j][s];
            auto on = [&](const float* q) { return __fadd_rn(__fmul_rn(es, q[s]), __fmul_rn(et, q[t])); };
            const float r = __fadd_rn(__fmul_rn(hs[s], fabsf(es)), __fmul_rn(hs[t], fabsf(et)));
            if (separated(on(v[0]), on(v[1]), on(v[2]), r)) return false;
        }
    }
    return true;
}

// ---------------------------------------------------------------------------
// grid geometry (one grid, or one cascade level)
// ---------------------------------------------------------------------------
struct DfGrid {
    int32_t n[3];
    int32_t lattice;
    int32_t ilo[3];
    float lo[3], h[3], hs[3];
    // conservative sample range of a triangle: origin, 1/h and a margin of a
    // small fraction of a voxel (much more than the rounding of the positions)
    float origin_f[3], ih_f[3], margin[3];
    int64_t count;
};

__device__ __forceinline__ void df_pos(const DfGrid& g, int64_t i, int64_t j, int64_t k, float* p)
{
    const int64_t ii[3] = {i, j, k};
#pragma unroll
    for (int a = 0; a < 3; ++a)
        p[a] = g.lattice ? __fmul_rn((float)(g.ilo[a] + ii[a]), g.h[a]) : __fmaf_rn((float)ii[a], g.h[a], g.lo[a]);
}

// Inside a build a site is a position in leaf order, so that a candidate's
// triangle is one load away; "best" compares input indices, which come with the
// triangle.  Sites that leave a build (rt_sdf_sites, the seeds of finer levels)
// are input indices.
struct Tris {
    const float4* tris;   // leaf order, 3 per triangle: v0.xyz | input index, v1.xyz, v2.xyz
    const int32_t* slot;  // input index -> leaf position
    int64_t n;
};

struct TriV {
    float a[3], b[3], c[3];
    int32_t id;  // input index
};

__device__ __forceinline__ TriV tri_verts(const Tris& T, int32_t k)
{
    const float4* p = T.tris + 3 * (int64_t)k;
    const float4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
    return {{a.x, a.y, a.z}, {b.x, b.y, b.z}, {c.x, c.y, c.z}, __float_as_int(a.w)};
}

// the better of two (squared distance, input index); id < 0: none
__device__ __forceinline__ bool site_better(float d2, int32_t id, float cur_d2, int32_t cur_id)
{
    return cur_id < 0 || d2 < cur_d2 || (d2 == cur_d2 && id < cur_id);
}

// Whether the triangle's box alone shows that tri_d2_rn(p, t) > d2.  The margins
// (4e-5 of d2, and the square of 1.4e-4 of the position, whose ulp rounds the
// closest point) are well above the roundings of both sides.
__device__ __forceinline__ bool tri_farther(const float* p, const TriV& t, float d2)
{
    float lb = 0.f, pp = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float lo = rtdev::min3f(t.a[k], t.b[k], t.c[k]), hi = rtdev::max3f(t.a[k], t.b[k], t.c[k]);
        const float e = rtdev::max3f(lo - p[k], p[k] - hi, 0.f);
        lb = fmaf(e, e, lb);
        pp = fmaf(p[k], p[k], pp);
    }
    return lb > fmaf(4e-5f, d2, d2) + 2e-8f * pp;
}

// samples whose voxels the triangle's bounds may reach: the range is widened by
// a small fraction of a voxel, far more than the rounding of the sample
// positions, and the separating-axis test decides
__device__ __forceinline__ bool tri_range(const DfGrid& g, const float* A, const float* B, const float* C,
                                          int32_t r0[3], int32_t r1[3])
{
    bool empty = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float lo_t = fminf(fminf(A[a], B[a]), C[a]) - g.hs[a];
        const float hi_t = fmaxf(fmaxf(A[a], B[a]), C[a]) + g.hs[a];
        const float x0f = ceilf((lo_t - g.origin_f[a] - g.margin[a]) * g.ih_f[a]);
        const float x1f = floorf((hi_t - g.origin_f[a] + g.margin[a]) * g.ih_f[a]);
        // clamp in float first: far-away triangles give values beyond the int range
        const int32_t x0 = (int32_t)fminf(fmaxf(x0f, 0.f), (float)g.n[a]);
        const int32_t x1 = (int32_t)fmaxf(fminf(x1f, (float)(g.n[a] - 1)), -1.f);
        r0[a] = x0;
        r1[a] = x1;
        empty = empty || x0 > x1 || x1f < 0.f || x0f > (float)(g.n[a] - 1);
    }
    return !empty;
}

// Test one (triangle, sample) pair and keep the better site of the sample.  On a
// coarse level thousands of triangles share a voxel: a pair that is no better
// than what the sample has needs neither the separating axes nor the atomic.
__device__ __forceinline__ void vox_pair(const DfGrid& g, const TriV& t, int32_t i, int32_t j, int32_t k,
                                         unsigned long long* keys)
{
    float p[3];
    df_pos(g, i, j, k, p);
    unsigned long long* at = keys + i + (int64_t)g.n[0] * (j + (int64_t)g.n[1] * k);
    const unsigned long long have = __ldcg(at);  // none yet: its distance is a NaN, which nothing exceeds
    if (tri_farther(p, t, __uint_as_float((uint32_t)(have >> 32)))) return;
    const float d2 = tri_d2_rn(p, t.a, t.b, t.c);
    const unsigned long long key = ((unsigned long long)__float_as_uint(d2) << 32) | (uint32_t)t.id;
    if (key >= have || !tri_box(p, g.hs, t.a, t.b, t.c)) return;
    atomicMin(at, key);
}

constexpr int64_t kSmallPairs = 64;  // a thread tests a triangle's voxels itself up to this many

// the grids voxelised by one pass over the triangles (all levels of a cascade at once)
struct VoxPass {
    DfGrid g[RT_MAX_LEVELS];
    unsigned long long* keys[RT_MAX_LEVELS];
    int32_t count;
};

// One thread per triangle, level by level: small ranges are tested here, large
// ones listed (leaf position, level) for k_df_vox_big; a full list leaves them
// to the thread.
__global__ void k_df_vox_small(const VoxPass vp, const Tris T, int2* big, unsigned* n_big, unsigned most_big)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T.n) return;
    const TriV v = tri_verts(T, (int32_t)t);
    for (int l = 0; l < vp.count; ++l) {
        const DfGrid& g = vp.g[l];
        int32_t r0[3], r1[3];
        if (!tri_range(g, v.a, v.b, v.c, r0, r1)) continue;
        const int64_t count = (int64_t)(r1[0] - r0[0] + 1) * (r1[1] - r0[1] + 1) * (r1[2] - r0[2] + 1);
        if (count > kSmallPairs) {
            const unsigned at = atomicAdd(n_big, 1u);
            if (at < most_big) {
                big[at] = make_int2((int)t, l);
                continue;
            }
        }
        for (int32_t k = r0[2]; k <= r1[2]; ++k)
            for (int32_t j = r0[1]; j <= r1[1]; ++j)
                for (int32_t i = r0[0]; i <= r1[0]; ++i) vox_pair(g, v, i, j, k, vp.keys[l]);
    }
}

// one block per listed (triangle, level), threads over its voxels
__global__ void k_df_vox_big(const VoxPass vp, const Tris T, const int2* big, const unsigned* n_big, unsigned most_big)
{
    const unsigned nb = min(*n_big, most_big);
    for (unsigned b = blockIdx.x; b < nb; b += gridDim.x) {
        const int2 e = big[b];
        const DfGrid& g = vp.g[e.y];
        const TriV v = tri_verts(T, e.x);
        int32_t r0[3], r1[3];
        tri_range(g, v.a, v.b, v.c, r0, r1);
        const int64_t sx = r1[0] - r0[0] + 1, sy = r1[1] - r0[1] + 1;
        const int64_t count = sx * sy * (r1[2] - r0[2] + 1);
        for (int64_t w = threadIdx.x; w < count; w += blockDim.x)
            vox_pair(g, v, r0[0] + (int32_t)(w % sx), r0[1] + (int32_t)((w / sx) % sy), r0[2] + (int32_t)(w / (sx * sy)),
                     vp.keys[e.y]);
    }
}

__device__ __forceinline__ int64_t floordiv(int64_t x, int64_t y)  // y > 0
{
    return x >= 0 ? x / y : -((-x + y - 1) / y);
}

// sites from the voxelisation; on a cascade level also the coarser level's site
// (an input index, like every site that a build leaves)
__global__ void k_df_seed(const DfGrid g, const Tris T, const unsigned long long* keys, const int32_t* coarse,
                          const DfGrid gc, int32_t* sites)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.count) return;
    const unsigned long long key = keys[s];
    int32_t cur = key == ~0ull ? -1 : (int32_t)(key & 0xffffffffull);
    if (coarse) {
        const int64_t ii[3] = {s % g.n[0], (s / g.n[0]) % g.n[1], s / ((int64_t)g.n[0] * g.n[1])};
        int64_t jc[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int64_t j = floordiv(g.ilo[a] + ii[a] + 1, 2) - gc.ilo[a];
            jc[a] = j < 0 ? 0 : (j > gc.n[a] - 1 ? gc.n[a] - 1 : j);
        }
        const int32_t t = coarse[jc[0] + (int64_t)gc.n[0] * (jc[1] + (int64_t)gc.n[1] * jc[2])];
        if (t >= 0 && t != cur) {
            float p[3];
            df_pos(g, ii[0], ii[1], ii[2], p);
            const TriV v = tri_verts(T, __ldg(T.slot + t));
            if (site_better(tri_d2_rn(p, v.a, v.b, v.c), t, __uint_as_float((uint32_t)(key >> 32)), cur)) cur = t;
        }
    }
    sites[s] = cur < 0 ? -1 : __ldg(T.slot + cur);
}

// One jump flooding step.  Triangles are small against the sample spacing, so the
// 27 neighbours mostly carry different sites, few of which can be the best.  A
// thread reads its neighbours' sites, all in flight together, takes its own
// sample's site first, and lists the other distinct ones (a candidate equal to
// one of the last kSiteCache listed is not listed again).  The warp then goes
// through the lists: a candidate whose box is farther than the best so far is
// done with; the (lane, candidate) pairs left are collected and evaluated 32 at a
// time, the smaller (squared distance, input index) winning by a 64-bit minimum
// in shared memory.  The result is the same minimum.
// What bounds it is issue.  64^3 samples of the frame scene, us a step: 37 with
// each candidate evaluated as it is met (once per neighbour for a few lanes at a
// time), 30 with every listed one evaluated.
constexpr int kSiteCache = 6;
constexpr int kJfaBlock = 128;

struct JfaShared {
    float4 pos[32];
    unsigned long long key[32];
    int32_t site[64];  // collected pairs: the candidate ...
    int32_t lane[64];  // ... and the lane whose sample it is for
};

__device__ __forceinline__ void jfa_pairs(const Tris& T, JfaShared& w, int first, int n)
{
    const int lane = (int)(threadIdx.x & 31u);
    if (lane < n) {
        const int to = w.lane[first + lane];
        const TriV v = tri_verts(T, w.site[first + lane]);
        const float4 q = w.pos[to];
        const float p[3] = {q.x, q.y, q.z};
        const float d2 = tri_d2_rn(p, v.a, v.b, v.c);
        atomicMin(&w.key[to], (unsigned long long)__float_as_uint(d2) << 32 | (uint32_t)v.id);
    }
    __syncwarp();
}

__global__ void __launch_bounds__(kJfaBlock) k_df_jfa(const DfGrid g, const Tris T, const int32_t* __restrict__ in,
                                                      int32_t* __restrict__ out, int32_t step)
{
    __shared__ int32_t list[26 * kJfaBlock];
    __shared__ JfaShared shared[kJfaBlock / 32];
    const unsigned full = 0xffffffffu;
    JfaShared& w = shared[threadIdx.x / 32];
    const int lane = (int)(threadIdx.x & 31u);
    const int64_t s = (int64_t)blockIdx.x * kJfaBlock + threadIdx.x;
    const bool on = s < g.count;
    const int64_t s0 = on ? s : 0;
    const int32_t nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int64_t jk = s0 / nx;
    const int32_t i = (int32_t)(s0 - jk * nx);
    const int32_t k = jk <= 0x7fffffff ? (int32_t)jk / ny : (int32_t)(jk / ny), j = (int32_t)(jk - (int64_t)k * ny);
    int32_t near[27];
#pragma unroll
    for (int q = 0; q < 27; ++q) {
        const int64_t x = i + (int64_t)(q % 3 - 1) * step, y = j + (int64_t)(q / 3 % 3 - 1) * step, z = k + (int64_t)(q / 9 - 1) * step;
        const bool inside = on && x >= 0 && x < nx && y >= 0 && y < ny && z >= 0 && z < nz;
        near[q] = inside ? __ldg(in + x + nx * (y + (int64_t)ny * z)) : -1;
    }
    const int32_t own = near[13];
    int listed = 0;
    int32_t seen[kSiteCache];
#pragma unroll
    for (int c = 0; c < kSiteCache; ++c) seen[c] = -1;
#pragma unroll
    for (int q = 0; q < 27; ++q) {
        const int32_t t = near[q];
        bool skip = t < 0 || t == own;
#pragma unroll
        for (int c = 0; c < kSiteCache; ++c) skip = skip || seen[c] == t;
        if (!skip) {
#pragma unroll
            for (int c = kSiteCache - 1; c > 0; --c) seen[c] = seen[c - 1];
            seen[0] = t;
            list[listed * kJfaBlock + threadIdx.x] = t;
            ++listed;
        }
    }
    float p[3];
    df_pos(g, i, j, k, p);
    w.pos[lane] = make_float4(p[0], p[1], p[2], 0.f);
    unsigned long long key = ~0ull;
    if (own >= 0) {
        const TriV v = tri_verts(T, own);
        key = (unsigned long long)__float_as_uint(tri_d2_rn(p, v.a, v.b, v.c)) << 32 | (uint32_t)v.id;
    }
    w.key[lane] = key;
    __syncwarp();
    const unsigned most = __reduce_max_sync(full, (unsigned)listed);
    int pairs = 0;
    for (unsigned c = 0; c < most; ++c) {
        bool near_enough = false;
        int32_t t = -1;
        if (c < (unsigned)listed) {
            t = list[c * kJfaBlock + threadIdx.x];
            // no site yet: the key's distance is a NaN, which nothing exceeds
            near_enough = !tri_farther(p, tri_verts(T, t), __uint_as_float((uint32_t)(w.key[lane] >> 32)));
        }
        const unsigned m = __ballot_sync(full, near_enough);
        if (near_enough) {
            const int at = pairs + __popc(m & ((1u << lane) - 1u));
            w.site[at] = t;
            w.lane[at] = lane;
        }
        pairs += __popc(m);
        __syncwarp();
        if (pairs >= 32) {
            pairs -= 32;
            jfa_pairs(T, w, pairs, 32);
        }
    }
    if (pairs) jfa_pairs(T, w, 0, pairs);
    if (!on) return;
    key = w.key[lane];
    out[s] = key == ~0ull ? -1 : __ldg(T.slot + (uint32_t)key);
}

// one thread per grid line along `axis`, walking in direction dir (+1 / -1).
// The line's sites are read eight at a time (independent loads in flight
// together); each is the value before this sweep reaches it, as in the
// sequential sweep, since the sweep only writes samples it has passed.
constexpr int kSweepChunk = 8;

__global__ void k_df_sweep(const DfGrid g, const Tris T, int32_t* sites, int axis, int dir)
{
    const int oa = axis == 0 ? 1 : 0, ob = axis == 2 ? 1 : 2;
    const int64_t line = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (line >= (int64_t)g.n[oa] * g.n[ob]) return;
    const int64_t n[3] = {g.n[0], g.n[1], g.n[2]};
    const int64_t stride[3] = {1, n[0], n[0] * n[1]};
    const int64_t ua = line % n[oa], ub = line / n[oa];
    const int64_t base = ua * stride[oa] + ub * stride[ob];
    const int64_t len = n[axis];
    int32_t prev = sites[base + (dir > 0 ? 0 : len - 1) * stride[axis]];
    for (int64_t c0 = 1; c0 < len; c0 += kSweepChunk) {
        int32_t buf[kSweepChunk];
#pragma unroll
        for (int u = 0; u < kSweepChunk; ++u) {
            const int64_t step = c0 + u;
            const int64_t q = dir > 0 ? step : len - 1 - step;
            buf[u] = step < len ? sites[base + q * stride[axis]] : -1;
        }
#pragma unroll
        for (int u = 0; u < kSweepChunk; ++u) {
            const int64_t step = c0 + u;
            if (step >= len) break;
            int32_t cur = buf[u];
            if (prev >= 0 && prev != cur) {  // otherwise nothing can change
                const int64_t q = dir > 0 ? step : len - 1 - step;
                int64_t ii[3];
                ii[axis] = q;
                ii[oa] = ua;
                ii[ob] = ub;
                float p[3];
                df_pos(g, ii[0], ii[1], ii[2], p);
                const TriV pv = tri_verts(T, prev);
                float cd2 = 0.f;
                int32_t cid = -1;
                if (cur >= 0) {
                    const TriV cv = tri_verts(T, cur);
                    cd2 = tri_d2_rn(p, cv.a, cv.b, cv.c);
                    cid = cv.id;
                }
                if (site_better(tri_d2_rn(p, pv.a, pv.b, pv.c), pv.id, cd2, cid)) {
                    cur = prev;
                    sites[base + q * stride[axis]] = cur;
                }
            }
            prev = cur;
        }
    }
}

// Both sweeps of one axis for one level, one warp per grid line (lines of one
// axis are independent, so the + sweep and then the - sweep of each line equal
// all + sweeps followed by all - sweeps).
//
// Triangles are small against the sample spacing, so most samples of a line have
// sites of their own and keep them.  A sample whose predecessor kept its site is
// offered that site: this is known for all samples in advance, so the warp tests
// 32 of them at a time.  Only where the offered site wins does the sweep go on in
// sequence: the winner is carried to the next samples, again tested 32 at a time,
// up to the first that keeps its own.  The triangles of the line's sites are read
// once, into shared memory, and so is each sample's distance to its own site; a
// sample holds the position of the sample its site came from.
//
// On a 64^3 level of the frame scene's cascade an axis took 50 to 210 us with one
// thread per line (4,096 lines, under one warp per SM, about 1.6 us a step), and
// 38 to 48 with the carried site tested ahead from every sample in turn.
constexpr int kLineMax = 1024;  // longest line swept in shared memory
constexpr int kLineBytes = 3 * 16 + 4 + 4;  // per sample: triangle (v0.w: input index), distance, site's origin

// the site that came from `carried` offered to sample q: whether it wins, and its distance there
__device__ __forceinline__ bool line_offer(const DfGrid& g, int32_t ii[3], int axis, const float4* tri, const float* d2,
                                           const int32_t* from, int q, int carried, float& d)
{
    const int own = from[q];
    const float4 a = tri[3 * carried], b = tri[3 * carried + 1], c = tri[3 * carried + 2];
    const int32_t id = __float_as_int(a.w), own_id = own >= 0 ? __float_as_int(tri[3 * own].w) : -1;
    if (own_id == id) return false;  // the same site: nothing changes
    float p[3];
    ii[axis] = q;
    df_pos(g, ii[0], ii[1], ii[2], p);
    const float va[3] = {a.x, a.y, a.z}, vb[3] = {b.x, b.y, b.z}, vc[3] = {c.x, c.y, c.z};
    d = tri_d2_rn(p, va, vb, vc);
    return site_better(d, id, d2[q], own_id);
}

__device__ __forceinline__ void sweep_line(const DfGrid& g, int32_t ii[3], int axis, const float4* tri, float* d2,
                                           int32_t* from, int len, int dir)
{
    const unsigned full = 0xffffffffu;
    const int lane = (int)(threadIdx.x & 31u);
    auto at = [&](int step) { return dir > 0 ? step : len - 1 - step; };
    int step = 1;
    while (step < len) {
        // the next 32 samples, each offered its predecessor's own site
        const bool valid = step + lane < len;
        const int q = valid ? at(step + lane) : 0;
        const int before = valid ? from[at(step + lane - 1)] : -1;
        float d = 0.f;
        const bool wins = valid && before >= 0 && line_offer(g, ii, axis, tri, d2, from, q, before, d);
        const unsigned m = __ballot_sync(full, wins);
        if (m == 0u) {  // every one keeps its own
            step += 32;
            continue;
        }
        const int first = __ffs(m) - 1;
        const int carried = __shfl_sync(full, before, first);
        if (lane == first) {
            from[q] = carried;
            d2[q] = d;
        }
        step += first + 1;
        __syncwarp();
        // the winner is carried on, up to the first sample that keeps its own site
        // (one with the same site neither changes nor stops it)
        while (step < len) {
            const bool ok = step + lane < len;
            const int r = ok ? at(step + lane) : 0;
            float e = 0.f;
            const bool takes = ok && line_offer(g, ii, axis, tri, d2, from, r, carried, e);
            const bool same = ok && from[r] >= 0 && __float_as_int(tri[3 * from[r]].w) == __float_as_int(tri[3 * carried].w);
            const unsigned stop = __ballot_sync(full, ok && !takes && !same);
            const int end = stop ? __ffs(stop) - 1 : 32;
            __syncwarp();
            if (takes && lane < end) {
                from[r] = carried;
                d2[r] = e;
            }
            step += stop ? end + 1 : 32;
            __syncwarp();
            if (stop) break;
        }
    }
}

__global__ void k_df_sweep_line(const DfGrid g, const Tris T, int32_t* sites, int axis)
{
    extern __shared__ float4 s_line[];
    const int oa = axis == 0 ? 1 : 0, ob = axis == 2 ? 1 : 2;
    const int warps = (int)blockDim.x / 32, warp = (int)threadIdx.x / 32, lane = (int)(threadIdx.x & 31u);
    const int64_t line = (int64_t)blockIdx.x * warps + warp;
    if (line >= (int64_t)g.n[oa] * g.n[ob]) return;
    const int len = g.n[axis];
    float4* tri = s_line + (size_t)warp * 3 * len;
    float* d2 = reinterpret_cast<float*>(s_line + (size_t)warps * 3 * len) + (size_t)warp * 2 * len;
    int32_t* from = reinterpret_cast<int32_t*>(d2 + len);
    const int64_t stride[3] = {1, g.n[0], (int64_t)g.n[0] * g.n[1]};
    int32_t ii[3];
    ii[oa] = (int32_t)(line % g.n[oa]);
    ii[ob] = (int32_t)(line / g.n[oa]);
    const int64_t base = ii[oa] * stride[oa] + ii[ob] * stride[ob];
    for (int q = lane; q < len; q += 32) {
        const int32_t k = sites[base + q * stride[axis]];
        from[q] = k >= 0 ? q : -1;
        d2[q] = 0.f;
        if (k >= 0) {
            const float4* v = T.tris + 3 * (int64_t)k;
            const float4 a = __ldg(v), b = __ldg(v + 1), c = __ldg(v + 2);
            tri[3 * q] = a;
            tri[3 * q + 1] = make_float4(b.x, b.y, b.z, __int_as_float(k));  // v1.w: leaf position
            tri[3 * q + 2] = c;
            float p[3];
            ii[axis] = q;
            df_pos(g, ii[0], ii[1], ii[2], p);
            const float va[3] = {a.x, a.y, a.z}, vb[3] = {b.x, b.y, b.z}, vc[3] = {c.x, c.y, c.z};
            d2[q] = tri_d2_rn(p, va, vb, vc);
        }
    }
    __syncwarp();
    sweep_line(g, ii, axis, tri, d2, from, len, 1);
    sweep_line(g, ii, axis, tri, d2, from, len, -1);
    for (int q = lane; q < len; q += 32) {
        const int o = from[q];
        if (o != q && o >= 0) sites[base + q * stride[axis]] = __float_as_int(tri[3 * o + 1].w);
    }
}

// The end of a level: its sites as input indices, and (grid non-null) the signed
// distance to each site's triangle (the exact bake's closest point and sign).
__global__ void k_df_finish(const DfGrid g, const Tris T, const float4* pn, const int32_t* sites, int32_t* ids, void* grid,
                            int32_t f16)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.count) return;
    const int32_t k = sites[s];
    ids[s] = k >= 0 ? __float_as_int(__ldg(&T.tris[3 * (int64_t)k].w)) : -1;
    if (!grid) return;
    float v = __int_as_float(0x7f800000);
    if (k >= 0) {
        float pp[3];
        df_pos(g, s % g.n[0], (s / g.n[0]) % g.n[1], s / ((int64_t)g.n[0] * g.n[1]), pp);
        const float3 p = make_float3(pp[0], pp[1], pp[2]);
        rtbake::Nearest nb = {__int_as_float(0x7f800000), -1, 0x7fffffff};
        rtbake::consider(nb, p, T.tris, k);
        v = rtbake::signed_distance(p, nb, T.tris, pn);
    }
    if (f16) reinterpret_cast<__half*>(grid)[s] = __float2half_rn(v);
    else reinterpret_cast<float*>(grid)[s] = v;
}

// geometry of the single grid, or of cascade level k
DfGrid df_grid(const rt_sdf* sdf, int k)
{
    DfGrid g;
    memset(&g, 0, sizeof(g));
    g.count = 1;
    for (int a = 0; a < 3; ++a) {
        g.n[a] = sdf->n[a];
        g.count *= sdf->n[a];
    }
    double origin[3];
    if (sdf->levels > 0) {
        const float hk = ldexpf(sdf->h0, k);
        g.lattice = 1;
        for (int a = 0; a < 3; ++a) {
            g.ilo[a] = sdf->ilo[k][a];
            g.h[a] = hk;
            origin[a] = (double)sdf->ilo[k][a] * (double)hk;
        }
    } else {
        for (int a = 0; a < 3; ++a) {
            g.lo[a] = sdf->lo[a];
            g.h[a] = sdf->h[a];
            origin[a] = sdf->lo[a];
        }
    }
    for (int a = 0; a < 3; ++a) {
        volatile float half = 0.5f * g.h[a];
        volatile float grow = g.h[a] * (1.f / 512.f);
        g.hs[a] = half + grow;
        g.ih_f[a] = 1.0f / g.h[a];
        g.margin[a] = (float)(1e-2 * g.h[a] + 1e-5 * (fabs(origin[a]) + g.n[a] * (double)g.h[a]));
        g.origin_f[a] = (float)origin[a];
    }
    return g;
}

unsigned blocks_for(int64_t n) { return (unsigned)((n + kBlock - 1) / kBlock); }

constexpr int64_t kBigMost = 1 << 18;  // large (triangle, level) pairs listed for a block each

// Steps 1..stage for the levels `lv[0..nl)` (0 for a single grid), given in
// the order they are built (coarsest first).  All levels are voxelised in one
// pass over the triangles (a level's voxel candidates do not depend on the
// other levels); then each level in turn is seeded (on a cascade also from the
// next coarser level's finished sites in `ids`), flooded and swept, leaving its
// sites in `ids` (one input index per sample of every level, device) before the
// next finer level reads them, and with `values` its field values in the grid.
rt_status df_build(const rt_scene* sc, const rt_sdf* sdf, const int* lv, int nl, int32_t stage, int32_t* ids, bool values,
                   cudaStream_t s)
{
    const Tris T = {sc->tris, sc->slot, sc->n_tris};
    const int64_t per = (int64_t)sdf->n[0] * sdf->n[1] * sdf->n[2];
    if (per > 0x7fffffffLL * (int64_t)kBlock) return rt_fail(RT_ERR_INVALID_ARG, "grid too large");
    const int cascade_levels = sdf->levels;

    // scratch: keys of every listed level, two site buffers, the large-triangle list
    auto align = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const unsigned most_big = (unsigned)(T.n * nl < kBigMost ? T.n * nl : kBigMost);
    const size_t keys_bytes = align((size_t)per * 8 * nl), sites_bytes = align((size_t)per * 4);
    const size_t big_bytes = align((size_t)most_big * sizeof(int2));
    void* scratch = nullptr;
    rt_status st = rt_scratch_alloc(&scratch, keys_bytes + 2 * sites_bytes + big_bytes + 256, s);
    if (st != RT_OK) return st;
    char* base = static_cast<char*>(scratch);
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(base);
    int32_t* work[2] = {reinterpret_cast<int32_t*>(base + keys_bytes), reinterpret_cast<int32_t*>(base + keys_bytes + sites_bytes)};
    int2* big = reinterpret_cast<int2*>(base + keys_bytes + 2 * sites_bytes);
    unsigned* n_big = reinterpret_cast<unsigned*>(base + keys_bytes + 2 * sites_bytes + big_bytes);

    cudaError_t e = cudaMemsetAsync(keys, 0xff, (size_t)per * 8 * nl, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(n_big, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) st = rt_cuda_fail(e, "cudaMemsetAsync");

    // 1. voxelisation of all listed levels
    if (st == RT_OK && T.n > 0) {
        VoxPass vp;
        memset(&vp, 0, sizeof(vp));
        vp.count = nl;
        for (int l = 0; l < nl; ++l) {
            vp.g[l] = df_grid(sdf, lv[l]);
            vp.keys[l] = keys + (size_t)l * per;
        }
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        k_df_vox_small<<<blocks_for(T.n), kBlock, 0, s>>>(vp, T, big, n_big, most_big);
        k_df_vox_big<<<(unsigned)(sms > 0 ? sms * 4 : 512), kBlock, 0, s>>>(vp, T, big, n_big, most_big);
    }
    // 2.-3. per level, coarsest first: seeding, jump flooding, the six sweeps
    const int64_t esz = sdf->dtype == RT_GRID_F16 ? 2 : 4;
    for (int l = 0; l < nl && st == RT_OK; ++l) {
        const int k = lv[l];
        const DfGrid g = df_grid(sdf, k);
        DfGrid gc;
        memset(&gc, 0, sizeof(gc));
        const int32_t* coarse = nullptr;
        if (cascade_levels > 0 && k + 1 < cascade_levels) {
            gc = df_grid(sdf, k + 1);
            coarse = ids + (int64_t)(k + 1) * per;
        }
        int32_t* sites = work[0];
        int32_t* other = work[1];
        k_df_seed<<<blocks_for(g.count), kBlock, 0, s>>>(g, T, keys + (size_t)l * per, coarse, gc, sites);
        if (stage >= 2) {
            int64_t nmax = g.n[0] > g.n[1] ? g.n[0] : g.n[1];
            if (g.n[2] > nmax) nmax = g.n[2];
            int64_t step = 1;
            while (2 * step < nmax) step *= 2;
            for (; step >= 1; step /= 2) {
                k_df_jfa<<<(unsigned)((g.count + kJfaBlock - 1) / kJfaBlock), kJfaBlock, 0, s>>>(g, T, sites, other, (int32_t)step);
                int32_t* t = sites;
                sites = other;
                other = t;
            }
        }
        if (stage >= 3) {
            for (int axis = 0; axis < 3 && st == RT_OK; ++axis) {
                const int oa = axis == 0 ? 1 : 0, ob = axis == 2 ? 1 : 2;
                const int64_t lines = (int64_t)g.n[oa] * g.n[ob];
                if (g.n[axis] <= kLineMax) {
                    // four lines a block while they fit in 48 KB of shared memory
                    const size_t line_bytes = (size_t)g.n[axis] * kLineBytes;
                    const int warps = 4 * line_bytes <= (48 << 10) ? 4 : (2 * line_bytes <= (48 << 10) ? 2 : 1);
                    const size_t smem = warps * line_bytes;
                    if (smem > 48 * 1024) {
                        e = cudaFuncSetAttribute(k_df_sweep_line, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                        if (e != cudaSuccess) st = rt_cuda_fail(e, "cudaFuncSetAttribute");
                    }
                    if (st == RT_OK)
                        k_df_sweep_line<<<(unsigned)((lines + warps - 1) / warps), 32 * warps, smem, s>>>(g, T, sites, axis);
                } else {
                    for (int dir = 1; dir >= -1; dir -= 2)
                        k_df_sweep<<<(unsigned)((lines + 63) / 64), 64, 0, s>>>(g, T, sites, axis, dir);
                }
            }
        }
        void* grid = values ? static_cast<char*>(const_cast<void*>(sdf->grid)) + k * per * esz : nullptr;
        if (st == RT_OK)
            k_df_finish<<<blocks_for(g.count), kBlock, 0, s>>>(g, T, sc->pn, sites, ids + (int64_t)k * per, grid,
                                                               sdf->dtype == RT_GRID_F16);
    }
    if (st == RT_OK) {
        e = cudaGetLastError();
        if (e != cudaSuccess) st = rt_cuda_fail(e, "field build launch");
    }
    e = cudaFreeAsync(scratch, s);
    if (st == RT_OK && e != cudaSuccess) st = rt_cuda_fail(e, "cudaFreeAsync");
    return st;
}

}  // namespace

// Sites of every sample after step `stage` (1..3), cascade levels one at a
// time, coarsest first (each seeded also from the next coarser level's sites
// after its steps 1..stage).
// d_sites holds levels * n^3 (or n0 n1 n2) entries.
rt_status rt_launch_df_sites(const rt_scene* sc, const rt_sdf* sdf, int32_t stage, int32_t* d_sites, cudaStream_t s)
{
    int lv[RT_MAX_LEVELS];
    const int nl = sdf->levels > 0 ? sdf->levels : 1;
    for (int l = 0; l < nl; ++l) lv[l] = nl - 1 - l;  // coarsest first
    return df_build(sc, sdf, lv, nl, stage, d_sites, false, s);
}

// The listed levels (all of them for a full build; the moved ones of a rolling
// update), coarsest first: finished sites into `ids` (kept by the handle: the
// seeds of finer levels later), field values from them.
rt_status rt_launch_df_levels(const rt_scene* sc, const rt_sdf* sdf, const int* lv, int nl, int32_t* ids, cudaStream_t s)
{
    if (nl <= 0) return RT_OK;
    return df_build(sc, sdf, lv, nl, 3, ids, true, s);
}
