// Distance-field bake: at every grid sample, the distance to the nearest
// triangle with the sign of the angle-weighted pseudonormal of the nearest
// feature (Baerentzen & Aanaes, IEEE TVCG 2005).  Positive on the side the
// triangle normals face.  The closest point on a triangle is found from the
// Voronoi regions of the triangle (Ericson, Real-Time Collision Detection,
// 5.1.5).  The paper builds its field by rasterised voxelisation, jump
// flooding and fast sweeping (Section 3, "Distance Field Generation"); this is
// the exact definition that those steps approximate.
//
// Two methods with the same result: brute force (every triangle, staged through
// shared memory in tiles) and a BVH-pruned nearest query, which a warp runs for
// up to 32 neighbouring samples together (k_bake_bricks), or, with few triangles,
// a thread for one sample (k_bake_threads).
#include <math.h>
#include <string.h>

#include "rt_bake_dev.cuh"
#include "rt_trace_dev.cuh"

namespace {

using namespace rtbake;

constexpr int kBakeBlock = 128;
constexpr int kBrickWarps = 2;  // bricks per block: few, as their times differ (1: 5 %, 4: 4 % slower at 256^3)
constexpr int kTile = 128;
constexpr unsigned kFull = 0xffffffffu;

struct BakeArgs {
    const BNode* nodes;
    const float4* tris;
    const float4* pn;
    const int32_t* slot;
    int64_t n_tris;
    void* grid;   // null: only the sites are wanted
    int32_t f16;
    float lo[3], h[3];
    int32_t n[3];
    int64_t count;
    // cascade level: samples at (ilo + i) * h[0], one rounding per coordinate,
    // so a sample's position depends only on its absolute lattice index
    int32_t lattice;
    int32_t ilo[3];
    // Source lattice: samples whose nearest triangle (ssrc) or value (bsrc) is
    // already known.  A sample at absolute lattice index a (a = ilo + i on a
    // cascade level, a = i otherwise) takes the source sample
    // j = clamp(round(a / bratio) - bilo, 0, bdim - 1), x fastest.
    //   ssrc  leaf position of the source's nearest triangle: the search starts
    //         from the distance to that triangle
    //   bsrc  value of the source (a field of this grid's type): the search
    //         starts from |phi(source)| + |p - source|, since the distance
    //         function is 1-Lipschitz
    // The nearest triangle found is the same as without either.
    const int32_t* ssrc;
    const void* bsrc;
    int32_t bratio;
    int32_t bilo[3], bdim[3];
    int32_t src_relative;  // 1: a = i on a cascade level too (the source counts from this grid's first sample)
    int32_t brute_sum;  // 1: the squared distance is summed as k_bake_brute's is (an ulp can differ)
    int32_t* sdst;  // nearest triangle (leaf position) of every sample visited, x fastest over its box; null: not wanted
};

// The samples a launch takes: up to three disjoint boxes of the grid, cut into
// bricks of 2^brick_log2 samples, one warp each.  Box samples are at stride `sub` (the
// coarse first pass of a bake takes every kSubStride-th sample per axis).
struct PacketBox {
    int32_t lo[3], dim[3], shift[3];  // brick edges 2^shift
    int64_t first;                    // number of bricks in the boxes before
};
struct PacketGrid {
    PacketBox box[3];
    int32_t boxes, sub, brick_log2;
    int64_t packets;
};

__device__ __forceinline__ float3 sample_pos(const BakeArgs& b, const int32_t ii[3])
{
    if (b.lattice)
        return make_float3(__fmul_rn((float)(b.ilo[0] + ii[0]), b.h[0]), __fmul_rn((float)(b.ilo[1] + ii[1]), b.h[0]),
                           __fmul_rn((float)(b.ilo[2] + ii[2]), b.h[0]));
    return make_float3(fmaf((float)ii[0], b.h[0], b.lo[0]), fmaf((float)ii[1], b.h[1], b.lo[1]),
                       fmaf((float)ii[2], b.h[2], b.lo[2]));
}

__device__ __forceinline__ void store(const BakeArgs& b, int64_t i, float v)
{
    if (b.f16) reinterpret_cast<__half*>(b.grid)[i] = __float2half_rn(v);
    else reinterpret_cast<float*>(b.grid)[i] = v;
}

__global__ void __launch_bounds__(kBakeBlock) k_bake_brute(const BakeArgs b)
{
    __shared__ float4 tile[3 * kTile];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = i < b.count;  // every thread stays for the barriers
    const int64_t i0 = live ? i : 0;
    const int32_t ii[3] = {(int32_t)(i0 % b.n[0]), (int32_t)((i0 / b.n[0]) % b.n[1]), (int32_t)(i0 / ((int64_t)b.n[0] * b.n[1]))};
    const float3 p = sample_pos(b, ii);
    Nearest nb = {__int_as_float(0x7f800000), -1, 0x7fffffff};
    for (int64_t t0 = 0; t0 < b.n_tris; t0 += kTile) {
        const int m = (int)min((int64_t)kTile, b.n_tris - t0);
        __syncthreads();
        for (int j = threadIdx.x; j < 3 * m; j += blockDim.x) tile[j] = __ldg(b.tris + 3 * t0 + j);
        __syncthreads();
        if (live) {
            for (int j = 0; j < m; ++j) {
                float3 q;
                closest_point(p, xyz(tile[3 * j]), xyz(tile[3 * j + 1]), xyz(tile[3 * j + 2]), q);
                float3 pq = sub(p, q);
                float d2 = dot(pq, pq);
                int32_t prim = __float_as_int(tile[3 * j].w);
                if (d2 < nb.d2 || (d2 == nb.d2 && prim < nb.prim)) {
                    nb.d2 = d2;
                    nb.k = (int32_t)(t0 + j);
                    nb.prim = prim;
                }
            }
        }
    }
    if (live) store(b, i, signed_distance(p, nb, b.tris, b.pn));
}

// squared distance from p to the box (lo.x, hi.x, lo.y, hi.y), (lo.z, hi.z)
__device__ __forceinline__ float box_d2(float lx, float hx, float ly, float hy, float lz, float hz, float3 p)
{
    const float dx = rtdev::max3f(lx - p.x, p.x - hx, 0.f);
    const float dy = rtdev::max3f(ly - p.y, p.y - hy, 0.f);
    const float dz = rtdev::max3f(lz - p.z, p.z - hz, 0.f);
    return dx * dx + dy * dy + dz * dz;
}

__device__ __forceinline__ float load_value(const void* g, int32_t f16, int64_t i)
{
    return f16 ? __half2float(reinterpret_cast<const __half*>(g)[i]) : reinterpret_cast<const float*>(g)[i];
}

__device__ __forceinline__ int64_t floordiv(int64_t x, int64_t y)  // y > 0
{
    return x >= 0 ? x / y : -((-x + y - 1) / y);
}

// the source sample of sample ii: its element and its squared distance
__device__ __forceinline__ int64_t source_of(const BakeArgs& b, const int32_t ii[3], float& d2)
{
    int64_t el = 0, stride = 1;
    d2 = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int64_t abs_i = (b.lattice && !b.src_relative ? b.ilo[a] : 0) + (int64_t)ii[a];
        int64_t j = floordiv(2 * abs_i + b.bratio, 2 * (int64_t)b.bratio) - b.bilo[a];  // round(abs_i / bratio)
        j = j < 0 ? 0 : (j > b.bdim[a] - 1 ? b.bdim[a] - 1 : j);
        const float gap = (float)(abs_i - (j + b.bilo[a]) * b.bratio) * b.h[a];
        d2 += gap * gap;
        el += j * stride;
        stride *= b.bdim[a];
    }
    return el;
}

// upper bound on the distance at a sample from the value of its source
__device__ __forceinline__ float distance_bound(const BakeArgs& b, const int32_t ii[3])
{
    if (!b.bsrc) return __int_as_float(0x7f800000);
    float d2;
    const int64_t el = source_of(b, ii, d2);
    const float phi = fabsf(load_value(b.bsrc, b.f16, el));
    // generous margin for the rounding of the stored value (float16 included)
    return (phi + sqrtf(d2)) * 1.002f + 1e-6f;
}

// ---------------------------------------------------------------------------
// Nearest triangle of a brick of S neighbouring samples, by one warp (S = 32, 8
// or 1).  The samples' positions and squared distances so far lie in shared
// memory, and the warp works on batches:
//   nodes   up to 32 nodes from the top of a stack, each by 32 / (their number)
//           lanes; a child is kept when any sample's distance reaches its box (a
//           coarser test, of spheres around four samples' searches, passed 3.5
//           times the leaves: 20.4 ms)
//   leaves  32 triangles are brought to shared memory; each (sample, triangle)
//           pair is tested against a disc that holds the triangle, 32 pairs at
//           a time, and the pairs left are collected
//   pairs   32 at a time, the exact distance; the smaller (squared distance,
//           input index) wins by a 64-bit minimum in shared memory
// So loads of 32 nodes or triangles are in flight together and every lane has
// work in each step.  One traversal per thread (lanes waiting at different
// nodes and in different regions of the closest point) took 31.3 ms for the
// 256^3 samples of the frame scene (2,050,412 triangles), one traversal per warp
// over 32 samples in lockstep 16.9 ms, this 11.0 ms; six moves of a 5 x 64^3
// cascade by one voxel, whose 11 new slabs each lasted as long as their slowest
// sample, 2.9 and 0.70 ms.  What bounds it now is issue: a brick visits 217 nodes
// and 100 leaves.
//
// The disc test (the triangle lies in a disc around its centroid) decides most
// pairs: 1,652 of a brick's 3,200 pairs passed a test against the plane alone.
// Boxes of tilted triangles reach towards the sample by about half an edge, so
// near the centre of a round object thousands of leaves pass the box test, while
// a disc's distance exceeds its triangle's only by the sagitta.  The test leaves
// a margin for every rounding in it and in closest_point_rn (4e-5 of the squared
// distance to the centroid and of the squared longest edge, the latter in pn.w,
// and the square of 1.4e-4 of the position, whose ulp rounds the closest point;
// badly shaped triangles have pn.w = inf and always pass), so the triangle found
// is the one found without it.
// ---------------------------------------------------------------------------
constexpr int kNodeStack = 384;   // a batch takes fewer nodes when this fills; depth first always fits
constexpr int kLeafQueue = 96;    // at most 31 left over and 64 from one batch

struct BrickShared {
    float4 sample[32];            // position, squared distance so far (-1: takes no part)
    unsigned long long key[32];   // squared distance bits << 32 | input index: the smaller is the nearer
    float4 v0[32], v1[32], v2[32];
    float4 normal[32], disc[32];  // face normal, margin; centroid, distance of the farthest vertex
    int32_t stack[kNodeStack];
    int32_t leaf[kLeafQueue];
    uint16_t pair[64];            // sample << 5 | triangle of the batch
};

// exact distances of the last n pairs (n <= 32)
__device__ __forceinline__ void brick_pairs(const BakeArgs& b, BrickShared& w, int first, int n)
{
    const int lane = (int)(threadIdx.x & 31u);
    if (lane < n) {
        const int e = w.pair[first + lane], i = e & 31, s = e >> 5;
        const float4 ps = w.sample[s], a = w.v0[i];
        const float3 p = xyz(ps);
        float3 q;
        closest_point_rn(p, xyz(a), xyz(w.v1[i]), xyz(w.v2[i]), q);
        const float d2 = gap2_rn(p, q, b.brute_sum);
        if (d2 <= ps.w) atomicMin(&w.key[s], (unsigned long long)__float_as_uint(d2) << 32 | __float_as_uint(a.w));
    }
    __syncwarp();
    if (w.sample[lane].w >= 0.f) w.sample[lane].w = __uint_as_float((uint32_t)(w.key[lane] >> 32));
    __syncwarp();
}

// the n leaves w.leaf[first ..] (n <= 32)
template <int LS>
__device__ __forceinline__ void brick_leaves(const BakeArgs& b, BrickShared& w, int first, int n)
{
    constexpr int S = 1 << LS;
    const int lane = (int)(threadIdx.x & 31u);
    if (lane < n) {
        const int64_t k = w.leaf[first + lane];
        const float4 a = __ldg(b.tris + 3 * k), bb = __ldg(b.tris + 3 * k + 1), c = __ldg(b.tris + 3 * k + 2);
        const float3 m = make_float3((a.x + bb.x + c.x) * (1.f / 3.f), (a.y + bb.y + c.y) * (1.f / 3.f), (a.z + bb.z + c.z) * (1.f / 3.f));
        const float3 ma = sub(xyz(a), m), mb = sub(xyz(bb), m), mc = sub(xyz(c), m);
        w.v0[lane] = a;
        w.v1[lane] = bb;
        w.v2[lane] = c;
        w.normal[lane] = __ldg(b.pn + 7 * k);
        w.disc[lane] = make_float4(m.x, m.y, m.z, sqrtf(rtdev::max3f(dot(ma, ma), dot(mb, mb), dot(mc, mc))));
    }
    __syncwarp();
    const int s = lane & (S - 1);
    const float3 p = xyz(w.sample[s]);
    const float coord = 2e-8f * dot(p, p);
    int pairs = 0;
    for (int i0 = 0; i0 < n; i0 += 32 / S) {
        const int i = i0 + (lane >> LS);
        bool near = false;
        if (i < n) {
            // the triangle lies in the disc of radius disc.w around disc.xyz in its plane
            const float best = w.sample[s].w;
            const float4 nn = w.normal[i], dc = w.disc[i];
            const float3 mp = sub(p, xyz(dc));
            const float h = dot(xyz(nn), mp), h2 = h * h, r2 = dot(mp, mp);
            const float out = fmaxf(sqrtf(fmaxf(r2 - h2, 0.f)) - dc.w, 0.f);
            near = best >= 0.f && !(fmaf(out, out, h2) > best + (fmaf(4e-5f, r2, nn.w) + coord));
        }
        const unsigned m = __ballot_sync(kFull, near);
        if (near) w.pair[pairs + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(s << 5 | i);
        pairs += __popc(m);
        if (pairs >= 32) {
            __syncwarp();
            pairs -= 32;
            brick_pairs(b, w, pairs, 32);
        }
    }
    __syncwarp();
    if (pairs) brick_pairs(b, w, 0, pairs);
}

// search the whole tree; w.sample and w.key set, w.leaf holding `leaves` (at most
// 32) triangles to look at first
template <int LS>
__device__ __forceinline__ void brick_search(const BakeArgs& b, BrickShared& w, int leaves)
{
    constexpr int S = 1 << LS;
    const int lane = (int)(threadIdx.x & 31u);
    brick_leaves<LS>(b, w, 0, leaves);
    leaves = 0;
    int nodes = 0;
    if (lane == 0) {
        if (b.n_tris > 1) w.stack[0] = 0;
        else w.leaf[0] = 0;
    }
    if (b.n_tris > 1) nodes = 1;
    else leaves = 1;
    __syncwarp();
    // bounded by the number of nodes; the guard stops only a corrupt structure
    for (uint32_t guard = 0; guard < (1u << 26); ++guard) {
        if (leaves >= 32 || (nodes == 0 && leaves > 0)) {
            const int n = min(leaves, 32);
            leaves -= n;
            brick_leaves<LS>(b, w, leaves, n);
            continue;
        }
        if (nodes == 0) break;
        // every node taken may leave two: near the stack's end take fewer, down to
        // one (depth first), whose path needs at most RT_STACK_DEPTH more entries
        int m = min(min(nodes, 32), max(1, kNodeStack - (RT_STACK_DEPTH + 2) - nodes));
        int lg = 31 - __clz(m);  // lanes per node: 32 >> lg
        if ((1 << lg) < m) {
            // with one sample every batch is one step; with more, idle lanes cost steps
            if (S == 1) ++lg;
            else m = 1 << lg;
        }
        const int per = 32 >> lg, mine = lane >> (5 - lg);
        nodes -= m;
        bool h0 = false, h1 = false;
        int32_t c0 = 0, c1 = 0;
        if (mine < m) {
            float v[8], u[8];
            rtdev::load_node(b.nodes, w.stack[nodes + mine], v, u);
            c0 = __float_as_int(u[4]);
            c1 = __float_as_int(u[5]);
#pragma unroll 2
            for (int s = lane & (per - 1); s < S; s += per) {
                const float4 q = w.sample[s];
                const float3 p = xyz(q);
                h0 = h0 | (box_d2(v[0], v[1], v[2], v[3], u[0], u[1], p) <= q.w);
                h1 = h1 | (box_d2(v[4], v[5], v[6], v[7], u[2], u[3], p) <= q.w);
            }
        }
        const unsigned g = (per == 32 ? 0xffffffffu : (1u << per) - 1u) << (mine * per & 31);
        const bool lead = (lane & (per - 1)) == 0;
        const unsigned a0 = __ballot_sync(kFull, h0), a1 = __ballot_sync(kFull, h1);
        h0 = lead && (a0 & g) != 0u;
        h1 = lead && (a1 & g) != 0u;
        const unsigned n0 = __ballot_sync(kFull, h0 && c0 >= 0), n1 = __ballot_sync(kFull, h1 && c1 >= 0);
        const unsigned l0 = __ballot_sync(kFull, h0 && c0 < 0), l1 = __ballot_sync(kFull, h1 && c1 < 0);
        const unsigned below = (1u << lane) - 1u;
        if (h0) {
            if (c0 >= 0) w.stack[nodes + __popc(n0 & below)] = c0;
            else w.leaf[leaves + __popc(l0 & below)] = ~c0;
        }
        if (h1) {
            if (c1 >= 0) w.stack[nodes + __popc(n0) + __popc(n1 & below)] = c1;
            else w.leaf[leaves + __popc(l0) + __popc(l1 & below)] = ~c1;
        }
        nodes += __popc(n0) + __popc(n1);
        leaves += __popc(l0) + __popc(l1);
        __syncwarp();
    }
}

// leaf reached from the root by always taking the child whose box is nearer to p
__device__ __forceinline__ int32_t greedy_leaf(const BakeArgs& b, float3 p)
{
    int32_t node = b.n_tris > 1 ? 0 : ~0;
    for (int depth = 0; node >= 0 && depth <= RT_STACK_DEPTH; ++depth) {
        float v[8], u[8];
        rtdev::load_node(b.nodes, node, v, u);
        node = box_d2(v[4], v[5], v[6], v[7], u[2], u[3], p) < box_d2(v[0], v[1], v[2], v[3], u[0], u[1], p)
                   ? __float_as_int(u[5]) : __float_as_int(u[4]);
    }
    return node < 0 ? ~node : 0;
}

// sample of this lane (lane mod S) in brick `packet`; false outside its box
template <int LS>
__device__ __forceinline__ bool packet_sample(const PacketGrid& pg, int64_t packet, int32_t ii[3], int64_t& box_el)
{
    int k = 0;
    while (k + 1 < pg.boxes && packet >= pg.box[k + 1].first) ++k;
    const PacketBox& bx = pg.box[k];
    const int64_t r = packet - bx.first;
    const int64_t nx = (bx.dim[0] + (1 << bx.shift[0]) - 1) >> bx.shift[0], ny = (bx.dim[1] + (1 << bx.shift[1]) - 1) >> bx.shift[1];
    const int s = (int)(threadIdx.x & 31u) & ((1 << LS) - 1);
    const int32_t j[3] = {(int32_t)(r % nx << bx.shift[0]) + (s & ((1 << bx.shift[0]) - 1)),
                          (int32_t)((r / nx) % ny << bx.shift[1]) + ((s >> bx.shift[0]) & ((1 << bx.shift[1]) - 1)),
                          (int32_t)(r / (nx * ny) << bx.shift[2]) + (s >> (bx.shift[0] + bx.shift[1]))};
    const bool in = j[0] < bx.dim[0] && j[1] < bx.dim[1] && j[2] < bx.dim[2];
    box_el = j[0] + (int64_t)bx.dim[0] * (j[1] + (int64_t)bx.dim[1] * j[2]);
#pragma unroll
    for (int a = 0; a < 3; ++a) ii[a] = in ? (bx.lo[a] + j[a]) * pg.sub : 0;
    return in;
}

__device__ __forceinline__ int64_t sample_index(const BakeArgs& b, const int32_t ii[3])
{
    return ii[0] + (int64_t)b.n[0] * (ii[1] + (int64_t)b.n[1] * ii[2]);
}

// 16 blocks (32 warps) an SM, 64 registers: 256^3 10.95 ms; the compiler's own 72
// registers 11.32, 18 blocks 11.07, 20 blocks (with spills) 12.02.
template <int LS>
__global__ void __launch_bounds__(32 * kBrickWarps, 16) k_bake_bricks(const BakeArgs b, const PacketGrid pg)
{
    constexpr int S = 1 << LS;
    __shared__ BrickShared shared[kBrickWarps];
    BrickShared& w = shared[threadIdx.x / 32];
    const int lane = (int)(threadIdx.x & 31u);
    const int64_t packet = (int64_t)blockIdx.x * kBrickWarps + threadIdx.x / 32;
    if (packet >= pg.packets) return;
    int32_t ii[3];
    int64_t box_el;
    const bool in = packet_sample<LS>(pg, packet, ii, box_el) && lane < S;
    const float3 p = sample_pos(b, ii);
    // where the search starts: a triangle near the sample's nearest one (the
    // source's, or the end of a greedy descent), and the source's value
    float bound = __int_as_float(0x7f800000);
    int32_t seed = -1;
    if (b.ssrc) {
        float gap2;
        seed = __ldg(b.ssrc + source_of(b, ii, gap2));
    } else {
        bound = distance_bound(b, ii);
    }
    if (seed < 0) seed = greedy_leaf(b, p);
    bool lost = in;
    for (int pass = 0; pass < 2; ++pass) {  // a second time, without the bound, where it held no triangle
        const float start = pass == 0 ? bound * bound : __int_as_float(0x7f800000);
        w.sample[lane] = make_float4(p.x, p.y, p.z, lost ? start : -1.f);
        w.key[lane] = (unsigned long long)__float_as_uint(start) << 32 | 0xffffffffu;
        // the brick's distinct seeds, looked at first by all its samples
        const unsigned same = __match_any_sync(kFull, in ? seed : -1);
        const bool first = in && (same & ((1u << lane) - 1u)) == 0u;
        const unsigned firsts = __ballot_sync(kFull, first);
        if (first) w.leaf[__popc(firsts & ((1u << lane) - 1u))] = seed;
        __syncwarp();
        brick_search<LS>(b, w, __popc(firsts));
        const uint32_t prim = (uint32_t)w.key[lane];
        if (lost && prim != 0xffffffffu) {
            Nearest nb = {__uint_as_float((uint32_t)(w.key[lane] >> 32)), __ldg(b.slot + prim), (int32_t)prim};
            if (b.sdst) b.sdst[box_el] = nb.k;
            if (b.grid) store(b, sample_index(b, ii), signed_distance_rn(p, nb, b.tris, b.pn));
            lost = false;
        }
        if (__ballot_sync(kFull, lost) == 0u) return;
        __syncwarp();
    }
    if (lost) {  // no triangle at a finite distance
        if (b.sdst) b.sdst[box_el] = -1;
        if (b.grid) store(b, sample_index(b, ii), __int_as_float(0x7f800000));
    }
}

// Few triangles (few_triangles): one traversal per thread, whose path is shorter than
// the fixed steps of a brick's search.  What bounds it is the latency of the nodes and
// triangles of the longest path.  A sample searches within the bound that its source's
// value gives, so no sites are kept and no scratch is needed: a bake that cannot have
// its scratch takes this too.
struct ThreadPass {
    int32_t sub;        // > 0: only the samples whose indices are multiples of it
    int32_t own;        // > 0: the source is this grid's own samples at that stride, which are left as they are
    const void* keep;   // rolling update: sample i takes the value of sample i + shift of it wherever that lies
    int32_t shift[3];   // inside the level (the level before the move)
};

// nearest triangle to p among those at most sqrt(d2_start) away; k = -1 when there is none
__device__ __forceinline__ Nearest nearest_triangle(const BakeArgs& b, float3 p, float d2_start)
{
    Nearest nb = {d2_start, -1, 0x7fffffff};
    int32_t stack[RT_STACK_DEPTH];
    float reach[RT_STACK_DEPTH];
    int sp = 0;
    int32_t node = b.n_tris > 1 ? 0 : ~0;
    // bounded by the number of nodes; the guard stops only a corrupt structure
    for (uint32_t guard = 0; guard < (1u << 26); ++guard) {
        if (node >= 0) {
            float v[8], u[8];
            rtdev::load_node(b.nodes, node, v, u);
            const float d0 = box_d2(v[0], v[1], v[2], v[3], u[0], u[1], p), d1 = box_d2(v[4], v[5], v[6], v[7], u[2], u[3], p);
            const int32_t c0 = __float_as_int(u[4]), c1 = __float_as_int(u[5]);
            const bool in0 = d0 <= nb.d2, in1 = d1 <= nb.d2;
            if (in0 && in1) {
                if (sp < RT_STACK_DEPTH) {
                    stack[sp] = d1 < d0 ? c0 : c1;
                    reach[sp++] = fmaxf(d0, d1);
                }
                node = d1 < d0 ? c1 : c0;
                continue;
            }
            if (in0 || in1) {
                node = in0 ? c0 : c1;
                continue;
            }
        } else {
            consider_rn(nb, p, b.tris, ~node, b.brute_sum);
        }
        bool more = false;
        while (sp > 0 && !more) {
            --sp;
            more = reach[sp] <= nb.d2;
        }
        if (!more) break;
        node = stack[sp];
    }
    return nb;
}

__global__ void __launch_bounds__(kBakeBlock) k_bake_threads(const BakeArgs b, const ThreadPass tp)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t step = tp.sub > 0 ? tp.sub : 1;
    const int64_t mx = (b.n[0] - 1) / step + 1, my = (b.n[1] - 1) / step + 1, mz = (b.n[2] - 1) / step + 1;
    if (t >= mx * my * mz) return;
    const int32_t ii[3] = {(int32_t)(t % mx) * step, (int32_t)((t / mx) % my) * step, (int32_t)(t / (mx * my)) * step};
    const int64_t i = sample_index(b, ii);
    if (tp.keep) {
        const int32_t x = ii[0] + tp.shift[0], y = ii[1] + tp.shift[1], z = ii[2] + tp.shift[2];
        if (x >= 0 && x < b.n[0] && y >= 0 && y < b.n[1] && z >= 0 && z < b.n[2]) {
            const int64_t src = x + (int64_t)b.n[0] * (y + (int64_t)b.n[1] * z);
            if (b.f16) reinterpret_cast<__half*>(b.grid)[i] = reinterpret_cast<const __half*>(tp.keep)[src];
            else reinterpret_cast<float*>(b.grid)[i] = reinterpret_cast<const float*>(tp.keep)[src];
            return;
        }
    }
    float bound;
    if (tp.own > 0) {
        // the nearest sample of the first pass, whose values stand in this grid
        int32_t src[3];
        float d2 = 0.f;
        bool self = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int32_t most = (b.n[a] - 1) / tp.own;
            const int32_t j = min((ii[a] + tp.own / 2) / tp.own, most);
            src[a] = j * tp.own;
            const float gap = (float)(ii[a] - src[a]) * b.h[a];
            d2 += gap * gap;
            self = self && src[a] == ii[a];
        }
        if (self) return;
        bound = (fabsf(load_value(b.grid, b.f16, sample_index(b, src))) + sqrtf(d2)) * 1.002f + 1e-6f;
    } else {
        bound = distance_bound(b, ii);
    }
    const float3 p = sample_pos(b, ii);
    Nearest nb = nearest_triangle(b, p, bound * bound);
    if (nb.k < 0 && !isinf(bound)) nb = nearest_triangle(b, p, __int_as_float(0x7f800000));  // a bound that held no triangle
    store(b, i, signed_distance_rn(p, nb, b.tris, b.pn));
}

// rolling update: sample i takes the value of sample i + shift of `keep` (the
// level before the move) wherever that lies inside the level
__global__ void k_roll(const void* keep, void* grid, int32_t f16, int32_t n, int3 shift)
{
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t j = (int32_t)blockIdx.y, k = (int32_t)blockIdx.z;
    const int32_t x = i + shift.x, y = j + shift.y, z = k + shift.z;
    if (i >= n || x < 0 || x >= n || y < 0 || y >= n || z < 0 || z >= n) return;
    const int64_t dst = i + (int64_t)n * (j + (int64_t)n * k), src = x + (int64_t)n * (y + (int64_t)n * z);
    if (f16) reinterpret_cast<__half*>(grid)[dst] = reinterpret_cast<const __half*>(keep)[src];
    else reinterpret_cast<float*>(grid)[dst] = reinterpret_cast<const float*>(keep)[src];
}

// The copies of a grid that the march reads (layouts: rt_internal.cuh), written in
// one pass: cell entries for j < ny-1, k < nz-1, and (pairs non-null) x-pairs for
// i < nx-1.  A thread takes the samples of kCopyRows successive rows at one i; a block
// takes a part of long rows, or short rows side by side.  us with one, two, four and
// eight rows a thread: 256^3 float32 123, 97, 90, 97; 5 x 200^3 float16 326, 244, 193,
// 175 (blocks of one row of a thread each: 109 and 290, and 277 for 2 x 700 x 700
// samples, now 10).  Bound by the bytes written: 256^3 float32 (67 MB read, 268 + 134 MB
// written; 69 us at the copy bandwidth).
constexpr int kCopyBlock = 128;
constexpr int kCopyRows = 4;

// how a block's threads lie over rows of nx samples: long rows are cut into equal
// parts of whole warps
struct CopyShape {
    int32_t width, rows, chunks;  // threads beside one another in a row, rows side by side, parts of a row
};
static CopyShape copy_shape(int32_t nx)
{
    CopyShape c;
    c.chunks = (nx + kCopyBlock - 1) / kCopyBlock;
    const int32_t part = (nx + c.chunks - 1) / c.chunks;
    if (part > 32) {
        c.width = (part + 31) / 32 * 32;
    } else {
        c.width = 2;
        while (c.width < part) c.width *= 2;
    }
    c.rows = kCopyBlock / c.width;
    return c;
}

template <class V2>
struct __align__(2 * sizeof(V2)) Quad {
    V2 a, b;
};
__device__ __forceinline__ Quad<__half2> quad(__half a, __half b, __half c, __half d)
{
    return {__halves2half2(a, b), __halves2half2(c, d)};
}
__device__ __forceinline__ Quad<float2> quad(float a, float b, float c, float d) { return {make_float2(a, b), make_float2(c, d)}; }

template <class T, class V2, class V4>
__global__ void __launch_bounds__(kCopyBlock) k_copies(const T* __restrict__ grid, int32_t nx, int32_t ny, int32_t nz,
                                                       CopyShape shape, int64_t samples, int64_t entries, int shift,
                                                       V4* __restrict__ cells, V2* __restrict__ pairs)
{
    static_assert(sizeof(V4) == sizeof(Quad<V2>), "one entry is two pairs");
    const uint32_t chunks = (uint32_t)shape.chunks, per = (uint32_t)shape.rows * kCopyRows;
    const uint64_t rows = (uint64_t)ny * (uint64_t)nz, total = chunks * ((rows + per - 1) / per);
    const bool wide = ((rows + per) | total) >> 32 != 0;  // (32-bit divisions wherever they suffice)
    const uint32_t mine = threadIdx.x / (uint32_t)shape.width, lane = threadIdx.x - mine * (uint32_t)shape.width;
    for (uint64_t at = blockIdx.x; at < total; at += gridDim.x) {
        const uint64_t group = wide ? at / chunks : (uint32_t)at / chunks;
        const uint64_t row0 = group * per + mine * kCopyRows;
        const int32_t i = (int32_t)((at - group * chunks) * (uint32_t)shape.width + lane);
        if (i >= nx || row0 >= rows) continue;
        int32_t k = (int32_t)(wide ? row0 / (uint32_t)ny : (uint32_t)row0 / (uint32_t)ny);
        int32_t j = (int32_t)(row0 - (uint64_t)k * (uint32_t)ny);
#pragma unroll
        for (int u = 0; u < kCopyRows; ++u) {
            const int64_t row = (int64_t)row0 + u;
            if ((uint64_t)row >= rows) break;
            const T* g = grid + blockIdx.y * samples + i + (int64_t)nx * row;
            const T v = g[0];
            if (pairs && i + 1 < nx) {
                const Quad<V2> q = quad(v, g[1], v, v);
                pairs[i + (int64_t)(nx - 1) * row] = q.a;
            }
            if (j + 1 < ny && k + 1 < nz) {
                const Quad<V2> q = quad(v, g[nx], g[(int64_t)nx * ny], g[(int64_t)nx * ny + nx]);
                const int64_t e = (blockIdx.y * entries + i + (int64_t)nx * (row - k)) << shift;  // (rtdev::cell_slot(i, j, k))
                cells[e] = *reinterpret_cast<const V4*>(&q);
                if (shift && i > 0) cells[e - 1] = *reinterpret_cast<const V4*>(&q);
            }
            if (++j == ny) {
                j = 0;
                ++k;
            }
        }
    }
}

// `levels` grids one after another from `grid` (pairs only for one)
rt_status launch_copies(const void* grid, int32_t dtype, const int32_t n[3], int levels, int shift, void* cells,
                        void* pairs, cudaStream_t s)
{
    const CopyShape shape = copy_shape(n[0]);
    const int block = shape.width * shape.rows;
    const int64_t per = shape.rows * kCopyRows, total = shape.chunks * (((int64_t)n[1] * n[2] + per - 1) / per);
    const dim3 blocks((unsigned)(total < 0x7fffffffLL ? total : 0x7fffffffLL), (unsigned)levels);
    const int64_t samples = (int64_t)n[0] * n[1] * n[2], entries = rtdev::cell_count(n[0], n[1], n[2]);
    if (dtype == RT_GRID_F16)
        k_copies<<<blocks, block, 0, s>>>(static_cast<const __half*>(grid), n[0], n[1], n[2], shape, samples, entries, shift,
                                          static_cast<uint2*>(cells), static_cast<__half2*>(pairs));
    else
        k_copies<<<blocks, block, 0, s>>>(static_cast<const float*>(grid), n[0], n[1], n[2], shape, samples, entries, shift,
                                          static_cast<float4*>(cells), static_cast<float2*>(pairs));
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

}  // namespace

// cell copies of levels first .. first + count - 1 of a cascade
rt_status rt_launch_cascade_cells(const rt_sdf* sdf, int first, int count, cudaStream_t s)
{
    const int64_t n = sdf->n[0], esz = sdf->dtype == RT_GRID_F16 ? 2 : 4;
    const void* grid = static_cast<const char*>(sdf->grid) + first * n * n * n * esz;
    void* cells = static_cast<char*>(sdf->cells) + first * rtdev::cell_count((int)n, (int)n, (int)n) * 4 * esz;
    return launch_copies(grid, sdf->dtype, sdf->n, count, 0, cells, nullptr, s);
}

// A call has written the handle's copies
rt_status rt_copies_written(rt_sdf* sdf, cudaStream_t s)
{
    ++sdf->version;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    RT_CUDA_TRY(cudaStreamIsCapturing(s, &capture));
    if (capture != cudaStreamCaptureStatusNone) sdf->replayed = true;
    return RT_OK;
}

// A handle's copies become visible to its traces together, and only once the
// launch that fills them is enqueued: a handle whose prepare failed is as before it.
rt_status rt_launch_prepare(rt_sdf* sdf, cudaStream_t s)
{
    const int64_t esz = sdf->dtype == RT_GRID_F16 ? 2 : 4;
    const int levels = sdf->levels > 0 ? sdf->levels : 1;
    const int64_t entries = rtdev::cell_count(sdf->n[0], sdf->n[1], sdf->n[2]);
    const int shift = sdf->levels > 0 ? 0 : rtdev::cell_shift(entries, sdf->dtype == RT_GRID_F16);
    const size_t pairs_bytes = sdf->levels > 0 ? 0 : (size_t)(sdf->n[0] - 1) * sdf->n[1] * sdf->n[2] * 2 * esz;
    void *cells = sdf->cells, *pairs = sdf->pairs;
    cudaError_t e = cudaSuccess;
    if (!cells) e = cudaMalloc(&cells, (size_t)levels * (size_t)(entries << shift) * 4 * esz);
    if (e == cudaSuccess && !pairs && pairs_bytes) e = cudaMalloc(&pairs, pairs_bytes);
    rt_status st = e == cudaSuccess ? launch_copies(sdf->grid, sdf->dtype, sdf->n, levels, shift, cells, pairs, s)
                                    : rt_cuda_fail(e, "allocating the copies of the grid");
    if (st != RT_OK) {
        if (cells && !sdf->cells) cudaFree(cells);
        if (pairs && !sdf->pairs) cudaFree(pairs);
        return st;
    }
    sdf->cells = cells;
    sdf->pairs = pairs;
    return rt_copies_written(sdf, s);
}

constexpr int kSubStride = 4;  // first-pass sub-lattice of a bake without a source

// log2 of a brick's samples.  Bricks of 32 samples (4 x 4 x 2) do the least work;
// bricks of one sample finish soonest.  A launch with few samples lasts as long as
// its slowest brick (one near the centre of a round object), so the fewer the
// samples the smaller the bricks: one sample up to 32,768, eight up to 2^19.  ms: a
// 5 x 32^3 cascade of the frame scene (32,768 samples a level) 0.90 with one, 1.31
// with eight; 41^3 to 64^3 grids 0.42-0.50 with eight, 0.92-1.0 with 32; 97^3
// samples, 1,213,548 triangles 2.0 with eight, 2.1 with 32; 256^3 samples 18.0 with
// eight, 11.2 with 32.
// With few triangles no brick is slow, and the number of bricks counts: one sample
// up to 6,144 and, where the search starts from a value and not from a triangle,
// eight up to 2^17.  us at 10,300 triangles (eight spheres), the limits above |
// these: 32^3 113 | 83, 5 x 32^3 401 | 280, moves of 5 x 64^3 by 1 and 40 samples 113
// | 106 and 476 | 463, of 5 x 128^3 by 10 542 | 395.  At 20,540 triangles moves of 5
// x 32^3 by 10 and of 5 x 64^3 by 40 were slower with them (250 | 283, 645 | 716).
constexpr int64_t kFewTriangles = 16384;
static int brick_log2(const BakeArgs& b, int64_t samples)
{
    const bool few = b.n_tris <= kFewTriangles;
    if (samples <= (few ? 6144 : 32768)) return 0;
    return samples <= (few && b.bsrc ? 131072 : 524288) ? 3 : 5;
}

// cut the box into bricks of 2^lg samples, as cubic as the box allows
static void set_bricks(PacketGrid& pg, PacketBox& bx, int lg)
{
    int left = lg;
    for (int c = 0; c < 3; ++c) bx.shift[c] = 0;
    while (left > 0) {  // x, y, z in turn, an axis only while the box is longer than its edge
        const int before = left;
        for (int c = 0; c < 3 && left > 0; ++c)
            if ((1 << bx.shift[c]) < bx.dim[c]) {
                ++bx.shift[c];
                --left;
            }
        if (left == before) {  // a box smaller than the brick
            bx.shift[0] += left;
            left = 0;
        }
    }
    bx.first = pg.packets;
    int64_t bricks = 1;
    for (int c = 0; c < 3; ++c) bricks *= (bx.dim[c] + (1 << bx.shift[c]) - 1) >> bx.shift[c];
    pg.packets += bricks;
}

// whole grid, or every `sub`-th sample of it
static PacketGrid whole_grid(const BakeArgs& b, int sub)
{
    PacketGrid pg;
    memset(&pg, 0, sizeof(pg));
    pg.boxes = 1;
    pg.sub = sub;
    int64_t samples = 1;
    for (int a = 0; a < 3; ++a) {
        pg.box[0].dim[a] = (b.n[a] - 1) / sub + 1;
        samples *= pg.box[0].dim[a];
    }
    pg.brick_log2 = brick_log2(b, samples);
    set_bricks(pg, pg.box[0], pg.brick_log2);
    return pg;
}

// the samples of an n^3 level that a move by `shift` samples brings in: an x slab,
// the y slab of the rest, the z slab of that rest
static PacketGrid new_slabs(const BakeArgs& b, const int32_t shift[3])
{
    const int32_t n = b.n[0];
    PacketGrid pg;
    memset(&pg, 0, sizeof(pg));
    pg.sub = 1;
    int32_t lo[3] = {0, 0, 0}, dim[3] = {n, n, n};  // what is left
    for (int a = 0; a < 3; ++a) {
        const int32_t thick = shift[a] < 0 ? -shift[a] : shift[a];
        if (thick == 0) continue;
        PacketBox& bx = pg.box[pg.boxes++];
        for (int c = 0; c < 3; ++c) {
            bx.lo[c] = lo[c];
            bx.dim[c] = dim[c];
        }
        bx.dim[a] = thick;
        bx.lo[a] = shift[a] > 0 ? n - thick : 0;
        lo[a] = shift[a] > 0 ? 0 : thick;
        dim[a] -= thick;
    }
    pg.brick_log2 = brick_log2(b, (int64_t)n * n * n - (int64_t)dim[0] * dim[1] * dim[2]);
    for (int k = 0; k < pg.boxes; ++k) set_bricks(pg, pg.box[k], pg.brick_log2);
    return pg;
}

// nearest-triangle search of the samples of pg
static rt_status launch_packets(const BakeArgs& b, const PacketGrid& pg, cudaStream_t s)
{
    if (pg.packets == 0) return RT_OK;
    const int64_t blocks = (pg.packets + kBrickWarps - 1) / kBrickWarps;
    if (blocks > 0x7fffffffLL) return rt_fail(RT_ERR_INVALID_ARG, "grid too large for one launch");
    switch (pg.brick_log2) {
    case 0: k_bake_bricks<0><<<(unsigned)blocks, 32 * kBrickWarps, 0, s>>>(b, pg); break;
    case 3: k_bake_bricks<3><<<(unsigned)blocks, 32 * kBrickWarps, 0, s>>>(b, pg); break;
    default: k_bake_bricks<5><<<(unsigned)blocks, 32 * kBrickWarps, 0, s>>>(b, pg); break;
    }
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

static rt_status launch_threads(const BakeArgs& b, const ThreadPass& tp, cudaStream_t s)
{
    int64_t samples = 1;
    for (int a = 0; a < 3; ++a) samples *= (b.n[a] - 1) / (tp.sub > 0 ? tp.sub : 1) + 1;
    const int64_t blocks = (samples + kBakeBlock - 1) / kBakeBlock;
    if (blocks > 0x7fffffffLL) return rt_fail(RT_ERR_INVALID_ARG, "grid too large for one launch");
    k_bake_threads<<<(unsigned)blocks, kBakeBlock, 0, s>>>(b, tp);
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

// the stride-4 sub-lattice first, then every other sample within the bound of its
// nearest sub-lattice sample
static rt_status launch_threads_two_pass(const BakeArgs& b, cudaStream_t s)
{
    ThreadPass tp = {};
    tp.sub = kSubStride;
    const rt_status st = launch_threads(b, tp, s);
    if (st != RT_OK) return st;
    tp.sub = 0;
    tp.own = kSubStride;
    return launch_threads(b, tp, s);
}

// device scratch of one bake, returned in stream order
struct BakeScratch {
    void* p = nullptr;
    cudaStream_t s;
    explicit BakeScratch(cudaStream_t st) : s(st) {}
    ~BakeScratch() { if (p) cudaFreeAsync(p, s); }
    rt_status take(size_t bytes) { return rt_scratch_alloc(&p, bytes, s); }
};

static size_t sub_sites_bytes(const int32_t n[3])
{
    size_t c = sizeof(int32_t);
    for (int a = 0; a < 3; ++a) c *= (size_t)((n[a] - 1) / kSubStride + 1);
    return (c + 255) & ~(size_t)255;
}

// BVH bake without a source: the nearest triangles of the stride-4 sub-lattice
// first, then every sample from its nearest sub-lattice sample's triangle.
// 256^3 samples, 2,050,412 triangles (the frame scene): 11.0 ms, the first pass
// 0.7 of them (31.3 ms with one traversal per thread and the source's value as
// the bound).
static rt_status launch_two_pass(BakeArgs b, int32_t* sub_sites, cudaStream_t s)
{
    void* const grid = b.grid;
    int32_t* const sdst = b.sdst;
    b.grid = nullptr;
    b.sdst = sub_sites;
    b.ssrc = nullptr;
    b.bsrc = nullptr;
    const PacketGrid coarse = whole_grid(b, kSubStride);
    rt_status st = launch_packets(b, coarse, s);
    if (st != RT_OK) return st;
    b.grid = grid;
    b.sdst = sdst;
    b.ssrc = sub_sites;
    b.bratio = kSubStride;
    b.src_relative = 1;
    for (int a = 0; a < 3; ++a) {
        b.bilo[a] = 0;
        b.bdim[a] = coarse.box[0].dim[a];
    }
    return launch_packets(b, whole_grid(b, 1), s);
}

static rt_status launch_brute(const BakeArgs& b, cudaStream_t s)
{
    const int64_t blocks = (b.count + kBakeBlock - 1) / kBakeBlock;
    if (blocks > 0x7fffffffLL) return rt_fail(RT_ERR_INVALID_ARG, "grid too large for one launch");
    k_bake_brute<<<(unsigned)blocks, kBakeBlock, 0, s>>>(b);
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

// RT_BAKE_AUTO gives the values of the brute force kernel up to 2^34 pairs of a
// sample and a triangle, and the BVH search's beyond.  The kernel itself is
// taken only for a few triangles: a pair costs it 2.8 ps, a sample costs the
// search 0.7 to 1.5 ns (123,000 samples: 344 triangles 0.12 and 0.10 ms, 11,748
// triangles 4.1 and 0.18 ms), and the search gives the same values.
constexpr int64_t kBruteMost = 256;
static bool brute_values(const BakeArgs& b, int32_t method)
{
    return method == RT_BAKE_BRUTE || (method == RT_BAKE_AUTO && (double)b.count * (double)b.n_tris <= 17179869184.0);
}
static bool pick_brute(BakeArgs& b, int32_t method)
{
    b.brute_sum = brute_values(b, method);
    return method == RT_BAKE_BRUTE || (b.brute_sum && b.n_tris <= kBruteMost);
}

// Up to 512 triangles, 1,024 on a cascade's levels and over 2^22 samples, a thread
// searches for a sample.
// us, threads | bricks, 24 triangles: 256^3 762 | 1,319, 5 x 64^3 141 | 399, its moves
// by 1 and 40 samples 74 | 87 and 143 | 190; 252 triangles: 256^3 1,441 | 1,734, 5 x
// 64^3 244 | 456, moves 86 | 96 and 214 | 242; 700 triangles: 32^3 201 | 66, 64^3 160 |
// 130, 256^3 1,384 | 1,584, 5 x 64^3 293 | 442, moves 87 | 92 and 210 | 247; 1,340
// triangles: 64^3 253 | 127, 5 x 64^3 556 | 494, moves 107 | 104 and 334 | 286.
static bool few_triangles(const BakeArgs& b, bool level) { return b.n_tris <= (level || b.count > (1 << 22) ? 1024 : 512); }

static BakeArgs bake_args(const rt_scene* sc, const rt_sdf* sdf)
{
    BakeArgs b;
    memset(&b, 0, sizeof(b));
    b.nodes = sc->nodes;
    b.tris = sc->tris;
    b.pn = sc->pn;
    b.slot = sc->slot;
    b.n_tris = sc->n_tris;
    b.f16 = sdf->dtype == RT_GRID_F16;
    b.bratio = 1;
    b.count = 1;
    for (int a = 0; a < 3; ++a) {
        b.n[a] = sdf->n[a];
        b.bdim[a] = sdf->n[a];
        b.count *= sdf->n[a];
    }
    return b;
}

static BakeArgs level_args(const rt_scene* sc, const rt_sdf* sdf, int k)
{
    BakeArgs b = bake_args(sc, sdf);
    const int64_t esz = sdf->dtype == RT_GRID_F16 ? 2 : 4;
    b.grid = static_cast<char*>(const_cast<void*>(sdf->grid)) + k * b.count * esz;
    b.lattice = 1;
    b.h[0] = b.h[1] = b.h[2] = ldexpf(sdf->h0, k);
    for (int a = 0; a < 3; ++a) b.ilo[a] = sdf->ilo[k][a];
    return b;
}

// the source of level k's samples: the next coarser level
static void coarser_source(BakeArgs& b, const rt_sdf* sdf, int k)
{
    b.bratio = 2;
    for (int a = 0; a < 3; ++a) b.bilo[a] = sdf->ilo[k + 1][a];
}

static void coarser_values(BakeArgs& b, const rt_sdf* sdf, int k)
{
    b.bsrc = static_cast<const char*>(sdf->grid) + (k + 1) * b.count * (b.f16 ? 2 : 4);
    coarser_source(b, sdf, k);
}

static rt_status whole_level_by_threads(BakeArgs b, const rt_sdf* sdf, int k, cudaStream_t s)
{
    if (k + 1 >= sdf->levels) return launch_threads_two_pass(b, s);
    coarser_values(b, sdf, k);
    return launch_threads(b, ThreadPass{}, s);
}

// Bake of cascade level k of a moved cascade: the kept samples from `keep` and
// the new slabs (keep non-null), or the whole level, bounded by the values of
// the next coarser level.  New samples get the values that the method of the
// cascade's last bake gives them, so that a rolled level equals a fresh one.
rt_status rt_launch_cascade_bake(const rt_scene* sc, const rt_sdf* sdf, int k, const void* keep, const int32_t shift[3],
                                 cudaStream_t s)
{
    BakeArgs b = level_args(sc, sdf, k);
    b.brute_sum = brute_values(b, sdf->bake_method);
    const int32_t n = sdf->n[0];
    const bool threads = few_triangles(b, true);
    if (keep) {
        if (threads) {
            b.bsrc = keep;
            ThreadPass tp = {};
            tp.keep = keep;
            for (int a = 0; a < 3; ++a) {
                tp.shift[a] = shift[a];
                b.bilo[a] = sdf->ilo[k][a] - shift[a];
            }
            return launch_threads(b, tp, s);
        }
        const unsigned threads = n >= 128 ? 128 : (n >= 64 ? 64 : 32);
        k_roll<<<dim3((n + threads - 1) / threads, n, n), threads, 0, s>>>(keep, b.grid, b.f16, n,
                                                                           make_int3(shift[0], shift[1], shift[2]));
        RT_CUDA_TRY(cudaGetLastError());
        // new samples are bounded by the nearest kept sample
        b.bsrc = keep;
        for (int a = 0; a < 3; ++a) b.bilo[a] = sdf->ilo[k][a] - shift[a];
        return launch_packets(b, new_slabs(b, shift), s);
    }
    if (threads) return whole_level_by_threads(b, sdf, k, s);
    if (k + 1 < sdf->levels) {
        coarser_values(b, sdf, k);
        return launch_packets(b, whole_grid(b, 1), s);
    }
    BakeScratch scratch(s);
    const rt_status st = scratch.take(sub_sites_bytes(b.n));
    if (st == RT_ERR_OOM) return whole_level_by_threads(b, sdf, k, s);
    if (st != RT_OK) return st;
    return launch_two_pass(b, static_cast<int32_t*>(scratch.p), s);
}

rt_status rt_launch_bake(const rt_scene* sc, const rt_sdf* sdf, int32_t method, cudaStream_t s)
{
    BakeScratch scratch(s);
    if (sdf->levels == 0) {
        BakeArgs b = bake_args(sc, sdf);
        b.grid = const_cast<void*>(sdf->grid);
        for (int k = 0; k < 3; ++k) {
            b.lo[k] = sdf->lo[k];
            b.h[k] = sdf->h[k];
        }
        if (pick_brute(b, method)) return launch_brute(b, s);
        if (few_triangles(b, false)) return launch_threads_two_pass(b, s);
        rt_status st = scratch.take(sub_sites_bytes(b.n));
        if (st == RT_ERR_OOM) return launch_threads_two_pass(b, s);
        if (st != RT_OK) return st;
        return launch_two_pass(b, static_cast<int32_t*>(scratch.p), s);
    }
    BakeArgs first = level_args(sc, sdf, 0);
    if (pick_brute(first, method)) {
        for (int k = sdf->levels - 1; k >= 0; --k) {
            rt_status st = launch_brute(level_args(sc, sdf, k), s);
            if (st != RT_OK) return st;
        }
        return RT_OK;
    }
    auto by_threads = [&] {
        // coarsest first: each level bounds the next finer one
        for (int k = sdf->levels - 1; k >= 0; --k) {
            BakeArgs b = level_args(sc, sdf, k);
            b.brute_sum = first.brute_sum;
            const rt_status st = whole_level_by_threads(b, sdf, k, s);
            if (st != RT_OK) return st;
        }
        return RT_OK;
    };
    if (few_triangles(first, true)) return by_threads();
    // coarsest first: each level starts from the nearest triangles of the next
    // coarser one, kept for two levels at a time
    const size_t sub_bytes = sub_sites_bytes(sdf->n);
    const size_t level_bytes = ((size_t)sdf->n[0] * sdf->n[1] * sdf->n[2] * sizeof(int32_t) + 255) & ~(size_t)255;
    rt_status st = scratch.take(sub_bytes + (sdf->levels > 1 ? 2 * level_bytes : 0));
    if (st == RT_ERR_OOM) return by_threads();
    if (st != RT_OK) return st;
    char* base = static_cast<char*>(scratch.p);
    for (int k = sdf->levels - 1; k >= 0; --k) {
        BakeArgs b = level_args(sc, sdf, k);
        b.brute_sum = first.brute_sum;
        int32_t* sites[2] = {reinterpret_cast<int32_t*>(base + sub_bytes),
                             reinterpret_cast<int32_t*>(base + sub_bytes + level_bytes)};
        b.sdst = k > 0 ? sites[k & 1] : nullptr;
        if (k == sdf->levels - 1) {
            st = launch_two_pass(b, reinterpret_cast<int32_t*>(base), s);
        } else {
            b.ssrc = sites[(k + 1) & 1];
            coarser_source(b, sdf, k);
            st = launch_packets(b, whole_grid(b, 1), s);
        }
        if (st != RT_OK) return st;
    }
    return RT_OK;
}
