// Internal data layout and device helpers of the combined ray query library.
//
// HBM layout (built once per scene / per grid):
//   nodes  : n_tris-1 internal BVH nodes, 64 B each, read as two 32-byte loads:
//              a = (c0.lo.x, c0.hi.x, c0.lo.y, c0.hi.y)
//              b = (c1.lo.x, c1.hi.x, c1.lo.y, c1.hi.y)
//              c = (c0.lo.z, c0.hi.z, c1.lo.z, c1.hi.z)
//              d = (child0, child1, -, -)   child >= 0: internal node,
//                                           child < 0 : leaf = triangle ~child
//   tris   : 48 B per triangle in leaf (Morton) order: v0.xyz|prim, v1.xyz|-, v2.xyz|-
//   wnodes : the same tree collapsed to 8-wide nodes of 80 B (five 16-byte vectors):
//              a  = (origin x, y, z, bits: exponent x | y << 8 | z << 16 | internal mask << 24)
//              b  = (first child node, first triangle, meta slots 0-3, meta slots 4-7)
//              q0 = (qlo.x[0..7], qlo.y[0..7]), q1 = (qlo.z[0..7], qhi.x[0..7]),
//              q2 = (qhi.y[0..7], qhi.z[0..7])   8-bit child bounds, box = origin + q * 2^(e-127)
//            meta byte: 0 empty, else leaf (count << 5 | first triangle offset) or, with the
//            internal-mask bit set, an inner child at first child + (inner children in lower slots)
//   wtris  : 48 B per triangle in wide-leaf order (each node's leaf triangles contiguous)
//   pn     : 112 B per triangle in leaf order: face normal, 3 edge and 3 vertex
//            pseudonormals (float4 each), read only by the distance bake; w of the
//            face normal: 4e-5 of the squared longest edge, the bake's margin for its
//            plane test (inf: a badly shaped triangle, never decided by its plane)
//   slot   : 4 B per triangle: input index -> leaf-order position (field build)
//   grid   : caller memory, dense n0*n1*n2 float32 or float16, x fastest
//   cells  : optional library copy of the grid with the four values of every cell
//            face across x stored together (16 B float32 / 8 B float16 per entry,
//            x fastest), so one march step is two adjacent vector loads instead
//            of eight scalar ones; a large float32 grid's copy holds both faces of
//            every cell (32 B); identical values, identical arithmetic
//   pairs  : optional library copy with the two x-neighbours (i, i+1) of every
//            sample stored together (8 B float32 / 4 B float16, (n0-1) x n1 x n2,
//            x fastest): a march step is four small loads from a copy twice the
//            grid's size, small enough to stay in L2 where the cell copy is not
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "../../include/rt_api.h"

#define RT_STACK_DEPTH 64

struct __align__(32) BNode {
    float4 a, b, c;
    int4 d;
};

struct __align__(16) WNode {
    float4 a;
    uint4 b, q0, q1, q2;
};

#define RT_WSTACK_DEPTH 32

struct rt_scene {
    int device;
    int64_t n_tris, n_verts, n_nodes;
    int32_t max_depth;
    BNode* nodes;
    float4* tris;   // 3 per triangle
    float4* pn;     // 7 per triangle
    int32_t* slot;  // input triangle index -> position in leaf order
    WNode* wnodes;  // null when the wide tree is not available
    float4* wtris;  // 3 per triangle
    int64_t n_wnodes;
    int32_t wide_depth;
    float lo[3], hi[3];
    int64_t bytes;
    void* block;    // the one allocation that holds all of the above
};

struct rt_sdf {
    const void* grid;
    int32_t dtype;
    float lo[3], hi[3], h[3], ih[3];  // one grid; on a cascade: the coarsest level's box
    int32_t n[3];
    void* cells;        // library-owned cell copy (null until rt_sdf_prepare)
    void* pairs;        // library-owned x-pair copy (null until rt_sdf_prepare)
    uint64_t version;   // how often the copies have been written (rt_sdf_version)
    bool replayed;      // a graph may write them again without this handle knowing
    int device;
    // cascade (levels > 0): level k holds n^3 samples at (ilo[k] + i) * h0 * 2^k,
    // stored at grid + k * n^3, its cells at cells + k * n (n-1)^2 entries
    int32_t levels;
    float h0;
    int32_t ilo[RT_MAX_LEVELS][3];
    void* scratch;      // one level, for rt_cascade_recenter
    int64_t scratch_bytes;
    int32_t bake_method;  // method of the last rt_sdf_bake (RT_BAKE_JFA: sites kept); a rolling update follows it
    int32_t* sites;       // finished site of every sample after a field build (RT_BAKE_JFA): the
                          // seeds of finer levels when a rolling update rebuilds them
    int64_t sites_count;
};

// geometry of cascade level k as the queries see it (float, rounded once each)
struct CascLevel {
    float lo[3], hi[3];
    float ih, h, eps_hit, eps_min;
};

// Query order (rt_tuning.order_bits): each window of consecutive queries
// stably sorted by the cell of a 2^bits lattice over the box
// lo + [0, 2^bits / scale] that holds the query's origin (rt_order.cu).
// bits = 0, or fewer than kOrderMin queries: no ordering.
struct OrderBox {
    float lo[3], scale[3];
    int32_t bits;
};
constexpr int32_t kOrderMaxBits = 5;
constexpr int64_t kOrderMin = 64;

// The query order is applied where it was measured to pay: to queries whose
// first sub-interval is the near triangle one (closest hit, a split with
// 0 < m_near < inf).  Triangles-only, field-only and any-hit calls start with
// a kernel whose time the order does not change, and pay only its cost.
inline bool rt_order_applies(const rt_split_params& p)
{
    return (p.mode == RT_MODE_SPLIT1 || p.mode == RT_MODE_SPLIT2) && p.any_hit == 0 && p.m_near > 0.f &&
           !isinf(p.m_near);
}

// Everything one trace kernel needs, passed by value.
struct TraceArgs {
    const BNode* nodes;
    const float4* tris;
    const WNode* wnodes;  // null: binary traversal
    const float4* wtris;
    int32_t root;        // 0 (internal), ~0 (single leaf) or INT32_MIN (no triangles)
    const void* grid;    // null: no field
    const void* cells;   // null: read the plain grid (or the pairs)
    const void* pairs;   // null: no x-pair copy
    int32_t grid_f16;
    float glo[3], ghi[3], gih[3];
    int32_t gn[3];
    float hsplit, eps_hit, eps_min;
    int32_t max_steps;
    int32_t mode, any_hit, refine_root;
    float m_near, m_far;
    int32_t levels;        // 0: one grid; > 0: a cascade read through its cell copy
    int64_t level_cells;   // entries of the cell copy per cascade level
    int64_t cell_row;      // one grid: bytes from a row of the cell copy to the next,
    int32_t cell_step;     // and from a cell to its neighbour in x
    CascLevel lv[RT_MAX_LEVELS];
    const float4* rays;
    rt_hit* hits;
    int64_t n;
    unsigned long long* counters;
    OrderBox ob;             // ob.bits = 0: queries in input order
    const int32_t* qorder;   // null: input order; else the first kernel's slot i traces query qorder[i]
};

// ---------------------------------------------------------------------------
// host-side error reporting (rt_api.cu)
// ---------------------------------------------------------------------------
rt_status rt_fail(rt_status s, const char* fmt, ...);
rt_status rt_cuda_fail(cudaError_t e, const char* what);
#define RT_CUDA_TRY(expr)                                         \
    do {                                                          \
        cudaError_t _e = (expr);                                  \
        if (_e != cudaSuccess) return rt_cuda_fail(_e, #expr);    \
    } while (0)

const rt_tuning& rt_current_tuning();

// which grid copy the march reads under a tuning: the cell copy, the x-pair copy
// or the plain grid (a copy is used only if rt_sdf_prepare has built it)
inline void rt_apply_layout(TraceArgs& a, const rt_tuning& tu)
{
    if (a.levels > 0) {  // a cascade has only its cell copy
        a.pairs = nullptr;
        return;
    }
    if (tu.grid_layout != RT_LAYOUT_CELLS) a.cells = nullptr;
    if (tu.grid_layout != RT_LAYOUT_PAIRS) a.pairs = nullptr;
}

// launchers implemented in the .cu files
// timing: when non-null, events[k] is recorded before launch k and events[n] after
// the last; kinds[k] receives the RT_STAGE_* of launch k; *n_launches the count
// Timed parts of one call (rt_trace_combined_timed): part k ran between
// events[2k] and events[2k+1], recorded on the stream that ran it.
constexpr int kMaxTimedParts = 6;
struct StageTiming {
    cudaEvent_t events[2 * kMaxTimedParts];
    int32_t kinds[kMaxTimedParts];
    int32_t n_launches;
};

// The queries' ray arrays as one index space: query g lies in segment b, the
// last with offset[b] <= g, at rays[b] + 2 (g - offset[b]).
struct OrderRays {
    const float4* rays[RT_MAX_BATCHES];
    int64_t offset[RT_MAX_BATCHES];
    int32_t count;
};
// Scratch bytes of the query order of n queries (a multiple of 256; 0 when
// there is nothing to order).
size_t rt_order_bytes(const OrderBox& ob, int64_t n);
// Order queries 0..n-1 of a (rt_order.cu) into `scratch` (rt_order_bytes,
// 256-byte aligned); on success a.qorder points into it.  Enqueued on s.
rt_status rt_launch_order(TraceArgs& a, const OrderRays& src, void* scratch, cudaStream_t s);
// The concurrent programs (rt_trace.cu for one call, rt_batch.cu for mixed
// batches): closest-hit near triangle sub-intervals run beside the field
// sub-intervals, which start at t_1 without waiting for the near result.  The
// near stage lists its hits; afterwards k_merge_hits writes each over the
// record the later stages left (a near hit lies before t_1, so it is the
// closest, Section 2).  A near miss that raised flags lists an entry with prim
// kFlagsOnly, whose flags are ORed into the record.
constexpr int32_t kFlagsOnly = -2;
struct HitEntry {
    rt_hit* dst;  // the query's record
    uint32_t flags;
    float t, u, v;
    int32_t prim;
    int32_t pad;
};
static_assert(sizeof(HitEntry) == 32, "one 32-byte entry per hit");
// Two library streams per device for the concurrent programs: near (highest
// priority) and field (lowest), with the events that fork and join them.
// Callers hold rt_conc_mutex() from the fork to the join.
struct ConcStreams {
    cudaStream_t near = nullptr, field = nullptr;
    cudaEvent_t fork = nullptr, ordered = nullptr, near_done = nullptr, field_done = nullptr;
    bool ready = false;
};
std::mutex& rt_conc_mutex();
// set 0: calls and batches; sets 1 .. kConcSets - 1: the pieces of
// rt_trace_combined_host, which would wait for one another on shared streams
constexpr int kConcSets = 5;
rt_status rt_conc_streams(int set, ConcStreams*& out);
// k_merge_hits over the *count entries of list, on s
rt_status rt_launch_merge_hits(const HitEntry* list, const unsigned* count, int sms, cudaStream_t s);
// Resident blocks of 128 threads per SM of the two concurrent stages when the
// tuning leaves them free.  Both kernels are persistent, so their blocks must
// fit in an SM side by side (registers: near 56, 64 for the batch kernel, field
// 40, times 128 threads, at most 65,536), or the later launch waits for the
// earlier one's end.  Measured, ms a call, near + field blocks: 1080p GI on one
// grid (256^3) 2 + 10 0.578, 2 + 9 0.594, 3 + 8 0.602, 4 + 7 0.649; on a 5 x 64^3
// cascade, whose near sub-intervals are several times longer, 5 + 5 0.806, 4 + 7
// 0.813, 3 + 8 0.837, 2 + 9 0.859; a mixed frame 3 + 8 1.946, 4 + 7 1.971, 2 + 9
// 1.992, 5 + 6 2.211.
// A copy with both faces of a cell (float32 grids of 2^26 entries on), 2 + 9 | 2 + 10:
// 420^3 GI 0.790 | 0.795, short AO rays 0.379 | 0.456; 512^3 0.854 | 0.866, 0.480 | 0.486.
constexpr int kConcNearBlocks = 2, kConcFieldBlocks = 10, kConcFieldBoth = 9;
constexpr int kConcNearCascade = 4, kConcFieldCascade = 7;
constexpr int kConcNearBatch = 3, kConcFieldBatch = 8;

// Device scratch in stream order (free it with cudaFreeAsync).  Up to
// kScratchKept bytes come from a pool of the library that keeps twice as much of
// what is freed (an allocation of the device's own costs 0.1 to 0.9 ms); more comes
// from the device's default pool, which gives it back.
constexpr size_t kScratchKept = (size_t)64 << 20;
rt_status rt_scratch_alloc(void** p, size_t bytes, cudaStream_t s);

// Queries up to which RT_KERNEL_AUTO takes one thread per query: about those
// resident at once (rt_launch_trace has the figures)
constexpr int64_t kSmallCall = 131072;
constexpr int64_t kSmallCallTriangles = 65536;  // calls that trace triangles only
// For batches, whose pipeline has more launches (those that trace triangles only:
// kSmallCall).  us, pipeline | one thread per query, frame scene, 256^3, at 150,000,
// 260,000 and 520,000 queries: GI 201 | 150, 240 | 218, 280 | 282; GI and shadow 257 |
// 155, 283 | 190, 328 | 274; the four kinds of a frame 213 | 147, 250 | 190, 272 | 207.
constexpr int64_t kSmallBatch = 524288;
constexpr int kSmallBlock = 128;                // their threads per block, whatever the tuning's

// conc_set: the set of library streams a concurrent program of this call uses
rt_status rt_launch_trace(const TraceArgs& a, bool counted, cudaStream_t s, StageTiming* timing = nullptr,
                          int conc_set = 0);
// at_record: the records' t are the roots of the copy that the march reads
rt_status rt_launch_backward(const TraceArgs& a, bool at_record, const float* grad_t, float* grad_grid, cudaStream_t s);
rt_status rt_build_scene(const float* verts, int64_t nv, const int32_t* tris, int64_t nt, cudaStream_t s,
                         rt_scene* out);
rt_status rt_launch_bake(const rt_scene* sc, const rt_sdf* sdf, int32_t method, cudaStream_t s);
// Arrays that share one allocation: counted first (base null), then handed out.
struct BuildArena {
    char* base = nullptr;
    size_t at = 0, size = 0;
    template <class T>
    T* take(int64_t count)
    {
        T* p = base ? reinterpret_cast<T*>(base + at) : nullptr;
        at += ((size_t)(count > 0 ? count : 1) * sizeof(T) + 255) & ~(size_t)255;
        if (at > size) size = at;
        return p;
    }
};

// Surface-area costs of the tree (rt_treelet.cu), every rounding written out: the
// restructured tree must not depend on how a compiler contracts these sums in one
// place or another (an ulp decides between two topologies of nearly equal cost).
namespace rttree {
constexpr float kCostNode = 1.2f;  // visiting a node ...
constexpr float kCostTri = 1.0f;   // ... and testing a triangle
__device__ __forceinline__ float half_area(float4 lo, float4 hi)
{
    const float dx = __fsub_rn(hi.x, lo.x), dy = __fsub_rn(hi.y, lo.y), dz = __fsub_rn(hi.z, lo.z);
    return __fmaf_rn(dz, dx, __fmaf_rn(dx, dy, __fmul_rn(dy, dz)));
}
__device__ __forceinline__ float node_cost(float4 lo, float4 hi, float c0, float c1)
{
    return __fadd_rn(__fmaf_rn(kCostNode, half_area(lo, hi), c0), c1);
}
}  // namespace rttree

// workspaces of the restructuring and of the wide tree's collapse
struct TreeletScratch {
    int* visit;      // one per internal node
    int* count;
    int32_t* pos;    // one per leaf, as the rest
    int32_t* order2;
    int32_t* par_l2;
    float4 *llo2, *lhi2;
};
struct WideScratch {
    int2* items[2];     // (binary node, wide node) pairs of one level
    unsigned* counters;
};
constexpr int kWideCounters = 4 + 260;  // nodes, triangles, error, -; then the items of each level
rt_status rt_build_wide(rt_scene* sc, const int2* child, const int2* range, const float4* node_lo,
                        const float4* node_hi, const float4* leaf_lo, const float4* leaf_hi, float pad,
                        const WideScratch& ws, cudaStream_t s);
rt_status rt_launch_prepare(rt_sdf* sdf, cudaStream_t s);
rt_status rt_copies_written(rt_sdf* sdf, cudaStream_t s);
rt_status rt_treelet_optimise(int64_t nt, int passes, int2* child, int2* range, int32_t* par_i, int32_t* par_l,
                              int32_t* order, float4* llo, float4* lhi, float4* nlo, float4* nhi, float* cost,
                              const TreeletScratch& ws, cudaStream_t s);
rt_status rt_fill_trace_args(TraceArgs& a, const rt_scene* sc, const rt_sdf* sdf, const rt_split_params* p);
void rt_cascade_geometry(const rt_sdf* sdf, int k, float lo[3], float hi[3], float* h, float* ih);
rt_status rt_launch_cascade_bake(const rt_scene* sc, const rt_sdf* sdf, int k, const void* keep, const int32_t shift[3],
                                 cudaStream_t s);
rt_status rt_launch_cascade_cells(const rt_sdf* sdf, int first, int count, cudaStream_t s);
rt_status rt_launch_df_sites(const rt_scene* sc, const rt_sdf* sdf, int32_t stage, int32_t* d_sites, cudaStream_t s);
rt_status rt_launch_df_levels(const rt_scene* sc, const rt_sdf* sdf, const int* lv, int nl, int32_t* ids, cudaStream_t s);
