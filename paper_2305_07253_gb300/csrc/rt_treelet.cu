// Treelet restructuring of the LBVH (Karras & Aila, "Fast Parallel
// Construction of High-Quality Bounding Volume Hierarchies", HPG 2013).
//
// The Morton-code hierarchy is fast to build but its splits ignore the
// surface-area cost that decides how many nodes a ray visits.  Each pass walks
// the tree bottom-up (one thread per leaf, a counter per node: the second
// thread to arrive continues), and every node reached this way becomes the
// root of a treelet: its leaves are found by repeatedly expanding the treelet
// leaf of largest surface area, up to 7 of them, and the binary topology over
// those leaves of least surface-area cost,
//     c(S) = C_node A(S) + min over splits S = P + (S \ P) of c(P) + c(S \ P),
// is found by dynamic programming over the 127 subsets, eight lanes per treelet.
// When it is cheaper the treelet is rewired with its own internal nodes.  The
// leaves are finally renumbered in depth-first order so that every subtree's
// triangles are contiguous again (the 8-wide collapse relies on that).
#include "rt_internal.cuh"

namespace {

constexpr int kBlock = 128;             // 4 warps (32 threads a block: 2 % slower rebuild)
constexpr int kWarps = kBlock / 32;
constexpr int kTreelet = 7;             // treelet leaves
constexpr int kSubsets = 1 << kTreelet;
constexpr int kGroup = 8;               // lanes that work on one treelet
constexpr int kGroups = 32 / kGroup;    // treelets a warp works on at a time
using rttree::half_area;
using rttree::kCostNode;
using rttree::kCostTri;
constexpr int kMaxWalk = 256;
// Leaves a lane of k_treelets walks up from, one after another: a lane whose walk
// ends takes its next leaf, so that more treelets are ready at a time for the
// warp's four groups.  Rebuild, ms, with 1, 2, 4, 8, 16: 11.0, 10.5, 10.3, 10.5, 10.7.
constexpr int kLeaves = 4;

// half the surface area of the subsets that the dynamic program compares (rounded as its sums always were)
__device__ __forceinline__ float subset_half_area(float4 lo, float4 hi)
{
    const float dx = __fsub_rn(hi.x, lo.x), dy = __fsub_rn(hi.y, lo.y), dz = __fsub_rn(hi.z, lo.z);
    return __fmaf_rn(dz, dx, __fmaf_rn(dy, dz, __fmul_rn(dx, dy)));
}

struct Tree {
    int2* child;
    int32_t* par_i;     // parent of an internal node (-1 for the root)
    int32_t* par_l;     // parent of a leaf
    const float4* llo;
    const float4* lhi;
    float4* nlo;
    float4* nhi;
    float* cost;        // surface-area cost of every internal node's subtree
    int* visit;
    int64_t n_leaves;
};

// One treelet's shared memory.  Its size is 32 bytes past a multiple of 128, so
// that the four treelets of a warp start eight banks apart.
struct Workspace {
    float4 lo[kTreelet], hi[kTreelet];  // boxes of the treelet's leaves
    float4 ulo[24], uhi[24];            // unions of leaves 0-2 (entries 0-7, by subset) and of leaves 3-6 (entries 8-23)
    float copt[kSubsets];
    unsigned char part[kSubsets];
    int leaf[kTreelet + 1];             // treelet leaves (node or ~leaf references)
    int inner[kTreelet + 1];            // the treelet's internal nodes, root first
    int set[kTreelet + 1], node[kTreelet + 1], ref0[kTreelet + 1], ref1[kTreelet + 1];  // the new topology, parents first
    int pad[32];
};
static_assert(sizeof(Workspace) % 128 == 32, "treelets of a warp eight banks apart");

// the non-empty subsets of kTreelet leaves ordered by size, then by value: those
// of size k among the first n leaves are the first C(n, k) of their size
__constant__ unsigned char kBySize[kSubsets] = {
    1, 2, 4, 8, 16, 32, 64, 3, 5, 6, 9, 10, 12, 17, 18, 20, 24, 33, 34, 36, 40, 48, 65, 66, 68, 72,
    80, 96, 7, 11, 13, 14, 19, 21, 22, 25, 26, 28, 35, 37, 38, 41, 42, 44, 49, 50, 52, 56, 67, 69, 70, 73,
    74, 76, 81, 82, 84, 88, 97, 98, 100, 104, 112, 15, 23, 27, 29, 30, 39, 43, 45, 46, 51, 53, 54, 57, 58, 60,
    71, 75, 77, 78, 83, 85, 86, 89, 90, 92, 99, 101, 102, 105, 106, 108, 113, 114, 116, 120, 31, 47, 55, 59, 61, 62,
    79, 87, 91, 93, 94, 103, 107, 109, 110, 115, 117, 118, 121, 122, 124, 63, 95, 111, 119, 123, 125, 126, 127, 0,
};

__host__ __device__ constexpr int choose(int n, int k)  // C(n, k), n <= 7
{
    int c = 1;
    for (int i = 0; i < k; ++i) c = c * (n - i) / (i + 1);
    return c;
}
__host__ __device__ constexpr int size_first(int k)  // position of the first subset of size k
{
    int at = 0;
    for (int j = 1; j < k; ++j) at += choose(kTreelet, j);
    return at;
}

__device__ __forceinline__ void subset_box(const Workspace& w, int S, float4& lo, float4& hi)
{
    const float4 a = w.ulo[S & 7], b = w.ulo[8 + (S >> 3)], c = w.uhi[S & 7], d = w.uhi[8 + (S >> 3)];
    lo = make_float4(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z), 0.f);
    hi = make_float4(fmaxf(c.x, d.x), fmaxf(c.y, d.y), fmaxf(c.z, d.z), 0.f);
}

// cost of subset S from the cost of its best split
__device__ __forceinline__ float subset_cost(const Workspace& w, int S, float split)
{
    float4 lo, hi;
    subset_box(w, S, lo, hi);
    return __fmaf_rn(kCostNode, subset_half_area(lo, hi), split);
}

// Best splits of the subsets of SIZE leaves, eight lanes over the subsets of one
// treelet.  The number of splits is a constant, so the loads of several splits
// are in flight together.
template <int SIZE>
__device__ __forceinline__ void best_splits(Workspace& w, const unsigned char* by_size, int n, int gl)
{
    const int count = SIZE < n ? choose(n, SIZE) : 0;
    for (int k = gl; k < count; k += kGroup) {
        const int S = by_size[size_first(SIZE) + k];
        const int low = S & -S, rest = S ^ low;
        float best = 3.4e38f;
        int bp = low, sub = rest;
        // P holds the lowest leaf of S, so every split is seen once
#pragma unroll
        for (int t = 0; t < (1 << (SIZE - 1)) - 1; ++t) {
            sub = (sub - 1) & rest;
            const int P = low | sub;
            const float c = w.copt[P] + w.copt[S ^ P];
            if (c < best) {
                best = c;
                bp = P;
            }
        }
        w.copt[S] = subset_cost(w, S, best);
        w.part[S] = (unsigned char)bp;
    }
    __syncwarp();
}

// Optimise up to four treelets, one per group of eight lanes (root < 0: the
// group has none).  All 32 lanes call it.
//
// What bounds it: issue slots (half of them used), mostly the 966 splits of a
// seven-leaf treelet.  One warp per treelet, with one lane growing it (about 40
// dependent L2 reads) and one lane on the full set's 63 splits, took 7.8 ms a
// pass over 2,050,412 triangles, nearly all of it latency.  Eight lanes hold a
// treelet's leaves in registers and fetch each new leaf's box, cost and children
// as soon as it is known, so growing costs one L2 latency per level; the splits
// of the full set are shared by the group; subset boxes are the union of two
// table entries; 2.1 to 2.4 ms a pass with one leaf a lane, the same trees.
__device__ void optimise_treelets(const Tree& T, int root, Workspace& w, const unsigned char* by_size)
{
    const unsigned full_mask = 0xffffffffu;
    const int gl = (int)(threadIdx.x & (kGroup - 1));  // lane in the group
    const bool on = root >= 0;
    __syncwarp();
    // grow the treelet: expand the leaf of largest area that is an internal node
    int n = on ? 2 : 0;
    int ref = 0;
    int2 kids = make_int2(0, 0);
    float area = -1.f, cost = 0.f;
    float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
    auto fetch = [&](int r) {
        ref = r;
        lo = __ldcg(r < 0 ? T.llo + ~r : T.nlo + r);
        hi = __ldcg(r < 0 ? T.lhi + ~r : T.nhi + r);
        if (r >= 0) {
            kids = __ldcg(T.child + r);
            cost = __ldcg(T.cost + r);
        }
        const float a = half_area(lo, hi);
        if (r < 0) cost = kCostTri * a;
        area = r >= 0 ? a : -1.f;  // only internal nodes are expanded
    };
    if (on) {
        const int2 c = __ldcg(T.child + root);
        if (gl == 0) w.inner[0] = root;
        if (gl < 2) fetch(gl == 0 ? c.x : c.y);
    }
    bool grow = on;
    for (int step = 2; step < kTreelet; ++step) {
        // the largest area of the group, the lowest lane among equals
        float best = gl < n && area > -1.f ? area : -1.f;
        int who = gl;
#pragma unroll
        for (int o = 1; o < kGroup; o <<= 1) {
            const float b = __shfl_xor_sync(full_mask, best, o);
            const int v = __shfl_xor_sync(full_mask, who, o);
            if (b > best || (b == best && v < who)) {
                best = b;
                who = v;
            }
        }
        const int node = __shfl_sync(full_mask, ref, who, kGroup);
        const int cx = __shfl_sync(full_mask, kids.x, who, kGroup), cy = __shfl_sync(full_mask, kids.y, who, kGroup);
        grow = grow && best > -1.f;
        if (grow) {
            if (gl == 0) w.inner[n - 1] = node;
            if (gl == who || gl == n) fetch(gl == who ? cx : cy);
            ++n;
        }
        if (__ballot_sync(full_mask, grow) == 0) break;
    }
    if (gl < n) {
        w.leaf[gl] = ref;
        w.lo[gl] = lo;
        w.hi[gl] = hi;
        w.copt[1 << gl] = cost;
    }
    __syncwarp();
    const int full = (1 << n) - 1;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int e = gl + r * kGroup;
        const int first = e < 8 ? 0 : 3, S = (e < 8 ? e : (e - 8) << 3) & full;
        float4 a = make_float4(3.4e38f, 3.4e38f, 3.4e38f, 0.f), b = make_float4(-3.4e38f, -3.4e38f, -3.4e38f, 0.f);
        for (int i = first; i < first + 4; ++i) {
            if (!(S & (1 << i))) continue;
            const float4 l = w.lo[i], h = w.hi[i];
            a = make_float4(fminf(a.x, l.x), fminf(a.y, l.y), fminf(a.z, l.z), 0.f);
            b = make_float4(fmaxf(b.x, h.x), fmaxf(b.y, h.y), fmaxf(b.z, h.z), 0.f);
        }
        w.ulo[e] = a;
        w.uhi[e] = b;
    }
    __syncwarp();
    // subsets by size, each by one lane: the best split of each
    const unsigned nmax = __reduce_max_sync(full_mask, (unsigned)n);
    if (nmax > 2) best_splits<2>(w, by_size, n, gl);
    if (nmax > 3) best_splits<3>(w, by_size, n, gl);
    if (nmax > 4) best_splits<4>(w, by_size, n, gl);
    if (nmax > 5) best_splits<5>(w, by_size, n, gl);
    if (nmax > 6) best_splits<6>(w, by_size, n, gl);
    // the full set: its splits, shared by the lanes, in the same order (the t-th
    // submask below `rest`); the first of the smallest wins
    bool better = false;
    {
        float best = 3.4e38f;
        int bt = 1 << kTreelet;
        const int splits = n >= 3 ? (1 << (n - 1)) - 1 : 0;
        for (int t = gl; t < splits; t += kGroup) {
            const int P = full - 2 * (t + 1);
            const float c = w.copt[P] + w.copt[full ^ P];
            if (c < best) { best = c; bt = t; }
        }
#pragma unroll
        for (int o = 1; o < kGroup; o <<= 1) {
            const float b = __shfl_xor_sync(full_mask, best, o);
            const int v = __shfl_xor_sync(full_mask, bt, o);
            if (b < best || (b == best && v < bt)) {
                best = b;
                bt = v;
            }
        }
        if (n >= 3) {
            const float c = subset_cost(w, full, best);
            better = c < __ldcg(T.cost + root) * (1.f - 1e-6f);
            if (gl == 0) w.part[full] = (unsigned char)(bt < splits ? full - 2 * (bt + 1) : 1);
        }
    }
    if (__ballot_sync(full_mask, better) == 0) return;
    __syncwarp();
    // rewire: internal nodes in the order they are assigned (parents first)
    if (better && gl == 0) {
        int sp = 0, next = 1, m = 0;
        int stack_set[kTreelet], stack_node[kTreelet];
        stack_set[sp] = full;
        stack_node[sp++] = root;
        while (sp > 0) {
            --sp;
            const int S = stack_set[sp], node = stack_node[sp];
            const int P = w.part[S];
            int ref2[2];
            for (int side = 0; side < 2; ++side) {
                const int X = side == 0 ? P : S ^ P;
                if (__popc(X) == 1) {
                    ref2[side] = w.leaf[__ffs(X) - 1];
                } else {
                    ref2[side] = w.inner[next++];
                    stack_set[sp] = X;
                    stack_node[sp++] = ref2[side];
                }
            }
            w.set[m] = S;
            w.node[m] = node;
            w.ref0[m] = ref2[0];
            w.ref1[m] = ref2[1];
            ++m;
        }
        // costs, children before parents (copt of the chosen sets becomes the nodes' cost)
        for (int i = m - 1; i >= 0; --i) {
            const int S = w.set[i], P = w.part[S];
            float4 lo2, hi2;
            subset_box(w, S, lo2, hi2);
            w.copt[S] = rttree::node_cost(lo2, hi2, w.copt[P], w.copt[S ^ P]);
        }
    }
    __syncwarp();
    if (better && gl < n - 1) {  // a treelet of n leaves has n - 1 internal nodes, one per lane
        const int S = w.set[gl], node = w.node[gl], r0 = w.ref0[gl], r1 = w.ref1[gl];
        float4 nl, nh;
        subset_box(w, S, nl, nh);
        T.child[node] = make_int2(r0, r1);
        if (r0 < 0) T.par_l[~r0] = node;
        else T.par_i[r0] = node;
        if (r1 < 0) T.par_l[~r1] = node;
        else T.par_i[r1] = node;
        T.nlo[node] = nl;
        T.nhi[node] = nh;
        T.cost[node] = w.copt[S];
        __threadfence();
    }
    __syncwarp();
}

// One restructuring pass: leaves walk up; each node whose second child finished
// is optimised by the warp of the thread that finished it, four at a time.  A
// node over two leaves has one topology only and is passed.  (Passing, in later
// passes, the nodes below and around which nothing had changed since they were
// last looked at saved nothing: few are left out.)
__global__ void __launch_bounds__(kBlock) k_treelets(Tree T)
{
    __shared__ Workspace ws[kWarps * kGroups];
    __shared__ unsigned char by_size[kSubsets];
    for (int i = (int)threadIdx.x; i < kSubsets; i += kBlock) by_size[i] = kBySize[i];
    __syncthreads();
    Workspace& w = ws[threadIdx.x / kGroup];
    const unsigned group = (threadIdx.x & 31u) / kGroup;
    // this lane's leaves: every 32nd of the warp's, taken in turn
    const int64_t warp0 = ((int64_t)blockIdx.x * kWarps + threadIdx.x / 32) * (32 * kLeaves);
    int64_t next = warp0 + (threadIdx.x & 31u);
    const int64_t end = min(warp0 + 32 * kLeaves, T.n_leaves);
    int32_t node = -1;
    bool active = false;
    for (int guard = 0; guard < kMaxWalk * kLeaves; ++guard) {
        bool ready = false, pick = false;
        if (!active && next < end) {
            node = T.par_l[next];
            next += 32;
            active = node >= 0;
        }
        if (active) {
            if (atomicAdd(&T.visit[node], 1) == 0) active = false;  // the sibling subtree is not finished
            else ready = true;
        }
        if (ready) {
            __threadfence();
            const int2 c = __ldcg(T.child + node);
            pick = c.x >= 0 || c.y >= 0;
        }
        unsigned todo = __ballot_sync(0xffffffffu, pick);
        if (todo == 0 && __ballot_sync(0xffffffffu, active || next < end) == 0) break;
        while (todo) {
            unsigned mine = todo;  // this group's root: the group-th of the lanes still to do
            for (unsigned g = 0; g < group; ++g) mine &= mine - 1;
            const int src = mine ? __ffs(mine) - 1 : 0;
            const int root = __shfl_sync(0xffffffffu, node, src);
            optimise_treelets(T, mine ? root : -1, w, by_size);
            for (int g = 0; g < kGroups; ++g) todo &= todo - 1;
        }
        if (ready) {
            node = __ldcg(T.par_i + node);
            active = node >= 0;
        }
    }
}

// leaves (and internal nodes) in depth-first order: the position of a node's
// first leaf is the number of leaves left of its path from the root
__global__ void k_counts(const int2* child, const int32_t* par_i, const int32_t* par_l, int64_t n_leaves, int* count,
                         int* visit)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_leaves) return;
    int32_t node = par_l[k];
    for (int guard = 0; node >= 0 && guard < kMaxWalk; ++guard) {
        if (atomicAdd(&visit[node], 1) == 0) return;
        __threadfence();
        const int2 c = child[node];
        count[node] = (c.x < 0 ? 1 : __ldcg(count + c.x)) + (c.y < 0 ? 1 : __ldcg(count + c.y));
        __threadfence();
        node = par_i[node];
    }
}

__device__ __forceinline__ int first_leaf(const int2* child, const int32_t* par_i, const int* count, int32_t self,
                                          int32_t parent)
{
    int pos = 0;
    for (int guard = 0; parent >= 0 && guard < kMaxWalk; ++guard) {
        const int2 c = child[parent];
        if (c.y == self) pos += c.x < 0 ? 1 : count[c.x];
        self = parent;
        parent = par_i[parent];
    }
    return pos;
}

__global__ void k_leaf_position(const int2* child, const int32_t* par_i, const int32_t* par_l, const int* count,
                                int64_t n_leaves, int32_t* pos)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_leaves) return;
    pos[k] = first_leaf(child, par_i, count, ~(int32_t)k, par_l[k]);
}

__global__ void k_node_range(const int2* child, const int32_t* par_i, const int* count, int64_t n_int, int2* range)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_int) return;
    const int first = first_leaf(child, par_i, count, (int32_t)i, par_i[i]);
    range[i] = make_int2(first, first + count[i] - 1);
}

// leaf k moves to position pos[k]: the triangle order, leaf boxes and references follow
__global__ void k_permute_leaves(const int32_t* pos, int64_t n_leaves, const int32_t* order, const float4* llo,
                                 const float4* lhi, int32_t* order2, float4* llo2, float4* lhi2, int32_t* par_l2,
                                 const int32_t* par_l)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_leaves) return;
    const int32_t p = pos[k];
    order2[p] = order[k];
    llo2[p] = llo[k];
    lhi2[p] = lhi[k];
    par_l2[p] = par_l[k];
}

__global__ void k_remap_children(int2* child, int64_t n_int, const int32_t* pos)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_int) return;
    int2 c = child[i];
    if (c.x < 0) c.x = ~pos[~c.x];
    if (c.y < 0) c.y = ~pos[~c.y];
    child[i] = c;
}

unsigned grid_for(int64_t n) { return (unsigned)((n + kBlock - 1) / kBlock); }

}  // namespace

rt_status rt_treelet_optimise(int64_t nt, int passes, int2* child, int2* range, int32_t* par_i, int32_t* par_l,
                              int32_t* order, float4* llo, float4* lhi, float4* nlo, float4* nhi, float* cost,
                              const TreeletScratch& ws, cudaStream_t s)
{
    if (nt < 3 || passes <= 0) return RT_OK;
    const int64_t ni = nt - 1;
    const Tree T = {child, par_i, par_l, llo, lhi, nlo, nhi, cost, ws.visit, nt};
    for (int pass = 0; pass < passes; ++pass) {
        RT_CUDA_TRY(cudaMemsetAsync(ws.visit, 0, ni * sizeof(int), s));
        k_treelets<<<(unsigned)((nt + kBlock * kLeaves - 1) / (kBlock * kLeaves)), kBlock, 0, s>>>(T);
    }
    // depth-first leaf order
    RT_CUDA_TRY(cudaMemsetAsync(ws.visit, 0, ni * sizeof(int), s));
    k_counts<<<grid_for(nt), kBlock, 0, s>>>(child, par_i, par_l, nt, ws.count, ws.visit);
    k_leaf_position<<<grid_for(nt), kBlock, 0, s>>>(child, par_i, par_l, ws.count, nt, ws.pos);
    k_node_range<<<grid_for(ni), kBlock, 0, s>>>(child, par_i, ws.count, ni, range);
    k_permute_leaves<<<grid_for(nt), kBlock, 0, s>>>(ws.pos, nt, order, llo, lhi, ws.order2, ws.llo2, ws.lhi2, ws.par_l2,
                                                     par_l);
    k_remap_children<<<grid_for(ni), kBlock, 0, s>>>(child, ni, ws.pos);
    RT_CUDA_TRY(cudaGetLastError());
    RT_CUDA_TRY(cudaMemcpyAsync(order, ws.order2, nt * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    RT_CUDA_TRY(cudaMemcpyAsync(par_l, ws.par_l2, nt * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    RT_CUDA_TRY(cudaMemcpyAsync(llo, ws.llo2, nt * sizeof(float4), cudaMemcpyDeviceToDevice, s));
    RT_CUDA_TRY(cudaMemcpyAsync(lhi, ws.lhi2, nt * sizeof(float4), cudaMemcpyDeviceToDevice, s));
    return RT_OK;
}
