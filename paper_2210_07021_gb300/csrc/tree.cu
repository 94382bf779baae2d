// The adaptive 12-root quad-tree of Sec. 3.1 and its box geometry.
//
// Division rule (Sec. 3.1, steps 1-3): the 12 HEALPix base boxes hold the
// particles by key; a box holding more than m particles is divided into its 4
// children (always 4, empty or not) until no box holds more than m, or the
// level reaches the maximum depth (r_max = 29 by default).  Built level by level
// from the key-sorted particles: a child's particle range is found by binary
// search inside its parent's range.  Nodes are numbered by level, then by
// pixel index.
//
// Geometry (Sec. 3.1 frame K_P, Sec. 3.5 radius): a box's centre is its HEALPix
// pixel centre; its frame has zenith e_r(centre) and azimuth reference
// e_theta(centre); its radius R is the largest angle from the centre to the
// pixel's 4 corners (the corners realise the covering radius of a HEALPix
// pixel), plus 2e-15 rad for the rounding of the keys.  r = tan(R/2) is the
// scale of the stereographic variable z = tan(theta/2) e^{i phi} inside the box.
#include "common.cuh"
#include "lookback.cuh"

#include <algorithm>

namespace sfmm {

namespace {

__constant__ int c_jrll[12] = {2, 2, 2, 2, 3, 3, 3, 3, 4, 4, 4, 4};
__constant__ int c_jpll[12] = {1, 3, 5, 7, 0, 2, 4, 6, 1, 3, 5, 7};

__device__ __forceinline__ int64_t lower_bound_u64(const uint64_t* a, int64_t lo, int64_t hi, uint64_t v)
{
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ uint64_t compact_bits(uint64_t v)
{
    v &= 0x5555555555555555ull;
    v = (v | (v >> 1)) & 0x3333333333333333ull;
    v = (v | (v >> 2)) & 0x0F0F0F0F0F0F0F0Full;
    v = (v | (v >> 4)) & 0x00FF00FF00FF00FFull;
    v = (v | (v >> 8)) & 0x0000FFFF0000FFFFull;
    v = (v | (v >> 16)) & 0x00000000FFFFFFFFull;
    return v;
}

// A node's centre and corners are points at face coordinates (X, Y) in [0, N_side]^2 of
// its base pixel (the inverse of the ang2pix mapping).  z and sin theta depend on X + Y
// alone, and in the belt the azimuth on X - Y alone: the centre and two corners lie on
// one ring, there the centre and the other two on one meridian, so five points take three
// rings and three (caps: five) azimuths.  FP64-bound; the divisions by 3 N_side^k are three
// instructions and a scaling, not a general division (10).  The tree of 1.6e7 clustered
// points: 0.64 -> 0.43 ms; 4096 points (one chain's latency): 49 -> 34 us.

// x / 3, correctly rounded: the product with the rounded reciprocal and one correction
// by the exact remainder (Markstein 1990)
__device__ __forceinline__ double third(double x)
{
    const double y = 1.0 / 3.0, q = x * y;
    return __fma_rn(__fma_rn(-3.0, q, x), y, q);
}

// The ring through the in-face point X + Y = const: nr, z and sin theta from
// jr = jrll N_side - X - Y (ns = N_side, ins = 1/N_side: powers of two, so scaling by them is exact)
struct Ring {
    double nr, z, s;
};
__device__ __forceinline__ Ring ring_of(double jr, double ns, double ins)
{
    Ring r;
    if (jr < ns || jr > 3.0 * ns) {
        r.nr = jr < ns ? jr : 4.0 * ns - jr;
        const double t = third(r.nr * r.nr) * (ins * ins);       // 1 - |z|
        r.z = jr < ns ? 1.0 - t : t - 1.0;
        r.s = sqrt(t * (2.0 - t));
    } else {
        r.nr = ns;
        r.z = third((2.0 * ns - jr) * 2.0) * ins;
        r.s = sqrt((1.0 - r.z) * (1.0 + r.z));
    }
    return r;
}
// cos phi and sin phi of the point X - Y = d of a ring
__device__ __forceinline__ void ring_phi(double jp, double d, const Ring& r, double ns, double ins, double* cp, double* sp)
{
    if (r.nr > 0.0) sincospi(0.25 * (jp + (r.nr == ns ? d * ins : d / r.nr)), sp, cp);
    else { *sp = 0.0; *cp = 1.0; }
}

__global__ void k_level0(const uint64_t* __restrict__ keys, int64_t n, uint64_t* prefix, int* level, int* first,
                         int* count, int* child0, int* parent)
{
    const int f = threadIdx.x;
    if (f >= 12) return;
    const uint64_t lo = (uint64_t)f << (2 * ORDER_MAX), hi = (uint64_t)(f + 1) << (2 * ORDER_MAX);
    const int64_t a = lower_bound_u64(keys, 0, n, lo);
    const int64_t b = lower_bound_u64(keys, a, n, hi);
    prefix[f] = (uint64_t)f;
    level[f] = 0;
    first[f] = (int)a;
    count[f] = (int)(b - a);
    child0[f] = -1;
    parent[f] = -1;
}

// Graph mode (dc != NULL): the level's bounds come from dc->level, the launch
// covers `width` (the level-width capacity) and the flags beyond the level are
// zero, so that a scan over the whole capacity is the scan of the level.
__global__ void k_split_flags(const int* count, int a, int b, int lvl, int m, int max_depth,
                              int64_t* flags, DevCounts* dc, int64_t width)
{
    after_previous();
    if (dc) {
        a = (int)dc->level[lvl];
        b = (int)dc->level[lvl + 1];
        if (blockIdx.x == 0 && threadIdx.x == 0 && b - a > width) dc->overflow = 1;
    } else {
        width = b - a;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < width; i += (int64_t)gridDim.x * blockDim.x)
        flags[i] = (i < b - a && count[a + i] > m && lvl < max_depth) ? 1 : 0;
}

__global__ void k_counts_init(DevCounts* dc)
{
    if (threadIdx.x < 32) dc->level[threadIdx.x] = threadIdx.x == 0 ? 0 : 12;
    if (threadIdx.x == 0) { dc->nn = 12; dc->n_leaves = 0; dc->n_items = 0; dc->overflow = 0; }
}

// Graph mode: the next level's end from the scan of the split flags (its total),
// or an overflow if the nodes would not fit the capacity (`last`: the deepest
// level the capacity allows; a split there is an overflow too).
__global__ void k_level_end(DevCounts* dc, int lvl, const int64_t* total, int64_t node_cap, int last)
{
    after_previous();
    const int64_t b = dc->level[lvl + 1];
    int64_t nb = b + 4 * *total;
    // after an overflow the tree stops growing: the nodes built so far stay a
    // consistent tree (unsplit nodes are leaves), so every later kernel stays in bounds
    if (dc->overflow || nb > node_cap || (last && *total > 0)) {
        dc->overflow = 1;
        nb = b;
    }
    dc->level[lvl + 2] = nb;
    dc->nn = nb;
}

struct NodeArrays {
    uint64_t* prefix;
    int *level, *first, *count, *child0, *parent;
};

// Child c = lane % 4 of a split node: its range by binary search of its first key
// inside the parent's range, its end from the next child (the four lanes of a
// node work together: one search's latency per node, not three).
__device__ __forceinline__ void make_child(const uint64_t* __restrict__ keys, const NodeArrays& N, int node, int c0,
                                           int lvl, bool split)
{
    const int c = threadIdx.x & 3;
    const int shift = 2 * (ORDER_MAX - (lvl + 1));
    uint64_t pf = 0;
    int64_t lo = 0, hi = 0, start = 0;
    if (split) {
        pf = N.prefix[node] * 4ull + c;
        lo = N.first[node];
        hi = lo + N.count[node];
        start = c == 0 ? lo : lower_bound_u64(keys, lo, hi, pf << shift);
    }
    const int64_t next = __shfl_down_sync(FULL, start, 1, 4);
    if (!split) return;
    const int64_t end = c == 3 ? hi : next;
    const int k = c0 + c;
    N.prefix[k] = pf;
    N.level[k] = lvl + 1;
    N.first[k] = (int)start;
    N.count[k] = (int)(end - start);
    N.child0[k] = -1;
    N.parent[k] = node;
    if (c == 0) N.child0[node] = c0;
}

__global__ void k_make_children(const uint64_t* keys, int a, int b, int lvl,
                                const int64_t* flags, const int64_t* pos, NodeArrays N,
                                const DevCounts* dc)
{
    after_previous();
    if (dc) {
        if (dc->overflow) return;
        a = (int)dc->level[lvl];
        b = (int)dc->level[lvl + 1];
    }
    const int64_t nt = 4 * (int64_t)(b - a), step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); t0 < nt; t0 += step) {
        const int64_t i = (t0 + (threadIdx.x & 31)) >> 2;
        const bool split = i < b - a && flags[i];
        make_child(keys, N, a + (int)i, split ? b + 4 * (int)pos[i] : 0, lvl, split);
    }
}

// The levels of the tree on the device: nodes of level l are [start[l], start[l + 1]),
// levels 0..lvl exist; done when no box of level lvl is to be split.
struct TreeLevels {
    int64_t lvl, done;
    int64_t start[ORDER_MAX + 3];
};

// One CTA builds the tree on from level lvl for as long as a level has at most
// TREE_NARROW boxes (and its children fit the node capacity): the flags, their
// scan and the children of all those levels in one launch and one host
// synchronisation.  A level at a time costs five launches and a synchronisation,
// 45 us: the tree of 1e4 clustered points (13 levels) took 0.58 ms without its
// geometry, and takes 0.06 ms.
constexpr int TREE_NARROW = 4096, TREE_T = 1024;

__global__ void __launch_bounds__(TREE_T) k_tree_narrow(const uint64_t* keys, int64_t n, int m,
                                                        int max_depth, int64_t node_cap, bool first, TreeLevels* L,
                                                        NodeArrays N)
{
    after_previous();
    __shared__ int s_node[TREE_NARROW];              // the level's split boxes in order
    __shared__ int s_warp[TREE_T / 32];
    __shared__ int s_total;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int lvl;
    int64_t a, b;
    if (first) {
        if (tid < 12) {
            const uint64_t lo = (uint64_t)tid << (2 * ORDER_MAX), hi = (uint64_t)(tid + 1) << (2 * ORDER_MAX);
            const int64_t f = lower_bound_u64(keys, 0, n, lo), e = lower_bound_u64(keys, f, n, hi);
            N.prefix[tid] = (uint64_t)tid;
            N.level[tid] = 0;
            N.first[tid] = (int)f;
            N.count[tid] = (int)(e - f);
            N.child0[tid] = -1;
            N.parent[tid] = -1;
        }
        lvl = 0;
        a = 0;
        b = 12;
        if (tid == 0) { L->start[0] = 0; L->start[1] = 12; }
        __syncthreads();
    } else {
        lvl = (int)L->lvl;
        a = L->start[lvl];
        b = L->start[lvl + 1];
    }
    bool done = false;
    while (b - a <= TREE_NARROW) {
        if (lvl >= max_depth) { done = true; break; }
        int splits = 0;
        for (int64_t i0 = a; i0 < b; i0 += TREE_T) {
            const bool f = i0 + tid < b && N.count[i0 + tid] > m;
            const unsigned mask = __ballot_sync(FULL, f);
            if (lane == 0) s_warp[warp] = __popc(mask);
            __syncthreads();
            if (warp == 0) {
                const int v = s_warp[lane];
                int inc = v;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(FULL, inc, o);
                    if (lane >= o) inc += t;
                }
                s_warp[lane] = inc - v;
                if (lane == 31) s_total = inc;
            }
            __syncthreads();
            if (f) s_node[splits + s_warp[warp] + __popc(mask & ((1u << lane) - 1u))] = (int)(i0 + tid);
            splits += s_total;
            __syncthreads();
        }
        if (splits == 0) { done = true; break; }
        if (b + 4 * (int64_t)splits > node_cap) break;
        for (int t0 = 0; t0 < 4 * splits; t0 += TREE_T) {
            const int j = (t0 + tid) >> 2;
            const bool split = j < splits;
            make_child(keys, N, split ? s_node[j] : 0, (int)b + 4 * j, lvl, split);
        }
        a = b;
        b += 4 * (int64_t)splits;
        ++lvl;
        if (tid == 0) L->start[lvl + 1] = b;
        __syncthreads();
    }
    if (tid == 0) {
        L->lvl = lvl;
        L->done = done;
    }
}

__global__ void k_geometry(int n_cap, const int64_t* d_nn, const uint64_t* prefix,
                           const int* level, double* geom)
{
    after_previous();
    const int64_t n_nodes = dcount(d_nn, n_cap);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_nodes; i += (int64_t)gridDim.x * blockDim.x) {
        const int order = level[i];
        const uint64_t pix = prefix[i];
        const int face = (int)(pix >> (2 * order));
        const uint64_t ipf = pix & ((1ull << (2 * order)) - 1ull);
        const double ix = (double)compact_bits(ipf), iy = (double)compact_bits(ipf >> 1);
        const double ns = __hiloint2double((1023 + order) << 20, 0), ins = __hiloint2double((1023 - order) << 20, 0);
        // the rings of the first corner, of the centre and two corners, of the last corner
        const double jr = c_jrll[face] * ns - ix - iy, d = ix - iy, jp = c_jpll[face];
        const Ring r0 = ring_of(jr, ns, ins), r1 = ring_of(jr - 1.0, ns, ins), r2 = ring_of(jr - 2.0, ns, ins);
        double cp, sp, c1, s1, c2, s2;
        ring_phi(jp, d, r1, ns, ins, &cp, &sp);
        ring_phi(jp, d + 1.0, r1, ns, ins, &c1, &s1);
        ring_phi(jp, d - 1.0, r1, ns, ins, &c2, &s2);
        double c0 = cp, s0 = sp, c3 = cp, s3 = sp;               // the same meridian in the belt
        if (r0.nr != r1.nr) ring_phi(jp, d, r0, ns, ins, &c0, &s0);
        if (r2.nr != r1.nr) ring_phi(jp, d, r2, ns, ins, &c3, &s3);
        const double ct = r1.z, st = r1.s, c[3] = {st * cp, st * sp, ct};
        const double vs[4] = {r0.s, st, st, r2.s}, vc[4] = {c0, c1, c2, c3}, vv[4] = {s0, s1, s2, s3}, vz[4] = {r0.z, ct, ct, r2.z};
        double chord2 = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double dx = __fma_rn(vs[k], vc[k], -c[0]), dy = __fma_rn(vs[k], vv[k], -c[1]), dz = vz[k] - c[2];
            chord2 = fmax(chord2, __fma_rn(dz, dz, __fma_rn(dy, dy, dx * dx)));
        }
        const double R = 2.0 * asin(fmin(1.0, 0.5 * sqrt(chord2))) + 2e-15;
        double* g = geom + (size_t)i * GEOM_STRIDE;
        g[0] = c[0]; g[1] = c[1]; g[2] = c[2];
        g[3] = ct * cp; g[4] = ct * sp; g[5] = -st;     // e_theta at the centre
        g[6] = -sp; g[7] = cp; g[8] = 0.0;              // e_phi at the centre
        g[9] = R;
        g[10] = tan(0.5 * R);
        g[11] = 0.0;
    }
}

__global__ void k_target_ranges(int n_cap, const int64_t* d_nn, const uint64_t* prefix,
                                const int* level, const uint64_t* tkeys, int64_t M,
                                int* tfirst, int* tcount)
{
    after_previous();
    const int64_t n_nodes = dcount(d_nn, n_cap);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_nodes; i += (int64_t)gridDim.x * blockDim.x) {
        const int shift = 2 * (ORDER_MAX - level[i]);
        const uint64_t lo = prefix[i] << shift, hi = (prefix[i] + 1ull) << shift;
        const int64_t a = lower_bound_u64(tkeys, 0, M, lo);
        const int64_t b = lower_bound_u64(tkeys, a, M, hi);
        tfirst[i] = (int)a;
        tcount[i] = (int)(b - a);
    }
}

// Evaluation items per node: a leaf's targets in chunks of 64, or (split) of 32
// where more than 32 are left.
__device__ __forceinline__ int64_t items_of(int tc, int split) { return split ? (tc + 31) / 32 : (tc + 63) / 64; }

// The source leaves (leaves holding sources, in node order) and the evaluation's
// items of all leaves holding targets, in one pass over the nodes: a tile of 1024
// nodes finds its places by looking back (words: leaves and items per tile).  A
// node with more than 4 items writes them by the whole warp (one leaf can hold
// every target of the problem).  out: the two counts, then the tile counter.
constexpr int CT = 256, CI = 4, CTILE = CT * CI;

__device__ __forceinline__ int2 make_item(int node, int tc, int64_t k, int split)
{
    if (!split) return make_int2(node, (int)(k * 64) | ITEM_A | ITEM_B);
    const int tb = (int)(k / 2) * 64;
    const int parts = (k & 1) ? ITEM_B : tc - tb > 32 ? ITEM_A : ITEM_A | ITEM_B;
    return make_int2(node, tb | parts);
}

__global__ void __launch_bounds__(CT) k_collect(int n_cap, const int64_t* d_nn, const int* child0,
                                                const int* count, const int* tcount,
                                                int split, int* leaves, int2* items,
                                                uint64_t* words, int64_t* n_leaves,
                                                int64_t* n_items, uint32_t* ticket, int limit)
{
    after_previous();
    __shared__ uint32_t s_tile;
    __shared__ int64_t s_warp[2][CT / 32], s_base[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nn = dcount(d_nn, n_cap);
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const int64_t tile = s_tile, ntiles = ((int64_t)n_cap + CTILE - 1) / CTILE;
    const int64_t i0 = tile * CTILE + (int64_t)threadIdx.x * CI;
    int tc[CI];
    bool lf[CI];
    int64_t nl = 0, ni = 0;
#pragma unroll
    for (int r = 0; r < CI; ++r) {
        const int64_t i = i0 + r;
        const bool leaf = i < nn && child0[i] < 0;
        lf[r] = leaf && count[i] > 0;
        tc[r] = leaf ? tcount[i] : 0;
        nl += lf[r];
        ni += items_of(tc[r], split);
    }
    int64_t il = nl, ii = ni;                       // inclusive sums over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t x = __shfl_up_sync(FULL, il, o), y = __shfl_up_sync(FULL, ii, o);
        if (lane >= o) { il += x; ii += y; }
    }
    if (lane == 31) { s_warp[0][warp] = il; s_warp[1][warp] = ii; }
    __syncthreads();
    int64_t bl = 0, bi = 0, tl = 0, ti = 0;
    for (int w = 0; w < CT / 32; ++w) {
        if (w < warp) { bl += s_warp[0][w]; bi += s_warp[1][w]; }
        tl += s_warp[0][w];
        ti += s_warp[1][w];
    }
    if (warp < 2) {                                 // warp 0: leaves, warp 1: items
        const int64_t own = warp == 0 ? tl : ti;
        uint64_t* w = words + 2 * tile + warp;
        if (lane == 0) lb_publish(w, 0, LB_OWN, own);
        int64_t before = 0;
        const bool ok = lb_before(words + warp, 2, tile, 0, limit, &before);
        if (!ok) {                                  // the wait ran out: count the earlier nodes
            before = 0;
            for (int64_t i = lane; i < tile * CTILE; i += 32)
                if (i < nn && child0[i] < 0) before += warp == 0 ? (count[i] > 0) : items_of(tcount[i], split);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(FULL, before, o);
        }
        if (lane == 0) {
            lb_publish(w, 0, LB_UPTO, before + own);
            s_base[warp] = before;
            if (tile == ntiles - 1) *(warp == 0 ? n_leaves : n_items) = before + own;
        }
    }
    __syncthreads();
    int64_t ol = s_base[0] + bl + il - nl, oi = s_base[1] + bi + ii - ni;
#pragma unroll
    for (int r = 0; r < CI; ++r) {
        const int64_t c = items_of(tc[r], split);
        if (lf[r]) leaves[ol++] = (int)(i0 + r);
        if (c <= 4)
            for (int64_t k = 0; k < c; ++k) items[oi + k] = make_item((int)(i0 + r), tc[r], k, split);
        for (unsigned big = __ballot_sync(FULL, c > 4); big; big &= big - 1) {
            const int l = __ffs(big) - 1;
            const int64_t cl = __shfl_sync(FULL, c, l), al = __shfl_sync(FULL, oi, l), node = __shfl_sync(FULL, i0 + r, l);
            const int tl2 = __shfl_sync(FULL, tc[r], l);
            for (int64_t k = lane; k < cl; k += 32) items[al + k] = make_item((int)node, tl2, k, split);
        }
        oi += c;
    }
}

inline unsigned grid_for(int64_t n, int threads = 256)
{
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 16) b = 152 * 16;
    return (unsigned)b;
}

}  // namespace

// Build the tree from the key-sorted source keys.  Grows the plan's node arrays
// as needed; fills plan->level_start and plan->n_nodes.  Synchronises the
// stream once per run of narrow levels and once per wide level (the next level's
// size is needed on the host).
//
// Graph mode (plan->gm): no synchronisation.  Every level up to the plan's level
// capacity is launched with grids sized by the level-width capacity; the level
// bounds and the node count live in the plan's DevCounts (k_level_end), and a
// tree that would not fit (more nodes, a wider level, or a split at the last
// level) sets the overflow flag.  plan->n_nodes is the node capacity.
cudaError_t build_tree(sfmm_plan_s* P, const uint64_t* keys, int64_t n, int m, int max_depth)
{
    cudaStream_t s = P->stream;
    cudaError_t e;
    auto grow = [&](int64_t need) -> cudaError_t {
        if (need <= P->node_cap) return cudaSuccess;
        int64_t cap = need + need / 2 + 1024;
        size_t keep = (size_t)P->n_nodes;
        cudaError_t r;
        if ((r = ensure_keep(P->n_prefix, cap * 8, keep * 8, s))) return r;
        if ((r = ensure_keep(P->n_level, cap * 4, keep * 4, s))) return r;
        if ((r = ensure_keep(P->n_first, cap * 4, keep * 4, s))) return r;
        if ((r = ensure_keep(P->n_count, cap * 4, keep * 4, s))) return r;
        if ((r = ensure_keep(P->n_child0, cap * 4, keep * 4, s))) return r;
        if ((r = ensure_keep(P->n_parent, cap * 4, keep * 4, s))) return r;
        P->node_cap = cap;
        return cudaSuccess;
    };
    auto arrays = [&]() {
        return NodeArrays{P->n_prefix.as<uint64_t>(), P->n_level.as<int>(), P->n_first.as<int>(),
                          P->n_count.as<int>(), P->n_child0.as<int>(), P->n_parent.as<int>()};
    };
    if (P->gm) {
        DevCounts* dc = P->dcnt.as<DevCounts>();
        const int64_t width = P->cap.width, levels = P->cap.levels;
        if ((e = grow(P->cap.nodes)) || (e = ensure(P->flags, (size_t)width * 8)) ||
            (e = ensure(P->pos, (size_t)width * 8)) || (e = ensure(P->tmp, scan_tmp_bytes(width))))
            return e;
        int64_t* flags = P->flags.as<int64_t>();
        int64_t* pos = P->pos.as<int64_t>();
        int64_t* total = P->small.as<int64_t>();
        k_level0<<<1, 32, 0, s>>>(keys, n, P->n_prefix.as<uint64_t>(), P->n_level.as<int>(), P->n_first.as<int>(),
                                  P->n_count.as<int>(), P->n_child0.as<int>(), P->n_parent.as<int>()); count_launch();
        k_counts_init<<<1, 32, 0, s>>>(dc); count_launch();
        for (int lvl = 0; lvl < levels; ++lvl) {
            launch_chained(k_split_flags, grid_for(width), 256, 0, s, P->n_count.as<int>(), 0, 0, lvl, m, max_depth, flags, dc,
                                                           width);
            if ((e = exclusive_scan_i64(flags, pos, width, total, P->tmp.p, s))) return e;
            launch_chained(k_level_end, 1, 1, 0, s, dc, lvl, total, P->cap.nodes, lvl == levels - 1);
            if (lvl < levels - 1) {
                launch_chained(k_make_children, grid_for(4 * width), 256, 0, s, keys, 0, 0, lvl, flags, pos, arrays(), dc);
            }
        }
        P->n_nodes = P->cap.nodes;
        return cudaGetLastError();
    }
    // narrow levels in runs by one CTA (k_tree_narrow), wide ones a level at a time
    P->n_nodes = 0;
    if ((e = grow(12 + 4 * 1024))) return e;
    TreeLevels* dL = reinterpret_cast<TreeLevels*>(P->small.as<int64_t>() + SM_TREE);
    TreeLevels* hL = reinterpret_cast<TreeLevels*>(P->h_small + SM_TREE);
    P->level_start.assign(1, 0);
    P->level_start.push_back(12);
    bool first = true;
    while (true) {
        launch_chained(k_tree_narrow, 1, TREE_T, 0, s, keys, n, m, max_depth, P->node_cap, first, dL, arrays());
        if ((e = cudaMemcpyAsync(hL, dL, sizeof *hL, cudaMemcpyDeviceToHost, s)) || (e = cudaStreamSynchronize(s)))
            return e;
        first = false;
        int lvl = (int)hL->lvl;
        P->level_start.resize(lvl + 2);
        for (int l = 0; l <= lvl + 1; ++l) P->level_start[l] = (int)hL->start[l];
        P->n_nodes = P->level_start[lvl + 1];
        if (hL->done) break;
        // this level (and the wide ones after it) with the whole GPU
        bool end = false;
        do {
            const int a = P->level_start[lvl], b = P->level_start[lvl + 1];
            const int64_t width = b - a;
            if (lvl >= max_depth) { end = true; break; }
            if ((e = ensure(P->flags, (size_t)width * 8)) || (e = ensure(P->pos, (size_t)width * 8)) ||
                (e = ensure(P->tmp, scan_tmp_bytes(width))))
                return e;
            int64_t* flags = P->flags.as<int64_t>();
            int64_t* pos = P->pos.as<int64_t>();
            int64_t* total = P->small.as<int64_t>() + SM_TOTAL;
            launch_chained(k_split_flags, grid_for(width), 256, 0, s, P->n_count.as<int>(), a, b, lvl, m, max_depth, flags,
                                                           nullptr, 0);
            if ((e = exclusive_scan_i64(flags, pos, width, total, P->tmp.p, s))) return e;
            int64_t* splits = P->h_small + SM_TOTAL;
            if ((e = cudaMemcpyAsync(splits, total, 8, cudaMemcpyDeviceToHost, s)) || (e = cudaStreamSynchronize(s)))
                return e;
            if (*splits == 0) { end = true; break; }
            if ((e = grow(b + 4 * *splits))) return e;
            launch_chained(k_make_children, grid_for(4 * width), 256, 0, s, keys, a, b, lvl, flags, pos, arrays(), nullptr);
            P->n_nodes = b + 4 * *splits;
            P->level_start.push_back((int)P->n_nodes);
            ++lvl;
        } while (P->level_start[lvl + 1] - P->level_start[lvl] > TREE_NARROW);
        if (end) break;
        // hand the levels so far back to the narrow kernel
        hL->lvl = lvl;
        for (int l = 0; l <= lvl + 1; ++l) hL->start[l] = P->level_start[l];
        if ((e = cudaMemcpyAsync(dL, hL, sizeof *hL, cudaMemcpyHostToDevice, s))) return e;
    }
    P->last_max_width = 12;
    for (size_t l = 0; l + 1 < P->level_start.size(); ++l)
        P->last_max_width = std::max<int64_t>(P->last_max_width, P->level_start[l + 1] - P->level_start[l]);
    return cudaGetLastError();
}

cudaError_t tree_geometry(sfmm_plan_s* P)
{
    cudaError_t e;
    const int64_t nn = P->n_nodes;
    if ((e = ensure(P->n_geom, (size_t)nn * GEOM_STRIDE * 8))) return e;
    launch_chained(k_geometry, grid_for(nn), 256, 0, P->stream, (int)nn, P->gm ? &P->dcnt.as<DevCounts>()->nn : nullptr,
                                                    P->n_prefix.as<uint64_t>(), P->n_level.as<int>(),
                                                    P->n_geom.as<double>());
    return cudaGetLastError();
}

cudaError_t tree_target_ranges(sfmm_plan_s* P, const uint64_t* tkeys, int64_t M)
{
    cudaError_t e;
    const int64_t nn = P->n_nodes;
    if ((e = ensure(P->n_tfirst, (size_t)nn * 4))) return e;
    if ((e = ensure(P->n_tcount, (size_t)nn * 4))) return e;
    launch_chained(k_target_ranges, grid_for(nn), 256, 0, P->stream, (int)nn, P->gm ? &P->dcnt.as<DevCounts>()->nn : nullptr,
                                                         P->n_prefix.as<uint64_t>(), P->n_level.as<int>(), tkeys, M,
                                                         P->n_tfirst.as<int>(), P->n_tcount.as<int>());
    return cudaGetLastError();
}

// The source leaves (plan->leaves_src) and the evaluation's work items (plan->items).
// Their counts stay on the device (*d_leaves, *d_items), the plan holds the
// capacities that launches over them are sized by: no host synchronisation.
// Chunks are split in two, at the price of staging a leaf's sources twice, when M
// targets make fewer full chunks than the GPU holds warps (152 SMs x 28) and most
// chunks are full (32 targets or more per node): 49,152 grid points over 447
// leaves.  Where the leaves hold about m targets each the halves only add staging
// (1e5 points at their own places: 1.80 ms whole, 1.84 ms split).
cudaError_t collect_leaves_items(sfmm_plan_s* P, int64_t M, int64_t* d_leaves, int64_t* d_items)
{
    cudaError_t e;
    const int64_t nn = P->n_nodes;
    cudaStream_t s = P->stream;
    const int split = M < 152 * 28 * (int64_t)ITEM_CHUNK && M >= 32 * nn;
    const int64_t cap = nn + M / (split ? 32 : 64) + 1;       // sum of ceilings over the leaves
    const int64_t ntiles = (nn + CTILE - 1) / CTILE;
    // the published words, then the tile counter
    const size_t wb = (size_t)(2 * ntiles + 1) * 8;
    if ((e = ensure(P->items, (size_t)cap * 8)) || (e = ensure(P->leaves_src, (size_t)nn * 4)) ||
        (e = ensure(P->cwords, wb)) || (e = cudaMemsetAsync(P->cwords.p, 0, wb, s)))
        return e;
    uint64_t* words = P->cwords.as<uint64_t>();
    launch_chained(k_collect, (unsigned)ntiles, CT, 0, s, (int)nn, P->gm ? &P->dcnt.as<DevCounts>()->nn : nullptr,
                                              P->n_child0.as<int>(), P->n_count.as<int>(), P->n_tcount.as<int>(), split,
                                              P->leaves_src.as<int>(), P->items.as<int2>(), words, d_leaves, d_items,
                                              reinterpret_cast<uint32_t*>(words + 2 * ntiles),
                                              P->opt.wait_limit > 0 ? P->opt.wait_limit : LB_POLLS);
    P->n_leaves = nn;
    P->n_items = cap;
    return cudaGetLastError();
}

}  // namespace sfmm
