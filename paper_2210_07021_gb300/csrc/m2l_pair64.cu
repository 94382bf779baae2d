// M2L (Lemma 3), P2M (Lemma 1) and the wide levels' M2M and L2L (Lemmas 2, 4) of the
// FP64 path.
//
// M2L, one thread per FMM-act pair, in the form of m2l_pair.cu: with
// u~_l = (a ph1)^l X_l and rho = g/(a b),
//     t_n = sum_{l >= n} C(l, n) u~_l,   o_l = sum_{n <= l} C(l-1, n-1) rho^n t_n,
//     Y_l = (b ph2)^l (-Q/l + o_l),      C' = C + 2 Q log sin(theta/2) + 2 Re t_0,  Q' = Q,
// both binomial sums as synthetic-division passes made of additions.  The FP64
// pipe bounds the translation (one warp instruction in about 19 cycles per SM),
// and this takes 2 p^2 + 21 p FP64 operations per pair, 87 warp instructions per
// pair at p = 32 with every lane busy; a warp per pair (its lanes' powers by
// prefix products, a multiply by a power in every term) took 185 (1e6
// clustered points, p = 32, 1.2e6 pairs: 13.3 -> 6.7 ms; 4096 points, 6488 pairs: 0.37 -> 0.10 ms).
//
// The pairs arrive grouped by target box.  A warp takes 32 consecutive pairs,
// stages their outputs in shared memory, and each lane sums one coefficient
// column over the runs of equal target.  A run that is its target's whole list
// is stored; the others go to two partial rows per warp (slot 0: a run that began
// before these 32 pairs, slot 1: one that goes on after them), which k_m2l_runs
// adds in order: no atomics, the same result every time.  Pairs with centres
// antipodal to rounding (left_out in xgeo.cuh) are listed for the warp kernel of
// expand.cu.
#include "common.cuh"
#include "dfops.cuh"
#include "xgeo.cuh"

namespace sfmm {

namespace {

constexpr int PW = 4;            // warps per CTA

// 1/l, l = 1..32
struct InvTab64 {
    double v[PMAX + 1];
};
constexpr InvTab64 make_inv64()
{
    InvTab64 t{};
    for (int l = 1; l <= PMAX; ++l) t.v[l] = 1.0 / l;
    return t;
}
__constant__ InvTab64 kInv64 = make_inv64();

__device__ __forceinline__ void cmul64(double& zr, double& zi, double xr, double xi)
{
    const double r = zr * xr - zi * xi;
    zi = zr * xi + zi * xr;
    zr = r;
}

// L lanes per pair (1 or 2): with two, each takes one part of the passes, which
// halves the time of a warp where the pairs are too few to fill the GPU.
template <int P, int L>
__global__ void __launch_bounds__(128, 3)
k_m2l_pair64(int64_t n_cap, const int64_t* d_n, const uint64_t* __restrict__ ptgt, const uint32_t* __restrict__ psrc,
             const int64_t* __restrict__ off, const XGeo* __restrict__ geo, const double* __restrict__ mpole, int p,
             double* __restrict__ local, double* __restrict__ part, uint32_t* __restrict__ leftover,
             uint32_t* __restrict__ n_left)
{
    constexpr int RS = 2 * P + 3;                 // row stride (odd: conflict-free row access)
    constexpr int CH = 32 / L;                    // pairs of a warp
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_tgt[PW][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int slot = lane / L, sub = lane % L;
    double* rows = reinterpret_cast<double*>(smem_raw) + (size_t)wid * CH * RS;
    double* row = rows + slot * RS;
    const int ncol = 2 * p + 2;
    const int64_t n_pairs = dcount(d_n, n_cap);
    for (int64_t chunk = (int64_t)blockIdx.x * nw + wid; chunk * CH < n_pairs; chunk += (int64_t)gridDim.x * nw) {
        const int64_t base = chunk * CH, k = base + slot;
        int tnode = -1;
        bool on = false;
        XGeo G;
        double rho = 0.0, C = 0.0, Q = 0.0, t0 = 0.0;
        const double* e = nullptr;
        if (k < n_pairs) {
            G = geo[k];
            tnode = (int)ptgt[k];
            on = !left_out(G);
            if (!on && sub == 0) leftover[atomicAdd(n_left, 1u)] = (uint32_t)k;
        }
        if (on) {
            rho = G.g / (G.a * G.b);
            e = mpole + (size_t)psrc[k] * EXP_STRIDE;
            C = e[0];
            Q = e[1];
            // u~_l = (a ph1)^l X_l into the row (zero for p < l <= P)
            const double ar = G.a * G.p1x, ai = G.a * G.p1y;
            double zr = ar, zi = ai;
#pragma unroll 1
            for (int l = 1; l <= P; ++l) {
                const double xr = l <= p ? e[2 * l] : 0.0, xi = l <= p ? e[2 * l + 1] : 0.0;
                if (L == 1 || sub == 0) row[2 * l] = zr * xr - zi * xi;
                if (L == 1 || sub == 1) row[2 * l + 1] = zr * xi + zi * xr;
                cmul64(zr, zi, ar, ai);
            }
            // both binomial stages, real then imaginary part (two lanes: a part each)
#pragma unroll 1
            for (int prt = sub; prt < 2; prt += L) {
                double c[P + 1];
                c[0] = 0.0;
#pragma unroll
                for (int l = 1; l <= P; ++l) c[l] = row[2 * l + prt];
                pascal_up<P>(c);
                if (prt == 0) t0 = c[0];
                double rp = rho;
#pragma unroll
                for (int n = 1; n <= P; ++n) {
                    c[n] *= rp;
                    if (n < P) rp *= rho;
                }
                pascal_down<P>(c);
#pragma unroll
                for (int l = 1; l <= P; ++l) row[2 * l + prt] = c[l];
            }
        }
        const unsigned onm = __ballot_sync(FULL, on);       // both lanes of a pair, or neither
        if (L > 1) __syncwarp();                            // each lane reads the part that the other wrote
        if (on) {
            // Y_l = (b ph2)^l (-Q/l + o_l)
            const double br = G.b * G.p2x, bi = G.b * G.p2y;
            double zr = br, zi = bi;
#pragma unroll 1
            for (int l = 1; l <= p; ++l) {
                const double orr = row[2 * l] - Q * kInv64.v[l], oi = row[2 * l + 1];
                if (L > 1) __syncwarp(onm);         // both lanes have read the pair's coefficient
                if (L == 1 || sub == 0) row[2 * l] = zr * orr - zi * oi;
                if (L == 1 || sub == 1) row[2 * l + 1] = zr * oi + zi * orr;
                cmul64(zr, zi, br, bi);
            }
            if (sub == 0) {
                row[0] = C + 2.0 * (Q * G.logk + t0);
                row[1] = Q;
            }
        } else {
            for (int c = sub; c < ncol; c += L) row[c] = 0.0;
        }
        if (sub == 0) s_tgt[wid][slot] = tnode;
        __syncwarp();
        // run sums of each coefficient column
        const int nrows = n_pairs - base < CH ? (int)(n_pairs - base) : CH;
        for (int c = lane; c < ncol; c += 32) {
            double a = 0.0;
            for (int r = 0; r < nrows; ++r) {
                a += rows[r * RS + c];
                const int t = s_tgt[wid][r];
                if (r + 1 == nrows || s_tgt[wid][r + 1] != t) {
                    const int64_t lo = off[t], hi = off[t + 1];
                    if (lo >= base && hi <= base + CH) local[(size_t)t * EXP_STRIDE + c] = a;
                    else part[(size_t)(2 * chunk + (lo < base ? 0 : 1)) * EXP_STRIDE + c] = a;
                    a = 0.0;
                }
            }
        }
        __syncwarp();
    }
}

// Locals of boxes whose list spans several warps' pairs: the sum of the partial
// rows in order; boxes without a list: zero.  One warp per box.
__global__ void __launch_bounds__(128) k_m2l_runs(TreeView T, const int64_t* __restrict__ off, int p, int ch,
                                                  const double* __restrict__ part, double* __restrict__ local)
{
    const int lane = threadIdx.x & 31;
    const int64_t nn = dcount(T.d_nn, T.n_nodes);
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < nn;
         t += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t lo = off[t], hi = off[t + 1];
        const int64_t c0 = lo / ch, c1 = (hi - 1) / ch;       // ch: pairs of a warp
        if (lo < hi && c0 == c1) continue;
        for (int c = lane; c < 2 * p + 2; c += 32) {
            double a = 0.0;
            if (lo < hi) {
                a = part[(size_t)(2 * c0 + 1) * EXP_STRIDE + c];
                for (int64_t k = c0 + 1; k <= c1; ++k) a += part[(size_t)(2 * k) * EXP_STRIDE + c];
            }
            local[(size_t)t * EXP_STRIDE + c] = a;
        }
    }
}

// few pairs or translations (one warp of single lanes for every SM sub-partition or
// less): two lanes for each, pairs in CTAs of one warp, so that they spread over the SMs'
// FP64 pipes
inline bool few_pairs(int64_t n) { return n <= 152 * 4 * 32; }

template <int P, int L>
cudaError_t launch_p(int64_t n_pairs, const int64_t* d_n, const uint64_t* ptgt, const uint32_t* psrc,
                     const int64_t* off, const XGeo* geo, const double* mpole, int p, double* local, double* part,
                     uint32_t* leftover, uint32_t* n_left, cudaStream_t s)
{
    const int nw = L == 2 ? 1 : PW, ch = 32 / L;
    const size_t smem = (size_t)nw * ch * (2 * P + 3) * sizeof(double);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_m2l_pair64<P, L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    const int64_t ctas = (n_pairs + nw * ch - 1) / (nw * ch);
    k_m2l_pair64<P, L><<<(unsigned)(ctas < (1 << 30) ? ctas : 1 << 30), nw * 32, smem, s>>>(
        n_pairs, d_n, ptgt, psrc, off, geo, mpole, p, local, part, leftover, n_left);
    count_launch();
    return cudaGetLastError();
}

// ------------------------------------------------------- M2M and L2L
// One thread per translation in the general form of expand.cu (a and b as multipliers
// of the passes: folded into the vectors they would underflow at deep levels):
//     u_l = ph1^l X_l,  v_n = sum_{l >= n} C(l, n) a^(l-n) u_l,  w_n = g^n v_n,
//     Y_l = ph2^l ( -Q b^l / l + sum_{n <= l} C(l-1, n-1) b^(l-n) w_n ),
//     C'  = C + 2 Q log k + 2 Re v_0,   Q' = Q,
// 88 FP64 warp instructions per translation at p = 32 against about 260 by a warp, which
// levels too narrow to fill the GPU keep (1e6 clustered points: M2M 1.77 -> 1.12 ms, L2L
// 2.21 -> 1.18 + 0.21 in the narrow ones; the whole call 29.4 -> 28.2 ms).  One lane
// would leave half of the sub-partitions idle at 4e3 to 2e4 nodes (1.64 and 1.72 ms);
// above that two lanes repeat the turns and cost more (4e6 points, levels over 2e4 nodes:
// 3.03 and 3.04 ms with two lanes, 2.47 and 2.59 with one).
// L lanes per translation (1 or 2, sub: this lane's): with two, each takes one part of
// the passes.  on: the lanes of the warp that translate, both of a pair or neither.
template <int P, int L>
__device__ __forceinline__ void translate_row64(double* row, int p, int sub, unsigned on, const XGeo& G, double C,
                                                double Q, double* Cout)
{
    {   // u_l, in place (the caller zeroes p < l <= P)
        double zr = G.p1x, zi = G.p1y;
#pragma unroll 1
        for (int l = 1; l <= p; ++l) {
            const double xr = row[2 * l], xi = row[2 * l + 1];
            if (L > 1) __syncwarp(on);
            if (L == 1 || sub == 0) row[2 * l] = zr * xr - zi * xi;
            if (L == 1 || sub == 1) row[2 * l + 1] = zr * xi + zi * xr;
            cmul64(zr, zi, G.p1x, G.p1y);
        }
    }
    double v0 = 0.0;
#pragma unroll 1
    for (int prt = sub; prt < 2; prt += L) {
        double c[P + 1];
        c[0] = 0.0;
#pragma unroll
        for (int l = 1; l <= P; ++l) c[l] = row[2 * l + prt];
        pascal_up_mul<P>(c, G.a);
        if (prt == 0) v0 = c[0];
        double gp = G.g;
#pragma unroll
        for (int n = 1; n <= P; ++n) {
            c[n] *= gp;
            if (n < P) gp *= G.g;
        }
        pascal_down_mul<P>(c, G.b);
#pragma unroll
        for (int l = 1; l <= P; ++l) row[2 * l + prt] = c[l];
    }
    if (L > 1) __syncwarp(on);
    {
        double zr = G.p2x, zi = G.p2y, bp = G.b;
#pragma unroll 1
        for (int l = 1; l <= p; ++l) {
            const double orr = row[2 * l] - Q * bp * kInv64.v[l], oi = row[2 * l + 1];
            if (L > 1) __syncwarp(on);
            if (L == 1 || sub == 0) row[2 * l] = zr * orr - zi * oi;
            if (L == 1 || sub == 1) row[2 * l + 1] = zr * oi + zi * orr;
            cmul64(zr, zi, G.p2x, G.p2y);
            bp *= G.b;
        }
    }
    *Cout = C + 2.0 * (Q * G.logk + v0);        // of sub == 0
}

// X_l of e into the row (zero for p < l <= P), by the translation's lanes
template <int P, int L>
__device__ __forceinline__ void ld_row64(double* row, const double* e, int p, int sub)
{
    for (int k = 2 + sub; k < 2 * P + 2; k += L) row[k] = k < 2 * p + 2 ? e[k] : 0.0;
}

// L lanes per child of a level; the four siblings' lanes sum their rows into the parent
template <int P, int L>
__global__ void __launch_bounds__(128, 3) k_m2m64(TreeView T, int c0, int c1, int lvl, int p,
                                                  const XGeo* geo, double* mpole)
{
    after_previous();
    if (T.d_level) {              // graph mode: the children are the nodes of level lvl + 1
        c0 = (int)T.d_level[lvl + 1];
        c1 = (int)T.d_level[lvl + 2];
    }
    constexpr int RS = 2 * P + 3, CH = 32 / L;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int slot = threadIdx.x / L, sub = threadIdx.x % L;
    double* rows = reinterpret_cast<double*>(smem_raw);
    double* row = rows + slot * RS;
    const int ncol = 2 * p + 2;
    const int64_t step = (int64_t)gridDim.x * (blockDim.x / L);
    // rounded up to whole warps, so that all lanes of a sibling group take part
    for (int64_t c = c0 + (int64_t)blockIdx.x * (blockDim.x / L) + slot; c - c0 < ((int64_t)(c1 - c0) + CH - 1) / CH * CH;
         c += step) {
        const bool use = c < c1 && T.count[c] > 0;
        const unsigned on = __ballot_sync(FULL, use);
        if (use) {
            const double* e = mpole + (size_t)c * EXP_STRIDE;
            ld_row64<P, L>(row, e, p, sub);
            if (L > 1) __syncwarp(on);
            double Cp;
            translate_row64<P, L>(row, p, sub, on, geo[c], e[0], e[1], &Cp);
            if (sub == 0) {
                row[0] = Cp;
                row[1] = e[1];
            }
        } else {
            for (int k = sub; k < ncol; k += L) row[k] = 0.0;
        }
        __syncwarp();
        const int r = threadIdx.x & (4 * L - 1);
        const double* g0 = rows + (slot & ~3) * RS;
        const int64_t first = c - (slot & 3);     // the group's first child
        if (first < c1) {
            double* out = mpole + (size_t)T.parent[first] * EXP_STRIDE;
            for (int k = r; k < ncol; k += 4 * L) out[k] = (g0[k] + g0[RS + k]) + (g0[2 * RS + k] + g0[3 * RS + k]);
        }
        __syncwarp();
    }
}

// L lanes per node of a level holding targets: local += the parent's local translated
template <int P, int L>
__global__ void __launch_bounds__(128, 3) k_l2l64(TreeView T, int a, int b, int lvl, int p,
                                                  const XGeo* geo, double* local)
{
    after_previous();
    if (T.d_level) {              // graph mode: the nodes of level lvl
        a = (int)T.d_level[lvl];
        b = (int)T.d_level[lvl + 1];
    }
    constexpr int RS = 2 * P + 3, CH = 32 / L;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int slot = threadIdx.x / L, sub = threadIdx.x % L;
    double* row = reinterpret_cast<double*>(smem_raw) + slot * RS;
    const int64_t step = (int64_t)gridDim.x * (blockDim.x / L);
    for (int64_t node = a + (int64_t)blockIdx.x * (blockDim.x / L) + slot;
         node - a < ((int64_t)(b - a) + CH - 1) / CH * CH; node += step) {
        const bool use = node < b && T.tcount[node] > 0 && T.parent[node] >= 0;
        const unsigned on = __ballot_sync(FULL, use);
        if (use) {
            const double* e = local + (size_t)T.parent[node] * EXP_STRIDE;
            double* out = local + (size_t)node * EXP_STRIDE;
            ld_row64<P, L>(row, e, p, sub);
            if (L > 1) __syncwarp(on);
            double Cp;
            translate_row64<P, L>(row, p, sub, on, geo[node], e[0], e[1], &Cp);
            if (L > 1) __syncwarp(on);
            if (sub == 0) {
                out[0] += Cp;
                out[1] += e[1];
            }
            for (int k = 2 + sub; k < 2 * p + 2; k += L) out[k] += row[k];
        }
        __syncwarp();
    }
}

template <int P, typename K, typename... Args>
cudaError_t level_p(K kern, int64_t n, int lanes, cudaStream_t s, Args... args)
{
    const int per = 128 / lanes;             // translations of a CTA
    const size_t smem = (size_t)per * (2 * P + 3) * sizeof(double);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    const int64_t blocks = (n + per - 1) / per;
    launch_chained(kern, (unsigned)(blocks < 152 * 16 ? blocks : 152 * 16), 128, smem, s, args...);
    return cudaGetLastError();
}

// ----------------------------------------------------------------- P2M
// One warp per leaf and one lane per source: the lane's row holds q, q log(1 - |D|^2/4)
// and q z^l, lane k then sums columns k, k + 32 and k + 64 over the leaf's sources.
// (One thread per leaf, every coefficient in its registers, was as fast on 7.7e4
// leaves, 1.09 ms, but waited for its serial chains on few: 195 leaves 0.29 -> 0.016 ms.)
constexpr double INV4PI = 0.079577471545947667884;
constexpr double LOG2 = 0.69314718055994530942;

template <int P>
__global__ void __launch_bounds__(128) k_p2m64_leaf(TreeView T, const int* __restrict__ leaves, int64_t n_cap,
                                                    const int64_t* d_nl, const double4_32a* __restrict__ src, int p,
                                                    double* __restrict__ mpole)
{
    constexpr int RS = 2 * P + 3;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double* rows = reinterpret_cast<double*>(smem_raw) + (size_t)wid * 32 * RS;
    double* row = rows + lane * RS;
    const int ncol = 2 * p + 2;
    const int64_t n_leaves = dcount(d_nl, n_cap);
    for (int64_t w = (int64_t)blockIdx.x * PW + wid; w < n_leaves; w += (int64_t)gridDim.x * PW) {
        const int node = leaves[w];
        const double* g = T.geom + (size_t)node * GEOM_STRIDE;
        const int f = T.first[node], n = T.count[node];
        double sc[3] = {0.0, 0.0, 0.0};
        for (int j0 = 0; j0 < n; j0 += 32) {
            if (j0 + lane < n) {
                const double4_32a y = src[f + j0 + lane];
                const double dx = y.x - g[0], dy = y.y - g[1], dz = y.z - g[2];
                const double d2 = dx * dx + dy * dy + dz * dz;
                const double s = 1.0 / ((2.0 - 0.5 * d2) * g[10]);       // 1/((1 + y.c) r)
                const double zr = (dx * g[3] + dy * g[4] + dz * g[5]) * s;
                const double zi = (dx * g[6] + dy * g[7] + dz * g[8]) * s;
                row[0] = y.w * log1p(-0.25 * d2);                         // 2 q log cos(theta/2)
                row[1] = y.w;
                double pr = y.w, pi = 0.0;
#pragma unroll 1
                for (int l = 1; l <= p; ++l) {
                    cmul64(pr, pi, zr, zi);
                    row[2 * l] = pr;
                    row[2 * l + 1] = pi;
                }
            }
            __syncwarp();
            const int nr = min(32, n - j0);
#pragma unroll
            for (int i = 0; i < 3; ++i)
                if (lane + 32 * i < ncol)
                    for (int r = 0; r < nr; ++r) sc[i] += rows[r * RS + lane + 32 * i];
            __syncwarp();
        }
        double* e = mpole + (size_t)node * EXP_STRIDE;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int k = lane + 32 * i;
            if (k < ncol) e[k] = k < 2 ? INV4PI * sc[i] : -INV4PI * kInv64.v[k >> 1] * sc[i];
        }
        __syncwarp();
        if (lane == 0) e[0] -= e[1] * LOG2;            // C = (1/4pi) sum q log(..) - Q log 2
        for (int k = ncol + lane; k < EXP_STRIDE; k += 32) e[k] = 0.0;
    }
}

template <int P>
cudaError_t p2m_p(const TreeView& T, const int* leaves, int64_t n_leaves, const int64_t* d_nl, const double4_32a* src,
                  int p, double* mpole, cudaStream_t s)
{
    const size_t smem = (size_t)PW * 32 * (2 * P + 3) * sizeof(double);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_p2m64_leaf<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    int64_t b = (n_leaves + PW - 1) / PW;
    if (b > 152 * 32) b = 152 * 32;
    k_p2m64_leaf<P><<<(unsigned)b, PW * 32, smem, s>>>(T, leaves, n_leaves, d_nl, src, p, mpole);
    count_launch();
    return cudaGetLastError();
}

#define SFMM_P_SWITCH(CALL)                                                                                 \
    switch ((p + 3) / 4 * 4) {                                                                              \
    case 4: return CALL(4); case 8: return CALL(8); case 12: return CALL(12); case 16: return CALL(16);     \
    case 20: return CALL(20); case 24: return CALL(24); case 28: return CALL(28); case 32: return CALL(32); \
    default: return cudaErrorInvalidValue;                                                                  \
    }

}  // namespace

// bytes of the partial rows for n pairs
size_t m2l64_part_bytes(int64_t n_pairs)
{
    const int64_t ch = few_pairs(n_pairs) ? 16 : 32;
    return (size_t)((n_pairs + ch - 1) / ch) * 2 * EXP_STRIDE * sizeof(double);
}

namespace {
cudaError_t m2l64(int64_t n_pairs, const int64_t* d_n, const uint64_t* ptgt, const uint32_t* psrc, const int64_t* off,
                  const XGeo* geo, const double* mpole, int p, double* local, double* part, uint32_t* leftover,
                  uint32_t* n_left, cudaStream_t s)
{
#define CALL(PP) few_pairs(n_pairs) ? launch_p<PP, 2>(n_pairs, d_n, ptgt, psrc, off, geo, mpole, p, local, part, \
                                                     leftover, n_left, s)                                   \
                                   : launch_p<PP, 1>(n_pairs, d_n, ptgt, psrc, off, geo, mpole, p, local, part, leftover, n_left, s)
    SFMM_P_SWITCH(CALL)
#undef CALL
}
}  // namespace

// Locals of every box = the sum of its M2Ls, but for the pairs put on the leftover list
// (*n_left of them, zero at the call).
cudaError_t launch_m2l_pair64(const TreeView& T, int64_t n_pairs, const int64_t* d_n, const uint64_t* ptgt,
                              const uint32_t* psrc, const int64_t* off, const void* geo, const double* mpole, int p,
                              double* local, double* part, uint32_t* leftover, uint32_t* n_left, cudaStream_t s)
{
    cudaError_t e;
    if (n_pairs > 0 && (e = m2l64(n_pairs, d_n, ptgt, psrc, off, static_cast<const XGeo*>(geo), mpole, p, local, part,
                                  leftover, n_left, s)))
        return e;
    int64_t b = ((int64_t)T.n_nodes + 3) / 4;
    if (b > 152 * 64) b = 152 * 64;
    k_m2l_runs<<<(unsigned)(b > 0 ? b : 1), 128, 0, s>>>(T, off, p, few_pairs(n_pairs) ? 16 : 32, part, local); count_launch();
    return cudaGetLastError();
}

// children c0..c1-1 (the nodes of level lvl + 1) -> their parents; nodes a..b-1 (level lvl).
// Graph mode: the bounds from the device, the given ones the capacity.
cudaError_t launch_m2m64(const TreeView& T, int c0, int c1, int lvl, int p, const void* geo, double* mpole,
                         cudaStream_t s)
{
    if (c1 <= c0) return cudaSuccess;
    const XGeo* G = static_cast<const XGeo*>(geo);
#define CALL(PP) few_pairs(c1 - c0) ? level_p<PP>(k_m2m64<PP, 2>, c1 - c0, 2, s, T, c0, c1, lvl, p, G, mpole) \
                                    : level_p<PP>(k_m2m64<PP, 1>, c1 - c0, 1, s, T, c0, c1, lvl, p, G, mpole)
    SFMM_P_SWITCH(CALL)
#undef CALL
}

cudaError_t launch_l2l64(const TreeView& T, int a, int b, int lvl, int p, const void* geo, double* local, cudaStream_t s)
{
    if (b <= a) return cudaSuccess;
    const XGeo* G = static_cast<const XGeo*>(geo);
#define CALL(PP) few_pairs(b - a) ? level_p<PP>(k_l2l64<PP, 2>, b - a, 2, s, T, a, b, lvl, p, G, local) \
                                  : level_p<PP>(k_l2l64<PP, 1>, b - a, 1, s, T, a, b, lvl, p, G, local)
    SFMM_P_SWITCH(CALL)
#undef CALL
}

cudaError_t launch_p2m64_leaf(const TreeView& T, const int* leaves, int64_t n_leaves, const int64_t* d_nl,
                              const double4_32a* src, int p, double* mpole, cudaStream_t s)
{
    if (n_leaves == 0) return cudaSuccess;
#define CALL(PP) p2m_p<PP>(T, leaves, n_leaves, d_nl, src, p, mpole, s)
    SFMM_P_SWITCH(CALL)
#undef CALL
}

}  // namespace sfmm
