// Device-wide exclusive scans and a stable LSD radix sort of (u64 key, u32 value).
//
// Scan: reduce-then-scan in three launches (per-tile sums, a single-CTA scan of
// the tile sums, per-tile scans with the tile offset added).
// Sort: 8-bit digits.  One launch counts the digits of every pass (the counts do
// not depend on the order); each pass is then one launch in which a tile of
// 1024 to 4096 keys ranks its keys stably (warp ballots, per-warp digit counters),
// finds where its runs start by looking back over the tiles before it (each
// publishes its digit counts, then their running totals), reorders itself by
// digit in shared memory and writes runs of equal digits.  That is 2 + passes
// launches; a histogram, a three-launch scan and a scatter per pass, latency-bound
// at these sizes, took 5 per pass (62-bit keys: 4096 230 -> 60 us, 262,144 255 -> 109,
// 1e6 285 -> 171).  Large sorts (RS_LARGE) count per tile and pass instead, in
// three launches per pass (3.1e6 keys 433 -> 375 us; 1.6e7 1385 -> 1373).
#include "common.cuh"

#include <algorithm>

namespace sfmm {

namespace {

constexpr int SC_T = 256, SC_I = 8, SC_TILE = SC_T * SC_I;

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// block-wide exclusive scan of one value per thread (256 threads); returns the
// exclusive prefix and writes the block total to *total.
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T* s_warp, T* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = warp_incl_scan(v, lane);
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < (SC_T / 32) ? s_warp[lane] : T(0);
        T wi = warp_incl_scan(w, lane);
        if (lane < (SC_T / 32)) s_warp[lane] = wi - w;
        if (lane == (SC_T / 32) - 1) *total = wi;
    }
    __syncthreads();
    return inc - v + s_warp[warp];
}

template <typename T>
__global__ void k_scan_reduce(const T* in, int64_t n, T* bsum)
{
    after_previous();
    __shared__ T s_warp[SC_T / 32];
    __shared__ T s_total;
    const int64_t base = (int64_t)blockIdx.x * SC_TILE;
    T acc = 0;
    for (int r = 0; r < SC_I; ++r) {
        int64_t e = base + (int64_t)r * SC_T + threadIdx.x;
        if (e < n) acc += in[e];
    }
    block_excl_scan(acc, s_warp, &s_total);
    if (threadIdx.x == 0) bsum[blockIdx.x] = s_total;
}

template <typename T>
__global__ void k_scan_top(T* bsum, int64_t nb, T* total)
{
    after_previous();
    __shared__ T s_warp[SC_T / 32];
    __shared__ T s_total;
    T carry = 0;
    for (int64_t c = 0; c < nb; c += SC_T) {
        int64_t e = c + threadIdx.x;
        T v = e < nb ? bsum[e] : T(0);
        T ex = block_excl_scan(v, s_warp, &s_total);
        if (e < nb) bsum[e] = ex + carry;
        carry += s_total;
        __syncthreads();
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

template <typename T>
__global__ void k_scan_down(const T* in, T* out, int64_t n, const T* bsum)
{
    after_previous();
    __shared__ T s_tile[SC_TILE];
    __shared__ T s_warp[SC_T / 32];
    __shared__ T s_total;
    const int64_t base = (int64_t)blockIdx.x * SC_TILE;
    for (int r = 0; r < SC_I; ++r) {
        int64_t e = base + (int64_t)r * SC_T + threadIdx.x;
        s_tile[r * SC_T + threadIdx.x] = e < n ? in[e] : T(0);
    }
    __syncthreads();
    T loc[SC_I];
    T acc = 0;
    for (int i = 0; i < SC_I; ++i) { loc[i] = acc; acc += s_tile[threadIdx.x * SC_I + i]; }
    T ex = block_excl_scan(acc, s_warp, &s_total) + bsum[blockIdx.x];
    __syncthreads();
    for (int i = 0; i < SC_I; ++i) s_tile[threadIdx.x * SC_I + i] = loc[i] + ex;
    __syncthreads();
    for (int r = 0; r < SC_I; ++r) {
        int64_t e = base + (int64_t)r * SC_T + threadIdx.x;
        if (e < n) out[e] = s_tile[r * SC_T + threadIdx.x];
    }
}

template <typename T>
cudaError_t exclusive_scan_t(const T* in, T* out, int64_t n, T* total, void* tmp, cudaStream_t s)
{
    if (n <= 0) {
        if (total) return cudaMemsetAsync(total, 0, sizeof(T), s);
        return cudaSuccess;
    }
    const int64_t nb = (n + SC_TILE - 1) / SC_TILE;
    T* bsum = static_cast<T*>(tmp);
    launch_chained(k_scan_reduce<T>, (unsigned)nb, SC_T, 0, s, in, n, bsum);
    launch_chained(k_scan_top<T>, 1, SC_T, 0, s, bsum, nb, total);
    launch_chained(k_scan_down<T>, (unsigned)nb, SC_T, 0, s, in, out, n, bsum);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- radix sort
// A tile is T threads x I keys; warp w owns keys [32 I w, 32 I (w + 1)) of it, loaded
// in I coalesced rounds of 32.
constexpr size_t RS_HEAD = 8 * 256 * 4 + 256;     // digit counts and tile counters in front of the tiles' words
constexpr int LOOK = 4;                           // tiles whose words a look-back reads at once
constexpr int RS_POLLS = 1 << 20;                 // polls of a look-back that found nothing new (each about 1 us)
// Sizes at which the tile and the way to the runs' starts change (62-bit keys, us per
// sort with the neighbouring choices): keys per thread 4 below 150,000 (4096 keys:
// 58, with 8: 76, with 16: 93; 1e5: 93 / 93 / 122), 8 below 500,000 (262,144: 109,
// with 16: 126), 16 above (1e6: 171, with 8: 230).  From RS_LARGE on the tiles in
// flight are many enough that their look-backs hold one another up, and counting
// launches take over (counting / look-back: 1.5e6 262 / 228, 2e6 295 / 300, 3.1e6
// 375 / 420, 1.6e7 1373 / 1388).
constexpr int64_t RS_SMALL = 150000, RS_MIDDLE = 500000, RS_LARGE = 2000000;
constexpr int RS_WC = 257;                        // per-warp digit counters (+1 slot for keys past n)
constexpr int RS_HT = 256;                        // threads of the counting kernel
// the tile's keys, then its values, reordered through one 8-byte-per-key buffer,
// plus the digit of every reordered slot
constexpr size_t rs_smem_bytes(int T, int I) { return (size_t)T * I * 9 + (size_t)(T / 32) * RS_WC * 4 + 2 * 256 * 4 + 64; }

// A tile's published word per digit (sorts below RS_LARGE keys): its own count of
// the digit, or the count of all keys up to and including the tile, with the flag
// in the top two bits.  One store carries both, so no fence orders them; zero
// means not published yet.
constexpr uint32_t RS_OWN = 1u << 30, RS_UPTO = 2u << 30, RS_COUNT = RS_OWN - 1;
static_assert(RS_LARGE < (int64_t)RS_COUNT, "counts and flags share a word");
__device__ __forceinline__ uint32_t ld_word(const uint32_t* p) { return *reinterpret_cast<const volatile uint32_t*>(p); }
__device__ __forceinline__ void st_word(uint32_t* p, uint32_t v) { *reinterpret_cast<volatile uint32_t*>(p) = v; }

// the digit counts of every pass: hist[pass][digit], zero at launch
__global__ void __launch_bounds__(RS_HT) k_rs_hist(const uint64_t* keys, int64_t n, int passes,
                                                  uint32_t* hist)
{
    after_previous();
    __shared__ uint32_t cnt[8][256];
    for (int i = threadIdx.x; i < 8 * 256; i += RS_HT) (&cnt[0][0])[i] = 0;
    __syncthreads();
    for (int64_t e = (int64_t)blockIdx.x * RS_HT + threadIdx.x; e < n; e += (int64_t)gridDim.x * RS_HT) {
        const uint64_t k = keys[e];
        for (int p = 0; p < passes; ++p) atomicAdd(&cnt[p][(k >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += RS_HT)
        if (const uint32_t c = (&cnt[0][0])[i]) atomicAdd(hist + i, c);
}

// exclusive prefix sum of one value per thread over the block's 256 threads
__device__ __forceinline__ uint32_t block_excl256(uint32_t v, uint32_t* s_warp, int lane, int warp)
{
    const uint32_t inc = warp_incl_scan(v, lane);
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < 7; ++w) before += w < warp ? s_warp[w] : 0u;
    __syncthreads();
    return before + inc - v;
}

// The keys of one digit in all tiles before `tile`, by looking back: LOOK tiles'
// words are read at once and added up until one holds a running total.  Tiles
// take their numbers in the order they start, so every word waited for belongs
// to a tile that is running or done; the wait is bounded all the same, and false
// is returned when `limit` polls found nothing (the caller then counts the keys
// itself).
__device__ __forceinline__ bool look_back(const uint32_t* __restrict__ words, int64_t tile, int digit, int limit,
                                          uint32_t* before)
{
    uint32_t sum = 0;
    int polls = 0;
    for (int64_t t = tile - 1; t >= 0;) {
        uint32_t w[LOOK];
#pragma unroll
        for (int i = 0; i < LOOK; ++i) w[i] = ld_word(words + (t - i < 0 ? 0 : t - i) * 256 + digit);
        int used = 0;
        bool go = true, done = false;
#pragma unroll
        for (int i = 0; i < LOOK; ++i) {
            go = go && !done && t - i >= 0 && w[i] != 0;
            if (go) {
                sum += w[i] & RS_COUNT;
                done = (w[i] & RS_UPTO) != 0;
                used = i + 1;
            }
        }
        if (done) break;
        if (used == 0 && ++polls >= limit) return false;
        t -= used;
    }
    *before = sum;
    return true;
}

// Sorts of RS_LARGE keys and more, per pass: the tiles' digit counts,
// counts[digit][tile], then one block per digit turns its row into exclusive
// sums over the tiles and writes the digit's total.
template <int T, int I>
__global__ void __launch_bounds__(T) k_rs_tile_counts(const uint64_t* keys, int64_t n, int shift,
                                                      uint32_t* counts, int64_t ntiles)
{
    after_previous();
    __shared__ uint32_t cnt[256];
    for (int i = threadIdx.x; i < 256; i += T) cnt[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (T * I);
#pragma unroll
    for (int r = 0; r < I; ++r) {
        const int64_t e = base + (int64_t)r * T + threadIdx.x;
        if (e < n) atomicAdd(&cnt[(keys[e] >> shift) & 255u], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += T) counts[(int64_t)i * ntiles + blockIdx.x] = cnt[i];
}

__global__ void __launch_bounds__(SC_T) k_rs_rows(uint32_t* counts, int64_t ntiles,
                                                  uint32_t* totals)
{
    after_previous();
    __shared__ uint32_t s_warp[SC_T / 32];
    __shared__ uint32_t s_total;
    uint32_t* row = counts + (int64_t)blockIdx.x * ntiles;
    uint32_t carry = 0;
    for (int64_t c = 0; c < ntiles; c += SC_TILE) {
        uint32_t v[SC_I], acc = 0;
        const int64_t e0 = c + (int64_t)threadIdx.x * SC_I;
#pragma unroll
        for (int i = 0; i < SC_I; ++i) v[i] = e0 + i < ntiles ? row[e0 + i] : 0u;
#pragma unroll
        for (int i = 0; i < SC_I; ++i) { const uint32_t x = v[i]; v[i] = acc; acc += x; }
        const uint32_t ex = block_excl_scan(acc, s_warp, &s_total) + carry;
#pragma unroll
        for (int i = 0; i < SC_I; ++i)
            if (e0 + i < ntiles) row[e0 + i] = v[i] + ex;
        carry += s_total;
        __syncthreads();
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// One tile: stable rank of every key among the tile's keys of its digit
// (warp-private counters advanced round by round; within a round the lanes of
// equal digit are found with eight ballots, one per digit bit), counts turned
// into per-warp offsets by a scan over (digit, warp), the start of each digit's
// run from the look-back, then the tile's keys and afterwards its values
// reordered by digit through one shared buffer and written out as runs per
// digit.  Only the digits (packed four to a register) and the
// ranks stay in registers between the phases; keys and values are read again
// (from L2) when they are reordered, which keeps four CTAs on an SM.
// words: this pass's published words (zero at launch), words_next: the next
// pass's, zeroed here tile by tile; ticket: this pass's tile counter (zero).
// LOOKB: the runs' starts by looking back (words, words_next, ticket, limit); else
// from the tiles' counts (words: their exclusive sums per digit row, limit: the
// tiles).  hist: the digits' totals in either case.
template <int RS_T, int RS_I, int CTAS, bool LOOKB>
__global__ void __launch_bounds__(RS_T, CTAS) k_rs_pass(const uint64_t* kin, const uint32_t* vin,
                                                    uint64_t* kout, uint32_t* vout,
                                                    int64_t n, int shift, const uint32_t* hist,
                                                    uint32_t* words, uint32_t* words_next,
                                                    uint32_t* ticket, int limit)
{
    after_previous();
    static_assert(RS_T == 256, "one thread per digit");
    constexpr int RS_TILE = RS_T * RS_I, RS_W = RS_T / 32;
    extern __shared__ __align__(16) unsigned char rs_smem[];
    uint64_t* sk = reinterpret_cast<uint64_t*>(rs_smem);
    uint32_t* sv = reinterpret_cast<uint32_t*>(rs_smem);   // the same bytes, once the keys are out
    uint32_t* wc = reinterpret_cast<uint32_t*>(sk + RS_TILE);   // [RS_W][RS_WC]
    uint32_t* tbase = wc + RS_W * RS_WC;                  // tile-local start of each digit
    uint32_t* gbase = tbase + 256;                        // global start of this tile's keys of each digit
    uint32_t* s_warp = gbase + 256;                       // scan scratch
    uint8_t* sdig = reinterpret_cast<uint8_t*>(s_warp + 16);   // digit of each reordered slot
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ uint32_t s_tile;
    __shared__ int s_lost;
    if (LOOKB) {
        if (tid == 0) {
            s_tile = atomicAdd(ticket, 1u);
            s_lost = 0;
        }
        __syncthreads();
    }
    const uint32_t tile = LOOKB ? s_tile : blockIdx.x;
    const int64_t tile0 = (int64_t)tile * RS_TILE;
    const int64_t w0 = tile0 + (int64_t)warp * (32 * RS_I);
    uint32_t dig[RS_I / 4];                               // digits, four to a register
    uint32_t loc[RS_I / 2];                               // slots (< 2^13), two to a register
#pragma unroll
    for (int r = 0; r < RS_I / 4; ++r) dig[r] = 0u;
#pragma unroll
    for (int r = 0; r < RS_I / 2; ++r) loc[r] = 0u;
#pragma unroll
    for (int r = 0; r < RS_I; ++r) {
        const int64_t e = w0 + r * 32 + lane;
        const uint32_t d = e < n ? (uint32_t)((kin[e] >> shift) & 255u) : 0u;
        dig[r >> 2] |= d << (8 * (r & 3));
    }
    for (int d = lane; d < RS_WC; d += 32) wc[warp * RS_WC + d] = 0;
    uint32_t* mine = words + (size_t)tile * 256 + tid;    // thread tid owns digit tid
    if (LOOKB) {
        // the tile's digit counts, published before the ranking so that later tiles find them
        words_next[(size_t)tile * 256 + tid] = 0;
        gbase[tid] = 0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < RS_I; ++r)
            if (w0 + r * 32 + lane < n) atomicAdd(&gbase[(dig[r >> 2] >> (8 * (r & 3))) & 255u], 1u);
        __syncthreads();
        if (tile > 0) st_word(mine, RS_OWN | gbase[tid]);
    } else {
        gbase[tid] = words[(size_t)tid * (unsigned)limit + (unsigned)tile];
    }
    __syncwarp();
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < RS_I; ++r) {
        const int64_t e = w0 + r * 32 + lane;
        const bool in = e < n;
        const int d = in ? (int)((dig[r >> 2] >> (8 * (r & 3))) & 255u) : 256;
        // lanes holding the same digit (keys past n: their own slot 256)
        unsigned peers = __ballot_sync(FULL, !in);
        peers = in ? ~peers : peers;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const unsigned m = __ballot_sync(FULL, (d >> b) & 1);
            peers &= ((d >> b) & 1) ? m : ~m;
        }
        const uint32_t before = wc[warp * RS_WC + d];
        __syncwarp();
        if ((peers & lt) == 0) wc[warp * RS_WC + d] = before + (uint32_t)__popc(peers);
        loc[r >> 1] |= (before + (uint32_t)__popc(peers & lt)) << (16 * (r & 1));
        __syncwarp();
    }
    __syncthreads();
    // thread tid = digit: per-warp exclusive offsets, then the tile's digit starts
    uint32_t tot = 0;
#pragma unroll
    for (int w = 0; w < RS_W; ++w) {
        const uint32_t c = wc[w * RS_WC + tid];
        wc[w * RS_WC + tid] = tot;
        tot += c;
    }
    tbase[tid] = block_excl256(tot, s_warp, lane, warp);
    const uint32_t run0 = block_excl256(hist[tid], s_warp, lane, warp);     // the digit's first place
    if (LOOKB) {
        uint32_t before = 0;
        if (!look_back(words, tile, tid, limit, &before)) s_lost = 1;
        __syncthreads();
        if (s_lost) {       // a wait ran out: count the keys before this tile directly
            gbase[tid] = 0;
            __syncthreads();
            for (int64_t e = tid; e < tile0; e += RS_T) atomicAdd(&gbase[(kin[e] >> shift) & 255u], 1u);
            __syncthreads();
            before = gbase[tid];
        }
        st_word(mine, RS_UPTO | (before + tot));
        gbase[tid] = run0 + before;
    } else {
        gbase[tid] += run0;
    }
    __syncthreads();
    // keys to their places in the tile's digit order (read again, from L2)
#pragma unroll
    for (int r = 0; r < RS_I; ++r) {
        const int64_t e = w0 + r * 32 + lane;
        if (e < n) {
            const int d = (int)((dig[r >> 2] >> (8 * (r & 3))) & 255u);
            loc[r >> 1] += (tbase[d] + wc[warp * RS_WC + d]) << (16 * (r & 1));
            const uint32_t slot = (loc[r >> 1] >> (16 * (r & 1))) & 0xFFFFu;
            sk[slot] = kin[e];
            sdig[slot] = (uint8_t)d;
        }
    }
    __syncthreads();
    // runs of equal digits go to consecutive global positions: keys, then values
    const int cnt = (int)((n - tile0) < RS_TILE ? (n - tile0) : RS_TILE);
    for (int i = tid; i < cnt; i += RS_T) {
        const int d = sdig[i];
        kout[gbase[d] + (uint32_t)i - tbase[d]] = sk[i];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_I; ++r) {
        const int64_t e = w0 + r * 32 + lane;
        if (e < n) sv[(loc[r >> 1] >> (16 * (r & 1))) & 0xFFFFu] = vin[e];
    }
    __syncthreads();
    for (int i = tid; i < cnt; i += RS_T) {
        const int d = sdig[i];
        vout[gbase[d] + (uint32_t)i - tbase[d]] = sv[i];
    }
}

inline int64_t rs_tile(int64_t n) { return n <= RS_SMALL ? 256 * 4 : n <= RS_MIDDLE ? 256 * 8 : 256 * 16; }

}  // namespace

size_t scan_tmp_bytes(int64_t n)
{
    int64_t nb = (n + SC_TILE - 1) / SC_TILE + 1;
    return (size_t)nb * sizeof(int64_t) + 256;
}

cudaError_t exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* total, void* tmp, cudaStream_t s)
{
    return exclusive_scan_t<int64_t>(in, out, n, total, tmp, s);
}

// the digit counts of 8 passes and the tile counters, then the tiles' words of even
// and of odd passes (counting sorts use the first half); never decreasing in n (a
// buffer sized for n serves every smaller sort)
size_t radix_tmp_bytes(int64_t n)
{
    auto need = [](int64_t m) {
        const int64_t ntiles = (m + rs_tile(m) - 1) / rs_tile(m);
        return RS_HEAD + (size_t)(2 * ntiles) * 256 * sizeof(uint32_t) + 512;
    };
    size_t b = need(n);
    if (n > RS_SMALL) b = std::max(b, need(RS_SMALL));
    if (n > RS_MIDDLE) b = std::max(b, need(RS_MIDDLE));
    return b;
}

namespace {

template <int I, bool LOOKB>
cudaError_t radix_sort_t(uint64_t* k1, uint32_t* v1, uint64_t* k2, uint32_t* v2, int64_t n, int bits, void* tmp,
                         cudaStream_t s, bool* in_alt, int limit)
{
    constexpr int T = 256;
    const int64_t ntiles = (n + T * I - 1) / (T * I);
    const int passes = (bits + 7) / 8;
    constexpr size_t smem = rs_smem_bytes(T, I);
    uint32_t* hist = reinterpret_cast<uint32_t*>((reinterpret_cast<uintptr_t>(tmp) + 255) & ~uintptr_t(255));
    uint32_t* tickets = hist + 8 * 256;
    uint32_t* words[2];
    words[0] = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(hist) + RS_HEAD);
    words[1] = words[0] + ntiles * 256;
    uint64_t *ka = k1, *kb = k2;
    uint32_t *va = v1, *vb = v2;
    bool alt = false;
    cudaError_t e;
    auto* pass = k_rs_pass<T, I, 4, LOOKB>;
    if ((e = cudaFuncSetAttribute(pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    if (LOOKB) {
        if ((e = cudaMemsetAsync(hist, 0, RS_HEAD + (size_t)ntiles * 256 * sizeof(uint32_t), s))) return e;
        const int64_t hb = (n + RS_HT * 8 - 1) / (RS_HT * 8);
        launch_chained(k_rs_hist, (unsigned)(hb < 152 * 8 ? hb : 152 * 8), RS_HT, 0, s, ka, n, passes, hist);
    }
    for (int p = 0; p < passes; ++p) {
        if constexpr (!LOOKB) {
            launch_chained(k_rs_tile_counts<T, I>, (unsigned)ntiles, T, 0, s, ka, n, 8 * p, words[0], ntiles);
            launch_chained(k_rs_rows, 256, SC_T, 0, s, words[0], ntiles, hist + 256 * p);
        }
        uint32_t *w = words[LOOKB ? p & 1 : 0], *wn = words[(p + 1) & 1];
        launch_chained(pass, (unsigned)ntiles, T, smem, s, ka, va, kb, vb, n, 8 * p, hist + 256 * p, w, wn, tickets + p,
                       LOOKB ? limit : (int)ntiles);
        std::swap(ka, kb);
        std::swap(va, vb);
        alt = !alt;
    }
    *in_alt = alt;
    return cudaGetLastError();
}

}  // namespace

cudaError_t radix_sort(uint64_t* k1, uint32_t* v1, uint64_t* k2, uint32_t* v2, int64_t n, int bits,
                       void* tmp, cudaStream_t s, bool* in_alt, int wait_limit)
{
    *in_alt = false;
    if (n <= 1 || bits <= 0) return cudaSuccess;
    const int limit = wait_limit > 0 ? wait_limit : RS_POLLS;
    if (n <= RS_SMALL) return radix_sort_t<4, true>(k1, v1, k2, v2, n, bits, tmp, s, in_alt, limit);
    if (n <= RS_MIDDLE) return radix_sort_t<8, true>(k1, v1, k2, v2, n, bits, tmp, s, in_alt, limit);
    if (n < RS_LARGE) return radix_sort_t<16, true>(k1, v1, k2, v2, n, bits, tmp, s, in_alt, limit);
    return radix_sort_t<16, false>(k1, v1, k2, v2, n, bits, tmp, s, in_alt, limit);
}

}  // namespace sfmm
