// Prefix sums across the tiles of one launch by looking back (single-pass scan
// with decoupled look-back, Merrill and Garland 2016): a tile publishes its own
// sum, adds up the sums of the tiles before it until it meets a running total,
// and publishes its own running total.  Tiles take their numbers from a counter
// in the order they start, so a tile waits only for tiles that run or are done;
// the wait is bounded all the same, and a caller whose wait ran out forms the
// sum of the earlier tiles from their inputs.
//
// A published word is 64 bits, so that state and value travel in one store and
// no fence orders them: 8 bits of epoch (the round a word belongs to: the words
// of an earlier round in the same buffer read as not published), 2 bits of
// state, 54 bits of value.  Words are zeroed before the first round.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace sfmm {

constexpr int LB_POLLS = 1 << 20;                  // default bound of a wait (about 1 us per poll)
constexpr uint64_t LB_OWN = 1ull << 54, LB_UPTO = 2ull << 54, LB_STATE = 3ull << 54, LB_VALUE = LB_OWN - 1;

__device__ __forceinline__ uint64_t lb_epoch(int round) { return (uint64_t)(round + 1) << 56; }
__device__ __forceinline__ void lb_publish(uint64_t* w, int round, uint64_t state, int64_t v)
{
    *reinterpret_cast<volatile uint64_t*>(w) = lb_epoch(round) | state | (uint64_t)v;
}

// The sum of the words of tiles 0..tile-1 (words[t * stride]), by one whole warp, 32
// tiles at a time; every lane gets the sum.  False when `limit` polls found nothing new.
__device__ __forceinline__ bool lb_before(const uint64_t* words, int stride, int64_t tile, int round, int limit,
                                          int64_t* before)
{
    const int lane = threadIdx.x & 31;
    int64_t sum = 0;
    int polls = 0;
    for (int64_t top = tile - 1; top >= 0;) {
        const int64_t t = top - lane;
        uint64_t w = LB_UPTO;                      // before the first tile: a running total of zero
        bool ok = true;
        if (t >= 0) {
            w = *reinterpret_cast<const volatile uint64_t*>(words + t * stride);
            ok = (w & (0xffull << 56)) == lb_epoch(round) && (w & LB_STATE) != 0;
        }
        const unsigned okm = __ballot_sync(0xffffffffu, ok), upm = __ballot_sync(0xffffffffu, ok && (w & LB_UPTO));
        const int run = okm == 0xffffffffu ? 32 : __ffs(~okm) - 1;      // tiles published without a gap
        const int first = upm ? __ffs(upm) - 1 : 32;                    // the nearest running total
        const int take = min(run, first + 1);
        int64_t v = lane < take ? (int64_t)(w & LB_VALUE) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        sum += v;
        if (first < run) break;
        if (take == 0 && ++polls >= limit) return false;
        top -= take;
    }
    *before = sum;
    return true;
}

}  // namespace sfmm
