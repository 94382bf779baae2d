// Order-29 nested HEALPix keys of unit vectors (Sec. 3.1; Gorski et al. 2005).
//
// This file is compiled with -fmad=false: every operation below is a single
// correctly rounded IEEE double operation (+, -, *, /, sqrt) in a fixed order,
// so the keys are bit-identical to any other implementation that evaluates the
// same published formulas in the same order.
//
// Azimuth, in quarter turns: octant reduction to t = min(|x|,|y|)/max(|x|,|y|);
// atan(t) from the Gregory series sum (-1)^k t^(2k+1)/(2k+1) after the
// reductions t -> (t-1)/(t+1) (adds pi/4) when t > tan(pi/8) and the
// half-angle identity atan(t) = 2 atan(t/(1+sqrt(1+t^2))), leaving
// |t| <= tan(pi/16) where 12 terms reach double precision.
// ang2pix_nest: the equatorial / polar-cap formulas of Gorski et al. (2005),
// with 1 - |z| = (x^2 + y^2)/(1 + |z|) in the caps.
//
// Fast path.  The same quantities are first computed with about 45 significant bits and
// without the FP64 pipe (FP64 arithmetic on this GPU runs at 1/64 of the FP32 rate):
// the coordinates are split into (hi, lo) FP32 pairs and compared through their bit
// patterns.  With D >= N the larger and the smaller of |x|, |y|, j = 128 N/D rounded and
// c = j/128 (exact),
//     atan(N/D) = atan(c) + atan(R),    R = (N - c D) / (D + c N),    |R| <= 1/256,
// one double-float division, atan(c) from a table, atan(R) = R - R^3/3 + R^5/5 - R^7/7.
// From there on fixed point, 2^-53 in 64 bits: octants, quadrants and the sums with
// z are exact.  In the caps sqrt(3 (x^2 + y^2)/(1 + |z|)) is an FP32 root corrected by the
// double-float residual 3 (x^2 + y^2) - s^2 (1 + |z|).  Every integer the key
// depends on is a floor of a non-negative value v (v = N_side (1/2 + tt -+ 3z/4),
// N_side tp sqrt(3(1-|z|)), ..., and tt itself in the caps); the fast path keeps
// floor(v) only when v lies at least 2^-14 from an integer.  Both its own
// error and that of the FP64 routine are below 2^-15 in these units, so the
// floors then agree; otherwise the point takes the FP64 routine above.  The
// keys are therefore those of the FP64 routine, bit for bit.  Issue-bound (about 500
// instructions per point, 36 bytes): 4e6 points 120 -> 68 us against the same quantities
// all in double-floats, with a division each for the ratio, R and 1 - |z| and
// conversions to 64-bit integers, which cost as much as FP64 instructions.
//
// The centres of a pixel grid all take the FP64 routine: a centre of N_side 2^k is a
// corner of order-29 pixels, both v's are whole.  The routine costs about 93 FP64
// instructions per point, more than half of them in three divisions, a square root, the
// comparisons and the conversions to integers.  key29_exact does these and the Gregory
// series' larger part on the integer and FP32 pipes with the same results (a correctly rounded
// quotient or root is the integer next to the exact one, which an integer remainder
// decides; products and differences are rounded from their exact bits) and leaves about
// 27 sums and products to the FP64 pipe: the 3.1e6 centres of N_side 512 600 -> 176 us.
#include "common.cuh"
#include "dfloat.cuh"

namespace sfmm {

namespace {

constexpr double TAN_PI_8 = 0.41421356237309503;
constexpr double TWO_OVER_PI = 0.6366197723675814;
constexpr double GREG0 = 1.0, GREG1 = -1.0 / 3.0, GREG2 = 1.0 / 5.0, GREG3 = -1.0 / 7.0,
                 GREG4 = 1.0 / 9.0, GREG5 = -1.0 / 11.0, GREG6 = 1.0 / 13.0, GREG7 = -1.0 / 15.0,
                 GREG8 = 1.0 / 17.0, GREG9 = -1.0 / 19.0, GREG10 = 1.0 / 21.0, GREG11 = -1.0 / 23.0;

__device__ __forceinline__ double atan_quarter_01(double t)
{
    const bool big = t > TAN_PI_8;
    const double t1 = big ? (t - 1.0) / (t + 1.0) : t;
    const double t2 = t1 / (1.0 + sqrt(1.0 + t1 * t1));
    const double s = t2 * t2;
    double p = GREG11;
    p = p * s + GREG10;
    p = p * s + GREG9;
    p = p * s + GREG8;
    p = p * s + GREG7;
    p = p * s + GREG6;
    p = p * s + GREG5;
    p = p * s + GREG4;
    p = p * s + GREG3;
    p = p * s + GREG2;
    p = p * s + GREG1;
    p = p * s + GREG0;
    const double a = (2.0 * t2) * p;
    const double v = a * TWO_OVER_PI;
    return big ? 0.5 + v : v;
}

__device__ __forceinline__ double phi_quarter(double x, double y)
{
    const double ax = fabs(x), ay = fabs(y);
    const bool swap = ay > ax;
    const double num = swap ? ax : ay;
    const double den = swap ? ay : ax;
    if (den == 0.0) return 0.0;
    const double u = atan_quarter_01(num / den);
    const double v = swap ? 1.0 - u : u;
    const bool xpos = x >= 0.0, ypos = y >= 0.0;
    double tt;
    if (xpos && ypos) tt = v;
    else if (!xpos && ypos) tt = 2.0 - v;
    else if (!xpos && !ypos) tt = 2.0 + v;
    else tt = 4.0 - v;
    return tt >= 4.0 ? tt - 4.0 : tt;
}

__device__ __forceinline__ uint64_t spread_bits(uint64_t v)
{
    v = (v | (v << 16)) & 0x0000FFFF0000FFFFull;
    v = (v | (v << 8)) & 0x00FF00FF00FF00FFull;
    v = (v | (v << 4)) & 0x0F0F0F0F0F0F0F0Full;
    v = (v | (v << 2)) & 0x3333333333333333ull;
    v = (v | (v << 1)) & 0x5555555555555555ull;
    return v;
}

__device__ __noinline__ uint64_t key29(double x, double y, double z)
{
    const int64_t ns = int64_t(1) << ORDER_MAX;
    const double nside = (double)ns;
    const double za = fabs(z);
    const double tt = phi_quarter(x, y);
    int64_t face, ix, iy;
    if (za <= 2.0 / 3.0) {
        const double temp1 = nside * (0.5 + tt);
        const double temp2 = nside * z * 0.75;
        const int64_t jp = (int64_t)(temp1 - temp2);
        const int64_t jm = (int64_t)(temp1 + temp2);
        const int64_t ifp = jp >> ORDER_MAX, ifm = jm >> ORDER_MAX;
        face = (ifp == ifm) ? (ifp | 4) : ((ifp < ifm) ? ifp : (ifm + 8));
        ix = jm & (ns - 1);
        iy = ns - (jp & (ns - 1)) - 1;
    } else {
        int64_t ntt = (int64_t)tt;
        if (ntt > 3) ntt = 3;
        const double tp = tt - (double)ntt;
        const double one_m_za = (x * x + y * y) / (1.0 + za);
        const double tmp = nside * sqrt(3.0 * one_m_za);
        int64_t jp = (int64_t)(tp * tmp);
        int64_t jm = (int64_t)((1.0 - tp) * tmp);
        if (jp > ns - 1) jp = ns - 1;
        if (jm > ns - 1) jm = ns - 1;
        if (z > 0.0) { face = ntt; ix = ns - jm - 1; iy = ns - jp - 1; }
        else         { face = ntt + 8; ix = jp; iy = jm; }
    }
    return ((uint64_t)face << (2 * ORDER_MAX)) | spread_bits((uint64_t)ix) | (spread_bits((uint64_t)iy) << 1);
}

// ------------------------------------------------------------- fast path
// Bit-pattern helpers: for finite doubles, |a| <= |b| exactly when the
// patterns with the sign cleared compare so as unsigned integers.  By the two words, so
// that no FP64 instruction (|v|, v == 0) is made of them.
__device__ __forceinline__ uint64_t abs_bits(double v)
{
    return ((uint64_t)((uint32_t)__double2hiint(v) & 0x7FFFFFFFu) << 32) | (uint32_t)__double2loint(v);
}
__device__ __forceinline__ double from_bits(uint64_t b) { return __hiloint2double((int)(b >> 32), (int)(uint32_t)b); }
__device__ __forceinline__ bool nonneg(double v)        // v >= 0.0 (true for -0.0 too)
{
    return __double2hiint(v) >= 0 || (((uint32_t)__double2hiint(v) << 1) | (uint32_t)__double2loint(v)) == 0;
}
// Conversions between integers and FP32 by the bits of x + 2^23 (0 <= x < 2^23) or
// x + 3 2^22 (|x| <= 2^22, rounding to nearest): the conversion instructions take as
// long as FP64 ones (FP32 -> integer) or a quarter of that.
__device__ __forceinline__ float float23(uint32_t v) { return __fsub_rn(__uint_as_float(v | 0x4B000000u), 8388608.f); }
__device__ __forceinline__ int round22(float x, float* whole)
{
    const float t = __fadd_rn(x, 12582912.f);
    *whole = __fsub_rn(t, 12582912.f);
    return __float_as_int(t) - 0x4B400000;
}
// bits 28 .. 6 of a significand (the rest of its FP32 part) plus half a unit of bit 6, in
// these units
__device__ __forceinline__ float sig_low(uint32_t l) { return __fsub_rn(__uint_as_float(((l >> 6) & 0x7FFFFFu) | 0x4B000000u), 8388607.5f); }

// |v| below 2^3 as (hi, lo): hi = the leading 24 bits of the significand (truncated),
// lo = the next 23 (relative error 2^-47).  Values below 2^-60 give 0 (the callers only
// need them to 2^-60 absolute).
__device__ __forceinline__ dflt dfl_from_abs(uint64_t b)
{
    const uint32_t h = (uint32_t)(b >> 32), l = (uint32_t)b;
    if (h < (1023u - 60) << 20) return dflt(0.f, 0.f);
    // exponent + 127 - 1023: adding 2^30 to the field moved to bit 23, mod 2^32
    const float hi = __uint_as_float(__funnelshift_l(l, h, 3) + 0x40000000u);
    return dflt(hi, __fmul_rn(sig_low(l), __uint_as_float(((h >> 20) - (1023 + 46 - 127)) << 23)));
}

// FP32 + FP32 of |h| < 2 and |l| <= 2^-23 -> units of 2^-52
__device__ __forceinline__ int64_t fixed52(float h, float l)
{
    const float a = __fmul_rn(h, 2097152.f);
    float w, w2, w3;
    const int k = round22(a, &w);
    const float f = __fmul_rn(__fadd_rn(__fsub_rn(a, w), __fmul_rn(l, 2097152.f)), 32768.f);     // below 2^15
    const int k2 = round22(f, &w2);
    const int k3 = round22(__fmul_rn(__fsub_rn(f, w2), 65536.f), &w3);
    return ((int64_t)k << 31) + (k2 * 65536 + k3);
}

// atan(j/128) as (hi, lo): atan t = t sum_k (prod_{i <= k} 2i/(2i+1)) t'^k / (1 + t^2), t' = t^2/(1 + t^2)
// (Euler's series)
struct AtanTab {
    float h[129], l[129];
};
constexpr AtanTab make_atan_tab()
{
    AtanTab T{};
    for (int j = 0; j <= 128; ++j) {
        const double t = j / 128.0, y = t * t / (1.0 + t * t);
        double term = t / (1.0 + t * t), sum = 0.0;
        for (int k = 1; term > 1e-20; ++k) {
            sum += term;
            term *= y * (2.0 * k) / (2.0 * k + 1.0);
        }
        T.h[j] = (float)sum;
        T.l[j] = (float)(sum - (double)T.h[j]);
    }
    return T;
}
__device__ constexpr AtanTab kAtan = make_atan_tab();
constexpr float TWO_OVER_PI_H = (float)TWO_OVER_PI, TWO_OVER_PI_L = (float)(TWO_OVER_PI - (double)(float)TWO_OVER_PI);

// 16 bits to the even positions of 32
__device__ __forceinline__ uint32_t spread16(uint32_t v)
{
    v = (v | (v << 8)) & 0x00FF00FFu;
    v = (v | (v << 4)) & 0x0F0F0F0Fu;
    v = (v | (v << 2)) & 0x33333333u;
    return (v | (v << 1)) & 0x55555555u;
}
// the key from floor(v) of both v's, in the equatorial belt and in the caps (there clamped
// to N_side - 1, ntt: the quadrant)
__device__ __forceinline__ uint64_t key_from_floors(bool cap, uint32_t jp, uint32_t jm, uint32_t ntt, bool north)
{
    const uint32_t top = (1u << ORDER_MAX) - 1;
    uint32_t ix, iy, face;
    if (cap) {
        jp = min(jp, top);
        jm = min(jm, top);
        ix = north ? top - jm : jp;
        iy = north ? top - jp : jm;
        face = north ? ntt : ntt + 8;
    } else {
        const uint32_t ifp = jp >> ORDER_MAX, ifm = jm >> ORDER_MAX;
        face = (ifp == ifm) ? (ifp | 4) : ((ifp < ifm) ? ifp : (ifm + 8));
        ix = jm & top;
        iy = ~jp & top;
    }
    const uint32_t lo = spread16(ix & 0xFFFFu) | (spread16(iy & 0xFFFFu) << 1);
    const uint32_t hi = spread16(ix >> 16) | (spread16(iy >> 16) << 1) | (face << (2 * ORDER_MAX - 32));
    return ((uint64_t)hi << 32) | lo;
}

constexpr int FX = 53, VF = FX - ORDER_MAX;                   // fraction bits of tt and of the v's
constexpr uint64_t FX_ONE = uint64_t(1) << FX, FX_MARGIN = uint64_t(1) << (VF - 14);

// v (VF fraction bits) at least 2^-14 from an integer
__device__ __forceinline__ bool floor_safe(uint64_t v)
{
    return (((uint32_t)v + (uint32_t)FX_MARGIN) & ((1u << VF) - 1)) >= 2 * (uint32_t)FX_MARGIN;
}

// Order-29 key by the fast path; false when a floor decision is too close to call
// or the point is not one of moderate size (the caller then uses key29_exact).
__device__ __forceinline__ bool key29_fast(double x, double y, double z, uint64_t* key)
{
    const uint64_t bx = abs_bits(x), by = abs_bits(y), bz = abs_bits(z);
    const bool swap = by > bx;                                        // |y| > |x|
    const uint64_t bnum = swap ? bx : by, bden = swap ? by : bx;
    // |x|, |y|, |z| below 4 (and no NaN), one of x, y at least 2^-60
    const uint32_t hd = (uint32_t)(bden >> 32);
    if (hd - ((1023u - 60) << 20) >= (62u << 20) || (uint32_t)(bz >> 32) >= (1025u << 20)) return false;
    const dflt N = dfl_from_abs(bnum), D = dfl_from_abs(bden);
    float cj;
    const int j = round22(fminf(__fdividef(__fmul_rn(N.h, 128.f), D.h), 128.f), &cj);
    const float c = __fmul_rn(cj, 1.f / 128.f);
    uint64_t tt;
    {
        // N - c D and D + c N
        const float p = __fmul_rn(D.h, c), pl = __fmaf_rn(D.l, c, __fmaf_rn(D.h, c, -p));
        const dflt n = dfl_two_sum(N.h, -p);
        const float nl = __fadd_rn(n.l, __fsub_rn(N.l, pl));
        const float g = __fmul_rn(N.h, c), gl = __fmaf_rn(N.l, c, __fmaf_rn(N.h, c, -g));
        const dflt d = dfl_fast_two_sum(D.h, g);
        const float dl = __fadd_rn(d.l, __fadd_rn(D.l, gl));
        const float inv = __fdividef(1.f, d.h);
        const float q1 = __fmul_rn(n.h, inv);
        const float q2 = __fmul_rn(__fmaf_rn(-q1, dl, __fadd_rn(__fmaf_rn(-q1, d.h, n.h), nl)), inv);
        const float r = __fadd_rn(q1, q2), r2 = __fmul_rn(r, r);
        const float tail = __fmul_rn(__fmul_rn(r, r2), __fmaf_rn(r2, __fmaf_rn(r2, -1.f / 7.f, 0.2f), -1.f / 3.f));
        const dflt A = dfl_fast_two_sum(kAtan.h[j], q1);
        const float al = __fadd_rn(__fadd_rn(q2, tail), __fadd_rn(A.l, kAtan.l[j]));
        const float u = __fmul_rn(A.h, TWO_OVER_PI_H);                // quarter turns, [0, 1/2]
        const float ul = __fmaf_rn(A.h, TWO_OVER_PI_L, __fmaf_rn(al, TWO_OVER_PI_H, __fmaf_rn(A.h, TWO_OVER_PI_H, -u)));
        uint64_t v = (uint64_t)fixed52(u, ul) * 2;
        if (swap) v = FX_ONE - v;
        const bool xpos = nonneg(x), ypos = nonneg(y);
        tt = (xpos ? (ypos ? 0 : 4 * FX_ONE) : 2 * FX_ONE) + (xpos == ypos ? v : 0 - v);
    }
    // tt wraps from 4 to 0 at phi = 2 pi: too close to the wrap, let the FP64 routine decide
    // (a tt of the fast path just below 0 is caught here too)
    if (tt >= 4 * FX_ONE - (FX_ONE >> 30)) return false;
    uint64_t vp, vm;
    uint32_t ntt = 0;
    const bool cap = bz > 0x3FE5555555555555ull;                     // |z| > 2/3 (the FP64 constant)
    if (!cap) {
        const int sh = min(1075 - FX - (int)(bz >> 52), 63);
        const uint64_t m = (bz & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
        uint64_t Z = (3 * m >> sh) >> 2;
        if (!nonneg(z)) Z = 0 - Z;
        vp = FX_ONE / 2 + tt - Z;
        vm = FX_ONE / 2 + tt + Z;
    } else {
        ntt = (uint32_t)(tt >> FX);
        const uint64_t tp = tt & (FX_ONE - 1);
        if (tp - FX_MARGIN >= FX_ONE - 2 * FX_MARGIN) return false;
        // S = 3 (x^2 + y^2) and 1 + |z|
        const float d2 = __fmul_rn(D.h, D.h), n2 = __fmul_rn(N.h, N.h);
        const float dl = __fmaf_rn(__fadd_rn(D.h, D.h), D.l, __fmaf_rn(D.h, D.h, -d2));
        const float nl = __fmaf_rn(__fadd_rn(N.h, N.h), N.l, __fmaf_rn(N.h, N.h, -n2));
        const dflt q = dfl_fast_two_sum(d2, n2);
        const float S = __fmul_rn(q.h, 3.f);
        const float Sl = __fmaf_rn(__fadd_rn(q.l, __fadd_rn(dl, nl)), 3.f, __fmaf_rn(q.h, 3.f, -S));
        const dflt zd = dfl_from_abs(bz);
        const dflt o = zd.h > 1.f ? dfl_fast_two_sum(zd.h, 1.f) : dfl_fast_two_sum(1.f, zd.h);
        const float ol = __fadd_rn(o.l, zd.l);
        // s0 = sqrt(S / o) to FP32, then the residual S - s0^2 o
        float inv = __fdividef(1.f, o.h);
        inv = __fmaf_rn(inv, __fmaf_rn(-inv, o.h, 1.f), inv);
        const float w = __fmul_rn(S, inv), y0 = rsqrtf(w);
        float s0 = __fmul_rn(w, y0);
        const float hy = __fmul_rn(0.5f, y0);
        s0 = __fmaf_rn(__fmaf_rn(-s0, s0, w), hy, s0);
        if (!(s0 < 1.5f)) return false;
        const float e = __fmul_rn(s0, s0), ee = __fmaf_rn(s0, s0, -e);
        const float P = __fmul_rn(e, o.h);
        const float Pl = __fmaf_rn(ee, o.h, __fmaf_rn(e, ol, __fmaf_rn(e, o.h, -P)));
        const float res = __fadd_rn(__fsub_rn(S, P), __fsub_rn(Sl, Pl));
        const uint64_t s = (uint64_t)fixed52(s0, __fmul_rn(res, __fmul_rn(hy, inv))) * 2;
        vp = __umul64hi(tp << (64 - FX), s);
        vm = s - vp;
    }
    *key = key_from_floors(cap, (uint32_t)(vp >> VF), (uint32_t)(vm >> VF), ntt, nonneg(z));
    return floor_safe(vp) && floor_safe(vm);
}

// ------------------------------------------------- the FP64 routine's values
// |v| of a finite double as significand and exponent: v = m 2^(e - 1075), m in [2^52, 2^53)
__device__ __forceinline__ uint64_t sig_bits(uint64_t b) { return (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull; }

// m 2^-52 of m in [2^52, 2^53) as a double-float (to 2^-47)
__device__ __forceinline__ dflt dfl_from_sig(uint64_t m)
{
    const float hi = __uint_as_float(((uint32_t)(m >> 29) & 0x7FFFFFu) | 0x3F800000u);
    return dfl_fast_two_sum(hi, __fmul_rn(sig_low((uint32_t)m), 1.f / 70368744177664.f));
}
// h + l -> units of 2^-sh (sh = 52 or 53) to about 2^8 of them: h in [1/2, 2], |l| <= 2^-24 h
__device__ __forceinline__ uint64_t sig_estimate(dflt v, int sh)
{
    const uint32_t b = __float_as_uint(v.h);
    const uint64_t h = (uint64_t)((b & 0x7FFFFFu) | 0x800000u) << ((b >> 23) - 126 + sh - 24);
    float w;
    return h + ((int64_t)round22(__fmul_rn(v.l, sh == 52 ? 17592186044416.f : 35184372088832.f), &w) << 8);
}

// a / b, correctly rounded, for b and a (or a = 0) of exponents that keep the quotient
// normal.  q = ma 2^sh / mb lies in [2^52, 2^53); the double-float quotient gives it to
// 2^10, the remainder ma 2^sh - q mb (below 2^63, so its low 64 bits are all of it) the
// rest.  A quotient of two 53-bit numbers is never halfway between two others.
__device__ __forceinline__ double div_rn(double a, double b)
{
    const uint64_t ba = abs_bits(a), bb = abs_bits(b);
    if (ba == 0) return 0.0;
    const uint64_t ma = sig_bits(ba), mb = sig_bits(bb);
    const bool ge = ma >= mb;
    const int sh = ge ? 52 : 53;
    const dflt A = dfl_from_sig(ma), B = dfl_from_sig(mb);
    float inv = __fdividef(1.f, B.h);
    inv = __fmaf_rn(inv, __fmaf_rn(-inv, B.h, 1.f), inv);
    const float q1 = __fmul_rn(A.h, inv);
    const dflt T = dfl_fast_two_sum(q1, __fmul_rn(__fmaf_rn(-q1, B.l, __fadd_rn(__fmaf_rn(-q1, B.h, A.h), A.l)), inv));
    uint64_t q = sig_estimate(T, sh);
    int64_t r = (int64_t)((ma << sh) - q * mb);
    float w;
    const int d = round22(__fdividef((float)(int)(r >> 32), float23((uint32_t)(mb >> 32))), &w);
    q += (int64_t)d;
    r -= (int64_t)((uint64_t)(int64_t)d * mb);              // |r| below 0.51 mb
    q += (uint64_t)(2 * r > (int64_t)mb) - (uint64_t)(2 * r < -(int64_t)mb);
    const uint64_t e = (ba >> 52) - (bb >> 52) + (ge ? 1023 : 1022);
    return from_bits((e << 52) + (q - 0x0010000000000000ull));
}

// sqrt(a), correctly rounded, for a normal a > 0: s = sqrt(m 2^52) in [2^52, 2^53) likewise
__device__ __forceinline__ double sqrt_rn(double a)
{
    const uint64_t ba = abs_bits(a);
    const int e = (int)(ba >> 52) - 1023;
    const uint64_t m = sig_bits(ba) << (e & 1);
    const dflt a1 = dfl_from_sig(sig_bits(ba));
    const float two = (e & 1) ? 2.f : 1.f, ah = __fmul_rn(a1.h, two), al = __fmul_rn(a1.l, two);
    const float s0 = sqrtf(ah), e2 = __fmul_rn(s0, s0);         // one correction from the residual a - s0^2
    const float res = __fadd_rn(__fsub_rn(__fsub_rn(ah, e2), __fmaf_rn(s0, s0, -e2)), al);
    int64_t s = (int64_t)sig_estimate(dfl_fast_two_sum(s0, __fdividef(res, __fadd_rn(s0, s0))), 52);
    int64_t r = (int64_t)((m << 52) - (uint64_t)s * (uint64_t)s);
    float w;
    const int64_t d = round22(__fdividef((float)(int)(r >> 32), float23((uint32_t)(s >> 31))), &w);
    r -= (2 * s + d) * d;
    s += d;
    s += (int64_t)(r > s) - (int64_t)(r <= -s);
    return from_bits(((uint64_t)(1022 + ((e - (e & 1)) >> 1)) << 52) + (uint64_t)s);
}

// x = m 2^e, m in [2^52, 2^53]
struct Soft {
    uint64_t m;
    int e;
};
__host__ __device__ constexpr Soft soft(uint64_t b)
{
    return Soft{(b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull, (int)(b >> 52) - 1075};
}

// a b, rounded to nearest even (m < 2^53): the top 64 bits of the 106-bit product, the
// others as one sticky bit
__device__ __forceinline__ Soft soft_mul(Soft a, Soft b)
{
    const uint64_t A = a.m << 11, B = b.m << 11;
    uint64_t hi = __umul64hi(A, B);
    const bool top = hi >> 63;
    hi = (top ? hi : hi << 1) | (A * B != 0);
    const uint32_t low = (uint32_t)hi & 0x7FFu;
    return Soft{(hi >> 11) + ((low + 0x3FFu + ((uint32_t)(hi >> 11) & 1u)) >> 11), a.e + b.e + (top ? 53 : 52)};
}

// c - x, rounded to nearest even, for x < c/2: ten guard bits, the last one sticky (odd
// when anything lies below it, so neither a tie nor exact)
__device__ __forceinline__ Soft soft_sub(Soft c, Soft x)
{
    const int d = min(c.e - x.e, 63);
    const uint64_t X = x.m << 10;
    uint64_t xs = X >> d;
    xs |= (xs << d) != X;
    uint64_t D = (c.m << 10) - xs;
    int e = c.e;
    if (!(D >> 62)) {
        D <<= 1;
        --e;
    }
    const uint64_t m = (D + 0x1FFu + ((uint32_t)(D >> 10) & 1u)) >> 10;
    const bool over = m >> 53;
    return Soft{over ? m >> 1 : m, e + over};
}

// the Gregory series' sum at s = t^2 <= tan(pi/16)^2, by Horner's rule with each product and
// each sum rounded: the terms alternate, so each step is 1/(2k+1) - s p
// its first steps on the FP64 pipe, the last GREG_SOFT on the others, which are then
// about equally busy (the 3.1e6 centres of N_side 512 with 4 / 5 / 6 / 7 / 8 / 11 of
// them: 204 / 193 / 181 / 176 / 182 / 200 us)
constexpr int GREG_SOFT = 7;
struct GregTab {
    double v[12];
};
__constant__ constexpr GregTab kGreg = {{GREG0, -GREG1, GREG2, -GREG3, GREG4, -GREG5, GREG6, -GREG7, GREG8, -GREG9, GREG10, -GREG11}};

__device__ __forceinline__ double gregory(double s)
{
    double q = kGreg.v[11];
#pragma unroll
    for (int k = 10; k >= GREG_SOFT; --k) q = kGreg.v[k] - s * q;
    const Soft S = soft(abs_bits(s));
    Soft p = soft(abs_bits(q));
#pragma unroll 1
    for (int k = GREG_SOFT - 1; k >= 0; --k) p = soft_sub(soft(abs_bits(kGreg.v[k])), soft_mul(p, S));
    return from_bits(((uint64_t)(p.e + 1074) << 52) + p.m);
}

// floor of |v| 2^sc for |v| 2^sc < 2^53
__device__ __forceinline__ int64_t trunc_scaled(double v, int sc)
{
    const uint64_t b = abs_bits(v);
    const int down = 1075 - sc - (int)(b >> 52);             // v 2^sc = m 2^-down
    return down > 52 ? 0 : (int64_t)(sig_bits(b) >> down);
}

// exponents between 2^-300 and 2^70
__device__ __forceinline__ bool mid_range(uint64_t b) { return (b >> 52) - 723u < 370u; }

// key29 with its divisions, roots, comparisons and conversions off the FP64 pipe: the
// same values in the same order.  Scaling by N_side is exact, so it is left to
// trunc_scaled.
__device__ __noinline__ uint64_t key29_exact(double x, double y, double z)
{
    const uint64_t bx = abs_bits(x), by = abs_bits(y), bz = abs_bits(z);
    const bool swap = by > bx;
    const uint64_t bnum = swap ? bx : by, bden = swap ? by : bx;
    if (!mid_range(bden) || (bnum && !mid_range(bnum)) || (bz && !mid_range(bz))) return key29(x, y, z);
    const double t = div_rn(from_bits(bnum), from_bits(bden));
    const bool big = abs_bits(t) > (uint64_t)__double_as_longlong(TAN_PI_8);
    const double t1 = big ? div_rn(1.0 - t, t + 1.0) : t;               // |t1|
    const double t2 = div_rn(t1, 1.0 + sqrt_rn(1.0 + t1 * t1));         // |t2|
    // (the factor 2 of 2 t2 is exact anywhere)
    const double w = abs_bits(t2) == 0 ? 0.0 : (t2 * gregory(t2 * t2)) * (2.0 * TWO_OVER_PI);
    double v = big ? 0.5 - w : w;                                       // t1 <= 0 where big
    if (swap) v = 1.0 - v;
    const bool xpos = nonneg(x), ypos = nonneg(y);
    double tt = v;
    if (!xpos || !ypos) tt = (xpos ? 4.0 : 2.0) + (xpos == ypos ? v : -v);
    if (abs_bits(tt) >= (uint64_t)__double_as_longlong(4.0)) tt = tt - 4.0;
    const bool cap = bz > (uint64_t)__double_as_longlong(2.0 / 3.0);
    double vp, vm;
    uint32_t ntt = 0;
    if (!cap) {
        vp = (0.5 + tt) - z * 0.75;
        vm = (0.5 + tt) + z * 0.75;
    } else {
        ntt = (uint32_t)trunc_scaled(tt, 0);                            // below 4
        const double tp = tt - (ntt > 1 ? (ntt > 2 ? 3.0 : 2.0) : (ntt > 0 ? 1.0 : 0.0));
        const double one_m_za = div_rn(x * x + y * y, 1.0 + from_bits(bz));
        const double tmp = sqrt_rn(3.0 * one_m_za);
        vp = tp * tmp;
        vm = (1.0 - tp) * tmp;
        // floors over N_side - 1 are clamped to it
        if (abs_bits(vp) > (uint64_t)__double_as_longlong(1.0)) vp = 1.0;
        if (abs_bits(vm) > (uint64_t)__double_as_longlong(1.0)) vm = 1.0;
    }
    return key_from_floors(cap, (uint32_t)trunc_scaled(vp, ORDER_MAX), (uint32_t)trunc_scaled(vm, ORDER_MAX), ntt, nonneg(z));
}

__global__ void __launch_bounds__(256) k_keys(const double* xyz, int64_t n, uint64_t* keys,
                                              uint32_t* iota)
{
    after_previous();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
        uint64_t k;
        if (!key29_fast(x, y, z, &k)) k = key29_exact(x, y, z);
        keys[i] = k;
        if (iota) iota[i] = (uint32_t)i;
    }
}

}  // namespace

cudaError_t launch_keys(const double* xyz, int64_t n, uint64_t* keys, uint32_t* iota, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    launch_chained(k_keys, (unsigned)blocks, 256, 0, s, xyz, n, keys, iota);
    return cudaGetLastError();
}

}  // namespace sfmm
