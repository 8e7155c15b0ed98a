// pairs_fixed.cuh -- integer accumulation of the plain (FP64) neighbour sums.
//
// On GB300 an FP64 operation occupies its pipe for 64 cycles per warp and quadrant, a 32-bit
// integer multiply-add into 64 bits for about 3.  The pair passes therefore form their sums
// sum_b q_b w_ab in integers, at or above FP64 precision:
//   * the pair's kernel value or gradient (dimensionless, |w| <= 1) as a fixed-point integer in
//     units of 2^-57, from the FP64 separation (pair_fixed);
//   * the particle's value q_b as its exact 53-bit mantissa (times 2) in two limbs
//     hi 2^29 + lo (lo balanced around 0) and its exponent;
//   * the particle's sums in units of the largest exponent E among its neighbours (a first look
//     over the exponents alone): w is shifted down by E - e_b and split into limbs, hi hi goes to
//     one 64-bit accumulator and the two cross products to another; the dropped lo lo is below
//     2^-54 of the largest q_b, with either sign;
//   * the lanes are added in integers, and each total becomes a double once.
// Against sums in FP64, whose additions round at 2^-53 of the partial sum, the error is smaller
// (the step's error against 64-bit values: 5.2e-16 of u on the ideal lattice with FP64 sums, 5.0e-16
// now), and it does not depend on the order of the additions.
// A non-finite q_b makes the particle's sums NaN.
#pragma once
#include "sph_internal.cuh"

namespace sphg {

constexpr int kFxBits = 57;   // units of the fixed-point kernel values
constexpr int kLimb = 29;
constexpr long long kLimbMask = (1LL << kLimb) - 1;
constexpr int kNonFinite = 0x7FF;
constexpr int kFoldEvery = 16;     // terms between folds of the cross accumulators
constexpr int kHeadroom = 128;     // terms a lane's high accumulator holds without a larger unit

// A lower bound of the distance along one axis from x, in cell c of side cell, to the cell c + o: 0
// for o = 0; the margin covers the rounding of the single-precision position and of c cell (each
// below 2^-24 of the position), so a cell left out at gap^2 > supp2_hi holds no neighbour.  NaN stays.
__device__ __forceinline__ float cell_gap(int o, float x, int c, float cell)
{
    if (o == 0) return 0.0f;
    const float g = o < 0 ? x - (float)c * cell : (float)(c + 1) * cell - x;
    const float m = g - 1e-6f * (fabsf(x) + cell);
    return m < 0.0f ? 0.0f : m;
}

// |v| 2^-s in units of 2^-61 (below 2^62), rounded to nearest
__device__ __forceinline__ unsigned long long abs_fixed(double v, int s)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int k = (int)(b >> 52 & 0x7FF) - (1075 - 61) - s;
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFULL) | (1ULL << 52);
    return k >= 0 ? m << min(k, 9) : (k > -60 ? (m + (1ULL << (-k - 1))) >> -k : 0ULL);
}

// A pair's kernel value and gradient in fixed point from its separation d and r2 = |d|^2 <= 4 h^2:
// w = (2-q)^3/4 - max(1-q, 0)^3 and g_k = w' d_k/r, w' = 3 max(1-q, 0)^2 - 3 (2-q)^2/4 <= 0, q = r/h,
// all in units of 2^-kFxBits.  r2 = m 4^s with m in [1, 4): a single-precision reciprocal square
// root y of m (relative error below 2^-21) is refined by one third-order Householder step, e =
// 1 - m y^2, c = e/2 + 3 e^2/8, 1/sqrt(m) = y (1 + c), with the remainder of order e^3 below 2^-60.
// Everything behind r2 is in 64-bit integers: a high product is about 10 integer instructions
// (25 cycles a warp), an FP64 operation 64 cycles; errors below 2^-56 of the kernel's maximum.
template <int D>
__device__ __forceinline__ void pair_fixed(const double (&d)[D], double r2, double inv_h, long long &w, long long (&g)[D])
{
    const unsigned hi = (unsigned)__double2hiint(r2), lo = (unsigned)__double2loint(r2);
    w = 1LL << kFxBits;  // coincident particles: W(0), no gradient
#pragma unroll
    for (int k = 0; k < D; ++k) g[k] = 0;
    if (hi - 0x00100000u >= 0x7FE00000u) return;  // zero (or below 2^-1022)
    const int E = (int)(hi >> 20) - 1023, s = E >> 1, odd = E & 1;
    const unsigned long long M = (((unsigned long long)(hi & 0xFFFFFu) | 0x100000u) << 32 | lo) << (10 + odd);  // m, 2^-62
    const float y = rsqrt_apx(__uint_as_float((__funnelshift_l(lo, hi, 3) & 0x7FFFFFu) | (unsigned)(127 + odd) << 23));
    const unsigned Y = __float2uint_rz(y * 33554432.0f);  // 2^-25, exact
    const long long e = (1LL << 61) - (long long)__umul64hi(M, (unsigned long long)Y * Y << 13);  // 2^-61, |e| < 2^-19
    const int e0 = (int)(e >> 21);
    const long long c = (e >> 1) + (((long long)e0 * e0 * 3) >> 22);
    const unsigned long long R = __umul64hi((unsigned long long)Y << 38, (1ULL << 63) + (unsigned long long)(c * 4)) << 1;  // 1/sqrt(m), 2^-63
    const unsigned long long hb = (unsigned long long)__double_as_longlong(inv_h);
    const unsigned long long H = (hb << 11) | (1ULL << 63);  // 1/h = H 2^t, 2^-63
    const int sh = s + (int)(hb >> 52 & 0x7FF) - 1023;
    const unsigned long long qr = __umul64hi(__umul64hi(M, R) << 1, H);  // q 2^-sh, 2^-61
    const long long Q = (long long)(sh >= 0 ? qr << min(sh, 63) : qr >> min(-sh, 63));
    // t = 2 - q and u = max(1 - q, 0), 2^-61
    const unsigned long long T = (unsigned long long)max((1LL << 62) - Q, 0LL), U = (unsigned long long)max((1LL << 61) - Q, 0LL);
    const unsigned long long T2 = __umul64hi(T, T), U2 = __umul64hi(U, U);  // 2^-58
    const unsigned long long T3 = __umul64hi(T2 << 3, T), U3 = __umul64hi(U2 << 3, U);
    w = ((long long)T3 - 4 * (long long)U3 + 4) >> 3;
    const unsigned long long n = (unsigned long long)max(48 * ((long long)(T2 >> 2) - (long long)U2), 0LL);  // -w', 2^-62
    const unsigned long long P = __umul64hi(n << 1, R) << 1;  // -w'/sqrt(m), 2^-63
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const long long a = (long long)((__umul64hi(P, abs_fixed(d[k], s) << 1) + 8) >> 4);
        g[k] = __double2hiint(d[k]) < 0 ? a : -a;
    }
}

// w >= 0 in units of 2^-kFxBits as a double, rounded to nearest (in integers: a conversion instruction
// occupies the FP64 pipe like an operation)
__device__ __forceinline__ double fixed_value(long long w)
{
    if (w <= 0) return 0.0;
    const int s = __clzll(w);
    const unsigned long long m = (unsigned long long)w << s;
    const unsigned long long b = ((unsigned long long)(1022 + 63 - kFxBits - s) << 52) + (m >> 11) + (m >> 10 & 1u);
    return __longlong_as_double((long long)b);
}

// The lanes' sums of up to 8 values: value k (of t[0..7]) over the warp in lane 4 k (and 4 k + 1 to
// 4 k + 3).  Halves exchange values first: 9 additions instead of 5 a value, in a fixed order.
__device__ __forceinline__ double warp_sums8(double (&t)[8], int lane)
{
#pragma unroll
    for (int h = 4, o = 16; h > 0; h >>= 1, o >>= 1)
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const bool up = lane & o;
            const double send = up ? t[k] : t[k + h];
            t[k] = (up ? t[k + h] : t[k]) + __shfl_xor_sync(0xFFFFFFFFu, send, o);
        }
    t[0] += __shfl_xor_sync(0xFFFFFFFFu, t[0], 2);
    return t[0] + __shfl_xor_sync(0xFFFFFFFFu, t[0], 1);
}

// biased exponent of v (zero and denormals: 1), kNonFinite for infinities and NaN
__device__ __forceinline__ int fx_exponent(double v)
{
    const int e = (__double2hiint(v) >> 20) & 0x7FF;
    return max(e, 1);
}
// v = (hi 2^29 + lo) 2^(E - 1076), E at least v's exponent (rounded down to that unit)
__device__ __forceinline__ int2 fx_limbs(double v, int E)
{
    const long long b = __double_as_longlong(v);
    const int e = (int)(b >> 52) & 0x7FF;
    long long m = ((b & 0xFFFFFFFFFFFFFLL) | (e > 0 ? 1LL << 52 : 0LL)) << 1;
    m = (b < 0 ? -m : m) >> min(E - max(e, 1), 63);
    const int lo = (int)((unsigned)m << (32 - kLimb)) >> (32 - kLimb);  // the low 29 bits, sign-extended
    return make_int2((int)((m - lo) >> kLimb), lo);
}

// one sum: value (hh 2^29 + x) 2^29 in units of 2^(E - 1076 - kFxBits)
struct FxSum {
    long long hh, x;
};
__device__ __forceinline__ void fx_add(FxSum &s, int whi, int wlo, int2 q)
{
    s.hh += (long long)whi * q.x;
    s.x += (long long)whi * q.y;
    s.x += (long long)wlo * q.x;
}
__device__ __forceinline__ void fx_fold(FxSum &s)
{
    s.hh += s.x >> kLimb;
    s.x &= kLimbMask;
}
// exponents of several values packed in 16-bit halves: the larger of each
__device__ __forceinline__ unsigned fx_max2(unsigned a, unsigned b) { return __vmaxu2(a, b); }
// packed exponents over the 16 lanes of a half warp
__device__ __forceinline__ unsigned fx_half_max2(unsigned e)
{
    for (int o = 8; o > 0; o >>= 1) e = fx_max2(e, __shfl_xor_sync(0xFFFFFFFFu, e, o));
    return e;
}
// the unit's exponent for sums over n entries (16 lanes): E, and more where a lane adds over
// kHeadroom terms
__device__ __forceinline__ int fx_room(int E, int n) { return E + (32 - __clz((n / 16) / kHeadroom)); }
// w shifted to a unit d exponents larger, in limbs
__device__ __forceinline__ void fx_split(long long w, int d, int &hi, int &lo)
{
    const long long t = w >> min(d, 63);
    hi = (int)(t >> kLimb);
    lo = (int)t & (int)kLimbMask;
}

// Sums over the 16 lanes of a half warp.  Each lane's (hh, x) goes into two words that cannot
// overflow (hh in high and low parts), reduced by recursive halving.
struct FxTotal {
    long long p, q;  // p 2^49 + q
};
__device__ __forceinline__ FxTotal fx_words(const FxSum &s)
{
    return FxTotal{s.hh >> 20, ((s.hh & 0xFFFFF) << kLimb) | s.x};
}
__device__ __forceinline__ FxTotal fx_exchange(const FxTotal &keep, const FxTotal &give, int mask)
{
    return FxTotal{keep.p + __shfl_xor_sync(0xFFFFFFFFu, give.p, mask), keep.q + __shfl_xor_sync(0xFFFFFFFFu, give.q, mask)};
}
__device__ __forceinline__ FxTotal fx_sel(bool c, const FxTotal &a, const FxTotal &b)
{
    return FxTotal{c ? a.p : b.p, c ? a.q : b.q};
}
// 8 values: lanes 2k, 2k + 1 of the half warp get the total of value k
__device__ __forceinline__ FxTotal fx_reduce8(const FxTotal (&v)[8], int lane)
{
    const bool b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
    FxTotal h[4], g[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = fx_exchange(fx_sel(b3, v[4 + i], v[i]), fx_sel(b3, v[i], v[4 + i]), 8);
#pragma unroll
    for (int i = 0; i < 2; ++i) g[i] = fx_exchange(fx_sel(b2, h[2 + i], h[i]), fx_sel(b2, h[i], h[2 + i]), 4);
    const FxTotal f = fx_exchange(fx_sel(b1, g[1], g[0]), fx_sel(b1, g[0], g[1]), 2);
    return fx_exchange(f, f, 1);
}
// 16 values: lane k of the half warp gets the total of value k
__device__ __forceinline__ FxTotal fx_reduce16(const FxTotal (&v)[16], int lane)
{
    const bool b3 = lane & 8, b2 = lane & 4, b1 = lane & 2, b0 = lane & 1;
    FxTotal o[8], h[4], g[2];
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] = fx_exchange(fx_sel(b3, v[8 + i], v[i]), fx_sel(b3, v[i], v[8 + i]), 8);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = fx_exchange(fx_sel(b2, o[4 + i], o[i]), fx_sel(b2, o[i], o[4 + i]), 4);
#pragma unroll
    for (int i = 0; i < 2; ++i) g[i] = fx_exchange(fx_sel(b1, h[2 + i], h[i]), fx_sel(b1, h[i], h[2 + i]), 2);
    return fx_exchange(fx_sel(b0, g[1], g[0]), fx_sel(b0, g[0], g[1]), 1);
}
// a total p 2^49 + q in units of 2^k as a double: k = fx_unit(E) for a group's sums, -kFxBits for
// sums of kernel values alone (x counting units of 2^-kFxBits)
__device__ __forceinline__ int fx_unit(int E) { return E - 1076 - kFxBits + kLimb; }
__device__ __forceinline__ double fx_value(const FxTotal &t, int k)
{
    const double v = fma((double)t.p, 562949953421312.0, (double)t.q);  // 2^49
    const int k1 = k / 2, k2 = k - k1;                                  // two normal factors
    return v * __hiloint2double((1023 + k1) << 20, 0) * __hiloint2double((1023 + k2) << 20, 0);
}
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7FF8000000000000LL); }

// The limbs of particle values for the pair passes, in planes of int4 (two values each) over the
// particles, so that the lanes' neighbours, mostly consecutive, load from few cache lines: values
// with an exponent each (S, N_B, N_S, N_Q; lane k < 4 of a group of lanes writes value k)
__device__ __forceinline__ void fx_store_value(int4 *Q, unsigned short *Qe, size_t n, size_t a, int k, double v)
{
    const int e = fx_exponent(v);
    reinterpret_cast<int2 *>(Q)[2 * ((k >> 1) * n + a) + (k & 1)] = fx_limbs(v, e);
    Qe[4 * a + k] = (unsigned short)e;
}
// the largest exponent of K components of one tensor or vector
template <int K>
__device__ __forceinline__ int fx_shared_exponent(const double (&v)[K])
{
    int e = 1;
#pragma unroll
    for (int k = 0; k < K; ++k) e = max(e, fx_exponent(v[k]));
    return e;
}
__device__ __forceinline__ int4 fx_limbs2(double v0, int e0, double v1, int e1)
{
    const int2 l0 = fx_limbs(v0, e0), l1 = fx_limbs(v1, e1);
    return make_int4(l0.x, l0.y, l1.x, l1.y);
}
__device__ __forceinline__ int2 lo_of(int4 v) { return make_int2(v.x, v.y); }
__device__ __forceinline__ int2 hi_of(int4 v) { return make_int2(v.z, v.w); }

}  // namespace sphg
