// pairs_fixed.cuh -- integer accumulation of the plain (FP64) neighbour sums.
//
// On GB300 an FP64 operation occupies its pipe for 64 cycles per warp and quadrant, a 32-bit
// integer multiply-add into 64 bits for about 3.  The pair passes therefore evaluate the kernel and
// form their sums sum_b q_b w_ab in integers, with the error of FP64 arithmetic or less in every term:
//   * the pair's kernel value or gradient component as a double, from the FP64 separation by 64-bit
//     integer operations (pair_kernel): relative error at most 2^-53 + 11 2^-60 / (2 - r/h), also
//     towards the kernel's rim and for a component much smaller than the others;
//   * the particle's value q_b as its exact 53-bit mantissa (times 2) in two limbs
//     hi 2^29 + lo (lo balanced around 0) and its exponent;
//   * each sum in units of the largest exponent E among its own terms' products q_b w_ab (a first
//     look over the exponents alone): w's mantissa is shifted down by E less the term's exponent
//     and split into limbs, hi hi goes to one 64-bit accumulator and the two cross products to another;
//     what is dropped is below 2^-53 of the largest term, and a sum in FP64 rounds at 2^-53 of its
//     partial sums, which reach half the largest term at least;
//   * the lanes are added in integers, and each total becomes a double once.
// So no value, charge or component is rounded against a larger one of another sum or of a neighbour
// that hardly counts, and the result does not depend on the order of the additions.
// A non-finite q_b makes the sums it enters NaN.
#pragma once
#include "sph_internal.cuh"

namespace sphg {

constexpr int kMant = 56;     // a kernel value's mantissa in units of its exponent: [2^56, 2^57),
constexpr int kGuard = 3;     // held times 2^3, so that a 32-bit word boundary parts the limbs
constexpr int kLimb = 29;
constexpr long long kLimbMask = (1LL << kLimb) - 1;
constexpr int kNonFinite = 0x3FFF;  // exponent of infinities and NaN: above every product's
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

// m 2^e as a double rounded to nearest (in integers: a conversion instruction occupies the FP64 pipe
// like an operation); m = 0 and results below 2^-1022: 0
__device__ __forceinline__ double pack_double(unsigned long long m, int e)
{
    const int s = __clzll((long long)m);
    m <<= s & 63;
    const int f = e - s + 63 + 1022;
    const unsigned long long b = ((unsigned long long)(unsigned)f << 52) + (m >> 11) + (m >> 10 & 1u);
    return __longlong_as_double(m == 0ULL || f < 0 ? 0LL : (long long)b);
}

// A pair's kernel value and gradient from its separation d and r2 = |d|^2 <= 4 h^2: w = (2-q)^3/4 -
// max(1-q, 0)^3 and g_k = w' d_k/r, w' = 3 max(1-q, 0)^2 - 3 (2-q)^2/4 <= 0, q = r/h.  r2 = m 4^s with
// m in [1, 4): a single-precision reciprocal square root y of m (relative error below 2^-21) is refined
// by one third-order Householder step, e = 1 - m y^2, c = e/2 + 3 e^2/8, 1/sqrt(m) = y (1 + c).
// Everything behind r2 is in 64-bit integers: a high product is about 10 integer instructions
// (25 cycles a warp), an FP64 operation 64 cycles.  q itself (q < 1) or t = 2 - q is normalised before
// its powers are taken, as are w'/r and d_k, so small results keep their leading bits: relative errors
// against 200-bit values at 60,000 separations stay below 2^-53 + 11 2^-60/(2 - q) for w and
// 2^-53 + 7.3 2^-60/(2 - q) for g_k (FP64 arithmetic: several 2^-53/(2 - q)).
template <int D>
__device__ __forceinline__ void pair_kernel(const double (&d)[D], double r2, double inv_h, double &w, double (&g)[D])
{
    const unsigned hi = (unsigned)__double2hiint(r2), lo = (unsigned)__double2loint(r2);
    w = 1.0;  // coincident particles: W(0), no gradient
#pragma unroll
    for (int k = 0; k < D; ++k) g[k] = 0.0;
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
    const unsigned long long Q = sh >= 0 ? qr << min(sh, 63) : qr >> min(-sh, 63);  // q, 2^-61
    const bool in = Q < (1ULL << 61);
    // v = X 2^ex: q itself for q < 1, t = 2 - q beyond, with all of its leading bits
    const unsigned long long v0 = in ? qr : (unsigned long long)max((1LL << 62) - (long long)Q, 0LL);
    const int lv = __clzll((long long)v0) & 63, ex = (in ? sh : 0) - 61 - lv;
    const unsigned long long X = v0 << lv, A = __umul64hi(X, X);
    // w = 1 - q^2 (3/2 - 3 q/4)  or  t^3/4;  -w' = 3 q (1 - 3 q/4)  or  3 t^2/4
    const unsigned long long B = __umul64hi(A, in ? 3 * ((1ULL << 62) - Q) : X);
    const unsigned long long w61 = (1ULL << 61) - (B >> min(-(126 + 2 * ex), 63));
    w = in ? pack_double(w61, -61) : pack_double(B, 126 + 3 * ex);
    unsigned long long N = in ? __umul64hi(X, (1ULL << 63) - 3 * Q) : A;
    N -= N >> 2;
    const int ln = __clzll((long long)N) & 63, en = (in ? ex + 1 : 62 + 2 * ex) + 2 - ln;
    const unsigned long long P = __umul64hi(N << ln, R);  // -w'/r = P 2^(en + 1 - s)
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const unsigned long long db = (unsigned long long)__double_as_longlong(d[k]);
        const int ed = (int)(db >> 52 & 0x7FF);
        const unsigned long long G = ed > 0 ? __umul64hi(P, (db << 11) | (1ULL << 63)) : 0ULL;
        const double a = pack_double(G, en - s + ed - 1021);
        g[k] = (long long)db < 0 ? a : -a;
    }
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
    return e == 0x7FF ? kNonFinite : max(e, 1);
}
// two exponents in the 16-bit halves of a word
__device__ __forceinline__ unsigned fx_pair(int lo, int hi) { return (unsigned)lo | ((unsigned)hi << 16); }
__device__ __forceinline__ int fx_lo(unsigned e) { return (int)(e & 0xFFFFu); }
__device__ __forceinline__ int fx_hi(unsigned e) { return (int)(e >> 16); }
// a kernel value (zero, or normal of magnitude up to 1) as mant 2^(exp - 1023 - kMant - kGuard)
__device__ __forceinline__ int fx_kexp(double w) { return (__double2hiint(w) >> 20) & 0x7FF; }
__device__ __forceinline__ long long fx_kmant(double w)
{
    const long long b = __double_as_longlong(w);
    const long long m = ((b & 0xFFFFFFFFFFFFFLL) | (1LL << 52)) << (kMant + kGuard - 52);
    return fx_kexp(w) == 0 ? 0LL : (b < 0 ? -m : m);
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

// one sum: value (hh 2^29 + x) 2^29 in units of 2^(E - 1076 - 1023 - kMant), E its products' exponent
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
// a mantissa shifted to a unit d exponents larger: as it is (units of kMant), and in limbs
__device__ __forceinline__ long long fx_shift(long long m, int d)
{
    long long t;  // amounts beyond 63 are clamped
    asm("shr.s64 %0, %1, %2;" : "=l"(t) : "l"(m), "r"(d));
    return t;
}
__device__ __forceinline__ void fx_split(long long m, int d, int &hi, int &lo)
{
    const long long t = fx_shift(m, d);
    hi = (int)(t >> 32);
    lo = (int)((unsigned)t >> kGuard);
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
// a total p 2^49 + q in units of 2^k as a double: k = fx_unit(E) for a sum of products, fx_kunit(E)
// for a sum of kernel values alone (x counting units); below 2^-1400 the total is zero as a double
__device__ __forceinline__ int fx_unit(int E) { return E - 1076 - 1023 - kMant + kLimb; }
__device__ __forceinline__ int fx_kunit(int E) { return E - 1023 - kMant; }
__device__ __forceinline__ double fx_value(const FxTotal &t, int k)
{
    const double v = fma((double)t.p, 562949953421312.0, (double)t.q);  // 2^49
    k = max(k, -1400);
    const int k1 = k / 2, k2 = k - k1;  // two normal factors
    return v * __hiloint2double((1023 + k1) << 20, 0) * __hiloint2double((1023 + k2) << 20, 0);
}
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7FF8000000000000LL); }

// limbs and pairs of words in 64 bits, four of them in a Limb4
__device__ __forceinline__ long long fx_word(unsigned lo, unsigned hi) { return (long long)(((unsigned long long)hi << 32) | lo); }
__device__ __forceinline__ long long fx_word(int2 v) { return fx_word((unsigned)v.x, (unsigned)v.y); }
__device__ __forceinline__ int2 fx_pair_of(long long w) { return make_int2((int)w, (int)(w >> 32)); }
__device__ __forceinline__ unsigned word_lo(long long w) { return (unsigned)w; }
__device__ __forceinline__ unsigned word_hi(long long w) { return (unsigned)(w >> 32); }
// S, N_B, N_S, N_Q (lane k < 4 of a group of lanes writes value k)
__device__ __forceinline__ void fx_store_value(Limb4 *Q, unsigned short *Qe, size_t a, int k, double v)
{
    const int e = fx_exponent(v);
    reinterpret_cast<int2 *>(Q)[4 * a + k] = fx_limbs(v, e);
    Qe[4 * a + k] = (unsigned short)e;
}

}  // namespace sphg
