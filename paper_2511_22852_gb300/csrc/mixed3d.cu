// mixed3d.cu -- the neighbour passes (rows a3, a5) of the 3+1D step in the mixed-precision
// form: positions relative to the origin of their cell in single precision, separations
// (r_a - r_b) - o (2h) formed from numbers of size <= 2h, a proven float error band around (2h)^2
// inside which the FP64 test r^2 < (2h)^2 (separately rounded products) decides -- the neighbour
// sets are those of the FP64 form.  The EoS inversion, equations of motion and reductions stay
// FP64 (step3d.cu).
//
// One warp takes two consecutive particles of a cell through the candidates of the 27 cells of
// side 2h around it, 32 candidates at a time, both particles in one packed two-wide FP32
// instruction.  The cells hold 216 h^3 of candidates for 33.5 h^3 of neighbours (6.4 to 1), so
// rejecting has to be cheap and the pair arithmetic must not run on rejected candidates: cells
// farther than 2h from both particles are left out (20.6 of 27 remain on average), accepted
// candidates are compacted into a queue (with their separation), and 32 at a time the kernel and
// the sums run on full warps.  Each lane sums at most kRun terms in plain FP32; the lanes' sums
// are then combined by error-free additions, one lane per sum over a transposed copy in shared
// memory, and converted to FP64 once.
//
// Bound: instruction issue (the rejection walk, about 1,500 warp instructions per particle and
// pass, against 900 for the accepted pairs of the density and 1,400 of the gradient pass); the
// gradient pass takes the accepted pairs from the list the density pass wrote (k_list_gradient3m),
// the walk is left for stages whose rows overflowed and for events without lists.
#include <algorithm>

#include "sph_internal.cuh"
#include "tiled_common.cuh"

namespace sphg {

namespace {

__device__ __forceinline__ double dist2_3e(double dx, double dy, double dz)
{
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}
__device__ __forceinline__ uint32_t key3m(const EvView &v, int cx, int cy, int cz)
{
    return v.spread[cx] | v.spread[1024 + cy] | v.spread[2048 + cz];
}

// cell-relative single-precision positions of the sorted particles, w: the cell's coordinates
// (10 bits per axis), and the density pass's per-particle values (S, N_B, N_S, N_Q) in FP32
__global__ void k_relpos3(EvView v, const double *__restrict__ y, const double *__restrict__ Nq,
                          float4 *__restrict__ rel, float4 *__restrict__ fq)
{
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= v.n) return;
    const size_t n = (size_t)v.n;
    const double cs = 2.0 * v.h;
    float r[3];
    int pk = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double xm = dec_double(v.sc->xmin_enc[d]);
        const double x = y[(size_t)d * n + j];
        const int c = cell_coord(x, xm, v.inv_cell);
        r[d] = __double2float_rn(__dsub_rn(__dsub_rn(x, xm), (double)c * cs));
        pk |= min(max(c, 0), (1 << v.B3[d]) - 1) << (10 * d);  // as the sort clamps it
    }
    rel[j] = make_float4(r[0], r[1], r[2], __int_as_float(pk));
    fq[j] = make_float4((float)y[6 * n + j], (float)Nq[j], (float)Nq[n + j], (float)Nq[2 * n + j]);
}

constexpr int kWW = 8;                // warps per block, two particles each
constexpr unsigned kFull = 0xFFFFFFFFu;

constexpr int kTag = 27;  // listed words: candidate index below, its cell's number (0-26) above
constexpr int kIndex = (1 << kTag) - 1;

struct WalkMem {
    float4 q[2][64];  // queued pairs of the two particles: separation and candidate index
};
// one particle's lane sums, transposed: NV values of 33 floats (over the queues when they are empty)
static_assert(sizeof(WalkMem) >= 15 * 33 * sizeof(float), "the sums fit over the queues");

// NV per-lane sums of one particle combined into lane v < NV (its running hi + lo), error-free:
// hi = TwoSum(hi, term) with the rounding errors in lo
template <int NV>
__device__ __forceinline__ void flush_sums(float *red, float (&s)[NV], int lane, bool mine, int slot, CSum &tot)
{
    __syncwarp();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        red[k * 33 + lane] = s[k];
        s[k] = 0.0f;
    }
    __syncwarp();
    if (mine) {
        float hi = tot.hi, lo = tot.lo;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const float x = red[slot * 33 + j];
            const float t = hi + x, bb = t - hi;
            lo += (hi - (t - bb)) + (x - bb);
            hi = t;
        }
        tot = CSum{hi, lo};
    }
    __syncwarp();
}

// The walk of one warp over the candidates of particles a0 and a1 = a0 + 1 (both in the cell of
// ra0; two = false: a0 alone).  pair(which, entry, place) receives an accepted pair per lane, the
// particle's pairs in order, 32 at a time; flush(mask) is called for a particle (bit) after every
// kRun of its batches and for both at the end, with the queues' memory free.
// nacc: accepted candidates (self included); shell: candidates decided by the FP64 test.  An
// entry's index word holds the candidate and, with TAG, its cell's number above bit kTag.
template <bool TAG, class Pair, class Flush>
__device__ __forceinline__ void walk27_two(const EvView &v, const double *__restrict__ y,
                                           const float4 *__restrict__ rel, const uint32_t *__restrict__ start,
                                           const uint32_t *__restrict__ cnt, int a0, bool two, float4 ra0, float4 ra1,
                                           WalkMem &M, int lane, int (&nacc)[2], unsigned &shell,
                                           Pair &&pair, Flush &&flush)
{
    const size_t n = (size_t)v.n;
    const unsigned lt = (1u << lane) - 1u;
    const float slo = v.shell_lo, shi = v.shell_hi, cell = v.cell_f;
    const int pk = __float_as_int(ra0.w);
    if (!two) ra1 = make_float4(kFar, kFar, kFar, 0.0f);  // never accepted
    // lane t < 27: the neighbour cell t, kept when it holds particles and its box lies within 2h
    // (with a margin far above the positions' rounding) of either particle
    int st = 0, len = 0;
    if (lane < 27) {
        const int o[3] = {lane % 3 - 1, (lane / 3) % 3 - 1, lane / 9 - 1};
        int c[3];
        bool in = true;
        float d0 = 0.0f, d1 = 0.0f;
        const float p0[3] = {ra0.x, ra0.y, ra0.z}, p1[3] = {ra1.x, ra1.y, ra1.z};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c[k] = ((pk >> (10 * k)) & 1023) + o[k];
            in = in && c[k] >= 0 && c[k] < (1 << v.B3[k]);
            const float g0 = o[k] < 0 ? p0[k] : (o[k] > 0 ? cell - p0[k] : 0.0f);
            const float g1 = o[k] < 0 ? p1[k] : (o[k] > 0 ? cell - p1[k] : 0.0f);
            d0 = fmaf(fmaxf(g0, 0.0f), g0, d0);
            d1 = fmaf(fmaxf(g1, 0.0f), g1, d1);
        }
        const float lim = shi * 1.0001f;
        // written so that a NaN position keeps the cell
        if (in && (!(d0 > lim) || (two && !(d1 > lim)))) {
            const uint32_t k = key3m(v, c[0], c[1], c[2]);
            st = (int)start[k];
            len = (int)cnt[k];
        }
    }
    unsigned cells = __ballot_sync(kFull, len > 0);
    const float2 ax = make_float2(ra0.x, ra1.x), ay = make_float2(ra0.y, ra1.y), az = make_float2(ra0.z, ra1.z);
    int qn[2] = {0, 0};  // queued; nacc - qn have been handed on
    while (cells) {
        const int o = __ffs(cells) - 1;
        cells &= cells - 1u;
        const int b0 = __shfl_sync(kFull, st, o), ln = __shfl_sync(kFull, len, o);
        const float ox = -(float)(o % 3 - 1) * cell, oy = -(float)((o / 3) % 3 - 1) * cell, oz = -(float)(o / 9 - 1) * cell;
        const int word = TAG ? (int)((unsigned)o << kTag) : 0;
        for (int base = 0; base < ln; base += 32) {
            const bool in = base + lane < ln;
            const int b = b0 + base + lane;
            float4 rb = make_float4(-kFar, -kFar, -kFar, 0.0f);
            if (in) rb = rel[b];
            // (r_a - r_b) - o (2h), rounded step by step as the shell bound assumes
            const float2 dx = __fadd2_rn(__fadd2_rn(ax, make_float2(-rb.x, -rb.x)), make_float2(ox, ox));
            const float2 dy = __fadd2_rn(__fadd2_rn(ay, make_float2(-rb.y, -rb.y)), make_float2(oy, oy));
            const float2 dz = __fadd2_rn(__fadd2_rn(az, make_float2(-rb.z, -rb.z)), make_float2(oz, oz));
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            bool acc0 = r2.x <= shi, acc1 = r2.y <= shi;
            if ((acc0 && r2.x >= slo) || (acc1 && r2.y >= slo)) {  // thin shell: the exact FP64 decision
                const double xb = y[b], yb = y[n + b], zb = y[2 * n + b];
                if (acc0 && r2.x >= slo) {
                    acc0 = dist2_3e(y[a0] - xb, y[n + a0] - yb, y[2 * n + a0] - zb) < v.supp2;
                    ++shell;
                }
                if (acc1 && r2.y >= slo) {
                    acc1 = dist2_3e(y[a0 + 1] - xb, y[n + a0 + 1] - yb, y[2 * n + a0 + 1] - zb) < v.supp2;
                    ++shell;
                }
            }
            const unsigned m0 = __ballot_sync(kFull, acc0), m1 = __ballot_sync(kFull, acc1);
            if (m0) {
                if (acc0) M.q[0][qn[0] + __popc(m0 & lt)] = make_float4(dx.x, dy.x, dz.x, __int_as_float(b | word));
                qn[0] += __popc(m0);
                nacc[0] += __popc(m0);
            }
            if (m1) {
                if (acc1) M.q[1][qn[1] + __popc(m1 & lt)] = make_float4(dx.y, dy.y, dz.y, __int_as_float(b | word));
                qn[1] += __popc(m1);
                nacc[1] += __popc(m1);
            }
            unsigned full = 0u;
#pragma unroll
            for (int p = 0; p < 2; ++p)
                if (qn[p] >= 32) {
                    __syncwarp();
                    pair(p, M.q[p][lane], nacc[p] - qn[p] + lane);
                    const float4 rest = M.q[p][32 + lane];
                    __syncwarp();
                    qn[p] -= 32;
                    if (lane < qn[p]) M.q[p][lane] = rest;
                    if (((nacc[p] - qn[p]) & (32 * kRun - 1)) == 0) full |= 1u << p;
                }
            if (full) {  // at most kRun plain terms per lane; the queues wait in registers
                __syncwarp();
                const float4 k0 = M.q[0][lane], k1 = M.q[1][lane];
                flush(full);
                M.q[0][lane] = k0;
                M.q[1][lane] = k1;
                __syncwarp();
            }
        }
    }
    __syncwarp();
    if (lane < qn[0]) pair(0, M.q[0][lane], nacc[0] - qn[0] + lane);
    if (lane < qn[1]) pair(1, M.q[1][lane], nacc[1] - qn[1] + lane);
    flush(3u);
}

// Density pass (row a3).  With lists (pl.total > 0) the accepted candidates go into the particles'
// rows for the gradient pass; a particle that outgrows its row flags the stage.
template <bool LIST>
__global__ void __launch_bounds__(32 * kWW, LIST ? 3 : 4) k_walk_density3m(EvView v, const double *__restrict__ y,
                                                             const float4 *__restrict__ rel,
                                                             const float4 *__restrict__ fq,
                                                             const uint32_t *__restrict__ start,
                                                             const uint32_t *__restrict__ cnt, PairBufs pl,
                                                             double *__restrict__ dens, int *__restrict__ nnb)
{
    __shared__ WalkMem mem[kWW];
    __shared__ unsigned s_pairs, s_shell;
    if (threadIdx.x == 0) s_pairs = s_shell = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t n = (size_t)v.n;
    WalkMem &M = mem[wid];
    float *red = reinterpret_cast<float *>(&M);
    const long long w = (long long)blockIdx.x * kWW + wid;
    const float ih = (float)v.inv_h;
    unsigned shell = 0u, pairs = 0u;
    for (int a0 = (int)min(2 * w, (long long)v.n), end = min(a0 + 2, v.n); a0 < end;) {  // warp-uniform
        const float4 ra0 = rel[a0], ra1 = rel[min(a0 + 1, end - 1)];
        const bool two = a0 + 1 < end && __float_as_int(ra0.w) == __float_as_int(ra1.w);
        float s0[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, s1[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
        CSum tot = {0.f, 0.f};  // lanes 0-4: a0's sums, 16-20: a1's
        int nacc[2] = {0, 0};
        int *row[2] = {nullptr, nullptr};
        int cap[2] = {0, 0};
        if (LIST)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int a = a0 + (two ? p : 0);
                const long long r0 = pl.off[a], r1 = pl.off[a + 1];
                row[p] = pl.L + r0;
                cap[p] = r1 <= pl.total ? (int)(r1 - r0) : 0;
            }
        auto pair = [&](int which, float4 e, int place) {
            const int word = __float_as_int(e.w);
            const float4 qb = fq[LIST ? word & kIndex : word];
            if (LIST && place < (which ? cap[1] : cap[0])) (which ? row[1] : row[0])[place] = word;
            const float r2 = fmaf(e.x, e.x, fmaf(e.y, e.y, e.z * e.z));
            const float q = sqrt_apx(r2) * ih;
            // w(q) = (2-q)^3/4 - max(1-q,0)^3 on 0 <= q <= 2
            const float t = 2.0f - q, u = fmaxf(1.0f - q, 0.0f);
            const float wv = fmaf(0.25f * (t * t), t, -(u * u) * u);
            float(&s)[5] = which ? s1 : s0;
            s[0] += wv;
            s[1] = fmaf(qb.x, wv, s[1]);
            s[2] = fmaf(qb.y, wv, s[2]);
            s[3] = fmaf(qb.z, wv, s[3]);
            s[4] = fmaf(qb.w, wv, s[4]);
        };
        auto flush = [&](unsigned m) {
            if (m & 1u) flush_sums<5>(red, s0, lane, lane < 5, lane, tot);
            if (two && (m & 2u)) flush_sums<5>(red, s1, lane, lane >= 16 && lane < 21, lane - 16, tot);
        };
        walk27_two<LIST>(v, y, rel, start, cnt, a0, two, ra0, ra1, M, lane, nacc, shell, pair, flush);
        const int k = lane & 15;
        if (k < 5 && (lane < 16 || two)) dens[(size_t)k * n + a0 + (lane >> 4)] = v.sigma_d * cval(tot);
        if (lane < (two ? 2 : 1)) {
            const int c = lane ? nacc[1] : nacc[0];
            nnb[a0 + lane] = c;
            pairs += (unsigned)c;
            if (LIST) {
                pl.cntF[a0 + lane] = c;
                if (pl.cnt_dst) pl.cnt_dst[a0 + lane] = c;  // sizes this particle's row in the next stage
                if (c > (lane ? cap[1] : cap[0])) atomicOr(&v.sc->pair_flag, 1u);
            }
        }
        a0 += two ? 2 : 1;
    }
    shell = __reduce_add_sync(kFull, shell);
    pairs = __reduce_add_sync(kFull, pairs);
    if (lane == 0) {
        atomicAdd(&s_pairs, pairs);
        if (shell) atomicAdd(&s_shell, shell);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_pairs) atomicAdd(&v.sc->pairs, (unsigned long long)s_pairs);
        if (s_shell) atomicAdd(&v.sc->shell_tests, (unsigned long long)s_shell);
    }
}

// Gradient pass (row a5).  gin rows: X^{ji}/sigma*^2 at 3 j + i, u^j/sigma* at 9 + j; gout rows:
// d_k u^j at 3 k + j, then F^i at 9 + i (the layout of the FP64 3+1D gradient pass).  The 15
// sums: 0-2 sum grad W, 3-5 sum_b X_b^{j i} grad_j W, 6 + 3 k + j sum_b u_b^j grad_k W.
__device__ __forceinline__ void add_gradient(float (&s)[15], float dx, float dy, float dz, float ih, const float4 *__restrict__ fx,
                                             size_t n, int b)
{
    const float4 f0 = fx[b], f1 = fx[n + b], f2 = fx[2 * n + b];
    const float row[12] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w, f2.x, f2.y, f2.z, f2.w};
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    // r = 0 (the particle itself) gives dw/dq = 0: a zero term
    const float ir = rsqrt_apx(fmaxf(r2, 1e-30f));
    const float q = (r2 * ir) * ih;
    const float t = 2.0f - q, u = fmaxf(1.0f - q, 0.0f);
    const float fac = fmaf(-0.75f, t * t, 3.0f * (u * u)) * ir;
    // rounded products: the list pass and the walk give the same sums
    const float g[3] = {__fmul_rn(fac, dx), __fmul_rn(fac, dy), __fmul_rn(fac, dz)};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        s[i] += g[i];
        s[3 + i] = fmaf(row[6 + i], g[2], fmaf(row[3 + i], g[1], fmaf(row[i], g[0], s[3 + i])));
    }
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) s[6 + 3 * k + j] = fmaf(row[9 + j], g[k], s[6 + 3 * k + j]);
}
// the totals of a0 (lanes 0-14) and a0 + 1 (lanes 16-30, with two) to gout
__device__ __forceinline__ void store_gradient(const EvView &v, int stage, const CSum &tot, int lane, int a0, bool two,
                                               const double *__restrict__ gin, double *__restrict__ gout)
{
    const size_t n = (size_t)v.n;
    const double d = cval(tot);
    const int k = lane & 15, first = lane & 16;
    const size_t a = (size_t)a0 + (lane >> 4);
    const double G0 = __shfl_sync(kFull, d, first), G1 = __shfl_sync(kFull, d, first + 1), G2 = __shfl_sync(kFull, d, first + 2);
    if (k >= 3 && k < 15 && (lane < 16 || two)) {
        const double cf = v.sigma_d * v.inv_h;
        if (k >= 6) {
            gout[(size_t)(k - 6) * n + a] = cf * d;
        } else {
            // minus the stress divergence: sum X_b grad W + X_a . sum grad W, times sqrt(-g)
            const double tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
            const double sqrtg = v.milne ? tau : 1.0;
            const int i = k - 3;
            double F = fma(gin[(size_t)i * n + a], G0, d);
            F = fma(gin[(size_t)(3 + i) * n + a], G1, F);
            F = fma(gin[(size_t)(6 + i) * n + a], G2, F);
            gout[(size_t)(9 + i) * n + a] = -sqrtg * cf * F;
        }
    }
}

// over the walk's candidates; fallback: the list pass ran first, and this one only does for a
// stage whose rows overflowed (counting it)
__global__ void __launch_bounds__(32 * kWW, 3) k_walk_gradient3m(EvView v, int stage, const double *__restrict__ y,
                                                              const float4 *__restrict__ rel,
                                                              const double *__restrict__ gin,
                                                              const float4 *__restrict__ fx,
                                                              const uint32_t *__restrict__ start,
                                                              const uint32_t *__restrict__ cnt,
                                                              double *__restrict__ gout, int fallback)
{
    if (fallback) {
        if (!v.sc->pair_flag) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&v.sc->pair_ovf, 1u);
    }
    __shared__ WalkMem mem[kWW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t n = (size_t)v.n;
    WalkMem &M = mem[wid];
    float *red = reinterpret_cast<float *>(&M);
    const float ih = (float)v.inv_h;
    for (long long w = (long long)blockIdx.x * kWW + wid; 2 * w < v.n; w += (long long)gridDim.x * kWW)
        for (int a0 = (int)(2 * w), end = min(a0 + 2, v.n); a0 < end;) {  // warp-uniform
            const float4 ra0 = rel[a0], ra1 = rel[min(a0 + 1, end - 1)];
            const bool two = a0 + 1 < end && __float_as_int(ra0.w) == __float_as_int(ra1.w);
            float s0[15], s1[15];
#pragma unroll
            for (int k = 0; k < 15; ++k) s0[k] = s1[k] = 0.0f;
            CSum tot = {0.f, 0.f};  // lanes 0-14: a0's sums, 16-30: a1's
            int nacc[2] = {0, 0};
            unsigned shell = 0u;
            auto pair = [&](int which, float4 e, int) {
                add_gradient(which ? s1 : s0, e.x, e.y, e.z, ih, fx, n, __float_as_int(e.w));
            };
            auto flush = [&](unsigned m) {
                if (m & 1u) flush_sums<15>(red, s0, lane, lane < 15, lane, tot);
                if (two && (m & 2u)) flush_sums<15>(red, s1, lane, lane >= 16 && lane < 31, lane - 16, tot);
            };
            walk27_two<false>(v, y, rel, start, cnt, a0, two, ra0, ra1, M, lane, nacc, shell, pair, flush);
            store_gradient(v, stage, tot, lane, a0, two, gin, gout);
            a0 += two ? 2 : 1;
        }
}

// over the rows the density pass listed, a warp for two particles in turn.
// Bound: the gathers (four 16-byte loads per pair, 9.5 GB a stage at 258,661 particles and 577
// neighbours, most from L1/L2).  Reading the list instead of testing the candidates again (about
// five per accepted pair): 0.74 ms a stage against 1.81 for the walk; writing the list adds 0.12 ms
// (1.44 to 1.56) to the density pass.
__global__ void __launch_bounds__(32 * kWW, 3) k_list_gradient3m(EvView v, int stage, const float4 *__restrict__ rel,
                                                              const double *__restrict__ gin,
                                                              const float4 *__restrict__ fx, PairBufs pl,
                                                              double *__restrict__ gout)
{
    if (v.sc->pair_flag) return;  // a row overflowed: the walk runs instead
    __shared__ float red_[kWW][15 * 33];
    __shared__ float4 shift[27];  // minus the cells' offsets
    if (threadIdx.x < 27) {
        const int o = threadIdx.x;
        shift[o] = make_float4(-(float)(o % 3 - 1) * v.cell_f, -(float)((o / 3) % 3 - 1) * v.cell_f, -(float)(o / 9 - 1) * v.cell_f, 0.0f);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t n = (size_t)v.n;
    float *red = red_[wid];
    const float ih = (float)v.inv_h;
    const long long a0l = 2 * ((long long)blockIdx.x * kWW + wid);
    if (a0l >= v.n) return;  // warp-uniform
    const int a0 = (int)a0l;
    const bool two = a0 + 1 < v.n;
    CSum tot = {0.f, 0.f};  // lanes 0-14: a0's sums, 16-30: a1's
    for (int p = 0; p < (two ? 2 : 1); ++p) {
        const int a = a0 + p, c = pl.cntF[a];
        const int *L = pl.L + pl.off[a];
        const float4 ra = rel[a];
        float s[15];
#pragma unroll
        for (int k = 0; k < 15; ++k) s[k] = 0.0f;
        const bool mine = p ? lane >= 16 && lane < 31 : lane < 15;
        int next = lane < c ? L[lane] : 0;
        for (int j = lane, it = 1; j - lane < c; j += 32, ++it) {  // warp-uniform trips
            const int word = next;
            next = j + 32 < c ? L[j + 32] : 0;
            if (j < c) {
                const int b = word & kIndex;
                const float4 rb = rel[b], sh = shift[(unsigned)word >> kTag];
                // (r_a - r_b) - o (2h), rounded as in the walk
                add_gradient(s, (ra.x - rb.x) + sh.x, (ra.y - rb.y) + sh.y, (ra.z - rb.z) + sh.z, ih, fx, n, b);
            }
            if ((it & (kRun - 1)) == 0) flush_sums<15>(red, s, lane, mine, lane - 16 * p, tot);
        }
        flush_sums<15>(red, s, lane, mine, lane - 16 * p, tot);
    }
    store_gradient(v, stage, tot, lane, a0, two, gin, gout);
}

inline int nblk(int n, int t) { return (n + t - 1) / t; }

}  // namespace

void launch_density3m(const EvView &v, const double *y, const double *Nq, CellBufs cb, double *dens, int *nnb,
                      cudaStream_t st)
{
    k_relpos3<<<nblk(v.n, 256), 256, 0, st>>>(v, y, Nq, cb.fpos3, cb.fq);
    const int grid = nblk(v.n, 2 * kWW);
    if (cb.pl.total > 0) {
        launch_pair_rows(v, cb, st);
        k_walk_density3m<true><<<grid, 32 * kWW, 0, st>>>(v, y, cb.fpos3, cb.fq, cb.start, cb.cnt, cb.pl, dens, nnb);
    } else {
        k_walk_density3m<false><<<grid, 32 * kWW, 0, st>>>(v, y, cb.fpos3, cb.fq, cb.start, cb.cnt, cb.pl, dens, nnb);
    }
}

void launch_gradient3m(const EvView &v, int stage, const double *y, const double *gin, CellBufs cb, double *gout,
                       cudaStream_t st)
{
    const int lists = cb.pl.total > 0, full = nblk(v.n, 2 * kWW);
    if (lists) k_list_gradient3m<<<full, 32 * kWW, 0, st>>>(v, stage, cb.fpos3, gin, cb.fx, cb.pl, gout);
    const int grid = lists ? std::min(full, 4 * device_sm_count()) : full;
    k_walk_gradient3m<<<grid, 32 * kWW, 0, st>>>(v, stage, y, cb.fpos3, gin, cb.fx, cb.start, cb.cnt, gout, lists);
}

}  // namespace sphg
