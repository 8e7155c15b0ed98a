// mixed2d.cu -- the neighbour passes (rows a3, a5) in the mixed-precision form, 2+1D.
//
// The pair arithmetic runs on the FP32 pipe (64x the FP64 rate on GB300):
//   * positions are stored relative to the origin of their cell, so a pair separation
//     dx = (r_a - r_b) - o * (2h) (o the cell offset, -1..1) is formed from numbers of
//     size <= 2h and its single-precision error is ~1e-7 fm regardless of where the
//     event sits;
//   * the neighbour decision stays exact: a proven bound err on the float r^2 classifies
//     candidates as certainly inside (r2f < (2h)^2 - err), certainly outside
//     (r2f > (2h)^2 + err), or in the thin shell between, where the FP64 test r^2 < (2h)^2
//     with separately rounded products decides -- the same set as the FP64 path.
// The EoS inversion, equations of motion and conservation reductions stay FP64.
//
// As in 3+1D (mixed3d.cu) one warp takes two consecutive particles of a cell through the
// candidates of the 3x3 cells of side 2h, 32 at a time, both particles in one packed two-wide FP32
// instruction; accepted candidates are compacted into queues, and the kernel and the sums run on
// full warps.  Each lane sums at most kRun terms in plain FP32; the lanes' sums are combined by
// error-free additions and converted to FP64 once.  A block per cell with the candidates in
// shared memory ran the kernel on all 2.9 candidates per neighbour, and where the matter has
// clumped (a few cells with many times the usual particles) waited for its largest cells: the
// 40 k event's density + gradient took 448 us per step at first and 1,070 us after 300 steps;
// now 366 and 408 us.
#include <algorithm>

#include "sph_internal.cuh"
#include "tiled_common.cuh"

namespace sphg {

namespace {

constexpr int kWW = 8;  // warps per block, two particles each
constexpr unsigned kFull = 0xFFFFFFFFu;

// the density pass's per-particle values (S, N_B, N_S, N_Q) in single precision, and u0 (row 5)
__global__ void k_fq2(EvView v, const double *__restrict__ y, const double *__restrict__ Nq, float4 *__restrict__ fq,
                      double *__restrict__ dens)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= v.n) return;
    const size_t n = (size_t)v.n;
    fq[j] = make_float4((float)y[4 * n + j], (float)Nq[j], (float)Nq[n + j], (float)Nq[2 * n + j]);
    const double ux = y[2 * n + j], uy = y[3 * n + j];
    dens[5 * n + j] = sqrt(fma(ux, ux, fma(uy, uy, 1.0)));
}

struct WalkMem2 {
    float4 q[2][66];  // queued pairs of the two particles: separation, r^2 and candidate index
};
// the lane sums of both particles, transposed (33 floats a value), over the queues when they are empty
static_assert(sizeof(WalkMem2) >= 2 * 8 * 33 * sizeof(float), "the sums fit over the queues");

// NV per-lane sums of each particle, combined error-free: lanes 2 k, 2 k + 1 add the two halves of
// value k (k < NV: a0's, k >= NV: a1's) and keep hi = TwoSum(hi, term) with the rounding errors in lo
template <int NV>
__device__ __forceinline__ void flush2(float *red, float (&s0)[NV], float (&s1)[NV], int lane, CSum &tot)
{
    __syncwarp();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        red[k * 33 + lane] = s0[k];
        red[(NV + k) * 33 + lane] = s1[k];
        s0[k] = s1[k] = 0.0f;
    }
    __syncwarp();
    if (lane < 4 * NV) {
        const float *r = red + (lane >> 1) * 33 + 16 * (lane & 1);
        float hi = tot.hi, lo = tot.lo;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float x = r[j];
            const float t = hi + x, bb = t - hi;
            lo += (hi - (t - bb)) + (x - bb);
            hi = t;
        }
        tot = CSum{hi, lo};
    }
    __syncwarp();
}
// value k's total in lanes 2 k, 2 k + 1
__device__ __forceinline__ double total2(const CSum &t)
{
    const float oh = __shfl_xor_sync(kFull, t.hi, 1), ol = __shfl_xor_sync(kFull, t.lo, 1);
    const float s = t.hi + oh, bb = s - t.hi;
    return (double)s + (double)((t.lo + ol) + ((t.hi - (s - bb)) + (oh - bb)));
}

// The walk of one warp over the candidates of particles a0 and a1 = a0 + 1 of cell (cx, cy) (two =
// false: a0 alone).  pair(which, entry) receives an accepted pair per lane; flush() is called before a
// particle has kRun batches behind it and at the end, with empty queues.
// nacc: accepted candidates (self included); shell: candidates decided by the FP64 test.
template <class Pair, class Flush>
__device__ __forceinline__ void walk9_two(const EvView &v, const double *__restrict__ y,
                                          const float2 *__restrict__ rel, const uint32_t *__restrict__ start,
                                          const uint32_t *__restrict__ cnt, int a0, bool two, int cx, int cy, float2 ra0,
                                          float2 ra1, WalkMem2 &M, int lane, int &nacc0, int &nacc1, unsigned &shell,
                                          Pair &&pair, Flush &&flush)
{
    const size_t n = (size_t)v.n;
    const unsigned lt = (1u << lane) - 1u;
    const float slo = v.shell_lo, shi = v.shell_hi, cell = v.cell_f;
    const int lim = 1 << v.B;
    if (!two) ra1 = make_float2(kFar, kFar);  // never accepted
    // lane t < 9: the neighbour cell t, kept when it holds particles and its box lies within 2h
    // (with a margin far above the positions' rounding) of either particle
    int st = 0, len = 0;
    if (lane < 9) {
        const int ox = lane % 3 - 1, oy = lane / 3 - 1, nx = cx + ox, ny = cy + oy;
        auto gap = [&](int o, float p) { return o < 0 ? p : (o > 0 ? cell - p : 0.0f); };
        auto dist = [&](float2 p) {
            const float gx = gap(ox, p.x), gy = gap(oy, p.y);
            return fmaf(fmaxf(gx, 0.0f), gx, fmaxf(gy, 0.0f) * gy);
        };
        const float lim2 = shi * 1.0001f;
        // written so that a NaN position keeps the cell
        if (nx >= 0 && nx < lim && ny >= 0 && ny < lim && (!(dist(ra0) > lim2) || (two && !(dist(ra1) > lim2)))) {
            const uint32_t k = morton2((uint32_t)nx, (uint32_t)ny);
            st = (int)start[k];
            len = (int)cnt[k];
        }
    }
    unsigned cells = __ballot_sync(kFull, len > 0);
    const float2 ax = make_float2(ra0.x, ra1.x), ay = make_float2(ra0.y, ra1.y);
    int qn0 = 0, qn1 = 0, nb = 0;
    while (cells) {
        const int o = __ffs(cells) - 1;
        cells &= cells - 1u;
        const int b0 = __shfl_sync(kFull, st, o), ln = __shfl_sync(kFull, len, o);
        const float ox = -(float)(o % 3 - 1) * cell, oy = -(float)(o / 3 - 1) * cell;
        for (int base = 0; base < ln; base += 32) {
            const int b = b0 + base + lane;
            float2 rb = make_float2(-kFar, -kFar);
            if (base + lane < ln) rb = rel[b];
            // (r_a - r_b) - o (2h), rounded step by step as the shell bound assumes
            const float2 dx = __fadd2_rn(__fadd2_rn(ax, make_float2(-rb.x, -rb.x)), make_float2(ox, ox));
            const float2 dy = __fadd2_rn(__fadd2_rn(ay, make_float2(-rb.y, -rb.y)), make_float2(oy, oy));
            const float2 r2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
            bool acc0 = r2.x <= shi, acc1 = r2.y <= shi;
            if ((acc0 && r2.x >= slo) || (acc1 && r2.y >= slo)) {  // thin shell: the exact FP64 decision
                const double xb = y[b], yb = y[n + b];
                if (acc0 && r2.x >= slo) {
                    acc0 = dist2_2d(y[a0] - xb, y[n + a0] - yb) < v.supp2;
                    ++shell;
                }
                if (acc1 && r2.y >= slo) {
                    acc1 = dist2_2d(y[a0 + 1] - xb, y[n + a0 + 1] - yb) < v.supp2;
                    ++shell;
                }
            }
            const unsigned m0 = __ballot_sync(kFull, acc0), m1 = __ballot_sync(kFull, acc1);
            if (acc0) M.q[0][qn0 + __popc(m0 & lt)] = make_float4(dx.x, dy.x, r2.x, __int_as_float(b));
            if (acc1) M.q[1][qn1 + __popc(m1 & lt)] = make_float4(dx.y, dy.y, r2.y, __int_as_float(b));
            qn0 += __popc(m0);
            qn1 += __popc(m1);
            nacc0 += __popc(m0);
            nacc1 += __popc(m1);
            if (qn0 >= 32) {
                __syncwarp();
                pair(0, M.q[0][lane]);
                const float4 rest = M.q[0][32 + lane];
                __syncwarp();
                qn0 -= 32;
                if (lane < qn0) M.q[0][lane] = rest;
                ++nb;
            }
            if (qn1 >= 32) {
                __syncwarp();
                pair(1, M.q[1][lane]);
                const float4 rest = M.q[1][32 + lane];
                __syncwarp();
                qn1 -= 32;
                if (lane < qn1) M.q[1][lane] = rest;
                ++nb;
            }
            if (nb >= kRun - 1) {  // at most kRun plain terms per lane and particle, these partial batches included
                __syncwarp();
                if (lane < qn0) pair(0, M.q[0][lane]);
                if (lane < qn1) pair(1, M.q[1][lane]);
                qn0 = qn1 = nb = 0;
                flush();
            }
        }
    }
    __syncwarp();
    if (lane < qn0) pair(0, M.q[0][lane]);
    if (lane < qn1) pair(1, M.q[1][lane]);
    flush();
}

// Density pass (row a3).
__global__ void __launch_bounds__(32 * kWW, 4) k_walk_density2m(EvView v, const double *__restrict__ y,
                                                             const float2 *__restrict__ rel,
                                                             const float4 *__restrict__ fq,
                                                             const uint32_t *__restrict__ start,
                                                             const uint32_t *__restrict__ cnt,
                                                             const uint32_t *__restrict__ key,
                                                             const uint32_t *__restrict__ perm,
                                                             double *__restrict__ dens, int *__restrict__ nnb)
{
    __shared__ WalkMem2 mem[kWW];
    __shared__ unsigned s_pairs, s_shell;
    if (threadIdx.x == 0) s_pairs = s_shell = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t n = (size_t)v.n;
    float *red = reinterpret_cast<float *>(&mem[wid]);
    const long long w = (long long)blockIdx.x * kWW + wid;
    const float ih = (float)v.inv_h;
    unsigned shell = 0u, pairs = 0u;
    for (int a0 = (int)min(2 * w, (long long)v.n), end = min(a0 + 2, v.n); a0 < end;) {  // warp-uniform
        const int a1 = min(a0 + 1, end - 1);
        const uint32_t k0 = key[perm[a0]], k1 = key[perm[a1]];
        const bool two = a1 > a0 && k0 == k1;
        float s0[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, s1[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
        CSum tot = {0.f, 0.f};
        int n0 = 0, n1 = 0;
        auto pair = [&](int which, float4 e) {
            const float4 qb = fq[__float_as_int(e.w)];
            const float q = sqrt_apx(e.z) * ih;
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
        auto flush = [&]() { flush2<5>(red, s0, s1, lane, tot); };
        walk9_two(v, y, rel, start, cnt, a0, two, (int)unspread2(k0), (int)unspread2(k0 >> 1), rel[a0], rel[a1], mem[wid],
                  lane, n0, n1, shell, pair, flush);
        const double d = v.sigma_d * total2(tot);
        const int k = lane >> 1;
        if (!(lane & 1) && k < (two ? 10 : 5)) dens[(size_t)(k < 5 ? k : k - 5) * n + a0 + (k < 5 ? 0 : 1)] = d;
        if (lane == 0) {
            nnb[a0] = n0;
            pairs += (unsigned)n0;
            if (two) {
                nnb[a0 + 1] = n1;
                pairs += (unsigned)n1;
            }
        }
        a0 += two ? 2 : 1;
    }
    shell = __reduce_add_sync(kFull, shell);
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

// Gradient pass (row a5).  The 8 sums: grad W (x, y), sum_b X_b grad W (x, y), sum_b u_b grad W
// (d_x u^x, d_x u^y, d_y u^x, d_y u^y).
__global__ void __launch_bounds__(32 * kWW, 4) k_walk_gradient2m(EvView v, int stage, const double *__restrict__ y,
                                                              const float2 *__restrict__ rel,
                                                              const double *__restrict__ gin,
                                                              const uint32_t *__restrict__ start,
                                                              const uint32_t *__restrict__ cnt,
                                                              const uint32_t *__restrict__ key,
                                                              const uint32_t *__restrict__ perm,
                                                              double *__restrict__ gout)
{
    __shared__ WalkMem2 mem[kWW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t n = (size_t)v.n;
    float *red = reinterpret_cast<float *>(&mem[wid]);
    const long long w = (long long)blockIdx.x * kWW + wid;
    const float ih = (float)v.inv_h;
    const float2 *fU = reinterpret_cast<const float2 *>(v.fX + n);
    for (int a0 = (int)min(2 * w, (long long)v.n), end = min(a0 + 2, v.n); a0 < end;) {  // warp-uniform
        const int a1 = min(a0 + 1, end - 1);
        const uint32_t k0 = key[perm[a0]], k1 = key[perm[a1]];
        const bool two = a1 > a0 && k0 == k1;
        float s0[8], s1[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) s0[k] = s1[k] = 0.0f;
        CSum tot = {0.f, 0.f};
        int n0 = 0, n1 = 0;
        unsigned shell = 0u;
        auto pair = [&](int which, float4 e) {
            const int b = __float_as_int(e.w);
            const float4 X = v.fX[b];
            const float2 U = fU[b];
            // r = 0 (the particle itself) gives dw/dq = 0: a zero term
            const float ir = rsqrt_apx(fmaxf(e.z, 1e-30f));
            const float q = (e.z * ir) * ih;
            const float t = 2.0f - q, u = fmaxf(1.0f - q, 0.0f);
            const float fac = fmaf(-0.75f, t * t, 3.0f * (u * u)) * ir;
            const float gx = fac * e.x, gy = fac * e.y;
            float(&s)[8] = which ? s1 : s0;
            s[0] += gx;
            s[1] += gy;
            s[2] = fmaf(X.x, gx, fmaf(X.z, gy, s[2]));
            s[3] = fmaf(X.y, gx, fmaf(X.w, gy, s[3]));
            s[4] = fmaf(U.x, gx, s[4]);
            s[5] = fmaf(U.y, gx, s[5]);
            s[6] = fmaf(U.x, gy, s[6]);
            s[7] = fmaf(U.y, gy, s[7]);
        };
        auto flush = [&]() { flush2<8>(red, s0, s1, lane, tot); };
        walk9_two(v, y, rel, start, cnt, a0, two, (int)unspread2(k0), (int)unspread2(k0 >> 1), rel[a0], rel[a1], mem[wid],
                  lane, n0, n1, shell, pair, flush);
        const double d = total2(tot);
        const int k = (lane >> 1) & 7, first = lane & 16;  // lanes 0-15: a0's values, 16-31: a1's
        const size_t a = (size_t)a0 + (lane >> 4);
        const double Gx = __shfl_sync(kFull, d, first), Gy = __shfl_sync(kFull, d, first + 2);
        if (!(lane & 1) && k >= 2 && (lane < 16 || two)) {
            const double c = v.sigma_d * v.inv_h;
            if (k >= 4) {
                gout[(size_t)(k - 4) * n + a] = c * d;
            } else {
                // minus the stress divergence: X_a . sum grad W + sum X_b grad W, times sqrt(-g)
                const double tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
                const double sqrtg = v.milne ? tau : 1.0;
                const double X0 = gin[(size_t)(k - 2) * n + a], X1 = gin[(size_t)k * n + a];
                gout[(size_t)(k + 2) * n + a] = -sqrtg * c * (X0 * Gx + X1 * Gy + d);
            }
        }
        a0 += two ? 2 : 1;
    }
}

inline int nblk(int n, int t) { return (n + t - 1) / t; }

}  // namespace

void launch_density2m(const EvView &v, const double *y, const double *Nq, CellBufs cb, double *dens, int *nnb,
                      cudaStream_t st)
{
    k_fq2<<<nblk(v.n, 256), 256, 0, st>>>(v, y, Nq, cb.fq, dens);
    k_walk_density2m<<<nblk(v.n, 2 * kWW), 32 * kWW, 0, st>>>(v, y, cb.fpos, cb.fq, cb.start, cb.cnt, cb.key, cb.perm, dens,
                                                              nnb);
}

void launch_gradient2m(const EvView &v, int stage, const double *y, const double *gin, CellBufs cb, double *gout,
                       cudaStream_t st)
{
    k_walk_gradient2m<<<nblk(v.n, 2 * kWW), 32 * kWW, 0, st>>>(v, stage, y, cb.fpos, gin, cb.start, cb.cnt, cb.key, cb.perm,
                                                               gout);
}

}  // namespace sphg
