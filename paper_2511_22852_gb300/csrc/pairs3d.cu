// pairs3d.cu -- plain 3D neighbour passes over half-pair lists: the 3D counterpart of the plain
// 2D passes (the same rows and fallback), over the 27 cells of the generalized Morton table.  Per
// accepted pair the forward pass evaluates W and grad W once (both depend on r_ab only; grad_b W_ba
// = -grad_a W_ab) and keeps them in both particles' rows; the sum and gradient passes
// add them in integers (pairs_fixed.cuh), independent of the order: reproducible.
#include "pairs_fixed.cuh"
#include "sph_internal.cuh"

namespace sphg {

namespace {

constexpr int kWarps = 4;
constexpr unsigned kFull = 0xFFFFFFFFu;

// Forward pass, a warp for two particles a.  Candidates of the cells from its own on (those within
// 2h of a) pass the single-precision prefilter; a candidate b > a is queued, and 32 at a time -- of
// both particles -- the exact test (where the float test left the pair undecided) and the kernel in
// integers (pair_kernel) run on full warps.  W and grad W go into a's row and, at a place taken
// from b's counter, into b's row.  The particles' own values go into limbs.
// (Listing b < a in a's own walk, and finding its W by a search in b's row, kept the sums waiting
// for memory: 258 k particles, sum pass 2.5 -> 0.9, gradient pass 3.4 -> 2.6 ms a stage, with the sums'
// units taken from the values alone.)
// Bound: the L2 sectors of the scattered writes to b's row.  The three components of grad W lie in
// one 32-byte sector and are written by one store (three 8-byte stores at a stride of 24 bytes
// wrote 7.6 sectors a pair against 4.4); with that and 6 FP64 operations per unordered pair (15
// with the kernel's distance in FP64), 258 k particles: both density passes 4.36 -> 3.24 ms a stage, the
// gradient pass, which reads 36 instead of 28 bytes an entry, 2.6 -> 2.9.  The integers alone gave
// nothing here (the stores bound it), the layout alone was not measured.  W in the record's fourth
// word, read by the sum pass at a stride of 32 bytes: both passes 2 ms a stage more at 1.01 M particles.
// Now 2.57 ms a stage at 258 k (3.5 with the sum pass).
__global__ void __launch_bounds__(32 * kWarps, 8) k_pairs3_fwd(EvView v, const double *__restrict__ y,
                                                           const float4 *__restrict__ fpos,
                                                           const double *__restrict__ Nq,
                                                           const uint32_t *__restrict__ start,
                                                           const uint32_t *__restrict__ cnt, PairBufs pl)
{
    __shared__ int queue[kWarps][64];
    // the two particles of a warp: position, first entry and size of the row
    __shared__ double pos_[kWarps][2][3];
    __shared__ long long row_[kWarps][2];
    __shared__ int cap_[kWarps][2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = v.n;
    const long long a0 = 2 * ((long long)blockIdx.x * kWarps + wid);
    if (a0 >= n) return;  // warp-uniform
    const int np = a0 + 1 < n ? 2 : 1;
    int *q = queue[wid];
    const double *X = y, *Y = y + n, *Z = y + 2 * (size_t)n, *S = y + 6 * (size_t)n;
    if (lane < 4 * np) {
        const size_t a = (size_t)a0 + (lane >> 2);
        const int k = lane & 3;
        fx_store_value(pl.Q, pl.Qe, a, k, k == 0 ? S[a] : Nq[(size_t)(k - 1) * n + a]);
    }
    const unsigned lt = (1u << lane) - 1u;
    const double (*pos)[3] = pos_[wid];
    const long long *row = row_[wid];
    const int *cap = cap_[wid];
    int nf[2] = {0, 0}, qn = 0;
    if (lane < 2) {
        const int a = (int)a0 + (lane < np ? lane : 0);
        pos_[wid][lane][0] = X[a];
        pos_[wid][lane][1] = Y[a];
        pos_[wid][lane][2] = Z[a];
        const long long r0 = pl.off[a], r1 = pl.off[a + 1];
        row_[wid][lane] = r0;
        cap_[wid][lane] = r1 <= pl.total ? (int)(r1 - r0) : 0;  // rows beyond the allocation write nothing
    }
    __syncwarp();
    // queued word: bit 31: the float test left the pair undecided (exact test needed), bit 30: of a0 + 1
    auto forward = [&](int qb, bool valid) {
        const int b = qb & 0x3FFFFFFF;
        const int p = qb >> 30 & 1;
        double dx = 0.0, dy = 0.0, dz = 0.0;
        bool acc = false;
        if (valid) {
            dx = pos[p][0] - X[b];
            dy = pos[p][1] - Y[b];
            dz = pos[p][2] - Z[b];
            acc = qb >= 0 || dist2_3d(dx, dy, dz) < v.supp2;
        }
        const unsigned m0 = __ballot_sync(kFull, acc && p == 0), m1 = __ballot_sync(kFull, acc && p == 1);
        if (acc) {
            // b's row and the place in it first: the loads and the atomic wait behind the arithmetic
            const long long rb = pl.off[b], rb1 = pl.off[b + 1];
            const int place = atomicAdd(&pl.cntB[b], 1);
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            double w, g[3];
            pair_kernel<3>({dx, dy, dz}, r2, v.inv_h, w, g);
            const int slot = (p ? nf[1] : nf[0]) + __popc((p ? m1 : m0) & lt);
            if (slot < cap[p]) {
                const long long i = row[p] + slot;
                pl.L[i] = b;
                pl.W[i] = w;
                pl.G3[i] = double4_32a{g[0], g[1], g[2], 0.0};
            }
            const long long i = rb1 - 1 - place;
            if (i >= rb && rb1 <= pl.total) {
                pl.L[i] = (int)a0 + p;
                pl.W[i] = w;
                pl.G3[i] = double4_32a{-g[0], -g[1], -g[2], 0.0};
            }
        }
        nf[0] += __popc(m0);
        nf[1] += __popc(m1);
    };
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        if (p >= np) break;
        const int a = (int)a0 + p, flag = p << 30;
        const float4 fa = fpos[a];
        const int ca = __float_as_int(fa.w);  // the packed cell coordinates
        const int c[3] = {ca & 1023, (ca >> 10) & 1023, (ca >> 20) & 1023};
        const uint32_t ka = key3(v, c[0], c[1], c[2]);
        // lane o < 27: the neighbour cell o, kept when it holds particles behind a within 2h of it
        uint32_t k = 0u, st = 0u, len = 0u;
        if (lane < 27) {
            const int o[3] = {lane % 3 - 1, (lane / 3) % 3 - 1, lane / 9 - 1};
            const float f[3] = {fa.x, fa.y, fa.z};
            bool in = true;
            float d = 0.0f;
            int m[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                m[i] = c[i] + o[i];
                in = in && m[i] >= 0 && m[i] < (1 << v.B3[i]);
                const float g = cell_gap(o[i], f[i], c[i], v.cell_f);
                d = fmaf(g, g, d);
            }
            if (in && !(d > v.supp2_hi)) {
                k = key3(v, m[0], m[1], m[2]);
                st = start[k];
                len = k < ka ? 0u : cnt[k];  // below ka: all of its particles come before a
            }
        }
        // batches of 32 candidates, each loaded while the one before is tested; b > a in all of them
        // (lanes past a cell's end hold NaN: never candidates)
        const float kNaN = __int_as_float(0x7FFFFFFF);
        unsigned cells = __ballot_sync(kFull, len > 0u);
        uint32_t base = 0u, b1 = 0u;
        auto next = [&]() {
            base += 32u;
            while (base >= b1 && cells) {
                const int o = __ffs(cells) - 1;
                cells &= cells - 1u;
                base = __shfl_sync(kFull, st, o);
                b1 = base + __shfl_sync(kFull, len, o);
                if (__shfl_sync(kFull, k, o) == ka) base = (uint32_t)a + 1u;
            }
            return base < b1;
        };
        auto load = [&](bool on) { return on && base + lane < b1 ? fpos[base + lane] : make_float4(kNaN, 0.0f, 0.0f, 0.0f); };
        bool more = next();
        float4 fn = load(more);
        while (more) {
            const uint32_t b = base + lane;
            const float4 fb = fn;
            more = next();
            fn = load(more);
            const float dx = fa.x - fb.x, dy = fa.y - fb.y, dz = fa.z - fb.z;
            const float r2f = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            const bool cand = r2f <= v.supp2_hi, sure = r2f < v.supp2_lo;
            const unsigned m = __ballot_sync(kFull, cand);
            if (cand) q[qn + __popc(m & lt)] = (int)(b | (sure ? 0u : 0x80000000u)) | flag;
            qn += __popc(m);
            __syncwarp();
            if (qn >= 32) {
                forward(q[lane], true);
                qn -= 32;
                __syncwarp();
                if (lane < qn) q[lane] = q[32 + lane];
                __syncwarp();
            }
        }
    }
    if (qn > 0) forward(lane < qn ? q[lane] : 0, lane < qn);
    if (lane == 0)
        for (int p = 0; p < np; ++p) pl.cntF[a0 + p] = nf[p];
}

// Gradient pass, half a warp per particle a, over the entries of its row, in integers
// (pairs_fixed.cuh): sum grad W (3), sum X_b^{j i} grad_j W (3), sum u_b^j grad_k W (9); the
// epilogue as the per-particle pass.
// Each sum in the unit of its own largest term, from a first look over the exponents.
// Bound: issue (59 %) and the gathers of four 32-byte words; 258 k particles: 3.7 ms a stage (2.9 with
// one unit for the stresses and one for u, from the values alone; 6.0 with 21 FP64 operations per
// pair).  4 blocks per SM (1.01 M particles: 3 took 1 % less, at 269 k 6 % more; 5 took 15 % more).  The
// first look without the gradients (looser units) takes 3 % less, without any look 13 %, one unit
// for all stresses and one for u 13 %; unrolling the look by 2 or 4, or prefetching it: none or worse.
__global__ void __launch_bounds__(32 * kWarps, 4) k_pairs3_gradient(EvView v, int stage, const double *__restrict__ gin,
                                                                 PairBufs pl, double *__restrict__ gout)
{
    if (v.sc->pair_flag) return;  // a list overflowed: the per-particle pass runs instead
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, l = lane & 15;
    const long long ap = 2 * ((long long)blockIdx.x * kWarps + wid) + (lane >> 4);
    if (ap - (lane >> 4) >= v.n) return;  // warp-uniform
    const bool on = ap < v.n;
    const int a = on ? (int)ap : v.n - 1;
    const size_t n = (size_t)v.n;
    const long long r0 = pl.off[a], r1 = pl.off[a + 1];
    const int nf = on ? pl.cntF[a] : 0, nt = on ? nf + pl.cntB[a] : 0;
    const int *L = pl.L + r0;
    const double4_32a *G = pl.G3 + r0;
    const int gap = (int)(r1 - r0) - nt;
    auto at = [&](int j) { return j + (j < nf ? 0 : gap); };  // entry j of a's row
    // the largest exponents among the terms of each sum, two in 16-bit halves: mG g_1 | g_2 and g_3, mH H_1 |
    // H_2, mD[k] H_3 (its terms of k) | u^k g_k, mU[k] the two u^j g_k with j != k, ascending
    unsigned mG[2] = {0u, 0u}, mH = 0u, mD[3] = {0u, 0u, 0u}, mU[3] = {0u, 0u, 0u};
    // u^j of j != k from the words (X^{j3} | u^j)
    auto others = [](const unsigned (&w)[3], int k) { return __byte_perm(w[k == 0 ? 1 : 0], w[k == 2 ? 1 : 2], 0x7632); };
    for (int j = l; j < nt; j += 16) {
        const int i = at(j);
        const int b = L[i];
        const double4_32a g = G[i];
        const Limb4 e = pl.X[3 * n + b];
        const unsigned eA[3] = {word_lo(e.x), word_lo(e.y), word_lo(e.z)}, eB[3] = {word_hi(e.x), word_hi(e.y), word_hi(e.z)};
        const int eg[3] = {fx_kexp(g.x), fx_kexp(g.y), fx_kexp(g.z)};
        mG[0] = fx_max2(mG[0], fx_pair(eg[0], eg[1]));
        mG[1] = fx_max2(mG[1], (unsigned)eg[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const unsigned g2 = fx_pair(eg[k], eg[k]);
            mH = fx_max2(mH, eA[k] + g2);
            mD[k] = fx_max2(mD[k], eB[k] + g2);
            mU[k] = fx_max2(mU[k], others(eB, k) + g2);
        }
    }
    mH = fx_half_max2(mH);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (k < 2) mG[k] = fx_half_max2(mG[k]);
        mD[k] = fx_half_max2(mD[k]);
        mU[k] = fx_half_max2(mU[k]);
    }
    {
        // one unit for H_3; room for rows of many entries
        const unsigned h3 = fx_max2(fx_max2(mD[0], mD[1]), mD[2]) & 0xFFFFu, room = (unsigned)fx_room(0, nt) * 0x10001u;
        mG[0] += room;
        mG[1] += room;
        mH += room;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            mD[k] = ((mD[k] & 0xFFFF0000u) | h3) + room;
            mU[k] += room;
        }
    }
    FxSum sG[3], sH[3], sU[9];  // sum g; sum_j X^{j i} g_j; 3 k + j: sum u^j g_k
#pragma unroll
    for (int k = 0; k < 3; ++k) sG[k] = sH[k] = sU[k] = sU[3 + k] = sU[6 + k] = FxSum{0, 0};
    auto fold = [&]() {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            fx_fold(sG[k]);
            fx_fold(sH[k]);
            fx_fold(sU[k]);
            fx_fold(sU[3 + k]);
            fx_fold(sU[6 + k]);
        }
    };
    // the next entry's index and gradient are loaded while the current one is added
    auto entry = [&](int j, int &b, double (&g)[3]) {
        b = a;
        g[0] = g[1] = g[2] = 0.0;
        if (j < nt) {
            const int i = at(j);
            b = L[i];
            const double4_32a e = G[i];
            g[0] = e.x;
            g[1] = e.y;
            g[2] = e.z;
        }
    };
    int b1;
    double g1[3];
    entry(l, b1, g1);
    for (int j = l, it = 1; j < nt; j += 16, ++it) {
        const int b = b1;
        const double g[3] = {g1[0], g1[1], g1[2]};
        const Limb4 x0 = pl.X[b], x1 = pl.X[n + b], x2 = pl.X[2 * n + b], e = pl.X[3 * n + b];
        entry(j + 16, b1, g1);
        const long long x[12] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w, x2.x, x2.y, x2.z, x2.w};
        const unsigned eA[3] = {word_lo(e.x), word_lo(e.y), word_lo(e.z)}, eB[3] = {word_hi(e.x), word_hi(e.y), word_hi(e.z)};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const long long m = fx_kmant(g[k]);
            const int eg = fx_kexp(g[k]);
            const unsigned g2 = fx_pair(eg, eg);
            // the shifts of the terms X^{k i} g_k and u^j g_k, two in a word (an entry past the end has m = 0)
            const unsigned dH = mH - eA[k] - g2, dD = mD[k] - eB[k] - g2, dU = mU[k] - others(eB, k) - g2;
            sG[k].x += fx_shift(m, (k == 0 ? fx_lo(mG[0]) : (k == 1 ? fx_hi(mG[0]) : fx_lo(mG[1]))) - eg + kGuard);
            auto term = [&](FxSum &s, int d, int i) {
                int hi, lo;
                fx_split(m, d, hi, lo);
                fx_add(s, hi, lo, fx_pair_of(x[i]));
            };
            term(sH[0], fx_lo(dH), 3 * k);
            term(sH[1], fx_hi(dH), 3 * k + 1);
            term(sH[2], fx_lo(dD), 3 * k + 2);
            term(sU[4 * k], fx_hi(dD), 9 + k);
            term(sU[3 * k + (k == 0 ? 1 : 0)], fx_lo(dU), 9 + (k == 0 ? 1 : 0));
            term(sU[3 * k + (k == 2 ? 1 : 2)], fx_hi(dU), 9 + (k == 2 ? 1 : 2));
        }
        if ((it & (kFoldEvery - 1)) == 0) fold();
    }
    fold();
    FxTotal t[16];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        t[k] = fx_words(sG[k]);
        t[3 + k] = fx_words(sH[k]);
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) t[6 + k] = fx_words(sU[k]);
    t[15] = FxTotal{0, 0};
    const FxTotal tt = fx_reduce16(t, lane);
    // the unit of the lane's sum: 0-2 g, 3-5 H, 6 + 3 k + j u^j g_k
    const int E[15] = {fx_lo(mG[0]), fx_hi(mG[0]), fx_lo(mG[1]), fx_lo(mH), fx_hi(mH), fx_lo(mD[0]), fx_hi(mD[0]), fx_lo(mU[0]),
                       fx_hi(mU[0]), fx_lo(mU[1]), fx_hi(mD[1]), fx_hi(mU[1]), fx_lo(mU[2]), fx_hi(mU[2]), fx_hi(mD[2])};
    int El = E[0];
#pragma unroll
    for (int i = 1; i < 15; ++i)
        if (l == i) El = E[i];
    double tot = fx_value(tt, l < 3 ? fx_kunit(El) : fx_unit(El));
    if (El >= kNonFinite) tot = fx_nan();
    const int h0 = lane & 16;
    const double G0 = __shfl_sync(kFull, tot, h0), G1 = __shfl_sync(kFull, tot, h0 + 1), G2 = __shfl_sync(kFull, tot, h0 + 2);
    if (on && l >= 3 && l < 15) {
        const double c = v.sigma_d * v.inv_h;
        if (l >= 6) {
            gout[(size_t)(l - 6) * n + a] = c * tot;  // d_k u^j at 3 k + j
        } else {
            // minus the stress divergence: H_i + sum_j X_a^{j i} G_j, times sqrt(-g)
            const int i = l - 3;
            const double tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
            const double sqrtg = v.milne ? tau : 1.0;
            double F = tot;
            F = fma(gin[(size_t)(0 + i) * n + a], G0, F);
            F = fma(gin[(size_t)(3 + i) * n + a], G1, F);
            F = fma(gin[(size_t)(6 + i) * n + a], G2, F);
            gout[(size_t)(9 + i) * n + a] = -sqrtg * c * F;
        }
    }
}

inline int nblk(int n, int t) { return (n + t - 1) / t; }

}  // namespace

void launch_pairs3_density(const EvView &v, const double *y, const double *Nq, CellBufs cb, double *dens, int *nnb,
                           cudaStream_t st)
{
    launch_pair_rows(v, cb, st);
    k_pairs3_fwd<<<nblk(v.n, 2 * kWarps), 32 * kWarps, 0, st>>>(v, y, cb.fpos3, Nq, cb.start, cb.cnt, cb.pl);
    launch_pairs_sum(v, cb, dens, nnb, st);
}

void launch_pairs3_gradient(const EvView &v, int stage, const double *y, const double *gin, CellBufs cb,
                            double *gout, cudaStream_t st)
{
    (void)y;
    k_pairs3_gradient<<<nblk(v.n, 2 * kWarps), 32 * kWarps, 0, st>>>(v, stage, gin, cb.pl, gout);
}

}  // namespace sphg
