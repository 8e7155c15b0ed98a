// pairs2d.cu -- plain 2D neighbour passes over half-pair lists.
//
// The density sums (Sec. "SPH formalism": sigma*, s*, n*_q as kernel sums) and the gradient sums
// (Sec. "SPH formalism", the n = 0 and n = -1 derivative forms) use W(r_ab) and dW/dr(r_ab) / r_ab
// of every accepted pair; both depend on r_ab only, so they are the same for (a, b) and (b, a).
// Each stage's forward pass evaluates them once per unordered pair -- on the pairs b > a of particle
// a (sorted index) -- and keeps them with the pair; the sum and gradient passes then add every pair's
// contribution to both of its particles in integers (pairs_fixed.cuh), which do not depend on the
// order, so results are reproducible run to run.
//
// FP64 operations per unordered pair fall from 56 (26 for the kernel, 10 for the density and 20 for
// the gradient sums of its two particles) to 4; the 40 k event's step 2,038 -> 1,272 us.
//
// Rows: a particle's row holds its previous neighbour count plus a margin (a prefix scan per
// stage); forward entries fill it from the start, backward entries from the end.
#include "pairs_fixed.cuh"
#include "sph_internal.cuh"

namespace sphg {

namespace {

constexpr int kWarps = 4;  // particles (warps) per block
constexpr unsigned kFull = 0xFFFFFFFFu;

// ---------------------------------------------------------------------------
// Row offsets: row j (sorted order) holds cnt_src[perm[j]] - 1 + margin entries (the previous
// neighbour count without the self pair); off = exclusive prefix sums, off[n] = entries needed.
constexpr int kScanThreads = 256, kScanPer = 8, kScanTile = kScanThreads * kScanPer;

__device__ __forceinline__ long long row_size(const PairBufs &pl, const uint32_t *perm, int j)
{
    const int c = pl.cnt_src[perm[j]];
    return (long long)(c > 1 ? c - 1 : 0) + pl.margin;
}

__global__ void __launch_bounds__(kScanThreads) k_rows_part(int n, const uint32_t *__restrict__ perm, PairBufs pl)
{
    __shared__ long long ws[kScanThreads / 32];
    const int base = blockIdx.x * kScanTile + threadIdx.x * kScanPer;
    long long t = 0;
    for (int k = 0; k < kScanPer; ++k)
        if (base + k < n) t += row_size(pl, perm, base + k);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long b = 0;
        for (int w = 0; w < kScanThreads / 32; ++w) b += ws[w];
        pl.part[blockIdx.x] = (unsigned long long)b;
    }
}

// exclusive scan of the block sums (one block); off[n] = total; rows beyond the allocation flag
// the stage (the per-particle passes run).  Bound: latency; 3.3 us (8.1 with one thread scanning the
// block's sums)
__global__ void __launch_bounds__(1024) k_rows_top(int n, int nparts, PairBufs pl, DevScalars *sc)
{
    __shared__ unsigned long long tot[32];
    const int t = threadIdx.x, lane = t & 31, per = (nparts + 1023) / 1024;
    const int b0 = min(t * per, nparts), b1 = min(b0 + per, nparts);
    unsigned long long s = 0;
    for (int i = b0; i < b1; ++i) s += pl.part[i];
    unsigned long long incl = s;  // over the warp, then over the warps
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long x = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) tot[t >> 5] = incl;
    __syncthreads();
    unsigned long long run = incl - s;
    for (int w = 0; w < (t >> 5); ++w) run += tot[w];
    if (t == 1023) {
        const long long all = (long long)(run + s);
        pl.off[n] = all;
        if (all > pl.total) atomicOr(&sc->pair_flag, 1u);
    }
    for (int i = b0; i < b1; ++i) {
        const unsigned long long x = pl.part[i];
        pl.part[i] = run;
        run += x;
    }
}

__global__ void __launch_bounds__(kScanThreads) k_rows_apply(int n, const uint32_t *__restrict__ perm, PairBufs pl)
{
    __shared__ long long ws[kScanThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int base = blockIdx.x * kScanTile + threadIdx.x * kScanPer;
    long long v[kScanPer], t = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        v[k] = base + k < n ? row_size(pl, perm, base + k) : 0;
        t += v[k];
    }
    long long incl = t;  // inclusive scan over the warp
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[wid] = incl;
    __syncthreads();
    long long wbase = 0;
    for (int w = 0; w < wid; ++w) wbase += ws[w];
    long long run = (long long)pl.part[blockIdx.x] + wbase + incl - t;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        if (base + k < n) {
            pl.off[base + k] = run;
            pl.cntB[base + k] = 0;  // counted up by the forward pass
        }
        run += v[k];
    }
}

// Forward pass, a warp for two particles a.  Candidates of the cells from its own on (those within
// 2h of a) pass the single-precision prefilter; a candidate b > a is queued, and 32 at a time -- of
// both particles -- the exact test (where the float test left the pair undecided) and the kernel in
// integers (pair_kernel) run on full warps.  W and grad W go into a's row and, at a place taken
// from b's counter, into b's row.  The particles' own values go into limbs.
// (Listing b < a in a's own walk, and finding its W by a search in b's row, kept the sums waiting
// for memory: 40 k event, sum pass 197 -> 92 us a stage, gradient pass 150 -> 137, with the sums' units
// taken from the values alone.)
// Bound: latency and the L2 sectors of the scattered writes (b's row: three sectors a pair).  4 FP64
// operations per unordered pair (12 with the kernel's distance in FP64, 31 with spline and sums).
// 40 k event: 195 us a stage (212 with the distance in FP64 and every cell walked, 325 with the
// spline in FP64).
__global__ void __launch_bounds__(32 * kWarps, 8) k_pairs_fwd(EvView v, const double *__restrict__ y,
                                                           const float2 *__restrict__ fpos,
                                                           const double *__restrict__ Nq,
                                                           const uint32_t *__restrict__ start,
                                                           const uint32_t *__restrict__ cnt,
                                                           const uint32_t *__restrict__ key,
                                                           const uint32_t *__restrict__ perm, PairBufs pl)
{
    __shared__ int queue[kWarps][64];
    // the two particles of a warp: position, first entry and size of the row
    __shared__ double pos_[kWarps][2][2];
    __shared__ long long row_[kWarps][2];
    __shared__ int cap_[kWarps][2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = v.n;
    const long long a0 = 2 * ((long long)blockIdx.x * kWarps + wid);
    if (a0 >= n) return;  // warp-uniform
    const int np = a0 + 1 < n ? 2 : 1;
    int *q = queue[wid];
    const double *X = y, *Y = y + n, *S = y + 4 * (size_t)n;
    if (lane < 4 * np) {
        const size_t a = (size_t)a0 + (lane >> 2);
        const int k = lane & 3;
        fx_store_value(pl.Q, pl.Qe, a, k, k == 0 ? S[a] : Nq[(size_t)(k - 1) * n + a]);
    }
    const unsigned lt = (1u << lane) - 1u;
    const double (*pos)[2] = pos_[wid];
    const long long *row = row_[wid];
    const int *cap = cap_[wid];
    int nf[2] = {0, 0}, qn = 0;
    if (lane < 2) {
        const int a = (int)a0 + (lane < np ? lane : 0);
        pos_[wid][lane][0] = X[a];
        pos_[wid][lane][1] = Y[a];
        const long long r0 = pl.off[a], r1 = pl.off[a + 1];
        row_[wid][lane] = r0;
        cap_[wid][lane] = r1 <= pl.total ? (int)(r1 - r0) : 0;  // rows beyond the allocation write nothing
    }
    __syncwarp();
    // queued word: bit 31: the float test left the pair undecided (exact test needed), bit 30: of a0 + 1
    auto forward = [&](int qb, bool valid) {
        const int b = qb & 0x3FFFFFFF;
        const int p = qb >> 30 & 1;
        double dx = 0.0, dy = 0.0;
        bool acc = false;
        if (valid) {
            dx = pos[p][0] - X[b];
            dy = pos[p][1] - Y[b];
            acc = qb >= 0 || dist2_2d(dx, dy) < v.supp2;
        }
        const unsigned m0 = __ballot_sync(kFull, acc && p == 0), m1 = __ballot_sync(kFull, acc && p == 1);
        if (acc) {
            // b's row and the place in it first: the loads and the atomic wait behind the arithmetic
            const long long rb = pl.off[b], rb1 = pl.off[b + 1];
            const int place = atomicAdd(&pl.cntB[b], 1);
            const double r2 = fma(dx, dx, dy * dy);
            double w, gk[2];
            pair_kernel<2>({dx, dy}, r2, v.inv_h, w, gk);
            const int slot = (p ? nf[1] : nf[0]) + __popc((p ? m1 : m0) & lt);
            const double2 g = make_double2(gk[0], gk[1]);
            if (slot < cap[p]) {
                const long long i = row[p] + slot;
                pl.L[i] = b;
                pl.W[i] = w;
                pl.G[i] = g;
            }
            const long long i = rb1 - 1 - place;
            if (i >= rb && rb1 <= pl.total) {
                pl.L[i] = (int)a0 + p;
                pl.W[i] = w;
                pl.G[i] = make_double2(-g.x, -g.y);
            }
        }
        nf[0] += __popc(m0);
        nf[1] += __popc(m1);
    };
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        if (p >= np) break;
        const int a = (int)a0 + p, flag = p << 30;
        const float2 fa = fpos[a];
        const uint32_t ka = key[perm[a]];
        const int cx = (int)unspread2(ka), cy = (int)unspread2(ka >> 1), lim = 1 << v.B;
        // lane o < 9: the neighbour cell o, kept when it holds particles behind a within 2h of it
        uint32_t k = 0u, st = 0u, len = 0u;
        if (lane < 9) {
            const int ox = lane % 3 - 1, oy = lane / 3 - 1, nx = cx + ox, ny = cy + oy;
            const float gx = cell_gap(ox, fa.x, cx, v.cell_f), gy = cell_gap(oy, fa.y, cy, v.cell_f);
            if (nx >= 0 && ny >= 0 && nx < lim && ny < lim && !(fmaf(gx, gx, gy * gy) > v.supp2_hi)) {
                k = morton2((uint32_t)nx, (uint32_t)ny);
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
        auto load = [&](bool on) { return on && base + lane < b1 ? fpos[base + lane] : make_float2(kNaN, 0.0f); };
        bool more = next();
        float2 fn = load(more);
        while (more) {
            const uint32_t b = base + lane;
            const float2 fb = fn;
            more = next();
            fn = load(more);
            const float dx = fa.x - fb.x, dy = fa.y - fb.y;
            const float r2f = fmaf(dx, dx, dy * dy);
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

// Density sums, half a warp per particle a, over the entries of its row, in integers, each in the unit
// of its own largest term (pairs_fixed.cuh).
// Bound: issue and the ALU pipe (67 and 66 % busy), then the latency of the gathers; 40 k event 95 us a
// stage, 3+1D event of 258 k particles 0.95 ms (92 and 0.92 with the units taken from the values alone,
// without the kernel value of the pair).
__global__ void __launch_bounds__(32 * kWarps, 7) k_pairs_sum(EvView v, PairBufs pl, double *__restrict__ dens,
                                                           int *__restrict__ nnb)
{
    if (v.sc->pair_flag) return;  // a list overflowed: the per-particle pass runs instead
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, l = lane & 15;
    const long long ap = 2 * ((long long)blockIdx.x * kWarps + wid) + (lane >> 4);
    if (ap - (lane >> 4) >= v.n) return;  // warp-uniform
    const bool on = ap < v.n;
    const int a = on ? (int)ap : v.n - 1;
    const size_t n = (size_t)v.n;
    const long long r0 = pl.off[a], r1 = pl.off[a + 1];
    const int nf = on ? pl.cntF[a] : 0, nb = on ? pl.cntB[a] : 0, nt = nf + nb;
    // the two ends met: the row does not hold a's entries (all listed values are pair values all the
    // same), and the per-particle passes run
    if (l == 0 && nt > (r1 <= pl.total ? (int)min(r1 - r0, (long long)nt) : 0)) atomicOr(&v.sc->pair_flag, 1u);
    const int fit = r1 <= pl.total && r1 - r0 >= nt ? nt : 0;
    // entry j of a's row
    auto at = [&](int j) { return j < nf ? r0 + j : r1 - nt + j; };
    const uint2 *Qe = reinterpret_cast<const uint2 *>(pl.Qe);
    // the largest exponents among the products q_b W of a (W = 1) and its neighbours (S | N_B << 16,
    // N_S | N_Q << 16)
    const unsigned one2 = fx_pair(1023, 1023);
    uint2 em = make_uint2(Qe[a].x + one2, Qe[a].y + one2);
    for (int j = l; j < fit; j += 16) {
        const long long i = at(j);
        const uint2 e = Qe[pl.L[i]];
        const int ew = fx_kexp(pl.W[i]);
        const unsigned w2 = fx_pair(ew, ew);
        em = make_uint2(fx_max2(em.x, e.x + w2), fx_max2(em.y, e.y + w2));
    }
    em = make_uint2(fx_half_max2(em.x), fx_half_max2(em.y));
    const int Em[4] = {fx_lo(em.x), fx_hi(em.x), fx_lo(em.y), fx_hi(em.y)};
    int E[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) E[k] = fx_room(Em[k], nt);
    FxSum sg = {0, 0};  // of W alone, the largest W(0) = 1: x in units of 2^-kMant
    FxSum s[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
    int it = 0;
    auto add = [&](double w, Limb4 q, uint2 e2) {
        const int e[4] = {fx_lo(e2.x), fx_hi(e2.x), fx_lo(e2.y), fx_hi(e2.y)};
        const long long qv[4] = {q.x, q.y, q.z, q.w};
        const long long m = fx_kmant(w);
        const int ew = fx_kexp(w);
        sg.x += fx_shift(m, 1023 - ew + kGuard);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            int whi, wlo;
            fx_split(m, E[k] - e[k] - ew, whi, wlo);
            fx_add(s[k], whi, wlo, fx_pair_of(qv[k]));
        }
    };
    // two entries at a time, their loads ahead of both; an entry past the end is a with weight 0
    auto add2 = [&](int b0, double w0, int b1, double w1) {
        const Limb4 q0 = pl.Q[b0], q1 = pl.Q[b1];
        const uint2 e0 = Qe[b0], e1 = Qe[b1];
        add(w0, q0, e0);
        add(w1, q1, e1);
        it += 2;
        if ((it & (kFoldEvery - 1)) == 0) {
            fx_fold(sg);
#pragma unroll
            for (int k = 0; k < 4; ++k) fx_fold(s[k]);
        }
    };
    if (l == 0 && on) add2(a, 1.0, a, 0.0);  // the self pair, W(0) = 1
    for (int j = l; j < fit; j += 32) {
        const bool two = j + 16 < fit;
        const long long i0 = at(j), i1 = at(j + 16);
        const int b0 = pl.L[i0], b1 = two ? pl.L[i1] : a;
        const double w0 = pl.W[i0], w1 = two ? pl.W[i1] : 0.0;
        add2(b0, w0, b1, w1);
    }
    fx_fold(sg);
    FxTotal t[8];
    t[0] = fx_words(sg);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        fx_fold(s[k]);
        t[1 + k] = fx_words(s[k]);
    }
    t[5] = t[6] = t[7] = FxTotal{0, 0};
    const FxTotal tot = fx_reduce8(t, lane);
    const int k = l >> 1;
    if (on && (l & 1) == 0 && k < 5) {
        // rows sigma*, lab-frame s* (divided by u0 sqrt(-g) in the EoS pass), n*_B, n*_S, n*_Q
        const int Ek = k <= 1 ? E[0] : (k == 2 ? E[1] : (k == 3 ? E[2] : E[3]));
        const bool bad = (k <= 1 ? Em[0] : (k == 2 ? Em[1] : (k == 3 ? Em[2] : Em[3]))) >= kNonFinite && k > 0;
        const double d = fx_value(tot, k == 0 ? -kMant : fx_unit(Ek));
        dens[(size_t)k * n + a] = bad ? fx_nan() : v.sigma_d * d;
    }
    if (on && l == 0) {
        const int c = 1 + nt;
        nnb[a] = c;
        if (pl.cnt_dst) pl.cnt_dst[a] = c;  // sizes this particle's row in the next stage
    }
    const unsigned c2 = __reduce_add_sync(kFull, on && l == 0 ? 1u + (unsigned)nt : 0u);
    // added to the event's counter by the pass that follows, unless a list overflowed
    if (lane == 0) atomicAdd(&v.sc->pairs_stage, (unsigned long long)c2);
}

// Gradient pass, half a warp per particle a, over the entries of its row with G = grad_a W_ab h /
// sigma_d, forming in integers the sums of the per-particle pass: sum grad W, sum X_b grad W, sum u_b grad W, each in
// the unit of its own largest term (a first look over the exponents).
// Bound: issue, then the latency of the gathers; 40 k event 161 us a stage (298 us with 10 FP64
// operations per pair; 137 with one unit for the stresses and one for u, from the values alone).  Two
// entries at a time; 5 blocks per SM: 4 took 5 % longer, 3 28 %.
__global__ void __launch_bounds__(32 * kWarps, 5) k_pairs_gradient(EvView v, int stage, const double *__restrict__ gin,
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
    auto at = [&](int j) { return j < nf ? r0 + j : r1 - nt + j; };  // entry j of a's row
    // the largest exponents among the terms of each sum: g_x | g_y, H_x | H_y, d_x u^x | d_x u^y, d_y u^x |
    // d_y u^y (16-bit halves)
    uint4 em = make_uint4(0u, 0u, 0u, 0u);
    for (int j = l; j < nt; j += 16) {
        const long long i = at(j);
        const longlong2 e = reinterpret_cast<const longlong2 *>(pl.X + n + pl.L[i])[1];
        const double2 g = pl.G[i];
        const int ex = fx_kexp(g.x), ey = fx_kexp(g.y);
        const unsigned x2 = fx_pair(ex, ex), y2 = fx_pair(ey, ey);
        em.x = fx_max2(em.x, fx_pair(ex, ey));
        em.y = fx_max2(em.y, fx_max2(word_lo(e.x) + x2, word_hi(e.x) + y2));
        em.z = fx_max2(em.z, word_lo(e.y) + x2);
        em.w = fx_max2(em.w, word_lo(e.y) + y2);
    }
    em = make_uint4(fx_half_max2(em.x), fx_half_max2(em.y), fx_half_max2(em.z), fx_half_max2(em.w));
    const int Em[8] = {fx_lo(em.x), fx_hi(em.x), fx_lo(em.y), fx_hi(em.y), fx_lo(em.z), fx_hi(em.z), fx_lo(em.w), fx_hi(em.w)};
    int E[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) E[k] = fx_room(Em[k], nt);
    FxSum sG[2] = {{0, 0}, {0, 0}};
    FxSum sH[2] = {{0, 0}, {0, 0}};                  // sum X^{x.} g, sum X^{y.} g
    FxSum sU[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};  // d_x u^x, d_x u^y, d_y u^x, d_y u^y
    int it = 0;
    auto add = [&](double2 g, Limb4 x, Limb4 u) {
        const long long mx = fx_kmant(g.x), my = fx_kmant(g.y);
        const int ex = fx_kexp(g.x), ey = fx_kexp(g.y);
        const unsigned eX0 = word_lo(u.z), eX1 = word_hi(u.z), eU = word_lo(u.w);
        sG[0].x += fx_shift(mx, E[0] - ex + kGuard);
        sG[1].x += fx_shift(my, E[1] - ey + kGuard);
        auto term = [&](FxSum &s, long long m, int d, long long q) {
            int hi, lo;
            fx_split(m, d, hi, lo);
            fx_add(s, hi, lo, fx_pair_of(q));
        };
        term(sH[0], mx, E[2] - ex - fx_lo(eX0), x.x);  // X^{xx} g_x
        term(sH[0], my, E[2] - ey - fx_lo(eX1), x.z);  // X^{yx} g_y
        term(sH[1], mx, E[3] - ex - fx_hi(eX0), x.y);  // X^{xy} g_x
        term(sH[1], my, E[3] - ey - fx_hi(eX1), x.w);  // X^{yy} g_y
        term(sU[0], mx, E[4] - ex - fx_lo(eU), u.x);
        term(sU[1], mx, E[5] - ex - fx_hi(eU), u.y);
        term(sU[2], my, E[6] - ey - fx_lo(eU), u.x);
        term(sU[3], my, E[7] - ey - fx_hi(eU), u.y);
    };
    auto fold = [&]() {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            fx_fold(sG[k]);
            fx_fold(sH[k]);
            fx_fold(sU[k]);
            fx_fold(sU[2 + k]);
        }
    };
    // two entries at a time, their loads ahead of both; an entry past the end is a with gradient 0
    auto add2 = [&](int b0, double2 g0, int b1, double2 g1) {
        const Limb4 x0 = pl.X[b0], u0 = pl.X[n + b0], x1 = pl.X[b1], u1 = pl.X[n + b1];
        add(g0, x0, u0);
        add(g1, x1, u1);
        it += 2;
        if ((it & (kFoldEvery - 1)) == 0) fold();
    };
    const double2 zero = make_double2(0.0, 0.0);
    for (int j = l; j < nt; j += 32) {
        const bool two = j + 16 < nt;
        const long long i0 = at(j), i1 = at(j + 16);
        add2(pl.L[i0], pl.G[i0], two ? pl.L[i1] : a, two ? pl.G[i1] : zero);
    }
    fold();
    FxTotal t[8] = {fx_words(sG[0]), fx_words(sG[1]), fx_words(sH[0]), fx_words(sH[1]),
                    fx_words(sU[0]), fx_words(sU[1]), fx_words(sU[2]), fx_words(sU[3])};
    const FxTotal tt = fx_reduce8(t, lane);
    const int k = l >> 1;
    int Ek = E[0], Emk = Em[0];
#pragma unroll
    for (int i = 1; i < 8; ++i)
        if (k == i) Ek = E[i], Emk = Em[i];
    double tot = fx_value(tt, k < 2 ? fx_kunit(Ek) : fx_unit(Ek));
    if (Emk >= kNonFinite) tot = fx_nan();
    // totals of lanes 2 k of the half warp: k = 0, 1: sum grad W; 2, 3: sum X_b grad W; 4-7: sum u_b grad W
    const double Sx = __shfl_sync(kFull, tot, lane & 16), Sy = __shfl_sync(kFull, tot, (lane & 16) + 2);
    if (on && (l & 1) == 0 && k >= 2) {
        const double c = v.sigma_d * v.inv_h;
        if (k >= 4) {
            gout[(size_t)(k - 4) * n + a] = c * tot;  // d_x u^x, d_x u^y, d_y u^x, d_y u^y
        } else {
            // minus the stress divergence: X_a . sum grad W + sum X_b grad W, times sqrt(-g)
            const double tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
            const double sqrtg = v.milne ? tau : 1.0;
            const double X0 = gin[(size_t)(k - 2) * n + a], X1 = gin[(size_t)k * n + a];
            gout[(size_t)(k + 2) * n + a] = -sqrtg * c * (X0 * Sx + X1 * Sy + tot);
        }
    }
}

inline int nblk(int n, int t) { return (n + t - 1) / t; }

}  // namespace

void launch_pair_rows(const EvView &v, CellBufs cb, cudaStream_t st)
{
    const int nparts = (v.n + kScanTile - 1) / kScanTile;
    k_rows_part<<<nparts, kScanThreads, 0, st>>>(v.n, cb.perm, cb.pl);
    k_rows_top<<<1, 1024, 0, st>>>(v.n, nparts, cb.pl, v.sc);
    k_rows_apply<<<nparts, kScanThreads, 0, st>>>(v.n, cb.perm, cb.pl);
}

void launch_pairs_density(const EvView &v, const double *y, const double *Nq, CellBufs cb, double *dens, int *nnb,
                          cudaStream_t st)
{
    launch_pair_rows(v, cb, st);
    k_pairs_fwd<<<nblk(v.n, 2 * kWarps), 32 * kWarps, 0, st>>>(v, y, cb.fpos, Nq, cb.start, cb.cnt, cb.key, cb.perm,
                                                             cb.pl);
    launch_pairs_sum(v, cb, dens, nnb, st);
}

void launch_pairs_sum(const EvView &v, CellBufs cb, double *dens, int *nnb, cudaStream_t st)
{
    k_pairs_sum<<<nblk(v.n, 2 * kWarps), 32 * kWarps, 0, st>>>(v, cb.pl, dens, nnb);
}

void launch_pairs_gradient(const EvView &v, int stage, const double *y, const double *gin, CellBufs cb,
                           double *gout, cudaStream_t st)
{
    (void)y;
    k_pairs_gradient<<<nblk(v.n, 2 * kWarps), 32 * kWarps, 0, st>>>(v, stage, gin, cb.pl, gout);
}

}  // namespace sphg
