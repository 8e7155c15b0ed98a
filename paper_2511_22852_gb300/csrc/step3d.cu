// step3d.cu -- the SPH step in three spatial dimensions: 3+1D Milne (tau, x, y, eta_s)
// and 3+1D Cartesian (t, x, y, z).  Same rows as the 2+1D kernels (a1-a8):
//   cells      generalized Morton key of the cell (per-axis bit counts, spread tables)
//   density    27-cell kernel sums, one warp per particle, single-precision prefilter
//   eos        u^0 = sqrt(1 - g_ij u^i u^j), rest-frame densities, inversion, X^{ji}/sigma*^2
//   gradient   27-cell n = 0 velocity gradients and n = -1 stress divergence
//   eom        covariant minimal Israel-Stewart equations with explicit Christoffel
//              symbols (Milne: Gamma^tau_{eta eta} = tau, Gamma^eta_{tau eta} = 1/tau),
//              every rate affine in the three acceleration components
// Distances are Euclidean in (x, y, eta) with eta taken in fm (Sec. "Kernel function").
// State rows (nv = 13): x^1..3, u^1..3, S, Pi/sigma, pi^{ij}/sigma for (11, 12, 13, 22, 23);
// pi^{33} follows from tracelessness, pi^{0 mu} from transversality.
#include "eos_device.cuh"
#include "pairs_fixed.cuh"
#include <algorithm>

#include "sph_internal.cuh"

namespace sphg {

namespace {

constexpr int kWarps3 = 4;

// ---------------------------------------------------------------------------
// a1: cell coordinates, keys and bucket counts
__global__ void k_cells3(EvView v, const double *__restrict__ y, uint32_t *key, uint32_t *cnt)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned act = __ballot_sync(0xFFFFFFFFu, i < v.n);
    if (i >= v.n) return;
    int c[3];
    bool bad = false;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        c[d] = cell_coord(y[(size_t)d * v.n + i], dec_double(v.sc->xmin_enc[d]), v.inv_cell);
        const int lim = 1 << v.B3[d];
        if (c[d] < 0 || c[d] >= lim) {
            bad = true;
            c[d] = min(max(c[d], 0), lim - 1);
        }
    }
    if (bad) atomicOr(&v.sc->err_flags, ERR_CELL_OVERFLOW);
    uint32_t k = key3(v, c[0], c[1], c[2]);
    key[i] = k;
    warp_count(cnt, k, act);
}

// the 27-cell candidate walk of one warp: prefilter, compaction, then `pair` on full warps
template <class Pair>
__device__ __forceinline__ void walk27(const EvView &v, const uint32_t *__restrict__ start,
                                       const uint32_t *__restrict__ cnt, const float4 *__restrict__ fpos, int a,
                                       const double *xa, int *q, Pair &pair)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const float4 fa = fpos[a];
    int c[3], lim[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        c[d] = cell_coord(xa[d], dec_double(v.sc->xmin_enc[d]), v.inv_cell);
        lim[d] = 1 << v.B3[d];
    }
    int qn = 0;
    for (int oz = -1; oz <= 1; ++oz) {
        const int nz = c[2] + oz;
        if (nz < 0 || nz >= lim[2]) continue;
        for (int oy = -1; oy <= 1; ++oy) {
            const int ny = c[1] + oy;
            if (ny < 0 || ny >= lim[1]) continue;
            for (int ox = -1; ox <= 1; ++ox) {
                const int nx = c[0] + ox;
                if (nx < 0 || nx >= lim[0]) continue;
                const uint32_t k = key3(v, nx, ny, nz);
                const uint32_t b0 = start[k], b1 = b0 + cnt[k];
                for (uint32_t base = b0; base < b1; base += 32) {
                    const uint32_t b = base + lane;
                    bool cand = false, sure = false;
                    if (b < b1) {
                        const float4 fb = fpos[b];
                        const float dx = fa.x - fb.x, dy = fa.y - fb.y, dz = fa.z - fb.z;
                        const float r2f = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                        cand = r2f <= v.supp2_hi;
                        sure = r2f < v.supp2_lo;
                    }
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, cand);
                    // bit 31 set: the float test left the pair undecided (exact test needed)
                    if (cand) q[qn + __popc(m & lt)] = sure ? (int)b : (int)(b | 0x80000000u);
                    qn += __popc(m);
                    __syncwarp();
                    if (qn >= 32) {
                        pair(q[lane]);
                        qn -= 32;
                        __syncwarp();
                        if (lane < qn) q[lane] = q[32 + lane];
                        __syncwarp();
                    }
                }
            }
        }
    }
    if (lane < qn) pair(q[lane]);
}

__device__ __forceinline__ double warp_sum(double x)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    return x;
}

// ---------------------------------------------------------------------------
// a3: kernel sums (lab frame); u^0 and the rest-frame division happen in the EoS pass.  Kernel values
// in integers and the lanes' sums by halves as in the 2D pass: 11 FP64 operations per pair (25).
__global__ void __launch_bounds__(32 * kWarps3) k_density3(EvView v, const double *__restrict__ y,
                                                           const float4 *__restrict__ fpos,
                                                           const double *__restrict__ Nq,
                                                           const uint32_t *__restrict__ start,
                                                           const uint32_t *__restrict__ cnt, double *__restrict__ dens,
                                                           int *__restrict__ nnb, int fallback, int *__restrict__ cnt_dst)
{
    // fallback = 1: the pair-list passes ran first; this pass only runs if one of their lists
    // overflowed (and counts such stages)
    if (fallback) {
        if (!v.sc->pair_flag) {
            if (blockIdx.x == 0 && threadIdx.x == 0) v.sc->pairs += v.sc->pairs_stage;
            return;
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&v.sc->pair_ovf, 1u);
    }
    __shared__ int queue[kWarps3][64];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // grid-stride over particles (one warp each): launched at a few blocks per SM when it is
    // only the fallback of the pair-list passes
    for (int a = blockIdx.x * kWarps3 + wid; a < v.n; a += gridDim.x * kWarps3) {  // warp-uniform
        const size_t n = (size_t)v.n;
        const double *X = y, *Y = y + n, *Z = y + 2 * n, *S = y + 6 * n;
        const double xa[3] = {X[a], Y[a], Z[a]};
        double sg = 0.0, ss = 0.0, sb = 0.0, sS = 0.0, sq = 0.0;
        int c = 0;
        auto pair = [&](int qb) {
            const int b = qb & 0x7FFFFFFF;
            const double dx = xa[0] - X[b], dy = xa[1] - Y[b], dz = xa[2] - Z[b];
            if (qb < 0 && !(dist2_3d(dx, dy, dz) < v.supp2)) return;
            {
                const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                double w, g[3];
                pair_kernel<3>({dx, dy, dz}, r2, v.inv_h, w, g);
                sg += w;
                ss = fma(S[b], w, ss);
                sb = fma(Nq[b], w, sb);
                sS = fma(Nq[n + b], w, sS);
                sq = fma(Nq[2 * n + b], w, sq);
                ++c;
            }
        };
        walk27(v, start, cnt, fpos, a, xa, queue[wid], pair);
        double t[8] = {sg, ss, sb, sS, sq, 0.0, 0.0, 0.0};
        const double tot = warp_sums8(t, lane);
        c = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)c);
        if ((lane & 3) == 0 && lane < 20) dens[(size_t)(lane >> 2) * n + a] = v.sigma_d * tot;
        if (lane == 0) {
            nnb[a] = c;
            if (cnt_dst) cnt_dst[a] = c;  // sizes the pair-list rows of the next stage
            atomicAdd(&v.sc->pairs, (unsigned long long)c);
        }
    }
}

// ---------------------------------------------------------------------------
// geometry of the stage: metric diag(1, -1, -1, g3), g3 = -tau^2 (Milne) or -1
struct Geo3 {
    double tau, g[4], gi[4], dg3, sqrtg;
    bool milne;
};
__device__ __forceinline__ Geo3 geo3(const EvView &v, int stage)
{
    Geo3 G;
    G.milne = v.milne != 0;
    G.tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
    G.g[0] = 1.0;
    G.g[1] = G.g[2] = -1.0;
    G.g[3] = G.milne ? -G.tau * G.tau : -1.0;
    for (int m = 0; m < 4; ++m) G.gi[m] = 1.0 / G.g[m];
    G.dg3 = G.milne ? -2.0 * G.tau : 0.0;
    G.sqrtg = G.milne ? G.tau : 1.0;
    return G;
}
// Christoffel symbols Gamma^a_{bc} of the Milne metric (zero in Cartesian coordinates)
__device__ __forceinline__ double gam(const Geo3 &G, int a, int b, int c)
{
    if (!G.milne) return 0.0;
    if (a == 0 && b == 3 && c == 3) return G.tau;
    if (a == 3 && ((b == 0 && c == 3) || (b == 3 && c == 0))) return 1.0 / G.tau;
    return 0.0;
}

// full contravariant pi^{mu nu} from the stored (11, 12, 13, 22, 23) components:
// pi^{33} from g_{mu nu} pi^{mu nu} = 0, pi^{0 nu} from u_mu pi^{mu nu} = 0; v_i = u_i / u_0 with
// u_1 = -u^1, u_2 = -u^2, u_3 = g_33 u^3 and iu0 = 1 / u^0
__device__ __forceinline__ void pi_full3(const Geo3 &G, const double *u, double iu0, const double *st, double pi[4][4])
{
    const double v1 = -u[1] * iu0, v2 = -u[2] * iu0, g3 = G.g[3], v3 = g3 * u[3] * iu0;
    pi[1][1] = st[0];
    pi[1][2] = pi[2][1] = st[1];
    pi[1][3] = pi[3][1] = st[2];
    pi[2][2] = st[3];
    pi[2][3] = pi[3][2] = st[4];
    const double known = v1 * v1 * st[0] + v2 * v2 * st[3] - (st[0] + st[3]) +
                         2.0 * (v1 * v2 * st[1] + v3 * (v1 * st[2] + v2 * st[4]));
    pi[3][3] = -known / (v3 * v3 + g3);
#pragma unroll
    for (int i = 1; i < 4; ++i) pi[0][i] = pi[i][0] = -(v1 * pi[1][i] + v2 * pi[2][i] + v3 * pi[3][i]);
    pi[0][0] = -(v1 * pi[1][0] + v2 * pi[2][0] + v3 * pi[3][0]);
}

// a4, first half: u^0, rest-frame densities, the search for (T, mu) (eos_device.cuh)
constexpr int kEosWarps3 = 4, kEosBlocks3 = 3;

struct Find3Ctx {
    const EvView &v;
    size_t n;
    double g3, sqrtg;
    const double *__restrict__ y;
    double *__restrict__ dens, *__restrict__ guess_out;
    uint32_t *__restrict__ status;
    const double *__restrict__ guess_in;
    __device__ bool load(int a, double &s, double nq[3], double g[4])
    {
        const double u1 = y[3 * n + a], u2 = y[4 * n + a], u3 = y[5 * n + a];
        const double u0 = sqrt(1.0 + (u1 * u1 + u2 * u2 - g3 * u3 * u3));
        const double ivol = 1.0 / (u0 * sqrtg);
        s = dens[n + a] * ivol;
        dens[n + a] = s;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            nq[q] = dens[(2 + q) * n + a] * ivol;
            dens[(2 + q) * n + a] = nq[q];
        }
        dens[5 * n + a] = u0;
#pragma unroll
        for (int k = 0; k < 4; ++k) g[k] = guess_in[k * n + a];
        return true;
    }
    __device__ void put(int a, const double x[4], uint32_t st)
    {
#pragma unroll
        for (int k = 0; k < 4; ++k) guess_out[k * n + a] = x[k];
        status[a] = st;
    }
    __device__ void keep(int a, const double g[4])
    {
#pragma unroll
        for (int k = 0; k < 4; ++k) guess_out[k * n + a] = g[k];
    }
    __device__ void mark(int a, uint32_t st) { status[a] = st; }
};

__global__ void __launch_bounds__(32 * kEosWarps3, kEosBlocks3)
    k_eos3_find(EvView v, int stage, const double *__restrict__ y, double *__restrict__ dens,
                uint32_t *__restrict__ status, const double *__restrict__ guess_in, double *__restrict__ guess_out)
{
    const Geo3 G = geo3(v, stage);
    Find3Ctx ctx{v, (size_t)v.n, G.g[3], G.sqrtg, y, dens, guess_out, status, guess_in};
    EosWork w = {0u, 0u, 0u};
    eos_find(v.eos, &v.sc->eos_claim, v.n, ctx, w);
    add_eos_work(v.sc, w, 0u);
}

// a4, second half: the EoS there, stress inputs of the gradient pass, work rate
__global__ void __launch_bounds__(64, 5) k_eos3_finish(EvView v, int stage, const double *__restrict__ y,
                                                    const double *__restrict__ dens, double *__restrict__ eos,
                                                    double *__restrict__ gin, uint32_t *__restrict__ status,
                                                    double *__restrict__ wpart, double *__restrict__ guess_out)
{
    __shared__ double red[2];
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    const size_t n = (size_t)v.n;
    double wcontrib = 0.0;
    EosWork w = {0u, 0u, 0u};
    unsigned st_or = 0u;
    if (a < v.n) {
        const Geo3 G = geo3(v, stage);
        const double u[4] = {dens[5 * n + a], y[3 * n + a], y[4 * n + a], y[5 * n + a]};
        const double isig = 1.0 / dens[a], iu0 = 1.0 / u[0];
        const double s = dens[n + a], nq[3] = {dens[2 * n + a], dens[3 * n + a], dens[4 * n + a]};
        const double g[4] = {guess_out[a], guess_out[n + a], guess_out[2 * n + a], guess_out[3 * n + a]};
        bool used = false;
        const EosOut o = eos_finish(v.eos, v.tr.cs2_cap, s, nq, g, status[a], used, w);
        guess_out[a] = used ? o.T : ((o.st & (PST_NOCONV | PST_NONFINITE | PST_BACKUP)) ? 0.0 : -o.T);
        for (int q = 0; q < 3; ++q) guess_out[(size_t)(1 + q) * n + a] = used ? o.mu[q] : 0.0;
        status[a] = o.st;
        st_or = o.st;
        eos[a] = o.T;
        for (int q = 0; q < 3; ++q) eos[(1 + q) * n + a] = o.mu[q];
        eos[4 * n + a] = o.p;
        eos[5 * n + a] = o.e;
        eos[6 * n + a] = o.ps;
        for (int q = 0; q < 3; ++q) eos[(7 + q) * n + a] = o.pn[q];
        eos[10 * n + a] = o.cs2;
        const double isg = G.milne ? 1.0 / G.sqrtg : 1.0;
        const double sigma = dens[a] * iu0 * isg;
        double Pi = 0.0, st[5] = {0, 0, 0, 0, 0};
        if (v.tr.viscous) {
            Pi = sigma * y[7 * n + a];
#pragma unroll
            for (int k = 0; k < 5; ++k) st[k] = sigma * y[(8 + k) * n + a];
        }
        double pi[4][4];
        pi_full3(G, u, iu0, st, pi);
        const double inv2 = isig * isig;
        const double P = o.p + Pi;
        double vv[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) vv[j] = u[1 + j] * iu0;
        double X[9], us[3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                double t = pi[1 + j][1 + i] - vv[j] * pi[0][1 + i];
                if (j == i) t += j < 2 ? P : P * (G.milne ? isg * isg : 1.0);  // -P g^{jj}
                X[3 * j + i] = t * inv2;
                gin[(size_t)(3 * j + i) * n + a] = X[3 * j + i];
            }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            us[j] = u[1 + j] * isig;
            gin[(size_t)(9 + j) * n + a] = us[j];
        }
        if (v.fX) {  // in single precision for the mixed form's
            v.fX[a] = make_float4((float)X[0], (float)X[1], (float)X[2], (float)X[3]);
            v.fX[n + a] = make_float4((float)X[4], (float)X[5], (float)X[6], (float)X[7]);
            v.fX[2 * n + a] = make_float4((float)X[8], (float)us[0], (float)us[1], (float)us[2]);
        }
        if (v.fxX) {  // the same in limbs for the pair-list gradient pass
            int e[12];
            long long w[12];
#pragma unroll
            for (int m = 0; m < 12; ++m) {
                const double x = m < 9 ? X[m] : us[m - 9];
                e[m] = fx_exponent(x);
                w[m] = fx_word(fx_limbs(x, e[m]));
            }
#pragma unroll
            for (int m = 0; m < 3; ++m) v.fxX[m * n + a] = Limb4{w[4 * m], w[4 * m + 1], w[4 * m + 2], w[4 * m + 3]};
            v.fxX[3 * n + a] = Limb4{fx_word(fx_pair(e[0], e[1]), fx_pair(e[2], e[9])), fx_word(fx_pair(e[3], e[4]), fx_pair(e[5], e[10])),
                                     fx_word(fx_pair(e[6], e[7]), fx_pair(e[8], e[11])), 0};
        }
        if (G.milne) {
            // sqrt(-g) Gamma^0_{33} T^{33} / sigma* = tau^2 T^{eta eta} / sigma*
            wcontrib = (G.tau * G.tau * ((o.e + P) * u[3] * u[3] + pi[3][3]) + P) * isig;
        }
    }
    add_eos_work(v.sc, w, st_or);
    wcontrib = warp_sum(wcontrib);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = wcontrib;
    __syncthreads();
    if (threadIdx.x == 0) wpart[blockIdx.x] = red[0] + red[1];
}

// ---------------------------------------------------------------------------
// a5: gradients.  gin rows: X^{ji}/sigma*^2 at 3 j + i, u^j/sigma* at 9 + j.
// gout rows: d_k u^j at 3 k + j, then F^i at 9 + i.
__global__ void __launch_bounds__(32 * kWarps3) k_gradient3(EvView v, int stage, const double *__restrict__ y,
                                                            const float4 *__restrict__ fpos,
                                                            const double *__restrict__ gin,
                                                            const uint32_t *__restrict__ start,
                                                            const uint32_t *__restrict__ cnt,
                                                            double *__restrict__ gout, int fallback)
{
    if (fallback && !v.sc->pair_flag) return;  // the pair-list pass did the work
    __shared__ int queue[kWarps3][64];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // grid-stride over particles (one warp each): launched at a few blocks per SM when it is
    // only the fallback of the pair-list passes
    for (int a = blockIdx.x * kWarps3 + wid; a < v.n; a += gridDim.x * kWarps3) {  // warp-uniform
        const size_t n = (size_t)v.n;
        const double *X = y, *Y = y + n, *Z = y + 2 * n;
        const double xa[3] = {X[a], Y[a], Z[a]};
        double G[3] = {0, 0, 0}, H[3] = {0, 0, 0}, du[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
        auto pair = [&](int qb) {
            const int b = qb & 0x7FFFFFFF;
            const double d[3] = {xa[0] - X[b], xa[1] - Y[b], xa[2] - Z[b]};
            if (qb < 0 && !(dist2_3d(d[0], d[1], d[2]) < v.supp2)) return;
            const double r2 = fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2]));
            if (r2 > 0.0) {
                const double ir = inv_sqrt(r2);
                const double fac = kernel_dw(r2 * ir * v.inv_h) * ir;
                double gw[3];
    #pragma unroll
                for (int k = 0; k < 3; ++k) {
                    gw[k] = fac * d[k];
                    G[k] += gw[k];
                }
    #pragma unroll
                for (int i = 0; i < 3; ++i) {
                    double h = H[i];
    #pragma unroll
                    for (int j = 0; j < 3; ++j) h = fma(gin[(size_t)(3 * j + i) * n + b], gw[j], h);
                    H[i] = h;
                }
    #pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const double ub = gin[(size_t)(9 + j) * n + b];
    #pragma unroll
                    for (int k = 0; k < 3; ++k) du[k][j] = fma(ub, gw[k], du[k][j]);
                }
            }
        };
        walk27(v, start, cnt, fpos, a, xa, queue[wid], pair);
    #pragma unroll
        for (int k = 0; k < 3; ++k) {
            G[k] = warp_sum(G[k]);
            H[k] = warp_sum(H[k]);
    #pragma unroll
            for (int j = 0; j < 3; ++j) du[k][j] = warp_sum(du[k][j]);
        }
        if (lane == 0) {
            const double tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
            const double sqrtg = v.milne ? tau : 1.0;
            const double c = v.sigma_d * v.inv_h;
    #pragma unroll
            for (int k = 0; k < 3; ++k)
    #pragma unroll
                for (int j = 0; j < 3; ++j) gout[(size_t)(3 * k + j) * n + a] = c * du[k][j];
    #pragma unroll
            for (int i = 0; i < 3; ++i) {
                double F = H[i];
    #pragma unroll
                for (int j = 0; j < 3; ++j) F = fma(gin[(size_t)(3 * j + i) * n + a], G[j], F);
                gout[(size_t)(9 + i) * n + a] = -sqrtg * c * F;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// a6/a7: equations of motion, minimal Israel-Stewart (the general form with DNMR is k_eom3).
//
// In the orthonormal frame along the coordinate axes (third components times tau in Milne
// coordinates: u^3 = tau u^eta, P^{13} = tau P^{x eta}, d_3 = d_eta / tau; h = 1/tau, 0 in
// Cartesian) the metric is Minkowski and the only connection terms are nabla_3 u^3 += h u^0,
// nabla_3 u^0 += h u^3.  With the unknowns A_i = du^i/dx^0 + delta_{i3} h u^3, Du^i = u^0 A_i and
// Du^0 = u^0 v.A, every rate is {c, x, y, z} = c + x A_1 + y A_2 + z A_3:
//   theta = th0 + v.A,
//   sigma^{ij} = -(N_ij + N_ji)/2 - u^0 (u^i A_j + u^j A_i)/2 + (delta_ij + u^i u^j) theta/3,
//   dS, dB, D and dP^{ij} as in the 2+1D form (dP^{ij} with the connection term
//     -h v^3 (delta_i3 P^{0j} + delta_j3 P^{0i})),
//   dP_lab^i = u^i D + (w/sigma) du^i + d(P^{0i}/u^0) = F^i - delta_i3 h P_lab^3.
// Bound: the FP64 pipe; about 470 FP64 operations a particle instead of 1,900 for the generic
// four-tensors (258 k particles: 828 -> 300 us a stage).
struct R4 {
    double c, x, y, z;
};
__device__ __forceinline__ double at4(const R4 &r, double a0, double a1, double a2)
{
    return fma(r.x, a0, fma(r.y, a1, fma(r.z, a2, r.c)));
}

__global__ void __launch_bounds__(64) k_eom3_min_is(EvView v, int stage, int mode, const double *__restrict__ ys,
                                                    const double *__restrict__ dens, const double *__restrict__ eos,
                                                    const double *__restrict__ gout, double *__restrict__ yout,
                                                    double *__restrict__ rates, uint32_t *__restrict__ status)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= v.n) return;
    const size_t n = (size_t)v.n;
    const bool milne = v.milne != 0;
    const double tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
    const double sqrtg = milne ? tau : 1.0, isqg = milne ? 1.0 / tau : 1.0, h = milne ? isqg : 0.0;
    const double g = dens[5 * n + a], T = eos[a], ig = 1.0 / g;
    const double u[3] = {ys[3 * n + a], ys[4 * n + a], ys[5 * n + a] * sqrtg};
    const double vv[3] = {u[0] * ig, u[1] * ig, u[2] * ig};
    const uint32_t st_in = status[a];
    double f[13];
    f[0] = vv[0];
    f[1] = vv[1];
    f[2] = vv[2] * isqg;
    double dN[3] = {0.0, 0.0, 0.0};  // charge rates dN_q/dx0 (charge sources only)
    uint32_t st = 0;
    if ((st_in & (PST_NOCONV | PST_NONFINITE)) || (v.tr.T_stop_GeV > 0.0 && T * kHbarc < v.tr.T_stop_GeV)) {
        // no EoS solution, or below the stop temperature: ballistic motion only, charges unchanged
#pragma unroll
        for (int k = 3; k < 13; ++k) f[k] = 0.0;
    } else {
        const double sig_star = dens[a], s = dens[n + a];
        const double p = eos[4 * n + a], e = eos[5 * n + a], ps = eos[6 * n + a];
        const double m0 = eos[n + a] + eos[7 * n + a], m1 = eos[2 * n + a] + eos[8 * n + a], m2 = eos[3 * n + a] + eos[9 * n + a];
        const double Q = m0 * dens[2 * n + a] + m1 * dens[3 * n + a] + m2 * dens[4 * n + a];
        const double isig = 1.0 / sig_star, sigma = sig_star * ig * isqg, isg = g * sqrtg * isig;
        const double ep = e + p, iT = 1.0 / T, third = 1.0 / 3.0;
        // N[k][j] = nabla_k u^j in the frame
        double N[3][3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                double d = gout[(size_t)(3 * k + j) * n + a];
                if (milne && k == 2 && j < 2) d *= isqg;
                if (milne && k < 2 && j == 2) d *= sqrtg;
                N[k][j] = d;
            }
        // d_k u^0 = v.d_k u before the connection is added
        double t0 = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) t0 = fma(vv[k], vv[0] * N[k][0] + vv[1] * N[k][1] + vv[2] * N[k][2], t0);
        N[2][2] = fma(h, g, N[2][2]);
        const double hu3 = h * u[2];
        const R4 th = {N[0][0] + N[1][1] + N[2][2] - t0 - vv[2] * hu3, vv[0], vv[1], vv[2]};
        double w = ep;
        R4 dS = {0.0, 0.0, 0.0, 0.0}, dB = dS, dP[3][3];
        double P[3][3], P0[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                P[i][j] = 0.0;
                dP[i][j] = R4{0.0, 0.0, 0.0, 0.0};
            }
        if (v.tr.viscous) {
            const double B = ys[7 * n + a], Pi = sigma * B;
            w += Pi;
            P[0][0] = ys[8 * n + a];
            P[0][1] = P[1][0] = ys[9 * n + a];
            P[0][2] = P[2][0] = ys[10 * n + a] * sqrtg;
            P[1][1] = ys[11 * n + a];
            P[1][2] = P[2][1] = ys[12 * n + a] * sqrtg;
            // P^{33} from tracelessness with P^{00} = v_i v_j P^{ij}
            const double known = fma(vv[0] * vv[0], P[0][0], vv[1] * vv[1] * P[1][1]) - P[0][0] - P[1][1] +
                                 2.0 * (vv[0] * vv[1] * P[0][1] + vv[2] * (vv[0] * P[0][2] + vv[1] * P[1][2]));
            P[2][2] = known / fma(-vv[2], vv[2], 1.0);
#pragma unroll
            for (int j = 0; j < 3; ++j) P0[j] = vv[0] * P[0][j] + vv[1] * P[1][j] + vv[2] * P[2][j];
            const double P00 = vv[0] * P0[0] + vv[1] * P0[1] + vv[2] * P0[2];
            const double eta = v.tr.eta_over_s * s;
            const double dTg = T * kHbarc - v.tr.zeta_T_GeV;
            const double zeta = v.tr.zeta_peak * exp(-dTg * dTg / (2.0 * v.tr.zeta_w_GeV * v.tr.zeta_w_GeV)) * s;
            const double itp = ep / (v.tr.tau_pi_coef * eta);  // 1/tau_pi; tau_Pi = ratio tau_pi
            const double q2 = ig * itp, q1 = 2.0 * eta * q2 * isg, q3 = third * ig;
            const R4 ev = {fma(q3, th.c, q2), q3 * vv[0], q3 * vv[1], q3 * vv[2]};
            double C[3][3];  // C^j = P^{0j} v.A - P^{jk} A_k
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k) C[j][k] = fma(P0[j], vv[k], -P[j][k]);
            R4 ps4 = {-B * th.c, -B * vv[0], -B * vv[1], -B * vv[2]};  // P:sigma - B theta
            const double hv3 = h * vv[2];
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = i; j < 3; ++j) {
                    const double cij = i == j ? fma(third * u[i], u[i], third) : third * u[i] * u[j];
                    R4 sg = {fma(cij, th.c, i == j ? -N[i][i] : -0.5 * (N[i][j] + N[j][i])), cij * vv[0], cij * vv[1], cij * vv[2]};
                    double *sk = &sg.x;
                    if (i == j) {
                        sk[i] -= g * u[i];
                    } else {
                        sk[j] = fma(-0.5 * g, u[i], sk[j]);
                        sk[i] = fma(-0.5 * g, u[j], sk[i]);
                    }
                    // P:sigma with the 0-components of both tensors written by their spatial ones
                    double M = P[i][j] - vv[i] * P0[j] - vv[j] * P0[i] + vv[i] * vv[j] * P00;
                    if (i != j) M *= 2.0;
                    ps4.c = fma(M, sg.c, ps4.c);
                    ps4.x = fma(M, sg.x, ps4.x);
                    ps4.y = fma(M, sg.y, ps4.y);
                    ps4.z = fma(M, sg.z, ps4.z);
                    R4 x = {q1 * sg.c - P[i][j] * ev.c, q1 * sg.x - P[i][j] * ev.x, q1 * sg.y - P[i][j] * ev.y,
                            q1 * sg.z - P[i][j] * ev.z};
                    if (i == j) {
                        const double t = -2.0 * u[i];
                        x.x = fma(t, C[i][0], x.x);
                        x.y = fma(t, C[i][1], x.y);
                        x.z = fma(t, C[i][2], x.z);
                    } else {
                        x.x -= u[i] * C[j][0] + u[j] * C[i][0];
                        x.y -= u[i] * C[j][1] + u[j] * C[i][1];
                        x.z -= u[i] * C[j][2] + u[j] * C[i][2];
                    }
                    if (j == 2) x.c = fma(i == 2 ? -2.0 * hv3 : -hv3, P0[i], x.c);
                    dP[i][j] = x;
                    dP[j][i] = x;
                }
            const double kS = ig * iT;
            dS = R4{kS * ps4.c, kS * ps4.x, kS * ps4.y, kS * ps4.z};
            const double kB = -(ig * isg) * (itp / v.tr.tau_Pi_ratio), kz = kB * zeta;
            dB = R4{fma(kz, th.c, kB * Pi), kz * vv[0], kz * vv[1], kz * vv[2]};
        }
        double Isrc[3] = {0.0, 0.0, 0.0}, Dsrc = 0.0;
        if (v.ntrack > 0 || v.nparton > 0) {
            // jet tracks (Cartesian) and partons: dP^i/dx0 gains sqrt(-g) I^i/sigma*, dS/dx0 gains
            // u_nu I^nu/(u^0 sigma T); parton charges: dN_q/dx0 = sqrt(-g) I_q/sigma*, and dS/dx0
            // gains -mu_q/T dN_q/dx0 (eq. dsdnrewr, R^S_q = -mu_q/T)
            double Is[4] = {0.0, 0.0, 0.0, 0.0}, Ik[4], Iq[3] = {0.0, 0.0, 0.0};
            if (v.ntrack > 0) {
                jet_deposit(v, tau, ys[a], ys[n + a], ys[2 * n + a], Ik);
                for (int k = 0; k < 4; ++k) Is[k] += Ik[k];
            }
            if (v.nparton > 0) {
                const double xa[3] = {ys[a], ys[n + a], ys[2 * n + a]};
                parton_deposit(v, tau, sqrtg, xa, Ik, Iq);
                for (int k = 0; k < 4; ++k) Is[k] += Ik[k];
            }
            Is[3] *= sqrtg;  // to the frame
            const double uI = g * Is[0] - u[0] * Is[1] - u[1] * Is[2] - u[2] * Is[3] -
                              (eos[n + a] * Iq[0] + eos[2 * n + a] * Iq[1] + eos[3 * n + a] * Iq[2]);
            dS.c += (ig * isg * iT) * uI;
            for (int c = 0; c < 3; ++c) {
                dN[c] = sqrtg * Iq[c] * isig;
                Isrc[c] = sqrtg * Is[1 + c] * isig;
            }
            Dsrc = m0 * dN[0] + m1 * dN[1] + m2 * dN[2];
        }
        const double Tps = T + ps, k3 = (isg * ig) * (ep - Tps * s - Q);
        const R4 D = {fma(Tps, dS.c, fma(k3, th.c, dB.c + Dsrc)), fma(Tps, dS.x, fma(k3, vv[0], dB.x)),
                      fma(Tps, dS.y, fma(k3, vv[1], dB.y)), fma(Tps, dS.z, fma(k3, vv[2], dB.z))};
        const double W = w * isg, ig2 = ig * ig;
        // M A = b: the lab momentum's rate, du^k = A_k - delta_k3 h u^3
        double A[3][3], b[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double hp = 2.0 * ig2 * P0[i];
            double cc = u[0] * dP[0][i].c + u[1] * dP[1][i].c + u[2] * dP[2][i].c - hu3 * P[2][i];
            double c = fma(u[i], D.c, fma(ig2, cc, hp * vv[2] * hu3));
            A[i][0] = fma(u[i], D.x, ig2 * (P[0][i] + u[0] * dP[0][i].x + u[1] * dP[1][i].x + u[2] * dP[2][i].x)) - hp * vv[0];
            A[i][1] = fma(u[i], D.y, ig2 * (P[1][i] + u[0] * dP[0][i].y + u[1] * dP[1][i].y + u[2] * dP[2][i].y)) - hp * vv[1];
            A[i][2] = fma(u[i], D.z, ig2 * (P[2][i] + u[0] * dP[0][i].z + u[1] * dP[1][i].z + u[2] * dP[2][i].z)) - hp * vv[2];
            A[i][i] += W;
            double F = gout[(size_t)(9 + i) * n + a];
            if (i == 2) {
                c -= W * hu3;
                F = F * sqrtg - h * fma(W, u[2], P0[2] * ig);
            }
            b[i] = F + Isrc[i] - c;
        }
        bool ok = true;
        double ipv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {  // partial pivoting on integer magnitudes
            int piv = c;
            long long best = mag_bits(A[c][c]);
#pragma unroll
            for (int r = c + 1; r < 3; ++r)
                if (mag_bits(A[r][c]) > best) {
                    best = mag_bits(A[r][c]);
                    piv = r;
                }
            if (best == 0 || best >= kInfBits) {
                ok = false;
                break;
            }
#pragma unroll
            for (int r = c + 1; r < 3; ++r)
                if (piv == r) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const double t = A[c][k];
                        A[c][k] = A[r][k];
                        A[r][k] = t;
                    }
                    const double t = b[c];
                    b[c] = b[r];
                    b[r] = t;
                }
            ipv[c] = 1.0 / A[c][c];
#pragma unroll
            for (int r = c + 1; r < 3; ++r) {
                const double q = A[r][c] * ipv[c];
#pragma unroll
                for (int k = c + 1; k < 3; ++k) A[r][k] = fma(-q, A[c][k], A[r][k]);
                b[r] = fma(-q, b[c], b[r]);
            }
        }
        // without a solution the acceleration du^i/dx^0 of the state's variables is zero
        double Av[3] = {0.0, 0.0, milne ? 2.0 * hu3 : 0.0};
        if (ok) {
            Av[2] = b[2] * ipv[2];
            Av[1] = fma(-A[1][2], Av[2], b[1]) * ipv[1];
            Av[0] = fma(-A[0][2], Av[2], fma(-A[0][1], Av[1], b[0])) * ipv[0];
        } else {
            st |= PST_SOLVE_FAIL;
        }
        f[3] = Av[0];
        f[4] = Av[1];
        f[5] = (Av[2] - 2.0 * hu3) * isqg;  // du^eta/dtau = (du^3/dtau - u^3/tau)/tau
        f[6] = at4(dS, Av[0], Av[1], Av[2]);
        f[7] = at4(dB, Av[0], Av[1], Av[2]);
        f[8] = at4(dP[0][0], Av[0], Av[1], Av[2]);
        f[9] = at4(dP[0][1], Av[0], Av[1], Av[2]);
        f[10] = (at4(dP[0][2], Av[0], Av[1], Av[2]) - h * P[0][2]) * isqg;
        f[11] = at4(dP[1][1], Av[0], Av[1], Av[2]);
        f[12] = (at4(dP[1][2], Av[0], Av[1], Av[2]) - h * P[1][2]) * isqg;
        bool fin = true;
#pragma unroll
        for (int k = 0; k < 13; ++k) fin = fin && isfinite(f[k]);
        if (!fin) st |= PST_NONFINITE;
        if (st) {
            status[a] = st_in | st;
            atomicOr(&v.sc->status_or, st);
        }
    }
    const double dt = v.dtau;
    if (mode == 0) {
#pragma unroll
        for (int k = 0; k < 13; ++k) yout[k * n + a] = ys[k * n + a] + dt * f[k];
    } else if (mode == 1) {
#pragma unroll
        for (int k = 0; k < 13; ++k) yout[k * n + a] = 0.5 * ((yout[k * n + a] + ys[k * n + a]) + dt * f[k]);
    } else {
#pragma unroll
        for (int k = 0; k < 13; ++k) rates[k * n + a] = f[k];
    }
    heun_charges(v, mode, n, a, dN);
}

// ---------------------------------------------------------------------------
// The general form (DNMR).  A3 = c + x a^1 + y a^2 + z a^3, affine in the acceleration.
struct A3 {
    double c, x, y, z;
};
__device__ __forceinline__ A3 k3(double c) { return {c, 0.0, 0.0, 0.0}; }
__device__ __forceinline__ A3 operator+(A3 a, A3 b) { return {a.c + b.c, a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ A3 operator-(A3 a, A3 b) { return {a.c - b.c, a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ A3 operator*(double s, A3 a) { return {s * a.c, s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ A3 operator+(A3 a, double s) { return {a.c + s, a.x, a.y, a.z}; }
__device__ __forceinline__ double at3(A3 a, const double *acc) { return fma(a.x, acc[0], fma(a.y, acc[1], fma(a.z, acc[2], a.c))); }

// the DNMR form (k_eom3_min_is is the minimal one)
__global__ void __launch_bounds__(64) k_eom3(EvView v, int stage, int mode, const double *__restrict__ ys,
                                             const double *__restrict__ dens, const double *__restrict__ eos,
                                             const double *__restrict__ gout, double *__restrict__ yout,
                                             double *__restrict__ rates, uint32_t *__restrict__ status)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= v.n) return;
    const size_t n = (size_t)v.n;
    const Geo3 G = geo3(v, stage);
    double u[4] = {dens[5 * n + a], ys[3 * n + a], ys[4 * n + a], ys[5 * n + a]};
    const double sig_star = dens[a], s = dens[n + a];
    const double nq[3] = {dens[2 * n + a], dens[3 * n + a], dens[4 * n + a]};
    const double T = eos[a], p = eos[4 * n + a], e = eos[5 * n + a], ps = eos[6 * n + a];
    const double mu[3] = {eos[n + a], eos[2 * n + a], eos[3 * n + a]};
    const double pn[3] = {eos[7 * n + a], eos[8 * n + a], eos[9 * n + a]};
    const double sigma = sig_star / (u[0] * G.sqrtg);
    const double ig = 1.0 / u[0], isg = 1.0 / sigma;
    const double vv[4] = {1.0, u[1] * ig, u[2] * ig, u[3] * ig};
    const bool visc = v.tr.viscous != 0;
    const double dt = v.dtau;
    const int nv = v.nv;
    if ((status[a] & (PST_NOCONV | PST_NONFINITE)) || (v.tr.T_stop_GeV > 0.0 && eos[a] * kHbarc < v.tr.T_stop_GeV)) {
        // no EoS solution, or below the stop temperature: ballistic motion only
        for (int k = 0; k < nv; ++k) {
            double fk = k < 3 ? vv[1 + k] : 0.0;
            if (mode == 0) yout[k * n + a] = ys[k * n + a] + dt * fk;
            else if (mode == 1) yout[k * n + a] = 0.5 * ((yout[k * n + a] + ys[k * n + a]) + dt * fk);
            else rates[k * n + a] = fk;
        }
        const double dN0[3] = {0.0, 0.0, 0.0};  // frozen: the charges stay as they are
        heun_charges(v, mode, n, a, dN0);
        return;
    }
    double Bv = 0.0, stv[5] = {0, 0, 0, 0, 0};
    if (visc) {
        Bv = ys[7 * n + a];
        for (int k = 0; k < 5; ++k) stv[k] = ys[(8 + k) * n + a];
    }
    const double Pi = sigma * Bv;
    double st[5];
    for (int k = 0; k < 5; ++k) st[k] = sigma * stv[k];
    double pi[4][4];
    pi_full3(G, u, ig, st, pi);
    // d_k u^j (spatial k, j) and d_k u^0
    double dku[4][4];
    for (int k = 1; k < 4; ++k) {
        double s0 = 0.0;
        for (int j = 1; j < 4; ++j) {
            dku[k][j] = gout[(size_t)(3 * (k - 1) + (j - 1)) * n + a];
            s0 += G.g[j] * u[j] * dku[k][j];
        }
        dku[k][0] = -s0 * ig;
    }
    const A3 acc[4] = {k3(0.0), {0.0, 1.0, 0.0, 0.0}, {0.0, 0.0, 1.0, 0.0}, {0.0, 0.0, 0.0, 1.0}};
    // du^0/dx^0 from u.u = 1
    A3 du0 = (-ig) * (G.g[1] * u[1] * acc[1] + G.g[2] * u[2] * acc[2] + G.g[3] * u[3] * acc[3] + 0.5 * G.dg3 * u[3] * u[3]);
    A3 dudt[4] = {du0, acc[1], acc[2], acc[3]};
    // nabla_0 u^nu (affine) and nabla_k u^nu (constant)
    A3 nab0[4];
    double nabk[4][4];
    for (int nu = 0; nu < 4; ++nu) {
        double conv = 0.0, chr = 0.0;
        for (int k = 1; k < 4; ++k) conv += vv[k] * dku[k][nu];
        for (int l = 0; l < 4; ++l) chr += gam(G, nu, 0, l) * u[l];
        nab0[nu] = dudt[nu] + (chr - conv);
        for (int k = 1; k < 4; ++k) {
            double c2 = 0.0;
            for (int l = 0; l < 4; ++l) c2 += gam(G, nu, k, l) * u[l];
            nabk[k][nu] = dku[k][nu] + c2;
        }
    }
    A3 th = nab0[0] + (nabk[1][1] + nabk[2][2] + nabk[3][3]);
    A3 Du[4];
    for (int nu = 0; nu < 4; ++nu) Du[nu] = u[0] * nab0[nu] + (u[1] * nabk[1][nu] + u[2] * nabk[2][nu] + u[3] * nabk[3][nu]);
    const A3 dsg = (-sigma * ig) * th;
    A3 dS = k3(0.0), dBv = k3(0.0), dPv[4][4];
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) dPv[i][j] = k3(0.0);
    if (visc) {
        // spatial shear tensor; the 0-components from transversality
        A3 sg[4][4];
        for (int i = 1; i < 4; ++i)
            for (int j = i; j < 4; ++j) {
                double sym = 0.5 * (G.gi[i] * nabk[i][j] + G.gi[j] * nabk[j][i]);
                double Delta = (i == j ? G.gi[i] : 0.0) - u[i] * u[j];
                A3 x = k3(sym) - 0.5 * (u[i] * Du[j] + u[j] * Du[i]) - (Delta / 3.0) * th;
                sg[i][j] = x;
                sg[j][i] = x;
            }
        for (int j = 1; j < 4; ++j) {
            A3 acc0 = k3(0.0);
            for (int k = 1; k < 4; ++k) acc0 = acc0 + (G.g[k] * u[k]) * sg[k][j];
            sg[0][j] = (-ig) * acc0;
            sg[j][0] = sg[0][j];
        }
        {
            A3 acc0 = k3(0.0);
            for (int k = 1; k < 4; ++k) acc0 = acc0 + (G.g[k] * u[k]) * sg[k][0];
            sg[0][0] = (-ig) * acc0;
        }
        A3 pisig = k3(0.0);
        for (int m = 0; m < 4; ++m)
            for (int l = 0; l < 4; ++l) pisig = pisig + (pi[m][l] * G.g[m] * G.g[l]) * sg[m][l];
        const double eta = v.tr.eta_over_s * s;
        const double dTg = T * kHbarc - v.tr.zeta_T_GeV;
        const double zeta = v.tr.zeta_peak * exp(-dTg * dTg / (2.0 * v.tr.zeta_w_GeV * v.tr.zeta_w_GeV)) * s;
        const double taupi = v.tr.tau_pi_coef * eta / (e + p);
        const double tauPi = v.tr.tau_Pi_ratio * taupi;
        dS = (ig * isg / T) * (pisig - Pi * th);
        // bulk (see the 2+1D equations of motion)
        const double cs2 = eos[10 * n + a];
        dBv = (ig * isg) * ((-1.0 / tauPi) * (zeta * th + Pi) + ((1.0 - v.tr.dnmr[0]) * Pi) * th +
                            (v.tr.dnmr[1] * (1.0 / 3.0 - cs2)) * pisig);
        double trB = 0.0;  // pi:pi
        for (int m = 0; m < 4; ++m)
            for (int l = 0; l < 4; ++l) trB += pi[m][l] * G.g[m] * G.g[l] * pi[m][l];
        A3 alow[4];
        for (int al = 0; al < 4; ++al) alow[al] = G.g[al] * Du[al];
        const double itp = 1.0 / taupi;
        for (int i = 1; i < 4; ++i)
            for (int j = i; j < 4; ++j) {
                double chr = 0.0;
                for (int m = 0; m < 4; ++m)
                    for (int l = 0; l < 4; ++l) chr += u[m] * (gam(G, i, m, l) * pi[l][j] + gam(G, j, m, l) * pi[i][l]);
                A3 pja = k3(0.0), pia = k3(0.0);
                for (int al = 0; al < 4; ++al) {
                    pja = pja + pi[j][al] * alow[al];
                    pia = pia + pi[i][al] * alow[al];
                }
                // - delta_pipi pi theta - tau_pipi <pi sigma> + phi_7 <pi pi> + lambda_piPi Pi sigma with
                // <A>^{ij} = (A^{ij} + A^{ji})/2 - Delta^{ij} tr A / 3 (pi, sigma transverse)
                A3 Aij = k3(0.0), Aji = k3(0.0);
                double Bij = 0.0;
                for (int l = 0; l < 4; ++l) {
                    Aij = Aij + (pi[i][l] * G.g[l]) * sg[j][l];
                    Aji = Aji + (pi[j][l] * G.g[l]) * sg[i][l];
                    Bij += pi[i][l] * G.g[l] * pi[j][l];
                }
                const double Dij = (i == j ? G.gi[i] : 0.0) - u[i] * u[j];
                const A3 PA = 0.5 * (Aij + Aji) - (Dij / 3.0) * pisig;
                const double PB = Bij - Dij * trB / 3.0;
                const A3 rhs = itp * (2.0 * eta * sg[i][j] + (-pi[i][j]) + k3(v.tr.dnmr[5] / p * PB)) -
                               (v.tr.dnmr[2] * pi[i][j]) * th - v.tr.dnmr[3] * PA + (v.tr.dnmr[4] * Pi) * sg[i][j];
                A3 dpi = ig * (rhs + (-chr) - (u[i] * pja + u[j] * pia));
                A3 x = isg * dpi - (pi[i][j] * isg * isg) * dsg;
                dPv[i][j] = x;
                dPv[j][i] = x;
            }
    }
    double Isrc[4] = {0.0, 0.0, 0.0, 0.0};
    double dN[3] = {0.0, 0.0, 0.0};  // charge rates dN_q/dx0 (charge sources only)
    if (v.ntrack > 0 || v.nparton > 0) {
        // jet tracks (Cartesian) and partons: dP^i/dx0 gains sqrt(-g) I^i/sigma*, dS/dx0 gains
        // u_nu I^nu/(u^0 sigma T); parton charges: dN_q/dx0 = sqrt(-g) I_q/sigma*, and dS/dx0
        // gains -mu_q/T dN_q/dx0 (eq. dsdnrewr, R^S_q = -mu_q/T)
        double Ik[4], Iq[3] = {0.0, 0.0, 0.0};
        if (v.ntrack > 0) {
            jet_deposit(v, G.tau, ys[a], ys[n + a], ys[2 * n + a], Ik);
            for (int k = 0; k < 4; ++k) Isrc[k] += Ik[k];
        }
        if (v.nparton > 0) {
            const double xa[3] = {ys[a], ys[n + a], ys[2 * n + a]};
            parton_deposit(v, G.tau, G.sqrtg, xa, Ik, Iq);
            for (int k = 0; k < 4; ++k) Isrc[k] += Ik[k];
        }
        double uI = 0.0;
        for (int k = 0; k < 4; ++k) uI += G.g[k] * u[k] * Isrc[k];
        uI -= mu[0] * Iq[0] + mu[1] * Iq[1] + mu[2] * Iq[2];
        dS = dS + k3((ig * isg / T) * uI);
        for (int c = 0; c < 3; ++c) dN[c] = G.sqrtg * Iq[c] / sig_star;
    }
    const A3 ds = sigma * dS + (s * isg) * dsg;
    const A3 dPi = sigma * dBv + Bv * dsg;
    // dn_q = N_q dsigma + sigma dN_q
    const A3 dw = (T + ps) * ds + (((mu[0] + pn[0]) * nq[0] + (mu[1] + pn[1]) * nq[1] + (mu[2] + pn[2]) * nq[2]) * isg) * dsg + dPi +
                  k3(sigma * ((mu[0] + pn[0]) * dN[0] + (mu[1] + pn[1]) * dN[1] + (mu[2] + pn[2]) * dN[2]));
    const double w = e + p + Pi;
    const double ig2 = ig * ig, ig3 = ig2 * ig;
    // T^{mu nu} for the Christoffel source of the momentum rate (i = eta in Milne)
    A3 M[3];
    double F[3], cvec[3];
    for (int i = 1; i < 4; ++i) {
        A3 t1 = k3(0.0);
        double t2 = 0.0;
        for (int j = 1; j < 4; ++j) {
            double Pvji = isg * pi[j][i];
            double dgj = (j == 3) ? G.dg3 : 0.0;
            t1 = t1 + k3(dgj * u[j] * Pvji) + (G.g[j] * Pvji) * acc[j] + (G.g[j] * u[j]) * dPv[j][i];
            t2 += G.g[j] * u[j] * Pvji;
        }
        A3 dpi0 = (-ig2) * t1 + (2.0 * t2 * ig3) * du0;
        A3 dP = (u[i] * isg) * dw + (w * isg) * acc[i] - (w * u[i] * isg * isg) * dsg + dpi0;
        double src = 0.0;
        for (int m = 0; m < 4; ++m)
            for (int l = 0; l < 4; ++l) {
                double gml = gam(G, i, m, l);
                if (gml != 0.0) {
                    double Delta = (m == l ? G.gi[m] : 0.0) - u[m] * u[l];
                    src += gml * (e * u[m] * u[l] - (p + Pi) * Delta + pi[m][l]);
                }
            }
        F[i - 1] = gout[(size_t)(9 + i - 1) * n + a] - G.sqrtg * src / sig_star + G.sqrtg * Isrc[i] / sig_star;
        M[i - 1] = dP;
        cvec[i - 1] = dP.c;
    }
    // solve M a = F - c (3x3, partial pivoting)
    double A[3][3] = {{M[0].x, M[0].y, M[0].z}, {M[1].x, M[1].y, M[1].z}, {M[2].x, M[2].y, M[2].z}};
    double b[3] = {F[0] - cvec[0], F[1] - cvec[1], F[2] - cvec[2]};
    uint32_t stt = 0;
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int piv = c;
        double best = fabs(A[c][c]);
#pragma unroll
        for (int r = c + 1; r < 3; ++r)
            if (fabs(A[r][c]) > best) {
                best = fabs(A[r][c]);
                piv = r;
            }
        if (!(best > 0.0) || !isfinite(best)) {
            ok = false;
            break;
        }
#pragma unroll
        for (int r = c + 1; r < 3; ++r)
            if (piv == r) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    double t = A[c][k];
                    A[c][k] = A[r][k];
                    A[r][k] = t;
                }
                double t = b[c];
                b[c] = b[r];
                b[r] = t;
            }
#pragma unroll
        for (int r = c + 1; r < 3; ++r) {
            double f = A[r][c] / A[c][c];
#pragma unroll
            for (int k = c; k < 3; ++k) A[r][k] = fma(-f, A[c][k], A[r][k]);
            b[r] = fma(-f, b[c], b[r]);
        }
    }
    double av[3] = {0.0, 0.0, 0.0};
    if (ok) {
#pragma unroll
        for (int r = 2; r >= 0; --r) {
            double t = b[r];
#pragma unroll
            for (int k = r + 1; k < 3; ++k) t = fma(-A[r][k], av[k], t);
            av[r] = t / A[r][r];
        }
    } else {
        stt |= PST_SOLVE_FAIL;
    }
    double f[13];
    for (int k = 0; k < 3; ++k) f[k] = vv[1 + k];
    for (int k = 0; k < 3; ++k) f[3 + k] = av[k];
    f[6] = at3(dS, av);
    f[7] = at3(dBv, av);
    f[8] = at3(dPv[1][1], av);
    f[9] = at3(dPv[1][2], av);
    f[10] = at3(dPv[1][3], av);
    f[11] = at3(dPv[2][2], av);
    f[12] = at3(dPv[2][3], av);
    bool fin = true;
    for (int k = 0; k < 13; ++k) fin = fin && isfinite(f[k]);
    if (!fin) stt |= PST_NONFINITE;
    if (stt) {
        status[a] |= stt;
        atomicOr(&v.sc->status_or, stt);
    }
    if (mode == 0) {
        for (int k = 0; k < nv; ++k) yout[k * n + a] = ys[k * n + a] + dt * f[k];
    } else if (mode == 1) {
        for (int k = 0; k < nv; ++k) yout[k * n + a] = 0.5 * ((yout[k * n + a] + ys[k * n + a]) + dt * f[k]);
    } else {
        for (int k = 0; k < nv; ++k) rates[k * n + a] = f[k];
    }
    heun_charges(v, mode, n, a, dN);
}

// a8: totals contributions in original order: [0] sqrt(-g) T^{00}/sigma*, [1] S
__global__ void k_totals3(EvView v, const double *__restrict__ y, const int *__restrict__ id,
                          const double *__restrict__ dens, const double *__restrict__ eos, double *__restrict__ contrib)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= v.n) return;
    const size_t n = (size_t)v.n;
    const Geo3 G = geo3(v, 1);
    double u[4] = {dens[5 * n + a], y[3 * n + a], y[4 * n + a], y[5 * n + a]};
    const double sig_star = dens[a];
    const double sigma = sig_star / (u[0] * G.sqrtg);
    double Pi = 0.0, st[5] = {0, 0, 0, 0, 0};
    if (v.tr.viscous) {
        Pi = sigma * y[7 * n + a];
        for (int k = 0; k < 5; ++k) st[k] = sigma * y[(8 + k) * n + a];
    }
    double pi[4][4];
    pi_full3(G, u, 1.0 / u[0], st, pi);
    const double p = eos[4 * n + a], e = eos[5 * n + a];
    const double T00 = (e + p + Pi) * u[0] * u[0] - (p + Pi) + pi[0][0];
    const int o = id[a];
    contrib[o] = G.sqrtg * T00 / sig_star;
    contrib[n + o] = y[6 * n + a];
}

// test support: neighbour pairs (pass 1 counts with offs == nullptr, pass 2 writes)
__global__ void k_neighbors3(EvView v, const double *__restrict__ y, const int *__restrict__ id,
                             const uint32_t *__restrict__ start, const uint32_t *__restrict__ cnt,
                             const long long *__restrict__ offs, int *count_out, int *pa, int *pb)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= v.n) return;
    const size_t n = (size_t)v.n;
    const double xa[3] = {y[a], y[n + a], y[2 * n + a]};
    int c[3], lim[3];
    for (int d = 0; d < 3; ++d) {
        c[d] = cell_coord(xa[d], dec_double(v.sc->xmin_enc[d]), v.inv_cell);
        lim[d] = 1 << v.B3[d];
    }
    long long w = offs ? offs[a] : 0;
    int m = 0;
    for (int oz = -1; oz <= 1; ++oz)
        for (int oy = -1; oy <= 1; ++oy)
            for (int ox = -1; ox <= 1; ++ox) {
                const int nx = c[0] + ox, ny = c[1] + oy, nz = c[2] + oz;
                if (nx < 0 || ny < 0 || nz < 0 || nx >= lim[0] || ny >= lim[1] || nz >= lim[2]) continue;
                const uint32_t k = key3(v, nx, ny, nz);
                for (uint32_t b = start[k]; b < start[k] + cnt[k]; ++b) {
                    double r2 = dist2_3d(xa[0] - y[b], xa[1] - y[n + b], xa[2] - y[2 * n + b]);
                    if (r2 < v.supp2) {
                        if (offs) {
                            pa[w + m] = id[a];
                            pb[w + m] = id[b];
                        }
                        ++m;
                    }
                }
            }
    if (!offs) count_out[a] = m;
}

__global__ void k_cell_coords3(EvView v, const double *__restrict__ y, const int *__restrict__ id, int *cell_orig)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= v.n) return;
    const int o = id[j];
    for (int d = 0; d < 3; ++d)
        cell_orig[(size_t)d * v.n + o] = cell_coord(y[(size_t)d * v.n + j], dec_double(v.sc->xmin_enc[d]), v.inv_cell);
}

inline int nblk(int n, int t) { return (n + t - 1) / t; }

}  // namespace

void launch_cells3(const EvView &v, const double *y, const int *id, CellBufs cb, cudaStream_t st)
{
    (void)id;
    k_cells3<<<nblk(v.n, 256), 256, 0, st>>>(v, y, cb.key, cb.cnt);
}

void launch_density3(const EvView &v, const double *y, const double *Nq, CellBufs cb, double *dens, int *nnb,
                     cudaStream_t st)
{
    if (v.mixed) {
        launch_density3m(v, y, Nq, cb, dens, nnb, st);
        return;
    }
    const int lists = cb.pl.total > 0;
    if (lists) launch_pairs3_density(v, y, Nq, cb, dens, nnb, st);
    // as the fallback of the pair-list passes it usually exits at once: a few blocks per SM
    const int grid = lists ? std::min(nblk(v.n, kWarps3), 8 * device_sm_count()) : nblk(v.n, kWarps3);
    k_density3<<<grid, 32 * kWarps3, 0, st>>>(v, y, cb.fpos3, Nq, cb.start, cb.cnt, dens, nnb, lists,
                                              lists ? cb.pl.cnt_dst : nullptr);
}

void launch_eos3(const EvView &v, int stage, const double *y, const double *dens, double *eos, double *gin,
                 uint32_t *status, double *wpart, const double *guess_in, double *guess_out, cudaStream_t st)
{
    const int sms = device_sm_count(), need = nblk(v.n, 32 * kEosWarps3);
    const int grid = need >= kEosBlocks3 * sms ? kEosBlocks3 * sms : (need >= sms ? (need / sms) * sms : std::max(1, need));
    k_eos3_find<<<grid, 32 * kEosWarps3, 0, st>>>(v, stage, y, const_cast<double *>(dens), status, guess_in, guess_out);
    k_eos3_finish<<<nblk(v.n, 64), 64, 0, st>>>(v, stage, y, dens, eos, gin, status, wpart, guess_out);
}

void launch_gradient3(const EvView &v, int stage, const double *y, const double *gin, CellBufs cb, double *gout,
                      cudaStream_t st)
{
    if (v.mixed) {
        launch_gradient3m(v, stage, y, gin, cb, gout, st);
        return;
    }
    const int lists = cb.pl.total > 0;
    if (lists) launch_pairs3_gradient(v, stage, y, gin, cb, gout, st);
    const int grid = lists ? std::min(nblk(v.n, kWarps3), 8 * device_sm_count()) : nblk(v.n, kWarps3);
    k_gradient3<<<grid, 32 * kWarps3, 0, st>>>(v, stage, y, cb.fpos3, gin, cb.start, cb.cnt, gout, lists);
}

void launch_eom3(const EvView &v, int stage, int mode, const double *ys, const double *dens, const double *eos,
                 const double *gout, double *yout, double *rates, uint32_t *status, cudaStream_t st)
{
    if (v.tr.model != 0) k_eom3<<<nblk(v.n, 64), 64, 0, st>>>(v, stage, mode, ys, dens, eos, gout, yout, rates, status);
    else k_eom3_min_is<<<nblk(v.n, 64), 64, 0, st>>>(v, stage, mode, ys, dens, eos, gout, yout, rates, status);
}

void launch_totals3(const EvView &v, const double *y, const int *id, const double *dens, const double *eos,
                    double *contrib, cudaStream_t st)
{
    k_totals3<<<nblk(v.n, 256), 256, 0, st>>>(v, y, id, dens, eos, contrib);
}

void launch_neighbors_list3(const EvView &v, const double *y, const int *id, CellBufs cb, const long long *offs,
                            int *pa, int *pb, cudaStream_t st)
{
    k_neighbors3<<<nblk(v.n, 128), 128, 0, st>>>(v, y, id, cb.start, cb.cnt, offs, offs ? nullptr : pa, pa, pb);
}

void launch_cell_coords3(const EvView &v, const double *y, const int *id, int *cell_orig, cudaStream_t st)
{
    k_cell_coords3<<<nblk(v.n, 256), 256, 0, st>>>(v, y, id, cell_orig);
}

}  // namespace sphg
