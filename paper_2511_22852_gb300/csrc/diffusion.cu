// diffusion.cu -- BSQ diffusion in 2+1D (Sec. "Equations of motion", eq. min_dif_rel, with the
// constant kappa_{qq'}/T^2 and tau_q T of Sec. "Transport coefficients"): the per-particle inputs
// and the neighbour sums of a stage.  The equations of motion (gradient_eom.cu) take them.
//
// Per particle a (sorted order of the stage):
//   alpha_q = mu_q / T; the flux of the lab charge relative to the particle, F^i_q = J^i_q -
//   v^i J^0_q (J^0 = u.J / u^0 from u_mu J^mu = 0), as F^i_q / sigma*^2; and d alpha_q / d(s, n)
//   = (d mu_q - alpha_q dT) / T with (dT, dmu) = H^-1 (ds, dn), H = d(s, n)/d(T, mu) of the EoS
//   branch that gave the particle's (T, mu) (the table, the closed form or the backup);
//   d_i alpha_q = (1 / sigma*_a) sum_b (alpha_qb - alpha_qa) d_i W_ab  (the SPH derivative with
//   n = 1: zero for a uniform alpha, so a uniform mu/T drives no current);
//   d(lab charge)/dx0 = -sqrt(-g) sum_b (F_a / sigma*_a^2 + F_b / sigma*_b^2) . grad W_ab (n = -1:
//   each pair moves charge from one particle to the other, so the total is conserved).
#include "sph_internal.cuh"
#include "eos_device.cuh"
#include "pairs_fixed.cuh"

namespace sphg {

namespace {

constexpr int kDiffWarps = 4;
constexpr unsigned kFull = 0xFFFFFFFFu;

__global__ void __launch_bounds__(128) k_diff_prep(EvView v, int stage, const double *__restrict__ y,
                                                   const double *__restrict__ dens, const double *__restrict__ eos,
                                                   const uint32_t *__restrict__ status)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= v.n) return;
    const size_t n = (size_t)v.n;
    const double tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
    const double sqrtg = v.milne ? tau : 1.0;
    const double sig_star = dens[a], u0 = dens[5 * n + a];
    const double sigma = sig_star / (u0 * sqrtg);
    const double ux = y[2 * n + a], uy = y[3 * n + a];
    const double vx = ux / u0, vy = uy / u0;
    const double T = eos[a];
    const uint32_t st = status[a];
    const bool ok = !(st & (PST_NOCONV | PST_NONFINITE)) && T > 0.0;
    const double i2 = 1.0 / (sig_star * sig_star);
    double al[3];
    double Fq[3][2];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double Jx = sigma * y[(kJRow + 2 * q) * n + a], Jy = sigma * y[(kJRow + 2 * q + 1) * n + a];
        const double J0 = (ux * Jx + uy * Jy) / u0;
        al[q] = ok ? eos[(1 + q) * n + a] / T : 0.0;
        v.dinp[q * n + a] = al[q];
        Fq[q][0] = (Jx - vx * J0) * i2;
        Fq[q][1] = (Jy - vy * J0) * i2;
        v.dinp[(3 + 2 * q) * n + a] = Fq[q][0];
        v.dinp[(4 + 2 * q) * n + a] = Fq[q][1];
    }
    if (v.dfx) {  // for the pair-list pass: alpha, and the fluxes in limbs
        unsigned ef[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int e0 = fx_exponent(Fq[q][0]), e1 = fx_exponent(Fq[q][1]);
            v.dfx[(2 + q) * n + a] = make_longlong2(fx_word(fx_limbs(Fq[q][0], e0)), fx_word(fx_limbs(Fq[q][1], e1)));
            ef[q] = fx_pair(e0, e1);
        }
        v.dfx[a] = make_longlong2(__double_as_longlong(al[0]), __double_as_longlong(al[1]));
        v.dfx[n + a] = make_longlong2(__double_as_longlong(al[2]), 0);
        v.dfe[a] = make_uint4(ef[0], ef[1], ef[2], 0u);
    }
    double dal[3][4];
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) dal[q][k] = 0.0;
    if (ok) {
        const EosDev &E = v.eos;
        const double x[4] = {T, eos[n + a], eos[2 * n + a], eos[3 * n + a]};
        double H[4][4];
        const bool backup = (st & PST_BACKUP) != 0;
        const bool table = !backup && E.has_table && !(st & (PST_FALLBACK | PST_OUT_OF_TABLE));
        if (backup) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) H[i][j] = 0.0;
            H[0][0] = 12.0 * E.cd_A0 * T * T;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const double m0 = E.cd_mu0[q];
                H[1 + q][1 + q] = 12.0 * E.cd_A0 * x[1 + q] * x[1 + q] / (m0 * m0 * m0 * m0);
            }
        } else if (table) {
            double sn[4];
            tab_eval(E, x, sn, H, nullptr);
        } else {
            double p, sn[4];
            an_eval(E, x[0], x + 1, p, sn, H);
        }
        bool act[4];
        act[0] = true;
#pragma unroll
        for (int q = 0; q < 3; ++q) act[1 + q] = table || backup || E.chi[q] > 0.0;
        // H^-1 over the active directions, one column at a time (inactive rows and columns of H
        // replaced by the identity, their entries of the inverse then set to zero)
        double Hi[4][4];
        bool good = true;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            double A[4][4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                b[i] = i == f ? 1.0 : 0.0;
#pragma unroll
                for (int j = 0; j < 4; ++j) A[i][j] = (act[i] && act[j]) ? H[i][j] : (i == j ? 1.0 : 0.0);
            }
            good = good && solve4(A, b);
#pragma unroll
            for (int i = 0; i < 4; ++i) Hi[i][f] = (act[i] && act[f]) ? b[i] : 0.0;
        }
        if (good)
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int f = 0; f < 4; ++f) dal[q][f] = (Hi[1 + q][f] - al[q] * Hi[0][f]) / T;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int f = 0; f < 4; ++f) v.dal[(4 * q + f) * n + a] = dal[q][f];
}

// the sums of particle a (lane 0 of its warp writes them): S = sum grad W, ga = sum (alpha_b -
// alpha_a) grad W, dv = sum F_b . grad W, lane partials reduced in a fixed butterfly order
__device__ __forceinline__ void diff_finish(const EvView &v, int stage, const double *__restrict__ dens, int a,
                                            int lane, double Gx, double Gy, double (&ga)[3][2], double (&dv)[3])
{
    const size_t n = (size_t)v.n;
    const double *F = v.dinp + 3 * n;
    for (int o = 16; o > 0; o >>= 1) {
        Gx += __shfl_xor_sync(0xFFFFFFFFu, Gx, o);
        Gy += __shfl_xor_sync(0xFFFFFFFFu, Gy, o);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            ga[q][0] += __shfl_xor_sync(0xFFFFFFFFu, ga[q][0], o);
            ga[q][1] += __shfl_xor_sync(0xFFFFFFFFu, ga[q][1], o);
            dv[q] += __shfl_xor_sync(0xFFFFFFFFu, dv[q], o);
        }
    }
    if (lane == 0) {
        const double tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
        const double sqrtg = v.milne ? tau : 1.0;
        const double c = v.sigma_d * v.inv_h;
        const double isig = 1.0 / dens[a];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            v.dout[(2 * q) * n + a] = c * ga[q][0] * isig;
            v.dout[(2 * q + 1) * n + a] = c * ga[q][1] * isig;
            const double div = F[(2 * q) * n + a] * Gx + F[(2 * q + 1) * n + a] * Gy + dv[q];
            v.dout[(6 + q) * n + a] = -sqrtg * c * div;
        }
    }
}

// pair-list form (plain 2D events): half a warp per particle over the entries of its row with the
// kernel gradient stored there (grad_a W_ab h / sigma_d), in integers (pairs_fixed.cuh) but for
// alpha_b - alpha_a, an FP64 subtraction; the fluxes are summed as the gradient pass sums the stresses.
// Bound: issue and the latency of the gathers; 40 k event: 295 us a stage (652 with 17 FP64 operations
// per pair; 223 with the differences and units taken from the values alone).  The values in planes of
// 32 bytes took 320.
__global__ void __launch_bounds__(32 * kDiffWarps, 4) k_diff_pairs(EvView v, int stage, const double *__restrict__ dens,
                                                                   PairBufs pl)
{
    if (v.sc->pair_flag) return;  // a list overflowed: the cell pass runs instead
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, l = lane & 15;
    const long long ap = 2 * ((long long)blockIdx.x * kDiffWarps + wid) + (lane >> 4);
    if (ap - (lane >> 4) >= v.n) return;  // warp-uniform
    const bool on = ap < v.n;
    const int a = on ? (int)ap : v.n - 1;
    const size_t n = (size_t)v.n;
    const long long r0 = pl.off[a], r1 = pl.off[a + 1];
    const int nf = on ? pl.cntF[a] : 0, nt = on ? nf + pl.cntB[a] : 0;
    auto at = [&](int j) { return j < nf ? r0 + j : r1 - nt + j; };  // entry j of a's row
    const double2 *alpha = reinterpret_cast<const double2 *>(v.dfx);
    const double aa[3] = {alpha[a].x, alpha[a].y, alpha[n + a].x};
    // the largest exponents among the terms of each sum, two in 16-bit halves: g_x | g_y, (alpha_b - alpha_a)_q
    // g_x | g_y, F_q^x g_x | F_q^y g_y
    unsigned mG = 0u, mA[3] = {0u, 0u, 0u}, mF[3] = {0u, 0u, 0u};
    for (int j = l; j < nt; j += 16) {
        const long long i = at(j);
        const int b = pl.L[i];
        const double2 g = pl.G[i], al0 = alpha[b], al1 = alpha[n + b];
        const uint4 e = v.dfe[b];
        const unsigned eg = fx_pair(fx_kexp(g.x), fx_kexp(g.y)), ef[3] = {e.x, e.y, e.z};
        const double al[3] = {al0.x, al0.y, al1.x};
        mG = fx_max2(mG, eg);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int ea = fx_exponent(al[q] - aa[q]);
            mA[q] = fx_max2(mA[q], fx_pair(ea, ea) + eg);
            mF[q] = fx_max2(mF[q], ef[q] + eg);
        }
    }
    mG = fx_half_max2(mG);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        mA[q] = fx_half_max2(mA[q]);
        mF[q] = fx_half_max2(mF[q]);
    }
    // exponents of the 11 sums: g (2), 2 + 2 q + i: (alpha_b - alpha_a) g_i, 8 + q: F_b . g
    const int Em[11] = {fx_lo(mG), fx_hi(mG), fx_lo(mA[0]), fx_hi(mA[0]), fx_lo(mA[1]), fx_hi(mA[1]), fx_lo(mA[2]), fx_hi(mA[2]),
                        max(fx_lo(mF[0]), fx_hi(mF[0])), max(fx_lo(mF[1]), fx_hi(mF[1])), max(fx_lo(mF[2]), fx_hi(mF[2]))};
    const int room = fx_room(0, nt);
    FxSum sG[2] = {{0, 0}, {0, 0}}, sA[3][2], sF[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) sA[q][0] = sA[q][1] = sF[q] = FxSum{0, 0};
    auto fold = [&]() {
        fx_fold(sG[0]);
        fx_fold(sG[1]);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            fx_fold(sA[q][0]);
            fx_fold(sA[q][1]);
            fx_fold(sF[q]);
        }
    };
    for (int j = l, it = 1; j < nt; j += 16, ++it) {
        const long long i = at(j);
        const int b = pl.L[i];
        const double2 g = pl.G[i], al0 = alpha[b], al1 = alpha[n + b];
        const uint4 e = v.dfe[b];
        const unsigned ef[3] = {e.x, e.y, e.z};
        const double al[3] = {al0.x, al0.y, al1.x};
        const long long m[2] = {fx_kmant(g.x), fx_kmant(g.y)};
        const int eg[2] = {fx_kexp(g.x) - room, fx_kexp(g.y) - room};
        int hi, lo;
#pragma unroll
        for (int k = 0; k < 2; ++k) sG[k].x += fx_shift(m[k], Em[k] - eg[k] + kGuard);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const double d = al[q] - aa[q];
            const int ea = fx_exponent(d);
            const int2 da = fx_limbs(d, ea);
            const longlong2 F = v.dfx[(2 + q) * n + b];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                fx_split(m[k], Em[2 + 2 * q + k] - eg[k] - ea, hi, lo);
                fx_add(sA[q][k], hi, lo, da);
                fx_split(m[k], Em[8 + q] - eg[k] - (k ? fx_hi(ef[q]) : fx_lo(ef[q])), hi, lo);
                fx_add(sF[q], hi, lo, fx_pair_of(k ? F.y : F.x));
            }
        }
        if ((it & (kFoldEvery - 1)) == 0) fold();
    }
    fold();
    FxTotal t[16];
    t[0] = fx_words(sG[0]);
    t[1] = fx_words(sG[1]);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        t[2 + 2 * q] = fx_words(sA[q][0]);
        t[3 + 2 * q] = fx_words(sA[q][1]);
        t[8 + q] = fx_words(sF[q]);
    }
#pragma unroll
    for (int k = 11; k < 16; ++k) t[k] = FxTotal{0, 0};
    const FxTotal tt = fx_reduce16(t, lane);
    // lane l: 0, 1 sum grad W; 2 + 2 q + i sum (alpha_b - alpha_a) grad_i W; 8 + q sum F_b . grad W
    const int q = l < 8 ? (l - 2) >> 1 : l - 8;
    int El = Em[0];
#pragma unroll
    for (int i = 1; i < 11; ++i)
        if (l == i) El = Em[i];
    double tot = fx_value(tt, l < 2 ? fx_kunit(El + room) : fx_unit(El + room));
    if (El >= kNonFinite) tot = fx_nan();
    const double Gx = __shfl_sync(kFull, tot, lane & 16), Gy = __shfl_sync(kFull, tot, (lane & 16) + 1);
    if (on && l >= 2 && l < 11) {
        const double c = v.sigma_d * v.inv_h;
        if (l < 8) {
            v.dout[(size_t)(l - 2) * n + a] = c * tot * (1.0 / dens[a]);
        } else {
            const double tau = v.sc->tau + (stage == 2 ? v.dtau : 0.0);
            const double sqrtg = v.milne ? tau : 1.0;
            const double *F = v.dinp + 3 * n;
            const double div = F[(2 * q) * n + a] * Gx + F[(2 * q + 1) * n + a] * Gy + tot;
            v.dout[(6 + q) * n + a] = -sqrtg * c * div;
        }
    }
}

// one warp per particle: the 3x3 cells of side 2h around its own, the exact FP64 test r < 2h on
// every candidate (the neighbour set of the other passes).  The mixed-precision form's pass,
// and the plain form's when a pair list overflowed (fallback: it returns at once otherwise).
__global__ void __launch_bounds__(32 * kDiffWarps) k_diff2(EvView v, int stage, const double *__restrict__ y,
                                                           const double *__restrict__ dens,
                                                           const uint32_t *__restrict__ start,
                                                           const uint32_t *__restrict__ cnt, int fallback)
{
    if (fallback && !v.sc->pair_flag) return;  // the pair-list pass did the work
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t n = (size_t)v.n;
    const double xmin0 = dec_double(v.sc->xmin_enc[0]), xmin1 = dec_double(v.sc->xmin_enc[1]);
    const int lim = 1 << v.B;
    const double *al = v.dinp, *F = v.dinp + 3 * n;
    for (int a = blockIdx.x * kDiffWarps + wid; a < v.n; a += gridDim.x * kDiffWarps) {  // warp-uniform
        const double xa = y[a], ya = y[n + a];
        const int cx = cell_coord(xa, xmin0, v.inv_cell), cy = cell_coord(ya, xmin1, v.inv_cell);
        const double aa[3] = {al[a], al[n + a], al[2 * n + a]};
        double ga[3][2] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}}, dv[3] = {0.0, 0.0, 0.0}, Gx = 0.0, Gy = 0.0;
        for (int oy = -1; oy <= 1; ++oy) {
            const int ny = cy + oy;
            if (ny < 0 || ny >= lim) continue;
            for (int ox = -1; ox <= 1; ++ox) {
                const int nx = cx + ox;
                if (nx < 0 || nx >= lim) continue;
                const uint32_t k = morton2((uint32_t)nx, (uint32_t)ny);
                const uint32_t b1 = start[k] + cnt[k];
                for (uint32_t b = start[k] + lane; b < b1; b += 32) {
                    const double dx = xa - y[b], dy = ya - y[n + b];
                    if (!(dist2_2d(dx, dy) < v.supp2)) continue;
                    const double r2 = fma(dx, dx, dy * dy);
                    if (!(r2 > 0.0)) continue;  // grad W = 0 at r = 0
                    const double ir = inv_sqrt(r2);
                    const double fac = kernel_dw(r2 * ir * v.inv_h) * ir;  // (dW/dr)/r without sigma_d/h
                    const double gx = fac * dx, gy = fac * dy;
                    Gx += gx;
                    Gy += gy;
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const double da = al[q * n + b] - aa[q];
                        ga[q][0] = fma(da, gx, ga[q][0]);
                        ga[q][1] = fma(da, gy, ga[q][1]);
                        dv[q] = fma(F[(2 * q) * n + b], gx, fma(F[(2 * q + 1) * n + b], gy, dv[q]));
                    }
                }
            }
        }
        diff_finish(v, stage, dens, a, lane, Gx, Gy, ga, dv);
    }
}

inline int nblk(int n, int t) { return (n + t - 1) / t; }

}  // namespace

void launch_diffusion(const EvView &v, int stage, const double *y, const double *dens, const double *eos,
                      const uint32_t *status, CellBufs cb, cudaStream_t st)
{
    if (!v.diff || v.n <= 0) return;
    k_diff_prep<<<nblk(v.n, 128), 128, 0, st>>>(v, stage, y, dens, eos, status);
    // the plain form keeps pair lists: the pass over them, with the cell pass standing by (at a
    // few blocks per SM) for a stage whose lists overflowed
    const int lists = !v.mixed && cb.pl.total > 0;
    if (lists) k_diff_pairs<<<nblk(v.n, 2 * kDiffWarps), 32 * kDiffWarps, 0, st>>>(v, stage, dens, cb.pl);
    const int grid = lists ? std::min(nblk(v.n, kDiffWarps), 8 * device_sm_count()) : nblk(v.n, kDiffWarps);
    k_diff2<<<grid, 32 * kDiffWarps, 0, st>>>(v, stage, y, dens, cb.start, cb.cnt, lists);
}

}  // namespace sphg
