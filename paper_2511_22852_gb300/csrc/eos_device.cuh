// eos_device.cuh -- device code of the EoS inversion (row a4), shared by the 2+1D and
// 3+1D EoS passes: closed-form EoS, quadrilinear table interpolation with derivatives,
// the damped table Newton, and the warm-started inversion (Sec. "EoS inverter").
#pragma once
#include "sph_internal.cuh"

namespace sphg {
namespace {

// closed-form EoS
__device__ __forceinline__ void an_shape(const EosDev &E, double T, double &f, double &fp, double &fpp)
{
    if (E.a1 == 0.0) {  // conformal: no crossover term
        f = E.a0;
        fp = fpp = 0.0;
        return;
    }
    double k = kHbarc / E.w_GeV;
    double th = tanh((T * kHbarc - E.Tc_GeV) / E.w_GeV);
    double sech2 = fma(-th, th, 1.0);
    f = E.a0 + 0.5 * E.a1 * (1.0 + th);
    fp = 0.5 * E.a1 * sech2 * k;
    fpp = -E.a1 * sech2 * th * k * k;
}

__device__ void an_eval(const EosDev &E, double T, const double *mu, double &p, double sn[4], double H[4][4])
{
    double f, fp, fpp;
    an_shape(E, T, f, fp, fpp);
    double cm2 = E.chi[0] * mu[0] * mu[0] + E.chi[1] * mu[1] * mu[1] + E.chi[2] * mu[2] * mu[2];
    double T2 = T * T, T3 = T2 * T, T4 = T2 * T2;
    p = T4 * f + 0.5 * T2 * cm2;
    sn[0] = 4.0 * T3 * f + T4 * fp + T * cm2;
    for (int q = 0; q < 3; ++q) sn[1 + q] = E.chi[q] * T2 * mu[q];
    H[0][0] = 12.0 * T2 * f + 8.0 * T3 * fp + T4 * fpp + cm2;
    for (int q = 0; q < 3; ++q) {
        double c = 2.0 * E.chi[q] * T * mu[q];
        H[0][1 + q] = c;
        H[1 + q][0] = c;
        for (int r = 0; r < 3; ++r) H[1 + q][1 + r] = (q == r) ? E.chi[q] * T2 : 0.0;
    }
}

// work counters of one inversion (reported as algorithmic work by the benchmark)
struct EosWork {
    unsigned resid, solve, g;
};

// a warp's work and status bits, to its event's counters
__device__ __forceinline__ void add_eos_work(DevScalars *sc, const EosWork &w, unsigned st_or)
{
    const unsigned wres = __reduce_add_sync(0xFFFFFFFFu, w.resid);
    const unsigned wsol = __reduce_add_sync(0xFFFFFFFFu, w.solve);
    const unsigned wg = __reduce_add_sync(0xFFFFFFFFu, w.g);
    const unsigned sor = __reduce_or_sync(0xFFFFFFFFu, st_or);
    if ((threadIdx.x & 31) == 0) {
        if (wres) atomicAdd(&sc->eos_resid, (unsigned long long)wres);
        if (wsol) atomicAdd(&sc->eos_solve, (unsigned long long)wsol);
        if (wg) atomicAdd(&sc->eos_g, (unsigned long long)wg);
        if (sor) atomicOr(&sc->status_or, sor);
    }
}

// g(T) = s(T, mu(T)) - s_target with mu_q(T) = n_q/(chi_q T^2)
__device__ __forceinline__ void an_g(const EosDev &E, double T, double s, double c, double &g, double &gp)
{
    double f, fp, fpp;
    an_shape(E, T, f, fp, fpp);
    const double iT = 1.0 / T, cT3 = c * (iT * iT * iT);  // one reciprocal for both quotients
    double T2 = T * T, T3 = T2 * T, T4 = T2 * T2;
    g = 4.0 * T3 * f + T4 * fp + cT3 - s;
    gp = 12.0 * T2 * f + 8.0 * T3 * fp + T4 * fpp - 3.0 * cT3 * iT;
}

// The closed form's root in single precision by the same bracketing and safeguarded Newton
// iteration as an_invert's (0: not found), as the start of the FP64 iteration: an FP64 evaluation
// of g is a chain of about 50 operations at 64 cycles each, a single-precision one costs 1/15 of it.
__device__ __forceinline__ void an_gf(float a0, float a1, float Tc, float iw, float k, float T, float s, float c,
                                      float &g, float &gp)
{
    const float th = tanhf((T * (float)kHbarc - Tc) * iw), sech2 = fmaf(-th, th, 1.0f);
    const float f = fmaf(0.5f * a1, 1.0f + th, a0), fp = 0.5f * a1 * sech2 * k, fpp = -a1 * sech2 * th * k * k;
    const float iT = 1.0f / T, cT3 = c * (iT * iT * iT), T2 = T * T, T3 = T2 * T;
    g = 4.0f * T3 * f + T2 * T2 * fp + cT3 - s;
    gp = 12.0f * T2 * f + 8.0f * T3 * fp + T2 * T2 * fpp - 3.0f * cT3 * iT;
}
__device__ __noinline__ float an_seed(const EosDev &E, double sd, double cd, double Tguess)
{
    const float a0 = (float)E.a0, a1 = (float)E.a1, Tc = (float)E.Tc_GeV, iw = 1.0f / (float)E.w_GeV,
                k = (float)kHbarc * iw, s = (float)sd, c = (float)cd, Tg = (float)Tguess;
    float Thi = cbrtf(s / (4.0f * a0));
    const bool warm = Tg > 0.0f && Tg < Thi;
    const float t0 = warm ? Tg : Thi, step = warm ? 0.99f : 0.8f;
    float g, gp, Tlo = t0, t = t0;
    an_gf(a0, a1, Tc, iw, k, t0, s, c, g, gp);
    if (g > 0.0f) {
        Thi = t0;
        float gprev = g;
        int j = 0;
        for (; j < 400; ++j) {
            Tlo *= step;
            float gl, gpl;
            an_gf(a0, a1, Tc, iw, k, Tlo, s, c, gl, gpl);
            if (gl <= 0.0f) break;
            if (!(gl <= gprev)) return 0.0f;
            gprev = gl;
        }
        if (j == 400) return 0.0f;
    }
    for (int it = 0; it < 40; ++it) {
        an_gf(a0, a1, Tc, iw, k, t, s, c, g, gp);
        if (g > 0.0f) Thi = t;
        else Tlo = t;
        float tn = t - g / gp;
        if (!(gp > 0.0f) || !(tn > Tlo && tn < Thi)) tn = 0.5f * (Tlo + Thi);
        const bool done = fabsf(tn - t) <= 4e-7f * t;
        t = tn;
        if (done) break;
    }
    return t;
}

// Tguess > 0: the particle's closed-form T of its previous stage (warm start of the bracket and of
// the Newton iteration; the root is the same)
__device__ uint32_t an_invert(const EosDev &E, double s, const double *n, double &T, double *mu, EosWork &w,
                              double Tguess = 0.0)
{
    if (!isfinite(s) || !isfinite(n[0]) || !isfinite(n[1]) || !isfinite(n[2])) return PST_NONFINITE | PST_NOCONV;
    if (!(s > 0.0)) return PST_NOCONV;
    double c = 0.0;
    for (int q = 0; q < 3; ++q) {
        if (E.chi[q] > 0.0) c += n[q] * n[q] / E.chi[q];
        else if (n[q] != 0.0) return PST_NOCONV;
    }
    {
        // FP64 Newton from the single-precision root (about 1e-7 of T off): a step below 1e-9 of T
        // leaves an error of its square, so two evaluations reach the root (measured on the ideal
        // Gubser event: 3 instead of 12 evaluations, EoS pass 303 -> 30 us a stage); anything
        // unexpected leaves the root to the bracketed iteration below
        const double t0 = (double)an_seed(E, s, c, Tguess);
        double t = t0;
        for (int it = 0; it < 5 && t > 0.0; ++it) {
            double g, gp;
            an_g(E, t, s, c, g, gp);
            ++w.g;
            const double d = g / gp, ad = fabs(d);
            if (!(gp > 0.0) || !(ad <= 1e-5 * t)) break;
            t -= d;
            if (ad <= 1e-9 * t) {
                T = t;
                const double it2 = 1.0 / (t * t);
                for (int q = 0; q < 3; ++q) mu[q] = E.chi[q] > 0.0 ? n[q] / E.chi[q] * it2 : 0.0;
                return 0u;
            }
        }
    }
    double Thi = cbrt(s / (4.0 * E.a0));
    // start: the bound cbrt(s / 4 a0) >= T, or a warm start below it
    const bool warm = Tguess > 0.0 && Tguess < Thi;
    const double t0 = warm ? Tguess : Thi;
    double g, gp;
    an_g(E, t0, s, c, g, gp);
    ++w.g;
    double Tlo = t0;
    if (g > 0.0) {  // the root lies below t0: step down to a lower bracket
        Thi = t0;
        const double f = warm ? 0.99 : 0.8;  // fine steps from a warm start
        double gprev = g;
        bool found = false;
        for (int k = 0; k < 400; ++k) {
            Tlo *= f;
            double gl, gpl;
            an_g(E, Tlo, s, c, gl, gpl);
            ++w.g;
            if (gl <= 0.0) {
                found = true;
                break;
            }
            if (gl > gprev) return PST_NOCONV;
            gprev = gl;
        }
        if (!found) return PST_NOCONV;
    }
    double t = t0;
    for (int it = 0; it < 200; ++it) {
        an_g(E, t, s, c, g, gp);
        ++w.g;
        if (g == 0.0) break;
        if (g > 0.0) Thi = t;
        else Tlo = t;
        double tn = t - g / gp;
        if (!(gp > 0.0) || !(tn > Tlo && tn < Thi)) tn = 0.5 * (Tlo + Thi);
        if (fabs(tn - t) <= 4e-16 * t) {
            t = tn;
            break;
        }
        t = tn;
    }
    T = t;
    for (int q = 0; q < 3; ++q) mu[q] = E.chi[q] > 0.0 ? n[q] / (E.chi[q] * t * t) : 0.0;
    return 0u;
}

// ---------------------------------------------------------------------------
// table: the quadrilinear interpolant reduced one axis at a time (mu_Q, mu_S inside each of the
// four (T, mu_B) corner patches, then mu_B, then T), carrying the partial derivatives along
// a non-negative int as a double, below 2^20 by its bits (a conversion between int and double costs
// as much as an FP64 operation)
__device__ __forceinline__ double int_double(int k)
{
    if (k >= (1 << 20)) return (double)k;
    const int e = 31 - __clz(k | 1);
    return k == 0 ? 0.0 : __hiloint2double(((e + 1023) << 20) | ((k << (20 - e)) & 0xFFFFF), 0);
}
// the cell of grid coordinate r and the position in it: the integer part of r >= 1 from its
// mantissa bits, clamped to [0, nx - 2]; r < 1 (negative too) lies in cell 0
__device__ __forceinline__ void locate_steps(double r, int nx, int &i, double &t)
{
    const int hi = __double2hiint(r);
    int k = 0;
    if (hi >= 0x3FF00000) {
        if (nx <= (1 << 20)) k = ((hi & 0xFFFFF) | 0x100000) >> max(0, 20 - ((hi >> 20) - 1023));
        else k = __double2int_rz(r);
    }
    k = min(k, nx - 2);
    i = k;
    t = r - int_double(k);
}
__device__ __forceinline__ void locate(double x, double x0, double inv, int nx, int &i, double &t)
{
    locate_steps((x - x0) * inv, nx, i, t);
}

// sn: interpolated (s, nB, nS, nQ); J[f][k] = d sn_f / d x_k per grid step of axis k (times
// inv_dT, inv_dmu[k-1] for the derivative per unit of x_k); p optional
__device__ void tab_eval_steps(const EosDev &E, const double *x, double sn[4], double J[4][4], double *p)
{
    int iT, iB, iS, iQ;
    double tT, tB, tS, tQ;
    locate(x[0], E.T0, E.inv_dT, E.nT, iT, tT);
    locate(x[1], E.mu0[0], E.inv_dmu[0], E.nmu[0], iB, tB);
    locate(x[2], E.mu0[1], E.inv_dmu[1], E.nmu[1], iS, tS);
    locate(x[3], E.mu0[2], E.inv_dmu[2], E.nmu[2], iQ, tQ);
    const int n3 = E.nmu[2], n23 = E.nmu[1] * E.nmu[2], n123 = E.nmu[0] * n23;
    const size_t node0 = (size_t)iT * n123 + (size_t)iB * n23 + (size_t)iS * n3 + iQ;
    // a node's four fields are 32 contiguous bytes: (s, n_B) and (n_S, n_Q) as two 16-byte loads
    // (the table is a cudaMalloc allocation, 256-byte aligned)
    const double2 *sn2 = reinterpret_cast<const double2 *>(E.sn);
#pragma unroll
    for (int fp = 0; fp < 2; ++fp) {  // a pair of fields at a time: their 16 corner values
        double lv[2][2], lb[2][2], ls[2][2], lq[2][2];  // [field][bT]: after the mu_B reduction
#pragma unroll
        for (int bT = 0; bT < 2; ++bT) {
            double pv[2][2], ps[2][2], pq[2][2];  // [field][bB]: (mu_S, mu_Q) patch value, d/dS, d/dQ
#pragma unroll
            for (int bB = 0; bB < 2; ++bB) {
                const size_t base = node0 + (size_t)bT * n123 + (size_t)bB * n23;
                const double2 q00 = __ldg(sn2 + 2 * base + fp), q01 = __ldg(sn2 + 2 * (base + 1) + fp);
                const double2 q10 = __ldg(sn2 + 2 * (base + n3) + fp), q11 = __ldg(sn2 + 2 * (base + n3 + 1) + fp);
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    const double c00 = g ? q00.y : q00.x, c01 = g ? q01.y : q01.x;
                    const double c10 = g ? q10.y : q10.x, c11 = g ? q11.y : q11.x;
                    const double d0 = c01 - c00, d1 = c11 - c10;  // along mu_Q
                    const double a0 = fma(tQ, d0, c00), a1 = fma(tQ, d1, c10);
                    const double ds = a1 - a0;  // along mu_S
                    pv[g][bB] = fma(tS, ds, a0);
                    ps[g][bB] = ds;
                    pq[g][bB] = fma(tS, d1 - d0, d0);
                }
            }
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const double db = pv[g][1] - pv[g][0];  // along mu_B
                lv[g][bT] = fma(tB, db, pv[g][0]);
                lb[g][bT] = db;
                ls[g][bT] = fma(tB, ps[g][1] - ps[g][0], ps[g][0]);
                lq[g][bT] = fma(tB, pq[g][1] - pq[g][0], pq[g][0]);
            }
        }
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const int f = 2 * fp + g;
            const double dt = lv[g][1] - lv[g][0];  // along T
            sn[f] = fma(tT, dt, lv[g][0]);
            J[f][0] = dt;
            J[f][1] = fma(tT, lb[g][1] - lb[g][0], lb[g][0]);
            J[f][2] = fma(tT, ls[g][1] - ls[g][0], ls[g][0]);
            J[f][3] = fma(tT, lq[g][1] - lq[g][0], lq[g][0]);
        }
    }
    if (p) {
        double lp[2];
#pragma unroll
        for (int bT = 0; bT < 2; ++bT) {
            double pb[2];
#pragma unroll
            for (int bB = 0; bB < 2; ++bB) {
                const size_t base = node0 + (size_t)bT * n123 + (size_t)bB * n23;
                const double p00 = __ldg(E.p + base), p01 = __ldg(E.p + base + 1);
                const double p10 = __ldg(E.p + base + n3), p11 = __ldg(E.p + base + n3 + 1);
                const double a0 = fma(tQ, p01 - p00, p00), a1 = fma(tQ, p11 - p10, p10);
                pb[bB] = fma(tS, a1 - a0, a0);
            }
            lp[bT] = fma(tB, pb[1] - pb[0], pb[0]);
        }
        *p = fma(tT, lp[1] - lp[0], lp[0]);
    }
}

// the same with the derivatives per unit of (T, mu_B, mu_S, mu_Q)
__device__ void tab_eval(const EosDev &E, const double *x, double sn[4], double J[4][4], double *p)
{
    tab_eval_steps(E, x, sn, J, p);
    const double sc[4] = {E.inv_dT, E.inv_dmu[0], E.inv_dmu[1], E.inv_dmu[2]};
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int k = 0; k < 4; ++k) J[f][k] *= sc[k];
}

// 4x4 Gaussian elimination with partial pivoting, fully unrolled so every index is a
// compile-time constant and the system stays in registers.  Row swaps are conditional
// moves; each pivot is inverted once (FP64 division is a multi-instruction sequence on
// the 1:64 FP64 pipe) and the back substitution multiplies by it.  Returns false on a
// zero or non-finite pivot.
// magnitude of a double as an integer: for non-negative doubles the IEEE bit patterns order as
// the values do (NaN above infinity), so the pivot search compares integers
__device__ __forceinline__ long long mag_bits(double v) { return __double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFLL; }
constexpr long long kInfBits = 0x7FF0000000000000LL;

__device__ __forceinline__ bool solve4(double A[4][4], double b[4])
{
    double ipv[4];  // reciprocal pivots, reused by the back substitution
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        int piv = c;
        long long best = mag_bits(A[c][c]);
#pragma unroll
        for (int r = c + 1; r < 4; ++r) {
            const long long v = mag_bits(A[r][c]);
            if (v > best) {
                best = v;
                piv = r;
            }
        }
        if (best == 0 || best >= kInfBits) return false;  // zero, infinite or NaN pivot
#pragma unroll
        for (int r = c + 1; r < 4; ++r) {
            if (piv == r) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    double t = A[c][k];
                    A[c][k] = A[r][k];
                    A[r][k] = t;
                }
                double t = b[c];
                b[c] = b[r];
                b[r] = t;
            }
        }
        double inv = 1.0 / A[c][c];
        ipv[c] = inv;
#pragma unroll
        for (int r = c + 1; r < 4; ++r) {
            double f = A[r][c] * inv;
#pragma unroll
            for (int k = c; k < 4; ++k) A[r][k] = fma(-f, A[c][k], A[r][k]);
            b[r] = fma(-f, b[c], b[r]);
        }
    }
#pragma unroll
    for (int r = 3; r >= 0; --r) {
        double acc = b[r];
#pragma unroll
        for (int k = r + 1; k < 4; ++k) acc = fma(-A[r][k], b[k], acc);
        b[r] = acc * ipv[r];
    }
    return true;
}

// order-preserving integer key of a double (its own inverse): negative values have their
// magnitude bits flipped, so signed integer comparisons order keys as the values
__device__ __forceinline__ long long okey(double v)
{
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFLL);
}
__device__ __forceinline__ double clamp_key(double v, double lo, double hi)
{
    const long long k = min(max(okey(v), okey(lo)), okey(hi));
    return __longlong_as_double(k ^ ((k >> 63) & 0x7FFFFFFFFFFFFFFFLL));
}

// the point into the table's box (exact: a comparison and a selection per bound, on integers)
__device__ __forceinline__ void clamp4(const EosDev &E, double *x)
{
    x[0] = clamp_key(x[0], E.T0, E.Tmax);
#pragma unroll
    for (int q = 0; q < 3; ++q) x[1 + q] = clamp_key(x[1 + q], E.mu0[q], E.mumax[q]);
}

__device__ double resid(const EosDev &E, const double *x, double s, double inv_s, const double *n, double r[4],
                        double J[4][4])
{
    double sn[4];
    tab_eval_steps(E, x, sn, J, nullptr);
    // J / s per unit of x: the grid-step scaling folded into the 1/s scaling
    const double sc[4] = {E.inv_dT * inv_s, E.inv_dmu[0] * inv_s, E.inv_dmu[1] * inv_s, E.inv_dmu[2] * inv_s};
    double tgt[4] = {s, n[0], n[1], n[2]};
    double m = 0.0;
    for (int k = 0; k < 4; ++k) {
        r[k] = (sn[k] - tgt[k]) * inv_s;
        m = isfinite(r[k]) ? fmax(m, fabs(r[k])) : __longlong_as_double(0x7FF0000000000000LL);
        for (int j = 0; j < 4; ++j) J[k][j] *= sc[j];
    }
    return m;
}

// Damped Newton on the table interpolant.  The Jacobian is factorised in place (it is
// not needed after the step); each line-search trial overwrites r and J with their values
// at the trial point, so the accepted point's residual and Jacobian are ready for the
// next iteration (the same sequence as a copy-on-accept scheme, with fewer registers).
// On convergence J holds d(s, n)/d(T, mu) / s at the returned x when *jx is set (the
// caller then needs only p there); otherwise it is stale.
__device__ bool tab_newton(const EosDev &E, double s, const double *n, double *x, EosWork &w, double J[4][4],
                           bool *jx)
{
    double r[4];
    *jx = false;
    const double inv_s = 1.0 / s;
    double rn = resid(E, x, s, inv_s, n, r, J);
    ++w.resid;
    for (int it = 0; it < E.maxit; ++it) {
        double d[4] = {-r[0], -r[1], -r[2], -r[3]};
        if (rn <= E.tol) {
            if (!E.polish) {
                *jx = true;
                return true;
            }
            ++w.solve;
            if (solve4(J, d)) {  // one polishing step, kept when its point still meets the tolerance
                double xn[4] = {x[0] + d[0], x[1] + d[1], x[2] + d[2], x[3] + d[3]};
                clamp4(E, xn);
                ++w.resid;
                if (resid(E, xn, s, inv_s, n, r, J) <= E.tol) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) x[k] = xn[k];
                    *jx = true;
                }
            }
            return true;
        }
        ++w.solve;
        if (!solve4(J, d)) return false;
        double lam = 1.0, xn[4], rnn = 0.0;
        for (int ls = 0; ls <= 8; ++ls) {
#pragma unroll
            for (int k = 0; k < 4; ++k) xn[k] = fma(lam, d[k], x[k]);
            clamp4(E, xn);
            rnn = resid(E, xn, s, inv_s, n, r, J);
            ++w.resid;
            if (rnn < rn) break;
            lam *= 0.5;
        }
        // no decrease along the Newton direction (the root lies beyond a clamped table
        // edge, or the interpolant is flat): the iteration has stalled and ends unconverged
        if (!(rnn < rn)) return false;
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = xn[k];
        rn = rnn;
    }
    return rn <= E.tol;
}

// quadrilinear interpolant of p alone
__device__ double tab_p(const EosDev &E, const double *x)
{
    int iT, iB, iS, iQ;
    double tT, tB, tS, tQ;
    locate(x[0], E.T0, E.inv_dT, E.nT, iT, tT);
    locate(x[1], E.mu0[0], E.inv_dmu[0], E.nmu[0], iB, tB);
    locate(x[2], E.mu0[1], E.inv_dmu[1], E.nmu[1], iS, tS);
    locate(x[3], E.mu0[2], E.inv_dmu[2], E.nmu[2], iQ, tQ);
    const int n3 = E.nmu[2], n23 = E.nmu[1] * E.nmu[2], n123 = E.nmu[0] * n23;
    double pv = 0.0;
    for (int bT = 0; bT < 2; ++bT)
        for (int bB = 0; bB < 2; ++bB) {
            double wT = bT ? tT : 1.0 - tT, wB = bB ? tB : 1.0 - tB;
            size_t base = (size_t)(iT + bT) * n123 + (size_t)(iB + bB) * n23 + (size_t)iS * n3 + iQ;
            double p00 = __ldg(E.p + base), p01 = __ldg(E.p + base + 1), p10 = __ldg(E.p + base + n3),
                   p11 = __ldg(E.p + base + n3 + 1);
            double a0 = p00 + tQ * (p01 - p00), a1 = p10 + tQ * (p11 - p10);
            pv = fma(wT * wB, a0 + tS * (a1 - a0), pv);
        }
    return pv;
}

// Offline inverter: the quadrilinear interpolant of the inverted table at (s, n_q / s); false
// outside the grid or where a corner holds no solution
__device__ bool inv_lookup(const EosDev &E, double s, const double *n, double *x)
{
    if (!(s > 0.0)) return false;
    const int K = E.inv_K, nd = E.inv_nd, nx = E.inv_nx;
    int d = (int)floor(log10(s / E.inv_p10[0]));
    if (d < 0 || d > nd) return false;
    double m = s / E.inv_p10[d];
    if (m >= 10.0 && d < nd) {
        m /= 10.0;
        d += 1;
    }
    if (m < 1.0 && d > 0) {
        m *= 10.0;
        d -= 1;
    }
    const double r = (m - 1.0) * K / 9.0;
    int j = (int)floor(r);
    j = max(0, min(j, K - 1));
    const long long i = (long long)d * K + j;
    if (i < 0 || i > (long long)K * nd - 1) return false;
    int ix[4];
    double t[4];
    ix[0] = (int)i;
    t[0] = r - j;
    if (!(t[0] >= 0.0 && t[0] <= 1.0)) return false;
    const double dxr = 2.0 * E.inv_xmax / (nx - 1);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double rr = (n[q] / s + E.inv_xmax) / dxr;
        if (!(rr >= 0.0 && rr <= (double)(nx - 1))) return false;
        const int k = min((int)floor(rr), nx - 2);
        ix[1 + q] = k;
        t[1 + q] = rr - k;
    }
    x[0] = x[1] = x[2] = x[3] = 0.0;
    const long long ns = (long long)K * nd + 1;
    for (int corner = 0; corner < 16; ++corner) {
        const int b0 = (corner >> 3) & 1, b1 = (corner >> 2) & 1, b2 = (corner >> 1) & 1, b3 = corner & 1;
        const long long node = (((long long)(ix[0] + b0) * nx + ix[1] + b1) * nx + ix[2] + b2) * nx + ix[3] + b3;
        const double w = (b0 ? t[0] : 1.0 - t[0]) * (b1 ? t[1] : 1.0 - t[1]) * (b2 ? t[2] : 1.0 - t[2]) *
                         (b3 ? t[3] : 1.0 - t[3]);
        const double2 *v = reinterpret_cast<const double2 *>(E.inv + 4 * node);
        const double2 a = __ldg(v), b = __ldg(v + 1);
        if (!isfinite(a.x)) return false;
        x[0] = fma(w, a.x, x[0]);
        x[1] = fma(w, a.y, x[1]);
        x[2] = fma(w, b.x, x[2]);
        x[3] = fma(w, b.y, x[3]);
    }
    (void)ns;
    return true;
}

struct EosOut {
    double T, mu[3], p, e, ps, pn[3], cs2;
    uint32_t st;
};

// the conformal-diagonal backup EoS (Sec. "Equation of state", backup EoS) inverted in closed
// form: s = 4 A0 T^3, n_q = 4 A0 mu_q^3 / mu_q0^4; e = 3 p; p_s = T/3, p_{n_q} = mu_q/3
__device__ __forceinline__ EosOut backup_eos(const EosDev &E, double s, const double *n)
{
    EosOut o;
    const double A0 = E.cd_A0;
    o.T = cbrt(s / (4.0 * A0));
    double pq = 0.0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double m0 = E.cd_mu0[q], m02 = m0 * m0;
        o.mu[q] = cbrt(n[q] * m02 * m02 / (4.0 * A0));
        const double r = o.mu[q] / m0, r2 = r * r;
        pq += r2 * r2;
        o.pn[q] = o.mu[q] / 3.0;
    }
    const double T2 = o.T * o.T;
    o.p = A0 * (T2 * T2 + pq);
    o.e = 3.0 * o.p;
    o.ps = o.T / 3.0;
    o.cs2 = 1.0 / 3.0;
    o.st = PST_BACKUP;
    return o;
}

__device__ __forceinline__ bool inside_table(const EosDev &E, const double *x)
{
    bool in = x[0] >= E.T0 && x[0] <= E.Tmax;
#pragma unroll
    for (int q = 0; q < 3; ++q) in = in && x[1 + q] >= E.mu0[q] && x[1 + q] <= E.mumax[q];
    return in;
}

// guess: this particle's table solution of the previous stage (T <= 0: none).  Attempts:
// table Newton from the guess; else the closed form, then table Newton from it; else the
// closed form (flagged).  used_table tells whether the table produced the result.
__device__ EosOut eos_invert(const EosDev &E, double cs2_cap, double s, const double *n, const double *guess,
                             bool &used_table, EosWork &w)
{
    EosOut o;
    o.T = 0.0;
    for (int q = 0; q < 3; ++q) o.mu[q] = 0.0, o.pn[q] = 0.0;
    o.p = o.e = o.ps = o.cs2 = 0.0;
    o.st = 0u;
    used_table = false;
    if (!isfinite(s) || !isfinite(n[0]) || !isfinite(n[1]) || !isfinite(n[2])) {
        o.st = PST_NONFINITE | PST_NOCONV;
        return o;
    }
    double x[4];
    double H[4][4];
    bool use_table = false, hx = false;
    if (E.offline && E.has_table && inv_lookup(E, s, n, x) && inside_table(E, x)) use_table = true;
    if (!use_table && E.has_table && guess[0] > 0.0 && inside_table(E, guess)) {
        double xt[4] = {guess[0], guess[1], guess[2], guess[3]};
        if (tab_newton(E, s, n, xt, w, H, &hx)) {
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = xt[k];
            use_table = true;
        }
    }
    if (!use_table) {
        // a negative guess is the particle's previous closed-form T
        o.st = an_invert(E, s, n, x[0], x + 1, w, guess[0] < 0.0 ? -guess[0] : 0.0);
        if (o.st && E.backup && s > 0.0) return backup_eos(E, s, n);
        if (o.st) return o;
        if (E.has_table) {
            if (inside_table(E, x)) {
                double xt[4] = {x[0], x[1], x[2], x[3]};
                if (tab_newton(E, s, n, xt, w, H, &hx)) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) x[k] = xt[k];
                    use_table = true;
                } else {
                    o.st |= PST_FALLBACK;
                }
            } else {
                o.st |= PST_OUT_OF_TABLE;
            }
        }
    }
    used_table = use_table;
    double p, sn[4];
    if (use_table && hx) {  // the Newton's last Jacobian is the one at the solution
        p = tab_p(E, x);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) H[i][j] *= s;
    } else if (use_table) {
        tab_eval(E, x, sn, H, &p);
        ++w.resid;
    } else {
        an_eval(E, x[0], x + 1, p, sn, H);
    }
    double e = x[0] * s + x[1] * n[0] + x[2] * n[1] + x[3] * n[2] - p;
    // (p_s, p_n) = H^-T (s, n) over the directions the EoS couples to; an uncoupled charge
    // direction (no table, chi_q = 0) becomes an identity row with zero right-hand side
    double A[4][4], z[4] = {s, n[0], n[1], n[2]};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool act_i = i == 0 || use_table || E.chi[i - 1] > 0.0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool act_j = j == 0 || use_table || E.chi[j - 1] > 0.0;
            A[i][j] = (act_i && act_j) ? H[j][i] : (i == j ? 1.0 : 0.0);
        }
        if (!act_i) z[i] = 0.0;
    }
    ++w.solve;
    if (!solve4(A, z)) {
        o.st |= PST_NOCONV;
        return o;
    }
    double cs2 = (s * z[0] + n[0] * z[1] + n[1] * z[2] + n[2] * z[3]) / (e + p);
    if (cs2 > cs2_cap) {
        double f = cs2_cap / cs2;
#pragma unroll
        for (int k = 0; k < 4; ++k) z[k] *= f;
        cs2 = cs2_cap;
        o.st |= PST_CS2_CAPPED;
    }
    o.T = x[0];
    for (int q = 0; q < 3; ++q) o.mu[q] = x[1 + q], o.pn[q] = z[1 + q];
    o.p = p;
    o.e = e;
    o.ps = z[0];
    o.cs2 = cs2;
    return o;
}

// ---------------------------------------------------------------------------
// The EoS pass in two halves.
//
// eos_find brings every particle to its (T, mu): the damped table Newton from the warm start,
// else from the closed form's solution, else the closed form.  A Newton step only has to reduce
// the residual, so it takes the residual (s, n_q) - target in FP64 and the Jacobian and the 4x4
// solve in FP32, from the same node values: an FP32 step is off by about 1e-6 of its length, and
// the point handed on is decided by FP64 residuals alone.  FP64 operations per evaluation fall from
// 360 (values, derivatives, p, solve) to about 110, and one evaluation fewer is needed: the last
// step is taken when the residual is below the hand-over bound, and eos_finish looks at its
// result.  The Newton's work varies from particle to particle, so the lanes refill: each lane
// holds its own particle and claims the next one as soon as its own is handed on.  Where FP32 does not
// do (rough_step, exact_step: charges that move together, differences that it does not resolve; a
// singular system; maxit steps), the particle is left to the general FP64 inversion from its own start.
//
// eos_finish evaluates p, e and (p_s, p_n) = H^-T (s, n) at that point in FP64, one thread per
// particle, all lanes alike.  A table point whose residual misses the tolerance there (a step
// across a cell boundary, rarely), or with polish the rounding level (kPolished: the FP32 step did not
// reduce the residual as an FP64 step does), goes through the general FP64 inversion from that point,
// and so do, from their starts, the particles that the search left to it.
//
// Bound: the FP64 pipe (64 cycles per warp instruction and quadrant).  Measured per stage on the
// 40 k viscous BSQ event: 111 us (196 in one pass with the derivatives and the solve of every
// evaluation in FP64), ideal Gubser lattice 31 (303), eight served events (437 k particles) 593 (772),
// 3+1D Milne event of 258 k particles, mixed form, 505 (976).
//
// Hand-over bounds on max |residual| / s: 1e-10 where the point has to be the root to rounding
// (polish), 1e-6 for the 1e-10 tolerance of the mixed and serving forms.
// status bits between the halves: the point is taken as it is; the general inversion from the start
constexpr uint32_t kNoVerify = 0x80000000u, kGeneral = 0x40000000u;
// max |residual| / s of a polished point: the rounding of the interpolant, about 20 operations of 2^-53 on node
// values of a few s
constexpr double kPolished = 8e-15;

// magnitude-truncated single-precision value of a double, from its bits (|v| < 2^-126: zero)
__device__ __forceinline__ float f32_bits(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v), m = hi & 0x7FFFFFFFu;
    const unsigned r = __funnelshift_l((unsigned)__double2loint(v), m - 0x38000000u, 3);
    return __uint_as_float((hi & 0x80000000u) | (m < 0x38100000u ? 0u : r));
}
// a float as a double by bits (denormals: zero; the exponent 255 becomes a large finite number)
__device__ __forceinline__ double f64_bits(float v)
{
    const unsigned b = __float_as_uint(v), m = b & 0x7FFFFFFFu;
    if (m < 0x00800000u) return 0.0;
    return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
}

// residual of (s, n_B, n_S, n_Q) at the grid coordinates xi in FP64 and its Jacobian per grid step in FP32
__device__ __forceinline__ void tab_resid_steps(const EosDev &E, const double *xi, const double *tgt, double r[4],
                                                float J[4][4])
{
    int iT, iB, iS, iQ;
    double tT, tB, tS, tQ;
    locate_steps(xi[0], E.nT, iT, tT);
    locate_steps(xi[1], E.nmu[0], iB, tB);
    locate_steps(xi[2], E.nmu[1], iS, tS);
    locate_steps(xi[3], E.nmu[2], iQ, tQ);
    const int n3 = E.nmu[2], n23 = E.nmu[1] * E.nmu[2], n123 = E.nmu[0] * n23;
    const size_t node0 = (size_t)iT * n123 + (size_t)iB * n23 + (size_t)iS * n3 + iQ;
    const double2 *sn2 = reinterpret_cast<const double2 *>(E.sn);
    const double uT = 1.0 - tT, uB = 1.0 - tB, uS = 1.0 - tS, uQ = 1.0 - tQ;
    const double w00 = uS * uQ, w01 = uS * tQ, w10 = tS * uQ, w11 = tS * tQ;
    const double wp[4] = {uT * uB, uT * tB, tT * uB, tT * tB};
    const float fT = f32_bits(tT), fB = f32_bits(tB), fS = f32_bits(tS), fQ = f32_bits(tQ);
#pragma unroll
    for (int fp = 0; fp < 2; ++fp) {
        double acc[2] = {-tgt[2 * fp], -tgt[2 * fp + 1]};
        float lv[2][2], lb[2][2], ls[2][2], lq[2][2];
#pragma unroll
        for (int bT = 0; bT < 2; ++bT) {
            float pv[2][2], ps[2][2], pq[2][2];
#pragma unroll
            for (int bB = 0; bB < 2; ++bB) {
                const size_t base = node0 + (size_t)bT * n123 + (size_t)bB * n23;
                const double2 q00 = __ldg(sn2 + 2 * base + fp), q01 = __ldg(sn2 + 2 * (base + 1) + fp);
                const double2 q10 = __ldg(sn2 + 2 * (base + n3) + fp), q11 = __ldg(sn2 + 2 * (base + n3 + 1) + fp);
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    const double c00 = g ? q00.y : q00.x, c01 = g ? q01.y : q01.x;
                    const double c10 = g ? q10.y : q10.x, c11 = g ? q11.y : q11.x;
                    acc[g] = fma(wp[2 * bT + bB], fma(w11, c11, fma(w10, c10, fma(w01, c01, w00 * c00))), acc[g]);
                    const float e00 = f32_bits(c00), e01 = f32_bits(c01), e10 = f32_bits(c10), e11 = f32_bits(c11);
                    const float d0 = e01 - e00, d1 = e11 - e10;
                    const float a0 = fmaf(fQ, d0, e00), a1 = fmaf(fQ, d1, e10), ds = a1 - a0;
                    pv[g][bB] = fmaf(fS, ds, a0);
                    ps[g][bB] = ds;
                    pq[g][bB] = fmaf(fS, d1 - d0, d0);
                }
            }
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                lb[g][bT] = pv[g][1] - pv[g][0];
                lv[g][bT] = fmaf(fB, lb[g][bT], pv[g][0]);
                ls[g][bT] = fmaf(fB, ps[g][1] - ps[g][0], ps[g][0]);
                lq[g][bT] = fmaf(fB, pq[g][1] - pq[g][0], pq[g][0]);
            }
        }
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const int f = 2 * fp + g;
            r[f] = acc[g];
            J[f][0] = lv[g][1] - lv[g][0];
            J[f][1] = fmaf(fT, lb[g][1] - lb[g][0], lb[g][0]);
            J[f][2] = fmaf(fT, ls[g][1] - ls[g][0], ls[g][0]);
            J[f][3] = fmaf(fT, lq[g][1] - lq[g][0], lq[g][0]);
        }
    }
}

// 4x4 Gaussian elimination with partial pivoting in FP32 (solve4's order)
__device__ __forceinline__ bool solve4f(float A[4][4], float b[4])
{
    float ipv[4];
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        int piv = c;
        float best = fabsf(A[c][c]);
#pragma unroll
        for (int r = c + 1; r < 4; ++r) {
            const float v = fabsf(A[r][c]);
            if (v > best) {
                best = v;
                piv = r;
            }
        }
        ok = ok && best > 0.0f && best < __int_as_float(0x7F800000);
#pragma unroll
        for (int r = c + 1; r < 4; ++r) {
            const bool sw = piv == r;
#pragma unroll
            for (int k = c; k < 4; ++k) {
                const float t = A[c][k];
                A[c][k] = sw ? A[r][k] : t;
                A[r][k] = sw ? t : A[r][k];
            }
            const float t = b[c];
            b[c] = sw ? b[r] : t;
            b[r] = sw ? t : b[r];
        }
        const float inv = __frcp_rn(A[c][c]);
        ipv[c] = inv;
#pragma unroll
        for (int r = c + 1; r < 4; ++r) {
            const float f = A[r][c] * inv;
#pragma unroll
            for (int k = c + 1; k < 4; ++k) A[r][k] = fmaf(-f, A[c][k], A[r][k]);
            b[r] = fmaf(-f, b[c], b[r]);
        }
    }
#pragma unroll
    for (int r = 3; r >= 0; --r) {
        float acc = b[r];
#pragma unroll
        for (int k = r + 1; k < 4; ++k) acc = fmaf(-A[r][k], b[k], acc);
        b[r] = acc * ipv[r];
    }
    return ok;
}

// inside_table on integer keys (an FP64 comparison costs an FP64 operation)
__device__ __forceinline__ bool inside_keys(const EosDev &E, const double *x)
{
    bool in = okey(x[0]) >= okey(E.T0) && okey(x[0]) <= okey(E.Tmax);
#pragma unroll
    for (int q = 0; q < 3; ++q) in = in && okey(x[1 + q]) >= okey(E.mu0[q]) && okey(x[1 + q]) <= okey(E.mumax[q]);
    return in;  // NaN keys lie beyond every bound
}
// max |r| as an integer magnitude; non-finite ones count as infinite
__device__ __forceinline__ long long resid_norm(const double *r)
{
    long long m = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) m = max(m, min(mag_bits(r[k]), kInfBits));
    return m;
}
__device__ __forceinline__ bool finite_bits(double v) { return mag_bits(v) < kInfBits; }

// the closed form as a call of its own: the lane loop keeps its registers for the table Newton
__device__ __noinline__ uint32_t an_invert_call(const EosDev &E, double s, const double *n, double *x, EosWork &w,
                                                double Tguess)
{
    return an_invert(E, s, n, x[0], x + 1, w, Tguess);
}

// upper grid coordinates as bit patterns (non-negative doubles order as integers)
__device__ __forceinline__ void grid_top(const EosDev &E, long long top[4])
{
    top[0] = __double_as_longlong(int_double(E.nT - 1));
#pragma unroll
    for (int q = 0; q < 3; ++q) top[1 + q] = __double_as_longlong(int_double(E.nmu[q] - 1));
}
// the trial point x + lam d in grid coordinates, clamped to the grid
__device__ __forceinline__ void trial_point(const long long *top, const double *x, const float *d, float lam, double *out)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const long long b = __double_as_longlong(x[k] + f64_bits(lam * d[k]));
        out[k] = __longlong_as_double(b < 0 ? 0LL : min(b, top[k]));
    }
}

// Whether the FP32 step d at residual norm r may not decrease the residual where the exact one does.  The
// Jacobian per grid step in FP32 is off by at most 2^-21 of the node values, and the elimination by about
// as much, so |J d + r| <= 2^-17 v sum |d_k| with v the node values, which the target and the residual
// bound (about 4 (|target| + r)): up to r/4 it does.
__device__ __forceinline__ bool rough_step(const float *d, float r, float target)
{
    const float sum = (fabsf(d[0]) + fabsf(d[1])) + (fabsf(d[2]) + fabsf(d[3]));
    return !(0x1p-15f * (target + r) * sum <= r);
}
// Whether the FP32 step d from a point with residual r and FP32 Jacobian J is the exact one to 1/32 of its
// length, so that a search along the one stalls as along the other: its error is J^-1 (E d) with |E_fk| <=
// 2^-20 v_f, v_f the node values of field f, bounded by the target, the residual and the differences.
// Four lanes in a row (f = lane & 3) with the same arguments take a column of the inverse each.
__device__ __forceinline__ bool exact_step(float (&J)[4][4], const double *r, const double *tgt, const float *d, int f)
{
    float rn = 0.f, sum = 0.f, top = 0.f, v = 0.f, e[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        rn = fmaxf(rn, fabsf(f32_bits(r[k])));
        sum += fabsf(d[k]);
        top = fmaxf(top, fabsf(d[k]));
        if (k == f) v = ((fabsf(J[k][0]) + fabsf(J[k][1])) + (fabsf(J[k][2]) + fabsf(J[k][3]))) + fabsf(f32_bits(tgt[k]));
        e[k] = k == f ? 1.f : 0.f;
    }
    v = 0x1p-18f * (v + rn) * sum;
    // a step below the single-precision range is zero here
    bool ok = solve4f(J, e) && top > 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float err = fabsf(e[i]) * v;
        err += __shfl_xor_sync(0xFFFFFFFFu, err, 1);
        err += __shfl_xor_sync(0xFFFFFFFFu, err, 2);
        ok = ok && err <= 0x1p-5f * top;
    }
    return ok;
}

// The line searches of a warp's lanes in todo after a full step without a decrease: the halvings
// 1/2 .. 1/2^8 of one particle at a time, a lane for each, and the largest that decreases the
// residual (the first that a search trial by trial would take).  xt: the point found; false: none, and
// exact says whether the step is an exact_step (the other lanes look, at the point itself).
// One trial a trip held the whole pass for particles beyond a table edge, whose searches fail
// every stage: 40 k event with three such particles, EoS pass 341 us per step, 270 with the trials side
// by side, 290 with the look at the step (after 1,200 steps, with 133 such particles, 346 and 359).
__device__ __noinline__ bool line_searches(const EosDev &E, unsigned todo, const double *xi, const float *d,
                                           const double *tgt, long long rn, double *xt, unsigned &trials, bool &exact)
{
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    bool found = false;
    long long top[4];
    grid_top(E, top);
    for (; todo; todo &= todo - 1u) {
        const int src = __ffs(todo) - 1;
        double xs[4], ts[4], xl[4];
        float ds[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            xs[k] = __shfl_sync(FULL, xi[k], src);
            ts[k] = __shfl_sync(FULL, tgt[k], src);
            ds[k] = __shfl_sync(FULL, d[k], src);
        }
        const long long rs = __shfl_sync(FULL, rn, src);
        double r[4];
        float J[4][4];
        if (lane < 8) trial_point(top, xs, ds, __int_as_float((126 - lane) << 23), xl);
#pragma unroll
        for (int k = 0; k < 4; ++k) xl[k] = lane < 8 ? xl[k] : xs[k];
        tab_resid_steps(E, xl, ts, r, J);
        const unsigned m = __ballot_sync(FULL, lane < 8 && resid_norm(r) < rs);
        const unsigned mx = m ? 0u : __ballot_sync(FULL, exact_step(J, r, ts, ds, lane & 3) && (lane >> 2) == 2);
        if (lane == src) {
            trials = m ? (unsigned)__ffs(m) : 8u;
            found = m != 0u;
            exact = mx == 0xF00u;
            if (m) trial_point(top, xi, d, __int_as_float((127 - __ffs(m)) << 23), xt);  // evaluated and accepted next
        }
    }
    return found;
}

// First half.  Ctx supplies  bool load(int a, double &s, double n[3], double g[4])  (false: not a
// particle of this pass; g: the warm start, T > 0 a table solution, T < 0 minus a closed-form T)
// void put(int a, const double x[4], uint32_t st): T > 0 a table point, T < 0 minus the closed form's
// T, 0 none (st tells why), and  void keep(int a, const double g[4]), which leaves the warm start where
// put leaves the result (kGeneral), and  void mark(int a, uint32_t st), the status alone.
// claim: the pass's particle counter.
// Every loop ends: a search takes at most maxit accepted points and one line search after each (its
// point has to be accepted next), from the warm start and from the closed form.
template <class Ctx>
__device__ void eos_find(const EosDev &E, unsigned int *claim, int limit, Ctx &ctx, EosWork &w)
{
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const double step[4] = {E.dT, E.dmu[0], E.dmu[1], E.dmu[2]};
    const double istep[4] = {E.inv_dT, E.inv_dmu[0], E.inv_dmu[1], E.inv_dmu[2]};
    const double org[4] = {E.T0, E.mu0[0], E.mu0[1], E.mu0[2]};
    long long top[4];
    grid_top(E, top);
    const double hand = E.polish ? 1e-10 : 1e-6;
    int a = -1, it = 0;
    bool more = true, first = false, cold = false, searched = false;  // searched: xt is a line search's
    long long rn = 0, tolb = 0, handb = 0;
    double xi[4] = {0.0, 0.0, 0.0, 0.0}, xt[4] = {0.0, 0.0, 0.0, 0.0}, tgt[4] = {0.0, 0.0, 0.0, 0.0}, Tcf = 0.0;
    float d[4] = {0.f, 0.f, 0.f, 0.f}, tmax = 0.f;
    for (;;) {
        // lanes without a particle claim the next ones (one atomic per warp)
        const unsigned need = __ballot_sync(FULL, a < 0 && more);
        if (need) {
            const int leader = __ffs(need) - 1;
            unsigned base = 0u;
            if (lane == leader) base = atomicAdd(claim, (unsigned)__popc(need));
            base = __shfl_sync(FULL, base, leader);
            bool closed = false;
            double g[4] = {0.0, 0.0, 0.0, 0.0};
            if (a < 0 && more) {
                const long long idx = (long long)base + __popc(need & ((1u << lane) - 1u));
                if (idx >= limit) {
                    more = false;
                } else if (ctx.load((int)idx, tgt[0], tgt + 1, g)) {
                    a = (int)idx;
                    const bool fin = finite_bits(tgt[0]) && finite_bits(tgt[1]) && finite_bits(tgt[2]) && finite_bits(tgt[3]);
                    closed = true;
                    if (!fin) {
                        const double z[4] = {0.0, 0.0, 0.0, 0.0};
                        ctx.put(a, z, PST_NONFINITE | PST_NOCONV);
                        a = -1;
                        closed = false;
                    } else if (E.has_table && E.offline) {
                        double x[4];
                        if (inv_lookup(E, tgt[0], tgt + 1, x) && inside_table(E, x)) {
                            ctx.put(a, x, kNoVerify);
                            a = -1;
                            closed = false;
                        }
                    }
                    if (closed && E.has_table && __double_as_longlong(g[0]) > 0 && inside_keys(E, g) &&
                        __double_as_longlong(tgt[0]) > 0) {
                        closed = cold = false;
#pragma unroll
                        for (int k = 0; k < 4; ++k) xt[k] = (g[k] - org[k]) * istep[k];
                    }
                }
            }
            if (closed) {
                double x[4] = {0.0, 0.0, 0.0, 0.0};
                const uint32_t st = an_invert_call(E, tgt[0], tgt + 1, x, w, __double_as_longlong(g[0]) < 0 ? -g[0] : 0.0);
                if (!st && E.has_table && inside_keys(E, x)) {
                    cold = true;
                    Tcf = x[0];
#pragma unroll
                    for (int k = 0; k < 4; ++k) xt[k] = (x[k] - org[k]) * istep[k];
                } else {
                    x[0] = st ? 0.0 : -x[0];
                    ctx.put(a, x, st ? (E.backup && tgt[0] > 0.0 ? PST_BACKUP : st) : (E.has_table ? PST_OUT_OF_TABLE : 0u));
                    a = -1;
                }
            }
            if (a >= 0 && ((need >> lane) & 1u)) {
                ctx.keep(a, g);
                first = true;
                searched = false;
                it = 0;
                tmax = fmaxf(fmaxf(fabsf(f32_bits(tgt[0])), fabsf(f32_bits(tgt[1]))), fmaxf(fabsf(f32_bits(tgt[2])), fabsf(f32_bits(tgt[3]))));
                tolb = __double_as_longlong(E.tol * tgt[0]);
                handb = max(tolb, __double_as_longlong(hand * tgt[0]));
            }
        }
        if (__ballot_sync(FULL, a >= 0 || more) == 0u) break;
        bool fail = false, general = false, step_on = false, last = false, search = false;
        if (a >= 0) {
            // one evaluation at the trial point
            double r[4];
            float J[4][4];
            tab_resid_steps(E, xt, tgt, r, J);
            ++w.resid;
            const long long rnn = resid_norm(r);
            if (first || rnn < rn) {
                it += first ? 0 : 1;
                first = searched = false;
#pragma unroll
                for (int k = 0; k < 4; ++k) xi[k] = xt[k];
                rn = rnn;
                if (rn <= tolb && (!E.polish || it >= E.maxit)) last = true;
                else if (it >= E.maxit) general = true;
                else if (rn <= handb) last = step_on = true;
                else step_on = true;
            } else if (searched) {
                general = true;
            } else {
                search = true;
            }
            if (step_on) {
                ++w.solve;
#pragma unroll
                for (int k = 0; k < 4; ++k) d[k] = -f32_bits(r[k]);
                const bool ok = solve4f(J, d);
                general = !ok || rough_step(d, f32_bits(__longlong_as_double(rn)), tmax);
                trial_point(top, xi, d, 1.0f, xt);
            }
        }
        // no decrease at the full step: the line searches of the warp's lanes, rarely
        const unsigned todo = __ballot_sync(FULL, search);
        if (todo) {
            double xs[4], ts[4], xo[4];
            float ds[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) xs[k] = xi[k], ts[k] = tgt[k], ds[k] = d[k], xo[k] = xt[k];
            unsigned trials = 0u;
            bool exact = false;
            const bool found = line_searches(E, todo, xs, ds, ts, rn, xo, trials, exact);
            w.resid += trials;
            if (search) {
                searched = true;
                fail = !found;  // no decrease along the Newton direction: stalled
                general = fail && !exact;
#pragma unroll
                for (int k = 0; k < 4; ++k) xt[k] = xo[k];
            }
        }
        if (general) {
            ctx.mark(a, kGeneral);
            a = -1;
        } else if (last) {
            double x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = fma(step_on ? xt[k] : xi[k], step[k], org[k]);
            clamp4(E, x);
            ctx.put(a, x, 0u);
            a = -1;
        } else if (fail) {
            double x[4] = {0.0, 0.0, 0.0, 0.0};
            if (!cold) {  // the table Newton from the warm start failed: from the closed form
                const uint32_t st = an_invert_call(E, tgt[0], tgt + 1, x, w, 0.0);
                if (!st && inside_keys(E, x)) {
                    cold = first = true;
                    searched = false;
                    Tcf = x[0];
                    it = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) xt[k] = (x[k] - org[k]) * istep[k];
                } else {
                    x[0] = st ? 0.0 : -x[0];
                    ctx.put(a, x, st ? (E.backup && tgt[0] > 0.0 ? PST_BACKUP : st) : PST_OUT_OF_TABLE);
                    a = -1;
                }
            } else {
                x[0] = -Tcf;
                ctx.put(a, x, PST_FALLBACK);
                a = -1;
            }
        }
    }
}

// the general inversion as a call of its own: the lane loop keeps its registers for the table
// Newton, the common path
__device__ __noinline__ EosOut eos_invert_call(const EosDev &E, double cs2_cap, double s, const double *n,
                                               const double *guess, bool &used_table, EosWork &w)
{
    return eos_invert(E, cs2_cap, s, n, guess, used_table, w);
}

// Second half: the EoS outputs of one particle at the point g handed on by eos_find with status
// st (see there).  used_table tells whether the table produced the result.
__device__ __forceinline__ EosOut eos_finish(const EosDev &E, double cs2_cap, double s, const double *n,
                                             const double *g, uint32_t st, bool &used_table, EosWork &w)
{
    EosOut o;
    o.T = o.p = o.e = o.ps = o.cs2 = 0.0;
#pragma unroll
    for (int q = 0; q < 3; ++q) o.mu[q] = o.pn[q] = 0.0;
    o.st = st & ~kNoVerify;
    used_table = false;
    if (st & kGeneral) return eos_invert_call(E, cs2_cap, s, n, g, used_table, w);
    const long long tb = __double_as_longlong(g[0]);
    if (tb == 0) {
        if (st & PST_BACKUP) return backup_eos(E, s, n);
        return o;
    }
    double x[4], H[4][4], b[4] = {s, n[0], n[1], n[2]}, p;
    if (tb > 0) {
        used_table = true;
        double sn[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = g[k];
        tab_eval_steps(E, x, sn, H, &p);
        ++w.resid;
        long long rn = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) rn = max(rn, min(mag_bits(sn[k] - b[k]), kInfBits));
        if (!(st & kNoVerify) && rn > __double_as_longlong((E.polish ? fmin(E.tol, kPolished) : E.tol) * s))
            return eos_invert_call(E, cs2_cap, s, n, g, used_table, w);
        const double istep[4] = {E.inv_dT, E.inv_dmu[0], E.inv_dmu[1], E.inv_dmu[2]};
#pragma unroll
        for (int i = 0; i < 4; ++i)  // H^T, per unit of (T, mu)
#pragma unroll
            for (int j = i; j < 4; ++j) {
                const double t = H[i][j];
                H[i][j] = H[j][i] * istep[i];
                H[j][i] = t * istep[j];
            }
    } else {
        double sn[4];
        x[0] = -g[0];
        const double it2 = 1.0 / (x[0] * x[0]);
#pragma unroll
        for (int q = 0; q < 3; ++q) x[1 + q] = E.chi[q] > 0.0 ? n[q] / E.chi[q] * it2 : 0.0;
        an_eval(E, x[0], x + 1, p, sn, H);  // symmetric
        // an uncoupled charge direction (chi_q = 0): an identity row with zero right-hand side
#pragma unroll
        for (int q = 1; q < 4; ++q)
            if (!(E.chi[q - 1] > 0.0)) {
#pragma unroll
                for (int j = 0; j < 4; ++j) H[q][j] = H[j][q] = q == j ? 1.0 : 0.0;
                b[q] = 0.0;
            }
    }
    ++w.solve;
    if (!solve4(H, b)) {
        o.st |= PST_NOCONV;
        return o;
    }
    const double e = x[0] * s + x[1] * n[0] + x[2] * n[1] + x[3] * n[2] - p;
    double cs2 = (s * b[0] + n[0] * b[1] + n[1] * b[2] + n[2] * b[3]) / (e + p);
    if (cs2 > cs2_cap) {
        const double f = cs2_cap / cs2;
#pragma unroll
        for (int k = 0; k < 4; ++k) b[k] *= f;
        cs2 = cs2_cap;
        o.st |= PST_CS2_CAPPED;
    }
    o.T = x[0];
#pragma unroll
    for (int q = 0; q < 3; ++q) o.mu[q] = x[1 + q], o.pn[q] = b[1 + q];
    o.p = p;
    o.e = e;
    o.ps = b[0];
    o.cs2 = cs2;
    return o;
}

}  // namespace
}  // namespace sphg
