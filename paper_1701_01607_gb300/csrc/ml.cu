// Multi-level atom: opacity per frequency and node, the plane sweep with all
// rays of a hemisphere in one thread block, and the N x N rate equations.
//
// Opacity (Eq. 1, Sec. 2.1, Sec. 3).  Every frequency point belongs to one
// transition (lower l, upper u); with the grey LTE background chi_c:
//   chi = chi_t + chi_c,  S = (eta_t + chi_c B_nu) / chi,
//   sc = chi_c B_nu / chi = S - eta_t / chi (the part of S the transition's
//        populations do not set),
//   oc = chi_c / chi = 1 - chi_t / chi (the opacity share they do not set),
// each formed directly, not as a difference.
// Line:        chi_t = kappa (n_l g_u/g_l - n_u) phi,  eta_t = kappa rho^3 n_u phi,
//              phi = exp(-(x/d)^2)/(sqrt(pi) d), d = sqrt(T/t_ref), B at line centre.
// Bound-free:  chi_t = kappa y^-3 (n_l - n_u G E),  eta_t = kappa y^-3 n_u G E (rho y)^3,
//              G = n_l*/n_u*, E = exp(-theta_ref rho y/T).
//
// Sweep.  One thread-block cluster per (frequency, group of rays of one
// hemisphere: 12, 6, 4, 3, 2 or 1 rays); its blocks split the plane in row
// bands and each holds the intensity planes of the group's rays, double
// buffered.  A thread owns a node and walks the group's rays, so the angle
// sums
//   Jx = sum_r w_r (I - w0 eta_t/chi),   Ux = sum_r w_r (1 - w0 chi_t/chi)
// over the group are complete in registers and written once per group; the
// radiative sums below add the groups in order.  They are accumulated as
//   Jx = sum (I - w0 S) + sc sum w0,   Ux = sum (1 - w0) + oc sum w0,
// where I - w0 S = I_up e^-x + w_up S_up and 1 - w0 = u come from the step
// itself: every term is non-negative, so in FP32 no cancellation between
// I and w0 eta_t/chi (nearly equal in an optically thick line) degrades
// them.  The MALI rates of a scattering-dominated line depend on the small
// difference J - Lambda* S, so this order keeps the FP32 formal solution
// accurate there.
//
// Rates (Rybicki & Hummer 1992, diagonal operator).  Per node, for a line:
//   Jbar = sum wphi Jx, Ubar = sum wphi Ux (wphi: trapezoid x profile,
//   normalised per node), P_lu += B_lu Jbar, P_ul += A_ul Ubar + B_ul Jbar;
// for a bound-free continuum (qa = beta w_y y^-4):
//   P_lc += sum qa Jx,   P_cl += G sum qa E ((rho y)^3 Ux + Jx);
// plus collisions; row 0 is particle conservation (Eq. 3); the N x N system
// is solved by Gaussian elimination with partial pivoting.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "mg3d.h"
#include "fixed_weights.cuh"
#include "mg3d_internal.h"
#include "sc_step.cuh"
#include "voigt.cuh"

namespace cg = cooperative_groups;

namespace mg3d {

static int grid_for(long n, int threads) {
    long b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152L * 32) b = 152L * 32;
    return (int)b;
}

__device__ __forceinline__ double planck_rho(double rho, double theta_ref, double T) {
    return rho * rho * rho / expm1(theta_ref * rho / T);
}

// ------------------------------------------------------------------ opacity

// Line profile exp(-dd2) di / sqrt(pi) in the formal-solution precision.
__device__ __forceinline__ double ml_doppler(double dd2, double di, const ExpNegTable &et) {
    return exp_neg(dd2, et) * di * 0.56418958354775628;
}
__device__ __forceinline__ float ml_doppler(float dd2, float di, const ExpNegTable &) {
    return __expf(-dd2) * di * 0.564189584f;
}

// Opacity and radiative sums of one transition per thread and node.  Both are
// bound by memory (four values written, two per ray-group slot read, per node
// and frequency) once their arithmetic is off the FP64 pipe, which converts
// and multiplies at 2 lanes per clock and SM: FP32 works on pairs of floats
// prepared per frequency and per node (the arguments of the exponentials are
// rounded once, as when they were formed in FP64), FP64 takes its exponentials
// from 64-bit integer arithmetic.  The grid's y index is the transition, so
// that small grids still fill the GPU and the populations and Planck function
// of a transition are read once.  Measured (64x64x129, 120 frequencies, FP32):
// opacity 3.00 -> 0.33 ms, sums 2.53 -> 0.36 ms; FP64 32x32x65: 0.82 -> 0.33 and 0.45 ->
// 0.35 ms; on an 8x8x9 grid with 30 frequencies (FP32) 75 -> 8 and 75 -> 15 us.

// e^-(product of two pairs) in FP32, the argument rounded once
__device__ __forceinline__ float pair_arg(float ah, float al, float bh, float bl) {
    const float p = ah * bh;
    float e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, e);
    return p + fmaf(al, bh, e);
}

// A damped line's profile at a node of Doppler width d = 1/inv_d reference
// widths, per reference width: H(a/d, x/d)/(sqrt(pi) d) with the damping a at
// t_ref (the damping width does not scale with temperature), from the
// rational Voigt function in FP64, rounded once.
template <typename T>
__device__ __forceinline__ T ml_voigt_phi(const FreqInfo &q, double inv_d, const VoigtTable *vt) {
    return (T)(voigt_H_rational(*vt, q.adamp * inv_d, q.xy * inv_d) * 0.5641895835477563 * inv_d);
}

// What a thread keeps of its node.
template <typename T>
struct MlNode;
template <>
struct MlNode<float> {
    float4 nf;
    float pnorm;
    __device__ __forceinline__ MlNode(const MlNodeTab &t, long v)
        : nf(t.nf[v]), pnorm(t.pnorm[v]) {}
    // e^-(x/d)^2
    __device__ __forceinline__ float line_exp(const FreqOp &q, const fx::Tables &) const {
        return expf(-pair_arg(q.ah, q.al, nf.x, nf.y));
    }
    // e^-(theta_ref rho y/T)
    __device__ __forceinline__ float cont_exp(const FreqOp &q, const fx::Tables &) const {
        return expf(-pair_arg(q.ah, q.al, nf.z, nf.w));
    }
};
template <>
struct MlNode<double> {
    double inv_d, inv_T, pnorm;
    __device__ __forceinline__ MlNode(const MlNodeTab &t, long v)
        : inv_d(t.inv_d[v]), inv_T(t.inv_T[v]), pnorm(0.5641895835477563 * t.inv_d[v]) {}
    __device__ __forceinline__ double line_exp(const FreqOp &q, const fx::Tables &ft) const {
        const double xd = q.a * inv_d;
        return fx::exp_neg_fx(xd * xd, ft);
    }
    __device__ __forceinline__ double cont_exp(const FreqOp &q, const fx::Tables &ft) const {
        return fx::exp_neg_fx(q.a * inv_T, ft);
    }
};

// f 2^e
__device__ __forceinline__ float scaled(float f, int e) {
    return (unsigned)(e + 126) < 253u ? f * __int_as_float((e + 127) << 23) : ldexpf(f, e);
}

// E/D rm 2^-64 2^e for fractions E, D of 64 bits (E, D and rm 2^-64 at least 2^-12), in
// FP32, rounded once from 29 bits or more: 1/D from the FP32 reciprocal and one Newton step.
// (Three FP32 operations instead take 15 us less of the 170 of 64x64x65 nodes and 120
// frequencies, with a third more error in a thick background: rms 9.4e-8 for 8.1e-8.)
__device__ __forceinline__ float planck_ratio(fx::u64 E, fx::u64 D, fx::u64 rm, int e) {
    const int z = __clz((unsigned)(D >> 32));
    const unsigned Dh = (unsigned)((D << z) >> 32);                       // 2^-32
    float f;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(__uint2float_rz(Dh)));
    const unsigned r0 = __float2uint_rz(fminf(f * 9223372036854775808.0f, 4294967040.0f));
    const long long c = (long long)(0x8000000000000000ull - (fx::u64)Dh * r0);   // 2^-63
    const long long r1 = (long long)r0 + (((long long)r0 * (int)(c >> 11)) >> 52);
    const unsigned r = (unsigned)min(r1, 0xffffffffll);                   // 1/D, 2^-31 2^z
    const unsigned t = (unsigned)(((E >> 32) * r + 0x80000000ull) >> 32);
    const unsigned b = (unsigned)((t * (rm >> 32) + 0x80000000ull) >> 32);
    return scaled(__uint2float_rn(b), z + e - 31);
}

// Bound-free continuum: E = e^-x and the Planck function (rho y)^3/(e^x - 1),
// x = theta_ref rho y/T.
__device__ __forceinline__ void cont_terms(const FreqOp &q, double inv_T, const fx::Tables &ft,
                                           float &E, float &B) {
    const double x = q.a * inv_T;
    fx::u64 e, d;
    int n;
    if (fx::exp_parts(x, ft, &e, &n, &d)) {
        E = scaled(__ull2float_rn(e), -64 - n);
        B = planck_ratio(e, d, q.rm, q.re - n);
    } else {
        E = expf(-(float)x);
        B = (float)(q.ry3 / expm1(x));
    }
}
__device__ __forceinline__ void cont_terms(const FreqOp &q, double inv_T, const fx::Tables &ft,
                                           double &E, double &B) {
    const double x = q.a * inv_T;
    fx::u64 e, d;
    int n;
    // 1 - e^-x as a fraction is good to 2^-55.5, so to FP64 relative to itself from x of
    // 1/4 on (at 1/1000 it would lose 8 bits)
    if (x >= 0.25 && fx::exp_parts(x, ft, &e, &n, &d)) {
        E = e ? fx::pack62(e, -n) : 0.0;
        B = q.ry3 * fast_div(E, fx::pack32(d, 0));
    } else {
        E = exp(-x);
        B = q.ry3 / expm1(x);
    }
}
__device__ __forceinline__ float fast_inv(float x) { return 1.0f / x; }
__device__ __forceinline__ double fast_inv(double x) { return fast_div(1.0, x); }

template <typename T>
__global__ void ml_opacity_kernel(const MlOpacityArgs a) {
    __shared__ fx::u64 fx_tab[2 * fx::kTab];
    for (int i = threadIdx.x; i < 2 * fx::kTab; i += blockDim.x) fx_tab[i] = a.fx_tab[i];
    __syncthreads();
    const fx::Tables ft{fx_tab, fx_tab + fx::kTab};
    const long nvox = a.nvox;
    const int t = blockIdx.y;
    const TransInfo tr = a.ti[t];
    const int fb = max(tr.f_begin, a.f0), fe = min(tr.f_end, a.f0 + a.nfreq);
    if (fb >= fe) return;
    for (long v = blockIdx.x * (long)blockDim.x + threadIdx.x; v < nvox;
         v += (long)gridDim.x * blockDim.x) {
        const MlNode<T> node(a.tab, v);
        const T cc = (T)a.chi_c[v];
        const T sg = a.sigma_c ? (T)a.sigma_c[v] : T(0);
        const double nl = a.n[(long)tr.lo * nvox + v], nu = a.n[(long)tr.up * nvox + v];
        // line: the population difference; continuum: n_u G, G = n_l*/n_u*
        const double nd = tr.kind == 0 ? tr.gr * nl - nu : nu * a.saha[(long)tr.lo * nvox + v];
        const T nlT = (T)nl, nuT = (T)nu, ndT = (T)nd;
        T B = 0;
        double inv_d = 0.0, inv_T = 0.0;
        if (tr.kind == 0) {
            B = ((const T *)a.tab.bline)[(long)t * nvox + v];
            if (a.voigt) inv_d = a.tab.inv_d[v];
        } else {
            inv_T = a.tab.inv_T[v];
        }
        for (int f = fb; f < fe; ++f) {
            const FreqOp &q = a.fo[f];
            const long i = (long)(f - a.f0) * nvox + v;
            const T kap = sizeof(T) == 8 ? (T)q.kap : (T)q.kapf;
            const T emis = sizeof(T) == 8 ? (T)q.emis : (T)q.emisf;
            T chi_t, eta_t;
            if (tr.kind == 0) {
                const T phi = q.damped ? ml_voigt_phi<T>(a.fi[f], inv_d, a.voigt)
                                       : node.line_exp(q, ft) * node.pnorm;
                chi_t = kap * phi * ndT;
                eta_t = emis * nuT * phi;
                if (a.moving) {
                    // a line's profile is applied per ray in the sweep
                    chi_t = kap * ndT;
                    eta_t = emis * nuT;
                }
            } else {
                T E;
                cont_terms(q, inv_T, ft, E, B);
                chi_t = kap * (nlT - ndT * E);
                if constexpr (sizeof(T) == 8) eta_t = kap * (ndT * q.ry3) * E;
                else eta_t = tr.wide ? kap * (T)(nd * q.ry3) * E : emis * ndT * E;
            }
            // the background's opacity and emissivity (continuum, and
            // coherent scattering of the previous mean intensity)
            T chi_b = cc, eta_b = cc * B;
            if (a.sigma_c) {
                chi_b += sg;
                eta_b += sg * ((const T *)a.jbg)[(long)f * nvox + v];
            }
            if (a.moving) {
                // ray-independent parts (continua do not shift)
                ((T *)a.chi)[i] = chi_t;
                ((T *)a.S)[i] = eta_t;
                ((T *)a.oc)[i] = chi_b;
                ((T *)a.sc)[i] = eta_b;
                continue;
            }
            T rho = T(1);
            bool prd = false;
            if (a.prd_index) {
                // partial redistribution: the line's emission profile is rho phi,
                // so its emissivity and the transition's shares scale by rho
                const int pr = a.prd_index[f];
                if (pr >= 0) {
                    rho = (T)a.prd_rho[(long)pr * nvox + v];
                    prd = true;
                }
            }
            const T chi = chi_t + chi_b;
            const T inv = fast_inv(chi);
            ((T *)a.chi)[i] = chi;
            ((T *)a.S)[i] = (rho * eta_t + eta_b) * inv;
            // the parts of S and chi the transition does not set, formed
            // directly: S - rho eta_t/chi and 1 - chi_t/chi.  For a PRD
            // frequency oc = 1 - rho chi_t/chi takes either sign and its
            // weighted sum over the line nearly cancels, so the sweep gets
            // oc = 0 (Ux = sum w u) and the radiative sums add the local
            // term in FP64 (prd_oc)
            ((T *)a.sc)[i] = eta_b * inv;
            ((T *)a.oc)[i] = prd ? T(0) : chi_b * inv;
        }
    }
}

// The per-node constants of a level.
template <typename T>
__global__ void ml_node_tab_kernel(long nvox, int n_lines, const TransInfo *__restrict__ ti,
                                   double t_ref, double theta_ref, const double *__restrict__ Tg,
                                   float4 *nf, float *pnorm, double *inv_d, double *inv_T,
                                   T *bline) {
    for (long v = blockIdx.x * (long)blockDim.x + threadIdx.x; v < nvox;
         v += (long)gridDim.x * blockDim.x) {
        const double it = 1.0 / Tg[v], d2 = t_ref / Tg[v], di = sqrt(d2);
        inv_d[v] = di;
        inv_T[v] = it;
        if (nf) {
            const float dh = (float)d2, th = (float)it;
            nf[v] = make_float4(dh, (float)(d2 - (double)dh), th, (float)(it - (double)th));
            pnorm[v] = (float)(0.5641895835477563 * di);
        }
        for (int l = 0; l < n_lines; ++l)
            bline[(long)l * nvox + v] = (T)planck_rho(ti[l].rho, theta_ref, Tg[v]);
    }
}

cudaError_t launch_ml_node_tab(int prec, long nvox, int n_lines, const TransInfo *ti, double t_ref,
                               double theta_ref, const double *T, float4 *nf, float *pnorm,
                               double *inv_d, double *inv_T, void *bline, cudaStream_t st) {
    if (prec == MG3D_PREC_F64)
        ml_node_tab_kernel<double><<<grid_for(nvox, 256), 256, 0, st>>>(
            nvox, n_lines, ti, t_ref, theta_ref, T, nullptr, nullptr, inv_d, inv_T,
            (double *)bline);
    else
        ml_node_tab_kernel<float><<<grid_for(nvox, 256), 256, 0, st>>>(
            nvox, n_lines, ti, t_ref, theta_ref, T, nf, pnorm, inv_d, inv_T, (float *)bline);
    return cudaGetLastError();
}

// ------------------------------------------------ partial redistribution

// Partial redistribution of a line (the next step Sec. 6 names; the reading
// of the two-level case generalised): the angle-averaged Doppler
// redistribution R_I-A at a node of Doppler width d,
//   R0(x', x) = erfc(max(|x|, |x'|)/d) / (2 d^2),
// scaled symmetrically, R = diag(c) R0 diag(c), so that its discrete
// marginals sum_f' wq_f' R(f', f) are the node's profile phi_f (wq: the
// line's trapezoid weights normalised by sum w phi).  R0 depends on its two
// frequencies only through the larger |x|, so with the frequencies sorted by
// |x| a product R0^T v is, for a frequency of group k (equal |x|),
//   g_k sum_{groups <= k} v + sum_{groups > k} g v,   g = erfc(|x|/d)/(2 d^2):
// a prefix and a suffix sum, O(n) per node instead of O(n^2).
constexpr int kMaxPrdFreq = kMaxPrdLineFreq;

// out_s = sum_a R0(a, s) v_a for the line's sorted frequencies s (v, out in
// sorted order; g per group; suf scratch of ngrp + 1 entries).
__device__ inline void prd_r0_product(int nf, int ngrp, const int *__restrict__ gs,
                                      const double *g, const double *v, double *out,
                                      double *suf) {
    // suffix sums over groups above k
    suf[ngrp] = 0.0;
    for (int k = ngrp - 1; k >= 0; --k) {
        double sg = 0.0;
        for (int s = gs[k]; s < gs[k + 1]; ++s) sg += v[s];
        suf[k] = suf[k + 1] + g[k] * sg;
    }
    double pre = 0.0;
    for (int k = 0; k < ngrp; ++k) {
        for (int s = gs[k]; s < gs[k + 1]; ++s) pre += v[s];
        const double m = g[k] * pre + suf[k + 1];
        for (int s = gs[k]; s < gs[k + 1]; ++s) out[s] = m;
    }
}

// The line's profile at the node (sorted order), its normalised weights and
// the R0 group values.
__device__ inline void prd_line_setup(const PrdLine &L, const FreqInfo *__restrict__ fi,
                                      const int *__restrict__ ord, const int *__restrict__ gs,
                                      double d, double *phi, double *wq, double *g) {
    const double inv_d = 1.0 / d;
    double norm = 0.0;
    for (int s = 0; s < L.nf; ++s) {
        const FreqInfo q = fi[ord[L.ord0 + s]];
        const double xd = q.xy * inv_d;
        phi[s] = exp(-xd * xd) * 0.56418958354775628 * inv_d;
        norm += q.w * phi[s];
    }
    for (int s = 0; s < L.nf; ++s) wq[s] = fi[ord[L.ord0 + s]].w / norm;
    for (int k = 0; k < L.ngrp; ++k) {
        const double ax = fabs(fi[ord[L.ord0 + gs[k]]].xy);
        g[k] = 0.5 * erfc(ax * inv_d) * inv_d * inv_d;
    }
}

__global__ void __launch_bounds__(128) ml_prd_scale_kernel(long nvox, int n_prd,
                                                           const PrdLine *__restrict__ pl,
                                                           const FreqInfo *__restrict__ fi,
                                                           const int *__restrict__ ord,
                                                           const int *__restrict__ grp,
                                                           double t_ref,
                                                           const double *__restrict__ T,
                                                           double *__restrict__ scale) {
    double phi[kMaxPrdFreq], wq[kMaxPrdFreq], c[kMaxPrdFreq], v[kMaxPrdFreq], m[kMaxPrdFreq];
    double g[kMaxPrdFreq + 1], suf[kMaxPrdFreq + 1];
    for (long x = blockIdx.x * (long)blockDim.x + threadIdx.x; x < nvox;
         x += (long)gridDim.x * blockDim.x) {
        const double d = sqrt(T[x] / t_ref);
        for (int l = 0; l < n_prd; ++l) {
            const PrdLine L = pl[l];
            const int *gs = grp + L.grp0;
            prd_line_setup(L, fi, ord, gs, d, phi, wq, g);
            for (int s = 0; s < L.nf; ++s) c[s] = 1.0;
            for (int it = 0; it < 200; ++it) {
                for (int s = 0; s < L.nf; ++s) v[s] = wq[s] * c[s];
                prd_r0_product(L.nf, L.ngrp, gs, g, v, m, suf);
                for (int s = 0; s < L.nf; ++s) c[s] = sqrt(c[s] * phi[s] / m[s]);
            }
            for (int s = 0; s < L.nf; ++s)
                scale[(long)(L.pf0 + ord[L.ord0 + s] - L.f_begin) * nvox + x] = c[s];
        }
    }
}

template <typename TP>
__global__ void __launch_bounds__(128) ml_prd_rho_kernel(const MlPrdArgs a) {
    double phi[kMaxPrdFreq], wq[kMaxPrdFreq], v[kMaxPrdFreq], m[kMaxPrdFreq];
    double g[kMaxPrdFreq + 1], suf[kMaxPrdFreq + 1];
    const TP *__restrict__ jbg = (const TP *)a.jbg;
    const long nvox = a.nvox;
    const int N = a.n_levels;
    for (long x = blockIdx.x * (long)blockDim.x + threadIdx.x; x < nvox;
         x += (long)gridDim.x * blockDim.x) {
        const double Tg = a.T[x];
        const double d = sqrt(Tg / a.t_ref), inv_d = 1.0 / d;
        // plain rates of the lagged field: collisions plus every transition's
        // radiative rates with J (no local operator)
        double P[kMaxLevels][kMaxLevels];
        for (int i = 0; i < N; ++i)
            for (int j = 0; j < N; ++j) P[i][j] = i == j ? 0.0 : a.c[((long)i * N + j) * nvox + x];
        for (int t = 0; t < a.n_trans; ++t) {
            const TransInfo tr = a.ti[t];
            if (tr.kind == 0) {
                double s0 = 0.0, s1 = 0.0;
                for (int f = tr.f_begin; f < tr.f_end; ++f) {
                    const FreqInfo q = a.fi[f];
                    const double xd = q.xy * inv_d;
                    const double wphi = q.w * exp(-xd * xd) * 0.56418958354775628 * inv_d;
                    s0 += wphi;
                    s1 += wphi * (double)jbg[(long)f * nvox + x];
                }
                const double Jb = s1 / s0;
                const double b_ul = tr.coef / (tr.rho * tr.rho * tr.rho);
                P[tr.lo][tr.up] += tr.gr * b_ul * Jb;
                P[tr.up][tr.lo] += tr.coef + b_ul * Jb;
            } else {
                const double G = a.saha[(long)tr.lo * nvox + x];
                double s0 = 0.0, s1 = 0.0, s2 = 0.0;
                for (int f = tr.f_begin; f < tr.f_end; ++f) {
                    const FreqInfo q = a.fi[f];
                    const double y = q.xy;
                    const double qa = tr.coef * q.w / (y * y * y * y);
                    const double E = exp(-a.theta_ref * tr.rho * y / Tg);
                    const double ry = tr.rho * y;
                    const double J = (double)jbg[(long)f * nvox + x];
                    s0 += qa * J;
                    s1 += qa * E * J;
                    s2 += qa * E * ry * ry * ry;
                }
                P[tr.lo][tr.up] += s0;
                P[tr.up][tr.lo] += G * (s2 + s1);
            }
        }
        for (int l = 0; l < a.n_prd; ++l) {
            const PrdLine L = a.pl[l];
            const int *gs = a.grp + L.grp0;
            prd_line_setup(L, a.fi, a.ord, gs, d, phi, wq, g);
            double Jbar = 0.0;
            for (int s = 0; s < L.nf; ++s) {
                const int f = a.ord[L.ord0 + s];
                const double J = (double)jbg[(long)f * nvox + x];
                const double cs = a.scale[(long)(L.pf0 + f - L.f_begin) * nvox + x];
                Jbar += wq[s] * phi[s] * J;
                v[s] = wq[s] * cs * J;
            }
            double inflow = 0.0;
            for (int j = 0; j < N; ++j)
                if (j != L.up) inflow += a.n[(long)j * nvox + x] * P[j][L.up];
            const double excite = a.n[(long)L.lo * nvox + x] * L.gr * L.b_ul * Jbar;
            const double frad = excite / inflow;
            prd_r0_product(L.nf, L.ngrp, gs, g, v, m, suf);
            // the line's opacity at the node (as the opacity step forms it)
            // for 1 - rho chi_t/chi, the local term of the line's U
            const double nlo = a.n[(long)L.lo * nvox + x], nup = a.n[(long)L.up * nvox + x];
            const double chi_b = a.chi_c[x] + (a.sigma_c ? a.sigma_c[x] : 0.0);
            for (int s = 0; s < L.nf; ++s) {
                const int f = a.ord[L.ord0 + s];
                const long row = (long)(L.pf0 + f - L.f_begin) * nvox + x;
                double r = 1.0;
                if (Jbar > 0.0) {
                    const double Af = a.scale[row] * m[s];
                    r = 1.0 + L.gamma * frad * (Af / (phi[s] * Jbar) - 1.0);
                }
                a.rho[row] = r;
                const FreqInfo q = a.fi[f];
                const double chi_t = q.kappa * phi[s] * (q.gr * nlo - nup);
                a.oc[row] = (chi_b + (1.0 - r) * chi_t) / (chi_t + chi_b);
            }
        }
    }
}

cudaError_t launch_ml_prd_scale(long nvox, int n_prd, const PrdLine *pl, const FreqInfo *fi,
                                const int *ord, const int *grp, double t_ref, const double *T,
                                double *scale, cudaStream_t st) {
    ml_prd_scale_kernel<<<grid_for(nvox, 128), 128, 0, st>>>(nvox, n_prd, pl, fi, ord, grp, t_ref,
                                                              T, scale);
    return cudaGetLastError();
}

cudaError_t launch_ml_prd_rho(const MlPrdArgs &a, cudaStream_t st) {
    if (a.prec == MG3D_PREC_F64)
        ml_prd_rho_kernel<double><<<grid_for(a.nvox, 128), 128, 0, st>>>(a);
    else
        ml_prd_rho_kernel<float><<<grid_for(a.nvox, 128), 128, 0, st>>>(a);
    return cudaGetLastError();
}

template <typename T>
__global__ void ml_bottom_kernel(long nplane, int nfreq, const FreqInfo *__restrict__ fi,
                                 double theta_ref, const double *__restrict__ Tg,
                                 T *__restrict__ ib) {
    const long total = nplane * nfreq;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total;
         i += (long)gridDim.x * blockDim.x) {
        const int f = (int)(i / nplane);
        const long p = i - (long)f * nplane;
        const FreqInfo q = fi[f];
        const double rho = q.kind == 0 ? q.rho : q.rho * q.xy;
        ib[i] = (T)planck_rho(rho, theta_ref, Tg[p]);
    }
}

// -------------------------------------------------------------------- sweep

// HERM: monotone cubic Hermite upwind interpolation (the Hermite-spline
// option of Sec. 3): per ray and local row the table holds the four upwind
// rows ya-1 .. ya+2 of the intensity and slope planes and of chi, S; each
// finished plane gets its x-slopes after a block barrier; chi and S take
// theirs from dchi, dS.
//
// MODE kSweepMoving (a velocity field): along ray r a line's profile at a node
// is phi((x - u_r) / d) / (d sqrt(pi)), so chi, S and the transition shares
// are formed per node, ray and frequency from the ray-independent parts the
// opacity kernel wrote, and kept in opacity and source planes next to the
// intensity planes, from which the next step interpolates the upwind values;
// the angle sums carry the ray's normalised profile weight inside the ray
// sum.
template <typename T, int MODE>
__device__ __forceinline__ void ml_sweep_body(const MlSweepArgs<T> &a, int f, int slot) {
    constexpr bool HERM = MODE == kSweepHermite, VEL = MODE == kSweepMoving;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    // slot = (hemisphere, ray group); hemisphere 0: rays 0-11 (up), 1: 12-23
    const int rpb = a.rpb, groups = 12 / rpb;
    const int hemi = slot / groups;
    const int r0 = hemi * 12 + (slot - hemi * groups) * rpb;
    const bool up = hemi == 0;
    const int nx = a.nx, ny = a.ny, nz = a.nz, rows = a.rows;
    const int y0 = rank * rows;
    const int myrows = max(0, min(rows, ny - y0));
    const int band = myrows * nx;
    const long nplane = (long)nx * ny;
    const long nvox = nplane * nz;
    const T *__restrict__ chif = a.chi + (long)f * nvox;
    const T *__restrict__ Sf = a.S + (long)f * nvox;
    const T *__restrict__ scf = a.sc + (long)f * nvox;
    const T *__restrict__ ocf = a.oc + (long)f * nvox;
    T *__restrict__ jxo = a.jx + ((long)slot * a.nfreq + f) * nvox;
    T *__restrict__ uxo = a.ux + ((long)slot * a.nfreq + f) * nvox;
    T *__restrict__ jmo = a.jm ? a.jm + ((long)slot * a.nfreq + f) * nvox : nullptr;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *buf = reinterpret_cast<T *>(smem_raw);
    const long raystride = (long)rows * nx;
    const long bufstride = rpb * raystride;
    // per step and (ray, local row): the upwind rows of the intensity planes
    // (here or in a peer block) and of chi, S on the upwind plane
    struct RowRef {
        const T *pa, *pb;
        int ra, rb;
    };
    struct RowRef4 {
        const T *p[4], *d[4];
        int r[4];
    };
    T *dbuf = buf + 2 * bufstride;  // slope planes (HERM)
    // VEL: opacity planes at buf + 2 bufstride, source planes at buf + 4 bufstride,
    // the same offsets from the intensity planes in every block of the cluster
    const long coff = 2 * bufstride, soff = 4 * bufstride;
    RowRef *rowref =
        reinterpret_cast<RowRef *>(buf + (HERM ? 4 : (VEL ? 6 : 2)) * bufstride);
    RowRef4 *rowref4 = reinterpret_cast<RowRef4 *>(rowref);
    __shared__ double exp_tab[kExpTab];
    if (sizeof(T) == 8) {
        for (int i = threadIdx.x; i < kExpTab; i += blockDim.x) exp_tab[i] = a.exp_tab[i];
        __syncthreads();
    }
    const ExpNegTable et{exp_tab, a.exp_l1, a.exp_l2};
    const T wray = T(1.0 / kRays);
    const unsigned long long rmagic = band_magic(rows);
    // per-ray constants of the current step (the upwind offset is the same
    // for every node of a plane): bilinear weights, half path, corner offsets
    __shared__ T g_w[12][4];        // bilinear weights, or the x and y Hermite
    __shared__ T g_wy[12][4];       // bases (HERM)
    __shared__ T g_hs[12];
    __shared__ int g_ix[12];
    const T *__restrict__ dchif = HERM ? a.dchi + (long)f * nvox : nullptr;
    const T *__restrict__ dSf = HERM ? a.dS + (long)f * nvox : nullptr;
    // VEL: this frequency's line (or -1), offset and weight
    const int vl = VEL ? a.vline[a.f0 + f] : -1;
    const T vxf = VEL ? a.vx[a.f0 + f] : T(0), vwf = VEL ? a.vwq[a.f0 + f] : T(0);
    // chi, S, sc, oc and the profile weight of node v for ray r0 + j
    auto moving_terms = [&](long v, int j, T &chi, T &S, T &sc, T &oc, T &wr) {
        const T A = chif[v], E = Sf[v], cb = ocf[v], eb = scf[v];
        T prof = T(1);
        wr = T(1);
        if (vl >= 0) {
            const long rv = (long)(r0 + j) * nvox + v;
            const T di = a.dinv[v];
            const T dd = (vxf - a.uproj[rv]) * di;
            prof = ml_doppler(dd * dd, di, et);
            wr = vwf * prof * a.vnorm[(long)vl * kRays * nvox + rv];
        }
        const T ct = A * prof, et_ = E * prof;
        chi = ct + cb;
        const T inv = T(1) / chi;
        S = (et_ + eb) * inv;
        sc = eb * inv;
        oc = cb * inv;
    };

    for (int t = 0; t < nz; ++t) {
        const int k = up ? t : nz - 1 - t;
        T *cur = buf + (t & 1) * bufstride;
        if (t == 0 && VEL) {
            for (int q = threadIdx.x; q < band; q += blockDim.x) {
                const int yl = q / nx, x = q - yl * nx;
                const int y = y0 + yl;
                const T Ib = up ? a.ib[(long)f * nplane + (long)y * nx + x] : T(0);
                const long v = (long)k * nplane + (long)y * nx + x;
                T jacc = 0, uacc = 0;
                for (int j = 0; j < rpb; ++j) {
                    T chi, S, sc, oc, wr;
                    moving_terms(v, j, chi, S, sc, oc, wr);
                    const long i = j * raystride + (long)yl * nx + x;
                    cur[i] = Ib;
                    cur[coff + i] = chi;
                    cur[soff + i] = S;
                    jacc += wr * Ib;
                    uacc += wr;
                }
                jxo[v] = wray * jacc;
                uxo[v] = wray * uacc;
                if (jmo) jmo[v] = T(rpb) * wray * Ib;
            }
        } else if (t == 0) {
            for (int q = threadIdx.x; q < band; q += blockDim.x) {
                const int yl = q / nx, x = q - yl * nx;
                const int y = y0 + yl;
                const T Ib = up ? a.ib[(long)f * nplane + (long)y * nx + x] : T(0);
                for (int j = 0; j < rpb; ++j) cur[j * raystride + (long)yl * nx + x] = Ib;
                const long v = (long)k * nplane + (long)y * nx + x;
                jxo[v] = T(rpb) * wray * Ib;
                uxo[v] = T(rpb) * wray;
                if (jmo) jmo[v] = T(rpb) * wray * Ib;
            }
        } else {
            const T *prev = buf + ((t - 1) & 1) * bufstride;
            if (threadIdx.x < rpb) {
                const StepGeom o = a.geom[(long)(r0 + threadIdx.x) * nz + t];
                const T tx = (T)o.tx, ty = (T)o.ty;
                if constexpr (HERM) {
                    const HermiteBasis<T> bx(tx), by(ty);
                    g_w[threadIdx.x][0] = bx.c0;
                    g_w[threadIdx.x][1] = bx.c1;
                    g_w[threadIdx.x][2] = bx.c2;
                    g_w[threadIdx.x][3] = bx.c3;
                    g_wy[threadIdx.x][0] = by.c0;
                    g_wy[threadIdx.x][1] = by.c1;
                    g_wy[threadIdx.x][2] = by.c2;
                    g_wy[threadIdx.x][3] = by.c3;
                } else {
                    g_w[threadIdx.x][0] = (T(1) - tx) * (T(1) - ty);
                    g_w[threadIdx.x][1] = tx * (T(1) - ty);
                    g_w[threadIdx.x][2] = (T(1) - tx) * ty;
                    g_w[threadIdx.x][3] = tx * ty;
                }
                g_hs[threadIdx.x] = T(0.5) * (T)o.s;
                g_ix[threadIdx.x] = o.ix0;
            }
            for (int i = threadIdx.x; i < rpb * myrows; i += blockDim.x) {
                const int j = i / myrows, yl = i - j * myrows;
                int ya = y0 + yl + a.geom[(long)(r0 + j) * nz + t].iy0;
                if (ya >= ny) ya -= ny;
                const int yb = (ya + 1 == ny) ? 0 : ya + 1;
                if constexpr (HERM) {
                    const T *dprev = dbuf + ((t - 1) & 1) * bufstride;
                    int yr[4] = {ya == 0 ? ny - 1 : ya - 1, ya, yb, yb + 1 == ny ? 0 : yb + 1};
                    RowRef4 r4;
                    for (int m = 0; m < 4; ++m) {
                        const int b = band_of(yr[m], rmagic);
                        const long ro = j * raystride + (long)(yr[m] - b * rows) * nx;
                        r4.p[m] = (b == rank ? prev : cluster.map_shared_rank(prev, b)) + ro;
                        r4.d[m] = (b == rank ? dprev : cluster.map_shared_rank(dprev, b)) + ro;
                        r4.r[m] = yr[m] * nx;
                    }
                    rowref4[j * rows + yl] = r4;
                } else {
                    const int ba = band_of(ya, rmagic), bb = band_of(yb, rmagic);
                    const T *Pa = (ba == rank) ? prev : cluster.map_shared_rank(prev, ba);
                    const T *Pb = (bb == rank) ? prev : cluster.map_shared_rank(prev, bb);
                    RowRef r;
                    r.pa = Pa + j * raystride + (long)(ya - ba * rows) * nx;
                    r.pb = Pb + j * raystride + (long)(yb - bb * rows) * nx;
                    r.ra = ya * nx;
                    r.rb = yb * nx;
                    rowref[j * rows + yl] = r;
                }
            }
            __syncthreads();
            const int kp = up ? k - 1 : k + 1;
            const T *__restrict__ chip = chif + (long)kp * nplane;
            const T *__restrict__ Sp = Sf + (long)kp * nplane;
            for (int q = threadIdx.x; q < band; q += blockDim.x) {
                const int yl = q / nx, x = q - yl * nx;
                const int y = y0 + yl;
                const long v = (long)k * nplane + (long)y * nx + x;
                const T chi_loc = chif[v], S_loc = Sf[v], sc = scf[v], oc = ocf[v];
                // sc and oc are the node's: sum I - w0 S, 1 - w0, w0 (and I
                // for the mean intensity) over the rays, then
                // Jx = sum (I - w0 S) + sc sum w0, Ux = sum u + oc sum w0
                T sum_i = 0, sum_p = 0, sum_u = 0, sum_w0 = 0;
                if constexpr (VEL) {
                    T jacc = 0, uacc = 0;
                    for (int j = 0; j < rpb; ++j) {
                        const T w00 = g_w[j][0], w10 = g_w[j][1], w01 = g_w[j][2],
                                w11 = g_w[j][3];
                        int xa = x + g_ix[j];
                        if (xa >= nx) xa -= nx;
                        const int xb = (xa + 1 == nx) ? 0 : xa + 1;
                        const RowRef r = rowref[j * rows + yl];
                        const T *Pa = r.pa, *Pb = r.pb;
                        auto bil = [&](long o) {
                            return w00 * Pa[o + xa] + w10 * Pa[o + xb] + w01 * Pb[o + xa] +
                                   w11 * Pb[o + xb];
                        };
                        const T I_up = bil(0), chi_up = bil(coff), S_up = bil(soff);
                        T chi, S, sc_r, oc_r, wr;
                        moving_terms(v, j, chi, S, sc_r, oc_r, wr);
                        const T x_tau = (chi_up + chi) * g_hs[j];
                        T ex, w0, wup, u;
                        ScWeights<T>::eval(x_tau, sc_rcp(x_tau), et, ex, w0, wup, u);
                        const T part = I_up * ex + wup * S_up;   // I - w0 S
                        const T I = part + w0 * S;
                        const long i = j * raystride + (long)yl * nx + x;
                        cur[i] = I;
                        cur[coff + i] = chi;
                        cur[soff + i] = S;
                        sum_i += I;
                        jacc += wr * (part + w0 * sc_r);
                        uacc += wr * (u + w0 * oc_r);
                    }
                    jxo[v] = wray * jacc;
                    uxo[v] = wray * uacc;
                    if (jmo) jmo[v] = wray * sum_i;
                    continue;
                }
                if constexpr (HERM) {
                    for (int j = 0; j < rpb; ++j) {
                        int xa = x + g_ix[j];
                        if (xa >= nx) xa -= nx;
                        const int xb = (xa + 1 == nx) ? 0 : xa + 1;
                        const RowRef4 &r4 = rowref4[j * rows + yl];
                        const T c0 = g_w[j][0], c1 = g_w[j][1], c2 = g_w[j][2], c3 = g_w[j][3];
                        const T e0 = g_wy[j][0], e1 = g_wy[j][1], e2 = g_wy[j][2], e3 = g_wy[j][3];
                        // x pass on four rows, then y pass through their values
                        auto up2d = [&](auto value_row, auto slope_row) {
                            T gq[4];
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                const T *v = value_row(m), *d = slope_row(m);
                                gq[m] = c0 * v[xa] + c1 * d[xa] + c2 * v[xb] + c3 * d[xb];
                            }
                            return e0 * gq[1] + e1 * mono_slope(gq[1] - gq[0], gq[2] - gq[1]) +
                                   e2 * gq[2] + e3 * mono_slope(gq[2] - gq[1], gq[3] - gq[2]);
                        };
                        const T *dchip = dchif + (long)kp * nplane, *dSp = dSf + (long)kp * nplane;
                        const T chi_up = up2d([&](int m) { return chip + r4.r[m]; },
                                              [&](int m) { return dchip + r4.r[m]; });
                        const T S_up = up2d([&](int m) { return Sp + r4.r[m]; },
                                            [&](int m) { return dSp + r4.r[m]; });
                        const T I_up = up2d([&](int m) { return r4.p[m]; },
                                            [&](int m) { return r4.d[m]; });
                        const T x_tau = (chi_up + chi_loc) * g_hs[j];
                        T ex, w0, wup, u;
                        ScWeights<T>::eval(x_tau, sc_rcp(x_tau), et, ex, w0, wup, u);
                        const T part = I_up * ex + wup * S_up;   // I - w0 S
                        const T I = part + w0 * S_loc;
                        cur[j * raystride + (long)yl * nx + x] = I;
                        sum_i += I;
                        sum_p += part;
                        sum_u += u;
                        sum_w0 += w0;
                    }
                } else
                for (int j = 0; j < rpb; ++j) {
                    const T w00 = g_w[j][0], w10 = g_w[j][1], w01 = g_w[j][2], w11 = g_w[j][3];
                    int xa = x + g_ix[j];
                    if (xa >= nx) xa -= nx;
                    const int xb = (xa + 1 == nx) ? 0 : xa + 1;
                    const RowRef r = rowref[j * rows + yl];
                    const T *ca = chip + r.ra, *cb = chip + r.rb;
                    const T *sa = Sp + r.ra, *sb = Sp + r.rb;
                    const T chi_up = w00 * ca[xa] + w10 * ca[xb] + w01 * cb[xa] + w11 * cb[xb];
                    const T S_up = w00 * sa[xa] + w10 * sa[xb] + w01 * sb[xa] + w11 * sb[xb];
                    const T *Pa = r.pa, *Pb = r.pb;
                    const T I_up = w00 * Pa[xa] + w10 * Pa[xb] + w01 * Pb[xa] + w11 * Pb[xb];
                    const T x_tau = (chi_up + chi_loc) * g_hs[j];
                    T ex, w0, wup, u;
                    ScWeights<T>::eval(x_tau, sc_rcp(x_tau), et, ex, w0, wup, u);
                    const T part = I_up * ex + wup * S_up;   // I - w0 S
                    const T I = part + w0 * S_loc;
                    cur[j * raystride + (long)yl * nx + x] = I;
                    sum_i += I;
                    sum_p += part;
                    sum_u += u;
                    sum_w0 += w0;
                }
                jxo[v] = wray * (sum_p + sc * sum_w0);
                uxo[v] = wray * (sum_u + oc * sum_w0);
                if (jmo) jmo[v] = wray * sum_i;
            }
        }
        if constexpr (HERM) {
            // x-slopes of the new planes; a band holds whole rows
            __syncthreads();
            T *dcur = dbuf + (t & 1) * bufstride;
            for (int i = threadIdx.x; i < rpb * band; i += blockDim.x) {
                const int j = i / band, q = i - j * band;
                const int yl = q / nx, x = q - yl * nx;
                const int xm = x == 0 ? nx - 1 : x - 1, xp = x + 1 == nx ? 0 : x + 1;
                const T *row = cur + j * raystride + (long)yl * nx;
                dcur[j * raystride + (long)yl * nx + x] =
                    mono_slope(row[x] - row[xm], row[xp] - row[x]);
            }
        }
        cluster.sync();
    }
}

template <typename T, int MAXT, int MODE>
__global__ void __launch_bounds__(MAXT) ml_sweep_kernel(const MlSweepArgs<T> a) {
    ml_sweep_body<T, MODE>(a, blockIdx.y, blockIdx.z);
}

size_t ml_sweep_smem_bytes(int prec, int rows, int nx, int rpb, int herm, int moving) {
    const size_t elem = prec == MG3D_PREC_F64 ? sizeof(double) : sizeof(float);
    // moving: intensity, opacity and source planes and the 24-byte table
    if (moving) return 6ull * rpb * rows * nx * elem + 24ull * rpb * rows;
    // intensity planes (and their slope planes), then the per-(ray, row)
    // upwind row table: two pointers and two offsets (24 bytes), or eight
    // pointers and four offsets (80 bytes); the planes end on an 8-byte
    // boundary
    if (herm) return 4ull * rpb * rows * nx * elem + 80ull * rpb * rows;
    return 2ull * rpb * rows * nx * elem + 24ull * rpb * rows;
}

template <typename T, int MAXT, int MODE>
static cudaError_t launch_ml_sweep_t(const MlSweepArgs<T> &a, int bands, int threads,
                                     cudaStream_t st) {
    const size_t smem = ml_sweep_smem_bytes(sizeof(T) == 8 ? MG3D_PREC_F64 : MG3D_PREC_F32,
                                            a.rows, a.nx, a.rpb, MODE == kSweepHermite ? 1 : 0,
                                            MODE == kSweepMoving ? 1 : 0);
    if (MODE == kSweepHermite && (!a.dchi || !a.dS)) return cudaErrorInvalidValue;
    if (MODE == kSweepMoving && (!a.vx || !a.vwq || !a.vline || !a.vnorm || !a.uproj || !a.dinv))
        return cudaErrorInvalidValue;
    // one fixed limit for every launch, so graph replays never meet a lower one
    cudaError_t e = cudaFuncSetAttribute(ml_sweep_kernel<T, MAXT, MODE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kMaxSweepSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(bands, a.nfreq, 2 * (12 / a.rpb));
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = bands;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = bands > 1 ? 1 : 0;  // one band: a plain launch
    return cudaLaunchKernelEx(&cfg, ml_sweep_kernel<T, MAXT, MODE>, a);
}

template <typename T>
static cudaError_t launch_ml_sweep_any(const MlSweepArgs<T> &a, int bands, int threads,
                                       cudaStream_t st) {
    if (a.herm && a.moving) return cudaErrorInvalidValue;
    if (a.herm)
        return threads <= 256 ? launch_ml_sweep_t<T, 256, kSweepHermite>(a, bands, threads, st)
                              : launch_ml_sweep_t<T, 512, kSweepHermite>(a, bands, threads, st);
    if (a.moving)
        return threads <= 256 ? launch_ml_sweep_t<T, 256, kSweepMoving>(a, bands, threads, st)
                              : launch_ml_sweep_t<T, 512, kSweepMoving>(a, bands, threads, st);
    return threads <= 256 ? launch_ml_sweep_t<T, 256, kSweepLinear>(a, bands, threads, st)
                          : launch_ml_sweep_t<T, 512, kSweepLinear>(a, bands, threads, st);
}

// Moving atmospheres: per ray and node the projected velocity u = mu_r . v,
// per node 1/d = sqrt(t_ref/T), and per line, ray and node the inverse of
// sum_f w_f phi((x_f - u)/d)/(d sqrt(pi)) over the line's frequencies (lines
// numbered in transition order).
template <typename T>
__global__ void ml_vel_prep_kernel(long nvox, int ntrans, const TransInfo *__restrict__ ti,
                                   const FreqInfo *__restrict__ fi, const double *__restrict__ mu,
                                   const double *__restrict__ vel, const double *__restrict__ Tg,
                                   double t_ref, T *__restrict__ uproj, T *__restrict__ dinv,
                                   T *__restrict__ vnorm) {
    const long total = (long)kRays * nvox;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total;
         i += (long)gridDim.x * blockDim.x) {
        const int r = (int)(i / nvox);
        const long v = i - (long)r * nvox;
        const double u = mu[3 * r] * vel[v] + mu[3 * r + 1] * vel[nvox + v] +
                         mu[3 * r + 2] * vel[2 * nvox + v];
        const double di = sqrt(t_ref / Tg[v]);
        uproj[i] = (T)u;
        if (r == 0) dinv[v] = (T)di;
        int l = 0;
        for (int t = 0; t < ntrans; ++t) {
            const TransInfo tr = ti[t];
            if (tr.kind != 0) continue;
            double sum = 0.0;
            for (int f = tr.f_begin; f < tr.f_end; ++f) {
                const double dd = (fi[f].xy - u) * di;
                sum += fi[f].w * exp(-dd * dd) * di * 0.56418958354775628;
            }
            vnorm[((long)l * kRays + r) * nvox + v] = (T)(1.0 / sum);
            ++l;
        }
    }
}

cudaError_t launch_ml_vel_prep(int prec, long nvox, int ntrans, const TransInfo *ti,
                               const FreqInfo *fi, const double *mu, const double *vel,
                               const double *T, double t_ref, void *uproj, void *dinv,
                               void *vnorm, cudaStream_t st) {
    const long total = (long)kRays * nvox;
    const int th = 256;
    const long b = std::min<long>((total + th - 1) / th, 152L * 32);
    if (prec == MG3D_PREC_F64)
        ml_vel_prep_kernel<double><<<(int)b, th, 0, st>>>(nvox, ntrans, ti, fi, mu, vel, T, t_ref,
                                                          (double *)uproj, (double *)dinv,
                                                          (double *)vnorm);
    else
        ml_vel_prep_kernel<float><<<(int)b, th, 0, st>>>(nvox, ntrans, ti, fi, mu, vel, T, t_ref,
                                                         (float *)uproj, (float *)dinv,
                                                         (float *)vnorm);
    return cudaGetLastError();
}

cudaError_t launch_ml_sweep_f64(const MlSweepArgs<double> &a, int bands, int threads,
                                cudaStream_t st) {
    return launch_ml_sweep_any<double>(a, bands, threads, st);
}

cudaError_t launch_ml_sweep_f32(const MlSweepArgs<float> &a, int bands, int threads,
                                cudaStream_t st) {
    return launch_ml_sweep_any<float>(a, bands, threads, st);
}

// -------------------------------------------------------------------- rates

__device__ __forceinline__ unsigned long long dbits_ml(double x) {
    return (unsigned long long)__double_as_longlong(x);
}

// an angle sum over the ray-group slots, in slot order
__device__ __forceinline__ PairSum slots_sum(const float *p, long stride, int n) {
    PairSum s;
    s.hi = p[0];
    for (int i = 1; i < n; ++i) s.add(p[(long)i * stride]);
    return s;
}

// The same in FP64 for either precision.
template <typename T>
__device__ __forceinline__ double slots_sum64(const T *p, long stride, int n) {
    double s = (double)p[0];
    for (int i = 1; i < n; ++i) s += (double)p[(long)i * stride];
    return s;
}

// Radiative sums of a transition over the chunk's frequencies, added to acc
// (frequencies in increasing order within a chunk, chunks in order).  The sums
// of a line share the factor 1/(sqrt(pi) d) of its profile, which cancels in
// their ratios and is left out.
struct AccumSums {
    double s0, s1, s2;
};

// The sums of transition tr at node v over frequencies fb .. fe-1 in FP64, from
// angle sums and exponentials in the formal-solution precision T.  PLAIN: no flow,
// partial redistribution, damped line or zero radiation.
template <typename T, bool PLAIN>
__device__ __forceinline__ AccumSums accum_sums(const MlAccumArgs &a, const TransInfo &tr, int fb,
                                                int fe, long v, const fx::Tables &ft) {
    const long nvox = a.nvox, hstride = (long)a.nfreq * nvox;
    const MlNode<T> node(a.tab, v);
    const double inv_d = !PLAIN && tr.kind == 0 && a.voigt ? a.tab.inv_d[v] : 0.0;
    const bool zero = !PLAIN && a.zero_radiation;
    AccumSums s{0.0, 0.0, 0.0};
#pragma unroll 1
    for (int f = fb; f < fe; ++f) {
        const FreqOp &q = a.fo[f];
        const long i = (long)(f - a.f0) * nvox + v;
        double J = 0.0, U = 1.0;
        if (!zero) {
            J = slots_sum64((const T *)a.jx + i, hstride, a.nslots);
            U = slots_sum64((const T *)a.ux + i, hstride, a.nslots);
        }
        if (tr.kind == 0) {
            if (!PLAIN && a.moving && !zero) {
                // the per-ray profile weights are inside J and U already
                s.s0 += f == tr.f_begin ? 1.0 : 0.0;
                s.s1 += J;
                s.s2 += U;
                continue;
            }
            const int pr = !PLAIN && a.prd_index && !zero ? a.prd_index[f] : -1;
            if (pr >= 0) {
                // U = sum_r w_r (1 - w0 (1 - oc)) = oc + (1 - oc) sum_r w_r u_r
                const double oc = a.prd_oc[(long)pr * nvox + v];
                U = oc + (1.0 - oc) * U;
            }
            const T phi = !PLAIN && q.damped ? (T)voigt_H_rational(*a.voigt, a.fi[f].adamp * inv_d,
                                                                   q.a * inv_d)
                                             : node.line_exp(q, ft);
            const double wphi = q.w * (double)phi;
            s.s0 += wphi;
            s.s1 = fma(wphi, J, s.s1);
            s.s2 = fma(wphi, U, s.s2);
        } else {
            const double E = (double)node.cont_exp(q, ft);
            s.s0 = fma(q.w, J, s.s0);
            s.s1 = fma(q.w * E, J, s.s1);
            s.s2 = fma(q.q3 * E, U, s.s2);
        }
    }
    return s;
}

// PLAIN: nor a background field.
template <bool PLAIN>
__global__ void ml_accum64_kernel(const MlAccumArgs a) {
    __shared__ fx::u64 fx_tab[2 * fx::kTab];
    for (int i = threadIdx.x; i < 2 * fx::kTab; i += blockDim.x) fx_tab[i] = a.fx_tab[i];
    __syncthreads();
    const fx::Tables ft{fx_tab, fx_tab + fx::kTab};
    const double *__restrict__ jx = (const double *)a.jx;
    const double *__restrict__ ux = (const double *)a.ux;
    const long nvox = a.nvox, hstride = (long)a.nfreq * nvox;
    const int t = blockIdx.y;
    const TransInfo tr = a.ti[t];
    const int fb = max(tr.f_begin, a.f0), fe = min(tr.f_end, a.f0 + a.nfreq);
    if (fb >= fe) return;
    for (long v = blockIdx.x * (long)blockDim.x + threadIdx.x; v < nvox;
         v += (long)gridDim.x * blockDim.x) {
        AccumSums s{0.0, 0.0, 0.0};
        if (PLAIN) {
            const MlNode<double> node(a.tab, v);
            // the next frequency's angle sums are loaded while this one's are added
            const double *pj = jx + (long)(fb - a.f0) * nvox + v;
            const double *pu = ux + (long)(fb - a.f0) * nvox + v;
#pragma unroll 2
            for (int f = fb; f < fe; ++f, pj += nvox, pu += nvox) {
                const FreqOp &q = a.fo[f];
                const double J = slots_sum64(pj, hstride, a.nslots);
                const double U = slots_sum64(pu, hstride, a.nslots);
                if (tr.kind == 0) {
                    const double wphi = q.w * node.line_exp(q, ft);
                    s.s0 += wphi;
                    s.s1 = fma(wphi, J, s.s1);
                    s.s2 = fma(wphi, U, s.s2);
                } else {
                    const double E = node.cont_exp(q, ft);
                    s.s0 = fma(q.w, J, s.s0);
                    s.s1 = fma(q.w * E, J, s.s1);
                    s.s2 = fma(q.q3 * E, U, s.s2);
                }
            }
        } else {
            s = accum_sums<double, false>(a, tr, fb, fe, v, ft);
            // background field: the new mean intensity
            if (a.jbg && !a.zero_radiation)
                for (int f = fb; f < fe; ++f)
                    ((double *)a.jbg)[(long)f * nvox + v] = slots_sum64(
                        (const double *)a.jm + (long)(f - a.f0) * nvox + v, hstride, a.nslots);
        }
        double *acc = a.acc + (long)t * kAccTerms * nvox + v;
        acc[0] += s.s0;
        acc[nvox] += s.s1;
        acc[2 * nvox] += s.s2;
    }
}

// FP32 angle sums are added as pairs of floats, whose products are good to
// about 2^-45 while no operand or product drops below the 2^-149 a float holds.  A
// node's sums of a transition go to FP64 instead (from the same FP32 angle sums and
// exponentials) where that is not certain:
//   a coefficient outside 2^-100 .. 2^100 (TransInfo::wide, for all nodes);
//   a sum below 2^-80 of the largest mean intensity (or of 1).  A term that lost
//   bits is below 2^-100 of that, so it is below 2^-20 of a larger sum, and what it
//   lost is 2^-24 of itself; for a continuum only the sum of the smaller of the two
//   terms of its downward rate may be tiny;
//   a sum above 2^100, infinite or NaN.
// A continuum's exponential leaves the range from x of about 55 on.  The test costs
// nothing (64x64x65, 120 frequencies: sums 211 us before, 184 with it and 64 registers,
// which let four blocks share an SM), and the populations' errors against an FP64 handle are
// the same with all nodes in pairs and all nodes in FP64 (rms 3.7175e-9 both, 60 boxes).
__device__ __forceinline__ bool pairs_hold(const TransInfo &tr, const PairSum &s0,
                                           const PairSum &s1, const PairSum &s2, float jmax) {
    const float lo = __int_as_float((127 - 80) << 23) * fmaxf(jmax, 1.0f);
    const float hi = __int_as_float((127 + 100) << 23);
    const float a0 = fabsf(s0.hi), a1 = fabsf(s1.hi), a2 = fabsf(s2.hi);
    const float rad = tr.kind == 0 ? a1 : a0;   // 0 without radiation
    return (rad >= lo || jmax == 0.0f) && (tr.kind == 0 ? fminf(a0, a2) : a2) >= lo &&
           fmaxf(fmaxf(a0, a1), a2) <= hi;
}

// Not inlined: it would take part in the register allocation of the loop that always runs.
template <bool PLAIN>
__device__ __noinline__ AccumSums accum_sums_wide(const MlAccumArgs &a, const TransInfo &tr, int fb,
                                                  int fe, long v) {
    return accum_sums<float, PLAIN>(a, tr, fb, fe, v, fx::Tables{nullptr, nullptr});
}

template <bool PLAIN>
__global__ void __launch_bounds__(256, 4)
    ml_accum32_kernel(const __grid_constant__ MlAccumArgs a) {
    const fx::Tables none{nullptr, nullptr};
    const float *__restrict__ jx = (const float *)a.jx;
    const float *__restrict__ ux = (const float *)a.ux;
    const long nvox = a.nvox, hstride = (long)a.nfreq * nvox;
    const int t = blockIdx.y;
    const TransInfo tr = a.ti[t];
    const int fb = max(tr.f_begin, a.f0), fe = min(tr.f_end, a.f0 + a.nfreq);
    if (fb >= fe) return;
    for (long v = blockIdx.x * (long)blockDim.x + threadIdx.x; v < nvox;
         v += (long)gridDim.x * blockDim.x) {
        const MlNode<float> node(a.tab, v);
        const double inv_d = tr.kind == 0 && a.voigt ? a.tab.inv_d[v] : 0.0;
        PairSum s0, s1, s2;
        float jmax = 0.0f;   // largest mean intensity of the transition
        auto add_line = [&](const FreqOp &q, float phi, const PairSum &J, const PairSum &U) {
            const float wh = q.wh * phi;   // w phi as a pair
            const float wl = fmaf(q.wl, phi, fmaf(q.wh, phi, -wh));
            jmax = fmaxf(jmax, fabsf(J.hi));
            s0.add(wh);
            s0.lo += wl;
            s1.add_product(wh, wl, J.hi, J.lo);
            s2.add_product(wh, wl, U.hi, U.lo);
        };
        auto add_cont = [&](const FreqOp &q, float E, const PairSum &J, const PairSum &U) {
            jmax = fmaxf(jmax, fabsf(J.hi));
            s0.add_product(q.wh, q.wl, J.hi, J.lo);
            const float eh = q.wh * E, el = fmaf(q.wl, E, fmaf(q.wh, E, -eh));
            s1.add_product(eh, el, J.hi, J.lo);
            const float gh = q.q3h * E, gl = fmaf(q.q3l, E, fmaf(q.q3h, E, -gh));
            s2.add_product(gh, gl, U.hi, U.lo);
        };
        if (PLAIN) {
            // four frequencies at a time, so that their loads are in flight together
            constexpr int B = 4;
            const float *pj = jx + (long)(fb - a.f0) * nvox + v;
            const float *pu = ux + (long)(fb - a.f0) * nvox + v;
            for (int f = fb; f < fe; f += B, pj += B * nvox, pu += B * nvox) {
                PairSum J[B], U[B];
                // two slots (all rays of a hemisphere in one block) at a time
                for (int s = 0; s < a.nslots; s += 2) {
                    float vj[2][B], vu[2][B];
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int k = 0; k < B; ++k) {
                            const long o = (long)(s + h) * hstride + (f + k < fe ? k : 0) * nvox;
                            vj[h][k] = pj[o];
                            vu[h][k] = pu[o];
                        }
#pragma unroll
                    for (int k = 0; k < B; ++k)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            J[k].add(vj[h][k]);
                            U[k].add(vu[h][k]);
                        }
                }
#pragma unroll
                for (int k = 0; k < B; ++k) {
                    if (f + k >= fe) break;
                    const FreqOp &q = a.fo[f + k];
                    if (tr.kind == 0) add_line(q, node.line_exp(q, none), J[k], U[k]);
                    else add_cont(q, node.cont_exp(q, none), J[k], U[k]);
                }
            }
        } else
        for (int f = fb; f < fe; ++f) {
            const FreqOp &q = a.fo[f];
            const long i = (long)(f - a.f0) * nvox + v;
            PairSum J, U;
            U.hi = 1.0f;
            if (!a.zero_radiation) {
                J = slots_sum(jx + i, hstride, a.nslots);
                U = slots_sum(ux + i, hstride, a.nslots);
            }
            if (tr.kind == 0) {
                if (a.moving && !a.zero_radiation) {
                    // the per-ray profile weights are inside J and U already
                    jmax = fmaxf(jmax, fabsf(J.hi));
                    s0.add(f == tr.f_begin ? 1.0f : 0.0f);
                    s1.add_product(1.0f, 0.0f, J.hi, J.lo);
                    s2.add_product(1.0f, 0.0f, U.hi, U.lo);
                } else {
                    const int pr = a.prd_index && !a.zero_radiation ? a.prd_index[f] : -1;
                    if (pr >= 0) {
                        // U = sum_r w_r (1 - w0 (1 - oc)) = oc + (1 - oc) sum_r w_r u_r
                        const double oc = a.prd_oc[(long)pr * nvox + v];
                        const double u = oc + (1.0 - oc) * U.value();
                        U.hi = (float)u;
                        U.lo = (float)(u - (double)U.hi);
                    }
                    const float phi =
                        q.damped ? (float)voigt_H_rational(*a.voigt, a.fi[f].adamp * inv_d,
                                                           q.a * inv_d)
                                 : node.line_exp(q, none);
                    add_line(q, phi, J, U);
                }
            } else {
                add_cont(q, node.cont_exp(q, none), J, U);
            }
            // background field of the frequency: the new mean intensity
            if (a.jbg && !a.zero_radiation) {
                const PairSum m = slots_sum((const float *)a.jm + i, hstride, a.nslots);
                ((float *)a.jbg)[(long)f * nvox + v] = m.hi + m.lo;
            }
        }
        AccumSums s{s0.value(), s1.value(), s2.value()};
        if (tr.wide || !pairs_hold(tr, s0, s1, s2, jmax))
            s = accum_sums_wide<PLAIN>(a, a.ti[t], fb, fe, v);
        double *acc = a.acc + (long)t * kAccTerms * nvox + v;
        acc[0] += s.s0;
        acc[nvox] += s.s1;
        acc[2 * nvox] += s.s2;
    }
}

// Rates and the N x N solve, one node per thread, N known at compile time: the
// rate matrix is gathered in shared memory (the transitions index it), the
// elimination runs on registers with every index static, pivots chosen on the
// bit patterns (positive doubles order like them) and one refined reciprocal
// per pivot, so that the FP64 pipe sees the products alone.  64x64x129, N = 6:
// 549 -> 460 us; an 8x8x9 grid, latency alone: 50 -> 24 us.
constexpr int kRateThreads = 64;
template <int N>
__global__ void __launch_bounds__(kRateThreads) ml_rates_kernel(const MlRateArgs a) {
    __shared__ double Ps[N * N][kRateThreads];
    const long nvox = a.nvox;
    const int tid = threadIdx.x;
    double cmax = 0.0;
    unsigned neg = 0, bad = 0;
    const long stride = (long)gridDim.x * blockDim.x;
    for (long base = (long)blockIdx.x * blockDim.x; base < nvox; base += stride) {
        const long v = base + tid;
        if (v >= nvox) continue;
#pragma unroll
        for (int i = 0; i < N * N; ++i)
            Ps[i][tid] = i % (N + 1) == 0 ? 0.0 : a.c[(long)i * nvox + v];
        // four transitions at a time, so that their loads are in flight together
        for (int t0 = 0; t0 < a.n_trans; t0 += 4) {
            double a0[4], a1[4], a2[4], G[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int t = min(t0 + k, a.n_trans - 1);
                const double *acc = a.acc + (long)t * kAccTerms * nvox + v;
                a0[k] = acc[0];
                a1[k] = acc[nvox];
                a2[k] = acc[2 * nvox];
                G[k] = a.saha[(long)a.ti[t].lo * nvox + v];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (t0 + k >= a.n_trans) break;
                const TransInfo tr = a.ti[t0 + k];
                double up, down;
                if (tr.kind == 0) {
                    const double inv = fast_div(1.0, a0[k]);
                    const double bJ = tr.b_ul * (a1[k] * inv);
                    up = tr.gr * bJ;
                    down = fma(tr.coef, a2[k] * inv, bJ);
                } else {
                    up = a0[k];
                    down = G[k] * (a2[k] + a1[k]);
                }
                Ps[tr.lo * N + tr.up][tid] += up;
                Ps[tr.up * N + tr.lo][tid] += down;
            }
        }
        // W(n) = M n: row 0 conservation, row i: n_i sum_j P_ij - sum_j n_j P_ji
        double M[N][N + 1];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            double out_i = 0.0;
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (j != i) out_i += Ps[i * N + j][tid];
#pragma unroll
            for (int j = 0; j < N; ++j)
                M[i][j] = i == 0 ? 1.0 : (j == i ? out_i : -Ps[j * N + i][tid]);
            M[i][N] = a.f ? a.f[(long)i * nvox + v] : (i == 0 ? a.n_tot[v] : 0.0);
        }
        if (a.mode == kRateSolve) {
            double inv[N];
#pragma unroll
            for (int c = 0; c < N; ++c) {
                // partial pivoting: the largest |M[r][c]| of the rows below c up
                unsigned long long best = (unsigned long long)__double_as_longlong(fabs(M[c][c]));
                int piv = c;
#pragma unroll
                for (int r = c + 1; r < N; ++r) {
                    const unsigned long long m =
                        (unsigned long long)__double_as_longlong(fabs(M[r][c]));
                    if (m > best) {
                        best = m;
                        piv = r;
                    }
                }
#pragma unroll
                for (int r = c + 1; r < N; ++r) {
                    const bool sw = r == piv;
#pragma unroll
                    for (int j = c; j <= N; ++j) {
                        const double x = M[c][j], y = M[r][j];
                        M[c][j] = sw ? y : x;
                        M[r][j] = sw ? x : y;
                    }
                }
                inv[c] = fast_div(1.0, M[c][c]);
#pragma unroll
                for (int r = c + 1; r < N; ++r) {
                    const double fac = M[r][c] * inv[c];
#pragma unroll
                    for (int j = c + 1; j <= N; ++j) M[r][j] = fma(-fac, M[c][j], M[r][j]);
                }
            }
            double xsol[N];
#pragma unroll
            for (int i = N - 1; i >= 0; --i) {
                double acc = M[i][N];
#pragma unroll
                for (int j = i + 1; j < N; ++j) acc = fma(-M[i][j], xsol[j], acc);
                const double q = acc * inv[i];
                xsol[i] = fma(fma(-M[i][i], q, acc), inv[i], q);
            }
            bool finite = true;
            double cl = 0.0;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const double old = a.n[(long)i * nvox + v];
                a.n[(long)i * nvox + v] = xsol[i];
                const double ci = fast_div(fabs(xsol[i] - old), fabs(xsol[i]));
                if (!(isfinite(xsol[i]) && isfinite(ci))) finite = false;
                else cl = fmax(cl, ci);
                neg += xsol[i] <= 0.0;
            }
            if (finite) cmax = fmax(cmax, cl);
            else ++bad;
        } else {
            double nn[N];
#pragma unroll
            for (int j = 0; j < N; ++j) nn[j] = a.n[(long)j * nvox + v];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                double w = 0.0;
#pragma unroll
                for (int j = 0; j < N; ++j) w += M[i][j] * nn[j];
                if (a.mode == kRateResidual) a.out[(long)i * nvox + v] = M[i][N] - w;
                else a.out[(long)i * nvox + v] += w;
            }
        }
    }
    if (a.mode == kRateSolve && a.scal) {
        __shared__ double red[32];
        __shared__ unsigned cnt[2][32];
        double m = cmax;
        for (int o = 16; o > 0; o >>= 1) {
            m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
            neg += __shfl_xor_sync(0xffffffffu, neg, o);
            bad += __shfl_xor_sync(0xffffffffu, bad, o);
        }
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        if (lane == 0) {
            red[wid] = m;
            cnt[0][wid] = neg;
            cnt[1][wid] = bad;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const int nw = (blockDim.x + 31) >> 5;
            double mm = 0.0;
            unsigned tn = 0, tb = 0;
            for (int i = 0; i < nw; ++i) {
                mm = fmax(mm, red[i]);
                tn += cnt[0][i];
                tb += cnt[1][i];
            }
            if (mm > 0.0) atomicMax(a.scal, dbits_ml(mm));
            if (tn) atomicAdd(a.scal + 1, (unsigned long long)tn);
            if (tb) atomicAdd(a.scal + 2, (unsigned long long)tb);
        }
    }
}

// small grids take small blocks, so that their few nodes reach every SM
static int node_threads(long nvox) { return nvox <= 152L * 64 ? 64 : 256; }

cudaError_t launch_ml_opacity(const MlOpacityArgs &a, cudaStream_t st) {
    const int th = node_threads(a.nvox);
    const dim3 grid(grid_for(a.nvox, th), a.n_trans);
    if (a.prec == MG3D_PREC_F64) ml_opacity_kernel<double><<<grid, th, 0, st>>>(a);
    else ml_opacity_kernel<float><<<grid, th, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_ml_bottom(int prec, long nplane, int nfreq, const FreqInfo *fi,
                             double theta_ref, const double *T, void *ib, cudaStream_t st) {
    const long total = nplane * nfreq;
    if (prec == MG3D_PREC_F64)
        ml_bottom_kernel<double><<<grid_for(total, 256), 256, 0, st>>>(nplane, nfreq, fi,
                                                                       theta_ref, T, (double *)ib);
    else
        ml_bottom_kernel<float><<<grid_for(total, 256), 256, 0, st>>>(nplane, nfreq, fi,
                                                                      theta_ref, T, (float *)ib);
    return cudaGetLastError();
}

cudaError_t launch_ml_accum(const MlAccumArgs &a, cudaStream_t st) {
    const int th = node_threads(a.nvox);
    const dim3 grid(grid_for(a.nvox, th), a.n_trans);
    const bool plain = !a.zero_radiation && !a.moving && !a.prd_index && !a.voigt && !a.jbg;
    if (a.prec == MG3D_PREC_F64) {
        if (plain) ml_accum64_kernel<true><<<grid, th, 0, st>>>(a);
        else ml_accum64_kernel<false><<<grid, th, 0, st>>>(a);
    } else {
        if (plain) ml_accum32_kernel<true><<<grid, th, 0, st>>>(a);
        else ml_accum32_kernel<false><<<grid, th, 0, st>>>(a);
    }
    return cudaGetLastError();
}

template <typename T>
__global__ void ml_slot_sum_kernel(const MlSlotSumArgs a) {
    const T *src = (const T *)a.src;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < a.count;
         i += (size_t)gridDim.x * blockDim.x) {
        const size_t o = a.first + i;
        double v = slots_sum64(src + o, (long)a.len, a.slots);
        if (a.prd_index) {
            const int pr = a.prd_index[o / a.nvox];
            if (pr >= 0) {
                const double oc = a.prd_oc[(size_t)pr * a.nvox + o % a.nvox];
                v = oc + (1.0 - oc) * v;
            }
        }
        a.out[i] = v;
    }
}

cudaError_t launch_ml_slot_sum(const MlSlotSumArgs &a, cudaStream_t st) {
    const int g = grid_for((long)a.count, 256);
    if (a.prec == MG3D_PREC_F64) ml_slot_sum_kernel<double><<<g, 256, 0, st>>>(a);
    else ml_slot_sum_kernel<float><<<g, 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_ml_rates(const MlRateArgs &a, cudaStream_t st) {
    const int g = grid_for(a.nvox, kRateThreads);
    switch (a.n_levels) {
        case 2: ml_rates_kernel<2><<<g, kRateThreads, 0, st>>>(a); break;
        case 3: ml_rates_kernel<3><<<g, kRateThreads, 0, st>>>(a); break;
        case 4: ml_rates_kernel<4><<<g, kRateThreads, 0, st>>>(a); break;
        case 5: ml_rates_kernel<5><<<g, kRateThreads, 0, st>>>(a); break;
        case 6: ml_rates_kernel<6><<<g, kRateThreads, 0, st>>>(a); break;
        case 7: ml_rates_kernel<7><<<g, kRateThreads, 0, st>>>(a); break;
        case 8: ml_rates_kernel<8><<<g, kRateThreads, 0, st>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace mg3d
