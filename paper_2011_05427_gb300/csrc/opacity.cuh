// opacity.cuh -- the group opacities and emission of one (cell, group): per-edge integrals,
// table evaluation (FP64 and FP32 pairs) and the per-cell terms they start from.  Used by
// the opacity kernels (physics.cu) and by the low-order kernels that evaluate the opacities
// where they need them (lo.cu).
#pragma once
#include "batch.cuh"

namespace trt {

// ---------------------------------------------------------------------------------------
// per-edge values
// ---------------------------------------------------------------------------------------
__host__ __device__ inline int series_terms(double x)
{
    return x < 0.125 ? 12 : x < 0.5 ? 18 : x < 1.0 ? 26 : 42;
}

// x < 2: P(x), Nt(x), D(x) by Horner
// The exponential of the group integrals: texp (table-driven, common.cuh) on the device,
// the C library's on the host (inflow spectra and initial state at creation).
struct Mx {
    const double *tab;
    ExpConsts c;
    __host__ __device__ double ex(double x) const
    {
#ifdef __CUDA_ARCH__
        return texp(x, tab, c);
#else
        return std::exp(x);
#endif
    }
};

__host__ __device__ inline void edge_series(double x, const SeriesTables &t, double &P,
                                            double &Nt, double &D)
{
    int n = series_terms(x);
    double sP = 0.0, sN = 0.0, sD = 0.0;
    for (int k = n - 1; k >= 0; --k) {
        sP = fma(sP, x, t.pP[k]);
        sN = fma(sN, x, t.pN[k]);
        sD = fma(sD, x, t.pD[k]);
    }
    double x3 = x * x * x;
    P = x3 * sP;
    Nt = x3 * sN;
    D = x3 * x * x * sD;
}

// x >= 2, every tail scaled by e^{x}:
//   TP = e^x (pi^4/15 - P(x)) = sum_k e^{-(k-1)x} 6 e3(kx)/k^4
//   TN = e^x x^4/(e^x - 1)    = x^4 / (1 - e^{-x})
//   TD = e^x (Dinf - D(x))    = sum_k k(k+1)/2 e^{-(k-1)x} 5040 e7(kx)/k^8
// with e_m(y) = sum_{j<=m} y^j/j!  (integration by parts of t^n e^{-kt}).
__host__ __device__ inline void edge_tail(double x, const SeriesTables &t, const Mx &mx, double &TP,
                                          double &TN, double &TD)
{
    const double e3 = 1.0 + x * (1.0 + x * (0.5 + x * (1.0 / 6.0)));
    const double e7 = 1.0 + x * (1.0 + x * (1.0 / 2 + x * (1.0 / 6 + x * (1.0 / 24 + x * (1.0 / 120
                      + x * (1.0 / 720 + x * (1.0 / 5040)))))));
    double sp = t.tP[1] * e3, sd = t.tD[1] * e7;
    if (x >= 40.0) {   // e^{-x} < 5e-18: one term, and 1 - e^{-x} = 1 in FP64
        TP = sp;
        TD = sd;
        TN = x * x * x * x;
        return;
    }
    const double q = mx.ex(-x);
    double ek = q;
    for (int k = 2; k <= 64 && ek >= 1e-18; ++k) {
        const double y = (double)k * x;
        const double f3 = 1.0 + y * (1.0 + y * (0.5 + y * (1.0 / 6.0)));
        const double f7 = 1.0 + y * (1.0 + y * (1.0 / 2 + y * (1.0 / 6 + y * (1.0 / 24 + y * (1.0 / 120
                          + y * (1.0 / 720 + y * (1.0 / 5040)))))));
        sp += ek * t.tP[k] * f3;
        sd += ek * t.tD[k] * f7;
        ek *= q;
    }
    TP = sp;
    TD = sd;
    TN = x * x * x * x * rcp64(-expm1(-x));
}

// Gauss rule on [xa, xb] for the three scaled integrands x^3 e^{xa-x}/(1-e^{-x}),
// x^4 e^{xa-x}/(1-e^{-x})^2, x^7 e^{xa-x}/(1-e^{-x})^3.  Their nearest singularities
// are the poles x = 2 pi i k, so an n-point rule on a half-width a converges like
// (a/4 pi)^(2n): 3 points reach 1e-16 for xb - xa <= 1/20, 4 points for xb - xa <= 1/4,
// 6 points for xb - xa <= 1.
template <int NP>
__host__ __device__ inline void gauss_group(double xa, double xb, const double *gx,
                                            const double *gw, const Mx &mx, double &dPs,
                                            double &Ns, double &Ds)
{
    // symmetric rule: the points mid -/+ hw xi_j share e^{xa-mid} and e^{+-hw xi_j}, so a
    // pair of points costs one exponential and one reciprocal; e^{-x} follows from
    // e^{-mid} the same way, and 1 - e^{-x} is formed directly where x >= 0.1 (relative
    // error <= eps/x) and by expm1 below
    const double hw = 0.5 * (xb - xa), mid = 0.5 * (xb + xa);
    const double E0 = mx.ex(xa - mid);
    const bool warm = mid - hw < 37.0;              // some point has 1 - e^{-x} != 1
    const double Em = warm ? mx.ex(-mid) : 0.0;
    double sp = 0.0, sn = 0.0, sd = 0.0;
#pragma unroll
    for (int j = NP / 2; j < NP; ++j) {
        const double t = hw * gx[j];
        const double ep = mx.ex(t), em = rcp64(ep);
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const double x = side ? mid + t : mid - t;
            const double ex = side ? E0 * em : E0 * ep;          // e^{xa - x}
            double u = 1.0;                                       // 1/(1 - e^{-x})
            if (warm && x <= 37.0) {
                const double omx = (x >= 0.1) ? 1.0 - Em * (side ? em : ep) : -expm1(-x);
                u = rcp64(omx);
            }
            const double x3 = x * x * x;
            const double eu = gw[j] * ex * x3 * u;
            sp += eu;
            sn += eu * x * u;
            sd += eu * x3 * x * u * u;
        }
    }
    dPs = hw * sp;
    Ns = hw * sn;
    Ds = hw * sd;
}

// e^{xa} [P]_{xa}^{xb}, e^{xa} [Nt]_{xa}^{xb}, e^{xa} [D]_{xa}^{xb}, and 1 - e^{-(xb-xa)}.
// Narrow groups -- xb - xa <= 1 and <= xa/4, where differences of edge values would
// cancel -- integrate the three integrands directly with a Gauss rule (over such a group
// the x^7 factor varies by at most (5/4)^7 and the rest is analytic within 2 pi);
// every other group differences the closed forms.
__host__ __device__ inline void group_integrals(double xa, double xb, bool binf,
                                                const SeriesTables &t, const Mx &mx,
                                                double &dPs, double &Ns, double &Ds,
                                                double &om)
{
    om = binf ? 1.0 : -expm1(-(xb - xa));
    const double w = xb - xa;
    if (!binf && w <= 0.25 * xa && w <= 1.0) {
        if (w <= 0.05)
            gauss_group<3>(xa, xb, t.g3x, t.g3w, mx, dPs, Ns, Ds);
        else if (w <= 0.25)
            gauss_group<4>(xa, xb, t.g4x, t.g4w, mx, dPs, Ns, Ds);
        else
            gauss_group<6>(xa, xb, t.g6x, t.g6w, mx, dPs, Ns, Ds);
        return;
    }
    if (xa >= kXSplit) {
        double TPa, TNa, TDa, TPb = 0.0, TNb = 0.0, TDb = 0.0, r = 0.0;
        edge_tail(xa, t, mx, TPa, TNa, TDa);
        if (!binf) {
            edge_tail(xb, t, mx, TPb, TNb, TDb);
            r = mx.ex(xa - xb);
        }
        dPs = TPa - r * TPb;
        Ns = (TNa - r * TNb) + 4.0 * dPs;
        Ds = TDa - r * TDb;
    } else {
        double Pa, Na, Da, Pb, Nb, Db;
        edge_series(xa, t, Pa, Na, Da);
        if (binf) {
            Pb = t.Pinf;
            Nb = 4.0 * t.Pinf;
            Db = t.Dinf;
        } else if (xb < kXSplit) {
            edge_series(xb, t, Pb, Nb, Db);
        } else {
            double TP, TN, TD;
            edge_tail(xb, t, mx, TP, TN, TD);
            double eb = mx.ex(-xb);
            Pb = t.Pinf - eb * TP;
            Nb = -eb * TN + 4.0 * Pb;
            Db = t.Dinf - eb * TD;
        }
        double ea = mx.ex(xa);
        dPs = ea * (Pb - Pa);
        Ns = ea * (Nb - Na);
        Ds = ea * (Db - Da);
    }
}

// One interval's series in the local coordinate t in [-1, 1], stored as monomial
// coefficients a_0 .. a_{kTabNC-1} (converted from the Chebyshev fit when the tables are
// built) and summed by Horner's rule: one FMA per term, half the FP64 operations of
// Clenshaw's recurrence on the Chebyshev coefficients.  The conversion is safe for the
// tabulated functions: sum |a_j| <= 1.45 min |p(t)| over every group and interval of the
// 17-, 256-, 1024- and 4096-group structures (the fits' coefficients decay much faster than
// the Chebyshev polynomials' monomial coefficients grow on intervals 0.125 wide in ln T).
// The terms from t^kTabLo on are at most 2.4e-6 of |p| there (1.9e-8 absolute for the
// logarithm of the emission factor), so they are summed in FP32 (a_k stored in FP32,
// between 3e-31 and 7.3e7: normal numbers) and joined to the FP64 Horner sum of the low
// terms; against the direct group integrals the split evaluation stays within 1e-12
// (sigma_E), the direct Rosseland quadrature's own 1.6e-11 (sigma_R) and 4e-14 absolute
// (emission logarithm) -- a CPU emulation of the split on every table entry at 9 points
// per interval -- for 3 FP32 FMAs and one exact conversion in place of 4 FP64 FMAs (the
// tail widened with integer instructions, widen_f32).
__device__ inline double horner(const double *__restrict__ a, const float *__restrict__ b,
                                double t, float tf)
{
    float q = b[kTabNC - kTabLo - 1];
#pragma unroll
    for (int k = kTabNC - kTabLo - 2; k >= 0; --k) q = fmaf(q, tf, b[k]);
    double p = widen_f32(q);
#pragma unroll
    for (int k = kTabLo - 1; k >= 0; --k) p = fma(p, t, a[k]);
    return p;
}

// Per-cell terms of the opacity evaluation: T, 1/T, 1/T^3, 27 s C_B T, the table interval
// m and local coordinate t of ln T (m < 0: outside the tables), and with the T_r option
// T_r and T_r / T.  The single-slab kernel reads them from an array that k_cell_terms
// fills once per evaluation (a logarithm and a reciprocal per cell, instead of once per
// block of 8 groups); the batched kernel stages its block's 32 cells with one row (warp),
// rotating with the block over the four sub-partitions.  Both use cell_vals: the same
// operations, the same bits.
struct CellVals {
    double T, iT, iT3, t, kET, Tr, rho;
    float tf;
    int m;
};

__device__ inline CellVals cell_vals(const OpacityArgs &a, int i)
{
    CellVals v;
    const double Ti = a.T[i];
    const double iT = rcp64(Ti);
    v.T = Ti;
    v.iT = iT;
    v.iT3 = iT * iT * iT;
    v.kET = a.kE * Ti;
    int m = -1;
    double t = 0.0;
    if (a.otab) {
        const double z = (log(Ti) - kTabU0) * (1.0 / kTabH);
        if (z >= 0.0 && z < (double)kTabNI) {
            m = min((int)z, kTabNI - 1);
            t = 2.0 * (z - (double)m) - 1.0;
        }
    }
    v.m = m;
    v.t = t;
    v.tf = (float)t;
    v.Tr = Ti;
    v.rho = 1.0;
    if (a.Erad) {   // T_r = (E/a_R)^{1/4}; T_r = T without a usable energy
        const double E = a.Erad[i];
        const double Tr = (E > 0.0 && isfinite(E)) ? sqrt(sqrt(E / kAR)) : Ti;
        v.Tr = Tr;
        v.rho = Tr * iT;
    }
    return v;
}

// the per-cell arrays of the single-slab kernel: [7][nx] doubles (T, 1/T, 1/T^3, t, 27 s
// C_B T, T_r, T_r/T), then tf [nx] floats and m [nx] ints
struct CellArrays {
    double *d;
    float *f;
    int *m;
    int nx;
    __device__ void put(int i, const CellVals &v) const
    {
        d[i] = v.T; d[nx + i] = v.iT; d[2 * nx + i] = v.iT3; d[3 * nx + i] = v.t;
        d[4 * nx + i] = v.kET; d[5 * nx + i] = v.Tr; d[6 * nx + i] = v.rho;
        f[i] = v.tf;
        m[i] = v.m;
    }
    __device__ CellVals get(int i) const
    {
        CellVals v;
        v.T = d[i]; v.iT = d[nx + i]; v.iT3 = d[2 * nx + i]; v.t = d[3 * nx + i];
        v.kET = d[4 * nx + i]; v.Tr = d[5 * nx + i]; v.rho = d[6 * nx + i];
        v.tf = f[i];
        v.m = m[i];
        return v;
    }
};

__device__ inline CellArrays cell_arrays(const OpacityArgs &a)
{
    return CellArrays{a.cterm, reinterpret_cast<float *>(a.cterm + 7 * (size_t)a.nx),
                      reinterpret_cast<int *>(a.cterm + 7 * (size_t)a.nx) + a.nx, a.nx};
}

// the pair form's per-cell terms (TRT_LO_PAIR): t, 1/T, 1/T^3, 27 s C_B T, h/2 split from
// the FP64 terms of cell_vals
struct CellPair {
    fpair t, iT, iT3, kET, hh;
};
__device__ inline CellPair cell_pair(const OpacityArgs &a, int i, const CellVals &v)
{
    return CellPair{fpair(v.t), fpair(v.iT), fpair(v.iT3), fpair(v.kET), fpair(0.5 * a.h[i])};
}

// The three quantities of group g in a cell with terms v outside the tables: direct group
// integrals (never inlined: a branch around them, not their code in every evaluation).
struct OpacVals {
    double sg, em, sR;
};
static __device__ __noinline__ OpacVals opacity_direct(double nu_a, double nu_b, double s, double T,
                                                       double iT, double iT3,
                                                       const SeriesTables *ser, const Mx &mx)
{
    const bool binf = isinf(nu_b);
    const double k27 = 27.0 * s;
    const double xa = nu_a * iT;
    const double xb = binf ? 0.0 : nu_b * iT;
    double dPs, Ns, Ds, om;
    group_integrals(xa, xb, binf, *ser, mx, dPs, Ns, Ds, om);
    OpacVals o;
    o.sg = k27 * om * iT3 * rcp64(dPs);
    o.sR = k27 * Ns * iT3 * rcp64(Ds);
    o.em = k27 * kCB * T * mx.ex(-xa) * om;
    return o;
}

// group g in a cell with terms v, FP64
__device__ inline OpacVals opacity_vals(const OpacityArgs &a, int g, const CellVals &v, const Mx &mx)
{
    const int m = v.m;
    if (m < 0)
        return opacity_direct(a.edges[g], a.edges[g + 1], a.s, v.T, v.iT, v.iT3, a.ser, mx);
    // tabulated: three polynomials in ln T on the cell's interval (the sigma series carry
    // the factor 27 s, kE = 27 s C_B)
    const double t = v.t;
    const float tf = v.tf;
    const double *c = a.otab + ((size_t)g * kTabNI + m) * kTabEntry;
    const float *ch = reinterpret_cast<const float *>(c + kTabNF * kTabLo);
    constexpr int kh = kTabNC - kTabLo;
    OpacVals o;
    o.sg = horner(c, ch, t, tf) * v.iT3;
    o.sR = horner(c + kTabLo, ch + kh, t, tf) * v.iT3;
    o.em = v.kET * mx.ex(horner(c + 2 * kTabLo, ch + 2 * kh, t, tf) - a.edges[g] * v.iT);
    return o;
}

// The same quantities in FP32-pair arithmetic (TRT_LO_PAIR; outputs FP64): the three
// Horner sums with their FP64 coefficients as pairs (the FP32 tails as in horner), sigma =
// sum / T^3, and the emission 27 s C_B T e^w, w = (the emission factor's logarithm) -
// nu_g/T, by pr_exp as a pair times 2^k -- the power of two goes into the exponent of the
// FP64 result (pr_join), so e_g keeps FP64's range.  Relative errors: about 1e-14 in the
// opacities, about 3 2^-47 max(1, |w|) in e_g (w's: nu_g, 1/T and their product each
// rounded to a pair; 1.6e-11 at the smallest e_g that FP64 holds, e^-746).  m, tf: the
// cell's table interval (>= 0) and FP32 local coordinate; cells outside the tables take
// opacity_body (the callers' choice), the T_r option k_opacity_tr.
__device__ inline fpair horner_pair(const fpair *__restrict__ a, const float *__restrict__ b,
                                   fpair t, float tf)
{
    float q = b[kTabNC - kTabLo - 1];
#pragma unroll
    for (int k = kTabNC - kTabLo - 2; k >= 0; --k) q = fmaf(q, tf, b[k]);
    fpair p(q, 0.f);
#pragma unroll
    for (int k = kTabLo - 1; k >= 0; --k) p = fma(p, t, a[k]);
    return p;
}

// sigma_E and sigma_R as pairs, the emission as a pair times 2^k
__device__ inline void opacity_vals_pair(const OpacityArgs &a, int g, int m, float tf,
                                         const CellPair &cp, const fpair *e2p, fpair &sg,
                                         fpair &em, int &k, fpair &sR)
{
    const fpair *c = a.otabp + ((size_t)g * kTabNI + m) * kTabEntry;
    const float *ch = reinterpret_cast<const float *>(c + kTabNF * kTabLo);
    constexpr int kh = kTabNC - kTabLo;
    sg = horner_pair(c, ch, cp.t, tf) * cp.iT3;
    sR = horner_pair(c + kTabLo, ch + kh, cp.t, tf) * cp.iT3;
    const fpair xa = a.otabp[(size_t)a.G * kTabNI * kTabEntry + g] * cp.iT;
    em = cp.kET * pr_exp(horner_pair(c + 2 * kTabLo, ch + 2 * kh, cp.t, tf) - xa, k, e2p);
}

// the pair form's terms of cell i from the arrays of k_cell_terms
__device__ inline CellPair cell_pair_at(const OpacityArgs &a, int i)
{
    const int n = a.nx;
    return CellPair{a.cpair[i], a.cpair[n + i], a.cpair[2 * n + i], a.cpair[3 * n + i],
                    a.cpair[4 * n + i]};
}

}  // namespace trt
