// lo.cu -- low-order QD systems (K3/K4), restriction between frequency grids (K4), grey
// LOQD + material energy balance Newton step (K5).
//
// One group of one level (eq. mloqd-d, eq. mloqd-d-gamma, Sec. 5) is
//   cell i:  (dx_i/dt)(E_i - Eold_i) + F_{i+1/2} - F_{i-1/2} + dx_i a_i E_i = dx_i s_i
//   face f:  (dx_f/(c dt))(F - Fold) + c (phiR E_right - phiL E_left) + sigR dx_f F = 0
// with a = c sigma_E, s = 2 sigma_B B on the group levels; phiR = phi_right + eta-hat,
// phiL = phi_left + eta-check; the boundary faces close a half cell with eq. mloqd-bcs
// (F = c C (E_face - E_in) + F_in, the face energy eliminated).  Eliminating F face by
// face, F_f = GD_f + PL_f E_{f-1} - PR_f E_f, gives a tridiagonal system in E that is
// column diagonally dominant (the dx/dt term), so elimination needs no pivoting.
//
// GB300 mapping.  A CTA of four warps (one per sub-partition, each with its own FP64 pipe)
// owns one system.  FP64 throughput on GB300 is a small fraction of FP32, so the solver
// keeps the FP64 work of plain Thomas elimination (one reciprocal per row) but splits the
// serial chain: each of P = min(128, n/2) threads eliminates its chunk of >= 2 consecutive
// rows (a "modified Thomas" pass down and up the chunk that leaves each row coupled only to
// the chunk's first and last unknowns); the chunks' last rows, then every other first row,
// are eliminated by cyclic reduction until at most 32 rows are left, which one warp solves
// by parallel cyclic reduction in registers; back substitution retraces the steps.  Rows are
// built from the level's fields into shared memory in a [row-in-chunk][chunk] layout
// (conflict free for the elimination).
#include <cmath>
#include "opacity.cuh"

namespace trt {

namespace {

template <typename R>
__device__ inline R rcpR(R d);
template <>
__device__ inline double rcpR<double>(double d) { return rcp64(d); }
template <>
__device__ inline float rcpR<float>(float d) { return __frcp_rn(d); }
template <>
__device__ inline fpair rcpR<fpair>(fpair d) { return prcp(d); }

// a/w: the refined reciprocal and one residual correction (the correctly rounded quotient
// but for rare last bits).  The weights of cold cells are subnormal, where 1/w overflows and
// a/w does not: an exponent outside +-900 divides, and a non-finite quotient is kept.
static __device__ __noinline__ double rquot_divide(double a, double w) { return a / w; }
__device__ inline double rquot(double a, double w)
{
    const unsigned ex = ((unsigned)__double2hiint(w) >> 20) & 0x7ffu;
    if (ex - 123u > 1800u) return rquot_divide(a, w);
    const double r = rcp64(w);
    const double q = a * r;
    if ((((unsigned)__double2hiint(q) >> 20) & 0x7ffu) == 0x7ffu) return q;
    return fma(fma(-q, w, a), r, q);
}

// Source terms of a group system (Eold, the emission, Fold, the boundary inflows) and its
// solution (E, F) in the pair form are held scaled by 2^-ks, ks the group's largest source
// exponent (lo_src_exp): the system is linear in them, and FP32's exponent range would
// otherwise cut the small groups' precision (values below 2^-103) or zero them (below
// 2^-126).  The coefficients are not scaled.  FP64 and FP32: ks is unused.
template <typename R>
__device__ inline R src_in(double v, int ks)
{
    if constexpr (is_pair<R>) return pr_split(v, ks);
    else return (R)v;
}
template <typename R>
__device__ inline double sol_out(R v, int ks)
{
    if constexpr (is_pair<R>) return pr_join(v, ks);
    else return (double)v;
}
// row constant j of kind k (the Problem::lopc order: 0 hf, 1 dxicdt, 2 fwl, 3 fwr, 4 hidt,
// 5 hc, 6 h2, 7 h): the pair form reads the pair copy, the others the FP64 array d
template <typename R>
__device__ inline R lc(const LoCtx &x, int k, int j, const double *d)
{
    if constexpr (is_pair<R>) return x.pc[(size_t)k * (x.nx + 1) + j];
    else return (R)d[j];
}
__device__ inline int bexp64(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
// the largest biased exponent of group q's source terms over this thread's cells and faces
// (threads t, t + nthr, ...); 0 when they are all zero
__device__ inline int lo_src_exp(const LoCtx &x, int q, int t, int nthr)
{
    const int n = x.nx;
    int m = 0;
    for (int i = t; i <= n; i += nthr) {
        if (i < n) {
            m = max(m, bexp64(x.L.Eold[(size_t)q * n + i]));
            m = max(m, bexp64(x.a_cell ? x.s_cell[i] : x.L.emis[(size_t)q * n + i]));
        }
        m = max(m, bexp64(x.L.Fold[(size_t)q * (n + 1) + i]));
    }
    if (t == 0)
        m = max(max(m, max(bexp64(x.L.Ein0[q]), bexp64(x.L.Fin0[q]))),
                max(bexp64(x.L.EinX[q]), bexp64(x.L.FinX[q])));
    return m;
}


// F_f = GD + PL E_{f-1} - PR E_f  (boundary faces: the face energy already eliminated).
// kW: GD is instead W = dx/(c dt) / D, the factor of Fold in GD, without the boundary
// inflow terms (the first pass of the pair staging, before the source scale is known).
// Every load comes before the arithmetic, the two boundaries in one branch: on a level of a
// few cells or groups a second round trip to L2, and a warp that holds both boundary faces
// taking two branches in turn, were a third of the staging's time.
template <typename R, bool kW = false>
__device__ inline void face_coef(const LoCtx &x, int q, int f, R &PL, R &PR, R &GD, int ks = 0)
{
    const int nx = x.nx;
    const bool lo = f == 0, hi = f == nx;
    const size_t fq = (size_t)q * (nx + 1) + f, cq = (size_t)q * nx;
    const double vL = *(lo ? x.L.phib0 + q : x.L.phi + cq + f - 1);
    const double vR = *(hi ? x.L.phibX + q : x.L.phi + cq + f);
    double Cb = 0.0, Ein = 0.0, Fin = 0.0, Fo = 0.0;
    if (lo || hi) {
        Cb = (lo ? x.L.C0 : x.L.CX)[q];
        if constexpr (!kW) {
            Ein = (lo ? x.L.Ein0 : x.L.EinX)[q];
            Fin = (lo ? x.L.Fin0 : x.L.FinX)[q];
        }
    }
    if constexpr (!kW) Fo = x.L.Fold[fq];
    const R dx = lc<R>(x, 0, f, x.hf);
    // dx (1/(c dt) + sigma_R,face) and dx Fold/(c dt) from the row constants: the face
    // opacity's dx-weighted mean folded into one FMA per cell opacity
    const R dxi = lc<R>(x, 1, f, x.dxicdt);
    R phiL = (R)vL, phiR = (R)vR, D;
    if (!x.L.fine) {
        const double eL = x.L.etaL[fq], eR = x.L.etaR[fq];
        D = fma(dx, (R)x.L.sigR[fq], dxi);
        phiL += (R)eL;
        phiR += (R)eR;
    } else {
        const double *sc = x.L.sigR + cq;
        const double sl = sc[max(f - 1, 0)], sr = sc[min(f, nx - 1)];
        D = lo || hi ? fma(dx, (R)(lo ? sr : sl), dxi)
                     : fma(lc<R>(x, 2, f, x.fwl), (R)sl, fma(lc<R>(x, 3, f, x.fwr), (R)sr, dxi));
    }
    R Gf;
    if constexpr (kW) Gf = dxi;
    else Gf = src_in<R>(Fo, ks) * dxi;
    const R c = (R)kC;
    if (lo || hi) {   // E_face = E_in + (F - F_in)/(c C)
        const R iC = rcpR<R>((R)Cb);
        const R s = lo ? phiL : -phiR;
        D -= s * iC;
        if constexpr (!kW) Gf += s * (c * src_in<R>(Ein, ks) - src_in<R>(Fin, ks) * iC);
    }
    const R iD = rcpR<R>(D);
    const R ciD = c * iD;
    PL = phiL * ciD;
    PR = phiR * ciD;
    GD = Gf * iD;
}

// row i of the cell equation, from the row constants h/dt, c h, 2 h: Ap = h (1/dt + a), Dp =
// h (s + Eold/dt)
template <typename R>
__device__ inline void cell_row(const LoCtx &x, int q, int i, R &Ap, R &Dp, int ks = 0)
{
    const size_t c = (size_t)q * x.nx + i;
    const R Eo = src_in<R>(x.L.Eold[c], ks);
    const R hidt = lc<R>(x, 4, i, x.hidt);
    if (x.a_cell) {
        const R hc = lc<R>(x, 7, i, x.h);
        Ap = fma(hc, (R)x.a_cell[i], hidt);
        Dp = fma(hidt, Eo, hc * src_in<R>(x.s_cell[i], ks));
    } else {
        Ap = fma(lc<R>(x, 5, i, x.hc), (R)x.L.sig[c], hidt);
        Dp = fma(hidt, Eo, lc<R>(x, 6, i, x.h2) * src_in<R>(x.L.emis[c], ks));
    }
}

// The face coefficients PL, PR, GD and the row parts dx/dt + dx a, dx s + dx Eold/dt of
// system q into the layout by `nthr` cooperating threads (index `t`).  n >= 2.
template <typename R>
__device__ void lo_stage(const LoCtx &x, int q, R *sm, int S, int t, int nthr, int ks = 0)
{
    const int n = x.nx;
    R *PLc = sm, *PRc = sm + S, *GDc = sm + 2 * S, *Ap = sm + 3 * S, *Dp = sm + 5 * S;
    for (int f = t; f <= n; f += nthr) {
        const int o = x.lo_slot[f];   // TriLayout's slots: a table built with the problem
        R PL, PR, GD;
        face_coef<R>(x, q, f, PL, PR, GD, ks);
        PLc[o] = PL;
        PRc[o] = PR;
        GDc[o] = GD;
        if (f < n) cell_row<R>(x, q, f, Ap[o], Dp[o], ks);
    }
}

// The same in the pair form by the CTA (t = threadIdx.x), with the group's source scale
// (src_in): pass 1 forms the coefficients PL, PR, Ap and the face factor W of Fold (a 7th
// array after the six of the solve) and parks the raw FP64 sources in slots the
// elimination fills later (Fold in GD's, Eold in Dp's, the emission in Cp's) while it
// takes their largest exponent; the CTA's maximum gives ks; pass 2 splits the parked
// sources at that scale into GD and Dp (the boundary faces are formed again whole, with
// their inflow terms).  Each slot is written and read again by one thread, so only the
// reduction needs a barrier.  Returns ks.  n >= 2.
__device__ int lo_stage_pair(const LoCtx &x, int q, fpair *sm, int S)
{
    const int n = x.nx;
    const int t = threadIdx.x, nthr = blockDim.x;
    fpair *PLc = sm, *PRc = sm + S, *GDc = sm + 2 * S, *Ap = sm + 3 * S, *Cp = sm + 4 * S,
          *Dp = sm + 5 * S, *Wc = sm + 6 * S;
    double *rawF = reinterpret_cast<double *>(GDc), *rawE = reinterpret_cast<double *>(Dp),
           *rawS = reinterpret_cast<double *>(Cp);
    int m = 0;
    for (int f = t; f <= n; f += nthr) {
        const int o = x.lo_slot[f];
        fpair PL, PR, W;
        face_coef<fpair, true>(x, q, f, PL, PR, W);
        PLc[o] = PL;
        PRc[o] = PR;
        Wc[o] = W;
        const double Fo = x.L.Fold[(size_t)q * (n + 1) + f];
        rawF[o] = Fo;
        m = max(m, bexp64(Fo));
        if (f < n) {
            const double Eo = x.L.Eold[(size_t)q * n + f];
            const double sv = x.a_cell ? x.s_cell[f] : x.L.emis[(size_t)q * n + f];
            rawE[o] = Eo;
            rawS[o] = sv;
            m = max(m, max(bexp64(Eo), bexp64(sv)));
            const fpair hidt = lc<fpair>(x, 4, f, x.hidt);
            Ap[o] = x.a_cell ? fma(lc<fpair>(x, 7, f, x.h), (fpair)x.a_cell[f], hidt)
                             : fma(lc<fpair>(x, 5, f, x.hc), (fpair)x.L.sig[(size_t)q * n + f], hidt);
        }
    }
    if (t == 0)
        m = max(max(m, max(bexp64(x.L.Ein0[q]), bexp64(x.L.Fin0[q]))),
                max(bexp64(x.L.EinX[q]), bexp64(x.L.FinX[q])));
    __shared__ int kw[32];
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((t & 31) == 0) kw[t >> 5] = m;
    __syncthreads();
    m = 0;
    for (int w = 0; w < (nthr >> 5); ++w) m = max(m, kw[w]);
    const int ks = (m == 0) ? 0 : m - 1023;
    for (int f = t; f <= n; f += nthr) {
        const int o = x.lo_slot[f];
        if (f == 0 || f == n) {
            fpair PL, PR, GD;
            face_coef<fpair>(x, q, f, PL, PR, GD, ks);
            GDc[o] = GD;
        } else {
            GDc[o] = pr_split(rawF[o], ks) * Wc[o];
        }
        if (f < n) {
            const fpair sv = pr_split(rawS[o], ks);
            const fpair Eo = pr_split(rawE[o], ks);
            Dp[o] = fma(lc<fpair>(x, 4, f, x.hidt), Eo,
                        (x.a_cell ? lc<fpair>(x, 7, f, x.h) : lc<fpair>(x, 6, f, x.h2)) * sv);
        }
    }
    return ks;
}

// One system on the staged arrays in sm (PL, PR, GD, Ap, Cp, Dp of y.S slots each; rb: 3 P
// more) by the whole block, of which the first P threads work: the solution x ends in Dp.
// n >= 2; ends with a barrier.
//   - chunks: rows normalised, row 0 of a chunk coupled to the last unknown of the chunk before
//     and its own last, the others to the chunk's first and last;
//   - the last rows are eliminated (a row needs its neighbours' three values: one exchange
//     through rb), then every other first row at strides 1, 2 until 32 or fewer are left;
//   - parallel cyclic reduction of those by warp 0 (rows kept with unit diagonals: one
//     reciprocal per row and level);
//   - back substitution.
// On the chain of one thread: 13 operations per chunk row (4 rows at n = 500), 12 per
// elimination step (3 + 5 there), about 170 in all, where one warp with 16-row chunks and
// PCR of 64 rows took 430; the operations in all are the same.  Measured against that one-warp
// form, 500 cells: 16 groups FP64 30.5 -> 20.3 us, 1024 groups FP64 (FP64-bound) 60 -> 61,
// 1024 groups pair (latency-bound) 41.8 -> 32.2; the grey kernel (four warps with 256 rows of
// PCR before) 23.0 -> 16.4.
template <typename R>
__device__ void tri_solve(R *sm, R *rb, int n, const TriLayout &y)
{
    const int t = threadIdx.x, P = y.P, S = y.S, LP = y.LP;
    R *PLc = sm, *PRc = sm + S, *GDc = sm + 2 * S;
    R *Ap = sm + 3 * S, *Cp = sm + 4 * S, *Dp = sm + 5 * S;
    R *rA = rb, *rC = rb + P, *rD = rb + 2 * P;
    const bool act = t < P;
    const int r0 = act ? (t * n) / P : n;
    const int r1 = act ? ((t + 1) * n) / P : n;
    const int m = r1 - r0;
    R A0 = 0, C0 = 0, D0 = 0, A1 = 0, C1 = 0, D1 = 0;   // the chunk's first and last row
    if (act) {
        R PLi = PLc[t], PRi = PRc[t], GDi = GDc[t];
        R ap = 0, cp = 0, dp = 0;
        for (int k = 0; k < m; ++k) {
            const int i = r0 + k, o = k * LP + t;
            const int on = (k + 1 < m) ? o + LP : (t + 1 < P) ? t + 1 : S - 1;   // face i + 1
            const R PL1 = PLc[on], PR1 = PRc[on], GD1 = GDc[on];
            const R di = Ap[o] + PL1 + PRi;
            const R rh = Dp[o] - GD1 + GDi;
            const R lo = (i > 0) ? -PLi : (R)0;
            const R up = (i < n - 1) ? -PR1 : (R)0;
            if (k < 2) {
                const R r = rcpR<R>(di);
                ap = lo * r;
                cp = up * r;
                dp = rh * r;
            } else {
                const R r = rcpR<R>(di - lo * cp);
                dp = r * (rh - lo * dp);
                ap = -r * lo * ap;
                cp = r * up;
            }
            if (k == 0) { A0 = ap; C0 = cp; D0 = dp; }
            Ap[o] = ap;
            Cp[o] = cp;
            Dp[o] = dp;
            PLi = PL1;
            PRi = PR1;
            GDi = GD1;
        }
        A1 = ap; C1 = cp; D1 = dp;
        // upwards: rows m-3 .. 1 coupled to the chunk's first and last unknown
        if (m >= 3) {
            const int o2 = (m - 2) * LP + t;
            R a = Ap[o2], c = Cp[o2], d = Dp[o2];   // the row below
            for (int k = m - 3; k >= 1; --k) {
                const int o = k * LP + t;
                const R ck = Cp[o];
                d = Dp[o] - ck * d;
                a = Ap[o] - ck * a;
                c = -ck * c;
                Dp[o] = d;
                Ap[o] = a;
                Cp[o] = c;
            }
            const R r = rcpR<R>((R)1 - C0 * a);
            D0 = r * (D0 - C0 * d);
            A0 = r * A0;
            C0 = -r * C0 * c;
        }
        rA[t] = A1;
        rC[t] = C1;
        rD[t] = D1;
    }
    __syncthreads();
    R lA = 0, lC = 0, lD = 0;   // the last row of the chunk before
    if (act && t > 0) { lA = rA[t - 1]; lC = rC[t - 1]; lD = rD[t - 1]; }
    __syncthreads();
    // row j with unit diagonal between rows l and u: A, C, D of the row at twice the distance
    const auto step = [](R &A, R &C, R &D, R lA, R lC, R lD, R uA, R uC, R uD) {
        const R al = -A, ga = -C;
        const R r = rcpR<R>((R)1 + al * lC + ga * uA);
        A = al * lA * r;
        C = ga * uC * r;
        D = (D + al * lD + ga * uD) * r;
    };
    if (act) {
        step(A0, C0, D0, lA, lC, lD, A1, C1, D1);
        rA[t] = A0;
        rC[t] = C0;
        rD[t] = D0;
    }
    __syncthreads();
    int s = 1;   // stride of the first rows still in play
    for (; (P + s - 1) / s > 32; s <<= 1) {
        const int j = t * 2 * s;
        if (j < P) {
            R A = rA[j], C = rC[j], D = rD[j];
            const bool hl = j > 0, hu = j + s < P;
            step(A, C, D, hl ? rA[j - s] : (R)0, hl ? rC[j - s] : (R)0, hl ? rD[j - s] : (R)0,
                 hu ? rA[j + s] : (R)0, hu ? rC[j + s] : (R)0, hu ? rD[j + s] : (R)0);
            rA[j] = A;   // no other thread reads row j: its neighbours are odd multiples of s
            rC[j] = C;
            rD[j] = D;
        }
        __syncthreads();
    }
    if (t < 32) {
        const int nr = (P + s - 1) / s, j = t * s;
        R A = 0, C = 0, D = 0;
        if (t < nr) { A = rA[j]; C = rC[j]; D = rD[j]; }
        for (int d = 1; d < nr; d <<= 1) {
            R pA = shfl_up(0xffffffffu, A, d), pC = shfl_up(0xffffffffu, C, d), pD = shfl_up(0xffffffffu, D, d);
            R uA = shfl_down(0xffffffffu, A, d), uC = shfl_down(0xffffffffu, C, d), uD = shfl_down(0xffffffffu, D, d);
            if (t < d) { pA = 0; pC = 0; pD = 0; }
            if (t + d > 31) { uA = 0; uC = 0; uD = 0; }
            step(A, C, D, pA, pC, pD, uA, uC, uD);
        }
        if (t < nr) rD[j] = D;
    }
    __syncthreads();
    for (s >>= 1; s >= 1; s >>= 1) {   // the eliminated first rows, odd multiples of s
        const int j = t * 2 * s + s;
        if (j < P) {
            R D = rD[j] - rA[j] * rD[j - s];
            if (j + s < P) D = D - rC[j] * rD[j + s];
            rD[j] = D;
        }
        __syncthreads();
    }
    if (act) {
        const R x0 = rD[t];
        R x1 = D1 - A1 * x0;
        if (t + 1 < P) x1 = x1 - C1 * rD[t + 1];
        Dp[t] = x0;
        for (int k = 1; k < m - 1; ++k) {
            const int o = k * LP + t;
            Dp[o] = Dp[o] - Ap[o] * x0 - Cp[o] * x1;
        }
        Dp[(m - 1) * LP + t] = x1;
    }
    __syncthreads();
}

// The outputs of system q by every thread of the CTA, from the solution (chunk layout, in
// the Dp array) and the face coefficients: consecutive threads take consecutive cells and
// faces (coalesced stores), each slot found through the slot table: F_f = GD_f + PL_f
// E_{f-1} - PR_f E_f, and the boundary face energies (the pair form in pair arithmetic, at
// the source scale).  n >= 2; called after a barrier that follows the elimination.
template <typename R>
__device__ void lo_outputs_cta(const LoCtx &x, int q, const R *sm, int S, int ks)
{
    const int n = x.nx;
    const R *PLc = sm, *PRc = sm + S, *GDc = sm + 2 * S, *Dp = sm + 5 * S;
    double *E = x.L.E + (size_t)q * n;
    double *F = x.L.F + (size_t)q * (n + 1);
    for (int f = threadIdx.x; f <= n; f += blockDim.x) {
        const int o = x.lo_slot[f];
        R Fv = GDc[o];
        if (f > 0) Fv += PLc[o] * Dp[x.lo_slot[f - 1]];
        if (f < n) {
            const R Ef = Dp[o];
            Fv -= PRc[o] * Ef;
            E[f] = sol_out<R>(Ef, ks);
        }
        F[f] = sol_out<R>(Fv, ks);
        if (f == 0 || f == n) {
            const double Ein = f == 0 ? x.L.Ein0[q] : x.L.EinX[q];
            const double Fin = f == 0 ? x.L.Fin0[q] : x.L.FinX[q];
            const double Cb = f == 0 ? x.L.C0[q] : x.L.CX[q];
            double Eb;
            if constexpr (is_pair<R>)
                Eb = pr_join(src_in<R>(Ein, ks) +
                                 (Fv - src_in<R>(Fin, ks)) * rcpR<R>((R)kC * (R)Cb), ks);
            else
                Eb = Ein + rquot((double)Fv - Fin, kC * Cb);
            (f == 0 ? x.L.Eb0 : x.L.EbX)[q] = Eb;
        }
    }
}

// One cell: the system is one equation, solved by one thread.
template <typename R>
__device__ void lo_one_cell(const LoCtx &x, int q, int ks = 0)
{
    double *E = x.L.E + q, *F = x.L.F + 2 * (size_t)q;
    R PL0, PR0, GD0, PL1, PR1, GD1, Ap0, Dp0;
    face_coef<R>(x, q, 0, PL0, PR0, GD0, ks);
    face_coef<R>(x, q, 1, PL1, PR1, GD1, ks);
    cell_row<R>(x, q, 0, Ap0, Dp0, ks);
    const R di = Ap0 + PL1 + PR0;
    const R rh = Dp0 - GD1 + GD0;
    const R e0 = rh / di;
    E[0] = sol_out<R>(e0, ks);
    const double F0d = sol_out<R>(GD0 - PR0 * e0, ks), F1d = sol_out<R>(GD1 + PL1 * e0, ks);
    F[0] = F0d;
    F[1] = F1d;
    x.L.Eb0[q] = x.L.Ein0[q] + (F0d - x.L.Fin0[q]) / (kC * x.L.C0[q]);
    x.L.EbX[q] = x.L.EinX[q] + (F1d - x.L.FinX[q]) / (kC * x.L.CX[q]);
}

// FP32 group solve refined to FP64 accuracy (mixed-precision iterative refinement).  The
// rows are staged in FP64 (s64) and converted to FP32 (s32), eliminated in FP32 (x0), then
// kLoRefine times the residual r = b - A x of the FP64 rows is formed in FP64, A d = r
// eliminated in FP32 and d added to x in FP64, all by the whole CTA; E = x, and the fluxes
// follow with the FP64 face coefficients.  Each step multiplies the error by about
// cond(A) eps_32 (the plain FP32 solve's error: 3.6e-6 in T on fc_1024, ~5e-5 in E on a
// 1000-cell random level, where one step left 2.6e-9); the eliminations, the part that is
// serial in cells, run on the FP32 pipes.
// Shared memory: 6 S doubles, 6 S + 3 P floats.
constexpr int kLoRefine = 2;

__device__ void lo_solve_refined(const LoCtx &x, int q)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = x.nx, t = threadIdx.x, nthr = blockDim.x;
    if (n < 2) {   // one cell: the FP64 form
        if (t == 0) lo_one_cell<double>(x, q);
        return;
    }
    const TriLayout y = tri_layout(n);
    const int S = y.S;
    double *s64 = reinterpret_cast<double *>(smem_raw);
    float *s32 = reinterpret_cast<float *>(s64 + 6 * S);
    const double *PL = s64, *PR = s64 + S, *GD = s64 + 2 * S, *Ap = s64 + 3 * S;
    double *X0 = s64 + 4 * S;   // the solution in FP64 (the unused Cp array of s64)
    double *Dp = s64 + 5 * S;   // right-hand sides, then E
    float *pl = s32, *pr = s32 + S, *gd = s32 + 2 * S, *ap = s32 + 3 * S, *dp = s32 + 5 * S;
    lo_stage<double>(x, q, s64, S, t, nthr);
    for (int f = t; f <= n; f += nthr) {   // the slots this thread staged
        const int o = x.lo_slot[f];
        pl[o] = (float)PL[o];
        pr[o] = (float)PR[o];
        gd[o] = (float)GD[o];
        if (f < n) {
            ap[o] = (float)Ap[o];
            dp[o] = (float)Dp[o];
        }
    }
    __syncthreads();
    tri_solve<float>(s32, s32 + 6 * S, n, y);   // x0 in dp
    for (int i = t; i < n; i += nthr) X0[x.lo_slot[i]] = (double)dp[x.lo_slot[i]];
    __syncthreads();
    for (int step = 0; step < kLoRefine; ++step) {
        // the correction system: the same matrix (its FP32 diagonal parts again: the
        // elimination overwrote them), the residual of row i as right-hand side, no face
        // sources:
        //   r = (Dp_i - GD_{i+1} + GD_i) - (Ap_i + PL_{i+1} + PR_i) x_i
        //       + PL_i x_{i-1} + PR_{i+1} x_{i+1}
        for (int i = t; i <= n; i += nthr) {
            const int o = x.lo_slot[i];
            gd[o] = 0.f;
            if (i == n) break;
            const int on = x.lo_slot[i + 1];
            const double di = Ap[o] + PL[on] + PR[o];
            const double rh = Dp[o] - GD[on] + GD[o];
            double r = rh - di * X0[o];
            if (i > 0) r = fma(PL[o], X0[x.lo_slot[i - 1]], r);
            if (i < n - 1) r = fma(PR[on], X0[on], r);
            ap[o] = (float)Ap[o];
            dp[o] = (float)r;
        }
        __syncthreads();
        tri_solve<float>(s32, s32 + 6 * S, n, y);   // the correction in dp
        for (int i = t; i < n; i += nthr) X0[x.lo_slot[i]] += (double)dp[x.lo_slot[i]];
        __syncthreads();
    }
    for (int i = t; i < n; i += nthr) Dp[x.lo_slot[i]] = X0[x.lo_slot[i]];
    __syncthreads();
    lo_outputs_cta<double>(x, q, s64, S, 0);
}

// One system per CTA (128 to 512 threads): all stage the rows (global loads and the face
// coefficients) and form and store the outputs, the first P eliminate.
template <typename R>
__device__ void lo_solve_body(const LoCtx &x, int q)
{
    if constexpr (std::is_same<R, float>::value) {   // FP32 group solves: refined to FP64 accuracy
        lo_solve_refined(x, q);
        return;
    }
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R *sm = reinterpret_cast<R *>(smem_raw);
    int ks = 0;
    if (x.nx >= 2) {
        const TriLayout y = tri_layout(x.nx);
        if constexpr (is_pair<R>) ks = lo_stage_pair(x, q, sm, y.S);
        else lo_stage<R>(x, q, sm, y.S, threadIdx.x, blockDim.x);
        __syncthreads();
        tri_solve<R>(sm, sm + 6 * y.S, x.nx, y);
        lo_outputs_cta<R>(x, q, sm, y.S, ks);
        return;
    }
    if constexpr (is_pair<R>) {   // one cell: one thread (the source scale from every thread)
        __shared__ int kw[32];
        int m = lo_src_exp(x, q, threadIdx.x, blockDim.x);
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((threadIdx.x & 31) == 0) kw[threadIdx.x >> 5] = m;
        __syncthreads();
        m = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = max(m, kw[w]);
        ks = (m == 0) ? 0 : m - 1023;
    }
    if (threadIdx.x == 0) lo_one_cell<R>(x, q, ks);
}

// The exponentials' tables in shared memory by the block (ends with a barrier).
__device__ inline Mx stage_exp(const OpacityArgs &a, double *e2, fpair *e2p)
{
    if (threadIdx.x < 32) {
        e2[threadIdx.x] = a.e2[threadIdx.x];
        e2p[threadIdx.x] = fpair(a.e2[threadIdx.x]);
    }
    __syncthreads();
    return Mx{e2, a.ec};
}
// where an evaluation takes its per-cell terms: 1, formed here (k_cell_terms did not run)
enum { OP_NONE = 0, OP_ARRAYS = 1, OP_HERE = 2 };
// the terms of a cell that the tabulated evaluation reads, and no more of CellVals: a lane
// keeps them over its members
template <bool kPair>
struct OpacCell {
    double t, iT, iT3, kET;
    float tf;
    int m;
};
template <>
struct OpacCell<true> {
    CellPair cp;
    float tf;
    int m;
};
template <bool kPair>
__device__ inline OpacCell<kPair> cell_terms(const OpacityArgs &a, int op, int i)
{
    const CellVals v = op == OP_HERE ? cell_vals(a, i) : cell_arrays(a).get(i);
    OpacCell<kPair> c;
    if constexpr (kPair) {
        c.cp = op == OP_HERE ? cell_pair(a, i, v) : cell_pair_at(a, i);
    } else {
        c.t = v.t; c.iT = v.iT; c.iT3 = v.iT3; c.kET = v.kET;
    }
    c.tf = v.tf;
    c.m = v.m;
    return c;
}
// sigma_E, e_g, sigma_R of group g in cell i with terms c; kIn: the cell is inside the tables
template <bool kPair, bool kIn = false>
__device__ inline OpacVals cell_opacities(const OpacityArgs &a, int g, int i, const OpacCell<kPair> &c,
                                          const Mx &mx, const fpair *e2p)
{
    if (!kIn && c.m < 0) {   // outside the tables: the temperature and its powers again (cell_vals' operations)
        const double T = a.T[i], iT = rcp64(T);
        return opacity_direct(a.edges[g], a.edges[g + 1], a.s, T, iT, iT * iT * iT, a.ser, mx);
    }
    if constexpr (kPair) {
        fpair sg, em, sR;
        int k;
        opacity_vals_pair(a, g, c.m, c.tf, c.cp, e2p, sg, em, k, sR);
        return OpacVals{pr_join(sg, 0), pr_join(em, k), pr_join(sR, 0)};
    } else {
        CellVals v;
        v.t = c.t; v.iT = c.iT; v.iT3 = c.iT3; v.kET = c.kET; v.tf = c.tf; v.m = c.m;
        return opacity_vals(a, g, v, mx);
    }
}
// the opacities of group g in every cell by the CTA, into the fine grid's arrays (ends with
// a barrier)
template <bool kPair>
__device__ void group_opacities(const OpacityArgs &a, int op, int g)
{
    __shared__ double e2[32];
    __shared__ fpair e2p[32];
    const Mx mx = stage_exp(a, e2, e2p);
    for (int i = threadIdx.x; i < a.nx; i += blockDim.x) {
        const OpacVals o = cell_opacities<kPair>(a, g, i, cell_terms<kPair>(a, op, i), mx, e2p);
        const size_t idx = (size_t)g * a.nx + i;
        a.sigE[idx] = o.sg;
        a.emis[idx] = o.em;
        a.sigR[idx] = o.sR;
    }
    __syncthreads();
}

// T threads.  128: 7 CTAs per SM (at most 72 registers), one wave of 1064 holds every group
// of a 1024-group level.  512 and 256: levels of few groups, whose staging and outputs (loads
// and ~60 operations per face) would be a chain of n/128 faces per thread; launch_lo_solve.
template <typename R, int T>
__global__ void __launch_bounds__(T, T == 128 ? 7 : T == 256 ? 3 : 1) k_lo_solve(LoCtx x)
{
    griddep_wait();
    if (x.gate && *x.gate) return;   // the phase's inner loop has ended
    lo_solve_body<R>(x, blockIdx.x);
}
// a fine grid whose opacities at a.T the CTA forms first, its own group's: a launch and a pass
// over the fields less than k_opacity and k_lo_solve (1024 groups x 500 cells FP64 84 us for
// both against 61 + 33; pair 40 against 32 + 15; 17 groups x 60 cells 12 against 9 + 6 + 3
// with k_cell_terms).  A kernel of its own: in one kernel the pair form's plain solve was 30%
// slower.
template <typename R, int T>
__global__ void __launch_bounds__(T, T == 128 ? 7 : T == 256 ? 3 : 1) k_lo_solve_opac(LoCtx x, OpacityArgs a,
                                                                                    int op)
{
    griddep_wait();
    if (x.gate && *x.gate) return;
    group_opacities<is_pair<R>>(a, op, blockIdx.x);
    lo_solve_body<R>(x, blockIdx.x);
}

template <typename R>
__global__ void __launch_bounds__(128) k_lo_solve_b(const int *__restrict__ meta, int N,
                                                    const LoCtx *__restrict__ xs)
{
    for (int b = blockIdx.x;; b += gridDim.x) {
        int s, bx, by;
        if (!bdecode(meta, N, b, s, bx, by)) break;
        const LoCtx x = xs[s];
        lo_solve_body<R>(x, bx);
        __syncthreads();
    }
}

// Per-cell terms of the grey Newton step (Sec. 5, eqs. eb-Gamma and f-derivative-d): from the
// grey opacity sig*, Q* = 2 e* and the group energy sum Esum of cell i at T*, the
// absorption w c sig*, the source w Q* - (1 - w) c_v (T* - Told)/dt and 1/Lambda.  Called
// by the grey kernel on the grey level's arrays, or by the restriction to that level on
// the same values it writes there (the same operations, the same bits).
// In two parts: what does not need the restricted sums (base = c_v/dt + Q'(T*), mT = c_v (T* -
// Told)/dt, rdT = 1/(T* - T_prev) or 0 without a secant), and the rest.
struct GreyNewtonIn {   // the cell's inputs of the first part
    double Ts, Told, Tp, sp;
};
__device__ inline GreyNewtonIn grey_newton_load(const GreyArgs &a, int have_prev, int i)
{
    GreyNewtonIn c;
    c.Ts = a.Tstar[i];
    c.Told = a.Told[i];
    c.Tp = have_prev ? a.T_prev[i] : c.Ts;
    c.sp = have_prev ? a.sig_prev[i] : 0.0;
    return c;
}
__device__ inline void grey_newton_first(const GreyArgs &a, const GreyNewtonIn &c, double &base,
                                         double &mT, double &rdT)
{
    const double cvdt = a.cvdt;
    const double k54 = a.k54;
    const double Ts = c.Ts;
    double dQ = k54;   // first edge at 0: (1 + x) e^{-x} = 1
    if (a.nu_first != 0.0 || !isinf(a.nu_last)) {
        const double iTs = rcp64(Ts);
        if (a.nu_first != 0.0) {
            const double x1 = a.nu_first * iTs;
            dQ = k54 * (1.0 + x1) * texp(-x1, a.e2, a.ec);
        }
        if (!isinf(a.nu_last)) {
            const double xL = a.nu_last * iTs;
            dQ -= k54 * (1.0 + xL) * texp(-xL, a.e2, a.ec);
        }
    }
    // T* != T_prev on the encodings (positive finite values: integer instructions, not an
    // FP64 compare); across grids only where |dT| is far above rounding (relative noise ~ eps
    // T/|dT|)
    rdT = 0.0;
    const bool moved = __double_as_longlong(Ts) != __double_as_longlong(c.Tp);
    const bool cut = __double_as_longlong(a.secant_cut) != 0ll;
    if (moved && (!cut || fabs(Ts - c.Tp) > a.secant_cut * Ts)) rdT = rcp64(Ts - c.Tp);
    base = cvdt + dQ;
    mT = cvdt * (Ts - c.Told);
}
__device__ inline void grey_newton_rest(const GreyArgs &a, double base, double mT, double rdT,
                                        double sp, double sig, double Q, double Esum, double &sa,
                                        double &ss, double &sL)
{
    double L = base;
    if (__double_as_longlong(rdT) != 0ll) L = base - kC * ((sig - sp) * rdT) * Esum;
    if (L < 0.5 * base) L = 0.5 * base;
    const double iL = rcp64(L);
    const double w = a.cvdt * iL;
    sa = w * kC * sig;
    ss = w * Q - (1.0 - w) * mT;
    sL = iL;
}

// ---- restriction (eqs. coeff-gamma, g-notation, eta-gamma / coeff-Gamma, g2G-notation,
// eta-Gamma, and the discrete compensation of eq. mloqd-d-gamma) ----
//
// One kernel per restriction.  Every sum over the members of a coarse group is an FP64
// operation, and GB300's FP64 pipe (a warp-wide operation holds its sub-partition's pipe for
// 64 cycles or more) bounds the kernel, so the split is by FP64 operations:
//   - a lane owns an extended position j = -1 .. n_x: cell j and face j, with the boundary
//     energies as "cells" -1 and n_x.  A warp covers 31 faces and the cell before its first
//     (lane 0), so that a face's sums of E_L and E_R are the cell sums of two neighbouring
//     lanes: no FP64 operation of their own.  A member's E_L is a second load: a shuffle
//     per member occupies the FP64 pipe as well (counters; 166 against 144 us below);
//   - one pass: the compensation is xi = dx (sum sigR F - sigR-bar sum F) + c (sum etaR E_R -
//     sum etaL E_L), equal to the two-pass sum up to rounding relative to the sigR dx F
//     terms.  12 operations per member and position (4 for the cell, 8 for the face), 2 more
//     for Eold and Fold where the target does not hold this step's sums yet, 2 more for the
//     compensation of a coarse source;
//   - the boundary means are the work of blocks of their own (bx = nt: 16 lanes are the 2
//     sides x 8 sums), not a second branch of the position blocks at the two ends;
//   - a quotient is a reciprocal and one residual correction (rquot), 6 operations.
// Modes (restrict_plan), one CTA = 4 warps, one per sub-partition:
//   0  a warp takes a whole coarse group (few members, many groups);
//   1  a CTA takes kc members of a coarse group, each warp every fourth; with more than one
//      chunk the partial sums go to scratch and the CTA that arrives last at a position
//      tile (a ticket) adds the chunks in a fixed order and forms the coefficients: no
//      second launch.
// Measured (warm, with the former two launches' times for the same work): 1024 members to
// the grey level, 500 cells 27.5 us (35.3 + 8.3); 4096 members to a few groups, 1000 cells
// 144 us (163 + 50; the FP64 pipe's own time is 106 us); 1024 to 256 groups, 500 cells 31 us
// (38); 256 members, 10 cells 13 us (21.6 + 5.6).
constexpr int kRV = 12;   // sums per position: the order of restrict_member's v
enum { R_PHI, R_SIG, R_EMIS, R_E, R_SW, R_W, R_SF, R_F, R_EOLD, R_FOLD, R_ETAR, R_ETAL };
constexpr int kRTile = 31;          // faces per position tile
constexpr int kRTickets = 2432;     // ints at the head of the scratch (nt * n_to < 1216 there)
constexpr int kRHead = kRTickets / 2;   // doubles

// sums over members p = p0, p0 + step, .. < pe of lane position i (clamped by the caller);
// kFine: S is the fine grid; kOld: Eold and Fold are summed too
template <bool kFine, bool kOld>
__device__ inline void restrict_members(const RestrictCtx &x, int p0, int pe, int step, int i,
                                        double (&v)[kRV])
{
    const Level &S = x.S;
    const int nx = x.nx;
    const int ic = min(max(i, 0), nx - 1);
    const size_t cs = (size_t)p0 * nx + ic, cd = (size_t)step * nx;
    const size_t fs = (size_t)p0 * (nx + 1) + max(i, 0), fd = cd + step;
    const bool in = i >= 0 && i < nx;
    const double *Ep = in ? S.E + cs : (i < 0 ? S.Eb0 : S.EbX) + p0;
    const size_t Ed = in ? cd : (size_t)step;
    const double *Lp = i > 0 ? S.E + (size_t)p0 * nx + i - 1 : S.Eb0 + p0;   // E left of face i
    const size_t Ld = i > 0 ? cd : (size_t)step;
    const double *ph = S.phi + cs, *sg = S.sig + cs, *em = S.emis + cs, *Fp = S.F + fs;
    const double *sb = S.sigR + (kFine ? cs : fs);
    const double *sa = kFine ? S.sigR + (size_t)p0 * nx + (in ? max(i - 1, 0) : ic) : nullptr;
    double wa = 0.0, wb = 1.0;
    if (kFine && i > 0) {   // the face opacity's dx-weighted mean; face n_x: its cell alone
        wa = i < nx ? x.h[i - 1] * x.ihf[i] : 1.0;
        wb = i < nx ? x.h[i] * x.ihf[i] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < kRV; ++k) v[k] = 0.0;
#pragma unroll 2
    for (int p = p0; p < pe; p += step) {
        const double E = *Ep, EL = *Lp, F = *Fp;
        v[R_PHI] = fma(*ph, E, v[R_PHI]);
        v[R_SIG] = fma(*sg, E, v[R_SIG]);
        v[R_EMIS] += *em;
        v[R_E] += E;
        double sR = *sb;
        if (kFine) sR = fma(wa, *sa, wb * sR);
        // |F| weight with a floor 1e-6 c E-bar: groups in local equilibrium carry
        // rounding-noise fluxes that must not decide the mean
        const double w = fma(0.5e-6 * kC, EL + E,
                             __longlong_as_double(__double_as_longlong(F) & 0x7fffffffffffffffll));
        v[R_SW] = fma(sR, w, v[R_SW]);
        v[R_W] += w;
        v[R_SF] = fma(sR, F, v[R_SF]);
        v[R_F] += F;
        if (!kFine) {
            const size_t fp = (size_t)p * (nx + 1) + max(i, 0);
            v[R_ETAR] = fma(S.etaR[fp], E, v[R_ETAR]);
            v[R_ETAL] = fma(S.etaL[fp], EL, v[R_ETAL]);
        }
        if (kOld) {
            v[R_EOLD] += S.Eold[(size_t)p * nx + ic];
            v[R_FOLD] += S.Fold[(size_t)p * (nx + 1) + max(i, 0)];
        }
        Ep += Ed; Lp += Ld; ph += cd; sg += cd; em += cd; Fp += fd;
        sb += kFine ? cd : fd;
        if (kFine) sa += cd;
    }
}
__device__ inline void restrict_members(const RestrictCtx &x, int p0, int pe, int step, int i,
                                        double (&v)[kRV])
{
    if (x.S.fine) {
        if (x.skip_old) restrict_members<true, false>(x, p0, pe, step, i, v);
        else restrict_members<true, true>(x, p0, pe, step, i, v);
    } else {
        if (x.skip_old) restrict_members<false, false>(x, p0, pe, step, i, v);
        else restrict_members<false, true>(x, p0, pe, step, i, v);
    }
}

// The same over a fine source whose opacities at a.T are formed here, per member and cell,
// instead of read (and stored for the other readers of the fine grid's arrays): the lane's
// per-cell terms stay in registers over the members.  A face's left opacity is the lane
// before's, through shared memory (xch: two rows of 33 for the warp, by turns).  The halo
// lane stores its cell's sigma_R too (the value that the tile before stores there): the
// plain mean of a face without flux weight (restrict_face) reads the members' sigma_R back,
// at the tile's first face the halo cell's, and nothing orders it after another tile's store.
// kFix: the sums that do not depend on the opacities (kFixed) are the caller's, from an
// earlier visit of the cycle.  kIn: every lane's cell is inside the tables.
template <bool kOld, bool kPair, bool kFix, bool kIn>
__device__ inline void restrict_members_opac(const RestrictCtx &x, const OpacityArgs &a, int op,
                                             const OpacCell<kPair> &cc, double (*xch)[33],
                                             const Mx &mx, const fpair *e2p, int p0, int pe,
                                             int step, int i, double (&v)[kRV])
{
    const Level &S = x.S;
    const int nx = x.nx, lane = threadIdx.x & 31;
    const int ic = min(max(i, 0), nx - 1);
    const size_t cd = (size_t)step * nx;
    size_t c = (size_t)p0 * nx + ic;
    const bool in = i >= 0 && i < nx, own = in && lane > 0;
    const double *Ep = in ? S.E + c : (i < 0 ? S.Eb0 : S.EbX) + p0;
    const size_t Ed = in ? cd : (size_t)step;
    const double *Lp = i > 0 ? S.E + (size_t)p0 * nx + i - 1 : S.Eb0 + p0;   // E left of face i
    const size_t Ld = i > 0 ? cd : (size_t)step;
    size_t f = (size_t)p0 * (nx + 1) + max(i, 0);
    double wa = 0.0, wb = 1.0;
    if (i > 0) {   // the face opacity's dx-weighted mean; face n_x: its cell alone
        wa = i < nx ? x.h[i - 1] * x.ihf[i] : 1.0;
        wb = i < nx ? x.h[i] * x.ihf[i] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < kRV; ++k) v[k] = 0.0;
    int par = 0;
    for (int p = p0; p < pe; p += step) {
        const double E = *Ep, EL = *Lp, F = S.F[f];
        double ph = 0.0;
        if (!kFix) ph = S.phi[c];
        const OpacVals o = cell_opacities<kPair, kIn>(a, p, ic, cc, mx, e2p);
        xch[par][lane] = o.sR;
        if (in) S.sigR[c] = o.sR;
        if (own) {
            S.sig[c] = o.sg;
            S.emis[c] = o.em;
        }
        __syncwarp();
        const double left = xch[par][max(lane - 1, 0)];
        par ^= 1;
        const double sR = fma(wa, left, wb * o.sR);
        v[R_SIG] = fma(o.sg, E, v[R_SIG]);
        v[R_EMIS] += o.em;
        if (!kFix) {
            v[R_PHI] = fma(ph, E, v[R_PHI]);
            v[R_E] += E;
        }
        const double w = fma(0.5e-6 * kC, EL + E,
                             __longlong_as_double(__double_as_longlong(F) & 0x7fffffffffffffffll));
        v[R_SW] = fma(sR, w, v[R_SW]);
        v[R_SF] = fma(sR, F, v[R_SF]);
        if (!kFix) {
            v[R_W] += w;
            v[R_F] += F;
        }
        if (kOld) {
            v[R_EOLD] += S.Eold[c];
            v[R_FOLD] += S.Fold[f];
        }
        Ep += Ed; Lp += Ld; c += cd; f += cd + step;
    }
}

// The form for a warp with a cell outside the tables, out of line: the direct integrals' call
// in the loop would cost every lane 32 to 48 registers.
template <bool kOld, bool kPair, bool kFix>
__device__ __noinline__ void restrict_members_direct(const RestrictCtx &x, const OpacityArgs &a,
                                                     int op, double (*xch)[33], const double *e2,
                                                     const fpair *e2p, int p0, int pe, int step,
                                                     int i, double *u)
{
    double v[kRV];
    const OpacCell<kPair> cc = cell_terms<kPair>(a, op, min(max(i, 0), x.nx - 1));
    restrict_members_opac<kOld, kPair, kFix, false>(x, a, op, cc, xch, Mx{e2, a.ec}, e2p, p0, pe, step,
                                                    i, v);
    for (int k = 0; k < kRV; ++k) u[k] = v[k];
}

// the E-weighted cell means of coarse group P at cell i
__device__ inline void restrict_cell(const RestrictCtx &x, int P, int i, double sphi, double ssig,
                                     double sE, double &sg)
{
    const Level &S = x.S;
    const int nx = x.nx;
    const size_t c = (size_t)P * nx + i;
    double ph;
    if (sE != 0.0) {
        ph = rquot(sphi, sE);
        sg = rquot(ssig, sE);
    } else {   // no energy in the coarse group: plain means of the members
        ph = sg = 0.0;
        for (int p = P * x.r; p < (P + 1) * x.r; ++p) {
            ph += S.phi[(size_t)p * nx + i];
            sg += __ldcg(S.sig + (size_t)p * nx + i);   // of this launch, perhaps
        }
        ph = rquot(ph, (double)x.r);
        sg = rquot(sg, (double)x.r);
    }
    x.T.phi[c] = ph;
    x.T.sig[c] = sg;
}

// the copied sums of coarse group P at position i
__device__ inline void restrict_sums(const RestrictCtx &x, int P, int i, double semis, double sE,
                                     double sEold, double sFold)
{
    const int nx = x.nx;
    if (i < nx) {
        const size_t c = (size_t)P * nx + i;
        x.T.emis[c] = semis;
        x.T.Esum[c] = sE;
        if (!x.skip_old) x.T.Eold[c] = sEold;
    }
    if (!x.skip_old) x.T.Fold[(size_t)P * (nx + 1) + i] = sFold;
}

// the face opacity and compensation of coarse group P at face i; sER, sEL: sums of E on
// either side
__device__ inline void restrict_face(const RestrictCtx &x, int P, int i, double sSW, double sW,
                                     double sSF, double sF, double sER, double sEL, double eR,
                                     double eL)
{
    const Level &S = x.S;
    const int nx = x.nx, nf = nx + 1;
    const double dxf = (i == 0) ? 0.5 * x.h[0] : (i == nx) ? 0.5 * x.h[nx - 1]
                                            : 0.5 * (x.h[i - 1] + x.h[i]);
    double sRP;
    if (sW != 0.0) {
        sRP = rquot(sSW, sW);
    } else {   // no flux weight: plain mean of the members' face opacities
        sRP = 0.0;
        for (int p = P * x.r; p < (P + 1) * x.r; ++p) {
            if (S.fine) {
                const double *sc = S.sigR + (size_t)p * nx;
                sRP += (i == 0) ? __ldcg(sc) : (i == nx) ? __ldcg(sc + nx - 1)
                       : (__ldcg(sc + i - 1) * x.h[i - 1] + __ldcg(sc + i) * x.h[i]) * x.ihf[i];
            } else {
                sRP += S.sigR[(size_t)p * nf + i];
            }
        }
        sRP = rquot(sRP, (double)x.r);
    }
    double xi = dxf * fma(-sRP, sF, sSF);
    if (!S.fine) xi = fma(kC, eR - eL, xi);
    const size_t f = (size_t)P * nf + i;
    const double side = xi > 0.0 ? sER : sEL;
    double eta = 0.0;
    if (xi != 0.0 && side != 0.0) eta = rquot(fabs(xi), kC * side);
    x.T.sigR[f] = sRP;
    x.T.etaR[f] = xi > 0.0 ? eta : 0.0;
    x.T.etaL[f] = xi < 0.0 ? eta : 0.0;
}

// lane side * 8 + k (< 16): sum k of the boundary means of one side over the members
__device__ inline double restrict_boundary(const RestrictCtx &x, int p0, int pe, int step, int l)
{
    const Level &S = x.S;
    const int side = l >> 3, k = l & 7;
    const double *ph = side ? S.phibX : S.phib0, *Eb = side ? S.EbX : S.Eb0,
                 *Cb = side ? S.CX : S.C0, *Ein = side ? S.EinX : S.Ein0,
                 *Fin = side ? S.FinX : S.Fin0;
    // phi Eb, phi, Eb, C Eo, C, Eo, Ein, Fin with Eo = Eb - Ein
    const double *pa = k < 2 ? ph : (k == 2 || k == 5) ? Eb : k < 5 ? Cb : k == 6 ? Ein : Fin;
    double s = 0.0;
    for (int p = p0; p < pe; p += step) {
        double a = pa[p], b = 1.0;
        if (k == 0) b = Eb[p];
        if (k == 3) b = Eb[p] - Ein[p];
        if (k == 5) a -= Ein[p];
        s = fma(a, b, s);
    }
    return s;
}
// the boundary means of coarse group P from the 16 sums on lanes 0 .. 15 of a warp
__device__ inline void restrict_boundary_out(const RestrictCtx &x, int P, int lane, double s)
{
    const int side = (lane >> 3) & 1, k = lane & 7;
    const double den = __shfl_sync(0xffffffffu, s, side * 8 + (k < 3 ? 2 : 5));
    const double pl = __shfl_sync(0xffffffffu, s, side * 8 + (k < 3 ? 1 : 4));
    if (lane >= 16) return;
    const Level &T = x.T;
    if (k == 0 || k == 3) {
        const double m = den != 0.0 ? rquot(s, den) : rquot(pl, (double)x.r);
        (k == 0 ? (side ? T.phibX : T.phib0) : (side ? T.CX : T.C0))[P] = m;
    }
    if (k == 6) (side ? T.EinX : T.Ein0)[P] = s;
    if (k == 7) (side ? T.FinX : T.Fin0)[P] = s;
}

// The sums that a later visit of the same grid in the same cycle would form again from the
// same fine solution (sum phi E, sum E, sum of the weights, sum F): x.fixed 1 stores them in
// x.fix ([n_to][4][32 nt]), 2 takes them from there.
__device__ inline int fixed_index(int k)
{
    return k == R_PHI ? 0 : k == R_E ? 1 : k == R_W ? 2 : k == R_F ? 3 : -1;
}
__device__ inline void restrict_fixed(const RestrictCtx &x, int P, int bx, int lane, int k, double &v)
{
    const int j = fixed_index(k);
    if (!x.fixed || j < 0) return;
    double *p = x.fix + ((size_t)P * 4 + j) * x.nt * 32 + bx * 32 + lane;
    if (x.fixed == 1) *p = v;
    else v = *p;
}

// last arrival of `n` CTAs at ticket t (which it resets): the partial sums written before
// by the others are visible to the CTA that gets true
__device__ inline bool restrict_last(int *t, int n)
{
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(t, 1) == n - 1;
        if (last) *t = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// block 128; grid (nt + 1, ceil(n_to / 4)) in mode 0, (nt + 1, n_to * nchunk) in mode 1;
// members(p0, pe, step, i, v): the sums over members
template <class Members>
__device__ void restrict_body(const RestrictCtx &x, int bx, int by, const Members &members)
{
    __shared__ double red[4][kRV][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nx = x.nx;
    const bool many = x.mode == 0;
    const int P = many ? by * 4 + warp : by / x.nchunk;
    const int ch = many ? 0 : by - P * x.nchunk;
    const int pb = P * x.r + ch * x.kc;
    const int pe = min(pb + x.kc, (P + 1) * x.r);

    if (bx == x.nt) {   // ---- boundary means ----
        const int l = lane & 15, half = lane >> 4;
        if (many) {
            if (P >= x.n_to) return;
            double s = restrict_boundary(x, pb + half, pe, 2, l);
            s += __shfl_xor_sync(0xffffffffu, s, 16);
            restrict_boundary_out(x, P, lane, s);
            return;
        }
        double *rb = &red[0][0][0];   // [8 slices][16]
        rb[(warp * 2 + half) * 16 + l] = restrict_boundary(x, pb + warp * 2 + half, pe, 8, l);
        __syncthreads();
        double s = 0.0;
        if (warp == 0)
            for (int k = 0; k < 8; ++k) s += rb[k * 16 + l];
        if (x.nchunk > 1) {
            if (threadIdx.x < 16) x.bpart[(size_t)by * 16 + l] = s;
            if (!restrict_last(x.ticket + P * (x.nt + 1) + bx, x.nchunk)) return;
            s = 0.0;
            if (warp == 0)
                for (int c = 0; c < x.nchunk; ++c)
                    s += __ldcg(x.bpart + ((size_t)P * x.nchunk + c) * 16 + l);
        }
        if (warp == 0) restrict_boundary_out(x, P, lane, s);
        return;
    }

    const int i = bx * kRTile - 1 + lane;   // extended position; lane 0 is the halo
    const bool face = lane > 0 && i <= nx, cell = lane > 0 && i < nx;
    double v[kRV];
    if (many) {
        if (P >= x.n_to) return;
        members(pb, pe, 1, min(i, nx), v);
#pragma unroll
        for (int k = 0; k < kRV; ++k) restrict_fixed(x, P, bx, lane, k, v[k]);
        const double sEL = __shfl_up_sync(0xffffffffu, v[R_E], 1);
        double sg;
        if (cell) restrict_cell(x, P, i, v[R_PHI], v[R_SIG], v[R_E], sg);
        if (face) {
            restrict_sums(x, P, i, v[R_EMIS], v[R_E], v[R_EOLD], v[R_FOLD]);
            restrict_face(x, P, i, v[R_SW], v[R_W], v[R_SF], v[R_F], v[R_E], sEL, v[R_ETAR],
                          v[R_ETAL]);
        }
        return;
    }
    // the grey visit's Newton terms are formed with the cell means: their inputs early
    GreyNewtonIn nin{};
    if (x.newton && warp == 3 && cell) nin = grey_newton_load(x.ga, x.ga.have_prev, i);
    members(pb + warp, pe, 4, min(i, nx), v);
#pragma unroll
    for (int k = 0; k < kRV; ++k) red[warp][k][lane] = v[k];
    __syncthreads();
    // the warps' partials, value k by warp k % 4 (the additions spread over the four FP64
    // pipes), then the chunks' in the same split
    const size_t np = (size_t)x.nt * 32;
    double *part = x.part + (size_t)by * kRV * np + bx * 32 + lane;
    const int kend = x.S.fine ? R_ETAR : kRV;   // a fine source has no compensation
    for (int k = warp; k < kend; k += 4) {
        if (x.skip_old && (k == R_EOLD || k == R_FOLD)) continue;
        if (x.fixed == 2 && fixed_index(k) >= 0) continue;
        const double s = (red[0][k][lane] + red[1][k][lane]) + (red[2][k][lane] + red[3][k][lane]);
        if (x.nchunk > 1) part[k * np] = s;
        else red[0][k][lane] = s;
    }
    if (x.nchunk > 1) {
        if (!restrict_last(x.ticket + P * (x.nt + 1) + bx, x.nchunk)) return;
        const double *all = x.part + (size_t)P * x.nchunk * kRV * np + bx * 32 + lane;
        for (int k = warp; k < kend; k += 4) {
            if (x.skip_old && (k == R_EOLD || k == R_FOLD)) continue;
            if (x.fixed == 2 && fixed_index(k) >= 0) continue;
            double s = 0.0;
#pragma unroll 8
            for (int c = 0; c < x.nchunk; ++c) s += __ldcg(all + ((size_t)c * kRV + k) * np);
            red[0][k][lane] = s;
        }
    }
    if (x.fixed)   // each value by the warp that summed it
        for (int k = warp; k < kend; k += 4) restrict_fixed(x, P, bx, lane, k, red[0][k][lane]);
    __syncthreads();
    const double(*sv)[32] = red[0];
    // the coefficients by four warps; warp 3 forms the first part of the Newton terms for warp 0
    if (warp == 0) {
        double sg = 0.0;
        if (cell) restrict_cell(x, P, i, sv[R_PHI][lane], sv[R_SIG][lane], sv[R_E][lane], sg);
        if (x.newton) {
            asm volatile("bar.sync 1, 64;" ::: "memory");
            if (cell) {
                double sa, ss, sL;
                grey_newton_rest(x.ga, red[1][0][lane], red[1][1][lane], red[1][2][lane],
                                 red[1][3][lane], sg, 2.0 * sv[R_EMIS][lane], sv[R_E][lane], sa, ss,
                                 sL);
                x.pre[i] = sa;
                x.pre[nx + i] = ss;
                x.pre[2 * (size_t)nx + i] = sL;
            }
        }
    } else if (warp == 3) {
        if (x.newton) {
            double base = 0.0, mT = 0.0, rdT = 0.0;
            if (cell) grey_newton_first(x.ga, nin, base, mT, rdT);
            red[1][0][lane] = base;
            red[1][1][lane] = mT;
            red[1][2][lane] = rdT;
            red[1][3][lane] = nin.sp;
            asm volatile("bar.sync 1, 64;" ::: "memory");
        }
    } else if (warp == 1) {
        if (face)
            restrict_sums(x, P, i, sv[R_EMIS][lane], sv[R_E][lane], sv[R_EOLD][lane], sv[R_FOLD][lane]);
    } else if (warp == 2) {
        if (face)
            restrict_face(x, P, i, sv[R_SW][lane], sv[R_W][lane], sv[R_SF][lane], sv[R_F][lane],
                          sv[R_E][lane], sv[R_E][lane - 1], sv[R_ETAR][lane], sv[R_ETAL][lane]);
    }
}

// ---------------------------------------------------------------------------------------
// grey LOQD + MEB: one Newton step on the grey level (single CTA)
// ---------------------------------------------------------------------------------------

// Block-wide maxima of non-negative values on their IEEE encodings: for x >= 0 (and +inf)
// the order of the doubles is the unsigned order of their bit patterns, so the reduction
// runs on the integer pipes (a warp-wide FP64 max takes a sub-partition's FP64 pipe for 64
// cycles on GB300).  NaN maps to 0, the value fmax would keep.  red: kGreyRed slots, at
// least 32 per value; the maxima are returned to thread 0 (each warp reduces its lanes by
// shuffles, then warp 0 reduces the warps' results the same way).

__device__ inline unsigned long long nn_bits(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return ((b & 0x7fffffffffffffffull) > 0x7ff0000000000000ull) ? 0ull : b;
}

__device__ inline unsigned long long umax64(unsigned long long a, unsigned long long b)
{
    return a > b ? a : b;
}

__device__ inline void block_max_bits(unsigned long long (&v)[kGreyNV], unsigned long long *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < kGreyNV; ++k)
        for (int o = 16; o > 0; o >>= 1) v[k] = umax64(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < kGreyNV; ++k) red[k * 32 + warp] = v[k];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < kGreyNV; ++k) {
            unsigned long long r = (lane < nw) ? red[k * 32 + lane] : 0ull;
            for (int o = 16; o > 0; o >>= 1) r = umax64(r, __shfl_xor_sync(0xffffffffu, r, o));
            v[k] = r;
        }
    }
}

// the grey level's outputs from the solution: E, the face fluxes F_f = GD_f + PL_f E_{f-1} -
// PR_f E_f and the boundary face energies
__device__ void grey_outputs(const LoCtx &x, const double *sm, int S, int n)
{
    const double *PL = sm, *PR = sm + S, *GD = sm + 2 * S, *Dp = sm + 5 * S;
    for (int f = threadIdx.x; f <= n; f += blockDim.x) {
        const int o = x.lo_slot[f];
        double Fv = GD[o];
        if (f > 0) Fv += PL[o] * Dp[x.lo_slot[f - 1]];
        if (f < n) {
            x.L.E[f] = Dp[o];
            Fv -= PR[o] * Dp[o];
        }
        x.L.F[f] = Fv;
        if (f == 0) x.L.Eb0[0] = x.L.Ein0[0] + (Fv - x.L.Fin0[0]) * rcp64(kC * x.L.C0[0]);
        if (f == n) x.L.EbX[0] = x.L.EinX[0] + (Fv - x.L.FinX[0]) * rcp64(kC * x.L.CX[0]);
    }
}

// what the update of a cell reads (loaded before the solve, whose chain hides the latency)
struct GreyCell {
    double Ts, Told, sig, emis, Tc, Ec, Tp, Ep;
};
__device__ inline GreyCell grey_cell_load(const GreyArgs &a, const Level &g, int i)
{
    GreyCell c{};
    c.Ts = a.Tstar[i];
    c.Told = a.Told[i];
    c.sig = g.sig[i];
    c.emis = g.emis[i];
    if (a.want_norms) {
        c.Tc = a.Tcyc[i];
        c.Ec = a.Ecyc[i];
        c.Tp = a.Tphase[i];
        c.Ep = a.Ephase[i];
    }
    return c;
}

// T at cell i from the grey solution E; the bad-value test and the norms' terms
__device__ inline void grey_update_cell(const GreyArgs &a, const GreyCell &c, int i, double sL,
                                        double E, unsigned long long (&v)[kGreyNV])
{
    const unsigned long long kInfBits = 0x7ff0000000000000ull;
    const double cvdt = a.cvdt;
    const double Ts = c.Ts;
    const double T = Ts + (kC * c.sig * E - 2.0 * c.emis - cvdt * (Ts - c.Told)) * sL;
    a.T[i] = T;
    const long long tb = __double_as_longlong(T);
    const unsigned long long eb = (unsigned long long)__double_as_longlong(E) & 0x7fffffffffffffffull;
    // T > 0 and finite: sign clear, not zero, below the infinity encoding
    if (tb <= 0 || (unsigned long long)tb >= kInfBits || eb >= kInfBits) v[0] = 1ull;
    if (a.want_norms) {
        v[1] = umax64(v[1], nn_bits(fabs(T - c.Tc)));
        v[2] = umax64(v[2], nn_bits(fabs(T)));
        v[3] = umax64(v[3], nn_bits(fabs(E - c.Ec)));
        v[4] = umax64(v[4], nn_bits(fabs(E)));
        v[5] = umax64(v[5], nn_bits(fabs(T - c.Tp)));
        v[6] = umax64(v[6], nn_bits(fabs(E - c.Ep)));
        if (a.T_out) a.T_out[i] = T;
        if (a.Tcyc_out) a.Tcyc_out[i] = T;
        if (a.Ecyc_out) a.Ecyc_out[i] = E;
    }
}

__device__ void grey_body(const GreyCtx &x)
{
    const int have_prev = x.a.have_prev_dev ? *x.a.have_prev_dev : x.a.have_prev;
    extern __shared__ __align__(16) double gsm[];
    const int nx = x.lo.nx;
    double *sa = gsm;            // absorption w c sig*
    double *ss = sa + nx;        // source w Q* - (1-w) cv (T* - Told)/dt
    double *sL = ss + nx;        // 1 / Lambda
    double *red = sL + nx;       // [kGreyRed] block maxima
    double *wsm = red + kGreyRed;   // the solver's rows (TriLayout) and its 3 P values more
    const GreyArgs &a = x.a;
    const Level &g = x.lo.L;
    const int t = threadIdx.x;
    GreyCell mine{};             // the thread's first cell
    if (t < nx) mine = grey_cell_load(a, g, t);
    double bad_before = 0.0;     // what thread 0 will test at the end
    int cycles = 0;
    if (t == 0 && a.want_norms && a.ctl) {
        bad_before = a.flags[0];
        cycles = a.ctl[1];
    }
    for (int i = t; i < nx; i += blockDim.x) {
        if (a.pre) {   // formed by the restriction before this kernel
            sa[i] = a.pre[i];
            ss[i] = a.pre[nx + i];
            sL[i] = a.pre[2 * (size_t)nx + i];
        } else {
            const GreyNewtonIn c = grey_newton_load(a, have_prev, i);
            double base, mT, rdT;
            grey_newton_first(a, c, base, mT, rdT);
            grey_newton_rest(a, base, mT, rdT, c.sp, g.sig[i], 2.0 * g.emis[i], g.Esum[i], sa[i], ss[i], sL[i]);
        }
        a.sig_prev_out[i] = g.sig[i];
        a.T_prev_out[i] = a.Tstar[i];
    }
    __syncthreads();
    LoCtx lc = x.lo;
    lc.a_cell = sa;
    lc.s_cell = ss;
    const TriLayout y = tri_layout(nx);
    if (nx >= 2) {
        lo_stage<double>(lc, 0, wsm, y.S, t, blockDim.x);
        __syncthreads();
        tri_solve<double>(wsm, wsm + 6 * y.S, nx, y);
        grey_outputs(lc, wsm, y.S, nx);
    } else {
        if (t == 0) lo_one_cell<double>(lc, 0);
        __syncthreads();
    }
    const double *Esol = nx >= 2 ? wsm + 5 * (size_t)y.S : g.E;
    // v: bad flag, max|T - Tcyc|, max|T|, max|E - Ecyc|, max|E|, max|T - Tphase|,
    // max|E - Ephase| as non-negative encodings (flags[0 .. 6])
    unsigned long long v[kGreyNV] = {};
    for (int i = t; i < nx; i += blockDim.x) {
        if (i != t) mine = grey_cell_load(a, g, i);
        grey_update_cell(a, mine, i, sL[i], Esol[nx >= 2 ? lc.lo_slot[i] : i], v);
    }
    block_max_bits(v, reinterpret_cast<unsigned long long *>(red));
    if (t == 0) {
        if (v[0] != 0ull) a.flags[0] = 1.0;
        if (a.want_norms) {
            a.flags[1] = __longlong_as_double((long long)v[1]);
            a.flags[2] = __longlong_as_double((long long)v[2]);
            a.flags[3] = __longlong_as_double((long long)v[3]);
            a.flags[4] = __longlong_as_double((long long)v[4]);
            a.flags[5] = __longlong_as_double((long long)v[5]);
            a.flags[6] = __longlong_as_double((long long)v[6]);
            if (a.ctl) {   // inner-loop control: this cycle ran; does the phase go on?
                const double f1 = __longlong_as_double((long long)v[1]);
                const double f2 = __longlong_as_double((long long)v[2]);
                const double f3 = __longlong_as_double((long long)v[3]);
                const double f4 = __longlong_as_double((long long)v[4]);
                const bool conv_in = f1 <= a.eps_in * f2 && f3 <= a.eps_in * f4;
                a.ctl[1] = cycles + 1;
                // a bad temperature of this visit or of an earlier visit of the cycle
                if (v[0] != 0ull || bad_before != 0.0 || (!a.fixed && conv_in)) a.ctl[0] = 1;
            }
        }
    }
    if (a.have_prev_dev && t == 0) *a.have_prev_dev = 1;   // after the reduction's barriers
}

// out_i = sum_q X[q][i]: block of 256 threads = 32 cells x 8 rows; row y sums the groups
// q = y (mod 8) of its cell, then one row adds the 8 partials in row order (fixed order,
// deterministic).  A single pass over the groups per cell would leave 32 cells per warp
// and few warps per SM on a serial FP64 chain.
__device__ void group_sum_body(const GroupSumArgs &a, int bx)
{
    __shared__ double part[8][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int i = bx * 32 + tx;
    double s = 0.0;
    if (i < a.nx)
        for (int q = ty; q < a.n; q += 8) s += a.X[(size_t)q * a.nx + i];
    part[ty][tx] = s;
    __syncthreads();
    if (ty == (bx & 7) && i < a.nx) {
        double t = part[0][tx];
        for (int y = 1; y < 8; ++y) t += part[y][tx];
        a.out[i] = t;
    }
}

// entry points: the single-slab kernels pass blockIdx; the batched ones walk a work list
// (single-slab entry points: return at entry while the driver's gate is set)
__device__ inline void restrict_run(const RestrictCtx &x, int bx, int by)
{
    restrict_body(x, bx, by, [&](int p0, int pe, int step, int i, double (&v)[kRV]) {
        restrict_members(x, p0, pe, step, i, v);
    });
}
__global__ void __launch_bounds__(128) k_restrict(RestrictCtx x)
{
    griddep_wait();
    if (x.gate && *x.gate) return;
    restrict_run(x, blockIdx.x, blockIdx.y);
}
// fine source, its opacities at a.T formed on the way (a coarse visit: every fine group's
// opacities, then the restriction onto the visit's grid).  The pair form's evaluation runs on
// the FP32 pipes under the sums' FP64 operations; one launch and a pass over three fields
// less than k_opacity and k_restrict.  A member is a chain of table loads and dependent
// operations, so the warps in flight decide: a kernel per form of the sums, the direct
// integrals out of line and only the terms that the tables need kept per lane (168 -> 96
// registers, 3 -> 5 CTAs per SM).  4096 groups x 1000 cells pair 163 us on a later visit of a
// cycle (FP64 pipe's own time 93), 198 us with the sums of phi E, E and the weights too,
// against 89 + 147 for the two kernels and 203 / 260 at 168 registers; 6 CTAs at 80 registers
// 168 / 192, 4 at 128 169 / 213.  1024 groups x 500 cells FP64 (all of it on the FP64 pipe)
// 59 us against 34 + 29, 63 with 3 CTAs and 57 to 60 with 5.
template <bool kPair, bool kOld, bool kFix>
__global__ void __launch_bounds__(128, kPair ? 5 : 4)
    k_restrict_opac(const __grid_constant__ RestrictCtx x, const __grid_constant__ OpacityArgs a, int op)
{
    griddep_wait();
    if (x.gate && *x.gate) return;
    __shared__ double e2[32], xch[4][2][33];
    __shared__ fpair e2p[32];
    const Mx mx = stage_exp(a, e2, e2p);
    restrict_body(x, blockIdx.x, blockIdx.y, [&](int p0, int pe, int step, int i, double (&v)[kRV]) {
        double(*xc)[33] = xch[threadIdx.x >> 5];
        const OpacCell<kPair> cc = cell_terms<kPair>(a, op, min(max(i, 0), x.nx - 1));
        if (__all_sync(0xffffffffu, cc.m >= 0)) {
            restrict_members_opac<kOld, kPair, kFix, true>(x, a, op, cc, xc, mx, e2p, p0, pe, step, i, v);
        } else {
            double u[kRV];
            restrict_members_direct<kOld, kPair, kFix>(x, a, op, xc, e2, e2p, p0, pe, step, i, u);
#pragma unroll
            for (int k = 0; k < kRV; ++k) v[k] = u[k];
        }
    });
}
__global__ void __launch_bounds__(1024) k_grey(GreyCtx x)
{
    griddep_wait();
    if (x.lo.gate && *x.lo.gate) return;
    grey_body(x);
}
__global__ void __launch_bounds__(256) k_group_sum(GroupSumArgs a) { group_sum_body(a, blockIdx.x); }

#define TRT_BATCHED(name, Ctx, bounds, minb, call)                                            \
    __global__ void __launch_bounds__(bounds, minb) name(const int *__restrict__ meta, int N,        \
                                                   const Ctx *__restrict__ xs)                 \
    {                                                                                          \
        for (int b = blockIdx.x;; b += gridDim.x) {                                            \
            int s, bx, by;                                                                     \
            if (!bdecode(meta, N, b, s, bx, by)) break;                                        \
            const Ctx x = xs[s];                                                               \
            call;                                                                              \
            __syncthreads();                                                                   \
        }                                                                                      \
    }
// (6 CTAs per SM: unbounded, the argument block held in registers leaves 3 and 64 slabs'
// restriction to the grey level takes 25% longer)
TRT_BATCHED(k_restrict_b, RestrictCtx, 128, 6, restrict_run(x, bx, by))
TRT_BATCHED(k_grey_b, GreyCtx, 1024, 1, grey_body(x))
TRT_BATCHED(k_group_sum_b, GroupSumArgs, 256, 1, group_sum_body(x, bx))
#undef TRT_BATCHED

__global__ void __launch_bounds__(256) k_copy_b(const int *__restrict__ meta, int N,
                                                const CopyArgs *__restrict__ xs)
{
    for (int b = blockIdx.x;; b += gridDim.x) {
        int s, bx, by;
        if (!bdecode(meta, N, b, s, bx, by)) break;
        const CopyArgs c = xs[s];
        const long i = (long)bx * blockDim.x + threadIdx.x;
        if (i < c.n) c.dst[i] = c.src[i];
    }
}

}  // namespace

namespace {
// h/dt per cell and hf/(c dt) per face (for step length dt); with pc (the pair form) the
// same two rows of Problem::lopc
__global__ void k_lo_consts(int nx, const double *__restrict__ h, const double *__restrict__ hf,
                            double idt, double icdt, double *hidt, double *dxicdt, fpair *pc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const size_t n1 = (size_t)nx + 1;
    if (i < nx) {
        const double v = h[i] * idt;
        hidt[i] = v;
        if (pc) pc[4 * n1 + i] = fpair(v);
    }
    if (i <= nx) {
        const double v = hf[i] * icdt;
        dxicdt[i] = v;
        if (pc) pc[n1 + i] = fpair(v);
    }
}

// the step-independent rows of Problem::lopc ([8][nx+1] pairs): hf, fwl, fwr (faces), hc,
// h2, h (cells); once per handle
__global__ void k_lo_pair_consts(int nx, const double *__restrict__ h, const double *__restrict__ hf,
                                 const double *__restrict__ hc, const double *__restrict__ h2,
                                 const double *__restrict__ fwl, const double *__restrict__ fwr,
                                 fpair *pc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const size_t n1 = (size_t)nx + 1;
    if (i < nx) {
        pc[5 * n1 + i] = fpair(hc[i]);
        pc[6 * n1 + i] = fpair(h2[i]);
        pc[7 * n1 + i] = fpair(h[i]);
    }
    if (i <= nx) {
        pc[i] = fpair(hf[i]);
        pc[2 * n1 + i] = fpair(fwl[i]);
        pc[3 * n1 + i] = fpair(fwr[i]);
    }
}

}  // namespace

cudaError_t launch_lo_pair_consts(const Problem &p)
{
    if (!p.lopc) return cudaSuccess;
    k_lo_pair_consts<<<(p.nx + 1 + 255) / 256, 256, 0, p.stream>>>(
        p.nx, p.h, p.hf, p.hc, p.h2, p.fwl, p.fwr, reinterpret_cast<fpair *>(p.lopc));
    return cudaGetLastError();
}

cudaError_t ensure_lo_consts(Problem &p, double dt)
{
    if (p.lo_dt == dt) return cudaSuccess;
    k_lo_consts<<<(p.nx + 1 + 255) / 256, 256, 0, p.stream>>>(
        p.nx, p.h, p.hf, 1.0 / dt, 1.0 / (kC * dt), p.hidt, p.dxicdt,
        reinterpret_cast<fpair *>(p.lopc));
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) p.lo_dt = dt;
    return e;
}

// (the LO row constants hidt, dxicdt must be those of dt: ensure_lo_consts first)
LoCtx make_lo_ctx(const Problem &p, double dt, const Level &L)
{
    LoCtx x;
    x.nx = p.nx; x.dt = dt; x.icdt = 1.0 / (kC * dt); x.idt = 1.0 / dt; x.h = p.h; x.ihf = p.ihf;
    x.hf = p.hf;
    x.hc = p.hc; x.h2 = p.h2; x.fwl = p.fwl; x.fwr = p.fwr; x.hidt = p.hidt; x.dxicdt = p.dxicdt;
    x.lo_slot = p.lo_slot;
    x.pc = reinterpret_cast<const fpair *>(p.lopc);
    x.L = L;
    x.a_cell = nullptr; x.s_cell = nullptr;
    x.gate = p.gate;
    return x;
}

// doubles of restriction scratch: tickets, boundary partials, position partials
static size_t restrict_doubles(int nt, int n_to, int nchunk)
{
    return kRHead + (size_t)n_to * nchunk * (16 + (size_t)kRV * nt * 32);
}

template <typename R, int T>
static cudaError_t lo_launch(const LoCtx &x, const OpacityArgs &a, int op, unsigned nb, size_t sm,
                             cudaStream_t st)
{
    const auto go = [&](auto kern, auto... more) {
        const cudaError_t e = allow_smem((const void *)kern, sm);
        return e != cudaSuccess ? e : launch_pdl(kern, dim3(nb), dim3(T), sm, st, x, more...);
    };
    return op == OP_NONE ? go(k_lo_solve<R, T>) : go(k_lo_solve_opac<R, T>, a, op);
}

// The opacities of a fine level inside a low-order kernel: its arguments, and the per-cell
// terms from k_cell_terms or, where `ctas` CTAs cannot fill the GPU and a launch costs more
// than a logarithm more per cell and CTA (3 us against 2), formed in place.
static cudaError_t fused_opacity(const Problem &p, const double *T, const Level &fine, long ctas,
                                 OpacityArgs &a, int &op)
{
    a = OpacityArgs{};
    op = OP_NONE;
    if (!T) return cudaSuccess;
    a = make_opacity_args(p, T, fine.sig, fine.emis, fine.sigR, nullptr, nullptr, 0.0);
    op = ctas <= 152 && p.nx <= 128 ? OP_HERE : OP_ARRAYS;
    return op == OP_HERE ? cudaSuccess : launch_cell_terms(p, a);
}

cudaError_t launch_lo_solve(const Problem &p, double dt, const Level &L, const double *Topac)
{
    const LoCtx x = make_lo_ctx(p, dt, L);
    OpacityArgs a;
    int op;
    const cudaError_t eo = fused_opacity(p, Topac, L, L.n, a, op);
    if (eo != cudaSuccess) return eo;
    const size_t sm = lo_smem(p.precision, p.nx);
    // 512 threads where every group has an SM of its own, 256 where the level fits the GPU at
    // three CTAs per SM, if the rows are more than 128 threads take at once.  128 against more
    // threads, measured: 16 groups x 500 cells FP64 20.3, 14.7 us; 4 groups x 1000 cells pair
    // 49.6, 21.4; 256 groups x 1000 cells pair 51.3, 31.8
    const int T = p.nx <= 128 || L.n > 456 ? 128 : L.n <= 152 ? 512 : 256;
    const auto go = [&](auto zero) {
        using R = decltype(zero);
        return T == 512   ? lo_launch<R, 512>(x, a, op, L.n, sm, p.stream)
               : T == 256 ? lo_launch<R, 256>(x, a, op, L.n, sm, p.stream)
                          : lo_launch<R, 128>(x, a, op, L.n, sm, p.stream);
    };
    return lo_pair(p.precision) ? go(fpair()) : lo_fp32(p.precision) ? go(0.f) : go(0.0);
}

cudaError_t launch_lo_solve_b(int precision, const BatchSmem &bs, const int *meta, int N,
                              const LoCtx *xs, int grid, cudaStream_t st)
{
    const size_t sm = bs.lo;
    cudaError_t e;
    if (lo_pair(precision)) {
        e = allow_smem((const void *)k_lo_solve_b<fpair>, sm);
        if (e != cudaSuccess) return e;
        k_lo_solve_b<fpair><<<grid, 128, sm, st>>>(meta, N, xs);
    } else if (!lo_fp32(precision)) {
        e = allow_smem((const void *)k_lo_solve_b<double>, sm);
        if (e != cudaSuccess) return e;
        k_lo_solve_b<double><<<grid, 128, sm, st>>>(meta, N, xs);
    } else {
        e = allow_smem((const void *)k_lo_solve_b<float>, sm);
        if (e != cudaSuccess) return e;
        k_lo_solve_b<float><<<grid, 128, sm, st>>>(meta, N, xs);
    }
    return cudaGetLastError();
}

RestrictPlan restrict_plan(const Problem &p, int n_from, int n_to)
{
    RestrictPlan q;
    const int r = n_from / n_to;
    q.nt = (p.nx + 1 + kRTile - 1) / kRTile;
    q.kc = r;
    q.nchunk = 1;
    const long units = (long)q.nt * n_to;
    // A warp per coarse group where that fills the GPU twice over (2 warps on each of the
    // 608 sub-partitions) and a warp's serial chain stays short; below, four warps share the
    // members.
    q.mode = (r < 16 && units >= 1216) ? 0 : 1;
    if (q.mode == 1 && r > 32 && units < 1216) {
        // Members in chunks: a warp's chain is 12 kc / 4 operations and the last CTA's 3 r / kc
        // (its 12 sums on 4 warps), least for kc = sqrt(r); no more than 16 CTAs per SM.
        int kc = 8;
        while (kc * kc < r) kc *= 2;
        while (kc < r && units * ((r + kc - 1) / kc) > 2432) kc *= 2;
        const int nc = (r + kc - 1) / kc;
        if (nc > 1 && restrict_doubles(q.nt, n_to, nc) <= p.rscratch_doubles) {
            q.kc = kc;
            q.nchunk = nc;
        }
    }
    q.gy = q.mode == 0 ? (n_to + 3) / 4 : n_to * q.nchunk;
    return q;
}

size_t restrict_head_doubles() { return kRHead; }

size_t restrict_scratch_doubles(const Problem &p)
{
    Problem t = p;
    t.rscratch_doubles = ~(size_t)0;
    size_t need = kRHead;
    for (int l = 0; l + 1 < p.nlev; ++l)
        for (int m = l + 1; m < p.nlev; ++m) {
            if (l > 0 && m + 1 < p.nlev) continue;   // fine to any grid, any grid to grey
            const RestrictPlan q = restrict_plan(t, p.levels[l], p.levels[m]);
            if (q.nchunk > 1) need = std::max(need, restrict_doubles(q.nt, p.levels[m], q.nchunk));
        }
    return need;
}

RestrictCtx make_restrict_ctx(const Problem &p, const Level &src, const Level &dst)
{
    RestrictCtx x;
    const RestrictPlan q = restrict_plan(p, src.n, dst.n);
    x.nx = p.nx; x.r = src.n / dst.n; x.n_to = dst.n; x.h = p.h; x.ihf = p.ihf;
    x.S = src; x.T = dst;
    x.gate = p.gate;
    x.mode = q.mode; x.nt = q.nt; x.kc = q.kc; x.nchunk = q.nchunk;
    x.ticket = reinterpret_cast<int *>(p.rscratch);
    x.bpart = p.rscratch + kRHead;
    x.part = x.bpart + (size_t)dst.n * q.nchunk * 16;
    x.newton = 0;
    x.ga = GreyArgs{};
    x.pre = nullptr;
    x.skip_old = 0;
    x.fixed = 0;
    x.fix = nullptr;
    return x;
}

size_t restrict_fix_doubles(int nx, int n_to)
{
    return (size_t)n_to * 4 * 32 * ((nx + 1 + kRTile - 1) / kRTile);
}

cudaError_t launch_restrict(const Problem &p, const Level &src, Level &dst,
                            const GreyArgs *newton, double *pre, bool skip_old, const double *Topac,
                            double *fix, int fixed)
{
    RestrictCtx x = make_restrict_ctx(p, src, dst);
    x.skip_old = skip_old ? 1 : 0;
    x.fix = fix;
    x.fixed = fix && Topac ? fixed : 0;
    if (newton) {
        x.newton = 1;
        x.ga = *newton;
        x.pre = pre;
    }
    const RestrictPlan q = restrict_plan(p, src.n, dst.n);
    const dim3 grid(q.nt + 1, q.gy);
    if (!Topac) return launch_pdl(k_restrict, grid, dim3(128), 0, p.stream, x);
    OpacityArgs a;
    int op;
    const cudaError_t e = fused_opacity(p, Topac, src, (long)q.nt * q.gy, a, op);
    if (e != cudaSuccess) return e;
    // a later visit of the cycle finds the step's Eold and Fold sums in the target too
    const int form = x.fixed == 2 ? 2 : x.skip_old ? 1 : 0;
    auto k = a.otabp ? (form == 2 ? k_restrict_opac<true, false, true>
                        : form == 1 ? k_restrict_opac<true, false, false>
                                    : k_restrict_opac<true, true, false>)
                     : (form == 2 ? k_restrict_opac<false, false, true>
                        : form == 1 ? k_restrict_opac<false, false, false>
                                    : k_restrict_opac<false, true, false>);
    return launch_pdl(k, grid, dim3(128), 0, p.stream, x, a, op);
}

cudaError_t launch_restrict_b(const int *meta, int N, const RestrictCtx *xs, int grid,
                              cudaStream_t st)
{
    k_restrict_b<<<grid, 128, 0, st>>>(meta, N, xs);
    return cudaGetLastError();
}

GreyArgs grey_args_ready(const Problem &p, const GreyArgs &a)
{
    GreyArgs r = a;
    r.cvdt = a.cv / a.dt;
    r.k54 = 54.0 * a.s * kCB;
    const SeriesTables &t = host_series();
    r.e2 = p.e2tab;
    r.ec = ExpConsts{t.einv, t.eL1, t.eL2};
    return r;
}

GreyCtx make_grey_ctx(const Problem &p, const Level &g, const GreyArgs &a)
{
    GreyCtx x;
    x.lo = make_lo_ctx(p, a.dt, g);
    x.a = grey_args_ready(p, a);
    return x;
}

// at least the solver's chunks (<= nx / 2), a warp at least
static int grey_threads(int nx) { return std::min(1024, std::max(32, (nx + 31) / 32 * 32)); }

cudaError_t launch_grey(const Problem &p, const Level &g, const GreyArgs &a)
{
    const GreyCtx x = make_grey_ctx(p, g, a);
    const size_t sm = grey_smem(p.nx);
    cudaError_t e = allow_smem((const void *)k_grey, sm);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_grey, dim3(1), dim3(grey_threads(p.nx)), sm, p.stream, x);
}

cudaError_t launch_grey_b(const BatchSmem &bs, const int *meta, int N, const GreyCtx *xs, int grid,
                          cudaStream_t st)
{
    const size_t sm = bs.grey;
    cudaError_t e = allow_smem((const void *)k_grey_b, sm);
    if (e != cudaSuccess) return e;
    k_grey_b<<<grid, grey_threads(bs.max_nx), sm, st>>>(meta, N, xs);
    return cudaGetLastError();
}

cudaError_t launch_group_sum(const Problem &p, int n, const double *X, double *out)
{
    GroupSumArgs a;
    a.n = n; a.nx = p.nx; a.X = X; a.out = out;
    k_group_sum<<<(p.nx + 31) / 32, 256, 0, p.stream>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_group_sum_b(const int *meta, int N, const GroupSumArgs *xs, int grid,
                               cudaStream_t st)
{
    k_group_sum_b<<<grid, 256, 0, st>>>(meta, N, xs);
    return cudaGetLastError();
}

cudaError_t launch_copy_b(const int *meta, int N, const CopyArgs *xs, int grid, cudaStream_t st)
{
    k_copy_b<<<grid, 256, 0, st>>>(meta, N, xs);
    return cudaGetLastError();
}

}  // namespace trt
