// sweep64.cu -- paired FP64 S_N sweep (kernel K2, FP64): the directions mu and -mu of one
// |mu| share their corner-system coefficients.
//
// Same discretisation as sweep.cu (eq. rt with implicit Euler, Sec. 5; simple corner
// balance in a 1D slab).  Per (cell, group, direction) the 2 x 2 corner system has
//   a = |mu|/2 + sigma_t h/2,  b = |mu|/2,  t = a/det,  s = b/det,  det = a^2 + b^2,
// and the solution is psi_out = s r_in + t r_out, psi_other = t r_in - s r_out with r the
// corner sources (the inflow corner's carrying |mu| psi_in).  a, b, det, t and s depend on
// |mu|, not on its sign: the sweeps of mu and -mu through a cell use the same t and s.
// On GB300 every FP64 instruction of this kernel holds an FP64 pipe for 64 cycles, and
// forming t and s (the determinant, a refined reciprocal and two products) is 7 of the
// ~17 FP64 instructions of an update, so each pair of directions forms them once.
//
// Schedule (meet in the middle).  A job is 32 groups (the lanes) and D values of |mu| with
// two sign groups of D warps: warps 0..D-1 sweep mu > 0 from x = 0, warps D..2D-1 sweep
// mu < 0 from x = X.  Phase 1: each sign group sweeps its first half of the slab ([0, mid)
// for mu > 0, [mid, nx) for mu < 0), forming t and s per cell and storing them, and its
// psi_L + psi_R, in a global scratch ts[|mu|][cell][3][ldG]; a CTA barrier; phase 2: each sign
// group sweeps the other half with the t and s the other group stored there, and the D
// directions' sums of both signs go into the two angular moments (a partial tile of D
// values of |mu|, summed in a fixed order by the finalize).  Every t, s is formed once and used
// twice, every moment takes both signs at once: 15 FP64 instructions per update in phase
// 1, 11 in phase 2, 13.0 on average.  The two groups never wait for each other inside a
// phase.  Within a sign group cells go in strips of S: intensity rows, the step's pre-scaled
// inputs sigma_t h/2 and h e/2 (FP64, [nx][ldG], written by k_prescale64 before the
// sweep) and, in phase 2, the partner's t, s, sum rows arrive by 16-byte cp.async NS - 1
// strips ahead.
//
// Balance.  A warp's chain over the cells is serial and a job cannot be spread over SMs, so
// one CTA per job leaves SMs idle (fc_1024, D = 4: 256 CTAs on 152 SMs, two on 104 of them
// and one on 48).  Where there are at least as many jobs as resident CTAs, the grid is the
// resident CTAs and the jobs' strips are dealt out evenly by McNaughton's wrap-around rule:
// CTA k takes the k-th equal share of the line of all strips, and a job that straddles two
// shares is split at a strip boundary.  The CTA on the right runs the job's first strips at
// its start and hands over psi; the CTA on the left runs the rest at its end.  A share is at
// least one job long, so the first part has ended long before the second begins; the second
// part waits for its flag all the same (bounded; a wait that runs out poisons psi with NaN,
// which a step reports as TRT_ENUMERIC).  The launch is cooperative: every CTA is resident.
//
// Bound by the FP64 pipe.  500 cells x 64 directions x 1024 groups, with prescale and
// finalize: 0.970 ms with one CTA of D = 4 per job and a partial tile per sign, 0.831 now
// (D = 2, 456 CTAs); 13.0 instructions per update at the measured FP64 rate are 0.807 ms.
#include <algorithm>
#include <atomic>
#include <type_traits>
#include "sweep.cuh"

namespace trt {

namespace {

// 1/d for the determinant d = a^2 + b^2 (normal, > 0): the hardware approximation refined
// by one third-order step (below FP64 rounding; see common.cuh's rcp64)
__device__ __forceinline__ double rcp_det(double d)
{
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(d));
    const double e = fma(-d, x, 1.0);
    return fma(x, fma(e, e, e), x);
}

__device__ __forceinline__ void cp16(void *smem, const void *gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}

// named barrier of one sign group (its D warps)
template <int D>
__device__ __forceinline__ void group_sync(int id)
{
    if (D == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(32 * D) : "memory");
}

template <int D, int S, int NS>
struct PairSmem {
    // per sign group (byte offsets within the group's section):
    static constexpr size_t it = 0;                                 // [NS][D][S][2][32] I_old rows
    static constexpr size_t tb = it + 8ull * NS * D * S * 64;       // [NS][D][S][3][32] t, s, sum rows
    static constexpr size_t tq = tb + 8ull * NS * D * S * 96;       // [NS][S][2][32] th, q rows
    static constexpr size_t kp = tq + 8ull * NS * S * 64;           // [NS][S] h/(2 c dt)
    static constexpr size_t ps = kp + 8ull * NS * S;                // [D][S][33] both signs' sums
    static constexpr size_t group = ps + 8ull * D * S * 33;
    static constexpr size_t total = 2 * group;
};

// strips of a phase, and the cost of a strip in the dealing (its FP64 instructions per update)
constexpr int kCost1 = 15, kCost2 = 11;
__host__ __device__ inline int pair_strips(int nx, int S) { return (nx - nx / 2 + S - 1) / S; }
// of a job whose first `units` of cost are cut off: the strips (of both phases) in that part
__device__ inline int pair_cut(long long units, int nst)
{
    if (units <= (long long)kCost1 * nst) return (int)(units / kCost1);
    return nst + (int)((units - (long long)kCost1 * nst) / kCost2);
}

template <int D, int S, int NS>
__global__ void __launch_bounds__(64 * D) k_sweep_pair(SweepArgs a)
{
    griddep_wait();
    using L = PairSmem<D, S, NS>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sg = warp / D, wi = warp % D, gtid = tid % (32 * D);
    unsigned char *base = smem_raw + sg * L::group;
    double *it = reinterpret_cast<double *>(base + L::it);
    double *tb = reinterpret_cast<double *>(base + L::tb);
    double *tq = reinterpret_cast<double *>(base + L::tq);
    double *kp = reinterpret_cast<double *>(base + L::kp);
    double *ps = reinterpret_cast<double *>(base + L::ps);

    const int nx = a.nx, N = a.N, G = a.G, ldG = a.ldG;
    const int mid = nx / 2, nst = pair_strips(nx, S);
    const size_t row = 2 * (size_t)ldG;      // one cell of one direction (two corner rows)
    const size_t trow = 3 * (size_t)ldG;     // one cell of one |mu| in the scratch
    const double *th64 = reinterpret_cast<const double *>(a.sigE);   // [nx][ldG]
    const double *q64 = reinterpret_cast<const double *>(a.emis);    // [nx][ldG], then kap [nx]
    const double *kap64 = q64 + (size_t)nx * ldG;
    double *part = reinterpret_cast<double *>(a.part);
    // this lane's 16-byte chunk of a cell's two 32-double rows: row rr, chunk ch
    const int rr = lane >> 4, ch = lane & 15;

    // strips s0 .. s1 - 1 of a job's 2 nst (phase 1, then phase 2); psi comes in from the strip
    // before s0 (the inflow at 0, the hand-over slot of `from` otherwise) and goes out to the
    // slot of `to` (or, after the last strip, to the exit intensities)
    auto run = [&](int job, int s0, int s1, int from, int to) {
        const int dtile = job % (N / D), gt = job / (N / D);
        const int gb = gt * 32, g = gb + lane;
        const int n = dtile * D + wi;            // |mu| index
        const int m = sg ? N + n : n;            // direction index (m >= N: mu < 0)
        const double am = fabs(a.mu[m]), b = 0.5 * am, bb = b * b;
        // moment weights of the D directions (w/2, w mu^2/2), the same for both signs
        double wt[D], wm[D];
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const int md = dtile * D + d;
            wt[d] = 0.5 * a.w[md];
            wm[d] = 0.5 * a.w[md] * a.mu[md] * a.mu[md];
        }
        const double *Iold = reinterpret_cast<const double *>(a.I_old) + (size_t)m * nx * row;
        double *Inew = reinterpret_cast<double *>(a.I_new) + (size_t)m * nx * row + g;
        double *ts = a.ts + (size_t)n * nx * trow;   // this |mu|'s t, s, sum rows
        double psi;
        if (from < 0) {
            psi = (g < G) ? (sg ? a.IinX[g] : a.Iin0[g]) : 0.0;
        } else {
            __shared__ int arrived;
            if (tid == 0) {
                int ok = 0;
                unsigned long long t0 = 0, t;
                for (;;) {
                    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(ok) : "l"(a.hand_flag + from) : "memory");
                    if (ok == a.hand_epoch) break;
                    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                    if (t0 == 0) t0 = t;
                    if (t - t0 > 1000000000ull) break;
                    __nanosleep(200);
                }
                arrived = ok == a.hand_epoch;
                if (arrived) a.hand_flag[from] = 0;   // one taker; a replayed launch starts at 0
            }
            __syncthreads();
            psi = arrived ? __ldcg(a.hand + ((size_t)from * 2 * D + warp) * 32 + lane)
                          : __longlong_as_double(0x7ff8000000000000ll);
        }
        for (int phase = 0; phase < 2; ++phase) {
            // this group's cells in this phase, in sweep order: mu > 0 ascending over [lo,
            // hi), mu < 0 descending; strips aligned at lo (mu > 0) or hi (mu < 0)
            const bool first = (phase == 0);
            const int lo = (first == (sg == 0)) ? 0 : mid;
            const int hi = (first == (sg == 0)) ? mid : nx;
            const int b0 = max(s0 - phase * nst, 0);
            const int b1 = min(min(s1 - phase * nst, nst), (hi - lo + S - 1) / S);
            auto range = [&](int st, int &c0, int &ns) {
                if (sg == 0) {
                    c0 = lo + st * S;
                    ns = min(S, hi - c0);
                } else {
                    const int c1 = hi - st * S;
                    c0 = max(c1 - S, lo);
                    ns = c1 - c0;
                }
            };
            auto prefetch = [&](int st) {
                const int bf = (st - b0) % NS;
                int c0, ns;
                range(st, c0, ns);
                double *itw = it + ((size_t)(bf * D + wi) * S) * 64;
                double *tbw = tb + ((size_t)(bf * D + wi) * S) * 96;
                for (int cc = 0; cc < ns; ++cc) {
                    const size_t src = (size_t)(c0 + cc) * row + rr * ldG + gb + 2 * ch;
                    cp16(itw + cc * 64 + rr * 32 + 2 * ch, Iold + src);
                    if (!first) {
                        const double *tsrc = ts + (size_t)(c0 + cc) * trow + gb + 2 * ch;
                        cp16(tbw + cc * 96 + rr * 32 + 2 * ch, tsrc + rr * ldG);
                        if (rr == (cc & 1)) cp16(tbw + cc * 96 + 64 + 2 * ch, tsrc + 2 * (size_t)ldG);
                    }
                }
                // th, q rows of the strip (phase 2: q alone): cells wi, wi + D, ... by warp wi
                double *tqb = tq + (size_t)bf * S * 64;
                for (int cc = wi; cc < ns; cc += D) {
                    const double *srcp = (rr ? q64 : th64) + (size_t)(c0 + cc) * ldG + gb + 2 * ch;
                    if (first || rr) cp16(tqb + cc * 64 + rr * 32 + 2 * ch, srcp);
                }
                if (gtid < ns) cp_async<8>(kp + bf * S + gtid, kap64 + c0 + gtid);
                cp_commit();
            };
            for (int k = 0; k < NS - 1; ++k) {
                if (b0 + k < b1)
                    prefetch(b0 + k);
                else
                    cp_commit();
            }
            for (int st = b0; st < b1; ++st) {
                const int bf = (st - b0) % NS;
                int c0, ns;
                range(st, c0, ns);
                cp_wait<NS - 2>();
                group_sync<D>(1 + sg);   // the strip's copies landed; the last reduction is done
                if (st + NS - 1 < b1)
                    prefetch(st + NS - 1);
                else
                    cp_commit();
                const double *itw = it + ((size_t)(bf * D + wi) * S) * 64 + lane;
                const double *tbw = tb + ((size_t)(bf * D + wi) * S) * 96 + lane;
                const double *tqb = tq + (size_t)bf * S * 64 + lane;
                const double *kpb = kp + bf * S;
                double *psw = ps + (size_t)wi * S * 33 + lane;
                double *tsw = ts + g;
                // one cell: FIRST forms t, s and stores them and its sum for the other sign
                // group; POS: the sign of mu (inflow on the left corner)
                auto cell = [&](auto first_c, auto pos_c, int cc) {
                    constexpr bool FIRST = decltype(first_c)::value, POS = decltype(pos_c)::value;
                    const int c = c0 + cc;
                    const double IL = itw[cc * 64], IR = itw[cc * 64 + 32];
                    const double q = tqb[cc * 64 + 32];
                    const double kap = kpb[cc];
                    double t, s;
                    if (FIRST) {
                        const double aa = b + tqb[cc * 64];
                        const double x = rcp_det(fma(aa, aa, bb));
                        t = aa * x;
                        s = b * x;
                        tsw[(size_t)c * trow] = t;
                        tsw[(size_t)c * trow + ldG] = s;
                    } else {
                        t = tbw[cc * 96];
                        s = tbw[cc * 96 + 32];
                    }
                    const double kL = fma(kap, IL, q), kR = fma(kap, IR, q);
                    double pL, pR;
                    if (POS) {
                        const double rL = fma(am, psi, kL);
                        pR = fma(s, rL, t * kR);
                        pL = fma(t, rL, -(s * kR));
                        psi = pR;
                    } else {
                        const double rR = fma(am, psi, kR);
                        pL = fma(s, rR, t * kL);
                        pR = fma(t, rR, -(s * kL));
                        psi = pL;
                    }
                    Inew[(size_t)c * row] = pL;
                    Inew[(size_t)c * row + ldG] = pR;
                    if (FIRST) tsw[(size_t)c * trow + 2 * (size_t)ldG] = pL + pR;
                    else psw[cc * 33] = (pL + pR) + tbw[cc * 96 + 64];
                };
                // full strips unrolled (the next cells' loads and independent products overlap
                // the recurrence of the current one), ragged strips in a loop
                auto strip = [&](auto first_c, auto pos_c) {
                    constexpr bool POS = decltype(pos_c)::value;
                    if (ns == S) {
#pragma unroll
                        for (int k = 0; k < S; ++k) cell(first_c, pos_c, POS ? k : S - 1 - k);
                    } else {
                        for (int k = 0; k < ns; ++k) cell(first_c, pos_c, POS ? k : ns - 1 - k);
                    }
                };
                using T_ = std::true_type;
                using F_ = std::false_type;
                if (first) {
                    if (sg == 0) strip(T_(), T_()); else strip(T_(), F_());
                    continue;
                }
                if (sg == 0) strip(F_(), T_()); else strip(F_(), F_());
                group_sync<D>(1 + sg);
                // both signs of the D directions summed per (cell, group) of the strip, in order
                for (int idx = gtid; idx < 32 * S; idx += 32 * D) {
                    const int gl = idx / S, cc = idx % S;
                    const int gg = gb + gl;
                    if (cc < ns && gg < G) {
                        double s0 = 0.0, s2 = 0.0;
#pragma unroll
                        for (int d = 0; d < D; ++d) {
                            const double v = ps[((size_t)d * S + cc) * 33 + gl];
                            s0 = fma(wt[d], v, s0);
                            s2 = fma(wm[d], v, s2);
                        }
                        const size_t o = ((size_t)(dtile * 2) * G + gg) * nx + c0 + cc;
                        part[o] = s0;
                        part[o + (size_t)G * nx] = s2;
                    }
                }
            }
            cp_wait<0>();
            // phase 1 -> 2: every t, s, sum of this CTA is stored (global writes before the
            // barrier are visible to the block after it) and every reduction has read ps
            __syncthreads();
        }
        if (to >= 0) {
            a.hand[((size_t)to * 2 * D + warp) * 32 + lane] = psi;
            __threadfence();   // psi and the strips' t, s, sum rows
            __syncthreads();
            if (tid == 0)
                asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(a.hand_flag + to), "r"(a.hand_epoch) : "memory");
        } else {
            reinterpret_cast<double *>(a.psi_exit)[(size_t)m * ldG + g] = psi;
        }
    };

    const int J = (N / D) * (ldG / 32), K = gridDim.x, k = blockIdx.x;
    if (K == J) {
        run(k, 0, 2 * nst, -1, -1);
        return;
    }
    // this CTA's share [u0, u1) of the line of J jobs of U units
    const long long U = (long long)(kCost1 + kCost2) * nst, tot = U * J;
    const long long u0 = tot * k / K, u1 = tot * (k + 1) / K;
    int j = (int)(u0 / U);
    if (u0 % U) {   // the first part of the job that the CTA before ends
        const int c = pair_cut((j + 1) * U - u0, nst);
        if (c > 0) run(j, 0, c, -1, k);
        ++j;
    }
    for (; (j + 1) * U <= u1; ++j) run(j, 0, 2 * nst, -1, -1);
    if (u1 % U && j * U < u1) {   // the rest of the job whose first part the next CTA ran
        const int c = pair_cut((j + 1) * U - u1, nst);
        run(j, c, 2 * nst, c > 0 ? k + 1 : -1, -1);
    }
}

// the paired sweep's pre-scaled FP64 inputs from sigma_E and e_g ([G][nx]): sigma_t h/2 and
// h e/2 as [nx][ldG] (zero in the padding groups), then h/(2 c dt) per cell; a 32 x 32 tile
// through shared memory so that both sides are read and written along rows
__global__ void k_prescale64(int nx, int G, int ldG, const double *__restrict__ h, double icdt,
                             const double *__restrict__ sigE, const double *__restrict__ emis,
                             double *th64, double *q64)
{
    griddep_wait();
    __shared__ double sth[32][33], sq[32][33];
    const int c0 = blockIdx.x * 32, g0 = blockIdx.y * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
    for (int r = ty; r < 32; r += 8) {   // read along cells: group g0 + r, cell c0 + tx
        const int g = g0 + r, c = c0 + tx;
        double vt = 0.0, vq = 0.0;
        if (g < G && c < nx) {
            const double hh = 0.5 * h[c];
            vt = hh * (sigE[(size_t)g * nx + c] + icdt);
            vq = hh * emis[(size_t)g * nx + c];
        }
        sth[r][tx] = vt;
        sq[r][tx] = vq;
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {   // write along groups: cell c0 + r, group g0 + tx
        const int c = c0 + r, g = g0 + tx;
        if (c < nx && g < ldG) {
            th64[(size_t)c * ldG + g] = sth[tx][r];
            q64[(size_t)c * ldG + g] = sq[tx][r];
        }
    }
    if (blockIdx.y == 0 && ty == 0 && c0 + tx < nx)
        q64[(size_t)nx * ldG + c0 + tx] = 0.5 * h[c0 + tx] * icdt;
}

}  // namespace

size_t pair_sweep_smem(int S, int NS)
{
    if (S == 8 && NS == 2) return PairSmem<4, 8, 2>::total;
    if (S == 4 && NS == 2) return PairSmem<4, 4, 2>::total;
    return 0;
}

int pair_default_D(int N, int ldG)
{
    // D = 2 (4 warps, one per sub-partition) deals out the finest jobs that still use every
    // FP64 pipe of an SM; one |mu| per CTA where even those leave SMs without a job (the
    // chain of a warp over the cells is the whole time there) or N is odd.
    const long jobs2 = (long)(N / 2) * (ldG / 32);
    return (N % 2 == 0 && jobs2 >= 152) ? 2 : 1;
}

// hand-over slots of 3 x 160 CTAs (psi of 8 warps), then their flags (ints)
constexpr size_t kHandSlots = 3 * 160;
size_t pair_hand_doubles() { return kHandSlots * (8 * 32) + kHandSlots / 2; }

cudaError_t launch_sweep_pair(int D, int S, int NS, const SweepArgs &a, int M, int ldG,
                              cudaStream_t st)
{
    if (D < 1 || a.N % D != 0 || !a.ts || !a.tab64 || !a.hand) return cudaErrorInvalidConfiguration;
    const double *sigE = reinterpret_cast<const double *>(a.sigE);
    const double *emis = reinterpret_cast<const double *>(a.emis);
    double *tab64 = a.tab64;
    const int nx = a.nx, G = a.G;
    cudaError_t e = launch_pdl(k_prescale64, dim3((nx + 31) / 32, (ldG + 31) / 32), dim3(32, 8),
                               0, st, nx, G, ldG, (const double *)a.h, a.icdt, sigE, emis, tab64,
                               tab64 + (size_t)nx * ldG);
    if (e != cudaSuccess) return e;
    SweepArgs x = a;
    x.sigE = tab64;
    x.emis = tab64 + (size_t)nx * ldG;
    x.hand_flag = reinterpret_cast<int *>(a.hand + kHandSlots * (8 * 32));
    static std::atomic<int> epoch{0};   // tells a launch's flags from those of any other
    x.hand_epoch = epoch.fetch_add(1) % 0x7ffffffe + 1;
    const int jobs = M / 2 / D * (ldG / 32);
    auto go = [&](auto kern, size_t sm) {
        cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sm);
        if (r != cudaSuccess) return r;
        int dev = 0, sms = 0, per_sm = 0;
        if ((r = cudaGetDevice(&dev)) != cudaSuccess) return r;
        if ((r = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return r;
        r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 64 * D, sm);
        if (r != cudaSuccess) return r;
        // resident CTAs per SM: as many as leave every CTA a job (3 at most: the hand-over
        // slots), none of them idle
        const int c = std::min(std::min(per_sm, 3), jobs / std::max(sms, 1));
        if (c < 1 || sms > 160 || jobs == c * sms)
            return launch_pdl(kern, dim3(jobs), dim3(64 * D), sm, st, x);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c * sms);
        cfg.blockDim = dim3(64 * D);
        cfg.dynamicSmemBytes = sm;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kern, x);
    };
    if (D == 4 && S == 8 && NS == 2) return go(k_sweep_pair<4, 8, 2>, PairSmem<4, 8, 2>::total);
    if (D == 4 && S == 4 && NS == 2) return go(k_sweep_pair<4, 4, 2>, PairSmem<4, 4, 2>::total);
    if (D == 2 && S == 4 && NS == 2) return go(k_sweep_pair<2, 4, 2>, PairSmem<2, 4, 2>::total);
    if (D == 1 && S == 4 && NS == 2) return go(k_sweep_pair<1, 4, 2>, PairSmem<1, 4, 2>::total);
    return cudaErrorInvalidConfiguration;
}

}  // namespace trt
