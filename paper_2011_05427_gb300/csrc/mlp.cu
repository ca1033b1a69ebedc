// mlp.cu -- the learned closure's network on the tensor cores: a BF16 GEMM on tcgen05
// (tensor memory accumulators, shared-memory operand descriptors, mbarrier-tracked
// commits) with fused epilogues, and the MLP's forward, backward, Adam and feature
// kernels built on it.  The paper has no learned component; see include/trt_mlp.h.
//
// GEMM tile: 128 rows x 256 columns per CTA, K in chunks of 64 through two shared-memory
// stages.  Four warps copy each chunk with cp.async into the canonical no-swizzle K-major
// layout of the tensor core (8-row x 16-byte core matrices, 128 contiguous bytes each; the
// 8 core matrices of a row group along K are adjacent, 128 bytes apart, and row groups are
// 1024 bytes apart -- either reading of the two descriptor strides stays inside the stage);
// one thread issues four tcgen05.mma (M 128, N 256, K 16) per chunk and commits them to
// the stage's mbarrier, which releases the stage for the chunk after next.  The 128 x 256
// FP32 accumulator lives in 256 tensor-memory columns; in the epilogue thread t owns row
// t (tensor-memory lane t) and reads its 256 values 32 at a time with tcgen05.ld.
#include <algorithm>
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include "common.cuh"
#include "../../include/trt_mlp.h"

namespace trt {

namespace {

typedef __nv_bfloat16 bf16;

constexpr int BM = 128, BN = 256, BK = 64;
constexpr int A_STAGE = BM * BK * 2;   // 16 KB
constexpr int B_STAGE = BN * BK * 2;   // 32 KB
constexpr int GEMM_SMEM = 2 * (A_STAGE + B_STAGE) + 256;
// core-matrix (row group r, K group k) of a stage at (r * 8 + k) * 128: leading-dimension
// (K) byte offset 128, stride-dimension (row group) byte offset 1024
constexpr uint32_t LBO = 128, SBO = 1024;
// instruction descriptor, kind::f16: D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9,
// 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                           ((uint32_t)(BM >> 4) << 24);
constexpr unsigned long long WAIT_NS = 1000000000ull;   // one second

__device__ int g_mlp_err = 0;

__device__ inline uint32_t su32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ inline unsigned long long gtime()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ inline void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(count));
}

__device__ inline bool mbar_test(uint64_t *bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(su32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait on a phase of an mbarrier: false after WAIT_NS without completion
__device__ inline bool mbar_wait(uint64_t *bar, unsigned parity)
{
    if (mbar_test(bar, parity)) return true;
    const unsigned long long t0 = gtime();
    while (!mbar_test(bar, parity))
        if (gtime() - t0 > WAIT_NS) return false;
    return true;
}

__device__ inline void cp16(void *dst, const void *src, unsigned bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(su32(dst)), "l"(src),
                 "r"(bytes));
}
__device__ inline void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ inline void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

__device__ inline void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ inline void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ inline void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory operand descriptor: start >> 4 (bits 0-13), leading-dimension byte offset
// >> 4 (16-29), stride-dimension byte offset >> 4 (32-45), descriptor version 1 (46-47),
// base offset 0, no swizzle (61-63 = 0)
__device__ inline uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) |
           ((uint64_t)(sbo >> 4) << 32) | (1ull << 46);
}

template <uint32_t kDesc = IDESC>
__device__ inline void umma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
        "l"(a), "l"(b), "r"(kDesc), "r"(acc));
}

__device__ inline void umma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     su32(bar))
                 : "memory");
}

// 32 consecutive FP32 columns of this warp's 32 tensor-memory lanes (one per thread)
__device__ inline void tmem_ld32(uint32_t taddr, float *v)
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// the same load without its wait (two loads may be in flight before one wait), and the
// wait tied to the loaded registers so that no use of them is scheduled before it
__device__ inline void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
}
__device__ inline void tmem_wait_tied(uint32_t (&r)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}
__device__ inline void reg_tie(uint32_t (&r)[32])
{
    asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]));
}

struct Epi {
    const float *bias;
    int relu;
    const bf16 *mask;
    float *out32;
    bf16 *out16, *out16T;
    int ldT;
    // head: z = sum_n act[n] w[n] + b, y = sigmoid(z)
    const float *head_w;
    const float *head_b;   // device pointer to the head's bias
    float *head_y;
};

__global__ void __launch_bounds__(128) k_gemm(int M, int N, int K, const bf16 *__restrict__ A,
                                              const bf16 *__restrict__ B, Epi e)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *sA = sm;
    unsigned char *sB = sm + 2 * A_STAGE;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + 2 * (A_STAGE + B_STAGE));
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 2);
    int *sfail = reinterpret_cast<int *>(tslot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    const int nk = K / BK;

    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        *sfail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         su32(tslot)),
                     "r"(256));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = *tslot;

    // chunk c of A (128 x 64) and B (256 x 64) into stage st in 16-byte pieces: piece p
    // is row p & 7 of core matrix (row group p >> 6, K group (p >> 3) & 7), i.e. shared
    // offset 16 p (conflict-free); rows of A past M are zero-filled
    auto load = [&](int c, int st) {
        const int k0 = c * BK;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int p = tid + 128 * j;
            const int r8 = p & 7, ki = (p >> 3) & 7, mi = p >> 6;
            const int row = m0 + mi * 8 + r8;
            const bf16 *src = A + (size_t)min(row, M - 1) * K + k0 + ki * 8;
            cp16(sA + st * A_STAGE + p * 16, src, row < M ? 16u : 0u);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int p = tid + 128 * j;
            const int r8 = p & 7, ki = (p >> 3) & 7, ni = p >> 6;
            const bf16 *src = B + (size_t)(n0 + ni * 8 + r8) * K + k0 + ki * 8;
            cp16(sB + st * B_STAGE + p * 16, src, 16u);
        }
    };

    load(0, 0);
    cp_commit();
    if (nk > 1) load(1, 1);
    cp_commit();
    bool ok = true;
    for (int c = 0; c < nk; ++c) {
        const int st = c & 1;
        if (c + 1 < nk)
            cp_wait<1>();
        else
            cp_wait<0>();
        fence_async_smem();   // this thread's copies -> visible to the tensor core
        __syncthreads();
        if (*sfail) { ok = false; break; }
        if (tid == 0) {
            tc_after();
            const uint32_t a0 = su32(sA + st * A_STAGE), b0 = su32(sB + st * B_STAGE);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)   // K = 16 per instruction: 2 core matrices
                umma(tmem, sdesc(a0 + kk * 2 * LBO, LBO, SBO), sdesc(b0 + kk * 2 * LBO, LBO, SBO),
                     (c | kk) != 0);
            umma_commit(&bar[st]);
        }
        if (c + 2 < nk) {
            // stage st takes chunk c + 2 once the MMAs of chunk c have read it
            if (!mbar_wait(&bar[st], (c >> 1) & 1)) *sfail = 1;
            __syncthreads();
            if (*sfail) { ok = false; break; }
            load(c + 2, st);
            cp_commit();
        }
    }
    if (ok && !mbar_wait(&bar[(nk - 1) & 1], ((nk - 1) >> 1) & 1)) ok = false;
    ok = !__syncthreads_or(!ok);   // CTA-uniform: the tensor-memory loads are warp-collective
    if (!ok) {
        cp_wait<0>();
        if (lane == 0) atomicExch(&g_mlp_err, TRT_ETIMEOUT);
    }
    tc_after();

    const int row = m0 + tid;
    if (ok) {
        float dot = 0.f;
        for (int ch = 0; ch < BN / 32; ++ch) {
            float v[32];
            tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + ch * 32, v);
            if (row >= M) continue;
            const int nb = n0 + ch * 32;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                float a = v[j];
                if (e.bias) a += e.bias[nb + j];
                if (e.relu) a = fmaxf(a, 0.f);
                v[j] = a;
            }
            if (e.mask) {
                const uint4 *mk = reinterpret_cast<const uint4 *>(e.mask + (size_t)row * N + nb);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint4 u = mk[q];
                    const bf16 *hb = reinterpret_cast<const bf16 *>(&u);
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (!(__bfloat162float(hb[j]) > 0.f)) v[q * 8 + j] = 0.f;
                }
            }
            if (e.out32) {
                float4 *o = reinterpret_cast<float4 *>(e.out32 + (size_t)row * N + nb);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
            if (e.out16) {
                uint4 *o = reinterpret_cast<uint4 *>(e.out16 + (size_t)row * N + nb);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint4 u;
                    bf16 *hb = reinterpret_cast<bf16 *>(&u);
#pragma unroll
                    for (int j = 0; j < 8; ++j) hb[j] = __float2bfloat16_rn(v[q * 8 + j]);
                    o[q] = u;
                }
            }
            if (e.out16T) {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    e.out16T[(size_t)(nb + j) * e.ldT + row] = __float2bfloat16_rn(v[j]);
            }
            if (e.head_w) {
#pragma unroll
                for (int j = 0; j < 32; ++j) dot = fmaf(v[j], e.head_w[nb + j], dot);
            }
        }
        if (e.head_w && row < M) {
            const float z = dot + *e.head_b;
            e.head_y[row] = 1.f / (1.f + __expf(-z));
        }
    }
    tc_before();
    __syncthreads();
    if (warp == 0) {
        tc_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256));
    }
}

// ---- fused inference: the whole network in one persistent kernel ----
// One CTA per SM, 576 threads: two groups of eight warps, a producer warp and an MMA warp.
// Each iteration takes 256 rows; group g (warps 8g .. 8g+7, thread = row = tensor-memory
// lane, four warps on columns 0 .. 127 and four on 128 .. 255) owns rows 128 g .. 128 g + 127
// of it, its activation tile A_g in shared memory and its 128 x 256 FP32 accumulator in
// tensor-memory columns 256 g .. 256 g + 255.  One thread (warp 16) streams the weights; one
// elected lane of warp 17 issues every MMA, in the order
//   layer 2 of group 0, layer 2 of group 1, layer 3 of group 0, layer 3 of group 1,
// so that while the tensor core multiplies for one group the other group's warps run its
// CUDA-core phase (layer 1, a ReLU/bias epilogue, the sigmoid head): the two groups work
// half a period apart and the MMAs of one hide the epilogues of the other.
//   Weights: 32-wide K chunks (16 KB, 256 rows x 32 K of W2 or W3) through a five-slot
// ring.  trt_mlp_refresh stores each chunk contiguously in the order the tensor core
// reads it (core matrices of 8 rows x 16 bytes; K groups 4096 bytes apart, row groups 128
// bytes apart), so one cp.async.bulk of 16 KB moves a chunk and completes on the slot's
// `full` mbarrier; the MMAs reading a slot commit to its `empty` mbarrier, which releases
// it for the chunk S later.  Every chunk is used by one group's layer, so each weight is
// streamed twice per 256 rows (from L2: the whole 256 KB image stays resident there).
//   The MMA thread never waits for a slot to drain (that is the producer's wait), so the
// tensor core always has the next chunk's MMAs queued behind the running ones.
//   What bounds it: shared memory.  The MMAs read 12 KB per 128 cycles and the epilogues'
// parameter reads (16 bytes broadcast to a warp cost two wavefronts or more) compete with
// them: without the epilogues' work the same MMA stream takes 67 us for 512,000 rows, without
// the weight copies it takes as long as with them.  So layer 1 reads each parameter once for
// four rows (a lane's rows 32 apart, 32 columns per warp) instead of once per row.  512,000
// rows: 104 us (floor at the measured BF16 GEMM rate 70); 117 with layer 1 reading its
// parameters once per row, 113 with chunks of 64 K in two slots.
//   Hand-offs: a group arrives on act[g] (256 arrivals) when A_g holds the next layer's
// input (after a proxy fence: the MMAs read it through the async proxy); the MMA thread
// commits the last MMA of a layer to acc[g], which the group waits on before it reads
// the accumulator.  Small parameters (layer-1 weights, biases, head) sit in shared
// memory.  Every mbarrier wait is bounded (one second); a wait that runs out stops the
// kernel's work and sets the device error flag (trt_mlp_status).
constexpr int FA_BYTES = 128 * 256 * 2;   // one activation tile
constexpr int FK = 32;                    // K width of a weight chunk
constexpr int FNC = 256 / FK;             // chunks per layer
constexpr int FW_BYTES = 256 * FK * 2;    // one weight chunk
constexpr int F_SLOTS = 5;
constexpr uint32_t FW_LBO = 4096, FW_SBO = 128;   // weight chunk: K groups, row groups
// small parameters in shared memory: W1^T [3][256], b1, b2, b3, w4, b4 (1793 floats)
constexpr int FP_W1 = 0, FP_B1 = 768, FP_B2 = 1024, FP_B3 = 1280, FP_W4 = 1536, FP_B4 = 1792;
constexpr int FP_BYTES = 1796 * 4;
constexpr int F_NBAR = 2 * F_SLOTS + 6;   // full[S], empty[S], act[2], acc[2], dotb[2]
constexpr int F_SMEM = 2 * FA_BYTES + F_SLOTS * FW_BYTES + FP_BYTES + 8 * F_NBAR + 32 + 2 * 128 * 4;
constexpr uint32_t FA_SBO = 4096;         // activation tiles: 32 K groups per row group
constexpr int F_THREADS = 576;

__device__ inline void mbar_init_n(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(count));
}
__device__ inline void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(bar)) : "memory");
}
__device__ inline void mbar_expect(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(bar)),
                 "r"(bytes)
                 : "memory");
}
// packed FP32 pairs (Blackwell f32x2 arithmetic: two lanes' worth of FP32 per instruction)
__device__ inline float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(*reinterpret_cast<unsigned long long *>(&d))
        : "l"(*reinterpret_cast<const unsigned long long *>(&a)),
          "l"(*reinterpret_cast<const unsigned long long *>(&b)),
          "l"(*reinterpret_cast<const unsigned long long *>(&c)));
    return d;
}
__device__ inline float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(*reinterpret_cast<unsigned long long *>(&d))
        : "l"(*reinterpret_cast<const unsigned long long *>(&a)),
          "l"(*reinterpret_cast<const unsigned long long *>(&b)));
    return d;
}
// relu of two FP32 values rounded to BF16 (nearest even) in one word, v.x in the low half:
// rounding keeps the sign, so rounding after the clamp equals clamping after rounding
__device__ inline uint32_t relu_bf16x2(float2 v)
{
    uint32_t d;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(v.y), "f"(v.x));
    return d;
}

// element (row, K group k8) of an activation tile: core matrix (row / 8, k8), row % 8 at
// 16 bytes
__device__ inline uint32_t a_off(int row, int k8)
{
    return (uint32_t)((row >> 3) * FA_SBO + k8 * 128 + (row & 7) * 16);
}

// layer 1, h1 = relu(W1 x + b1), of the four rows r, r + 32, r + 64, r + 96 with inputs v,
// columns 8 k0 .. 8 k1 - 1 into the activation tile: W1^T rows and b1 as broadcast float4
// reads of shared memory, once for the four rows, pairs of columns by packed FP32 FMAs, ReLU
// fused in the BF16 pack.  kMax: clamped first by fmax, which turns a NaN into 0 as the GEMM
// epilogue does (the pack's ReLU keeps it)
template <bool kMax>
__device__ inline void layer1_rows4(const float *sP, const float (&v)[4][3], unsigned char *A, int r,
                                    int k0, int k1)
{
    const float4 *pw = reinterpret_cast<const float4 *>(sP + FP_W1);
    const float4 *pb = reinterpret_cast<const float4 *>(sP + FP_B1);
    for (int k8 = k0; k8 < k1; ++k8) {
        uint4 u[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = k8 * 2 + h;
            const float4 b = pb[k], w0 = pw[k], w1 = pw[64 + k], w2 = pw[128 + k];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 X0 = make_float2(v[j][0], v[j][0]), X1 = make_float2(v[j][1], v[j][1]),
                             X2 = make_float2(v[j][2], v[j][2]);
                float2 a = make_float2(b.x, b.y), c = make_float2(b.z, b.w);
                a = fma2(make_float2(w0.x, w0.y), X0, a);
                c = fma2(make_float2(w0.z, w0.w), X0, c);
                a = fma2(make_float2(w1.x, w1.y), X1, a);
                c = fma2(make_float2(w1.z, w1.w), X1, c);
                a = fma2(make_float2(w2.x, w2.y), X2, a);
                c = fma2(make_float2(w2.z, w2.w), X2, c);
                if (kMax) {
                    a = make_float2(fmaxf(a.x, 0.f), fmaxf(a.y, 0.f));
                    c = make_float2(fmaxf(c.x, 0.f), fmaxf(c.y, 0.f));
                }
                (h ? u[j].z : u[j].x) = relu_bf16x2(a);
                (h ? u[j].w : u[j].y) = relu_bf16x2(c);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4 *>(A + a_off(r + 32 * j, k8)) = u[j];
    }
}

// small parameters into shared memory (W1 transposed, b1, b2, b3, w4, b4) by threads
// 0 .. 255; P of any alignment
__device__ inline void stage_params(float *sP, const float *P, int tid)
{
    for (int k = 0; k < 3; ++k) sP[FP_W1 + k * 256 + tid] = __ldg(P + TRT_MLP_W1 + 3 * tid + k);
    sP[FP_B1 + tid] = __ldg(P + TRT_MLP_B1 + tid);
    sP[FP_B2 + tid] = __ldg(P + TRT_MLP_B2 + tid);
    sP[FP_B3 + tid] = __ldg(P + TRT_MLP_B3 + tid);
    sP[FP_W4 + tid] = __ldg(P + TRT_MLP_W4 + tid);
    if (tid == 0) sP[FP_B4] = __ldg(P + TRT_MLP_B4);
}

// one lane of a converged warp, the same at every call
__device__ inline bool elect_one()
{
    unsigned p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// one contiguous bulk copy global -> this CTA's shared memory, completing (bytes) on `bar`
__device__ inline void bulk_copy(void *dst, const void *src, unsigned bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     su32(dst)),
                 "l"(src), "r"(bytes), "r"(su32(bar))
                 : "memory");
}

__global__ void __launch_bounds__(F_THREADS, 1) k_mlp_fused(int rows, const float *__restrict__ x,
                                                            const float *__restrict__ P,
                                                            const bf16 *__restrict__ Wimg,
                                                            float *__restrict__ y)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *sW = sm + 2 * FA_BYTES;   // F_SLOTS weight chunks
    float *sP = reinterpret_cast<float *>(sW + F_SLOTS * FW_BYTES);
    uint64_t *bar = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(sP) + FP_BYTES);
    uint64_t *full = bar, *empty = bar + F_SLOTS, *act = bar + 2 * F_SLOTS, *acc = act + 2;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + F_NBAR);
    int *sfail = reinterpret_cast<int *>(tslot + 1);
    int *sprod = sfail + 1, *scons = sfail + 2;   // chunks copied / expected (failure drain)
    uint64_t *dotb = acc + 2;
    float *sdot = reinterpret_cast<float *>(bar + F_NBAR) + 8;   // [2][128] head sums of columns 128 ..

    const int tid = threadIdx.x, warp = tid >> 5;
    const int ntiles = (rows - 1) / 256 + 1;
    const int mine = (int)blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

    if (tid == 0) {
        for (int k = 0; k < F_SLOTS; ++k) {
            mbar_init_n(&full[k], 1);
            mbar_init_n(&empty[k], 1);   // the commit of the MMAs that read the slot
        }
        for (int g = 0; g < 2; ++g) {
            mbar_init_n(&act[g], 256);
            mbar_init_n(&acc[g], 1);
            mbar_init_n(&dotb[g], 128);
        }
        *sfail = 0;
        *sprod = 0;
        *scons = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         su32(tslot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid < 256) stage_params(sP, P, tid);
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = *tslot;
    bool ok = true;

    const int Q = 4 * FNC * mine;   // weight chunks: 4 layer-jobs of FNC chunks per iteration
    if (warp == 16) {
        // ---------------- producer thread ----------------
        if ((tid & 31) == 0) {
            int q = 0, slot = 0;
            unsigned ph = 1;   // the slot's reuse waits for the phase before
            for (; q < Q; ++q) {   // chunk q: job q / FNC, K chunk q % FNC
                if (q >= F_SLOTS && !mbar_wait(&empty[slot], ph)) {
                    *sfail = 1;
                    break;
                }
                const int layer = (q / FNC) % 4 >= 2 ? 1 : 0;
                mbar_expect(&full[slot], FW_BYTES);
                bulk_copy(sW + slot * FW_BYTES,
                          Wimg + layer * 65536 + (q % FNC) * (FW_BYTES / 2), FW_BYTES,
                          &full[slot]);
                if (++slot == F_SLOTS) {
                    slot = 0;
                    ph ^= 1u;
                }
            }
            *sprod = q;
        }
    } else if (warp == 17) {
        // ---------------- MMA warp: one elected lane issues ----------------
        // the warp walks the chunks together, so that addresses and descriptors are uniform
        // values (a branch for one thread makes every operand of an MMA a register move)
        const bool lead = elect_one();
        unsigned pact = 0, ph = 0;   // bit g: parity of act[g]'s next phase; of the ring's
        int q = 0, slot = 0;
        const uint64_t wd = sdesc(su32(sW), FW_LBO, FW_SBO);
        for (int it = 0; it < mine && ok; ++it) {
            for (int job = 0; job < 4 && ok; ++job) {
                const int g = job & 1;
                if (!__all_sync(0xffffffffu, mbar_wait(&act[g], (pact >> g) & 1u))) { ok = false; break; }
                pact ^= 1u << g;
                tc_after();
                const uint64_t ad = sdesc(su32(sm + g * FA_BYTES), LBO, FA_SBO);
                const uint32_t d = tmem + (uint32_t)(g * 256);
#pragma unroll
                for (int c = 0; c < FNC; ++c, ++q) {
                    if (!__all_sync(0xffffffffu, mbar_wait(&full[slot], ph))) {
                        ok = false;
                        break;
                    }
                    const uint64_t bd = wd + (uint64_t)(slot * (FW_BYTES >> 4));
                    if (lead) {
#pragma unroll
                        for (int kk = 0; kk < FK / 16; ++kk)
                            umma(d, ad + (uint64_t)(((c * (FK / 8) + kk * 2) * 128) >> 4),
                                 bd + (uint64_t)((kk * 2 * FW_LBO) >> 4), (c | kk) != 0);
                        // the slot is free for chunk q + S once the MMAs reading it are done
                        umma_commit(&empty[slot]);
                    }
                    if (++slot == F_SLOTS) {
                        slot = 0;
                        ph ^= 1u;
                    }
                }
                if (!ok) break;
                if (lead) umma_commit(&acc[g]);   // the group's accumulator is complete
            }
        }
        if (lead) {
            if (!ok) *sfail = 1;
            *scons = q;   // chunks that have landed
        }
    } else {
        // -------- a group of eight warps: 128 rows, columns 128 half .. 128 half + 127 --------
        const int g = warp >> 3, half = (warp >> 2) & 1, r = tid & 127;
        unsigned char *myA = sm + g * FA_BYTES;
        const uint32_t tb = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(g * 256);
        unsigned pacc = 0, pdot = 0;
        auto wait_acc = [&]() {
            if (!mbar_wait(&acc[g], pacc)) {
                *sfail = 1;
                return false;
            }
            pacc ^= 1u;
            tc_after();
            return true;
        };
        auto hand_off = [&]() {   // A_g holds the next layer's input
            tc_before();
            fence_async_smem();
            mbar_arrive(&act[g]);
        };
        // layer 1: rows lane + 32 j, columns 32 w8 .. 32 w8 + 31 (w8: the warp within its group)
        const int lane = tid & 31, w8 = warp & 7;
        float xn[4][3];   // the tile's inputs (0 past the last row)
        // rows unsigned: a tile's last may lie past 2^31, and three values a row past 2^32
        auto load_x = [&](unsigned base) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const unsigned row = base + lane + 32 * j;
                const float *xr = x + 3 * (size_t)row;
#pragma unroll
                for (int k = 0; k < 3; ++k) xn[j][k] = row < (unsigned)rows ? xr[k] : 0.f;
            }
        };
        if (mine > 0) load_x(blockIdx.x * 256 + g * 128);
        for (int it = 0; it < mine && ok; ++it) {
            const unsigned base = (blockIdx.x + it * gridDim.x) * 256 + g * 128, row = base + r;
            const bool rv = row < (unsigned)rows;
            layer1_rows4<false>(sP, xn, myA, lane, 4 * w8, 4 * w8 + 4);
            // the next tile's inputs, in flight during the two layers
            if (it + 1 < mine) load_x(base + gridDim.x * 256);
            hand_off();
            if (!(ok = wait_acc())) break;
            // ---- epilogue of layer 2: h2 = relu(acc + b2) over h1 ----
            for (int ch = 4 * half; ch < 4 * half + 4; ch += 2) {   // 64 columns per tensor-memory wait
                uint32_t ra[32], rb[32];
                tmem_ld32_issue(tb + ch * 32, ra);
                tmem_ld32_issue(tb + ch * 32 + 32, rb);
                tmem_wait_tied(ra);
                reg_tie(rb);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const uint32_t *rr = k ? rb : ra;
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) {
                        const float4 *b2 = reinterpret_cast<const float4 *>(sP + FP_B2) + (ch + k) * 8 + qq * 2;
                        const float4 p0 = b2[0], p1 = b2[1];
                        const uint32_t *vq = rr + qq * 8;
                        uint4 u;
                        u.x = relu_bf16x2(add2(make_float2(__uint_as_float(vq[0]), __uint_as_float(vq[1])), make_float2(p0.x, p0.y)));
                        u.y = relu_bf16x2(add2(make_float2(__uint_as_float(vq[2]), __uint_as_float(vq[3])), make_float2(p0.z, p0.w)));
                        u.z = relu_bf16x2(add2(make_float2(__uint_as_float(vq[4]), __uint_as_float(vq[5])), make_float2(p1.x, p1.y)));
                        u.w = relu_bf16x2(add2(make_float2(__uint_as_float(vq[6]), __uint_as_float(vq[7])), make_float2(p1.z, p1.w)));
                        *reinterpret_cast<uint4 *>(myA + a_off(r, (ch + k) * 4 + qq)) = u;
                    }
                }
            }
            hand_off();
            if (!(ok = wait_acc())) break;
            // ---- epilogue of layer 3 and the head: y = sigmoid(w4 . relu(acc + b3) + b4) ----
            float2 dot = make_float2(0.f, 0.f);   // even and odd columns
            for (int ch = 4 * half; ch < 4 * half + 4; ch += 2) {   // 64 columns per tensor-memory wait
                uint32_t ra[32], rb[32];
                tmem_ld32_issue(tb + ch * 32, ra);
                tmem_ld32_issue(tb + ch * 32 + 32, rb);
                tmem_wait_tied(ra);
                reg_tie(rb);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const uint32_t *rr = k ? rb : ra;
#pragma unroll
                    for (int j4 = 0; j4 < 8; ++j4) {
                        const float4 b3 = reinterpret_cast<const float4 *>(sP + FP_B3)[(ch + k) * 8 + j4];
                        const float4 w4 = reinterpret_cast<const float4 *>(sP + FP_W4)[(ch + k) * 8 + j4];
                        float2 a = add2(make_float2(__uint_as_float(rr[4 * j4]), __uint_as_float(rr[4 * j4 + 1])),
                                        make_float2(b3.x, b3.y));
                        float2 c = add2(make_float2(__uint_as_float(rr[4 * j4 + 2]), __uint_as_float(rr[4 * j4 + 3])),
                                        make_float2(b3.z, b3.w));
                        a = make_float2(fmaxf(a.x, 0.f), fmaxf(a.y, 0.f));
                        c = make_float2(fmaxf(c.x, 0.f), fmaxf(c.y, 0.f));
                        dot = fma2(a, make_float2(w4.x, w4.y), dot);
                        dot = fma2(c, make_float2(w4.z, w4.w), dot);
                    }
                }
            }
            // the other half's sum through shared memory: its next write is a layer hand-off
            // later, which this half joins after it has read
            if (half) {
                sdot[g * 128 + r] = dot.x + dot.y;
                mbar_arrive(&dotb[g]);
            } else {
                if (!mbar_wait(&dotb[g], pdot)) {
                    *sfail = 1;
                    ok = false;
                    break;
                }
                pdot ^= 1u;
                const float z = (dot.x + dot.y) + sdot[g * 128 + r];
                if (rv) y[row] = 1.f / (1.f + __expf(-(z + sP[FP_B4])));
            }
        }
    }
    tc_before();
    __syncthreads();
    if (*sfail && tid == 0) {
        atomicExch(&g_mlp_err, TRT_ETIMEOUT);
        // let the producer's copies in flight land (bounded)
        for (int r = *scons; r < *sprod; ++r) mbar_wait(&full[r % F_SLOTS], (r / F_SLOTS) & 1);
    }
    __syncthreads();   // the drain above ends before TMEM is released
    if (warp == 0) {
        tc_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

// ---- training: forward, backward and weight gradients of 128 rows per CTA ----
// One CTA takes 128 rows through the whole step: the activations and layer gradients stay
// in two 64 KB shared-memory tiles (core-matrix layout of the fused inference kernel), the
// accumulators in tensor memory, and only the CTA's partial parameter gradients (FP32, one
// value per parameter) go to global memory; k_train_reduce adds the CTAs' partials in a
// fixed order.  Products per CTA (M 128, K 16 per instruction, BF16 in, FP32 accumulate):
//   h2 = relu(h1 W2^T), h3 = relu(h2 W3^T)          weights K-major from the streaming image
//   d2 = (d3 W3) [h2 > 0], d1 = (d2 W2) [h1 > 0]    the same image read MN-major: a K chunk
//                                                   (32 outputs) is a box of 32 rows of 512
//                                                   bytes, one tensor-map copy
//   dW3 = d3^T h2, dW2 = d2^T h1                    both operands MN-major from the tiles
// The weight gradients are 256 x 256: two halves of 128 output features, one after the other
// in columns 256 .. 511; the layers' accumulator is columns 0 .. 255.
// Warps 0-7 (thread = tensor-memory lane of quadrant warp & 3, columns 128 (warp >> 2) ..)
// run the layers' epilogues, warps 8-15 (the same lanes and columns) the column sums of the
// layer gradients and the weight gradients' way out, off the layers' chain; warp 16 streams
// weights through a ring of F_TSLOTS chunks, warp 17 issues the MMAs.  h1 is formed twice (3
// FMAs a value) because three tiles would leave the ring too small.  The loss head sums a
// row's 256 terms in column order in one chain, as the inference GEMM's epilogue does.
// What bounds it: 8192 rows are 64 CTAs of the 152 SMs, each a serial chain of 4 layer
// products (1 us each at the tensor rate) with their epilogues; the floor at the measured
// BF16 GEMM rate is 3.4 us.  Measured (8192 rows, gradient and Adam step): 39 us, against
// 1249 us for one GEMM launch per product, whose two weight gradients ran on two CTAs over K =
// 8192 (500 us) and whose column sums ran on 8 and 1 CTAs (520 us).
constexpr int F_TSLOTS = 5;
constexpr int F_TRING = F_TSLOTS * FW_BYTES;
constexpr int T_THREADS = 576;
constexpr int TNBAR = 2 * F_TSLOTS + 7;   // full, empty, act, acc, wac, drn, w3d, d3r, d2r
constexpr int T_SMEM = 2 * FA_BYTES + F_TRING + FP_BYTES + 128 * 16 + 3 * 128 * 4 + 8 * TNBAR + 32;
constexpr uint32_t IDESC_BT = IDESC | (1u << 16);                  // B MN-major
constexpr uint32_t IDESC_ABT = IDESC | (1u << 15) | (1u << 16);    // A and B MN-major
// one CTA's partials: dW2 and dW3 as float4 [i / 4][o] (stored by lanes that own o), then the
// other gradients at their parameter offsets less the matrices, b4, the loss
constexpr int TP_DW2 = 0, TP_DW3 = 65536, TP_W1 = 131072, TP_B1 = TP_W1 + 768, TP_B2 = TP_B1 + 256,
              TP_B3 = TP_B2 + 256, TP_W4 = TP_B3 + 256, TP_B4 = TP_W4 + 256, TP_LOSS = TP_B4 + 1,
              TP_N = TP_B4 + 4;

__device__ inline void bar_epi() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// sums over the 128 rows of the tile's 256 columns (each row times wr[row], or 1): warp w
// takes K groups 4 w .. 4 w + 3, lane = (K group & 3) * 8 + row % 8 (conflict-free 16-byte
// reads), 16 rows per lane, then the 8 lanes of a K group
template <bool kW>
__device__ inline void tile_colsum(const unsigned char *A, int warp, int lane, const float *wr,
                                   float *out)
{
    const int kg = warp * 4 + (lane >> 3), r8 = lane & 7;
    float s[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) s[j] = 0.f;
#pragma unroll 4
    for (int rg = 0; rg < 16; ++rg) {
        const uint4 u = *reinterpret_cast<const uint4 *>(A + a_off(rg * 8 + r8, kg));
        const float f = kW ? wr[rg * 8 + r8] : 1.f;
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float lo = __uint_as_float(w[j] << 16), hi = __uint_as_float(w[j] & 0xffff0000u);
            s[2 * j] = kW ? fmaf(lo, f, s[2 * j]) : s[2 * j] + lo;
            s[2 * j + 1] = kW ? fmaf(hi, f, s[2 * j + 1]) : s[2 * j + 1] + hi;
        }
    }
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) s[j] += __shfl_xor_sync(0xffffffffu, s[j], o);
        if (r8 == j) v = s[j];
    }
    out[kg * 8 + r8] = v;
}

// a box of 32 rows of 256 elements of the weight images (tensor map of launch_train), at
// element x of its rows y ..: one tile copy into shared memory, completing on `bar`
__device__ inline void tile_copy(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
                 "[%1, {%2, %3}], [%4];" ::"r"(su32(dst)),
                 "l"(map), "r"(x), "r"(y), "r"(su32(bar))
                 : "memory");
}

__global__ void __launch_bounds__(T_THREADS, 1) k_mlp_train(int rows, const float *__restrict__ x,
                                                            const float *__restrict__ target,
                                                            const float *__restrict__ P,
                                                            const bf16 *__restrict__ Wimg,
                                                            const __grid_constant__ CUtensorMap map,
                                                            float *__restrict__ part)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *A0 = sm, *A1 = sm + FA_BYTES, *ring = sm + 2 * FA_BYTES;
    float *sP = reinterpret_cast<float *>(ring + F_TRING);
    float4 *sx = reinterpret_cast<float4 *>(reinterpret_cast<unsigned char *>(sP) + FP_BYTES);
    float *sdot = reinterpret_cast<float *>(sx + 128), *sdz = sdot + 128, *ssq = sdz + 128;
    uint64_t *bar = reinterpret_cast<uint64_t *>(ssq + 128);
    uint64_t *full = bar, *empty = bar + F_TSLOTS, *act = bar + 2 * F_TSLOTS, *acc = act + 1,
             *wac = act + 2, *drn = act + 3;   // layer product, weight gradient half, its columns read
    // single-phase barriers of the two groups of warps, neither of which waits on the other's
    // every phase: dW3 formed, d3 in A0, d2 in A0
    uint64_t *w3d = act + 4, *d3r = act + 5, *d2r = act + 6;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + TNBAR);
    volatile int *sfail = reinterpret_cast<int *>(tslot + 1);
    volatile int *sprod = sfail + 1, *scons = sfail + 2;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row0 = blockIdx.x * 128;
    float *pt = part + (size_t)blockIdx.x * TP_N;

    if (tid == 0) {
        for (int k = 0; k < F_TSLOTS; ++k) {
            mbar_init_n(&full[k], 1);
            mbar_init_n(&empty[k], 1);
        }
        mbar_init_n(act, 256);
        mbar_init_n(acc, 1);
        mbar_init_n(wac, 1);
        mbar_init_n(drn, 256);
        mbar_init_n(w3d, 1);
        mbar_init_n(d3r, 256);
        mbar_init_n(d2r, 256);
        *sfail = 0;
        *sprod = 0;
        *scons = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         su32(tslot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    griddep_wait();   // the parameters and their image are the previous step's
    if (tid < 256) stage_params(sP, P, tid);
    if (tid < 128) {
        const size_t r = (size_t)(row0 + tid) * 3;
        sx[tid] = make_float4(x[r], x[r + 1], x[r + 2], 0.f);
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = *tslot;
    bool ok = true;

    constexpr int Q = 4 * FNC;   // chunks: W2, W3 (forward), W3, W2 (backward)
    if (warp == 16) {
        // ---------------- producer thread ----------------
        int q = 0;
        for (; lane == 0 && q < Q; ++q) {
            const int slot = q % F_TSLOTS, job = q / FNC, c = q % FNC;
            if (q >= F_TSLOTS && !mbar_wait(&empty[slot], ((q - F_TSLOTS) / F_TSLOTS) & 1)) {
                *sfail = 1;
                break;
            }
            const int layer = (job == 1 || job == 2) ? 1 : 0;
            unsigned char *dst = ring + slot * FW_BYTES;
            mbar_expect(&full[slot], FW_BYTES);
            if (job < 2)
                bulk_copy(dst, Wimg + layer * 65536 + c * (FW_BYTES / 2), FW_BYTES, &full[slot]);
            else   // inputs 8 i .. 8 i + 7 (box row i) of outputs 32 c .. 32 c + 31
                tile_copy(dst, &map, c * 256, layer * 32, &full[slot]);
        }
        if (lane == 0) *sprod = q;
    } else if (warp == 17) {
        // ---------------- MMA thread ----------------
        if (lane == 0) {
            int q = 0;
            unsigned pact = 0, pdrn = 0;
            const uint32_t a0 = su32(A0), a1 = su32(A1);
            auto wait_act = [&]() {
                if (ok && !mbar_wait(act, pact)) ok = false;
                pact ^= 1u;
                tc_after();
            };
            auto wait_drn = [&]() {
                if (ok && !mbar_wait(drn, pdrn)) ok = false;
                pdrn ^= 1u;
                tc_after();
            };
            // one layer product into columns 0 .. 255: A = a tile (K-major), B = 8 chunks
            auto layer = [&](uint32_t a, bool back) {
                for (int c = 0; c < FNC && ok; ++c, ++q) {
                    const int slot = q % F_TSLOTS;
                    if (!mbar_wait(&full[slot], (q / F_TSLOTS) & 1)) {
                        ok = false;
                        break;
                    }
                    const uint32_t w = su32(ring + slot * FW_BYTES);
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk) {
                        const uint64_t ad = sdesc(a + (c * 4 + kk * 2) * 128, LBO, FA_SBO);
                        if (back)   // outputs (K) 8 apart at 128 bytes, inputs (N) at 512
                            umma<IDESC_BT>(tmem, ad, sdesc(w + kk * 256, 128, 512), (c | kk) != 0);
                        else
                            umma(tmem, ad, sdesc(w + kk * 2 * FW_LBO, FW_LBO, FW_SBO), (c | kk) != 0);
                    }
                    umma_commit(&empty[slot]);
                }
                if (ok) umma_commit(acc);
            };
            // half hf (output features 128 hf ..) of A0^T A1 over the tile's 128 rows
            auto wgrad = [&](int hf) {
                if (!ok) return;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)   // rows 16 kk ..: row groups 4096 bytes apart
                    umma<IDESC_ABT>(tmem + 256, sdesc(a0 + hf * 2048 + kk * 8192, FA_SBO, 128),
                                    sdesc(a1 + kk * 8192, FA_SBO, 128), kk != 0);
                umma_commit(wac);
            };
            wait_act();             // h1 in A0
            layer(a0, false);
            wait_act();             // h2 in A1
            layer(a1, false);
            wait_act();             // d3 in A0
            wgrad(0);
            layer(a0, true);
            wait_drn();             // columns 256 .. 511 read
            wgrad(1);
            if (ok) umma_commit(w3d);
            wait_act();             // d2 in A0, h1 in A1
            layer(a0, true);
            wait_drn();
            wgrad(0);
            wait_drn();
            wgrad(1);
            if (!ok) *sfail = 1;
            *scons = q;
        }
    } else {
        // ---------------- epilogue warps ----------------
        const bool side = warp >= 8;   // the column sums and weight gradients
        const int qd = warp & 3, hf = (warp >> 2) & 1;
        const int r = qd * 32 + lane;       // the tile row, or the output feature of a gradient
        const uint32_t tb = tmem + ((uint32_t)(qd * 32) << 16);
        auto wait_bar = [&](uint64_t *b, unsigned &ph) {
            if (ok && !mbar_wait(b, ph)) {
                ok = false;
                *sfail = 1;
            }
            ph ^= 1u;
            __syncwarp();
            tc_after();
        };
        unsigned pacc = 0, pwac = 0, pw3 = 0, pd3 = 0, pd2 = 0;
        auto hand_off = [&]() {
            tc_before();
            fence_async_smem();
            mbar_arrive(act);
        };
        auto load32 = [&](uint32_t col, uint32_t (&v)[32]) {
            tmem_ld32_issue(tb + col, v);
            tmem_wait_tied(v);
        };
        // this thread's 128 columns of feature 128 half + r of a weight gradient
        auto drain = [&](int tp, int half) {
            wait_bar(wac, pwac);
            float4 *o = reinterpret_cast<float4 *>(pt + tp) + half * 128 + r;
#pragma unroll 1
            for (int ch = 4 * hf; ch < 4 * hf + 4; ++ch) {
                uint32_t v[32];
                load32(256 + ch * 32, v);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    o[(size_t)(ch * 8 + j) * 256] =
                        make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                    __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
            }
            tc_before();
            mbar_arrive(drn);
        };
        if (side) {
            wait_bar(d3r, pd3);
            tile_colsum<false>(A0, warp - 8, lane, nullptr, pt + TP_B3);
            drain(TP_DW3, 0);
            drain(TP_DW3, 1);
            wait_bar(d2r, pd2);
            tile_colsum<false>(A0, warp - 8, lane, nullptr, pt + TP_B2);
            drain(TP_DW2, 0);
            drain(TP_DW2, 1);
        } else {
        // layer 1: rows lane + 32 j, columns 32 warp .. 32 warp + 31
        const auto layer1 = [&](unsigned char *A) {
            float xr[4][3];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 X = sx[lane + 32 * j];
                xr[j][0] = X.x;
                xr[j][1] = X.y;
                xr[j][2] = X.z;
            }
            layer1_rows4<true>(sP, xr, A, lane, 4 * warp, 4 * warp + 4);
        };
        layer1(A0);
        hand_off();
        // ---- h2 = relu(acc + b2) ----
        wait_bar(acc, pacc);
#pragma unroll 1
        for (int ch = 4 * hf; ch < 4 * hf + 4; ++ch) {
            uint32_t v[32];
            load32(ch * 32, v);
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
                uint4 u;
                uint32_t *hw = reinterpret_cast<uint32_t *>(&u);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 b = *reinterpret_cast<const float2 *>(sP + FP_B2 + ch * 32 + qq * 8 + 2 * j);
                    const float2 a = add2(make_float2(__uint_as_float(v[qq * 8 + 2 * j]),
                                                      __uint_as_float(v[qq * 8 + 2 * j + 1])), b);
                    hw[j] = relu_bf16x2(make_float2(fmaxf(a.x, 0.f), fmaxf(a.y, 0.f)));
                }
                *reinterpret_cast<uint4 *>(A1 + a_off(r, ch * 4 + qq)) = u;
            }
        }
        hand_off();
        // ---- h3 = relu(acc + b3) into A0, the head in column order: the first half's
        // threads take columns 0 .. 127, the second half's go on from their sums ----
        wait_bar(acc, pacc);
        float dot = 0.f;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
            for (int ch = 4 * hf; ch < 4 * hf + 4; ++ch) {
                if (pass == 1 && hf == 0) break;
                uint32_t v[32];
                load32(ch * 32, v);
                float a[32];
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    a[j] = fmaxf(__uint_as_float(v[j]) + sP[FP_B3 + ch * 32 + j], 0.f);
                if (pass == 0) {
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) {
                        uint4 u;
                        uint32_t *hw = reinterpret_cast<uint32_t *>(&u);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            hw[j] = relu_bf16x2(make_float2(a[qq * 8 + 2 * j], a[qq * 8 + 2 * j + 1]));
                        *reinterpret_cast<uint4 *>(A0 + a_off(r, ch * 4 + qq)) = u;
                    }
                }
                if (pass == hf) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) dot = fmaf(a[j], sP[FP_W4 + ch * 32 + j], dot);
                }
            }
            if (pass == 0) {
                if (hf == 0) sdot[r] = dot;
                bar_epi();
                if (hf == 1) dot = sdot[r];
            }
        }
        if (hf == 1) {
            const float scale = 2.f / rows;
            const float z = dot + sP[FP_B4];
            const float y = 1.f / (1.f + __expf(-z));
            const float d = y - target[row0 + r];
            sdz[r] = scale * d * y * (1.f - y);
            ssq[r] = 0.5f * scale * d * d;
        }
        bar_epi();
        tile_colsum<true>(A0, warp, lane, sdz, pt + TP_W4);   // dw4 = sum dz h3
        if (warp == 0) {
            float s = (sdz[lane] + sdz[lane + 32]) + (sdz[lane + 64] + sdz[lane + 96]);
            float t = (ssq[lane] + ssq[lane + 32]) + (ssq[lane + 64] + ssq[lane + 96]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, o);
                t += __shfl_xor_sync(0xffffffffu, t, o);
            }
            if (lane == 0) {
                pt[TP_B4] = s;
                pt[TP_LOSS] = t;
            }
        }
        bar_epi();
        // ---- d3 = dz w4 [h3 > 0] over h3 ----
        {
            const float dz = sdz[r];
#pragma unroll 4
            for (int k8 = 16 * hf; k8 < 16 * hf + 16; ++k8) {
                uint4 *p = reinterpret_cast<uint4 *>(A0 + a_off(r, k8));
                uint4 u = *p;
                uint32_t *hw = reinterpret_cast<uint32_t *>(&u);
#pragma unroll
                for (int j = 0; j < 4; ++j) {   // h3 >= 0: positive where not zero
                    const float2 w = *reinterpret_cast<const float2 *>(sP + FP_W4 + k8 * 8 + 2 * j);
                    const __nv_bfloat162 g = __floats2bfloat162_rn((hw[j] & 0x7fffu) ? dz * w.x : 0.f,
                                                                   (hw[j] & 0x7fff0000u) ? dz * w.y : 0.f);
                    hw[j] = *reinterpret_cast<const uint32_t *>(&g);
                }
                *p = u;
            }
        }
        mbar_arrive(d3r);
        hand_off();
        // ---- d2 = acc [h2 > 0] over d3, h1 again over h2, once dW3 has read both (its second
        // half follows the column sums' read of d3) ----
        wait_bar(acc, pacc);
        wait_bar(w3d, pw3);
#pragma unroll 1
        for (int ch = 4 * hf; ch < 4 * hf + 4; ++ch) {
            uint32_t v[32];
            load32(ch * 32, v);
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
                const uint4 m = *reinterpret_cast<const uint4 *>(A1 + a_off(r, ch * 4 + qq));
                const uint32_t mw[4] = {m.x, m.y, m.z, m.w};
                uint4 u;
                uint32_t *hw = reinterpret_cast<uint32_t *>(&u);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const __nv_bfloat162 g = __floats2bfloat162_rn(
                        (mw[j] & 0x7fffu) ? __uint_as_float(v[qq * 8 + 2 * j]) : 0.f,
                        (mw[j] & 0x7fff0000u) ? __uint_as_float(v[qq * 8 + 2 * j + 1]) : 0.f);
                    hw[j] = *reinterpret_cast<const uint32_t *>(&g);
                }
                *reinterpret_cast<uint4 *>(A0 + a_off(r, ch * 4 + qq)) = u;
            }
        }
        mbar_arrive(d2r);
        bar_epi();   // every row's h2 has been read
        layer1(A1);
        hand_off();
        bar_epi();   // h1 of every row is in place for the mask below
        // ---- d1 = acc [h1 > 0] (FP32): its column sums, plain (b1) and times x (W1).  The
        // ring is free (the last layer product has read it): a warp stages 32 rows x 32
        // columns, lane = column sums its 32 rows, then the four row quadrants meet ----
        wait_bar(acc, pacc);
        float *stage = reinterpret_cast<float *>(ring) + warp * (32 * 33);
        float *quad = reinterpret_cast<float *>(ring) + 8 * 32 * 33;   // [4 sums][4 quadrants][256]
#pragma unroll 1
        for (int ch = 4 * hf; ch < 4 * hf + 4; ++ch) {
            uint32_t v[32];
            load32(ch * 32, v);
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
                const uint4 m = *reinterpret_cast<const uint4 *>(A1 + a_off(r, ch * 4 + qq));
                const uint32_t mw[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    stage[lane * 33 + qq * 8 + 2 * j] =
                        (mw[j] & 0x7fffu) ? __uint_as_float(v[qq * 8 + 2 * j]) : 0.f;
                    stage[lane * 33 + qq * 8 + 2 * j + 1] =
                        (mw[j] & 0x7fff0000u) ? __uint_as_float(v[qq * 8 + 2 * j + 1]) : 0.f;
                }
            }
            __syncwarp();
            float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 8
            for (int k = 0; k < 32; ++k) {
                const float dv = stage[k * 33 + lane];
                const float4 xr = sx[qd * 32 + k];
                s0 += dv;
                s1 = fmaf(dv, xr.x, s1);
                s2 = fmaf(dv, xr.y, s2);
                s3 = fmaf(dv, xr.z, s3);
            }
            const int c = ch * 32 + lane;
            quad[(0 * 4 + qd) * 256 + c] = s0;
            quad[(1 * 4 + qd) * 256 + c] = s1;
            quad[(2 * 4 + qd) * 256 + c] = s2;
            quad[(3 * 4 + qd) * 256 + c] = s3;
            __syncwarp();
        }
        bar_epi();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float *qs = quad + k * 1024 + tid;
            const float s = (qs[0] + qs[256]) + (qs[512] + qs[768]);
            if (k == 0) pt[TP_B1 + tid] = s;
            else pt[TP_W1 + 3 * tid + k - 1] = s;
        }
        }
    }
    tc_before();
    __syncthreads();
    if (*sfail && tid == 0) {
        atomicExch(&g_mlp_err, TRT_ETIMEOUT);
        for (int q = *scons; q < *sprod; ++q)   // the copies in flight land (bounded)
            mbar_wait(&full[q % F_TSLOTS], (q / F_TSLOTS) & 1);
    }
    __syncthreads();
    if (warp == 0) {
        tc_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

// grad and loss from the CTAs' partials: 64 float4 positions x 4 slices per block, slice s
// adds CTAs s, s + 4, ..., then the slices in order (fixed order, deterministic)
__global__ void __launch_bounds__(256) k_train_reduce(int nt, const float *__restrict__ part,
                                                      float *__restrict__ grad,
                                                      float *__restrict__ loss)
{
    __shared__ float4 red[4][64];
    griddep_wait();
    const int l = threadIdx.x & 63, sl = threadIdx.x >> 6;
    const int p = blockIdx.x * 64 + l;   // float4 index
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p < TP_N / 4) {
        const float4 *src = reinterpret_cast<const float4 *>(part) + p;
#pragma unroll 8
        for (int t = sl; t < nt; t += 4) {
            const float4 v = __ldcg(src + (size_t)t * (TP_N / 4));
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
    }
    red[sl][l] = s;
    __syncthreads();
    if (sl != 0 || p >= TP_N / 4) return;
#pragma unroll
    for (int k = 1; k < 4; ++k) {
        const float4 v = red[k][l];
        s.x += v.x;
        s.y += v.y;
        s.z += v.z;
        s.w += v.w;
    }
    if (p < TP_W1 / 4) {   // a matrix: float4 i4 of output o
        const int m = p >> 14, i4 = (p >> 8) & 63, o = p & 255;
        float *g = grad + (m ? TRT_MLP_W3 : TRT_MLP_W2) + o * 256 + i4 * 4;
        g[0] = s.x;
        g[1] = s.y;
        g[2] = s.z;
        g[3] = s.w;
        return;
    }
    const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int k = 4 * p + j;
        if (k < TP_B2) grad[TRT_MLP_W1 + k - TP_W1] = v[j];              // W1, then b1
        else if (k < TP_B3) grad[TRT_MLP_B2 + k - TP_B2] = v[j];
        else if (k < TP_LOSS) grad[TRT_MLP_B3 + k - TP_B3] = v[j];       // b3, w4, b4
        else if (k == TP_LOSS) *loss = v[j];
    }
}

// the weight images as a matrix of 64 rows (32 input groups of W2, then of W3; 4096 bytes: 256
// outputs x 8 inputs) for boxes of 32 rows x 32 outputs
cudaError_t image_map(const bf16 *img, CUtensorMap *map)
{
    typedef CUresult (*Encode)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                               const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                               CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                               CUtensorMapFloatOOBfill);
    static Encode encode = nullptr;   // the driver's entry point, the same for every device
    if (!encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                         cudaEnableDefault, &q);
        if (e != cudaSuccess) return e;
        if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        encode = reinterpret_cast<Encode>(fn);
    }
    const cuuint64_t dim[2] = {2048, 64}, pitch[1] = {4096};
    const cuuint32_t box[2] = {256, 32}, one[2] = {1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(img), dim,
                              pitch, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

int g_num_sms = 0;

cudaError_t mlp_fused(int rows, const float *x, const float *P, const bf16 *W, float *y,
                      cudaStream_t st)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t r = cudaFuncSetAttribute(k_mlp_fused,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, F_SMEM);
        if (r != cudaSuccess) return r;
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        attr = true;
    }
    // one persistent CTA per SM, no more CTAs than row tiles (a CTA left for a second wave
    // would double the time)
    const int ntiles = (rows - 1) / 256 + 1;
    const int grid = std::max(1, std::min(ntiles, g_num_sms > 0 ? g_num_sms : 148));
    k_mlp_fused<<<grid, F_THREADS, F_SMEM, st>>>(rows, x, P, (const bf16 *)(W + 4 * 65536), y);
    return cudaGetLastError();
}

cudaError_t gemm(int M, int N, int K, const bf16 *A, const bf16 *B, const Epi &e,
                 cudaStream_t st)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t r = cudaFuncSetAttribute(k_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             GEMM_SMEM);
        if (r != cudaSuccess) return r;
        attr = true;
    }
    dim3 grid((M + BM - 1) / BM, N / BN);
    k_gemm<<<grid, 128, GEMM_SMEM, st>>>(M, N, K, A, B, e);
    return cudaGetLastError();
}

// ---- MLP pieces on CUDA cores ----

// h1 = relu(W1 x + b1) per row (FP32), stored BF16 row-major
__global__ void k_layer1(int R, const float *__restrict__ x, const float *__restrict__ P,
                         bf16 *__restrict__ h1)
{
    __shared__ float w[TRT_MLP_HIDDEN * 4];
    for (int i = threadIdx.x; i < TRT_MLP_HIDDEN; i += blockDim.x) {
        w[4 * i + 0] = P[TRT_MLP_W1 + 3 * i + 0];
        w[4 * i + 1] = P[TRT_MLP_W1 + 3 * i + 1];
        w[4 * i + 2] = P[TRT_MLP_W1 + 3 * i + 2];
        w[4 * i + 3] = P[TRT_MLP_B1 + i];
    }
    __syncthreads();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    const float x0 = x[3 * r], x1 = x[3 * r + 1], x2 = x[3 * r + 2];
    uint4 *o = reinterpret_cast<uint4 *>(h1 + (size_t)r * TRT_MLP_HIDDEN);
    for (int q = 0; q < TRT_MLP_HIDDEN / 8; ++q) {
        uint4 u;
        bf16 *hb = reinterpret_cast<bf16 *>(&u);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = q * 8 + j;
            float a = w[4 * c + 3];
            a = fmaf(w[4 * c + 0], x0, a);
            a = fmaf(w[4 * c + 1], x1, a);
            a = fmaf(w[4 * c + 2], x2, a);
            hb[j] = __float2bfloat16_rn(fmaxf(a, 0.f));
        }
        o[q] = u;
    }
}

// W2, W3 (BF16), their transposes and their streaming images (the 16 KB chunks of the
// fused kernel, each laid out as it lands in shared memory) from the FP32 parameters
__device__ inline void store_w16(bf16 *w16, int layer, int o, int i, float v)
{
    const bf16 b = __float2bfloat16_rn(v);
    w16[layer * 65536 + o * 256 + i] = b;                 // W [out][in]
    w16[(2 + layer) * 65536 + i * 256 + o] = b;           // W^T [in][out]
    const int c = i >> 5, kg = (i >> 3) & 3, j = i & 7;   // chunk, K group, element
    w16[(4 + layer) * 65536 + c * 8192 + kg * 2048 + o * 8 + j] = b;
}

__global__ void k_refresh(const float *__restrict__ P, bf16 *__restrict__ w16)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;   // 2 x 65536
    if (idx >= 2 * 65536) return;
    const int layer = idx >> 16, o = (idx >> 8) & 255, i = idx & 255;
    store_w16(w16, layer, o, i, P[(layer ? TRT_MLP_W3 : TRT_MLP_W2) + o * 256 + i]);
}

// one Adam step, and the BF16 copies of the matrix elements it updated (k_refresh's, saving
// its launch and its read of the parameters)
__global__ void k_adam(int n, float *__restrict__ P, const float *__restrict__ g,
                       float *__restrict__ m, float *__restrict__ v, float lr, float b1,
                       float b2, float eps, float c1, float c2, bf16 *__restrict__ w16)
{
    griddep_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float p = P[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    P[i] = p;
    const int layer = i >= TRT_MLP_W3 ? 1 : 0;
    const int e = i - (layer ? TRT_MLP_W3 : TRT_MLP_W2);
    if (e >= 0 && e < 65536) store_w16(w16, layer, e >> 8, e & 255, p);
}

__global__ void k_features(int nx, int G, const double *__restrict__ T,
                           const double *__restrict__ sigE, const double *__restrict__ Eg,
                           const double *__restrict__ Ecell, float *__restrict__ x)
{
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)G * nx) return;
    const int i = (int)(idx % nx);
    const double t = fmax(T[i], 1e-30);
    const double s = fmax(sigE[idx], 1e-300);
    const double r = fmax(Eg[idx], 1e-300) / fmax(Ecell[i], 1e-300);
    x[3 * idx + 0] = (float)((log(t) + 3.5) * 0.5);
    x[3 * idx + 1] = (float)((log(s) - 10.0) * 0.1);
    x[3 * idx + 2] = (float)((log(r) + 10.0) * 0.1);
}

inline size_t al256(size_t x) { return (x + 255) / 256 * 256; }

struct Scratch {
    bf16 *h1, *h2;   // inference
    float *part;     // training: the CTAs' partial gradients
    size_t bytes;
};

Scratch carve_scratch(void *base, int R, int training)
{
    Scratch s{};
    char *p = reinterpret_cast<char *>(base);
    size_t o = 0;
    auto take = [&](size_t n) { char *q = p ? p + o : nullptr; o += al256(n); return q; };
    if (training) {
        s.part = reinterpret_cast<float *>(take((size_t)((R + 127) / 128) * TP_N * sizeof(float)));
    } else {
        s.h1 = reinterpret_cast<bf16 *>(take((size_t)R * TRT_MLP_HIDDEN * sizeof(bf16)));
        s.h2 = reinterpret_cast<bf16 *>(take((size_t)R * TRT_MLP_HIDDEN * sizeof(bf16)));
    }
    s.bytes = o;
    return s;
}

bool al16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

}  // namespace trt

using namespace trt;

extern "C" {

int trt_gemm_bf16(int M, int N, int K, const void *A, const void *B, const float *bias, int relu,
                  const void *mask, float *out32, void *out16, void *out16T, int ldT,
                  void *stream)
{
    if (M < 1 || N < BN || N % BN || K < BK || K % BK || !A || !B) return TRT_EINVAL;
    if (out16T && ldT < M) return TRT_EINVAL;
    if (!al16(A) || !al16(B) || !al16(mask) || !al16(out32) || !al16(out16)) return TRT_EINVAL;
    Epi e{};
    e.bias = bias;
    e.relu = relu;
    e.mask = reinterpret_cast<const bf16 *>(mask);
    e.out32 = out32;
    e.out16 = reinterpret_cast<bf16 *>(out16);
    e.out16T = reinterpret_cast<bf16 *>(out16T);
    e.ldT = ldT;
    cudaError_t r = gemm(M, N, K, reinterpret_cast<const bf16 *>(A),
                         reinterpret_cast<const bf16 *>(B), e, reinterpret_cast<cudaStream_t>(stream));
    return r == cudaSuccess ? TRT_OK : TRT_ECUDA;
}

size_t trt_mlp_scratch_bytes(int rows, int training)
{
    if (rows < 1) return 0;
    return carve_scratch(nullptr, rows, training).bytes;
}

int trt_mlp_refresh(const float *params, void *w16, void *stream)
{
    if (!params || !w16) return TRT_EINVAL;
    k_refresh<<<512, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        params, reinterpret_cast<bf16 *>(w16));
    return cudaGetLastError() == cudaSuccess ? TRT_OK : TRT_ECUDA;
}

int trt_mlp_forward_fused(int rows, const float *x, const float *params, const void *w16,
                          float *y, void *stream)
{
    if (rows < 1 || !x || !params || !w16 || !y) return TRT_EINVAL;
    if (!al16(params) || !al16(w16)) return TRT_EINVAL;   // w16: 16-byte pieces of the bulk copies
    return mlp_fused(rows, x, params, reinterpret_cast<const bf16 *>(w16), y,
                     reinterpret_cast<cudaStream_t>(stream)) == cudaSuccess
               ? TRT_OK
               : TRT_ECUDA;
}

int trt_mlp_forward(int rows, const float *x, const float *params, const void *w16,
                    void *scratch, size_t scratch_bytes, float *y, void *stream)
{
    if (rows < 1 || !x || !params || !w16 || !scratch || !y) return TRT_EINVAL;
    Scratch s = carve_scratch(scratch, rows, 0);
    if (scratch_bytes < s.bytes || !al16(scratch) || !al16(w16)) return TRT_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const bf16 *W = reinterpret_cast<const bf16 *>(w16);
    k_layer1<<<(rows + 127) / 128, 128, 0, st>>>(rows, x, params, s.h1);
    if (cudaGetLastError() != cudaSuccess) return TRT_ECUDA;
    Epi e2{};
    e2.bias = params + TRT_MLP_B2;
    e2.relu = 1;
    e2.out16 = s.h2;
    if (gemm(rows, 256, 256, s.h1, W, e2, st) != cudaSuccess) return TRT_ECUDA;
    Epi e3{};
    e3.bias = params + TRT_MLP_B3;
    e3.relu = 1;
    e3.head_w = params + TRT_MLP_W4;
    e3.head_b = params + TRT_MLP_B4;
    e3.head_y = y;
    if (gemm(rows, 256, 256, s.h2, W + 65536, e3, st) != cudaSuccess) return TRT_ECUDA;
    return TRT_OK;
}

int trt_mlp_grad(int rows, const float *x, const float *target, const float *params,
                 const void *w16, void *scratch, size_t scratch_bytes, float *grad, float *loss,
                 void *stream)
{
    if (rows < 128 || rows % 128 || !x || !target || !params || !w16 || !scratch || !grad ||
        !loss)
        return TRT_EINVAL;
    Scratch s = carve_scratch(scratch, rows, 1);
    if (scratch_bytes < s.bytes || !al16(scratch) || !al16(w16)) return TRT_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const bf16 *img = reinterpret_cast<const bf16 *>(w16) + 4 * 65536;
    const int nt = rows / 128;
    CUtensorMap map;
    if (image_map(img, &map) != cudaSuccess ||
        cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, T_SMEM) !=
            cudaSuccess ||
        launch_pdl(k_mlp_train, dim3(nt), dim3(T_THREADS), T_SMEM, st, rows, x, target, params, img,
                   map, s.part) != cudaSuccess ||
        launch_pdl(k_train_reduce, dim3((TP_N / 4 + 63) / 64), dim3(256), 0, st, nt,
                   (const float *)s.part, grad, loss) != cudaSuccess)
        return TRT_ECUDA;
    return TRT_OK;
}

int trt_mlp_adam(float *params, const float *grad, float *m, float *v, int t, float lr,
                 float beta1, float beta2, float eps, void *w16, void *stream)
{
    if (!params || !grad || !m || !v || t < 1 || !w16) return TRT_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const float c1 = 1.f - powf(beta1, (float)t), c2 = 1.f - powf(beta2, (float)t);
    return launch_pdl(k_adam, dim3((TRT_MLP_NPARAM + 255) / 256), dim3(256), 0, st, TRT_MLP_NPARAM,
                      params, grad, m, v, lr, beta1, beta2, eps, c1, c2,
                      reinterpret_cast<bf16 *>(w16)) == cudaSuccess
               ? TRT_OK
               : TRT_ECUDA;
}

int trt_mlp_features(int nx, int G, const double *T, const double *sigE, const double *Eg,
                     const double *E, float *x, void *stream)
{
    if (nx < 1 || G < 1 || !T || !sigE || !Eg || !E || !x) return TRT_EINVAL;
    const long n = (long)G * nx;
    k_features<<<(unsigned)((n + 255) / 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        nx, G, T, sigE, Eg, E, x);
    return cudaGetLastError() == cudaSuccess ? TRT_OK : TRT_ECUDA;
}

int trt_mlp_status(void)
{
    int v = 0, zero = 0;
    if (cudaDeviceSynchronize() != cudaSuccess) return TRT_ECUDA;
    if (cudaMemcpyFromSymbol(&v, g_mlp_err, sizeof(int)) != cudaSuccess) return TRT_ECUDA;
    if (cudaMemcpyToSymbol(g_mlp_err, &zero, sizeof(int)) != cudaSuccess) return TRT_ECUDA;
    return v;
}

}  // extern "C"
