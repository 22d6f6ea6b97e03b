// Kernels of the convolutional neural operator used as the learned surrogate
// of the LB step: 3x3 convolutions as implicit GEMMs on the sm_100-family
// tensor cores (tcgen05.mma, BF16 operands, FP32 accumulators in tensor
// memory, operands staged by TMA), plus the elementwise, reduction and
// optimiser kernels of training.
//
// Conventions (the same as the FP64 reference of the network):
//   activations NHWC bf16, channels a multiple of 64 (one 128-byte row);
//   weights W[o][t][i] bf16, tap t = 3 (dy + 1) + (dx + 1), zero padding;
//   y[n,h,w,o] = b[o] + sum_{t,i} x[n,h+dy,w+dx,i] W[o,t,i];
//   lrelu(z) = z (z > 0), z / 16 otherwise.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace cnok {

typedef __nv_bfloat16 bf16;

constexpr int BM = 128;             // tile rows of a GEMM (pixels, or output channels in wgrad)
constexpr int KB = 64;              // K elements per stage: 64 bf16 = one 128-byte swizzle row
constexpr int ROW_BYTES = 128;
constexpr int SUB_BYTES = 64 * ROW_BYTES;   // one 64-row x 128-byte TMA box
constexpr float LRELU_SLOPE = 0.0625f;
constexpr unsigned long long WAIT_NS = 4000000000ull;  // bound of every barrier wait

// status bits
constexpr unsigned ST_TIMEOUT_PRODUCER = 1u, ST_TIMEOUT_MMA = 2u, ST_TIMEOUT_EPILOGUE = 4u;

// --------------------------------------------------------------------------
// PTX wrappers
// --------------------------------------------------------------------------
// Programmatic dependent launch: the blocks of a kernel may be resident before the
// kernel in front of it has ended.  grid_begin waits for that kernel's end (its
// writes are then visible) and only then lets the kernel behind this one start its
// blocks, so at most two are ever in flight.  Every kernel launched that way calls
// it before its first access to global memory.  Its inputs may be written while it
// is resident, so it must not read them as read-only data: no __ldg, and no
// "const T *__restrict__" input, which lets the compiler choose such a load and move
// it over the wait (__restrict__ on what it writes is enough to overlap its loads).
__device__ __forceinline__ void grid_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase `parity` of a barrier to complete, for at most limit_ns;
// gives up early when another CTA has already reported a failure.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, const unsigned *status,
                                          unsigned long long limit_ns = WAIT_NS)
{
    if (mbar_try_wait(bar, parity))
        return true;
    const unsigned long long t0 = global_ns();
    for (unsigned it = 1;; it++) {
        if (mbar_try_wait(bar, parity))
            return true;
        if ((it & 63u) == 0u) {
            if (*(volatile const unsigned *)status != 0u)
                return false;
            if (global_ns() - t0 > limit_ns)
                return false;
        }
    }
}


// A CTA in which a wait was given up may have loads under way into its shared memory and
// MMAs that read it; it must not end before they are over.  Each role sets the abort
// flag when it gives up, and then the issuing threads wait for what they issued, by
// time alone (the status is set by then).  A CTA that ran to its end has seen the
// end of both: the MMAs waited for every load, and the epilogue for every MMA.
__device__ __noinline__ void mbar_drain(uint64_t *bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity))
        return;
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity) && global_ns() - t0 < WAIT_NS) {
    }
}
// The last load of each slot of a ring whose slots were filled `fills` times in turn.
template <int SLOTS>
__device__ __forceinline__ void drain_loads(uint64_t *full, int fills)
{
    for (int s = 0; s < SLOTS && s < fills; s++)
        mbar_drain(&full[s], ((fills - 1 - s) / SLOTS) & 1);
}

__device__ __forceinline__ void fence_barrier_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Self-test of the bounded wait: one thread waits on a barrier that nothing
// arrives at; the wait must give up after limit_ns and report it in out[0]
// (1: gave up), with the elapsed time in out[1] (ns).
__global__ void wait_selftest_kernel(unsigned long long limit_ns, const unsigned *status,
                                     unsigned long long *out)
{
    __shared__ uint64_t bar;
    mbar_init(&bar, 1);
    fence_barrier_init();
    const unsigned long long t0 = global_ns();
    const bool ok = mbar_wait(&bar, 0, status, limit_ns);
    out[0] = ok ? 0ull : 1ull;
    out[1] = global_ns() - t0;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2,
                                            int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t *holder, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(holder)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D (tensor memory, FP32) = A * B^T (+ D if accumulate): BF16 operands from
// shared memory descriptors, shape and majors in idesc.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrive on a barrier once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// All MMAs that this thread has issued (bar: used for nothing else).
__device__ __forceinline__ void drain_mmas(uint64_t *bar)
{
    umma_commit(bar);
    mbar_drain(bar, 0);
}

// 32 consecutive FP32 columns of the warp's 32 tensor-memory lanes.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; i++)
        v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor of a tcgen05 operand in the 128-byte
// swizzled layout: start address, leading- and stride-dimension byte offsets,
// descriptor version 1 (bits 46-48), swizzle mode 2 = 128 B (bits 61-63).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor of kind::f16 with BF16 A and B, FP32 D, M x N; a_mn /
// b_mn select the MN-major form of an operand (0: K-major).
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int a_mn, int b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ float lrelu(float z) { return z > 0.0f ? z : LRELU_SLOPE * z; }
__device__ __forceinline__ float lrelu_slope(float y) { return y > 0.0f ? 1.0f : LRELU_SLOPE; }

// --------------------------------------------------------------------------
// Convolution forward and data gradient: D[pixel][o] = sum_k A[pixel][k] B[o][k]
// with k = (tap, input channel), A gathered by TMA from the shifted input
// (zero fill outside the image), B the weight matrix.  A tile is 128 pixels
// (wt x ht of one image) by BN output channels.
//
// Persistent: each CTA takes tiles blockIdx.x, blockIdx.x + gridDim.x, ...
// Warp roles (6 warps): warp 0 lane 0 issues the TMA loads into a ring of
// stages, warp 1 owns the tensor memory and its lane 0 issues the MMAs, warps
// 2-5 run the epilogue, warp w reading tensor-memory lanes 32 (w % 4) ...
// 32 (w % 4) + 31.  Two accumulators in tensor memory alternate between tiles,
// so the epilogue of one tile overlaps the main loop of the next.
// --------------------------------------------------------------------------
enum { EPI_BIAS = 0, EPI_BIAS_LRELU = 1, EPI_SLOPE = 2, EPI_PLAIN = 3 };

struct ConvArgs {
    int n, h, w, cin, cout;
    int wt, ht, tiles_w, tiles_h, tiles;
    int kblocks, cblocks;
    int epi;
    const float *bias;          // EPI_BIAS*
    const bf16 *slope_src;      // EPI_SLOPE: y whose lrelu slope multiplies the result (NHWC, cout channels)
    void *out;                  // NHWC, out_cs channels per pixel
    int out_cs, n_store, out_f32;
    int ksteps;                 // conv64_kernel: 16-channel steps of a tap that can be non-zero (4: all)
    float *out2;                // FP32 outputs only: the first n2 <= min(8, n_store) channels again, out2_cs per pixel
    int out2_cs, n2;
    unsigned *status;
};

template <int BN>
struct ConvShape {
    static constexpr int A_BYTES = BM * ROW_BYTES;
    static constexpr int B_BYTES = BN * ROW_BYTES;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    // BN = 64: three CTAs per SM with 3 stages of 24 KB each (measured 4 % faster
    // over the whole forward pass than two CTAs with 4 stages); BN = 128: two
    // CTAs per SM, 96 KB of stages each (their accumulators fill the 512
    // tensor-memory columns); BN = 256: one CTA per SM, 4 stages
    static constexpr int CTAS_PER_SM = BN >= 256 ? 1 : (BN == 64 ? 3 : 2);
    static constexpr int STAGES = BN >= 256 ? 4 : (BN == 64 ? 3 : ((96 * 1024 / STAGE) < 2 ? 2 : (96 * 1024 / STAGE)));
    static constexpr int BAR_BYTES = 256;
    static constexpr int SMEM = STAGES * STAGE + 1024 /* alignment */ + BAR_BYTES + BN * 4 /* bias */;
    static constexpr int TMEM_COLS = 2 * BN;  // two FP32 accumulators
};

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// (At BN = 64 the bound keeps the kernel at 96 registers: with 104 a scheduler's
// register file holds four warps instead of five, so two CTAs fit instead of three
// and the 64-channel layers take 25 % longer.)
template <int BN>
__global__ void __launch_bounds__(192, ConvShape<BN>::CTAS_PER_SM)
    conv_fprop_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                      const ConvArgs a)
{
    using S = ConvShape<BN>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + S::STAGES * S::STAGE);
    uint64_t *empty = full + S::STAGES;
    uint64_t *acc_full = empty + S::STAGES;  // [2]: the MMAs of a tile are done
    uint64_t *acc_empty = acc_full + 2;      // [2]: the epilogue has read the accumulator
    uint64_t *drained = acc_empty + 2;
    uint32_t *tmem_holder = (uint32_t *)(drained + 1);
    volatile int *abort_flag = (volatile int *)(tmem_holder + 1);
    float *sbias = (float *)(smem + S::STAGES * S::STAGE + S::BAR_BYTES);

    grid_begin();
    if (*(volatile unsigned *)a.status != 0u)
        return;  // an earlier launch failed: leave the output untouched

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.y * BN;
    const bool has_bias = a.epi == EPI_BIAS || a.epi == EPI_BIAS_LRELU;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S::STAGES; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);  // one arrival per epilogue warp
        }
        mbar_init(drained, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp >= 2 && has_bias)
        for (int c = threadIdx.x - 64; c < BN; c += 128)
            sbias[c] = a.bias[n0 + c];
    if (warp == 1)
        tmem_alloc(tmem_holder, S::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_holder;
    uint32_t loads = 0;  // stages filled by this thread

    if (warp == 0 && lane == 0) {
        // producer: the stage ring runs on across tiles
        for (int tile = blockIdx.x; tile < a.tiles && !*abort_flag; tile += gridDim.x) {
            int t = tile;
            const int tw = t % a.tiles_w;
            t /= a.tiles_w;
            const int th = t % a.tiles_h;
            const int img = t / a.tiles_h;
            const int w0 = tw * a.wt, h0 = th * a.ht;
            int cb = 0, dx = -1, dy = -1;  // channel block and tap of kb
            for (int kb = 0; kb < a.kblocks; kb++, loads++) {
                const int s = loads % S::STAGES;
                const uint32_t use = loads / S::STAGES;
                if (use > 0 && !mbar_wait(&empty[s], (use - 1) & 1, a.status)) {
                    atomicOr(a.status, ST_TIMEOUT_PRODUCER);
                    *abort_flag = 1;
                    break;
                }
                uint8_t *sa = smem + s * S::STAGE;
                mbar_expect_tx(&full[s], S::STAGE);
                tma_load_4d(sa, &map_x, &full[s], cb * KB, w0 + dx, h0 + dy, img);
                tma_load_2d(sa + S::A_BYTES, &map_w, &full[s], kb * KB, n0);
                if (++cb == a.cblocks) {
                    cb = 0;
                    if (++dx == 2) {
                        dx = -1;
                        dy++;
                    }
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = idesc_bf16(BM, BN, 0, 0);
        uint32_t kc = 0;
        int it = 0;
        for (int tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, it++) {
            const int acc = it & 1, use = it >> 1;
            if (*abort_flag || (use > 0 && !mbar_wait(&acc_empty[acc], (use - 1) & 1, a.status))) {
                atomicOr(a.status, ST_TIMEOUT_MMA);
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const uint32_t dt = tmem + (uint32_t)(acc * BN);
            bool ok = true;
            for (int kb = 0; kb < a.kblocks; kb++, kc++) {
                const int s = kc % S::STAGES;
                if (*abort_flag || !mbar_wait(&full[s], (kc / S::STAGES) & 1, a.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t sa = smem_u32(smem + s * S::STAGE);
                const uint32_t sb = sa + S::A_BYTES;
#pragma unroll
                for (int k = 0; k < KB / 16; k++) {
                    // K-major, 128-byte swizzle: rows 128 B apart, 8-row groups 1024 B
                    // apart; the k-th 16-element slice starts 32 B further in.
                    const uint64_t ad = sw128_desc(sa + 32 * k, 16, 1024);
                    const uint64_t bd = sw128_desc(sb + 32 * k, 16, 1024);
                    umma_bf16(dt, ad, bd, idesc, (kb | k) != 0);
                }
                umma_commit(&empty[s]);
            }
            if (!ok) {
                atomicOr(a.status, ST_TIMEOUT_MMA);
                *abort_flag = 1;
                break;
            }
            umma_commit(&acc_full[acc]);
        }
    } else if (warp >= 2) {
        const int q = warp & 3;
        const int r = 32 * q + lane;
        int it = 0;
        for (int tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, it++) {
            const int acc = it & 1, use = it >> 1;
            // the tensor-memory loads are warp-collective: take the decision per warp
            const bool ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[acc], use & 1, a.status));
            if (!ok) {
                if (lane == 0) {
                    atomicOr(a.status, ST_TIMEOUT_EPILOGUE);
                    *abort_flag = 1;
                }
                break;
            }
            tc_fence_after();
            int t = tile;
            const int tw = t % a.tiles_w;
            t /= a.tiles_w;
            const int th = t % a.tiles_h;
            const int img = t / a.tiles_h;
            const int px = tw * a.wt + r % a.wt, py = th * a.ht + r / a.wt;
            const bool valid = px < a.w && py < a.h;
            const long long pix = ((long long)img * a.h + py) * a.w + px;
#pragma unroll 1
            for (int c0 = 0; c0 < BN; c0 += 32) {
                float v[32];
                tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * BN + c0), v);
                const int oc = n0 + c0;
                if (!valid || oc >= a.n_store)
                    continue;
                if (has_bias) {
#pragma unroll
                    for (int i = 0; i < 32; i++) {
                        const float z = v[i] + sbias[c0 + i];
                        v[i] = a.epi == EPI_BIAS_LRELU ? lrelu(z) : z;
                    }
                } else if (a.epi == EPI_SLOPE) {
                    const uint4 *ys = (const uint4 *)(a.slope_src + pix * a.cout + oc);
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        uint4 u = ys[j];
                        const bf16 *yb = (const bf16 *)&u;
#pragma unroll
                        for (int e = 0; e < 8; e++)
                            v[8 * j + e] *= lrelu_slope(__bfloat162float(yb[e]));
                    }
                }
                const int nst = min(32, a.n_store - oc);
                if (a.out_f32) {
                    if (a.out2 && oc == 0) {
                        float *o2 = a.out2 + pix * a.out2_cs;
#pragma unroll
                        for (int i = 0; i < 8; i++)
                            if (i < a.n2)
                                o2[i] = v[i];
                    }
                    float *o = (float *)a.out + pix * a.out_cs + oc;
                    if (nst == 8 && (a.out_cs & 3) == 0) {
                        ((float4 *)o)[0] = make_float4(v[0], v[1], v[2], v[3]);
                        ((float4 *)o)[1] = make_float4(v[4], v[5], v[6], v[7]);
                    } else if (nst == 32 && (a.out_cs & 3) == 0) {
#pragma unroll
                        for (int j = 0; j < 8; j++)
                            ((float4 *)o)[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; i++)
                            if (i < nst)
                                o[i] = v[i];
                    }
                } else {
                    bf16 *o = (bf16 *)a.out + pix * a.out_cs + oc;
                    if (nst == 32 && (a.out_cs & 7) == 0) {
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            uint4 u;
                            __nv_bfloat162 *p2 = (__nv_bfloat162 *)&u;
#pragma unroll
                            for (int e = 0; e < 4; e++)
                                p2[e] = __floats2bfloat162_rn(v[8 * j + 2 * e], v[8 * j + 2 * e + 1]);
                            ((uint4 *)o)[j] = u;
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; i++)
                            if (i < nst)
                                o[i] = __float2bfloat16_rn(v[i]);
                    }
                }
            }
            // the accumulator is read: hand it back to the MMA warp
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&acc_empty[acc]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (__builtin_expect(*abort_flag, 0)) {
        if (warp == 0 && lane == 0) {
            drain_loads<S::STAGES>(full, loads);
        } else if (warp == 1 && lane == 0) {
            drain_mmas(drained);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, S::TMEM_COLS);
    }
}

// --------------------------------------------------------------------------
// The same convolutions for 64 input channels (the full-resolution layers).  K is
// only 576, so conv_fprop_kernel moves 24 KB from L2 for every 128 x 64 x 64 step
// (each input pixel nine times, the weights once per tile) and is bound by that:
// 92 us for 1024^2 pixels, the tensor pipe 31 % active.  Here
//   - the weights (nine taps of BN x 64, 72 KB at BN = 64) stay in shared memory;
//   - a tile is 8 x 16 pixels and its input with the halo, 10 x 18 pixels, is one TMA
//     box of 23 KB.  Tap (dy, dx) is the same box read from pixel (dx, dy): the eight
//     pixels of an image row are one 8-row group of the operand (128 bytes a
//     pixel, swizzled by their address), and the groups lie 10 pixels (1280 bytes)
//     apart.  24 KB a tile instead of 216 KB;
//   - bf16 results go through shared memory and leave by TMA, one box of 8 x 4 pixels
//     per epilogue warp, and the activations whose slope multiplies a data gradient
//     come in by TMA: whole lines both ways, no masks.
// One persistent CTA per SM: TMA warp, MMA warp, four epilogue warps, two
// accumulators.  The taps are added in the same order as in conv_fprop_kernel, so
// the results are the same bits.  BN = 16 serves the head of small images, of whose 64
// outputs at most 16 are stored.
// --------------------------------------------------------------------------
constexpr int C64_W = 8, C64_H = 16;              // pixels of a tile
constexpr int C64_HW = C64_W + 2, C64_HH = C64_H + 2;

template <int BN, bool SLOPE>
struct Conv64Shape {
    static constexpr int A_BYTES = C64_HW * C64_HH * ROW_BYTES;
    static constexpr int A_STAGE = (A_BYTES + 1023) / 1024 * 1024;
    static constexpr int STAGES = SLOPE ? 3 : 4;
    static constexpr int TAP_BYTES = BN * ROW_BYTES;
    static constexpr int TILE_BYTES = BM * ROW_BYTES;  // 128 pixels of 64 bf16 channels
    static constexpr int OFF_A = 9 * TAP_BYTES;
    static constexpr int OFF_OUT = OFF_A + STAGES * A_STAGE;            // two staged output tiles
    static constexpr int OFF_SLOPE = OFF_OUT + (BN == 64 ? 2 : 0) * TILE_BYTES;  // two slope tiles
    static constexpr int OFF_BAR = OFF_SLOPE + (SLOPE ? 2 : 0) * TILE_BYTES;
    static constexpr int SMEM = OFF_BAR + 256 + BN * 4 + 1024 /* alignment */;
    static constexpr int TMEM_COLS = 2 * BN;
};

__device__ __forceinline__ void tma_store_4d(const CUtensorMap *map, const void *src, int c0, int c1, int c2, int c3)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(
                     (uint64_t)map),
                 "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(src))
                 : "memory");
}

// 16 consecutive FP32 columns of the warp's 32 tensor-memory lanes.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++)
        v[i] = __uint_as_float(r[i]);
}

template <int BN, bool SLOPE>
__global__ void __launch_bounds__(192, 1)
    conv64_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                  const __grid_constant__ CUtensorMap map_out, const __grid_constant__ CUtensorMap map_slope,
                  const ConvArgs a)
{
    using S = Conv64Shape<BN, SLOPE>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + S::OFF_BAR);
    uint64_t *empty = full + S::STAGES;
    uint64_t *w_full = empty + S::STAGES;
    uint64_t *acc_full = w_full + 1;    // [2]
    uint64_t *acc_empty = acc_full + 2; // [2]
    uint64_t *sl_full = acc_empty + 2;  // [2]
    uint64_t *sl_empty = sl_full + 2;   // [2]
    uint64_t *drained = sl_empty + 2;
    uint32_t *tmem_holder = (uint32_t *)(drained + 1);
    volatile int *abort_flag = (volatile int *)(tmem_holder + 1);
    float *sbias = (float *)(smem + S::OFF_BAR + 256);

    grid_begin();
    if (*(volatile unsigned *)a.status != 0u)
        return;  // an earlier launch failed: leave the output untouched

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.y * 64;
    const bool has_bias = a.epi == EPI_BIAS || a.epi == EPI_BIAS_LRELU;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S::STAGES; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(w_full, 1);
        for (int b = 0; b < 2; b++) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);
            mbar_init(&sl_full[b], 1);
            mbar_init(&sl_empty[b], 4);
        }
        mbar_init(drained, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp >= 2 && has_bias)
        for (int c = threadIdx.x - 64; c < BN; c += 128)
            sbias[c] = a.bias[n0 + c];
    if (warp == 1)
        tmem_alloc(tmem_holder, S::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_holder;
    int loads = 0, slopes = 0;  // tiles and slopes loaded by this thread

    auto place = [&](int tile, int &w0, int &h0, int &img) {
        const int tw = tile % a.tiles_w, r = tile / a.tiles_w;
        w0 = tw * C64_W;
        h0 = (r % a.tiles_h) * C64_H;
        img = r / a.tiles_h;
    };

    if (warp == 0 && lane == 0) {
        mbar_expect_tx(w_full, 9 * S::TAP_BYTES);
        for (int t = 0; t < 9; t++)
            tma_load_2d(smem + t * S::TAP_BYTES, &map_w, w_full, t * KB, n0);
        int it = 0;
        for (int tile = blockIdx.x; tile < a.tiles && !*abort_flag; tile += gridDim.x, it++) {
            int w0, h0, img;
            place(tile, w0, h0, img);
            const int s = it % S::STAGES, use = it / S::STAGES;
            if (use > 0 && !mbar_wait(&empty[s], (use - 1) & 1, a.status)) {
                atomicOr(a.status, ST_TIMEOUT_PRODUCER);
                *abort_flag = 1;
                break;
            }
            loads = it + 1;
            mbar_expect_tx(&full[s], S::A_BYTES);
            tma_load_4d(smem + S::OFF_A + s * S::A_STAGE, &map_x, &full[s], 0, w0 - 1, h0 - 1, img);
            if (SLOPE) {
                const int b = it & 1;
                if (it >= 2 && !mbar_wait(&sl_empty[b], ((it >> 1) - 1) & 1, a.status)) {
                    atomicOr(a.status, ST_TIMEOUT_PRODUCER);
                    *abort_flag = 1;
                    break;
                }
                slopes = it + 1;
                mbar_expect_tx(&sl_full[b], S::TILE_BYTES);
                tma_load_4d(smem + S::OFF_SLOPE + b * S::TILE_BYTES, &map_slope, &sl_full[b], n0, w0, h0, img);
            }
        }
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = idesc_bf16(BM, BN, 0, 0);
        const uint32_t sw = smem_u32(smem);
        int it = 0;
        bool ok = mbar_wait(w_full, 0, a.status);
        for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x, it++) {
            const int acc = it & 1, use = it >> 1, s = it % S::STAGES;
            ok = !*abort_flag && (use == 0 || mbar_wait(&acc_empty[acc], (use - 1) & 1, a.status)) &&
                 mbar_wait(&full[s], (it / S::STAGES) & 1, a.status);
            if (!ok)
                break;
            tc_fence_after();
            const uint32_t dt = tmem + (uint32_t)(acc * BN);
            const uint32_t sa = sw + S::OFF_A + s * S::A_STAGE;
#pragma unroll
            for (int t = 0; t < 9; t++) {
                // K-major, 128-byte swizzle; the k-th 16-element slice starts 32 B further in
                const uint64_t ad = sw128_desc(sa + ((t / 3) * C64_HW + t % 3) * ROW_BYTES, 16, C64_HW * ROW_BYTES);
                const uint64_t bd = sw128_desc(sw + t * S::TAP_BYTES, 16, 1024);
#pragma unroll
                for (int k = 0; k < KB / 16; k++)
                    if (k < a.ksteps)
                        umma_bf16(dt, ad + 2 * k, bd + 2 * k, idesc, (t | k) != 0);
            }
            umma_commit(&empty[s]);
            umma_commit(&acc_full[acc]);
        }
        if (!ok) {
            atomicOr(a.status, ST_TIMEOUT_MMA);
            *abort_flag = 1;
        }
    } else if (warp >= 2) {
        const int q = warp & 3;
        const int r = 32 * q + lane, px = r % C64_W, py = r / C64_W;
        int it = 0;
        for (int tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, it++) {
            const int acc = it & 1, use = it >> 1;
            // the tensor-memory loads are warp-collective: take the decision per warp
            bool ok = mbar_wait(&acc_full[acc], use & 1, a.status);
            if (SLOPE)
                ok = ok && mbar_wait(&sl_full[acc], use & 1, a.status);
            if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0) {
                    atomicOr(a.status, ST_TIMEOUT_EPILOGUE);
                    *abort_flag = 1;
                }
                break;
            }
            tc_fence_after();
            int w0, h0, img;
            place(tile, w0, h0, img);
            const uint32_t td = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * BN);
            if constexpr (BN == 64) {
                // this warp's 32 pixels (8 x 4) of the staged tile; the store two tiles ago has read them
                uint8_t *stage = smem + S::OFF_OUT + acc * S::TILE_BYTES + q * 32 * ROW_BYTES;
                const uint8_t *slope = smem + S::OFF_SLOPE + acc * S::TILE_BYTES + r * ROW_BYTES;
                if (lane == 0)
                    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                __syncwarp();
#pragma unroll
                for (int c0 = 0; c0 < BN; c0 += 32) {
                    float v[32];
                    tmem_ld32(td + (uint32_t)c0, v);
                    if (has_bias) {
#pragma unroll
                        for (int i = 0; i < 32; i++) {
                            const float z = v[i] + sbias[c0 + i];
                            v[i] = a.epi == EPI_BIAS_LRELU ? lrelu(z) : z;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const int chunk = ((c0 / 8 + j) ^ (lane & 7)) * 16;
                        if (SLOPE) {
                            const uint4 u = *(const uint4 *)(slope + chunk);
                            const bf16 *yb = (const bf16 *)&u;
#pragma unroll
                            for (int e = 0; e < 8; e++)
                                v[8 * j + e] *= lrelu_slope(__bfloat162float(yb[e]));
                        }
                        uint4 u;
                        __nv_bfloat162 *p2 = (__nv_bfloat162 *)&u;
#pragma unroll
                        for (int e = 0; e < 4; e++)
                            p2[e] = __floats2bfloat162_rn(v[8 * j + 2 * e], v[8 * j + 2 * e + 1]);
                        *(uint4 *)(stage + lane * ROW_BYTES + chunk) = u;
                    }
                }
                tc_fence_before();
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&acc_empty[acc]);
                    if (SLOPE)
                        mbar_arrive(&sl_empty[acc]);
                    if (h0 + 4 * q < a.h)
                        tma_store_4d(&map_out, stage, n0, w0, h0 + 4 * q, img);
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            } else {
                float v[16];
                tmem_ld16(td, v);
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(&acc_empty[acc]);
                if (w0 + px < a.w && h0 + py < a.h) {
                    const long long pix = ((long long)img * a.h + h0 + py) * a.w + w0 + px;
#pragma unroll
                    for (int i = 0; i < 16; i++) {
                        const float z = v[i] + (has_bias ? sbias[i] : 0.0f);
                        v[i] = a.epi == EPI_BIAS_LRELU ? lrelu(z) : z;
                    }
                    float *o = (float *)a.out + pix * a.out_cs;
                    if (a.n_store == 8 && (a.out_cs & 3) == 0) {
                        ((float4 *)o)[0] = make_float4(v[0], v[1], v[2], v[3]);
                        ((float4 *)o)[1] = make_float4(v[4], v[5], v[6], v[7]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; i++)
                            if (i < a.n_store)
                                o[i] = v[i];
                    }
                    if (a.out2) {
                        float *o2 = a.out2 + pix * a.out2_cs;
#pragma unroll
                        for (int i = 0; i < 8; i++)
                            if (i < a.n2)
                                o2[i] = v[i];
                    }
                }
            }
        }
        if (BN == 64 && lane == 0)
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    if (__builtin_expect(*abort_flag, 0)) {
        if (warp == 0 && lane == 0) {
            mbar_drain(w_full, 0);
            drain_loads<S::STAGES>(full, loads);
            drain_loads<2>(sl_full, slopes);
        } else if (warp == 1 && lane == 0) {
            drain_mmas(drained);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, S::TMEM_COLS);
    }
}

// --------------------------------------------------------------------------
// The same convolutions for 64 CB input channels (CB = 1, 2) and 128 output channels a
// tile, with the weights streamed: the input tile with its halo stays in shared memory (23 KB
// per 64 channels, read once instead of nine times), the weights come through a
// ring of G K blocks (a K block: 64 input channels of one tap) a stage.
// conv_fprop_kernel moves 32 KB per K block and was bound by that (600 cycles a
// block, 54 bytes a cycle and SM from L2, where the four N = 128 MMAs take 260);
// here it is 18.6 KB, and waiting for a stage and committing it, some 250 cycles of
// the issuing thread, is shared by G blocks.  Results and slopes pass through shared
// memory by TMA as in conv64_kernel, 64 channels at a time.  Same order of additions,
// same bits.  At 512^2, before -> now (us): 64 -> 128 channels 48.7 -> 34.1, 128 -> 128 74.6 -> 65.5,
// data gradient of 128 -> 128 with slopes 85.0 -> 66.4.  With 64 output channels a tile or four
// input blocks (one tile buffer) it was slower than conv_fprop_kernel: 128 -> 64 50.5 -> 57.9,
// 256 -> 256 at 256^2 57.5 -> 63.8.
// Warps: 0 weights, 1 MMAs, 2-5 epilogue, 6 input tiles.
// --------------------------------------------------------------------------
template <int CB>
struct ConvHaloShape {
    static constexpr int BN = 128;
    static constexpr int A_BYTES = C64_HW * C64_HH * ROW_BYTES;    // 64 channels of a tile
    static constexpr int A_BLOCK = (A_BYTES + 1023) / 1024 * 1024;
    static constexpr int A_BUFS = 2;
    static constexpr int B_BLOCK = BN * ROW_BYTES;
    static constexpr int G = CB == 1 ? 3 : 2;
    static constexpr int B_STAGES = 3;
    static constexpr int HALF_BYTES = BM * ROW_BYTES;              // 64 output channels of a tile
    static constexpr int OFF_B = A_BUFS * CB * A_BLOCK;
    static constexpr int OFF_OUT = OFF_B + B_STAGES * G * B_BLOCK; // two of them staged
    static constexpr int OFF_BAR = OFF_OUT + 2 * HALF_BYTES;
    static constexpr int SMEM = OFF_BAR + 256 + BN * 4 + 1024 /* alignment */;
    static constexpr int TMEM_COLS = 2 * BN;
    static_assert(9 * CB % G == 0, "a tile is whole stages");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

template <int CB, bool SLOPE>
__global__ void __launch_bounds__(224, 1)
    conv_halo_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                     const __grid_constant__ CUtensorMap map_out, const __grid_constant__ CUtensorMap map_slope,
                     const ConvArgs a)
{
    using S = ConvHaloShape<CB>;
    constexpr int BN = S::BN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *a_full = (uint64_t *)(smem + S::OFF_BAR);  // [2]
    uint64_t *a_empty = a_full + 2;                      // [2]
    uint64_t *b_full = a_empty + 2;                      // [3]
    uint64_t *b_empty = b_full + S::B_STAGES;            // [3]
    uint64_t *acc_full = b_empty + S::B_STAGES;          // [2]
    uint64_t *acc_empty = acc_full + 2;                  // [2]
    uint64_t *sl_full = acc_empty + 2;                   // [4 warps][2]
    uint64_t *drained = sl_full + 8;
    uint32_t *tmem_holder = (uint32_t *)(drained + 1);
    volatile int *abort_flag = (volatile int *)(tmem_holder + 1);
    float *sbias = (float *)(smem + S::OFF_BAR + 256);

    grid_begin();
    if (*(volatile unsigned *)a.status != 0u)
        return;  // an earlier launch failed: leave the output untouched

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.y * BN;
    const bool has_bias = a.epi == EPI_BIAS || a.epi == EPI_BIAS_LRELU;

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; b++) {
            mbar_init(&a_full[b], 1);
            mbar_init(&a_empty[b], 1);
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);
        }
        for (int s = 0; s < S::B_STAGES; s++) {
            mbar_init(&b_full[s], 1);
            mbar_init(&b_empty[s], 1);
        }
        for (int k = 0; k < 8; k++)
            mbar_init(&sl_full[k], 1);
        mbar_init(drained, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp >= 2 && warp < 6 && has_bias)
        for (int c = threadIdx.x - 64; c < BN; c += 128)
            sbias[c] = a.bias[n0 + c];
    if (warp == 1)
        tmem_alloc(tmem_holder, S::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_holder;
    int loads = 0;  // tiles, weight stages or slopes loaded by this thread

    auto place = [&](int tile, int &w0, int &h0, int &img) {
        const int tw = tile % a.tiles_w, r = tile / a.tiles_w;
        w0 = tw * C64_W;
        h0 = (r % a.tiles_h) * C64_H;
        img = r / a.tiles_h;
    };
    constexpr int NST = 9 * CB / S::G;  // weight stages of a tile

    if (warp == 6 && lane == 0) {
        int it = 0;
        for (int tile = blockIdx.x; tile < a.tiles && !*abort_flag; tile += gridDim.x, it++) {
            const int b = it % S::A_BUFS, use = it / S::A_BUFS;
            if (use > 0 && !mbar_wait(&a_empty[b], (use - 1) & 1, a.status)) {
                atomicOr(a.status, ST_TIMEOUT_PRODUCER);
                *abort_flag = 1;
                break;
            }
            int w0, h0, img;
            place(tile, w0, h0, img);
            loads = it + 1;
            mbar_expect_tx(&a_full[b], CB * S::A_BYTES);
            for (int c = 0; c < CB; c++)
                tma_load_4d(smem + (b * CB + c) * S::A_BLOCK, &map_x, &a_full[b], c * KB, w0 - 1, h0 - 1, img);
        }
    } else if (warp == 0 && lane == 0) {
        int s = 0, phase = 1;  // the first wait for an empty slot passes at once
        for (int tile = blockIdx.x; tile < a.tiles && !*abort_flag; tile += gridDim.x) {
            for (int st = 0; st < NST; st++) {
                if (!mbar_wait(&b_empty[s], phase, a.status)) {
                    atomicOr(a.status, ST_TIMEOUT_PRODUCER);
                    *abort_flag = 1;
                    break;
                }
                loads++;
                mbar_expect_tx(&b_full[s], S::G * S::B_BLOCK);
#pragma unroll
                for (int g = 0; g < S::G; g++)
                    tma_load_2d(smem + S::OFF_B + (s * S::G + g) * S::B_BLOCK, &map_w, &b_full[s],
                                (st * S::G + g) * KB, n0);
                if (++s == S::B_STAGES) {
                    s = 0;
                    phase ^= 1;
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = idesc_bf16(BM, BN, 0, 0);
        const uint32_t sw = smem_u32(smem);
        int it = 0, s = 0, phase = 0;
        bool ok = true;
        for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x, it++) {
            const int acc = it & 1, use = it >> 1, b = it % S::A_BUFS;
            ok = !*abort_flag && (use == 0 || mbar_wait(&acc_empty[acc], (use - 1) & 1, a.status)) &&
                 mbar_wait(&a_full[b], (it / S::A_BUFS) & 1, a.status);
            const uint32_t dt = tmem + (uint32_t)(acc * BN);
            int kb = 0;
            for (int st = 0; ok && st < NST; st++) {
                ok = mbar_wait(&b_full[s], phase, a.status);
                if (!ok)
                    break;
                tc_fence_after();
#pragma unroll
                for (int g = 0; g < S::G; g++, kb++) {
                    const int tap = kb / CB, c = kb % CB, dy = tap / 3;
                    const uint64_t ad = sw128_desc(sw + (b * CB + c) * S::A_BLOCK + (dy * (C64_HW - 3) + tap) * ROW_BYTES,
                                                   16, C64_HW * ROW_BYTES);
                    const uint64_t bd = sw128_desc(sw + S::OFF_B + (s * S::G + g) * S::B_BLOCK, 16, 1024);
#pragma unroll
                    for (int k = 0; k < KB / 16; k++)
                        umma_bf16(dt, ad + 2 * k, bd + 2 * k, idesc, (kb | k) != 0);
                }
                umma_commit(&b_empty[s]);
                if (++s == S::B_STAGES) {
                    s = 0;
                    phase ^= 1;
                }
            }
            if (ok) {
                umma_commit(&a_empty[b]);
                umma_commit(&acc_full[acc]);
            }
        }
        if (!ok) {
            atomicOr(a.status, ST_TIMEOUT_MMA);
            *abort_flag = 1;
        }
    } else if (warp >= 2 && warp < 6) {
        const int q = warp & 3;
        int it = 0;
        for (int tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, it++) {
            const int acc = it & 1;
            int w0, h0, img;
            place(tile, w0, h0, img);
            // staged output, 64 channels of this warp's 32 pixels (8 x 4): buffer (it * BN / 64 + hf) & 1
            auto stage = [&](int hf) {
                return smem + S::OFF_OUT + ((it * (BN / 64) + hf) & 1) * S::HALF_BYTES + q * 32 * ROW_BYTES;
            };
            if (SLOPE && lane == 0) {
                // the slopes into the staging buffers, once the stores have read them
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
#pragma unroll
                for (int hf = 0; hf < BN / 64; hf++) {
                    uint64_t *bar = &sl_full[2 * q + ((it * (BN / 64) + hf) & 1)];
                    loads++;
                    mbar_expect_tx(bar, 32 * ROW_BYTES);
                    tma_load_4d(stage(hf), &map_slope, bar, n0 + 64 * hf, w0, h0 + 4 * q, img);
                }
            }
            // the tensor-memory loads are warp-collective: take the decision per warp
            bool ok = mbar_wait(&acc_full[acc], (it >> 1) & 1, a.status);
#pragma unroll
            for (int hf = 0; hf < BN / 64; hf++)
                if (SLOPE) {
                    const int u = it * (BN / 64) + hf;  // use of the buffer u & 1
                    ok = ok && mbar_wait(&sl_full[2 * q + (u & 1)], (u >> 1) & 1, a.status);
                }
            if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0) {
                    atomicOr(a.status, ST_TIMEOUT_EPILOGUE);
                    *abort_flag = 1;
                }
                break;
            }
            tc_fence_after();
            const uint32_t td = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * BN);
#pragma unroll 1
            for (int hf = 0; hf < BN / 64; hf++) {
                uint8_t *row = stage(hf) + lane * ROW_BYTES;
                if (!SLOPE) {
                    if (lane == 0)
                        asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    __syncwarp();
                }
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 32) {
                    float v[32];
                    tmem_ld32(td + (uint32_t)(64 * hf + c0), v);
                    if (has_bias) {
#pragma unroll
                        for (int i = 0; i < 32; i++) {
                            const float z = v[i] + sbias[64 * hf + c0 + i];
                            v[i] = a.epi == EPI_BIAS_LRELU ? lrelu(z) : z;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        uint4 *at = (uint4 *)(row + ((c0 / 8 + j) ^ (lane & 7)) * 16);
                        if (SLOPE) {
                            const uint4 u = *at;
                            const bf16 *yb = (const bf16 *)&u;
#pragma unroll
                            for (int e = 0; e < 8; e++)
                                v[8 * j + e] *= lrelu_slope(__bfloat162float(yb[e]));
                        }
                        uint4 u;
                        __nv_bfloat162 *p2 = (__nv_bfloat162 *)&u;
#pragma unroll
                        for (int e = 0; e < 4; e++)
                            p2[e] = __floats2bfloat162_rn(v[8 * j + 2 * e], v[8 * j + 2 * e + 1]);
                        *at = u;
                    }
                }
                fence_proxy_async_smem();
                if (hf == BN / 64 - 1)
                    tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (hf == BN / 64 - 1)
                        mbar_arrive(&acc_empty[acc]);
                    if (h0 + 4 * q < a.h)
                        tma_store_4d(&map_out, stage(hf), n0 + 64 * hf, w0, h0 + 4 * q, img);
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            }
        }
        if (lane == 0)
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    if (__builtin_expect(*abort_flag, 0)) {
        if (lane == 0) {
            if (warp == 0)
                drain_loads<S::B_STAGES>(b_full, loads);
            else if (warp == 1)
                drain_mmas(drained);
            else if (warp == 6)
                drain_loads<S::A_BUFS>(a_full, loads);
            else
                drain_loads<2>(sl_full + 2 * (warp & 3), loads);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, S::TMEM_COLS);
    }
}

// --------------------------------------------------------------------------
// Weight gradient of one tap: D[o][i] = sum_p dz[p][o] x[p + s_tap][i] over a
// range of 64-pixel K blocks.  Both operands are loaded from the NHWC tensors
// as they are, so they are MN-major (the 64 channels of one pixel form one
// 128-byte row, consecutive pixels are consecutive K).  M = 128 output
// channels (two 64-channel boxes; a missing second box stays zero), N = BN
// input channels (BN / 64 boxes).  Each CTA writes its FP32 partial sum; a
// second kernel adds the partials of all pixel ranges in a fixed order.
// --------------------------------------------------------------------------
struct WgradArgs {
    int n, h, w, cin, cout;
    int wt, ht, tiles_w, tiles_h;   // 64-pixel K blocks: wt x ht pixels of one image
    int kb_total, kb_per_split, splits;
    int mtiles, ntiles;
    float *partial;                 // [splits][cout][9 cin]
    unsigned *status;
};

template <int BN>
struct WgradShape {
    static constexpr int A_BYTES = 2 * SUB_BYTES;
    static constexpr int B_BYTES = (BN / 64) * SUB_BYTES;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int STAGES = (96 * 1024 / STAGE) < 2 ? 2 : (96 * 1024 / STAGE);
    static constexpr int SMEM = STAGES * STAGE + 1024 + 256;
    static constexpr int TMEM_COLS = BN < 32 ? 32 : BN;
};

template <int BN>
__global__ void __launch_bounds__(192, 1)
    conv_wgrad_kernel(const __grid_constant__ CUtensorMap map_dz, const __grid_constant__ CUtensorMap map_x,
                      const WgradArgs a)
{
    using S = WgradShape<BN>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + S::STAGES * S::STAGE);
    uint64_t *empty = full + S::STAGES;
    uint64_t *done = empty + S::STAGES;
    uint64_t *drained = done + 1;
    uint32_t *tmem_holder = (uint32_t *)(drained + 1);
    volatile int *abort_flag = (volatile int *)(tmem_holder + 1);

    grid_begin();
    if (*(volatile unsigned *)a.status != 0u)
        return;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int b = blockIdx.x;
    const int tap = b % 9;
    b /= 9;
    const int mt = b % a.mtiles;
    const int nt = b / a.mtiles;
    const int m0 = mt * BM, n0 = nt * BN;
    const int dy = tap / 3 - 1, dx = tap % 3 - 1;
    const int split = blockIdx.y;
    const int kb_lo = split * a.kb_per_split;
    const int kb_hi = min(a.kb_total, kb_lo + a.kb_per_split);
    const bool two_m = m0 + 64 < a.cout;       // second 64-channel box of A present

    if (!two_m) {
        // the second half of every A stage stays zero (no TMA writes it)
        for (int s = 0; s < S::STAGES; s++) {
            uint4 *z = (uint4 *)(smem + s * S::STAGE + SUB_BYTES);
            for (int i = threadIdx.x; i < SUB_BYTES / 16; i += blockDim.x)
                z[i] = make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async_smem();
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < S::STAGES; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        mbar_init(drained, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1)
        tmem_alloc(tmem_holder, S::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_holder;
    const int nk = kb_hi - kb_lo;
    int loads = 0;  // stages filled by this thread

    if (warp == 0 && lane == 0) {
        const uint32_t bytes = (two_m ? 2 : 1) * SUB_BYTES + S::B_BYTES;
        // the K block's place, kept instead of divided for
        int tw = kb_lo % a.tiles_w, th = kb_lo / a.tiles_w % a.tiles_h, img = kb_lo / a.tiles_w / a.tiles_h;
        for (int j = 0; j < nk && !*abort_flag; j++) {
            const int s = j % S::STAGES, it = j / S::STAGES;
            if (j >= S::STAGES && !mbar_wait(&empty[s], (it - 1) & 1, a.status)) {
                atomicOr(a.status, ST_TIMEOUT_PRODUCER);
                *abort_flag = 1;
                break;
            }
            const int pw = tw * a.wt, ph = th * a.ht;
            uint8_t *st = smem + s * S::STAGE;
            loads = j + 1;
            mbar_expect_tx(&full[s], bytes);
            tma_load_4d(st, &map_dz, &full[s], m0, pw, ph, img);
            if (two_m)
                tma_load_4d(st + SUB_BYTES, &map_dz, &full[s], m0 + 64, pw, ph, img);
#pragma unroll
            for (int q = 0; q < BN / 64; q++)
                tma_load_4d(st + S::A_BYTES + q * SUB_BYTES, &map_x, &full[s], n0 + 64 * q, pw + dx, ph + dy, img);
            if (++tw == a.tiles_w) {
                tw = 0;
                if (++th == a.tiles_h) {
                    th = 0;
                    img++;
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = idesc_bf16(BM, BN, 1, 1);
        bool ok = true;
        for (int j = 0; j < nk; j++) {
            const int s = j % S::STAGES, it = j / S::STAGES;
            if (*abort_flag || !mbar_wait(&full[s], it & 1, a.status)) {
                atomicOr(a.status, ST_TIMEOUT_MMA);
                *abort_flag = 1;
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + s * S::STAGE);
            const uint32_t sb = sa + S::A_BYTES;
#pragma unroll
            for (int k = 0; k < KB / 16; k++) {
                // MN-major, 128-byte swizzle: 64 channels per 128-byte row, the
                // next 64 channels one box (8 KB) further (LBO); 8 pixel rows per
                // 1024-byte group (SBO); 16 pixels (2 KB) per MMA.
                const uint64_t ad = sw128_desc(sa + 2048 * k, SUB_BYTES, 1024);
                const uint64_t bd = sw128_desc(sb + 2048 * k, SUB_BYTES, 1024);
                umma_bf16(tmem, ad, bd, idesc, (j | k) != 0);
            }
            umma_commit(&empty[s]);
        }
        if (ok && nk > 0)
            umma_commit(done);
    } else if (warp >= 2) {
        const int q = warp & 3;
        const int o = m0 + 32 * q + lane;
        const int ldk = 9 * a.cin;
        float *dst = a.partial + ((long long)split * a.cout + o) * ldk + tap * a.cin + n0;
        if (nk == 0) {
            if (o < a.cout)
                for (int c = 0; c < BN; c++)
                    dst[c] = 0.0f;
        } else if (!__all_sync(0xffffffffu, mbar_wait(done, 0, a.status))) {
            if (lane == 0) {
                atomicOr(a.status, ST_TIMEOUT_EPILOGUE);
                *abort_flag = 1;
            }
        } else {
            tc_fence_after();
            for (int c0 = 0; c0 < BN; c0 += 32) {
                float v[32];
                tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0, v);
                if (o < a.cout) {
#pragma unroll
                    for (int j = 0; j < 8; j++)
                        ((float4 *)(dst + c0))[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (__builtin_expect(*abort_flag, 0)) {
        if (warp == 0 && lane == 0) {
            drain_loads<S::STAGES>(full, loads);
        } else if (warp == 1 && lane == 0) {
            drain_mmas(drained);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, S::TMEM_COLS);
    }
}

// --------------------------------------------------------------------------
// Weight gradient for 64 input channels, three taps of one image row offset dy at a
// time.  An MMA with M = 128 reads its A operand for about 64 cycles per 16 pixels
// whatever N <= 128 is, and conv_wgrad_kernel spends one on each tap, half of M
// empty at 64 output channels, loading 16 KB of pixels for four of them: 160 us for 16 x 256^2,
// 480 TFLOP/s.  Here M = 128 holds x at two column offsets a, N = 128 holds dz at
// two column offsets b, and the tap is dx = a - b:
//   D[(a, i)][(b, o)] = sum_p x[p + a + dy][i] dz[p + b][o],  a, b in {-1, 0}
//   (-1, 0): dx = -1;  (0, 0): dx = 0;  (0, -1): dx = +1;  (-1, -1): dx = 0 again, not used.
// Both offsets are the same staged pixels read one 128-byte row further on (the
// leading-dimension offset of the operands).  dz[-1] is the zero fill of the
// load, and the one pixel pair per row that no block holds, x[w] dz[w-1], is zero.
// A K block is 64 pixels: wt x ht of one image, loaded with one column more.
// Partials per pixel range as in conv_wgrad_kernel: [split][o][9 cin].
// --------------------------------------------------------------------------
// A stage is G K blocks: waiting for a stage and committing it costs the issuing
// thread some 250 cycles, an MMA 70 (at one block a stage, 148 us for 16 x 256^2; with
// half the loads, or with twice the stages, as long).  G = 4 where the CTAs fit
// one per SM, else G = 2 and two per SM.
template <int G>
struct Wgrad64Shape {
    static constexpr int SLOT = 9 * 1024;  // (wt + 1) ht <= 72 pixels of 128 bytes
    static constexpr int BLOCK = 2 * SLOT; // x, then dz
    static constexpr int STAGE = G * BLOCK;
    static constexpr int STAGES = 3;
    static constexpr int SMEM = STAGES * STAGE + 1024 + 256;
    static constexpr int TMEM_COLS = 128;
};

template <int G>
__global__ void __launch_bounds__(192, G == 4 ? 1 : 2)
    wgrad64_kernel(const __grid_constant__ CUtensorMap map_dz, const __grid_constant__ CUtensorMap map_x,
                   const WgradArgs a)
{
    using S = Wgrad64Shape<G>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + S::STAGES * S::STAGE);
    uint64_t *empty = full + S::STAGES;
    uint64_t *done = empty + S::STAGES;
    uint64_t *drained = done + 1;
    uint32_t *tmem_holder = (uint32_t *)(drained + 1);
    volatile int *abort_flag = (volatile int *)(tmem_holder + 1);

    grid_begin();
    if (*(volatile unsigned *)a.status != 0u)
        return;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int dy = (int)(blockIdx.x % 3) - 1, o0 = (int)(blockIdx.x / 3) * 64;
    const int split = blockIdx.y;
    const int kb_lo = split * a.kb_per_split;
    const int nk = min(a.kb_total, kb_lo + a.kb_per_split) - kb_lo;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S::STAGES; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        mbar_init(drained, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1)
        tmem_alloc(tmem_holder, S::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_holder;
    int loads = 0;  // stages filled by this thread
    const int pitch = (a.wt + 1) * ROW_BYTES;  // bytes of a staged image row

    // The two issuing threads keep their positions instead of dividing for them (which
    // took longer than a block's MMAs).
    if (warp == 0 && lane == 0) {
        const uint32_t bytes = 2 * pitch * a.ht;
        int tw = kb_lo % a.tiles_w, th = kb_lo / a.tiles_w % a.tiles_h, img = kb_lo / a.tiles_w / a.tiles_h;
        int s = 0, phase = 1;  // the parity of an empty slot's first wait is passed at once
        for (int j = 0; j < nk; j += G) {
            if (!mbar_wait(&empty[s], phase, a.status)) {
                atomicOr(a.status, ST_TIMEOUT_PRODUCER);
                *abort_flag = 1;
                break;
            }
            uint8_t *st = smem + s * S::STAGE;
            const int blocks = min(G, nk - j);
            loads++;
            mbar_expect_tx(&full[s], blocks * bytes);
            for (int g = 0; g < blocks; g++, st += S::BLOCK) {
                const int pw = tw * a.wt, ph = th * a.ht;
                tma_load_4d(st, &map_x, &full[s], 0, pw - 1, ph + dy, img);
                tma_load_4d(st + S::SLOT, &map_dz, &full[s], o0, pw - 1, ph, img);
                if (++tw == a.tiles_w) {
                    tw = 0;
                    if (++th == a.tiles_h) {
                        th = 0;
                        img++;
                    }
                }
            }
            if (++s == S::STAGES) {
                s = 0;
                phase ^= 1;
            }
        }
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = idesc_bf16(BM, 128, 1, 1);
        // 16 pixels per MMA: of one image row, or (wt = 8) eight of two rows each
        const uint32_t sbo = a.wt >= 16 ? 1024 : pitch;
        // MN-major, 128-byte swizzle: the two 64-channel halves are one pixel (128 B) apart
        const uint64_t base = sw128_desc(smem_u32(smem), ROW_BYTES, sbo);
        uint32_t off[4];  // of the block's k-th 16 pixels, in the descriptor's 16-byte units
#pragma unroll
        for (int k = 0; k < 4; k++)
            off[k] = (16 * k / a.wt * pitch + 16 * k % a.wt * ROW_BYTES) >> 4;
        int s = 0, phase = 0;
        bool ok = true;
        for (int j = 0; j < nk; j += G) {
            if (!mbar_wait(&full[s], phase, a.status)) {
                atomicOr(a.status, ST_TIMEOUT_MMA);
                *abort_flag = 1;
                ok = false;
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int g = 0; g < G; g++) {
                if (j + g >= nk)
                    break;
                const uint64_t at = base + (uint64_t)((s * S::STAGE + g * S::BLOCK) >> 4);
#pragma unroll
                for (int k = 0; k < 4; k++)
                    umma_bf16(tmem, at + off[k], at + off[k] + (S::SLOT >> 4), idesc, (j | g | k) != 0);
            }
            umma_commit(&empty[s]);
            if (++s == S::STAGES) {
                s = 0;
                phase ^= 1;
            }
        }
        if (ok && nk > 0)
            umma_commit(done);
    } else if (warp >= 2) {
        const int q = warp & 3;
        const int i = 32 * (q & 1) + lane;  // input channel; q / 2: column offset a + 1 of x
        const int ldk = 9 * 64, tap0 = 3 * (dy + 1);
        float *dst = a.partial + ((long long)split * a.cout + o0) * ldk + i;
        const bool have = nk > 0;
        const bool ok = !have || __all_sync(0xffffffffu, mbar_wait(done, 0, a.status));
        if (!ok) {
            if (lane == 0) {
                atomicOr(a.status, ST_TIMEOUT_EPILOGUE);
                *abort_flag = 1;
            }
        } else {
            tc_fence_after();
#pragma unroll 1
            for (int c0 = 0; c0 < 128; c0 += 32) {
                // columns (b + 1, o): b = -1 in 0 .. 63, b = 0 in 64 .. 127
                const int dx = (q >> 1) - (c0 >> 6);  // a - b
                if (c0 < 64 && q < 2)
                    continue;  // (-1, -1)
                float v[32];
                if (have)
                    tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0, v);
                float *d = dst + (long long)(c0 & 63) * ldk + (tap0 + dx + 1) * 64;
#pragma unroll
                for (int e = 0; e < 32; e++)
                    d[(long long)e * ldk] = have ? v[e] : 0.0f;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (__builtin_expect(*abort_flag, 0)) {
        if (warp == 0 && lane == 0) {
            drain_loads<S::STAGES>(full, loads);
        } else if (warp == 1 && lane == 0) {
            drain_mmas(drained);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, S::TMEM_COLS);
    }
}

__device__ __forceinline__ void unpack8(uint4 u, float (&f)[8])
{
    const __nv_bfloat162 *p = (const __nv_bfloat162 *)&u;
#pragma unroll
    for (int e = 0; e < 4; e++) {
        float2 t = __bfloat1622float2(p[e]);
        f[2 * e] = t.x;
        f[2 * e + 1] = t.y;
    }
}

__device__ __forceinline__ uint4 pack8(const float (&f)[8])
{
    uint4 u;
    __nv_bfloat162 *p = (__nv_bfloat162 *)&u;
#pragma unroll
    for (int e = 0; e < 4; e++)
        p[e] = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
    return u;
}

// dW[i] = sum over splits s (in order) of partial[s][i]; eight reads in flight
__global__ void __launch_bounds__(256) sum_partials_kernel(const float *partial, int splits,
                                                           long long count, float *__restrict__ out)
{
    grid_begin();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        float s = 0.0f;
        int k = 0;
        for (; k + 8 <= splits; k += 8) {
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; e++)
                v[e] = partial[(k + e) * count + i];
#pragma unroll
            for (int e = 0; e < 8; e++)
                s += v[e];
        }
        for (; k < splits; k++)
            s += partial[k * count + i];
        out[i] = s;
    }
}

// Bias gradient, first pass: block b adds dz (npix x c, bf16) over its pixel
// range [b * ppb, (b + 1) * ppb) per channel into partial[b][c].  Thread t reads
// 8 channels (16 bytes) of pixel p0 + t / (c / 8) + k * (256 / (c / 8)), so a
// warp's loads are contiguous; the threads of one channel group are then added
// in shared memory in a fixed order.  Bound by the read of dz: each thread keeps
// eight loads in flight (with one, 50 us for 134 MB, 2.7 TB/s).
__global__ void __launch_bounds__(256) channel_sum_kernel(const bf16 *dz, long long npix, int c,
                                                          long long ppb, float *__restrict__ partial)
{
    grid_begin();
    __shared__ float red[256][9];
    const int groups = c / 8;                 // 16-byte channel groups (c <= 2048)
    const int lanes_per_pix = groups;
    const int pix_step = 256 / lanes_per_pix; // pixels per sweep of the block (>= 1)
    const int g = threadIdx.x % lanes_per_pix, r = threadIdx.x / lanes_per_pix;
    const long long p0 = (long long)blockIdx.x * ppb;
    const long long p1 = min(npix, p0 + ppb);
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    auto add = [&](uint4 u) {
        float f[8];
        unpack8(u, f);
#pragma unroll
        for (int e = 0; e < 8; e++)
            acc[e] += f[e];
    };
    if (r < pix_step) {
        const uint4 *src = (const uint4 *)(dz + 8 * g);
        long long p = p0 + r;
        for (; p + 7 * pix_step < p1; p += 8 * pix_step) {
            uint4 u[8];
#pragma unroll
            for (int j = 0; j < 8; j++)
                u[j] = src[(p + j * pix_step) * groups];
#pragma unroll
            for (int j = 0; j < 8; j++)
                add(u[j]);
        }
        for (; p < p1; p += pix_step)
            add(src[p * groups]);
    }
#pragma unroll
    for (int e = 0; e < 8; e++)
        red[threadIdx.x][e] = acc[e];
    __syncthreads();
    for (int ch = threadIdx.x; ch < c; ch += 256) {
        const int gg = ch / 8, e = ch % 8;
        float sum = 0.0f;
        for (int rr = 0; rr < pix_step; rr++)
            sum += red[rr * lanes_per_pix + gg][e];
        partial[(long long)blockIdx.x * c + ch] = sum;
    }
}

// Bias gradient, second pass: db[ch] = sum of partial[b][ch] over the blocks, one
// block of 32 channels x 32 block groups, added in a fixed order.
__global__ void __launch_bounds__(1024) channel_total_kernel(const float *partial, int blocks, int c,
                                                             float *__restrict__ db)
{
    grid_begin();
    __shared__ float red[32][33];
    const int lane = threadIdx.x & 31, j = threadIdx.x >> 5, ch = blockIdx.x * 32 + lane;
    float s = 0.0f;
    if (ch < c)
        for (int b = j; b < blocks; b += 32)
            s += partial[(long long)b * c + ch];
    red[j][lane] = s;
    __syncthreads();
    // warp j adds the 32 group sums of channel j by a tree
    float t = red[lane][j];
    for (int o = 16; o > 0; o >>= 1)
        t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0 && blockIdx.x * 32 + j < c)
        db[blockIdx.x * 32 + j] = t;
}

// --------------------------------------------------------------------------
// Elementwise kernels on NHWC bf16 tensors, 8 channels (16 bytes) per thread.
// --------------------------------------------------------------------------
// y[n][h][w] = mean of x[n][2h..2h+1][2w..2w+1]; x is n x 2ho x 2wo
__global__ void pool2_kernel(const bf16 *x, int n, int ho, int wo, int c, bf16 *__restrict__ y)
{
    grid_begin();
    const int cv = c / 8;
    const long long total = (long long)n * ho * wo * cv;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i % cv);
        long long p = i / cv;
        const int ww = (int)(p % wo);
        p /= wo;
        const int hh = (int)(p % ho);
        const int nn = (int)(p / ho);
        const int wi = 2 * wo;
        float s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int dy = 0; dy < 2; dy++)
#pragma unroll
            for (int dxx = 0; dxx < 2; dxx++) {
                const long long q = (((long long)nn * 2 * ho + 2 * hh + dy) * wi + 2 * ww + dxx) * c + 8 * k;
                float f[8];
                unpack8(*(const uint4 *)(x + q), f);
#pragma unroll
                for (int e = 0; e < 8; e++)
                    s[e] += f[e];
            }
#pragma unroll
        for (int e = 0; e < 8; e++)
            s[e] *= 0.25f;
        *(uint4 *)(y + i * 8) = pack8(s);
    }
}

// u = up2(x) + skip; x is n x h/2 x w/2, skip and u n x h x w
__global__ void up_add_kernel(const bf16 *x, const bf16 *skip, int n, int h, int w, int c,
                              bf16 *__restrict__ u)
{
    grid_begin();
    const int cv = c / 8;
    const long long total = (long long)n * h * w * cv;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i % cv);
        long long p = i / cv;
        const int ww = (int)(p % w);
        p /= w;
        const int hh = (int)(p % h);
        const int nn = (int)(p / h);
        const long long q = (((long long)nn * (h / 2) + hh / 2) * (w / 2) + ww / 2) * c + 8 * k;
        float a[8], b[8];
        unpack8(*(const uint4 *)(x + q), a);
        unpack8(*(const uint4 *)(skip + i * 8), b);
#pragma unroll
        for (int e = 0; e < 8; e++)
            a[e] += b[e];
        *(uint4 *)(u + i * 8) = pack8(a);
    }
}

// Backward of u = up2(x) + skip followed by x = lrelu(.): dz[p] = slope(y[p]) *
// sum of du over the 2x2 block of p (y = x, the coarse activation)
__global__ void up_bwd_kernel(const bf16 *du, const bf16 *y, int n, int ho, int wo, int c,
                              bf16 *__restrict__ dz)
{
    grid_begin();
    const int cv = c / 8;
    const long long total = (long long)n * ho * wo * cv;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i % cv);
        long long p = i / cv;
        const int ww = (int)(p % wo);
        p /= wo;
        const int hh = (int)(p % ho);
        const int nn = (int)(p / ho);
        const int wi = 2 * wo;
        float s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int dy = 0; dy < 2; dy++)
#pragma unroll
            for (int dxx = 0; dxx < 2; dxx++) {
                const long long q = (((long long)nn * 2 * ho + 2 * hh + dy) * wi + 2 * ww + dxx) * c + 8 * k;
                float f[8];
                unpack8(*(const uint4 *)(du + q), f);
#pragma unroll
                for (int e = 0; e < 8; e++)
                    s[e] += f[e];
            }
        float yy[8];
        unpack8(*(const uint4 *)(y + i * 8), yy);
#pragma unroll
        for (int e = 0; e < 8; e++)
            s[e] *= lrelu_slope(yy[e]);
        *(uint4 *)(dz + i * 8) = pack8(s);
    }
}

// Backward at an encoder output e that feeds both a skip addition (gradient
// du) and pooling (gradient dp, at half resolution), followed by e = lrelu(.):
// dz[p] = slope(e[p]) * (du[p] + dp[p / 2] / 4)
__global__ void pool_bwd_kernel(const bf16 *du, const bf16 *dp, const bf16 *e,
                                int n, int h, int w, int c, bf16 *__restrict__ dz)
{
    grid_begin();
    const int cv = c / 8;
    const long long total = (long long)n * h * w * cv;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i % cv);
        long long p = i / cv;
        const int ww = (int)(p % w);
        p /= w;
        const int hh = (int)(p % h);
        const int nn = (int)(p / h);
        const long long q = (((long long)nn * (h / 2) + hh / 2) * (w / 2) + ww / 2) * c + 8 * k;
        float a[8], b[8], ee[8];
        unpack8(*(const uint4 *)(du + i * 8), a);
        unpack8(*(const uint4 *)(dp + q), b);
        unpack8(*(const uint4 *)(e + i * 8), ee);
#pragma unroll
        for (int j = 0; j < 8; j++)
            a[j] = lrelu_slope(ee[j]) * (a[j] + 0.25f * b[j]);
        *(uint4 *)(dz + i * 8) = pack8(a);
    }
}

// --------------------------------------------------------------------------
// Sums to FP64's accuracy from FP32 operations.  FP64 is the scarce pipe of this
// GPU (2 lane operations a cycle and SM).  A sum is held as three floats, h + m + l;
// sums and products of floats are exact as pairs (Knuth's TwoSum; an FMA for the
// product), so what is added to it loses nothing down to about 2^-68 of the sum.
// Products are exact as long as their rounding error does not underflow: the
// callers send operands too small or too large for that to FP64.
// --------------------------------------------------------------------------
struct f2 {
    float s, e;  // s + e: the result rounded, and its rounding error
};
struct f3 {
    float h, m, l;
};
__device__ __forceinline__ f2 two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ f2 two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
// a += x
__device__ __forceinline__ void f3_add(f3 &a, float x)
{
    const f2 s = two_sum(a.h, x), t = two_sum(a.m, s.e), r = two_sum(s.s, t.s);
    a.h = r.s;
    a.m = r.e;
    a.l = __fadd_rn(a.l, t.e);
}
// a += x + x1 + x2, each small beside the one before it
__device__ __forceinline__ void f3_add(f3 &a, float x, float x1, float x2 = 0.0f)
{
    const f2 s = two_sum(a.h, x), t = two_sum(a.m, s.e), u = two_sum(t.s, x1), r = two_sum(s.s, u.s);
    a.h = r.s;
    a.m = r.e;
    a.l = __fadd_rn(a.l, __fadd_rn(__fadd_rn(t.e, u.e), x2));
}
// a += x c
__device__ __forceinline__ void f3_add_product(f3 &a, float x, float c)
{
    const f2 p = two_prod(x, c);
    f3_add(a, p.s, p.e);
}
// The warp's sums in lane 0, in a fixed order.
__device__ __forceinline__ void f3_warp_sum(f3 &a, int lanes = 32)
{
    for (int o = lanes / 2; o > 0; o >>= 1)
        f3_add(a, __shfl_down_sync(0xffffffffu, a.h, o), __shfl_down_sync(0xffffffffu, a.m, o),
               __shfl_down_sync(0xffffffffu, a.l, o));
}
__device__ __forceinline__ double f3_value(const f3 &a) { return (double)a.h + ((double)a.m + (double)a.l); }

// Mean squared error over the first nf <= 8 channels of out (FP32, 8 per pixel)
// against target (FP32, nf per pixel).  dout (bf16, c per pixel) gets 2 (out -
// target) / count on those channels and 0 elsewhere; each block adds its squared
// errors into partial[block] (FP64).  A warp takes 32 pixels: each lane forms the
// gradient of its pixel, and the warp writes the pixels' rows in order, 512
// contiguous bytes per store.  The squares are exact pairs, added as above; a
// difference beyond 2^-48 .. 1e12 (NaN too) is squared and added in FP64.  Bound by
// the write of dout; in FP64, one row per thread, this took 259 us for 16 x 256^2
// (134 MB).
constexpr float SQUARE_MIN = 3.5527137e-15f, SQUARE_MAX = 1e12f;  // 2^-48
__global__ void __launch_bounds__(256) mse_kernel(const float *out, const float *target,
                                                  int nf, long long npix, int c, double inv_count,
                                                  bf16 *__restrict__ dout, double *__restrict__ partial)
{
    grid_begin();
    __shared__ f3 red[8];
    __shared__ double wred[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, cv = c / 8;
    const float scale = (float)(2.0 * inv_count);
    f3 sum = {0.0f, 0.0f, 0.0f};
    double wide = 0.0;  // squares taken in FP64
    for (long long g = blockIdx.x * 8LL + w; 32 * g < npix; g += gridDim.x * 8LL) {
        const long long p = 32 * g + lane;
        float d[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (p < npix) {
            const float4 a = ((const float4 *)out)[2 * p], b = ((const float4 *)out)[2 * p + 1];
            const float o[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int k = 0; k < 8; k++)
                if (k < nf)
                    d[k] = o[k] - target[p * nf + k];
        }
        float gr[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            gr[k] = scale * d[k];
            if (fabsf(d[k]) >= SQUARE_MIN && fabsf(d[k]) < SQUARE_MAX)
                f3_add_product(sum, d[k], d[k]);
            else if (d[k] != 0.0f)
                wide += (double)d[k] * (double)d[k];
        }
        const uint4 mine = pack8(gr);
        uint4 *row = (uint4 *)dout + 32 * g * cv;
        for (int j = 0; j < cv; j++) {
            const int q = 32 * j + lane, pix = q / cv, chunk = q - pix * cv;
            uint4 u;
            u.x = __shfl_sync(0xffffffffu, mine.x, pix);
            u.y = __shfl_sync(0xffffffffu, mine.y, pix);
            u.z = __shfl_sync(0xffffffffu, mine.z, pix);
            u.w = __shfl_sync(0xffffffffu, mine.w, pix);
            if (32 * g + pix < npix)
                row[q] = chunk == 0 ? u : make_uint4(0u, 0u, 0u, 0u);
        }
    }
    // the warps, then the block, in a fixed order
    f3_warp_sum(sum);
    if (__any_sync(0xffffffffu, wide != 0.0))  // true for NaN
        for (int o = 16; o > 0; o >>= 1)
            wide += __shfl_down_sync(0xffffffffu, wide, o);
    if (lane == 0) {
        red[w] = sum;
        wred[w] = wide;
    }
    __syncthreads();
    if (w == 0) {
        f3 s = red[lane & 7];
        f3_warp_sum(s, 8);
        if (lane == 0) {
            double t = f3_value(s);
            for (int j = 0; j < 8; j++)
                if (wred[j] != 0.0)
                    t += wred[j];
            partial[blockIdx.x] = t;
        }
    }
}

// Adam (Kingma and Ba, Algorithm 1) on FP32 master parameters; omb1 = 1 - beta1,
// omb2 = 1 - beta2, c1 = 1 - beta1^t, c2 = 1 - beta2^t, all rounded from FP64 on
// the host so that omb1 / c1 = omb2 / c2 = 1 exactly at t = 1.
__global__ void adam_kernel(float *__restrict__ p, const float *g, float *__restrict__ m,
                            float *__restrict__ v, long long count, float lr, float beta1, float beta2, float omb1,
                            float omb2, float eps, float c1, float c2)
{
    grid_begin();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = beta1 * m[i] + omb1 * gi;
        const float vi = beta2 * v[i] + omb2 * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// bf16 copies of FP32 weights W[o][t][i]: the forward matrix (same layout) and the
// data-gradient matrix Wd[i][t][o] = W[o][8 - t][i].  One launch takes the layers of
// a network (each block works on one of them; twelve launches of a few
// microseconds each took 51 us a training step).
constexpr int MAX_LAYERS = 12;
struct WeightLayers {
    int n;
    int block0[MAX_LAYERS + 1];  // first block of a layer
    int cout[MAX_LAYERS], cin[MAX_LAYERS];
    const float *w[MAX_LAYERS];
    bf16 *wf[MAX_LAYERS], *wd[MAX_LAYERS];
};

__global__ void __launch_bounds__(256) weights_to_bf16_kernel(const __grid_constant__ WeightLayers a)
{
    grid_begin();
    int l = 0;
    while (l + 1 < a.n && (int)blockIdx.x >= a.block0[l + 1])
        l++;
    const int cout = a.cout[l], cin = a.cin[l];
    const float *w = a.w[l];
    bf16 *__restrict__ wf = a.wf[l], *__restrict__ wd = a.wd[l];
    const long long total = (long long)cout * 9 * cin, step = (long long)(a.block0[l + 1] - a.block0[l]) * blockDim.x;
    for (long long idx = (blockIdx.x - a.block0[l]) * (long long)blockDim.x + threadIdx.x; idx < total; idx += step) {
        const int i = (int)(idx % cin);
        const int t = (int)((idx / cin) % 9);
        const int o = (int)(idx / (9LL * cin));
        const bf16 b = __float2bfloat16_rn(w[idx]);
        wf[idx] = b;
        wd[((long long)i * 9 + (8 - t)) * cout + o] = b;
    }
}

}  // namespace cnok
