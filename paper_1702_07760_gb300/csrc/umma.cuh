// Dense BF16 contraction on the 5th-generation tensor cores (tcgen05) for
// the learned surrogate: C = A B^T with A (M x K) and B (N x K) row-major
// BF16, FP32 accumulation in tensor memory (TMEM), fused epilogue.
//
// Per CTA: one 128-row tile of C and all N <= 256 columns.  K is consumed in
// chunks of up to 64; each chunk of A and B is brought to shared memory by the
// tensor memory accelerator (cp.async.bulk.tensor, one 2-D box of rows x 8
// elements per 8-wide k group) in the tensor core's K-major layout without
// swizzle ([k group][row][16 B]: core matrices of 8 rows x 16 bytes, 128 B
// apart along M and rows x 16 B apart along K), double buffered, and contracted by one thread issuing tcgen05.mma (M = 128, N,
// K = 16) into a TMEM accumulator of N columns.  The same thread issues the
// copies: a chunk's arrival and the completion of its MMAs (tcgen05.commit)
// are each signalled through an mbarrier; every wait gives up after one
// second, raising an error flag, and the CTA waits (again bounded) for its
// copies in flight and still releases its TMEM.  The accumulator is read with tcgen05.ld
// (each warp its 32-lane quarter) and stored as FP32, or added with
// atomics when K is split across CTAs.  That is k_gemm, for any K and N; the
// network's node layers run in k_layer (whole K in shared memory, persistent,
// with the layers' epilogues) and its weight gradients in k_wgrad (operands as
// stored, no transposes).
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

namespace umma {

constexpr int BM = 128;       // rows of a tile (MMA M)
constexpr int BK = 64;        // K of a staged chunk
constexpr int THREADS = 256;  // 8 warps: loads and epilogue (warps w and w+4 share a lane quarter)
constexpr unsigned ERR_TIMEOUT = 1u;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of a K-major operand without swizzle:
// start address, leading-dimension byte offset (between core matrices
// adjacent in K), stride-dimension byte offset (between 8-row groups), the
// descriptor version bit of tcgen05 (bit 46); base offset, offset mode and
// swizzle mode 0.
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo & 0x3FFFFu) >> 4) << 16;
    d |= (uint64_t)((sbo & 0x3FFFFu) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// Shared-memory matrix descriptor with the 128-byte swizzle (bits 61-63 = 2).
// K-major operand (rows of 64 BF16 = 128 bytes along K, 8-row atoms of 1024
// bytes): sbo = 1024 between 8-row groups, lbo unused; a K step of 16 starts
// 32 bytes further along the row.  M/N-major operand (rows of 64 features =
// 128 bytes, one row per K): lbo between 64-feature groups, sbo = 1024
// between 8-row K groups.  Atoms are 1024-byte aligned.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return desc_kmajor(saddr, lbo, sbo) | ((uint64_t)2 << 61);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), A
// and B BF16 (bits 7-9 and 10-12 = 1), both K-major (bits 15, 16 = 0),
// N >> 3 at bits 17-22, M >> 4 at bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t *mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *mbar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ bool mbar_try_wait(uint64_t *mbar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(mbar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Waits for the completion of the mbarrier phase with the given parity; false
// after one second without it.
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity)
{
    if (mbar_try_wait(mbar, parity)) return true;
    const unsigned long long t0 = now_ns();
    while (!mbar_try_wait(mbar, parity))
        if (now_ns() - t0 > 1000000000ull) return false;
    return true;
}

__device__ __forceinline__ void tmem_alloc(uint32_t *dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive FP32 accumulator columns of this thread's TMEM lane, the load
// and its wait in one statement, so that nothing that uses the values can be moved
// between them.  Both need the whole warp converged.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Expects `bytes` more transaction bytes on the mbarrier and arrives once.
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes)
                 : "memory");
}

// 2-D tensor copy global -> shared of the box at (x, y) = (k, row) of the
// tensor map; completion counted in bytes on the mbarrier.  x is a multiple
// of 8 elements (16 bytes) and dst 128-byte aligned.
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *mbar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(smem_u32(dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(mbar))
        : "memory");
}

__device__ __forceinline__ float silu(float z) { return z / (1.f + __expf(-z)); }

__device__ __forceinline__ float dsilu(float z)
{
    const float s = 1.f / (1.f + __expf(-z));
    return s * (1.f + z * (1.f - s));
}

// Arguments of one contraction C = A B^T (+ epilogue).
struct GemmArgs {
    const __nv_bfloat16 *A;
    int lda;                    // M x K, row-major, lda % 8 == 0
    const __nv_bfloat16 *B;
    int ldb;                    // N x K, row-major, ldb % 8 == 0
    int M, N, K;                // N in {16, 32, 64, 128, 256}; K % 16 == 0
    int k_split;                // K range of one CTA (multiple of 64); >= K: no split
    float *Cf;                  // FP32 output (or NULL)
    int ldcf;
    // from here to the fold for k_layer alone: k_gemm stores or adds the accumulator into Cf
    __nv_bfloat16 *Cb;          // BF16 output (or NULL); FP16 (__half) with the fold
    int ldcb;
    const float *bias;          // per column (or NULL)
    const float *row_scale;     // C[r][c] += row_scale[r] * row_bias[c] (or NULL)
    const float *row_bias;
    float *Z;                   // pre-activation output, FP32 (or NULL)
    int ldz;
    const float *residual;      // added after the activation (or NULL)
    int ldr;
    const float *residual2;     // added to the residual first (or NULL)
    int ldr2;
    int act;                    // 0 none, 1 SiLU, 2 multiply by SiLU'(dact) (backward)
    const float *dact;          // pre-activation for act == 2
    int lddact;
    int atomic;                 // 1: atomicAdd the accumulator into Cf (k_gemm; split K)
    unsigned *err;              // error word (ERR_TIMEOUT)
    // k_layer<256, 128> only: the result [P | Q] (128 columns each, rounded to
    // FP16 as Cb holds it) with the linear form s = W3d . f of the row's node
    // quantities f added to P and taken from Q, as FP16, to fold_out
    const float4 *fold_f;       // per row: up to three vector components and (w) a scalar (or NULL)
    const float *fold_w;        // 128 rows of fold_ldw: the vector's weights at fold_v, the scalar's at fold_s
    int fold_ldw, fold_v, fold_s, fold_dim;
    __half *fold_out;
    int fold_ld;
};

__device__ __forceinline__ bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// 16 consecutive FP32 values: four 16-byte accesses when aligned, else element by element.
__device__ __forceinline__ void store16(float *p, const float (&v)[16])
{
    if (aligned16(p)) {
#pragma unroll
        for (int q = 0; q < 4; ++q) ((float4 *)p)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) p[j] = v[j];
    }
}

// Issues the copies of K chunk [k0, k0 + kc) of A (rows row0...) and B into
// one buffer pair: kc / 8 boxes each, [k group][row][16 B].
template <int BN>
__device__ __forceinline__ void tma_chunk(uint8_t *a, uint8_t *b, const CUtensorMap *mA, const CUtensorMap *mB,
                                          int row0, int k0, int kc, uint64_t *bar)
{
    const int KG = kc / 8;
    mbar_arrive_expect_tx(bar, (uint32_t)(KG * (BM + BN) * 16));
    for (int kg = 0; kg < KG; ++kg) {
        tma_load_2d(a + kg * BM * 16, mA, k0 + kg * 8, row0, bar);
        tma_load_2d(b + kg * BN * 16, mB, k0 + kg * 8, 0, bar);
    }
}

template <int BN>
__global__ void __launch_bounds__(THREADS, 1)
    k_gemm(const __grid_constant__ GemmArgs g, const __grid_constant__ CUtensorMap mapA,
           const __grid_constant__ CUtensorMap mapB)
{
    constexpr int NCOLS = BN < 32 ? 32 : BN;
    constexpr int A_BYTES = BM * BK * 2;
    constexpr int B_BYTES = BN * BK * 2;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    // buffer b: A at smem + b * (A_BYTES + B_BYTES), B right after it
    auto bufA = [&](int b) { return smem + b * (A_BYTES + B_BYTES); };
    auto bufB = [&](int b) { return smem + b * (A_BYTES + B_BYTES) + A_BYTES; };
    __shared__ __align__(8) uint64_t mbar[2];   // MMAs of the chunk in buffer b complete
    __shared__ __align__(8) uint64_t lbar[2];   // copies into buffer b complete
    __shared__ uint32_t tmem_base;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row0 = blockIdx.x * BM;
    const int k_begin = blockIdx.y * g.k_split;
    const int k_end = min(g.K, k_begin + g.k_split);
    const int nchunks = (k_end - k_begin + BK - 1) / BK;

    if (warp == 0) {
        tmem_alloc(&tmem_base, NCOLS);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        mbar_init(&mbar[0], 1);
        mbar_init(&mbar[1], 1);
        mbar_init(&lbar[0], 1);
        mbar_init(&lbar[1], 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = tmem_base;
    const uint32_t idesc = idesc_bf16(BM, BN);

    bool failed = false;
    if (nchunks > 0) {
        if (threadIdx.x == 0) {
            // copies issued into each buffer (their arrivals are waited on by
            // phase parity (uses - 1) & 1)
            int issued[2] = {0, 0}, landed[2] = {0, 0};
            int committed = -1;  // last chunk whose MMAs were committed
            tma_chunk<BN>(bufA(0), bufB(0), &mapA, &mapB, row0, k_begin, min(BK, k_end - k_begin), &lbar[0]);
            issued[0] = 1;
            for (int c = 0; c < nchunks; ++c) {
                const int b = c & 1;
                if (c + 1 < nchunks) {
                    // buffer b^1 held chunk c-1: its MMAs must be complete before it is overwritten
                    if (c >= 1 && !mbar_wait(&mbar[b ^ 1], ((c - 1) >> 1) & 1)) {
                        failed = true;
                        break;
                    }
                    const int k0 = k_begin + (c + 1) * BK;
                    tma_chunk<BN>(bufA(b ^ 1), bufB(b ^ 1), &mapA, &mapB, row0, k0, min(BK, k_end - k0), &lbar[b ^ 1]);
                    issued[b ^ 1] += 1;
                }
                if (!mbar_wait(&lbar[b], (c >> 1) & 1)) {
                    failed = true;
                    break;
                }
                landed[b] += 1;
                tc_fence_after();
                const int k0 = k_begin + c * BK;
                const int kc = min(BK, k_end - k0);
                const uint32_t a0 = smem_u32(bufA(b)), b0 = smem_u32(bufB(b));
                for (int kk = 0; kk < kc / 16; ++kk) {
                    const uint64_t ad = desc_kmajor(a0 + kk * 2 * BM * 16, BM * 16, 128);
                    const uint64_t bd = desc_kmajor(b0 + kk * 2 * BN * 16, BN * 16, 128);
                    mma_bf16(taddr, ad, bd, idesc, (c > 0 || kk > 0) ? 1u : 0u);
                }
                mma_commit(&mbar[b]);
                committed = c;
            }
            if (failed) {
                // copies still in flight write this CTA's shared memory and
                // MMAs in flight its TMEM: wait for them (bounded) before the
                // CTA releases either (the last commit covers every MMA)
                for (int bb = 0; bb < 2; ++bb)
                    for (int u = landed[bb]; u < issued[bb]; ++u) mbar_wait(&lbar[bb], u & 1);
                if (committed >= 0) mbar_wait(&mbar[committed & 1], (committed >> 1) & 1);
            }
        }
        if (!__syncthreads_or(failed)) {
            const int last = nchunks - 1;
            failed = !mbar_wait(&mbar[last & 1], (last >> 1) & 1);
        }
        failed = __syncthreads_or(failed);
    }
    if (failed) {
        if (threadIdx.x == 0) atomicOr(g.err, ERR_TIMEOUT);
    } else {
        tc_fence_after();
        const int quarter = warp & 3;
        const int half = warp >> 2;
        const int row = row0 + quarter * 32 + lane;
        constexpr int COLS_PER_HALF = BN >= 32 ? BN / 2 : BN;
        const bool active = BN >= 32 || half == 0;
        if (active) {
            for (int cc = 0; cc < COLS_PER_HALF; cc += 16) {
                const int c0 = half * COLS_PER_HALF + cc;
                float v[16];
                __syncwarp();   // the lanes without a row came round ahead of the others
                if (nchunks > 0) {
                    tmem_ld16(taddr + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, v);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = 0.f;
                }
                if (row >= g.M) continue;
                // 16-byte vector accesses where the row's address allows them
                float *dst = g.Cf + (size_t)row * g.ldcf + c0;
                if (!g.atomic) {
                    store16(dst, v);
                } else if (aligned16(dst)) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        atomicAdd((float4 *)dst + q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) atomicAdd(dst + j, v[j]);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(taddr, NCOLS);
}

// ---------------------------------------------------------------------------
// One dense layer over many rows: C = A B^T with the whole K of both operands
// in shared memory (K = 16, 128 or 256), for the network's node layers.
//
// These contractions are bound by HBM (K <= 256: 64 to 128 flops a byte), so
// what counts is bytes in flight.  Persistent blocks keep the weights B in
// shared memory for all their 128-row tiles; a tile of A arrives by TMA in
// 128-byte swizzled rows (one box per 64 K columns; k_gemm's 16-byte boxes
// reach a tenth of the rate), the copy of the next tile is issued as soon as
// the MMAs have read this one and runs under the epilogue, and the blocks of
// an SM (two or more where the shared memory allows, else one block of 16
// warps) overlap each other's waits.  Epilogue: each warp moves 32 rows x 32
// columns of the accumulator from tensor memory to a 4 KB square of its own in
// shared memory (16-byte chunks XORed with the row: no bank conflicts either
// way) and reads it back with eight lanes a row, so every global access
// of the outputs, the residual and the pre-activation is a whole 128-byte
// line; a thread per row, as k_gemm stores, touches 32 lines an instruction.
// MMAs in ascending K, 16 at a time, as in k_gemm: the same bits.
// Measured (GB300, profiler, cold caches, 656 600 rows; k_gemm before): 128 ->
// 128 plain or FP32 + BF16 out 86 us on average (245), with the residual stream
// in and out 165 us (1.0 GB, 0.92 of the copy rate), 128 -> 16 35 us (82); the
// SiLU layers (111 to 147 us) and the folded P, Q layer (231 us; 288 and a
// pass of 321 us for the fold) are bound by their epilogues' instructions.  On
// 3 220 rows 6 to 12 us a layer (31).
template <int BN, int K>
struct LayerShape {
    static constexpr int NCOLS = BN < 32 ? 32 : BN;
    static constexpr int WARPS = BN == 16 ? 4 : (BN + K > 256 ? 16 : 8);
    static constexpr int BLOCKS = BN + K > 256 ? 1 : 2;   // resident blocks an SM
    static constexpr int A_BYTES = BM * K * 2;
    static constexpr int B_BYTES = BN * K * 2;
    static constexpr int B_ALIGNED = (B_BYTES + 1023) / 1024 * 1024;
    static constexpr int SMEM = A_BYTES + B_ALIGNED + WARPS * 4096 + 1024;
};

// Copies a tile of ROWS rows and the whole K: K = 16 as two 8-wide boxes
// without swizzle ([k group][row][16 B]), else one 128-byte swizzled box per
// 64 columns.
template <int ROWS, int K>
__device__ __forceinline__ void layer_load(uint8_t *dst, const CUtensorMap *map, int row0, uint64_t *bar)
{
    mbar_arrive_expect_tx(bar, (uint32_t)(ROWS * K * 2));
    if constexpr (K == 16) {
        tma_load_2d(dst, map, 0, row0, bar);
        tma_load_2d(dst + ROWS * 16, map, 8, row0, bar);
    } else {
#pragma unroll
        for (int c = 0; c < K / 64; ++c) tma_load_2d(dst + c * ROWS * 128, map, c * 64, row0, bar);
    }
}

// Epilogues of k_layer (compiled apart, so that each carries only its own loads).
enum LayerEpi { EPI_PLAIN, EPI_SILU, EPI_DSILU, EPI_RESIDUAL, EPI_FOLD };

template <int BN, int K, int EPI>
__global__ void __launch_bounds__(LayerShape<BN, K>::WARPS * 32, LayerShape<BN, K>::BLOCKS)
    k_layer(const __grid_constant__ GemmArgs g, const __grid_constant__ CUtensorMap mapA,
            const __grid_constant__ CUtensorMap mapB)
{
    using L = LayerShape<BN, K>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sA = smem, *sB = smem + L::A_BYTES;
    __shared__ __align__(8) uint64_t abar, bbar, mbar;   // tile of A in, weights in, MMAs done
    __shared__ uint32_t tmem_base;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntiles = (g.M + BM - 1) / BM;
    if (warp == 0) {
        tmem_alloc(&tmem_base, L::NCOLS);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        mbar_init(&abar, 1);
        mbar_init(&bbar, 1);
        mbar_init(&mbar, 1);
        fence_mbar_init();
        layer_load<BN, K>(sB, &mapB, 0, &bbar);
        layer_load<BM, K>(sA, &mapA, blockIdx.x * BM, &abar);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = tmem_base;
    const uint32_t idesc = idesc_bf16(BM, BN);
    float4 *const sq = (float4 *)(smem + L::A_BYTES + L::B_ALIGNED + warp * 4096);
    const int quarter = warp & 3, group = warp >> 2;
    constexpr int GROUPS = L::WARPS / 4;
    const int rsub = lane >> 3, c4 = lane & 7;   // read-back: row within four, 16-byte chunk

    bool failed = false;
    int it = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        bool ok = true;
        if (threadIdx.x == 0) {
            if (it == 0) ok = mbar_wait(&bbar, 0);
            ok = mbar_wait(&abar, it & 1) && ok;
            if (ok) {
                tc_fence_after();
                const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
#pragma unroll
                for (int kk = 0; kk < K / 16; ++kk) {
                    uint64_t ad, bd;
                    if constexpr (K == 16) {
                        ad = desc_kmajor(a0, BM * 16, 128);
                        bd = desc_kmajor(b0, BN * 16, 128);
                    } else {
                        ad = desc_sw128(a0 + (kk / 4) * BM * 128 + (kk % 4) * 32, 16, 1024);
                        bd = desc_sw128(b0 + (kk / 4) * BN * 128 + (kk % 4) * 32, 16, 1024);
                    }
                    mma_bf16(taddr, ad, bd, idesc, kk > 0 ? 1u : 0u);
                }
                mma_commit(&mbar);
                ok = mbar_wait(&mbar, it & 1);
                // the MMAs have read this tile: the next one's copy runs under the epilogue
                if (ok && tile + (int)gridDim.x < ntiles)
                    layer_load<BM, K>(sA, &mapA, (tile + gridDim.x) * BM, &abar);
            }
        }
        failed = __syncthreads_or(!ok);
        if (failed) break;
        tc_fence_after();
        const int row0 = tile * BM + quarter * 32;
#pragma unroll 1
        for (int c0 = group * 32; c0 < BN; c0 += GROUPS * 32) {
            if constexpr (BN >= 32) {
                float v[32];
                tmem_ld32(taddr + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    sq[lane * 8 + (q ^ (lane & 7))] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            } else {
                float v[16];
                tmem_ld16(taddr + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    sq[lane * 8 + (q ^ (lane & 7))] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
            __syncwarp();
            const int col = c0 + 4 * c4;
            if (col < BN) {
                float bias[4] = {0.f, 0.f, 0.f, 0.f}, rb4[4] = {0.f, 0.f, 0.f, 0.f};
                if (g.bias) *(float4 *)bias = *(const float4 *)(g.bias + col);
                if (g.row_scale) *(float4 *)rb4 = *(const float4 *)(g.row_bias + col);
                float wf[4][4];
                if constexpr (EPI == EPI_FOLD) {
                    const int f = col & 127;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float *w = g.fold_w + (size_t)(f + j) * g.fold_ldw;
                        wf[j][0] = w[g.fold_v];
                        wf[j][1] = w[g.fold_v + 1];
                        wf[j][2] = g.fold_dim == 3 ? w[g.fold_v + 2] : 0.f;
                        wf[j][3] = w[g.fold_s];
                    }
                }
                // rows in batches of 4 x RB: what the batch reads from global memory is asked for
                // before any of it is used (the outputs may alias the inputs, so loads do not
                // move above stores by themselves)
                constexpr int RB = 4;
#pragma unroll 1
                for (int rb = 0; rb < 32; rb += 4 * RB) {
                    float4 in[RB], in2[RB];
                    float scale[RB];
#pragma unroll
                    for (int t = 0; t < RB; ++t) {
                        const int row = min(row0 + rb + 4 * t + rsub, g.M - 1);
                        if constexpr (EPI == EPI_DSILU) in[t] = *(const float4 *)(g.dact + (size_t)row * g.lddact + col);
                        if constexpr (EPI == EPI_RESIDUAL) {
                            in[t] = *(const float4 *)(g.residual + (size_t)row * g.ldr + col);
                            if (g.residual2) in2[t] = *(const float4 *)(g.residual2 + (size_t)row * g.ldr2 + col);
                        }
                        if constexpr (EPI == EPI_FOLD) in[t] = g.fold_f[row];
                        if constexpr (EPI == EPI_PLAIN) scale[t] = g.row_scale ? g.row_scale[row] : 0.f;
                    }
#pragma unroll
                    for (int t = 0; t < RB; ++t) {
                        const int r = rb + 4 * t + rsub, row = row0 + r;
                        const float4 acc = sq[r * 8 + (c4 ^ (r & 7))];
                        if (row >= g.M) continue;
                        float v[4] = {acc.x, acc.y, acc.z, acc.w};
                        if (g.bias)
#pragma unroll
                            for (int j = 0; j < 4; ++j) v[j] += bias[j];
                        if constexpr (EPI == EPI_PLAIN)
                            if (g.row_scale)
#pragma unroll
                                for (int j = 0; j < 4; ++j) v[j] = fmaf(scale[t], rb4[j], v[j]);
                        if constexpr (EPI == EPI_SILU) {
                            if (g.Z) *(float4 *)(g.Z + (size_t)row * g.ldz + col) = make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
                            for (int j = 0; j < 4; ++j) v[j] = silu(v[j]);
                        }
                        if constexpr (EPI == EPI_DSILU) {
                            v[0] *= dsilu(in[t].x);
                            v[1] *= dsilu(in[t].y);
                            v[2] *= dsilu(in[t].z);
                            v[3] *= dsilu(in[t].w);
                        }
                        if constexpr (EPI == EPI_RESIDUAL) {
                            float4 q = in[t];
                            if (g.residual2) {
                                q.x += in2[t].x;
                                q.y += in2[t].y;
                                q.z += in2[t].z;
                                q.w += in2[t].w;
                            }
                            v[0] += q.x;
                            v[1] += q.y;
                            v[2] += q.z;
                            v[3] += q.w;
                        }
                        if (g.Cf) *(float4 *)(g.Cf + (size_t)row * g.ldcf + col) = make_float4(v[0], v[1], v[2], v[3]);
                        if constexpr (EPI == EPI_FOLD) {
                            const __half2 a = __floats2half2_rn(v[0], v[1]), b = __floats2half2_rn(v[2], v[3]);
                            if (g.Cb)
                                *(uint2 *)((__half *)g.Cb + (size_t)row * g.ldcb + col) =
                                    make_uint2(*(const uint32_t *)&a, *(const uint32_t *)&b);
                            const float4 f = in[t];
                            const float2 x = __half22float2(a), y = __half22float2(b);
                            float o[4] = {x.x, x.y, y.x, y.y};
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                float sd = __fmul_rn(wf[j][3], f.w);
                                sd = fmaf(wf[j][0], f.x, sd);
                                sd = fmaf(wf[j][1], f.y, sd);
                                if (g.fold_dim == 3) sd = fmaf(wf[j][2], f.z, sd);
                                o[j] = col < 128 ? o[j] + sd : o[j] - sd;
                            }
                            const __half2 oa = __floats2half2_rn(o[0], o[1]), ob = __floats2half2_rn(o[2], o[3]);
                            *(uint2 *)(g.fold_out + (size_t)row * g.fold_ld + col) =
                                make_uint2(*(const uint32_t *)&oa, *(const uint32_t *)&ob);
                        } else if (g.Cb) {
                            const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]),
                                                 b = __floats2bfloat162_rn(v[2], v[3]);
                            *(uint2 *)(g.Cb + (size_t)row * g.ldcb + col) =
                                make_uint2(*(const uint32_t *)&a, *(const uint32_t *)&b);
                        }
                    }
                }
            }
            __syncwarp();
        }
        // every warp has read the accumulator before the next tile's MMAs overwrite it
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }
    if (failed && threadIdx.x == 0) {
        atomicOr(g.err, ERR_TIMEOUT);
        // copies and MMAs in flight are waited for (bounded) before the memory is given up
        mbar_wait(&bbar, 0);
        mbar_wait(&abar, it & 1);
        mbar_wait(&mbar, it & 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(taddr, L::NCOLS);
}

// ---------------------------------------------------------------------------
// Weight gradient: dW (128 or fewer rows x BN columns) += sum over nodes of
// dY[node][row] X[node][col], both operands read as they are stored, one node
// a row: the tensor core takes them M/N-major (128-byte swizzled rows of 64
// features, one row per K), so no transposed copies are made.  (The transposes
// this replaces were 24 launches and 1.2 ms of a training step on 193 496
// particles, and the split kernel read them back in 16-byte boxes; 128 x 128 of
// that size now takes 27 us.)  Each
// block takes k_split nodes in chunks of 64 through a ring of
// WG_STAGES buffers, one thread issuing the copies and another the MMAs, and
// adds its sum to dW with FP32 atomics; blocks along y take 128 rows of dY
// each.  Rows and features beyond the arrays read as zero.  Same split and
// order of the nodes as k_gemm on the transposed copies.
constexpr int WG_STAGES = 4;
constexpr int WG_KC = 64;

struct WgradArgs {
    float *C;        // dW
    int ldc;
    int rows;        // rows of dW stored by the first block row (<= 128)
    int cols;        // columns stored (<= BN)
    int n;           // nodes
    int k_split;     // nodes of one block, a multiple of 64
    float *C2;       // dW of the second 128 features of dY (blockIdx.y == 1)
    unsigned *err;
};

template <int BN>
__global__ void __launch_bounds__(256, 1)
    k_wgrad(const __grid_constant__ WgradArgs g, const __grid_constant__ CUtensorMap mapY,
            const __grid_constant__ CUtensorMap mapX)
{
    constexpr int NCOLS = BN < 32 ? 32 : BN;
    constexpr int NB = (BN + 63) / 64;             // 64-feature groups of X
    constexpr int GB = WG_KC * 128;                // bytes of one group of a chunk
    constexpr int STAGE = (2 + NB) * GB;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[WG_STAGES], empty[WG_STAGES], done;
    __shared__ uint32_t tmem_base;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k0 = blockIdx.x * g.k_split, k1 = min(g.n, k0 + g.k_split);
    const int nchunks = (k1 - k0 + WG_KC - 1) / WG_KC;   // >= 1 (the grid covers the nodes)
    if (warp == 0) {
        tmem_alloc(&tmem_base, NCOLS);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < WG_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = tmem_base;
    // both operands M/N-major: bits 15 (A) and 16 (B)
    const uint32_t idesc = idesc_bf16(BM, BN) | (1u << 15) | (1u << 16);
    bool ok = true;
    if (threadIdx.x == 0) {
        int c = 0;
        for (; c < nchunks; ++c) {
            const int s = c % WG_STAGES, u = c / WG_STAGES;
            if (u > 0 && !(ok = mbar_wait(&empty[s], (u - 1) & 1))) break;
            uint8_t *st = smem + s * STAGE;
            mbar_arrive_expect_tx(&full[s], STAGE);
            const int y = k0 + c * WG_KC, f = blockIdx.y * BM;
            tma_load_2d(st, &mapY, f, y, &full[s]);
            tma_load_2d(st + GB, &mapY, f + 64, y, &full[s]);
#pragma unroll
            for (int q = 0; q < NB; ++q) tma_load_2d(st + (2 + q) * GB, &mapX, q * 64, y, &full[s]);
        }
        // every copy issued has landed before the block may end (bounded)
        for (int q = max(0, c - WG_STAGES); q < c; ++q) ok = mbar_wait(&full[q % WG_STAGES], (q / WG_STAGES) & 1) && ok;
    } else if (threadIdx.x == 32) {
        for (int c = 0; c < nchunks; ++c) {
            const int s = c % WG_STAGES, u = c / WG_STAGES;
            if (!(ok = mbar_wait(&full[s], u & 1))) break;
            tc_fence_after();
            const uint32_t a0 = smem_u32(smem + s * STAGE), b0 = a0 + 2 * GB;
#pragma unroll
            for (int kk = 0; kk < WG_KC / 16; ++kk)
                mma_bf16(taddr, desc_sw128(a0 + kk * 2048, GB, 1024), desc_sw128(b0 + kk * 2048, GB, 1024), idesc,
                         c > 0 || kk > 0 ? 1u : 0u);
            mma_commit(&empty[s]);
        }
        mma_commit(&done);
        ok = mbar_wait(&done, 0) && ok;
    }
    const bool failed = __syncthreads_or(!ok);
    if (failed) {
        if (threadIdx.x == 0) atomicOr(g.err, ERR_TIMEOUT);
    } else {
        tc_fence_after();
        const int quarter = warp & 3, half = warp >> 2;
        const int row = quarter * 32 + lane;
        float *const C = blockIdx.y == 0 ? g.C : g.C2;
        constexpr int PER_HALF = BN >= 32 ? BN / 2 : BN;
        if (BN >= 32 || half == 0) {
            for (int cc = 0; cc < PER_HALF; cc += 16) {
                const int c0 = half * PER_HALF + cc;
                float v[16];
                __syncwarp();   // the lanes without a row came round ahead of the others
                tmem_ld16(taddr + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, v);
                if (row >= g.rows) continue;
                float *dst = C + (size_t)row * g.ldc + c0;
                if (c0 + 16 <= g.cols && aligned16(dst)) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        atomicAdd((float4 *)dst + q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (c0 + j < g.cols) atomicAdd(dst + j, v[j]);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(taddr, NCOLS);
}

inline size_t gemm_smem_bytes(int BN) { return 2 * (size_t)(BM * BK * 2 + BN * BK * 2) + 1024; }

// cuTensorMapEncodeTiled of the driver, looked up once through the runtime.
inline PFN_cuTensorMapEncodeTiled_v12000 encode_tiled()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    });
    return fn;
}

// Tensor map of a row-major BF16 matrix (rows x cols, ld elements between
// rows) read in boxes of box_rows rows x box_cols elements: 8 without swizzle
// or 64 (128 bytes) with the 128-byte swizzle; rows beyond `rows` and
// columns beyond `cols` read as zero.  False when the base is not 16-byte
// aligned, ld not a multiple of 8, or the driver refuses the map.
inline bool make_map(CUtensorMap *m, const __nv_bfloat16 *base, int rows, int cols, int ld, int box_rows,
                     int box_cols = 8)
{
    const PFN_cuTensorMapEncodeTiled_v12000 fn = encode_tiled();
    if (!fn || ((uintptr_t)base & 15u) || ld % 8 != 0 || rows <= 0 || cols <= 0) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    const cuuint32_t step[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)base, dims, strides, box, step,
              CU_TENSOR_MAP_INTERLEAVE_NONE, box_cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, int K, int EPI>
inline cudaError_t launch_layer(const GemmArgs &g, cudaStream_t stream)
{
    using L = LayerShape<BN, K>;
    CUtensorMap mapA{}, mapB{};
    const int box = K == 16 ? 8 : 64;
    if (!make_map(&mapA, g.A, g.M, g.K, g.lda, BM, box) || !make_map(&mapB, g.B, g.N, g.K, g.ldb, g.N, box))
        return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_layer<BN, K, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM);
    if (e != cudaSuccess) return e;
    const int ntiles = (g.M + BM - 1) / BM;
    const int grid = ntiles < sms * L::BLOCKS ? ntiles : sms * L::BLOCKS;
    k_layer<BN, K, EPI><<<grid, L::WARPS * 32, L::SMEM, stream>>>(g, mapA, mapB);
    return cudaGetLastError();
}

using LayerLaunch = cudaError_t (*)(const GemmArgs &, cudaStream_t);

// The launch of the contraction by k_layer, NULL where it is not k_layer's.  The table holds the
// shapes and epilogues of the network (and the plain product of each shape); besides, every
// operand of the epilogue is on 16-byte boundaries in every row, and K is not split.  Plain and
// accumulated products with other N or K, a split K, odd leading dimensions or addresses are
// k_gemm's.
inline LayerLaunch layer_for(const GemmArgs &g)
{
    auto ok = [](const void *p, int ld) { return !p || ((uintptr_t)p % 16 == 0 && ld % 4 == 0); };
    if (g.atomic || g.k_split < g.K || !ok(g.Cf, g.ldcf) || !ok(g.Cb, g.ldcb) || !ok(g.Z, g.ldz) ||
        !ok(g.residual, g.ldr) || !ok(g.residual2, g.ldr2) || !ok(g.dact, g.lddact) || !ok(g.bias, 0) ||
        !ok(g.row_bias, 0))
        return nullptr;
    // one of activation, residual and fold; a pre-activation only with SiLU, a row-scaled bias with none
    const int kinds = (g.act != 0) + (g.residual != nullptr) + (g.fold_out != nullptr);
    if (kinds > 1 || (g.Z && g.act != 1) || (g.row_scale && kinds)) return nullptr;
    const int epi = g.fold_out ? EPI_FOLD
                               : (g.residual ? EPI_RESIDUAL : (g.act == 1 ? EPI_SILU : (g.act == 2 ? EPI_DSILU : EPI_PLAIN)));
#define SPH_LAYER_CASE(BN, KK, EPI) \
    if (g.N == BN && g.K == KK && epi == EPI) return launch_layer<BN, KK, EPI>;
    SPH_LAYER_CASE(128, 16, EPI_PLAIN)
    SPH_LAYER_CASE(128, 16, EPI_SILU)
    SPH_LAYER_CASE(128, 16, EPI_DSILU)
    SPH_LAYER_CASE(128, 128, EPI_PLAIN)
    SPH_LAYER_CASE(128, 128, EPI_SILU)
    SPH_LAYER_CASE(128, 128, EPI_DSILU)
    SPH_LAYER_CASE(128, 128, EPI_RESIDUAL)
    SPH_LAYER_CASE(128, 256, EPI_PLAIN)
    SPH_LAYER_CASE(128, 256, EPI_SILU)
    SPH_LAYER_CASE(128, 256, EPI_RESIDUAL)
    SPH_LAYER_CASE(256, 128, EPI_PLAIN)
    SPH_LAYER_CASE(256, 128, EPI_FOLD)
    SPH_LAYER_CASE(16, 128, EPI_PLAIN)
#undef SPH_LAYER_CASE
    return nullptr;
}

// dW += dY^T X over n nodes: dY has fy features (rows of dW, 128 to a block
// row: dW, then dW2), X has fx = 16, 128 or 256 (cols of them stored).
inline cudaError_t wgrad(const __nv_bfloat16 *dY, int ldy, int fy, const __nv_bfloat16 *X, int ldx, int fx, int n,
                         float *dW, float *dW2, int ldc, int rows, int cols, int k_split, unsigned *err,
                         cudaStream_t stream)
{
    if (n <= 0) return cudaSuccess;
    CUtensorMap mapY{}, mapX{};
    if (k_split % WG_KC || !make_map(&mapY, dY, n, fy, ldy, WG_KC, 64) || !make_map(&mapX, X, n, fx, ldx, WG_KC, 64))
        return cudaErrorInvalidValue;
    WgradArgs g{dW, ldc, rows, cols, n, k_split, dW2, err};
    const dim3 grid((n + k_split - 1) / k_split, dW2 ? 2 : 1);
    cudaError_t e = cudaSuccess;
    switch (fx) {
#define SPH_WGRAD_CASE(BN)                                                                                 \
    case BN: {                                                                                             \
        const int smem = WG_STAGES * (2 + (BN + 63) / 64) * WG_KC * 128 + 1024;                            \
        e = cudaFuncSetAttribute(k_wgrad<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);         \
        if (e != cudaSuccess) return e;                                                                    \
        k_wgrad<BN><<<grid, 256, smem, stream>>>(g, mapY, mapX);                                           \
        break;                                                                                             \
    }
        SPH_WGRAD_CASE(16)
        SPH_WGRAD_CASE(128)
        SPH_WGRAD_CASE(256)
#undef SPH_WGRAD_CASE
    default:
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// Launches C = A B^T, stored in Cf or (atomic) added to it, on `stream`; returns a cudaError_t.
inline cudaError_t gemm(const GemmArgs &g, cudaStream_t stream)
{
    if (g.M <= 0) return cudaSuccess;
    if (g.K % 16 != 0 || g.lda % 8 != 0 || g.ldb % 8 != 0 || g.k_split % BK != 0 || g.k_split <= 0)
        return cudaErrorInvalidValue;
    if (const LayerLaunch l = layer_for(g)) return l(g, stream);
    const dim3 grid((g.M + BM - 1) / BM, (g.K + g.k_split - 1) / g.k_split);
    const size_t smem = gemm_smem_bytes(g.N);
    CUtensorMap mapA{}, mapB{};
    if (g.K > 0 && (!make_map(&mapA, g.A, g.M, g.K, g.lda, BM) || !make_map(&mapB, g.B, g.N, g.K, g.ldb, g.N)))
        return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    switch (g.N) {
#define SPH_GEMM_CASE(BN)                                                                                  \
    case BN:                                                                                              \
        e = cudaFuncSetAttribute(k_gemm<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);    \
        if (e != cudaSuccess) return e;                                                                   \
        k_gemm<BN><<<grid, THREADS, smem, stream>>>(g, mapA, mapB);                                       \
        break;
        SPH_GEMM_CASE(16)
        SPH_GEMM_CASE(32)
        SPH_GEMM_CASE(64)
        SPH_GEMM_CASE(128)
        SPH_GEMM_CASE(256)
#undef SPH_GEMM_CASE
    default:
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace umma
