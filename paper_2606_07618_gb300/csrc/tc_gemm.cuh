// fp32 GEMM on the 5th-generation tensor cores (tcgen05) for the LDLQ error
// feedback and its factorization (Appendix A.2, GPTQ paragraph): C[M, N] += alpha *
// A[M, K] B[N, K]^T with fp32 accumulation, three TF32 products per term
// ("3xTF32"):
//
//   a ~ a_hi + a_lo, both TF32 values (split_tf32), a*b ~ a_hi*b_hi + a_hi*b_lo +
//   a_lo*b_hi, dropping a_lo*b_lo (~2^-22 relative): products to ~2^-21 relative,
//   against 2^-24 for one fp32 FMA.
//
// The sums decide the error, not the products: each MMA adds its 8-term sum to an
// accumulator without rounding to nearest, and that error follows the accumulator's
// size.  So the two small products go to an accumulator of their own, K goes in two parts
// with a pair of accumulators each, and the epilogue adds them in fp32 (both kernels the
// same).  LDLQ's targets against 64 bits, over 24 shapes of 535 to 3820 rows and 256 to
// 3760 columns: 0.28 to 0.36 of the error with all products in one accumulator, 0.47 to
// 0.87 of that of FP32 multiply-adds (one part: up to 1.09).  The factor's D at n = 4096:
// 1.5e-5 in one accumulator, 3.5e-6.  Time, with one accumulator and now: weights of 4096
// x 4096 0.924 / 0.964 ms, 14336 x 4096 2.66 / 2.75, 4096 x 14336 6.45 / 6.75; factors of
// n = 4096 1.591 / 1.603 ms, n = 14336 20.7 / 20.7.
//
// The operands arrive already split, K-major (K contiguous): the kernels that
// produce them (the panel walk, the panel solve, a transpose of U) write the hi and lo
// arrays, a few words per element once, so the GEMM's main loop is TMA and MMA only.
// (Splitting and transposing raw operands inside the GEMM, by all of its warps
// between two barriers per stage, took 2.7k cycles per stage of K = 32; the MMAs
// take 0.9k and shared memory 1.25k: 64 KB landing, 96 KB read.)
//
// One CTA of 256 threads computes a 128 x 128 tile of C:
//   * one thread loads operand stages of K = 32 fp32 (128 bytes, one swizzle row)
//     by TMA (cp.async.bulk.tensor) into a three-stage ring of 128-byte-swizzled
//     shared memory: A hi, A lo, B hi, B lo, 64 KB per stage;
//   * one thread issues 4 k-steps x 3 tcgen05.mma.kind::tf32 (M = 128, N = 128,
//     K = 8) per stage into 128-column fp32 accumulators in tensor memory, and
//     tcgen05.commit frees the stage's slot;
//   * the C tile arrives by TMA in the first slot that no stage needs any more; the
//     epilogue reads the accumulators with tcgen05.ld (warps w and w + 4 read TMEM
//     lanes 32(w%4).. = rows, 64 columns each), forms C = fma(alpha, acc, C) in
//     shared memory and TMA stores the tile.
//
// Updates of several tiles per SM take gemm_strip_kernel: up to four tiles to a CTA,
// loads, MMAs and epilogue in warps of their own.
//
// Every mbarrier wait is bounded by the global timer (1 s).  On a timeout the
// CTA sets bit 4 (16) of the status word, stops issuing, waits (bounded again)
// for the copies and MMAs it has in flight, frees its tensor memory and
// returns without writing (the rest of) C.
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "nvfp4_device.cuh"

namespace nvfp4 {
namespace tc {

constexpr int kTileM = 128;
constexpr int kTileN = 128;
constexpr int kStageK = 32;                               // fp32 per swizzle row (128 bytes)
constexpr int kEpiThreads = 256;                          // warps w, w + 4 read TMEM lanes 32(w % 4)..
constexpr int kThreads = 256;
constexpr int kStripThreads = kEpiThreads + 64;           // a warp for the loads and one for the MMAs
constexpr int kOpBytes = kTileM * kStageK * 4;            // one operand tile: 16 KB
constexpr int kStages = 3;
constexpr int kStageBytes = 4 * kOpBytes;                 // A hi, A lo, B hi, B lo
constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 128;   // + alignment, barriers
constexpr int kStripSmem = kSmemBytes + 2 * kOpBytes;     // + boxes of C
constexpr int kPairCols = 2 * kTileN;                     // fp32 accumulators: the large products, the small ones
constexpr int kTmemCols = 2 * kPairCols;                  // a pair for each part of K
// Stages of the first part of K: all but a quarter, or all of a short K.  Even parts are
// a fifth more exact, but the strips' second pair then waits for the epilogue (4096 x
// 14336 6.91 ms, 6.75 so, 6.50 with one part; 7 of 8 stages 6.71).
__host__ __device__ constexpr int first_stages(int nst) { return nst >= 4 ? nst - nst / 4 : nst; }
constexpr unsigned long long kWaitNs = 1000000000ull;
constexpr int kStatusTimeout = 16;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ---- mbarriers
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Wait for the phase with the given parity to complete; false after ~1 s.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = now_ns();
    while (!mbar_try_wait(bar, parity))
        if (now_ns() - t0 > kWaitNs) return false;
    return true;
}

// ---- TMA: a 2-D box of the tensor map into shared memory, completion on bar
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int c0, int c1, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(src)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// The committed stores have read shared memory / have completed.
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// ---- tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t holder, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Generic-proxy writes to shared memory become visible to the async proxy
// (the tensor core reading its operands).
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}
// 16 consecutive fp32 accumulator columns of this thread's TMEM lane; the values are
// there after tmem_wait_ld, which names them so that no use moves above it.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
          "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld(float (&a)[16], float (&b)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]), "+f"(a[6]), "+f"(a[7]),
                   "+f"(a[8]), "+f"(a[9]), "+f"(a[10]), "+f"(a[11]), "+f"(a[12]), "+f"(a[13]), "+f"(a[14]), "+f"(a[15])
                 :: "memory");
    asm volatile("" : "+f"(b[0]), "+f"(b[1]), "+f"(b[2]), "+f"(b[3]), "+f"(b[4]), "+f"(b[5]), "+f"(b[6]), "+f"(b[7]),
                      "+f"(b[8]), "+f"(b[9]), "+f"(b[10]), "+f"(b[11]), "+f"(b[12]), "+f"(b[13]), "+f"(b[14]), "+f"(b[15]));
}
// The two accumulators at taddr and taddr + gap, added.
__device__ __forceinline__ void tmem_sum16(uint32_t taddr, uint32_t gap, float (&v)[16]) {
    float l[16];
    tmem_ld16(taddr, v);
    tmem_ld16(taddr + gap, l);
    tmem_wait_ld(v, l);
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __fadd_rn(v[i], l[i]);
}

// Shared-memory matrix descriptor of a K-major 128-byte-swizzled operand tile:
// start address >> 4 (bits 0-13), leading-dimension byte offset >> 4 (16-29),
// stride-dimension byte offset >> 4 (32-45), descriptor version 1 (46-47),
// base offset 0 (tiles are 1024-byte aligned), swizzle mode 2 = 128 bytes
// (61-63).  Rows of 128 bytes, SBO = 1024 between 8-row groups.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor of tcgen05.mma.kind::tf32 with both operands
// K-major: D fp32 (bits 4-5 = 1), A and B TF32 (bits 7-9, 10-12 = 2), N >> 3
// (bits 17-22), M >> 4 (bits 24-28).
__host__ __device__ constexpr uint32_t idesc_tf32() {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(kTileN >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
}

}  // namespace tc
}  // namespace nvfp4

namespace nvfp4 {
namespace tc {

// x ~ hi + lo, both TF32 values: hi is x with its low 13 mantissa bits cleared, lo the
// rest rounded to nearest (half of the last place away from zero).  Left to the MMA,
// which drops the bits past its eleven, lo would be too small by 2^-23 of x on average.
__device__ __forceinline__ void split_tf32(float x, float& hi, float& lo) {
    hi = __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
    lo = __uint_as_float((__float_as_uint(__fsub_rn(x, hi)) + 0x1000u) & 0xFFFFE000u);
}
__device__ __forceinline__ void split4(const float4& x, float4& h, float4& l) {
    split_tf32(x.x, h.x, l.x);
    split_tf32(x.y, h.y, l.y);
    split_tf32(x.z, h.z, l.z);
    split_tf32(x.w, h.w, l.w);
}

// C[M, N] (row-major, ldc) += alpha * (Ah + Al)[M, K] (Bh + Bl)[N, K]^T.  The operand
// maps have a box of 32 fp32 along K (128 bytes, 128-byte swizzle) by 128 rows; what
// lies outside a matrix reads as zero.  LOWER skips tiles entirely above the diagonal.
//
// Thread 0 loads stage s into slot s % 3 once the MMAs of stage s - 3 have read it;
// thread 32 issues the MMAs of s once it has landed.
template <bool LOWER>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl,
                const __grid_constant__ CUtensorMap tmC, int K, float alpha, int* status, int starve) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_abort, s_issued;
    __shared__ uint32_t s_tmem;
    const int m0 = (int)blockIdx.y * kTileM, n0 = (int)blockIdx.x * kTileN;
    grid_launch_dependents();                                    // a dependent launch waits for this grid's end
    if (LOWER && n0 > m0 + kTileM - 1) return;
    const int nst = (K + kStageK - 1) / kStageK;
    const int first = first_stages(nst);
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + kStages * kStageBytes);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kStages);
    const uint32_t cbar = smem_u32(bars + 2 * kStages), dbar = smem_u32(bars + 2 * kStages + 1);

    if (warp == 0) tmem_alloc(smem_u32(&s_tmem), kTmemCols);
    if (tid == 0) {
        for (int b = 0; b < kStages; b++) {
            mbar_init(full0 + 8 * b, 1 + starve);
            mbar_init(empty0 + 8 * b, 1);
        }
        mbar_init(cbar, 1);
        mbar_init(dbar, 1);
        s_abort = 0;
        s_issued = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    uint8_t* cbase = base + (nst % kStages) * kStageBytes;       // the C tile's slot: that of stage nst - 3

    if (tid == 0) {
        bool ok = true;
        int s = 0;
        for (; s < nst; s++) {
            const int r = s % kStages;
            if (s >= kStages && !mbar_wait(empty0 + 8 * r, (s / kStages - 1) & 1)) {
                ok = false;
                break;
            }
            const uint32_t bar = full0 + 8 * r, st = smem_u32(base + r * kStageBytes);
            mbar_expect_tx(bar, kStageBytes);
            tma_load_2d(st, &tmAh, s * kStageK, m0, bar);
            tma_load_2d(st + kOpBytes, &tmAl, s * kStageK, m0, bar);
            tma_load_2d(st + 2 * kOpBytes, &tmBh, s * kStageK, n0, bar);
            tma_load_2d(st + 3 * kOpBytes, &tmBl, s * kStageK, n0, bar);
        }
        if (ok && nst >= kStages && !mbar_wait(empty0 + 8 * (nst % kStages), (nst / kStages - 1) & 1)) ok = false;
        if (ok) {
            mbar_expect_tx(cbar, kTileM * kTileN * 4);
#pragma unroll
            for (int j = 0; j < kTileN / 32; j++)
                tma_load_2d(smem_u32(cbase + j * kOpBytes), &tmC, n0 + 32 * j, m0, cbar);
        }
        s_issued = s + (ok ? 1000 : 0);
        if (!ok) atomicOr(&s_abort, 1);
    } else if (tid == 32) {
        constexpr uint32_t idesc = idesc_tf32();
        bool ok = true;
        for (int s = 0; s < nst; s++) {
            const int r = s % kStages;
            if (!mbar_wait(full0 + 8 * r, (s / kStages) & 1)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t st = smem_u32(base + r * kStageBytes);
            const uint32_t acc = tmem + (s < first ? 0 : kPairCols);
            const int i = s < first ? s : s - first;             // the stage within its part
#pragma unroll
            for (int kk = 0; kk < kStageK / 8; kk++) {           // the k-step's 32 bytes of each 128-byte row
                const uint64_t ahi = smem_desc(st + kk * 32, 16, 1024);
                const uint64_t alo = smem_desc(st + kOpBytes + kk * 32, 16, 1024);
                const uint64_t bhi = smem_desc(st + 2 * kOpBytes + kk * 32, 16, 1024);
                const uint64_t blo = smem_desc(st + 3 * kOpBytes + kk * 32, 16, 1024);
                mma_tf32(acc, ahi, bhi, idesc, i | kk);
                mma_tf32(acc + kTileN, ahi, blo, idesc, i | kk);
                mma_tf32(acc + kTileN, alo, bhi, idesc, 1);
            }
            mma_commit(empty0 + 8 * r);
        }
        mma_commit(dbar);                                        // after every MMA issued, also on a timeout
        if (!ok) atomicOr(&s_abort, 1);
    }
    __syncthreads();
    const bool c_loaded = s_issued >= 1000;
    if (!mbar_wait(dbar, 0)) atomicOr(&s_abort, 1);              // the MMAs have written the accumulator
    if (c_loaded && !mbar_wait(cbar, 0)) atomicOr(&s_abort, 1);
    if (s_abort && tid == 0)                                     // copies still in flight: bounded wait
        for (int s = 0; s < s_issued % 1000; s++)
            if (s + kStages >= s_issued % 1000) (void)mbar_wait(full0 + 8 * (s % kStages), (s / kStages) & 1);
    tc_fence_after();
    __syncthreads();
    if (!s_abort) {
        // C += alpha * acc in shared memory (thread = row; the box rows are
        // 128-byte swizzled, so the eight lanes of a quarter warp touch eight
        // distinct 16-byte chunks), then TMA stores the tile (out-of-range
        // rows and columns are not written)
        const int q = warp & 3, r = 32 * q + lane;               // TMEM lane quarter q = rows 32q..32q+31
#pragma unroll 1
        for (int j = 2 * (warp >> 2); j < 2 * (warp >> 2) + 2; j++) {   // warps 0-3: boxes 0-1, 4-7: 2-3
            float v[32];
            const uint32_t at = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(32 * j);
#pragma unroll
            for (int e = 0; e < 32; e += 16) {
                float a[16];
                tmem_sum16(at + e, kTileN, a);                   // .sync.aligned
                if (nst > first) {
                    float b[16];
                    tmem_sum16(at + kPairCols + e, kTileN, b);
#pragma unroll
                    for (int i = 0; i < 16; i++) a[i] = __fadd_rn(a[i], b[i]);
                }
#pragma unroll
                for (int i = 0; i < 16; i++) v[e + i] = a[i];
            }
            uint8_t* box = cbase + j * kOpBytes + r * 128;
#pragma unroll
            for (int g = 0; g < 8; g++) {
                float4* c = reinterpret_cast<float4*>(box + (((g ^ r) & 7) << 4));
                float4 o = *c;
                o.x = __fmaf_rn(alpha, v[4 * g], o.x);
                o.y = __fmaf_rn(alpha, v[4 * g + 1], o.y);
                o.z = __fmaf_rn(alpha, v[4 * g + 2], o.z);
                o.w = __fmaf_rn(alpha, v[4 * g + 3], o.w);
                *c = o;
            }
        }
        fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
#pragma unroll
            for (int j = 0; j < kTileN / 32; j++)
                tma_store_2d(&tmC, n0 + 32 * j, m0, smem_u32(cbase + j * kOpBytes));
            tma_store_commit();
            tma_store_wait();
        }
    } else if (tid == 0 && status) {
        atomicOr(status, kStatusTimeout);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

// The warps that add accumulators to C.
__device__ __forceinline__ void epi_barrier() {
    __syncwarp();
    asm volatile("barrier.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
}

// The same with a CTA for up to `tiles` tiles of C side by side, for updates of several
// tiles per SM: loads, MMAs and the update of C run beside each other.  Stages run on through them: warp
// 8's first thread loads stage s into slot s % 3 once the MMAs of stage s - 3 have
// read it, warp 9's issues the MMAs of s once it has landed, alternating between two
// pairs of accumulators, one for each part of K; the other eight warps take the first
// part into registers beside the second one's MMAs and add both to C, 32 columns
// at a time through two boxes that thread 0 loads and stores, beside the next tile's
// MMAs.
template <bool LOWER>
__global__ void __launch_bounds__(kStripThreads, 1)
    gemm_strip_kernel(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl,
                const __grid_constant__ CUtensorMap tmC, int N, int K, int tiles, float alpha, int* status, int starve) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_abort, s_lost;                              // a wait ran out: of the other two warps, of these eight
    __shared__ uint32_t s_tmem;
    const int m0 = (int)blockIdx.y * kTileM, nb = (int)blockIdx.x * tiles * kTileN;
    grid_launch_dependents();                                    // a dependent launch waits for this grid's end
    if (LOWER && nb > m0 + kTileM - 1) return;
    const int last = LOWER ? min(N - 1, m0 + kTileM - 1) : N - 1;                // last column of this CTA's rows
    const int nt = min(tiles, (last - nb) / kTileN + 1);
    const int nst = (K + kStageK - 1) / kStageK;
    const int first = first_stages(nst), parts = first < nst ? 2 : 1;
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* cbox = base + kStages * kStageBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(cbox + 2 * kOpBytes);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kStages, cfull0 = empty0 + 8 * kStages;
    const uint32_t accf0 = cfull0 + 16, acce0 = accf0 + 16, dbar = acce0 + 16;

    if (warp == 0) tmem_alloc(smem_u32(&s_tmem), kTmemCols);
    if (tid == 0) {
        for (int b = 0; b < kStages; b++) {
            mbar_init(full0 + 8 * b, 1 + starve);
            mbar_init(empty0 + 8 * b, 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(cfull0 + 8 * b, 1);
            mbar_init(accf0 + 8 * b, 1);
            mbar_init(acce0 + 8 * b, kEpiThreads / 32);
        }
        mbar_init(dbar, 1);
        s_abort = s_lost = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (tid == kEpiThreads) {
        int s = 0;
        for (; s < nt * nst; s++) {
            const int r = s % kStages;
            if (s >= kStages && !mbar_wait(empty0 + 8 * r, (s / kStages - 1) & 1)) {
                atomicOr(&s_abort, 1);
                break;
            }
            const uint32_t bar = full0 + 8 * r, st = smem_u32(base + r * kStageBytes);
            const int k = s % nst * kStageK, n0 = nb + s / nst * kTileN;
            mbar_expect_tx(bar, kStageBytes);
            tma_load_2d(st, &tmAh, k, m0, bar);
            tma_load_2d(st + kOpBytes, &tmAl, k, m0, bar);
            tma_load_2d(st + 2 * kOpBytes, &tmBh, k, n0, bar);
            tma_load_2d(st + 3 * kOpBytes, &tmBl, k, n0, bar);
        }
        for (int i = s < kStages ? 0 : s - kStages; i < s; i++)  // none in flight at the end (bounded)
            if (!mbar_wait(full0 + 8 * (i % kStages), (i / kStages) & 1)) atomicOr(&s_abort, 1);
    } else if (tid == kEpiThreads + 32) {
        constexpr uint32_t idesc = idesc_tf32();
        bool ok = true;
        for (int u = 0; ok && u < nt * parts; u++) {
            const int t = u / parts, from = u % parts ? first : 0, to = u % parts ? nst : first;
            const uint32_t acc = tmem + (uint32_t)((u & 1) * kPairCols);
            if (u >= 2 && !mbar_wait(acce0 + 8 * (u & 1), (u / 2 - 1) & 1)) ok = false;
            tc_fence_after();
            for (int i = from; ok && i < to; i++) {
                const int s = t * nst + i, r = s % kStages;
                if (!mbar_wait(full0 + 8 * r, (s / kStages) & 1)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t st = smem_u32(base + r * kStageBytes);
#pragma unroll
                for (int kk = 0; kk < kStageK / 8; kk++) {       // the k-step's 32 bytes of each 128-byte row
                    const uint64_t ahi = smem_desc(st + kk * 32, 16, 1024);
                    const uint64_t alo = smem_desc(st + kOpBytes + kk * 32, 16, 1024);
                    const uint64_t bhi = smem_desc(st + 2 * kOpBytes + kk * 32, 16, 1024);
                    const uint64_t blo = smem_desc(st + 3 * kOpBytes + kk * 32, 16, 1024);
                    mma_tf32(acc, ahi, bhi, idesc, (i - from) | kk);
                    mma_tf32(acc + kTileN, ahi, blo, idesc, (i - from) | kk);
                    mma_tf32(acc + kTileN, alo, bhi, idesc, 1);
                }
                mma_commit(empty0 + 8 * r);
            }
            if (ok) mma_commit(accf0 + 8 * (u & 1));
        }
        mma_commit(dbar);                                        // after every MMA issued, also on a timeout
        if (!ok) atomicOr(&s_abort, 1);
        if (!mbar_wait(dbar, 0)) atomicOr(&s_abort, 1);
    } else if (tid < kEpiThreads) {
        // C += alpha * acc in shared memory (thread = row and half of the box's columns;
        // the box rows are 128-byte swizzled, so the eight lanes of a quarter warp touch
        // eight distinct 16-byte chunks), then TMA stores the box (out-of-range rows and
        // columns are not written)
        const int q = warp & 3, h = warp >> 2, r = 32 * q + lane;    // TMEM lane quarter q = rows 32q..32q+31
        constexpr int kBoxes = kTileN / 32;
        auto load_c = [&](int c) {
            mbar_expect_tx(cfull0 + 8 * (c & 1), kOpBytes);
            tma_load_2d(smem_u32(cbox + (c & 1) * kOpBytes), &tmC, nb + 32 * c, m0, cfull0 + 8 * (c & 1));
        };
        int issued = 0;                                          // thread 0: boxes loaded
        if (tid == 0)
            for (; issued < 2; issued++) load_c(issued);
        // the pair of accumulators of one part, columns 32 j + 16 h .., added
        auto pair_sum = [&](int u, int j, float (&v)[16]) {
            tmem_sum16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)((u & 1) * kPairCols + 32 * j + 16 * h), kTileN, v);
        };
        auto pair_read = [&](int u) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce0 + 8 * (u & 1));
        };
        int c = 0;
        bool lost = false;
        for (int t = 0; !lost && t < nt; t++) {
            const int ul = t * parts + parts - 1;                // the tile's last part
            bool ok = true;
            float v[kBoxes][16];
            if (parts == 2) {                                    // the first one, beside the second one's MMAs
                ok = mbar_wait(accf0 + 8 * ((ul - 1) & 1), ((ul - 1) >> 1) & 1);
                tc_fence_after();
                __syncwarp();
#pragma unroll
                for (int j = 0; j < kBoxes; j++) pair_sum(ul - 1, j, v[j]);
                pair_read(ul - 1);
            }
            ok = ok && mbar_wait(accf0 + 8 * (ul & 1), (ul >> 1) & 1);
#pragma unroll
            for (int j = 0; j < kBoxes; j++) {
                ok = ok && mbar_wait(cfull0 + 8 * (c & 1), (c >> 1) & 1);
                if (!ok) atomicOr(&s_lost, 1);
                epi_barrier();                                   // one decision for all eight warps: s_lost is
                if (*reinterpret_cast<volatile int*>(&s_lost)) {     // written before this barrier, read before the next
                    lost = true;
                    break;
                }
                tc_fence_after();
                __syncwarp();
                float w[16];
                pair_sum(ul, j, w);
                if (parts == 2)
#pragma unroll
                    for (int i = 0; i < 16; i++) w[i] = __fadd_rn(v[j][i], w[i]);
                uint8_t* box = cbox + (c & 1) * kOpBytes + r * 128;
#pragma unroll
                for (int g = 0; g < 4; g++) {
                    float4* o4 = reinterpret_cast<float4*>(box + (((4 * h + g) ^ r) & 7) * 16);
                    float4 o = *o4;
                    o.x = __fmaf_rn(alpha, w[4 * g], o.x);
                    o.y = __fmaf_rn(alpha, w[4 * g + 1], o.y);
                    o.z = __fmaf_rn(alpha, w[4 * g + 2], o.z);
                    o.w = __fmaf_rn(alpha, w[4 * g + 3], o.w);
                    *o4 = o;
                }
                if (j == kBoxes - 1) pair_read(ul);
                fence_proxy_async();
                epi_barrier();
                if (tid == 0) {
                    tma_store_2d(&tmC, nb + 32 * c, m0, smem_u32(cbox + (c & 1) * kOpBytes));
                    tma_store_commit();
                    if (issued < nt * kBoxes) {
                        tma_store_wait_read();
                        load_c(issued++);
                    }
                }
                c++;
            }
        }
        if (tid == 0) {
            for (; c < issued; c++) (void)mbar_wait(cfull0 + 8 * (c & 1), (c >> 1) & 1);   // after a timeout: bounded
            tma_store_wait();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && (s_abort | s_lost) && status) atomicOr(status, kStatusTimeout);
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

}  // namespace tc
}  // namespace nvfp4

#include <atomic>

namespace nvfp4 {
namespace tc {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime
// (no link against libcuda); nullptr if the driver does not provide it.
inline EncodeTiledFn encode_fn() {
    static std::atomic<void*> fn{nullptr};
    static std::atomic<int> looked{0};
    if (!looked.load(std::memory_order_acquire)) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        fn.store(p, std::memory_order_release);
        looked.store(1, std::memory_order_release);
    }
    return reinterpret_cast<EncodeTiledFn>(fn.load(std::memory_order_acquire));
}

// A row-major fp32 matrix of `outer` rows of `inner` elements (row stride ld
// elements) as a TMA tensor map with a box of 32 x box_outer and 128-byte
// swizzle; out-of-range elements of a box read as zero.
inline bool make_map(CUtensorMap* m, const float* ptr, int64_t inner, int64_t outer, int64_t ld, uint32_t box_outer) {
    const EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
    const cuuint32_t box[2] = {32, box_outer};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A split operand: hi and lo, both [rows][K] with row stride ld.
struct Split {
    const float *hi, *lo;
    int64_t ld;
};

// C[M, N] += alpha * A B^T on the tensor cores (3xTF32), A [M, K] and B [N, K] split.
// starve: 1 makes the wait for the operands run out (self-test).  Returns
// cudaErrorNotSupported (nothing launched) where a base or row stride is not
// 16-byte aligned, a size is beyond the tensor maps' limits, or the driver has none.
template <bool LOWER>
cudaError_t launch_gemm(float* C, int64_t ldc, const Split& A, const Split& B, int64_t M, int64_t N, int K, float alpha,
                        int* status, int starve, int sms, cudaStream_t s) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    auto al = [](const void* p, int64_t ld) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && ld % 4 == 0 && ld < (1ll << 35); };
    if (!al(A.hi, A.ld) || !al(A.lo, A.ld) || !al(B.hi, B.ld) || !al(B.lo, B.ld) || !al(C, ldc) || M >= (1ll << 30) ||
        N >= (1ll << 30) || encode_fn() == nullptr)
        return cudaErrorNotSupported;
    CUtensorMap mah, mal, mbh, mbl, mc;
    if (!make_map(&mah, A.hi, K, M, A.ld, kTileM) || !make_map(&mal, A.lo, K, M, A.ld, kTileM) ||
        !make_map(&mbh, B.hi, K, N, B.ld, kTileN) || !make_map(&mbl, B.lo, K, N, B.ld, kTileN) ||
        !make_map(&mc, C, N, M, ldc, kTileM))
        return cudaErrorNotSupported;
    static std::atomic<bool> attr_set[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute(gemm_kernel<LOWER>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(gemm_strip_kernel<LOWER>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStripSmem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_release);
    }
    const int64_t tm = (M + kTileM - 1) / kTileM, tn = (N + kTileN - 1) / kTileN;
    // Tiles per SM.  One tile to a CTA spends almost half its time filling the ring and
    // adding to C (9 us at K = 256, 5 of them loads and MMAs); two or four overlap that,
    // but leave the SMs less evenly filled and later for a waiting walk or factor.
    // Passes with one / from 2 / from 3 / from 4 tiles per SM on: 4096 x 4096 966 / 954 /
    // 949 / 953 us, 14336 x 4096 2.92 / 2.72 / 2.72 / 2.72 ms, 4096 x 14336 7.54 / 6.68 /
    // 6.68 / 6.68; the factor at n = 4096 1.607 / 1.628 / 1.605 / 1.606 and n = 14336 22.3 /
    // 20.8 / 20.8 / 20.8.  Four tiles from 4 per SM on: 4096 x 4096 966; never: 4096 x 14336 7.01.
    const int64_t waves = (LOWER ? tm * tn / 2 : tm * tn) / sms;
    if (waves < 3) {
        gemm_kernel<LOWER><<<dim3((unsigned)tn, (unsigned)tm), kThreads, kSmemBytes, s>>>(mah, mal, mbh, mbl, mc, K, alpha,
                                                                                          status, starve);
    } else {
        const int tiles = waves < 8 ? 2 : 4;
        gemm_strip_kernel<LOWER><<<dim3((unsigned)((tn + tiles - 1) / tiles), (unsigned)tm), kStripThreads, kStripSmem, s>>>(
            mah, mal, mbh, mbl, mc, (int)N, K, tiles, alpha, status, starve);
    }
    return cudaGetLastError();
}

}  // namespace tc
}  // namespace nvfp4
