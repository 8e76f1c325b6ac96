// Optimal real-valued block scale (Appendix C of the ScaleSweep paper) and the
// FP8-quantised optimal scale, per block, on the GPU.  Analysis kernels: they
// measure how far AbsMax, 4/6 and ScaleSweep are from the best possible FP32
// block scale (the paper's Figs. 1 and 4), not part of the quantisation path.
//
// In the S-normalised domain (a_i = |fl(x_i * fl(1/S))|, weights w_i) the loss
// L(s) = sum_i w_i (a_i - s g_i(s))^2, g_i(s) = RN_E2M1(a_i / s), is piecewise
// quadratic with breakpoints b = a_i / mu_k (mu_k the 7 midpoints of the E2M1
// grid); on the segment just above a breakpoint every g_i is fixed, the segment's
// quadratic A - 2Bs + Cs^2 is minimised at s* = B/C, and its value there is
// sum_i w_i (a_i - s* g_i)^2.  For any fixed assignment that value is an upper
// bound on L(s*) (per-element rounding can only do better), and for the segment
// holding the global minimum it is the minimum itself, so the minimum over all
// segments' values is min_s L(s) -- no sorting of breakpoints is needed.  The
// assignment above breakpoint (i, k) gives element i the lower neighbour of mu_k
// and every other element the grid point nearest to a_j / b, with quotients at
// or within ~1e-6 (relative) of a midpoint sent to the lower neighbour -- the
// segment just above b also when breakpoints coincide (equal magnitudes); only
// segments narrower than ~1e-6 relative can be skipped, and their neighbours,
// which share their endpoints, are enumerated.
//
// The minimum can be attained at several scales; the smallest is reported.
// FP8-quantised optimum: the better of floor_E4M3(s*) and ceil_E4M3(s*) (ties
// to the floor), each scored with the sweep's arithmetic contract.
//
// One thread per block, in two passes over the 7n segments.  The first screens:
// the value of a segment's quadratic at its minimum is A - B^2/C (A = sum w a^2),
// so B and C alone rank it, to a few fp32 roundings of A.  The seven segments of
// one element run together, two to a packed f32x2 operation, over magnitudes and
// weights kept in shared memory (a column per thread, no bank conflicts); a
// segment that could still be the minimum is noted in a short list.  The second
// pass scores the list's remaining segments (about one per block) exactly, in
// element order and in fp32 sums of w e^2, and takes the smallest.  See screen_ok
// and screen_limit for why the first pass cannot lose the second one's answer.
// Bound by instruction issue: about 33 (MSE) or 37 (WMSE) instructions for each pair of
// elements (i, j) of a block, against about 15 times that when every segment was
// scored in full with the rounding done by selects.
#include "nvfp4_device.cuh"
#include "nvfp4_kernels.h"

namespace nvfp4 {

constexpr int kOptThreads = 128;
constexpr int kOptList = 24;          // segments noted by the screen; more: every segment is scored

__constant__ float kMid[8] = {0.25f, 0.75f, 1.25f, 1.75f, 2.5f, 3.5f, 5.0f, 5.0f};
__constant__ float kGrid[8] = {0.0f, 0.5f, 1.0f, 1.5f, 2.0f, 3.0f, 4.0f, 6.0f};

// Nearest E2M1 magnitudes of a pair of t >= 0 (ties to even), as f16x2.
__device__ __forceinline__ void rn_grid2(float tl, float th, float& gl, float& gh) {
    uint32_t h2;
    asm("{\n\t.reg .b8 q;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 q, %1, %2;\n\t"
        "cvt.rn.f16x2.e2m1x2 %0, q;\n\t}"
        : "=r"(h2) : "f"(th), "f"(tl));
    gl = f16bits_to_f32((uint16_t)(h2 & 0xFFFFu));
    gh = f16bits_to_f32((uint16_t)(h2 >> 16));
}
__device__ __forceinline__ float rn_grid(float t) {
    float g, unused;
    rn_grid2(t, 0.0f, g, unused);
    return g;
}

// A thread's block in shared memory: element j at [j * kOptThreads].
template <int OBJ>
struct Column {
    const float* a;
    const float* w;
    __device__ __forceinline__ float mag(int j) const { return a[j * kOptThreads]; }
    __device__ __forceinline__ float wt(int j) const { return OBJ ? w[j * kOptThreads] : 1.0f; }
};

// Loss of E4M3 scale code c under the sweep's contract (t = fl(y*fl(1/v)),
// q = RNE_E2M1(t), e = fl(y - q*v), fp32 accumulation in element order); the
// loss of a magnitude is that of either sign.
template <int BLOCK, int OBJ>
__device__ __noinline__ float contract_loss(Column<OBJ> col, int c) {
    const float v = f16bits_to_f32(e4m3_to_f16bits((uint32_t)c));
    const float r = __frcp_rn(v);
    float L = 0.0f;
#pragma unroll 8
    for (int i = 0; i < BLOCK; i++) {
        const float a = col.mag(i);
        const float e = __fmaf_rn(-rn_grid(__fmul_rn(a, r)), v, a);
        L = __fmaf_rn(OBJ ? __fmul_rn(col.wt(i), e) : e, e, L);
    }
    return L;
}

// ~ 1/b for b = a_i / mu_k, shrunk by 2^-20 so that quotients at (or within
// ~1e-6 of) a midpoint take the lower neighbour: the assignment just above b
// even when breakpoints coincide (equal magnitudes are common in bf16 blocks).
__device__ __forceinline__ float segment_rcp(float mid, float ra) {
    return __fmul_rn(__fmul_rn(mid, ra), 1.0f - 9.5367431640625e-07f);
}

// One segment in full: its least-squares scale and loss, and the running best.
// The optimum can be attained on several segments (e.g. one dominant element
// that can sit on 6, 4, 3, ... grid points while the rest round to 0): the
// smallest such scale is kept, within fp32 ties.
template <int BLOCK, int OBJ>
__device__ __noinline__ void score_segment(Column<OBJ> col, int i, int k, float& best, float& best_s) {
    const float ai = col.mag(i);
    if (!(ai > 0.0f)) return;
    const float r = segment_rcp(kMid[k], __frcp_rn(ai));
    float B = 0.0f, C = 0.0f;
#pragma unroll 8
    for (int j = 0; j < BLOCK; j++) {
        const float a = col.mag(j), w = col.wt(j);
        const float g = (j == i) ? kGrid[k] : rn_grid(__fmul_rn(a, r));
        B = __fmaf_rn(__fmul_rn(w, a), g, B);
        C = __fmaf_rn(__fmul_rn(w, g), g, C);
    }
    if (!(C > 0.0f)) return;
    const float s = __fdiv_rn(B, C);
    float L = 0.0f;
#pragma unroll 8
    for (int j = 0; j < BLOCK; j++) {
        const float a = col.mag(j);
        const float g = (j == i) ? kGrid[k] : rn_grid(__fmul_rn(a, r));
        const float e = __fmaf_rn(-s, g, a);
        L = __fmaf_rn(__fmul_rn(col.wt(j), e), e, L);
    }
    if (L < best * (1.0f - 1e-6f) || (L <= best * (1.0f + 1e-6f) && s < best_s)) {
        best = fminf(best, L);
        best_s = s;
    }
}

// The seven segments of element i one after the other, with the operations of
// score_segment, two segments to a packed one and four pairs to a pass: what blocks
// without a screen take for all of their elements.  One segment at a time those were
// slower than before there was a screen (512 x 8192 bf16 WMSE: one weight in ten
// negative 540 -> 674 us, all magnitudes equal 530 -> 623; so 446 and 432).
template <int BLOCK, int OBJ>
__device__ __noinline__ void score_element(Column<OBJ> col, int i, float& best, float& best_s) {
    const float ai = col.mag(i);
    if (!(ai > 0.0f)) return;
    const float ra = __frcp_rn(ai);
    u64 r2[4], B2[4], C2[4], L2[4], ns2[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        r2[q] = pack2(segment_rcp(kMid[2 * q], ra), segment_rcp(kMid[2 * q + 1], ra));
        B2[q] = C2[q] = L2[q] = 0ull;
    }
    auto grid2 = [&](int j, u64 a2, int q) -> u64 {
        float tl, th, gl, gh;
        unpack2(mul2(a2, r2[q]), tl, th);
        rn_grid2(tl, th, gl, gh);
        return j == i ? pack2(kGrid[2 * q], kGrid[2 * q + 1]) : pack2(gl, gh);
    };
#pragma unroll 4
    for (int j = 0; j < BLOCK; j++) {
        const float a = col.mag(j), w = col.wt(j);
        const float wa = OBJ ? __fmul_rn(w, a) : a;
        const u64 a2 = pack2(a, a), wa2 = pack2(wa, wa), w2 = pack2(w, w);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const u64 g2 = grid2(j, a2, q);
            B2[q] = fma2(wa2, g2, B2[q]);
            C2[q] = fma2(OBJ ? mul2(w2, g2) : g2, g2, C2[q]);
        }
    }
    float b[8], c[8], L[8];                          // [7]: no segment
#pragma unroll
    for (int q = 0; q < 4; q++) {
        unpack2(B2[q], b[2 * q], b[2 * q + 1]);
        unpack2(C2[q], c[2 * q], c[2 * q + 1]);
#pragma unroll
        for (int h = 2 * q; h < 2 * q + 2; h++) b[h] = __fdiv_rn(b[h], c[h]);        // the scale
        ns2[q] = pack2(-b[2 * q], -b[2 * q + 1]);
    }
#pragma unroll 4
    for (int j = 0; j < BLOCK; j++) {
        const float a = col.mag(j), w = col.wt(j);
        const u64 a2 = pack2(a, a), w2 = pack2(w, w);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const u64 e2 = fma2(ns2[q], grid2(j, a2, q), a2);
            L2[q] = fma2(OBJ ? mul2(w2, e2) : e2, e2, L2[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; q++) unpack2(L2[q], L[2 * q], L[2 * q + 1]);
#pragma unroll
    for (int h = 0; h < 7; h++)
        if (c[h] > 0.0f && (L[h] < best * (1.0f - 1e-6f) || (L[h] <= best * (1.0f + 1e-6f) && b[h] < best_s))) {
            best = fminf(best, L[h]);
            best_s = b[h];
        }
}

// How far the screen's A - B^2/C can lie from the scored loss, relative to A:
// B and C carry at most n + 1 roundings each and B^2/C <= A (Cauchy-Schwarz), so
// 3(n + 1) + 4 roundings of A, and the list entry drops 2^-14 of its own value
// (covered by the factor 1 + 2^-9 beside it).  n 2^-20 is over four times that.
// The scored pass compares losses within 1e-6, so anything farther than that
// from the least loss leaves no trace in its result: a better segment replaces
// it whichever comes first.
template <int BLOCK>
__device__ __forceinline__ float screen_limit(float least, float A) {
    return __fmaf_rn(A, BLOCK * 9.5367431640625e-07f, least * 1.001953125f);
}

template <int DT, int OBJ, int BLOCK>
__global__ void __launch_bounds__(kOptThreads) optimal_scale_kernel(OptParams p) {
    extern __shared__ float smem[];
    float* sa = smem + threadIdx.x;
    float* sw = sa + BLOCK * kOptThreads;
    uint32_t* list = reinterpret_cast<uint32_t*>(sa + (OBJ ? 2 : 1) * BLOCK * kOptThreads);
    const Column<OBJ> col{sa, sw};
    const float S = __ldg(p.S);
    const float E = __frcp_rn(S);
    const bool usable = (S > 0.0f) && isfinite(S) && isfinite(E);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t blk = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; blk < p.nblocks; blk += stride) {
        const int64_t row = blk / p.kb, kbi = blk - row * p.kb;
        const int64_t off = row * p.cols + kbi * BLOCK;
        const float* wp = p.w + row * p.w_row_stride + kbi * BLOCK;
        // s -> infinity: everything rounds to 0;  s -> 0+: every non-zero element saturates at 6
        float best = 0.0f, B0 = 0.0f, C0 = 0.0f;
        bool sane = true;
#pragma unroll 16
        for (int i = 0; i < BLOCK; i++) {
            const float xv = DT == 0 ? __uint_as_float((uint32_t)(static_cast<const uint16_t*>(p.x)[off + i]) << 16)
                                     : static_cast<const float*>(p.x)[off + i];
            const float a = fabsf(usable ? __fmul_rn(xv, E) : 0.0f);
            const float w = OBJ ? __ldg(wp + i) : 1.0f;
            sa[i * kOptThreads] = a;
            if (OBJ) sw[i * kOptThreads] = w;
            const float wa = __fmul_rn(w, a), g = a > 0.0f ? 6.0f : 0.0f;
            best = __fmaf_rn(wa, a, best);
            B0 = __fmaf_rn(wa, g, B0);
            C0 = __fmaf_rn(__fmul_rn(w, g), g, C0);
            sane = sane && (a == 0.0f || a > 1e-15f) && (!OBJ || w == 0.0f || (w > 1e-18f && w < 1e30f));
        }
        const float A = best;
        float best_s = 0.0f;
        if (C0 > 0.0f) {
            const float s = __fdiv_rn(B0, C0);
            float L = 0.0f;
#pragma unroll 16
            for (int i = 0; i < BLOCK; i++) {
                const float a = col.mag(i);
                const float e = __fmaf_rn(-s, a > 0.0f ? 6.0f : 0.0f, a);
                L = __fmaf_rn(__fmul_rn(col.wt(i), e), e, L);
            }
            if (L < best) {
                best = L;
                best_s = s;
            }
        }
        // The screen's bound holds for non-negative weights and sums far from
        // overflow and underflow; other blocks (NaN and inf among them) are scored in full.
        const bool screen_ok = sane && A > 1e-25f && A < 1e30f;
        int noted = 0;
        float least = best;
        if (screen_ok) {
            for (int i = 0; i < BLOCK; i++) {
                const float ai = col.mag(i);
                const float ra = ai > 0.0f ? __frcp_rn(ai) : 0.0f;      // zero: every code is 0, C = 0, not noted
                u64 r2[4], B2[4], C2[4];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    r2[q] = pack2(segment_rcp(kMid[2 * q], ra), segment_rcp(kMid[2 * q + 1], ra));
                    B2[q] = C2[q] = 0ull;
                }
#pragma unroll 4
                for (int j = 0; j < BLOCK; j++) {
                    const float a = col.mag(j), w = col.wt(j);
                    const u64 a2 = pack2(a, a);
                    const float wa = OBJ ? __fmul_rn(w, a) : a;
                    const u64 wa2 = pack2(wa, wa), w2 = pack2(w, w);
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        float tl, th, gl, gh;
                        unpack2(mul2(a2, r2[q]), tl, th);
                        rn_grid2(tl, th, gl, gh);
                        const u64 g2 = pack2(gl, gh);
                        B2[q] = fma2(wa2, g2, B2[q]);
                        C2[q] = fma2(OBJ ? mul2(w2, g2) : g2, g2, C2[q]);
                    }
                }
#pragma unroll
                for (int k = 0; k < 7; k++) {
                    float b0, b1, c0, c1;
                    unpack2(B2[k >> 1], b0, b1);
                    unpack2(C2[k >> 1], c0, c1);
                    const float B = (k & 1) ? b1 : b0, C = (k & 1) ? c1 : c0;
                    const float est = fmaxf(__fmaf_rn(-B, __fdividef(B, C), A), 0.0f);   // NaN for C = 0: 0 by fmaxf
                    if (C > 0.0f && est <= screen_limit<BLOCK>(least, A)) {
                        if (noted < kOptList)
                            list[noted * kOptThreads] = (__float_as_uint(est) & ~511u) | (uint32_t)(i * 7 + k);
                        noted++;
                        least = fminf(least, est);
                    }
                }
            }
        }
        if (!screen_ok || noted > kOptList) {
            for (int i = 0; i < BLOCK; i++) score_element<BLOCK, OBJ>(col, i, best, best_s);
        } else {
            const float limit = screen_limit<BLOCK>(least, A);
            for (int n = 0; n < noted; n++) {
                const uint32_t e = list[n * kOptThreads];
                if (__uint_as_float(e & ~511u) > limit) continue;
                const int id = (int)(e & 511u);
                score_segment<BLOCK, OBJ>(col, id / 7, id % 7, best, best_s);
            }
        }
        p.s_opt[blk] = best_s;
        p.loss_opt[blk] = best;
        if (p.fp8_code) {
            int code = 0;
            float Lf = best;
            if (best_s > 0.0f) {
                int fl = e4m3_floor_code(best_s);
                if (fl < 1) fl = 1;
                int ce = fl;
                const float vfl = f16bits_to_f32(e4m3_to_f16bits((uint32_t)fl));
                if (vfl < best_s && fl < 126) ce = fl + 1;
                const float Lfl = contract_loss<BLOCK, OBJ>(col, fl);
                const float Lce = ce == fl ? Lfl : contract_loss<BLOCK, OBJ>(col, ce);
                code = (Lce < Lfl) ? ce : fl;
                Lf = (Lce < Lfl) ? Lce : Lfl;
            }
            p.fp8_code[blk] = (uint8_t)code;
            if (p.loss_fp8) p.loss_fp8[blk] = Lf;
        }
    }
}

template <int DT, int OBJ, int BLOCK>
static cudaError_t opt_launch(const OptParams& p, int sms, cudaStream_t s) {
    constexpr int smem = ((OBJ ? 2 : 1) * BLOCK + kOptList) * kOptThreads * (int)sizeof(float);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(optimal_scale_kernel<DT, OBJ, BLOCK>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    int64_t grid = (p.nblocks + kOptThreads - 1) / kOptThreads;
    if (grid > (int64_t)sms * 64) grid = (int64_t)sms * 64;
    optimal_scale_kernel<DT, OBJ, BLOCK><<<(int)grid, kOptThreads, smem, s>>>(p);
    return cudaGetLastError();
}

template <int DT, int OBJ>
static cudaError_t opt_block(const OptParams& p, int block, int sms, cudaStream_t s) {
    switch (block) {
        case 16: return opt_launch<DT, OBJ, 16>(p, sms, s);
        case 32: return opt_launch<DT, OBJ, 32>(p, sms, s);
        default: return opt_launch<DT, OBJ, 64>(p, sms, s);
    }
}

cudaError_t launch_optimal_scale(const OptParams& p, int dtype, int obj, int block, int sms, cudaStream_t s) {
    if (p.nblocks <= 0) return cudaSuccess;
    if (dtype == 0) return obj ? opt_block<0, 1>(p, block, sms, s) : opt_block<0, 0>(p, block, sms, s);
    return obj ? opt_block<1, 1>(p, block, sms, s) : opt_block<1, 0>(p, block, sms, s);
}

}  // namespace nvfp4
