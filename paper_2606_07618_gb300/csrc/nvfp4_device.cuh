// Device helpers for the NVFP4 ScaleSweep kernels (sm_103a).
//
// Number formats (Sec. 3.2, Appendix A of the ScaleSweep paper): FP4 E2M1
// elements {0, 0.5, 1, 1.5, 2, 3, 4, 6} with a sign bit, FP8 E4M3 block scales
// (bias 7, codes 1..126 positive finite, 0x7F NaN), FP32 global scale.
// Rounding is done by the native converts, which round to nearest-even and
// saturate: cvt.rn.satfinite.e2m1x2.f32 (element codes) and
// cvt.rn.satfinite.e4m3x2.f32 (AbsMax scale).  Every float op whose rounding the
// arithmetic contract fixes is written with an explicit _rn intrinsic or PTX
// instruction so that nvcc cannot contract it into an FMA.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace nvfp4 {

typedef unsigned long long u64;

__device__ __forceinline__ u64 pack2(float lo, float hi) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(u64 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Eight fp32 (four packed pairs) -> a word of eight E2M1 codes, the first in the
// lowest nibble: the converts' bytes are assembled by the conversions themselves.
__device__ __forceinline__ uint32_t e2m1x8(u64 t0, u64 t1, u64 t2, u64 t3) {
    uint32_t r;
    asm("{\n\t.reg .b8 a, b, c, d;\n\t.reg .b32 l0, h0, l1, h1, l2, h2, l3, h3;\n\t"
        "mov.b64 {l0, h0}, %1;\n\tmov.b64 {l1, h1}, %2;\n\tmov.b64 {l2, h2}, %3;\n\tmov.b64 {l3, h3}, %4;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 a, h0, l0;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b, h1, l1;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 c, h2, l2;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 d, h3, l3;\n\t"
        "mov.b32 %0, {a, b, c, d};\n\t}"
        : "=r"(r) : "l"(t0), "l"(t1), "l"(t2), "l"(t3));
    return r;
}

// One candidate step on an element pair: from t = fl(y*r), q = RNE_E2M1(t),
// e = fl(y - q*v) computed as fma(q, -v, y) with q and -v as exact f16
// operands, returned packed {e_lo, e_hi}.  nv = f16 bit pattern of -v_c.
__device__ __forceinline__ u64 err2_of_t(u64 t2, u64 y2, uint16_t nv) {
    u64 e2;
    asm("{\n\t"
        ".reg .b32 tl, th, yl, yh, h2, el, eh;\n\t"
        ".reg .b16 ql, qh;\n\t"
        ".reg .b8 q;\n\t"
        "mov.b64 {tl, th}, %1;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 q, th, tl;\n\t"
        "cvt.rn.f16x2.e2m1x2 h2, q;\n\t"
        "mov.b32 {ql, qh}, h2;\n\t"
        "mov.b64 {yl, yh}, %2;\n\t"
        "fma.rn.f32.f16 el, ql, %3, yl;\n\t"
        "fma.rn.f32.f16 eh, qh, %3, yh;\n\t"
        "mov.b64 %0, {el, eh};\n\t"
        "}"
        : "=l"(e2) : "l"(t2), "l"(y2), "h"(nv));
    return e2;
}
__device__ __forceinline__ u64 cand_err2(u64 y2, u64 r2, uint16_t nv) { return err2_of_t(mul2(y2, r2), y2, nv); }

// E4M3 code -> f16 bit pattern of its value (exact), via the native decode.
__device__ __forceinline__ uint16_t e4m3_to_f16bits(uint32_t code) {
    uint32_t h2;
    uint16_t c16 = (uint16_t)(code & 0xFF);
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(c16));
    return (uint16_t)(h2 & 0xFFFF);
}

__device__ __forceinline__ float f16bits_to_f32(uint16_t h) {
    float f;
    asm("cvt.f32.f16 %0, %1;" : "=f"(f) : "h"(h));
    return f;
}

// RN_E4M3 (ties to even, saturating at 448) of a non-negative fp32, as a code.
__device__ __forceinline__ uint32_t e4m3_rn_code(float s) {
    uint16_t d;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(d) : "f"(0.0f), "f"(s));
    return (uint32_t)(d & 0xFF);
}

// floor_E4M3 of a non-negative fp32 as a code: the largest code in 0..126 with
// value <= s (Sec. 3.1 notation, s_base^FP8 of Sec. 4.2.2).  Normal E4M3 values
// truncate the fp32 mantissa to 3 bits; subnormal ones are floor(s * 2^9).
__device__ __forceinline__ int e4m3_floor_code(float s) {
    if (s >= 448.0f) return 126;
    if (!(s >= 0.001953125f)) return 0;           // below 2^-9 (or NaN)
    uint32_t b = __float_as_uint(s);
    int e = (int)(b >> 23) - 127;
    if (e >= -6) return ((e + 7) << 3) | (int)((b >> 20) & 7u);
    return (int)__fmul_rn(s, 512.0f);                // 1..7, exact scaling then truncation
}

// fl(m / 6) for m >= 0 without the division: a correctly rounded quotient by one
// residual step (compared with the division over every mantissa; below the normal
// range it may differ, where every caller's result is the smallest scale anyway).
__device__ __forceinline__ float sixth(float m) {
    const float q = __fmul_rn(m, 0.16666667163372039794921875f);
    return __fmaf_rn(__fmaf_rn(-6.0f, q, m), 0.16666667163372039794921875f, q);
}

// e4m3_floor_code(fl(m / 6)) for m >= 0 (NaN and inf give 126): m >= 6 v_c exactly
// when the product of m and fl(1/6), which is a third of an ulp above 1/6, rounded
// towards zero reaches v_c -- compared with the division for every fp32 m from the
// octave of the smallest 6 v_c to that of the largest.  Normal codes are the top bits of that
// product, those below 2^-5 its integer part in units of 2^-9.
__device__ __forceinline__ int e4m3_floor_code_of_sixth(float m) {
    const float s = __fmul_rz(m, 0.16666667163372039794921875f);
    const int sub = (int)(__float_as_uint(__fmaf_rz(s, 512.0f, 8388608.0f)) & 0xFFu);
    const int top = (int)(__float_as_uint(s) >> 20) - 960;
    return min(s < 0.03125f ? sub : top, 126);
}

// Byte offset of scale (row r, scale column k) in the 128x4-atom swizzled
// layout read by block-scaled MMA (kpad4 = ceil(kblocks/4)).
__device__ __forceinline__ int64_t swizzle_offset(int64_t r, int64_t k, int64_t kpad4) {
    return ((r >> 7) * kpad4 + (k >> 2)) * 512 + (r & 31) * 16 + ((r >> 5) & 3) * 4 + (k & 3);
}

// The same with 32-bit row, column and atom index (rows * scale columns < 2^32).
__device__ __forceinline__ int64_t swizzle_offset32(uint32_t r, uint32_t k, uint32_t kpad4) {
    return (int64_t)((r >> 7) * kpad4 + (k >> 2)) * 512 + (int)((r & 31) * 16 + ((r >> 5) & 3) * 4 + (k & 3));
}

// Loads of what an earlier kernel may have written: not the non-coherent form, which
// the compiler may move above, and the hardware serve from before, a programmatic
// dependent launch's wait (every one is volatile and stays below it).
__device__ __forceinline__ float ld_f32(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_u32(const void* p) {
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
// Streaming 16-byte load that bypasses L1 allocation (each byte is read once).  NC:
// the non-coherent form, for data that nothing writes while the kernel is scheduled
// (any launch but a programmatic dependent of the data's producer; 0.5% on the sweeps).
template <bool NC = true>
__device__ __forceinline__ uint4 ld_stream16(const void* p) {
    uint4 v;
    if (NC)
        asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    else
        asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// 32 bytes at once (32-byte aligned).  A lane that reads its 32-byte sector in two
// 16-byte halves makes two requests per line and, past L1, fetches the sector twice.
template <bool NC>
__device__ __forceinline__ void ld_stream32(const void* p, uint4& a, uint4& b) {
    if (NC)
        asm volatile("ld.global.nc.L1::no_allocate.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p));
    else
        asm volatile("ld.global.L1::no_allocate.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p));
}
template <bool NC>
__device__ __forceinline__ uint4 ld_ro16(const void* p) {
    uint4 v;
    if (NC)
        asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    else
        asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// Programmatic dependent launch: the running grid lets a kernel launched after
// it with cudaLaunchAttributeProgrammaticStreamSerialization be scheduled once
// every CTA of this grid has executed launch_dependents (or exited); that
// kernel's griddepcontrol.wait returns once this grid has completed and its
// writes are visible (and at once when it was launched the ordinary way).
__device__ __forceinline__ void grid_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch of `kernel` on `s` as a programmatic dependent of the kernel before it on
// the stream: it is scheduled while that one drains, builds what depends on nothing
// and waits (grid_dependency_wait) before it touches memory.  Saves the launch
// latency and the table build of back-to-back calls (2-3 us each).
template <typename... P, typename... Args>
inline cudaError_t launch_dependent_smem(void (*kernel)(P...), int64_t grid, int threads, int smem, cudaStream_t s,
                                         Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

template <typename... P, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(P...), int64_t grid, int threads, cudaStream_t s, Args... args) {
    return launch_dependent_smem(kernel, grid, threads, 0, s, args...);
}

__device__ __forceinline__ float bf16lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

}  // namespace nvfp4
