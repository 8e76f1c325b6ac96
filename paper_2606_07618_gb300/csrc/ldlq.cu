// LDLQ (GPTQ's error-feedback pass) with fixed NVFP4 block scales and static
// reordering -- Appendix A.2 of the ScaleSweep paper: GPTQ run as LDLQ (QuIP),
// damping 0.01 x the mean Hessian diagonal, block scales fixed beforehand by
// ScaleSweep, input channels processed in descending order of diag(H).
//
// Prepare (depends on H only):
//   lambda = damp * mean(diag H); perm = channels by (diag desc, index asc);
//   A = J H_pi J + lambda I (J reverses the order), A = L L^T by a blocked
//   right-looking Cholesky (64-wide panels: diagonal block factor and inverse
//   in one CTA, panel solve by the inverse and update of the next block column in
//   one kernel, the rest of the trailing update by a K<=64 GEMM on lower tiles
//   only); then, in place,
//   H_pi = (U + I) D (U + I)^T with U_ik = L[n-1-i][n-1-k] / L[n-1-k][n-1-k]
//   (J L J is upper triangular) and D_k = L[n-1-k][n-1-k]^2.
// Quantize (rows independent):
//   T = W_pi (fp32); per 256-column super-panel, one lane per row walks the
//   columns in order -- What_k = Q(T_k) at the element's fixed scale, e_k = W_k -
//   What_k, T_j += e_k U_kj for the later columns of the super-panel -- then the
//   later columns get T += E U (the GEMM); finally the nibbles are scattered back
//   to the original column order.
// Q follows the sweep's float32 contract: y = fl(t*E), q = RNE_E2M1(fl(y*r_c)),
// What = fl(fl(q*v_c)*S); a zero-scale block or an unusable S gives signed
// zeros; an exactly zero y takes the +0 code.
#include <atomic>
#include <mutex>
#include <type_traits>

#include <cuda_bf16.h>

#include "nvfp4_device.cuh"
#include "ldlq_kernels.h"
#include "nvfp4_kernels.h"
#include "tc_gemm.cuh"

namespace nvfp4 {

namespace {

constexpr int kP = 64;                // Cholesky panel width
constexpr int kLd = 132;              // GEMM smem row stride (floats): 128 + 4, 16-byte rows

inline int64_t imin64(int64_t a, int64_t b) { return a < b ? a : b; }

__device__ __forceinline__ float sort_key(float v) { return isnan(v) ? -INFINITY : v; }

// d = diag(H), lambda = damp * mean(d) (double sum); bit 4 if any diagonal entry is not finite.
__global__ void __launch_bounds__(1024) diag_kernel(const float* H, int64_t n, float damp, float* d, float* lam,
                                                    int* status) {
    double s = 0.0;
    int bad = 0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const float v = H[i * n + i];
        d[i] = v;
        if (isfinite(v)) s += (double)v; else bad = 1;
    }
    __shared__ double ss[32];
    __shared__ int sb[32];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    bad = __reduce_or_sync(0xffffffffu, (unsigned)bad);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        ss[warp] = s;
        sb[warp] = bad;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        int b = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            t += ss[w];
            b |= sb[w];
        }
        lam[0] = (float)((double)damp * t / (double)n);
        if (b && status) atomicOr(status, 4);
    }
}

// perm[rank(i)] = i, rank by (key desc, index asc): a total order, so perm is a
// permutation of 0..n-1 whatever the keys.  A warp per channel, its lanes over the
// others (one thread per channel left 16 CTAs walking 4096 keys each: 85 us at n =
// 4096).
__global__ void __launch_bounds__(256) rank_kernel(const float* d, int64_t n, int32_t* perm) {
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= n) return;
    const float di = sort_key(d[i]);
    unsigned rank = 0;
#pragma unroll 4
    for (int64_t j = lane; j < n; j += 32) {
        const float dj = sort_key(__ldg(d + j));
        rank += (dj > di) || (dj == di && j < i);
    }
    rank = __reduce_add_sync(0xffffffffu, rank);
    if (lane == 0) perm[rank] = (int32_t)i;
}

// A[a][b] = H[p(a)][p(b)] (+ lambda on the diagonal) for b <= a, p(a) = perm[n-1-a];
// nothing reads the upper part.
__global__ void __launch_bounds__(256) gather_h_kernel(const float* H, int64_t n, const int32_t* perm,
                                                       const float* lam, float* A) {
    const float l = lam[0];
    for (int64_t a = blockIdx.x; a < n; a += gridDim.x) {
        const float* hrow = H + (int64_t)perm[n - 1 - a] * n;
        float* arow = A + a * n;
        for (int64_t b = threadIdx.x; b <= a; b += blockDim.x) {
            float v = hrow[perm[n - 1 - b]];
            if (a == b) v = __fadd_rn(v, l);
            arow[b] = v;
        }
    }
}

// out[r][c] = sum_{k < K} x[r][k] y[c][k] for the rows r = r0 + RS i and columns
// c = c0 + CS j of a thread's 4 x 4 tile; x and y in shared memory, kPad words per
// row, K a multiple of 4.  Even and odd k are summed apart (packed fp32).
constexpr int kPad = kP + 4;          // rows 4 banks apart: eight lanes' 16-byte reads cover all banks
// LOW (CS = 16): y is lower triangular, so column group j ends at k = 16 j + 15.
template <int RS, int CS, bool LOW = false>
__device__ __forceinline__ void tile_dot(const float* x, int r0, const float* y, int c0, int K, float (&out)[4][4]) {
    u64 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = 0ull;
    auto chunk = [&](int k, int j0) {
        float4 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; i++) a[i] = *reinterpret_cast<const float4*>(x + (r0 + RS * i) * kPad + k);
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (j >= j0) b[j] = *reinterpret_cast<const float4*>(y + (c0 + CS * j) * kPad + k);
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (j >= j0) {
                    acc[i][j] = fma2(pack2(a[i].x, a[i].y), pack2(b[j].x, b[j].y), acc[i][j]);
                    acc[i][j] = fma2(pack2(a[i].z, a[i].w), pack2(b[j].z, b[j].w), acc[i][j]);
                }
    };
    if (LOW) {
#pragma unroll
        for (int j0 = 0; j0 < 4; j0++)
#pragma unroll 2
            for (int k = 16 * j0; k < 16 * j0 + 16; k += 4) chunk(k, j0);
    } else {
#pragma unroll 2
        for (int k = 0; k < K; k += 4) chunk(k, 0);
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
            float lo, hi;
            unpack2(acc[i][j], lo, hi);
            out[i][j] = __fadd_rn(lo, hi);
        }
}

// 1/p to an ulp without the branches of the rounded form: the hardware's
// approximation and, where its residual is a normal number, one Newton step.
__device__ __forceinline__ float rcp_fast(float p) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(p));
    return p > 1e-37f ? __fmaf_rn(r, __fmaf_rn(-p, r, 1.0f), r) : r;
}

constexpr int kPotrfThreads = 544;
// All of potrf_kernel's warps, from either role's code.
__device__ __forceinline__ void potrf_barrier() {
    __syncwarp();
    asm volatile("barrier.sync 1, %0;" ::"n"(kPotrfThreads) : "memory");
}

__device__ __forceinline__ float sum2(u64 v) {
    float lo, hi;
    unpack2(v, lo, hi);
    return __fadd_rn(lo, hi);
}

// One panel's sequential part, in one CTA: the Cholesky factor of the nb x nb
// diagonal block at k0 (lower, in place), its inverse Linv (64 x 64, lower), and the
// solved panel of the next 64 rows, Xtop = A[k0 + nb .., k0 ..] Linv^T, element (r, c) at
// r xr + c xc.
//
// The block is padded to 64 with an identity and held as 4 x 4 tiles in registers.
// Warp J < 16 holds tile column J: lanes (I, h) have rows 2h, 2h + 1 of tile (I, J)
// of the block for I > J and, for I < J, of tile (J, I) of X = M^-1, transposed; lane
// T of the last warp holds both diagonal tiles T.  The pivots stay unscaled, A = M
// diag(p) M^T with M unit lower triangular.  Block step b: the last warp factors
// tile b and publishes M_bb and 1/p; after a barrier warp b's tiles become
// W = A M_bb^-T and the multipliers -W / p, and the tiles of X's row b take the same
// steps; after another, every remaining tile takes its rank-4 update, tile -= m_I W_J^T
// or X^T tile -= X_b^T m_I^T (the same code), the last warp's first of all.  Then
// L = M diag(sqrt p) and Linv = diag(1/sqrt p) X.  A pivot that is not positive and
// finite sets bit 4 of the status word and is replaced by 1 so the values stay finite.
//
// Bound by latency: 16 steps of a 4-pivot chain (370 cycles alone: a reciprocal, two
// dependent multiply-adds and a test per pivot), two barriers, the solve (150-300)
// and the diagonal tiles' update (300).  A column per warp lets one full warp do the
// solve while the others wait; with a tile row per warp every warp went through it on
// two lanes (n = 4096: 1605 us for the whole factorization, with it 1579).  The
// update's shared-memory reads (24 words a thread) take the other warps about as long
// as the next tile's factor.  One column per step (64 barriers, every thread updating a
// tile of both matrices) took 17.8 us a block without Xtop, this 13 us; one warp
// factoring 16 x 16 blocks, the column going round by shuffles or through shared
// memory, 480-560 cycles per column.  Holding the workers back until the diagonal
// tiles have read their operands: no gain.
__global__ void __launch_bounds__(kPotrfThreads) potrf_kernel(float* A, int64_t n, int64_t k0, int nb, float* Linv,
                                                              float* Xtop, int64_t xr, int64_t xc, int* status) {
    extern __shared__ __align__(16) float psm[];
    float* sl = psm;                                 // [64][kPad] Linv
    float* st = psm + kP * kPad;                     // [64][kPad] the next 64 rows of the panel
    // W, -W / p, X_b^T: entry i of tile T at [i][T], so that a warp's tiles lie in distinct banks
    // (one array, indexed: a pointer chosen between arrays would make the accesses generic)
    constexpr int kW = 0, kMul = 4, kX = 8;
    __shared__ __align__(16) float4 sb[12][16];
    __shared__ __align__(16) float sm[8], sip[4];
    __shared__ float piv[kP];
    const int tid = threadIdx.x, lane = tid & 31;
    const bool dwarp = tid >= 512;
    const int I = tid & 15, J = (tid >> 5) & 15, h = 2 * ((tid >> 4) & 1);
    const bool low = J < I, off = J != I;
    const int R = low ? I : J, C = low ? J : I;      // a worker's tile: (R, C) of A (low) or of X
    const int nt = (int)(n - k0 - nb < kP ? n - k0 - nb : kP);          // rows of Xtop
    // the previous panel's kernel updated this block column
    grid_dependency_wait();
    if (!dwarp) {
        // every load before the first store to shared memory: one trip to L2
        float v[kP * kP / 512], w[kP * kP / 512];
#pragma unroll
        for (int e = 0; e < kP * kP / 512; e++) {
            const int r = e * 8 + (tid >> 6), c = tid & 63;
            v[e] = r < nb && c <= r ? A[(k0 + r) * n + k0 + c] : r == c ? 1.0f : 0.0f;
            w[e] = r < nt ? A[(k0 + nb + r) * n + k0 + c] : 0.0f;
        }
#pragma unroll
        for (int e = 0; e < kP * kP / 512; e++) {
            const int r = e * 8 + (tid >> 6), c = tid & 63;
            sl[r * kPad + c] = v[e];
            st[r * kPad + c] = w[e];
        }
    }
    potrf_barrier();
    int bad = 0;
    if (dwarp) {
        u64 t2[4][4];                                // lane T: A's diagonal tile, each entry as two sums
        float t[4][4], xd[4][4];                     // factored, and X's diagonal tile
        const int T = lane & 15;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const float4 q = *reinterpret_cast<const float4*>(sl + (4 * T + i) * kPad + 4 * T);
            t2[i][0] = pack2(q.x, 0.0f);
            t2[i][1] = pack2(q.y, 0.0f);
            t2[i][2] = pack2(q.z, 0.0f);
            t2[i][3] = pack2(q.w, 0.0f);
#pragma unroll
            for (int j = 0; j < 4; j++) t[i][j] = xd[i][j] = i == j ? 1.0f : 0.0f;
        }
#pragma unroll 1
        for (int b = 0; b < kP / 4; b++) {
            if (lane == b) {
                float p[4], ip[4], m[4][4];
#pragma unroll
                for (int i = 0; i < 4; i++)
#pragma unroll
                    for (int j = 0; j <= i; j++) t[i][j] = sum2(t2[i][j]);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const bool ok = __float_as_uint(t[j][j]) - 1u < 0x7f7fffffu;      // positive and finite
                    bad |= !ok;
                    p[j] = ok ? t[j][j] : 1.0f;
                    ip[j] = rcp_fast(p[j]);
#pragma unroll
                    for (int i = j + 1; i < 4; i++) m[i][j] = __fmul_rn(t[i][j], ip[j]);
#pragma unroll
                    for (int i = j + 1; i < 4; i++)
#pragma unroll
                        for (int l = j + 1; l <= i; l++) t[i][l] = __fmaf_rn(-m[i][j], t[l][j], t[i][l]);
                }
                *reinterpret_cast<float4*>(sip) = make_float4(ip[0], ip[1], ip[2], ip[3]);
                *reinterpret_cast<float4*>(sm) = make_float4(m[1][0], m[2][0], m[2][1], m[3][0]);
                *reinterpret_cast<float2*>(sm + 4) = make_float2(m[3][1], m[3][2]);
#pragma unroll
                for (int j = 0; j < 4; j++) t[j][j] = p[j];
#pragma unroll
                for (int i = 1; i < 4; i++)
#pragma unroll
                    for (int j = 0; j < i; j++) t[i][j] = m[i][j];     // M_bb stays in the tile
            }
            potrf_barrier();
            if (lane == b) {
                // X's diagonal tile M_bb^-1 (unit lower), transposed for the update
                xd[1][0] = -t[1][0];
                xd[2][1] = -t[2][1];
                xd[3][2] = -t[3][2];
                xd[2][0] = __fmaf_rn(t[2][1], t[1][0], -t[2][0]);
                xd[3][1] = __fmaf_rn(t[3][2], t[2][1], -t[3][1]);
                xd[3][0] = __fmaf_rn(-t[3][2], xd[2][0], __fmaf_rn(-t[3][1], xd[1][0], -t[3][0]));
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    sb[kX + j][b] = make_float4(xd[0][j], xd[1][j], xd[2][j], xd[3][j]);
                    piv[4 * b + j] = t[j][j];
                }
            }
            potrf_barrier();
            if (T > b) {
                float4 mr[4], yc[4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    mr[i] = sb[kMul + i][T];
                    yc[i] = sb[kW + i][T];
                }
#pragma unroll
                for (int i = 0; i < 4; i++)
#pragma unroll
                    for (int j = 0; j <= i; j++) {
                        t2[i][j] = fma2(pack2(mr[i].x, mr[i].y), pack2(yc[j].x, yc[j].y), t2[i][j]);
                        t2[i][j] = fma2(pack2(mr[i].z, mr[i].w), pack2(yc[j].z, yc[j].w), t2[i][j]);
                    }
            }
        }
        potrf_barrier();
        potrf_barrier();                             // the workers' sqrt p and 1 / sqrt p
        const float* sq = &sb[0][0].x;
        if (lane < 16) {
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j <= i; j++)
                    sl[(4 * T + i) * kPad + 4 * T + j] = i == j ? sq[4 * T + j] : __fmul_rn(t[i][j], sq[4 * T + j]);
        }
        potrf_barrier();
        potrf_barrier();                             // L is read
        if (lane < 16) {
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const int r = 4 * T + i;
                float o[4];
#pragma unroll
                for (int j = 0; j < 4; j++) o[j] = j <= i ? __fmul_rn(xd[i][j], sq[kP + r]) : 0.0f;
                const float4 x = make_float4(o[0], o[1], o[2], o[3]);
                *reinterpret_cast<float4*>(sl + r * kPad + 4 * T) = x;
                *reinterpret_cast<float4*>(Linv + r * kP + 4 * T) = x;
            }
        }
    } else {
        u64 t2[2][4];                                // rows h, h + 1 of the tile, each entry as two sums
#pragma unroll
        for (int i = 0; i < 2; i++) {
            float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (low) q = *reinterpret_cast<const float4*>(sl + (4 * R + h + i) * kPad + 4 * C);
            t2[i][0] = pack2(q.x, 0.0f);
            t2[i][1] = pack2(q.y, 0.0f);
            t2[i][2] = pack2(q.z, 0.0f);
            t2[i][3] = pack2(q.w, 0.0f);
        }
        float t[2][4] = {};                          // solved
#pragma unroll 1
        for (int b = 0; b < kP / 4; b++) {
            if (J == b) {
#pragma unroll
                for (int i = 0; i < 2; i++)
#pragma unroll
                    for (int j = 0; j < 4; j++) t[i][j] = sum2(t2[i][j]);
            }
            potrf_barrier();
            // W = A M_bb^-T below the block; X's row b, held transposed, takes the same steps
            if (J == b && off) {
                const float4 ma = *reinterpret_cast<const float4*>(sm), ip = *reinterpret_cast<const float4*>(sip);
                const float2 mb = *reinterpret_cast<const float2*>(sm + 4);
                const int dst = (low ? kW : kX) + h;
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    t[i][1] = __fmaf_rn(-t[i][0], ma.x, t[i][1]);
                    t[i][2] = __fmaf_rn(-t[i][0], ma.y, t[i][2]);
                    t[i][3] = __fmaf_rn(-t[i][0], ma.w, t[i][3]);
                    t[i][2] = __fmaf_rn(-t[i][1], ma.z, t[i][2]);
                    t[i][3] = __fmaf_rn(-t[i][1], mb.x, t[i][3]);
                    t[i][3] = __fmaf_rn(-t[i][2], mb.y, t[i][3]);
                    sb[dst + i][I] = make_float4(t[i][0], t[i][1], t[i][2], t[i][3]);
                    if (low)                         // (X's tiles have no multipliers)
                        sb[kMul + h + i][I] = make_float4(__fmul_rn(t[i][0], -ip.x), __fmul_rn(t[i][1], -ip.y),
                                                          __fmul_rn(t[i][2], -ip.z), __fmul_rn(t[i][3], -ip.w));
                }
            }
            potrf_barrier();
            if (low ? J > b : off && J > b && I <= b) {
                // A: t[i][j] -= m_(R i) . W_(C j);  X^T: t[i][j] -= X_b^T_(C i) . m_(R j)
                const int u = (low ? kMul : kX) + h, y = low ? kW : kMul;
                float4 mr[2], yc[4];
#pragma unroll
                for (int i = 0; i < 2; i++) mr[i] = sb[u + i][I];
#pragma unroll
                for (int j = 0; j < 4; j++) yc[j] = sb[y + j][J];
#pragma unroll
                for (int i = 0; i < 2; i++)
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        t2[i][j] = fma2(pack2(mr[i].x, mr[i].y), pack2(yc[j].x, yc[j].y), t2[i][j]);
                        t2[i][j] = fma2(pack2(mr[i].z, mr[i].w), pack2(yc[j].z, yc[j].w), t2[i][j]);
                    }
            }
        }
        // L into the block, Linv = diag(1 / sqrt p) X into shared and global memory
        potrf_barrier();
        float* sq = &sb[0][0].x;                     // sqrt p, then 1 / sqrt p
        if (tid < kP) {
            sq[tid] = __fsqrt_rn(piv[tid]);
            sq[kP + tid] = __frsqrt_rn(piv[tid]);
        }
        potrf_barrier();
        if (low) {
            // W = M p, so below the diagonal tile L = M sqrt p = W / sqrt p
            const float4 q = *reinterpret_cast<const float4*>(sq + kP + 4 * C);
#pragma unroll
            for (int i = 0; i < 2; i++)
                *reinterpret_cast<float4*>(sl + (4 * R + h + i) * kPad + 4 * C) =
                    make_float4(__fmul_rn(t[i][0], q.x), __fmul_rn(t[i][1], q.y), __fmul_rn(t[i][2], q.z),
                                __fmul_rn(t[i][3], q.w));
        }
        potrf_barrier();
#pragma unroll
        for (int e = 0; e < kP * kP / 512; e++) {
            const int r = e * 8 + (tid >> 6), c = tid & 63;
            if (r < nb && c <= r) A[(k0 + r) * n + k0 + c] = sl[r * kPad + c];
        }
        potrf_barrier();
        if (!low && off) {
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int r = 4 * R + j;
                const float2 x = make_float2(__fmul_rn(t[0][j], sq[kP + r]), __fmul_rn(t[1][j], sq[kP + r]));
                *reinterpret_cast<float2*>(sl + r * kPad + 4 * C + h) = x;
                *reinterpret_cast<float2*>(Linv + r * kP + 4 * C + h) = x;
            }
            const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);       // the upper part
#pragma unroll
            for (int i = 0; i < 2; i++) {
                *reinterpret_cast<float4*>(sl + (4 * C + h + i) * kPad + 4 * R) = z;
                *reinterpret_cast<float4*>(Linv + (4 * C + h + i) * kP + 4 * R) = z;
            }
        }
    }
    if (bad && status) atomicOr(status, 4);
    potrf_barrier();
    // Xtop: rows r + 16 i, columns J + 16 j of the solved panel
    if (nt > 0 && tid < 256) {
        float o[4][4];
        const int r = tid >> 4, c = tid & 15;
        tile_dot<16, 16, true>(st, r, sl, c, kP, o);
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (r + 16 * i < nt) Xtop[(r + 16 * i) * xr + (c + 16 * j) * xc] = o[i][j];
    }
}

// The rows i >= k0 + 64 of one panel, 32 per CTA: the solved panel X = A Linv^T (in
// place, and, unless Lh is null, split into TF32 halves Lh, Ll [n, 64] for the trailing
// update), then the next panel's block column, A[i][k0 + 64 ..] -= X Xtop^T, up to column i.  Everything in fp32 from shared memory; a separate panel solve and a
// tensor-core update of a 64-wide column spent 14 us here on launches, tile fills
// and half-empty tiles.
constexpr int kPanelRows = 32;
constexpr int kPanelSmem = (2 * kP + 2 * kPanelRows) * kPad * 4;
template <bool VEC>
__global__ void __launch_bounds__(128) panel_kernel(float* A, int64_t n, int64_t k0, const float* Linv, const float* Xtop,
                                                    int64_t xr, int64_t xc, float* Lh, float* Ll) {
    grid_launch_dependents();                        // the next diagonal factor waits for this grid's end
    extern __shared__ __align__(16) float psm[];
    float* sl = psm;                                 // [64][kPad] Linv
    float* st = sl + kP * kPad;                      // [64][kPad] Xtop
    float* sa = st + kP * kPad;                      // [32][kPad] the rows
    float* sx = sa + kPanelRows * kPad;              // [32][kPad] the solved rows
    const int64_t i0 = k0 + kP + (int64_t)blockIdx.x * kPanelRows;
    const int rows = (int)(n - i0 < kPanelRows ? n - i0 : kPanelRows);
    // every load before the first store to shared memory: one trip to L2
    constexpr int kQ = kP / 4;
    float4 vl[kP * kQ / 128], vt[kP * kQ / 128], va[kPanelRows * kQ / 128];
#pragma unroll
    for (int u = 0; u < kPanelRows * kQ / 128; u++) {
        const int e = threadIdx.x + 128 * u, r = e / kQ, c = 4 * (e % kQ);
        va[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (r < rows) {
            const float* a = A + (i0 + r) * n + k0 + c;
            if (VEC) va[u] = *reinterpret_cast<const float4*>(a);
            else va[u] = make_float4(a[0], a[1], a[2], a[3]);
        }
    }
#pragma unroll
    for (int u = 0; u < kP * kQ / 128; u++) {
        vl[u] = reinterpret_cast<const float4*>(Linv)[threadIdx.x + 128 * u];
        const int e = threadIdx.x + 128 * u, r = e / kQ, c = 4 * (e % kQ);
        vt[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (k0 + kP + r < n) {
            const float* x = Xtop + r * xr + c * xc;
            if (xc == 1) vt[u] = *reinterpret_cast<const float4*>(x);
            else vt[u] = make_float4(x[0], x[xc], x[2 * xc], x[3 * xc]);
        }
    }
#pragma unroll
    for (int u = 0; u < kPanelRows * kQ / 128; u++) {
        const int e = threadIdx.x + 128 * u;
        *reinterpret_cast<float4*>(sa + (e / kQ) * kPad + 4 * (e % kQ)) = va[u];
    }
#pragma unroll
    for (int u = 0; u < kP * kQ / 128; u++) {
        const int e = threadIdx.x + 128 * u;
        *reinterpret_cast<float4*>(sl + (e / kQ) * kPad + 4 * (e % kQ)) = vl[u];
        *reinterpret_cast<float4*>(st + (e / kQ) * kPad + 4 * (e % kQ)) = vt[u];
    }
    __syncthreads();
    // thread: rows ty + 8 i, columns 4 tx .. (phase 1: Linv's row c ends at column c) or tx + 16 j
    const int ty = threadIdx.x & 7, tx = threadIdx.x >> 3;
    float o[4][4];
    tile_dot<8, 1>(sa, ty, sl, 4 * tx, 4 * tx + 4, o);
#pragma unroll
    for (int i = 0; i < 4; i++)
        *reinterpret_cast<float4*>(sx + (ty + 8 * i) * kPad + 4 * tx) = make_float4(o[i][0], o[i][1], o[i][2], o[i][3]);
    __syncthreads();
    // the solved rows, and the block column's values, which the products below come off
    float4 vc[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int64_t r = i0 + ty + 8 * i, c0 = k0 + kP + 4 * tx;
        vc[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (r >= n) continue;
        float* a = A + r * n + k0 + 4 * tx;
        if (VEC) {
            const float4 x = make_float4(o[i][0], o[i][1], o[i][2], o[i][3]);
            *reinterpret_cast<float4*>(a) = x;
            if (Lh) {                                 // the trailing update's operands
                float4 h, l;
                tc::split4(x, h, l);
                *reinterpret_cast<float4*>(Lh + r * kP + 4 * tx) = h;
                *reinterpret_cast<float4*>(Ll + r * kP + 4 * tx) = l;
            }
            if (c0 + 3 <= r) vc[i] = *reinterpret_cast<const float4*>(A + r * n + c0);
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++) a[j] = o[i][j];
        }
    }
    tile_dot<8, 1>(sx, ty, st, 4 * tx, kP, o);
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int64_t r = i0 + ty + 8 * i, c0 = k0 + kP + 4 * tx;
        if (r >= n) continue;
        float* c = A + r * n + c0;
        if (VEC && c0 + 3 <= r) {
            *reinterpret_cast<float4*>(c) = make_float4(__fsub_rn(vc[i].x, o[i][0]), __fsub_rn(vc[i].y, o[i][1]),
                                                        __fsub_rn(vc[i].z, o[i][2]), __fsub_rn(vc[i].w, o[i][3]));
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (c0 + j <= r) c[j] = __fsub_rn(c[j], o[i][j]);
        }
    }
}

// C[M, N] += alpha * A * op(B), A [M, K] row-major; op(B) = B [K, N] row-major, or
// (BT) B^T with B stored [N, K] row-major.  128 x 128 tiles, 256 threads, 8 x 8 outputs per
// thread, K in stages of 32 through two shared buffers filled by cp.async
// (global to shared without registers) while the other stage is multiplied.
// LOWER skips tiles entirely above the diagonal (n0 > m0 + 127).  VEC: C rows
// and the column base are 16-byte aligned, so the epilogue moves float4s.
constexpr int kBK = 32;

__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool valid) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    const int n = valid ? 4 : 0;                    // 0: zero-fill, nothing is read
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

template <bool BT, bool LOWER, bool VEC>
__global__ void __launch_bounds__(256, 2) gemm_kernel(float* C, int64_t ldc, const float* A, int64_t lda,
                                                      const float* B, int64_t ldb, int64_t M, int64_t N, int K,
                                                      float alpha) {
    extern __shared__ __align__(16) float smem[];
    float* As = smem;                         // [2][kBK][kLd]: As[b][k][m]
    float* Bs = smem + 2 * kBK * kLd;         // [2][kBK][kLd]: Bs[b][k][n]
    const int64_t m0 = (int64_t)blockIdx.y * 128, n0 = (int64_t)blockIdx.x * 128;
    if (LOWER && n0 > m0 + 127) return;
    const int tid = threadIdx.x;
    // element e = tid + 256*i of a 128 x 32 (A) or 32 x 128 (B) stage tile
    auto issue = [&](int k0, int b) {
        float* as = As + b * kBK * kLd;
        float* bs = Bs + b * kBK * kLd;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const int e = tid + 256 * i;
            {
                const int mm = e / kBK, k = e % kBK;
                const bool ok = k0 + k < K && m0 + mm < M;
                cp_async4(as + k * kLd + mm, ok ? A + (m0 + mm) * lda + k0 + k : A, ok);
            }
            if (BT) {
                const int nn = e / kBK, k = e % kBK;
                const bool ok = k0 + k < K && n0 + nn < N;
                cp_async4(bs + k * kLd + nn, ok ? B + (n0 + nn) * ldb + k0 + k : B, ok);
            } else {
                const int k = e / 128, nn = e % 128;
                const bool ok = k0 + k < K && n0 + nn < N;
                cp_async4(bs + k * kLd + nn, ok ? B + (int64_t)(k0 + k) * ldb + n0 + nn : B, ok);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int tx = tid & 15, ty = tid >> 4;
    // 8 x 8 outputs per thread as 8 x 4 packed pairs: one fma.rn.f32x2 per pair
    // (per lane the same IEEE fma as the scalar form, at twice the operands per
    // register read).
    u64 acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = 0ull;
    const int nst = (K + kBK - 1) / kBK;
    issue(0, 0);
    for (int st = 0; st < nst; st++) {
        const int b = st & 1;
        if (st + 1 < nst) {
            issue((st + 1) * kBK, b ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float* as = As + b * kBK * kLd;
        const float* bs = Bs + b * kBK * kLd;
#pragma unroll 8
        for (int k = 0; k < kBK; k++) {
            const float4 a0 = *reinterpret_cast<const float4*>(as + k * kLd + ty * 4);
            const float4 a1 = *reinterpret_cast<const float4*>(as + k * kLd + 64 + ty * 4);
            const float4 b0 = *reinterpret_cast<const float4*>(bs + k * kLd + tx * 4);
            const float4 b1 = *reinterpret_cast<const float4*>(bs + k * kLd + 64 + tx * 4);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const u64 bp[4] = {pack2(b0.x, b0.y), pack2(b0.z, b0.w), pack2(b1.x, b1.y), pack2(b1.z, b1.w)};
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const u64 ap = pack2(av[i], av[i]);
#pragma unroll
                for (int j = 0; j < 4; j++) acc[i][j] = fma2(ap, bp[j], acc[i][j]);
            }
        }
        __syncthreads();                           // buffer b is refilled by the next issue
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const int64_t r = m0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + i - 4);
        if (r >= M) continue;
        float* crow = C + r * ldc;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int64_t c = n0 + h * 64 + tx * 4;
            float o[4];
            unpack2(acc[i][2 * h], o[0], o[1]);
            unpack2(acc[i][2 * h + 1], o[2], o[3]);
            if (VEC && c + 3 < N) {
                float4 v = *reinterpret_cast<float4*>(crow + c);
                v.x = __fmaf_rn(alpha, o[0], v.x);
                v.y = __fmaf_rn(alpha, o[1], v.y);
                v.z = __fmaf_rn(alpha, o[2], v.z);
                v.w = __fmaf_rn(alpha, o[3], v.w);
                *reinterpret_cast<float4*>(crow + c) = v;
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (c + j < N) crow[c + j] = __fmaf_rn(alpha, o[j], crow[c + j]);
            }
        }
    }
}

template <bool BT, bool LOWER, bool VEC>
cudaError_t launch_gemm_t(float* C, int64_t ldc, const float* A, int64_t lda, const float* B, int64_t ldb, int64_t M,
                          int64_t N, int K, float alpha, cudaStream_t s) {
    constexpr int kSmem = 4 * kBK * kLd * (int)sizeof(float);
    static std::atomic<bool> attr_set[64];        // per device: the shared-memory opt-in is done
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute(gemm_kernel<BT, LOWER, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_release);
    }
    const dim3 grid((unsigned)((N + 127) / 128), (unsigned)((M + 127) / 128));
    gemm_kernel<BT, LOWER, VEC><<<grid, 256, kSmem, s>>>(C, ldc, A, lda, B, ldb, M, N, K, alpha);
    return cudaGetLastError();
}

template <bool BT, bool LOWER>
cudaError_t launch_gemm(float* C, int64_t ldc, const float* A, int64_t lda, const float* B, int64_t ldb, int64_t M,
                        int64_t N, int K, float alpha, cudaStream_t s) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    const bool vec = (ldc % 4 == 0) && ((reinterpret_cast<uintptr_t>(C) & 15) == 0);
    return vec ? launch_gemm_t<BT, LOWER, true>(C, ldc, A, lda, B, ldb, M, N, K, alpha, s)
               : launch_gemm_t<BT, LOWER, false>(C, ldc, A, lda, B, ldb, M, N, K, alpha, s);
}

__global__ void diag_d_kernel(const float* A, int64_t n, float* D) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) {
        const float l = A[(n - 1 - k) * n + (n - 1 - k)];
        D[k] = __fmul_rn(l, l);
    }
}

// In place: U[n-1-a][n-1-b] = L[a][b] / L[b][b] for a > b; L[a][b] = 0.  Every
// thread reads its own lower entry and a diagonal entry and writes its own lower
// entry and one upper entry that nothing reads, so the threads do not race.
__global__ void __launch_bounds__(256) flip_kernel(float* A, int64_t n) {
    for (int64_t a = blockIdx.x; a < n; a += gridDim.x) {
        for (int64_t b = threadIdx.x; b < a; b += blockDim.x) {
            const float v = __fdiv_rn(A[a * n + b], A[b * n + b]);
            A[(n - 1 - a) * n + (n - 1 - b)] = v;
            A[a * n + b] = 0.0f;
        }
    }
}

__global__ void zero_diag_kernel(float* A, int64_t n) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) A[k * n + k] = 0.0f;
}

// ---------------------------------------------------------------- quantize

__device__ __forceinline__ int32_t checked_index(int32_t p, int64_t n, int* status) {
    if ((uint32_t)p >= (uint64_t)n) {
        if (status) atomicOr(status, 8);
        return 0;
    }
    return p;
}

__global__ void __launch_bounds__(256) invperm_kernel(const int32_t* perm, int64_t n, int32_t* inv, int* status) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) inv[checked_index(perm[k], n, status)] = (int32_t)k;
}

template <int DT>
__device__ __forceinline__ float load_w(const void* W, int64_t idx) {
    if (DT == 0) return __uint_as_float((uint32_t)(static_cast<const uint16_t*>(W)[idx]) << 16);
    return static_cast<const float*>(W)[idx];
}

// T[r][k] = Wp[r][k] = W[r][perm[k]] (fp32) and sfp[r][k] = sf[r][perm[k] / block],
// one row at a time straight from global memory: rows too long for gather_w_kernel.
template <int DT>
__global__ void __launch_bounds__(256) gather_w_long_kernel(LdlqParams p) {
    for (int64_t r = blockIdx.x; r < p.rows; r += gridDim.x)
        for (int64_t k = threadIdx.x; k < p.n; k += blockDim.x) {
            const int64_t c = checked_index(p.perm[k], p.n, p.status);
            const float v = load_w<DT>(p.W, r * p.n + c);
            p.T[r * p.n + k] = v;
            p.Wp[r * p.n + k] = v;
            uint8_t code = p.sf[r * p.kb + c / p.block];
            p.sfp[r * p.n + k] = code > 126 ? 0 : code;      // 0x7F (NaN) and above: a zero scale
        }
}

// The same through shared memory, kGatherRows rows at a time: the rows come in
// coalesced and the random reads are shared-memory ones.  Straight from global memory
// every gathered word is a cache-line lookup of its own, which bound it (54 us at
// 4096 x 4096 bf16, where writing the targets and weights takes 20).
constexpr int kGatherRows = 4;
template <int DT>
__host__ __device__ inline int64_t gather_row_bytes(int64_t n) {        // a row's weights, 16 bytes apart
    return n * (DT == 0 ? 2 : 4);
}
template <int DT>
__global__ void __launch_bounds__(256) gather_w_kernel(LdlqParams p, int shift) {
    extern __shared__ __align__(16) uint8_t gsm[];
    const int64_t rb = gather_row_bytes<DT>(p.n);
    uint8_t* ssf = gsm + kGatherRows * rb;                              // [kGatherRows][kb]
    const bool wide = (reinterpret_cast<uintptr_t>(p.W) & 15) == 0;     // then every row is: n is a multiple of 16
    for (int64_t r0 = (int64_t)blockIdx.x * kGatherRows; r0 < p.rows; r0 += (int64_t)gridDim.x * kGatherRows) {
        const int nr = (int)(p.rows - r0 < kGatherRows ? p.rows - r0 : kGatherRows);
        __syncthreads();                                                // the last rows are read
        if (wide) {
            const uint4* src = reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(p.W) + r0 * rb);
            for (int i = threadIdx.x; i < (int)(nr * rb / 16); i += 256) reinterpret_cast<uint4*>(gsm)[i] = src[i];
        } else {
            for (int i = threadIdx.x; i < (int)(nr * p.n); i += 256) {
                if (DT == 0) reinterpret_cast<uint16_t*>(gsm)[i] = static_cast<const uint16_t*>(p.W)[r0 * p.n + i];
                else reinterpret_cast<float*>(gsm)[i] = static_cast<const float*>(p.W)[r0 * p.n + i];
            }
        }
        for (int i = threadIdx.x; i < (int)(nr * p.kb); i += 256) ssf[i] = p.sf[r0 * p.kb + i];
        __syncthreads();
        for (int64_t k = 4 * threadIdx.x; k < p.n; k += 4 * 256) {
            int c[4];
#pragma unroll
            for (int j = 0; j < 4; j++) c[j] = (int)checked_index(p.perm[k + j], p.n, p.status);
#pragma unroll
            for (int i = 0; i < kGatherRows; i++) {
                if (i >= nr) break;
                float v[4];
                uint32_t codes = 0;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    if (DT == 0) v[j] = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(gsm + i * rb)[c[j]] << 16);
                    else v[j] = reinterpret_cast<const float*>(gsm + i * rb)[c[j]];
                    const uint32_t code = ssf[i * p.kb + (c[j] >> shift)];
                    codes |= (code > 126 ? 0u : code) << (8 * j);       // 0x7F (NaN) and above: a zero scale
                }
                const int64_t at = (r0 + i) * p.n + k;
                const float4 q = make_float4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<float4*>(p.T + at) = q;
                *reinterpret_cast<float4*>(p.Wp + at) = q;
                *reinterpret_cast<uint32_t*>(p.sfp + at) = codes;
            }
        }
    }
}

// One super-panel of up to 256 columns (a multiple of 8): every column is
// quantized in order and its error fed to the later columns of the super-panel.
//
// A CTA takes 32 rows, one per lane, in every one of its 8 warps, and walks the
// super-panel in sub-panels of 64 columns, a group of 8 to a warp.  At step o of a
// sub-panel warp o walks its group alone -- the chain quantize -> error -> update
// never leaves the lane -- and publishes the 8 errors of its 32 rows; one barrier
// ends the step.  The later warps then apply these errors to their own groups by
// fp32 multiply-adds (U, the same for all lanes, was read into registers before
// the barrier), so the next walk starts after 32 packed operations.  Beside the
// walk every other warp applies published errors to its groups of the later
// sub-panels with mma.sync (K = 8, three TF32 products per term as the trailing
// GEMM), a group's 32 x 8 sums being two accumulator fragments: the last
// published errors to the next sub-panel, those of the sub-panel before to the
// ones after it.  A walking warp makes up the one step it missed when the
// sub-panel is done, and turns its next group's fragments into rows (through
// shared memory, 12-word rows).
//
// The error sums start from zero, those of 8 errors in the MMA and their running sum
// in fp32, and meet the target, which is many times larger, in one addition when its
// group is walked.  (An MMA does not round its sum to nearest: accumulating on the
// targets themselves put them 1.14e-6 from 64 bits at 4096 x 4096 bf16, this 1.3e-7.)
//
// Bound by the chain: 35 cycles of dependent arithmetic per column (52 with the
// rest of a column's instructions), and a barrier and the last group's update per
// 8 columns.  An mma.sync takes 8.5 cycles of its quarter of the SM and about 70
// until its result is there, so none of them is on the chain but two or three per
// sub-panel.  Splitting a row's columns over lanes instead (eight or sixteen
// threads per row, a shuffle per column, panels of 64 with a GEMM between them)
// repeats the quantize step once per row rather than once per 32 rows and was
// issue-bound at 520 cycles per column; applying all errors by multiply-adds on
// broadcast reads of U was bound by the shared-memory returns (a word per lane
// and multiply-add) at 260, all by mma.sync by its latency at 220.
//
// The upper triangle of the super-panel's U block is staged by one bulk copy per
// row (the wait for it is bounded: status bit 16, as the trailing GEMM's waits).
constexpr int kGroupCols = 8;
constexpr int kWalkWarps = 8;
constexpr int kWalkRows = 32;
constexpr int kWalkThreads = 32 * kWalkWarps;
constexpr int kSubCols = kGroupCols * kWalkWarps;                       // 64
constexpr int kSubs = kLdlqPanel / kSubCols;                            // 4
constexpr int kErrStride = 40;                                          // words per column of errors: conflict-free A fragments
constexpr int kErrSlot = kGroupCols * kErrStride;
constexpr int kTurnStride = 12;                                         // words per row of a group's targets
constexpr int kUWords = 8 * (3 * 264 + 4 * (232 + 200 + 168 + 136 + 104 + 72 + 40) + 8);   // see u_row
constexpr int kWalkSmem = (kUWords + 2 * kWalkWarps * kErrSlot + kWalkWarps * kWalkRows * kTurnStride + 128) * 4;

// The staged upper triangle of U: row 8 g + j holds columns 8 g .. 255, its pitch
// rounded up to 8 words modulo 32 (the rows of B fragments then lie in distinct
// banks): 264 words for g < 3, then 32 fewer every four groups.
__device__ __forceinline__ int u_pitch(int g) { return g < 3 ? 264 : 232 - 32 * ((g - 3) >> 2); }
__device__ __forceinline__ int u_row(int g) {                           // word offset of row 8 g
    if (g < 3) return 8 * 264 * g;
    const int m = (g - 3) >> 2;
    return 8 * (3 * 264 + 4 * (232 * m - 16 * m * (m - 1)) + ((g - 3) & 3) * (232 - 32 * m));
}

// Untiled bulk copy to shared memory (16-byte aligned, a multiple of 16 bytes), completion on bar.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Every warp arrives once per step, the walking one from its own branch.
__device__ __forceinline__ void step_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }

// tc::split_tf32 as bit patterns, lo not masked (the MMA reads its top 11 bits).
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
    hi = __float_as_uint(x) & 0xFFFFE000u;
    lo = __float_as_uint(__fsub_rn(x, __uint_as_float(hi))) + 0x1000u;
}
__device__ __forceinline__ void mma_16n8k8_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// UVEC: U is 16-byte aligned (its rows then are too: n is a multiple of 16).
template <bool UVEC>
__global__ void __launch_bounds__(kWalkThreads, 1) walk_kernel(LdlqParams p, int64_t s0, int span, float* Eh,
                                                               float* El) {
    extern __shared__ __align__(16) float dsm[];
    __shared__ __align__(8) uint64_t s_ubar;
    float* ut = dsm;                                              // U, see u_row
    float* es = dsm + kUWords;                                    // [2][kWalkWarps][8][kErrStride]: two sub-panels' errors
    float* turn = es + 2 * kWalkWarps * kErrSlot;                 // [kWalkWarps][kWalkRows][kTurnStride]
    float* rtab = turn + kWalkWarps * kWalkRows * kTurnStride;    // [128] fl(1/v) of each code, 0 for a zero scale
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ng = span / kGroupCols;
    const int wc = warp * kGroupCols;                             // this warp's columns within a sub-panel

    const int64_t row0 = (int64_t)blockIdx.x * kWalkRows, last = p.rows - 1;
    const int64_t r = row0 + lane;
    const bool active = r <= last;
    const int64_t rbase = (active ? r : last) * p.n + s0;         // lanes past the last row repeat it and store nothing
    float* tw = turn + warp * kWalkRows * kTurnStride;
    // the sums of errors on the row's targets in the group to be walked, packed pairs
    u64 t[4] = {0ull, 0ull, 0ull, 0ull};
    auto set_rows = [&](const float* src) {
        const float4 a = *reinterpret_cast<const float4*>(src);
        const float4 b = *reinterpret_cast<const float4*>(src + 4);
        t[0] = pack2(a.x, a.y);
        t[1] = pack2(a.z, a.w);
        t[2] = pack2(b.x, b.y);
        t[3] = pack2(b.z, b.w);
    };
    // operands of the warp's next walk: original weights, scale codes and, written by the
    // update before this grid, the targets without the super-panel's own errors
    float4 wa, wb, ta, tb;
    uint2 cd;
    auto fetch = [&](int q) {
        const int c = q * kSubCols + wc;
        if (c < span) {
            wa = *reinterpret_cast<const float4*>(p.Wp + rbase + c);
            wb = *reinterpret_cast<const float4*>(p.Wp + rbase + c + 4);
            cd = *reinterpret_cast<const uint2*>(p.sfp + rbase + c);
        }
    };
    auto fetch_targets = [&](int q) {
        const int c = q * kSubCols + wc;
        if (c < span) {
            ta = *reinterpret_cast<const float4*>(p.T + rbase + c);
            tb = *reinterpret_cast<const float4*>(p.T + rbase + c + 4);
        }
    };
    fetch(0);
    // row i of the super-panel's U from column 8 (i / 8) on: one bulk copy per row,
    // or 4-byte copies where U is not 16-byte aligned
    const uint32_t ubar = tc::smem_u32(&s_ubar);
    if (UVEC) {
        if (tid == 0) {
            tc::mbar_init(ubar, 1 + (p.starve & kStarveWalk));
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            tc::mbar_expect_tx(ubar, (uint32_t)(32 * kGroupCols * ng * (ng + 1) / 2));   // 8 rows of 32 (ng - g) bytes per group
        }
        __syncthreads();
        if (tid < span) {
            const int g = tid >> 3;
            bulk_load(tc::smem_u32(ut + u_row(g) + (tid & 7) * u_pitch(g)), p.U + (s0 + tid) * p.n + s0 + 8 * g,
                      (uint32_t)(span - 8 * g) * 4, ubar);
        }
    } else {
        for (int i = warp; i < span; i += kWalkWarps) {
            const int g = i >> 3;
            const float* src = p.U + (s0 + i) * p.n + s0;
            float* dst = ut + u_row(g) + (i & 7) * u_pitch(g) - 8 * g;
            for (int c = 8 * g + lane; c < span; c += 32) cp_async4(dst + c, src + c, true);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const float S = __ldg(p.S);
    const float Einv = __frcp_rn(S);
    const bool usable = (S > 0.0f) && isfinite(S) && isfinite(Einv);
    const float E = usable ? Einv : 1.0f;
    const float Sq = usable ? S : 0.0f;               // an unusable S reconstructs zeros (q is a signed zero then)
    // an unusable S or a zero code: r = 0 turns every target into a signed zero
    if (tid < 128)
        rtab[tid] = (usable && tid >= 1 && tid <= 126) ? __frcp_rn(f16bits_to_f32(e4m3_to_f16bits((uint32_t)tid))) : 0.0f;

    // all of the above is older than the update of these columns, which the targets come
    // from and the only grid this one may start before the end of
    grid_dependency_wait();
    fetch_targets(0);
    // the errors' sums for this warp's groups in sub-panels 1.. as accumulator fragments:
    // rows 16 m + lane / 4 (+ 8), columns 2 (lane % 4), + 1
    float acc[kSubs][2][4] = {};
    float rs[kGroupCols];
    uint16_t vh[kGroupCols];
    auto scales = [&]() {
#pragma unroll
        for (int j = 0; j < kGroupCols; j++) {
            const uint32_t code = ((j < 4 ? cd.x : cd.y) >> (8 * (j & 3))) & 0x7Fu;
            rs[j] = rtab[code];
            vh[j] = e4m3_to_f16bits(code);
        }
    };
    // the errors of group g as A fragments (row = row of the CTA, k = column of the group)
    auto load_errors = [&](uint32_t (&ah)[2][4], uint32_t (&al)[2][4], int g) {
        const float* e = es + (g & (2 * kWalkWarps - 1)) * kErrSlot + (lane & 3) * kErrStride + (lane >> 2);
#pragma unroll
        for (int m = 0; m < 2; m++) {
            split_tf32(e[16 * m], ah[m][0], al[m][0]);
            split_tf32(e[16 * m + 8], ah[m][1], al[m][1]);
            split_tf32(e[16 * m + 4 * kErrStride], ah[m][2], al[m][2]);
            split_tf32(e[16 * m + 4 * kErrStride + 8], ah[m][3], al[m][3]);
        }
    };
    // the rows of group g of U as a B fragment, for the columns of this warp's group in sub-panel q
    auto load_u = [&](uint32_t (&bh)[2], uint32_t (&bl)[2], int g, int q) {
        const int up = u_pitch(g);
        const float* u = ut + u_row(g) + (lane & 3) * up + (lane >> 2) + q * kSubCols + wc - 8 * g;
        split_tf32(u[0], bh[0], bl[0]);
        split_tf32(u[4 * up], bh[1], bl[1]);
    };
    auto products = [&](float (&c)[2][4], const uint32_t (&ah)[2][4], const uint32_t (&al)[2][4], const uint32_t (&bh)[2],
                        const uint32_t (&bl)[2]) {
        float d[2][4] = {};
#pragma unroll
        for (int m = 0; m < 2; m++) mma_16n8k8_tf32(d[m], al[m], bh);
#pragma unroll
        for (int m = 0; m < 2; m++) mma_16n8k8_tf32(d[m], ah[m], bl);
#pragma unroll
        for (int m = 0; m < 2; m++) mma_16n8k8_tf32(d[m], ah[m], bh);
#pragma unroll
        for (int m = 0; m < 2; m++)
#pragma unroll
            for (int i = 0; i < 4; i++) c[m][i] = __fadd_rn(c[m][i], d[m][i]);
    };

    bool staged = true;
    if (UVEC) staged = tc::mbar_wait(ubar, 0);
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (__syncthreads_or(!staged)) {
        // U never arrived: report it, give the copies a second bounded wait (they must not
        // land in a later CTA's shared memory) and leave zero errors and zero codes, so
        // that nothing stale from the workspace reaches the updates or the result
        if (tid == 0 && p.status) atomicOr(p.status, tc::kStatusTimeout);
        if (UVEC) (void)tc::mbar_wait(ubar, 0);
        const int nr = (int)min((int64_t)kWalkRows, p.rows - row0);
        for (int i = tid; i < nr * span; i += kWalkThreads) {
            const int64_t rr = row0 + i / span;
            const int c = i % span;
            Eh[rr * kLdlqPanel + c] = 0.0f;
            if (El) El[rr * kLdlqPanel + c] = 0.0f;
            p.qb[rr * p.n + s0 + c] = 0;
        }
        return;
    }
    scales();
#pragma unroll
    for (int q = 0; q < kSubs; q++) {
        const int nq = min(kWalkWarps, ng - q * kWalkWarps);      // groups of this sub-panel
        if (nq <= 0) break;
        // acc[q + 1] += errors of group g of this sub-panel
        auto near = [&](int o) {
            if ((q + 1) * kSubCols + wc < span) {
                uint32_t ah[2][4], al[2][4], bh[2], bl[2];
                load_u(bh, bl, q * kWalkWarps + o, q + 1);
                load_errors(ah, al, q * kWalkWarps + o);
                products(acc[q + 1 < kSubs ? q + 1 : 0], ah, al, bh, bl);
            }
        };
        // acc[q + 1 ..] += errors of group o of the sub-panel before
        auto far = [&](int o) {
            if (q > 0 && (q + 1) * kSubCols + wc < span) {
                uint32_t ah[2][4], al[2][4], bh[kSubs][2], bl[kSubs][2];
#pragma unroll
                for (int q2 = q + 1; q2 < kSubs; q2++)
                    if (q2 * kSubCols + wc < span) load_u(bh[q2], bl[q2], (q - 1) * kWalkWarps + o, q2);
                load_errors(ah, al, (q - 1) * kWalkWarps + o);
#pragma unroll
                for (int q2 = q + 1; q2 < kSubs; q2++)
                    if (q2 * kSubCols + wc < span) products(acc[q2], ah, al, bh[q2], bl[q2]);
            }
        };
        float4 un[2 * kGroupCols];                     // U: rows of the group being walked, columns of this warp's
#pragma unroll 1
        for (int o = 0; o < nq; o++) {                 // errors up to group o - 1 are published
            const int g = q * kWalkWarps + o;
            if (o > 0 && warp >= o && warp < nq) {
                const float* ep = es + ((g - 1) & (2 * kWalkWarps - 1)) * kErrSlot + lane;
#pragma unroll
                for (int j = 0; j < kGroupCols; j++) {
                    const float ej = ep[j * kErrStride];
                    const u64 e2 = pack2(ej, ej);
                    t[0] = fma2(e2, pack2(un[2 * j].x, un[2 * j].y), t[0]);
                    t[1] = fma2(e2, pack2(un[2 * j].z, un[2 * j].w), t[1]);
                    t[2] = fma2(e2, pack2(un[2 * j + 1].x, un[2 * j + 1].y), t[2]);
                    t[3] = fma2(e2, pack2(un[2 * j + 1].z, un[2 * j + 1].w), t[3]);
                }
            }
            if (warp == o) {
                float tt[8], ev[8];
                const float tw8[8] = {ta.x, ta.y, ta.z, ta.w, tb.x, tb.y, tb.z, tb.w};
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    unpack2(t[h], tt[2 * h], tt[2 * h + 1]);
                    tt[2 * h] = __fadd_rn(tw8[2 * h], tt[2 * h]);
                    tt[2 * h + 1] = __fadd_rn(tw8[2 * h + 1], tt[2 * h + 1]);
                }
                const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
                float* e = es + (g & (2 * kWalkWarps - 1)) * kErrSlot + lane;
                const float* ud = ut + u_row(g);
                const int dp = u_pitch(g);
                uint32_t packed[2] = {0u, 0u};
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    // What = fl(fl(q v) S) with q = RNE_E2M1(fl(y r)), y = fl(t E); q v is
                    // exact, formed by one mixed fma with a +0 addend (a zero q gives +0)
                    const float y = __fmul_rn(tt[j], E);
                    uint32_t nib;
                    float qv;
                    asm("{\n\t.reg .b8 b;\n\t.reg .b32 h2;\n\t.reg .b16 ql, qh;\n\t"
                        "cvt.rn.satfinite.e2m1x2.f32 b, %4, %2;\n\t"
                        "cvt.rn.f16x2.e2m1x2 h2, b;\n\tmov.b32 {ql, qh}, h2;\n\t"
                        "fma.rn.f32.f16 %0, ql, %3, %4;\n\t"
                        "cvt.u32.u8 %1, b;\n\t}"
                        : "=f"(qv), "=r"(nib) : "f"(__fmul_rn(y, rs[j])), "h"(vh[j]), "f"(0.0f));
                    ev[j] = __fsub_rn(w[j], __fmul_rn(qv, Sq));
                    if (j < 7) {
                        const float4 u0 = *reinterpret_cast<const float4*>(ud + j * dp);
                        const float4 u1 = *reinterpret_cast<const float4*>(ud + j * dp + 4);
                        const float uv[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
                        for (int c = j + 1; c < 8; c++) tt[c] = __fmaf_rn(ev[j], uv[c], tt[c]);
                    }
                    e[j * kErrStride] = ev[j];
                    // an exactly zero target takes the +0 code
                    packed[j >> 2] |= (y == 0.0f ? 0u : nib & 0xFu) << (8 * (j & 3));
                }
                step_barrier();                        // publish before the global stores
                if (active) {
                    // the trailing update's operands, [rows, kLdlqPanel]: TF32 halves, or the error itself
                    const int64_t at = r * kLdlqPanel + g * kGroupCols;
#pragma unroll
                    for (int j = 0; j < 8; j += 4) {
                        float4 h = make_float4(ev[j], ev[j + 1], ev[j + 2], ev[j + 3]), l;
                        if (El) {
                            tc::split4(h, h, l);
                            *reinterpret_cast<float4*>(El + at + j) = l;
                        }
                        *reinterpret_cast<float4*>(Eh + at + j) = h;
                    }
                    *reinterpret_cast<uint2*>(p.qb + rbase + g * kGroupCols) = make_uint2(packed[0], packed[1]);
                }
                fetch(q + 1);
                fetch_targets(q + 1);
                continue;
            }
            if (warp > o && warp < nq) {
                const float* u = ut + u_row(g) + (warp - o) * kGroupCols;
                const int up = u_pitch(g);
#pragma unroll
                for (int j = 0; j < 2 * kGroupCols; j++) un[j] = *reinterpret_cast<const float4*>(u + (j >> 1) * up + 4 * (j & 1));
            }
            if (o > 0) near(o - 1);
            far(o);
            step_barrier();
        }
        // here sub-panel q + 1 exists only if this one is full; its rows need the last
        // group's errors, and what this warp missed while it walked
        if (q + 1 < kSubs && (q + 1) * kSubCols + wc < span) {
            far(warp);
            if (warp > 0) near(warp - 1);
            near(kWalkWarps - 1);
            const float (&c)[2][4] = acc[q + 1 < kSubs ? q + 1 : 0];
#pragma unroll
            for (int m = 0; m < 2; m++)
#pragma unroll
                for (int h = 0; h < 2; h++)
                    *reinterpret_cast<float2*>(tw + (16 * m + 8 * h + (lane >> 2)) * kTurnStride + 2 * (lane & 3)) =
                        make_float2(c[m][2 * h], c[m][2 * h + 1]);
            __syncwarp();
            set_rows(tw + lane * kTurnStride);
            __syncwarp();
            scales();
        }
    }
}

// The TF32 halves of U's rows s0 .. s0 + 255, columns c0 .. n - 1, transposed: Bh, Bl
// [n - c0, kLdlqPanel], the trailing update's second operand.  32 x 32 tiles.
__global__ void __launch_bounds__(256) split_u_kernel(const float* U, int64_t n, int64_t s0, int64_t c0, float* Bh, float* Bl) {
    __shared__ float t[32][33];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int64_t c = c0 + (int64_t)blockIdx.x * 32;
    const int k = (int)blockIdx.y * 32;
#pragma unroll
    for (int i = 0; i < 32; i += 8) t[y + i][x] = c + x < n ? U[(s0 + k + y + i) * n + c + x] : 0.0f;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 32; i += 8)
        if (c + y + i < n) {
            float h, l;
            tc::split_tf32(t[x][y + i], h, l);
            const int64_t at = (c + y + i - c0) * kLdlqPanel + k + x;
            Bh[at] = h;
            Bl[at] = l;
        }
}

// codes[r][c/2]: nibble of original column c from qb[r][inv[c]]; rows too long for pack_kernel.
__global__ void __launch_bounds__(256) pack_long_kernel(const uint8_t* qb, const int32_t* inv, int64_t rows, int64_t n,
                                                        uint8_t* codes, int* status) {
    const int64_t half = n / 2;
    for (int64_t r = blockIdx.x; r < rows; r += gridDim.x)
        for (int64_t c2 = threadIdx.x; c2 < half; c2 += blockDim.x) {
            const uint8_t lo = qb[r * n + checked_index(inv[2 * c2], n, status)];
            const uint8_t hi = qb[r * n + checked_index(inv[2 * c2 + 1], n, status)];
            codes[r * half + c2] = (uint8_t)((lo & 0xF) | ((hi & 0xF) << 4));
        }
}

// The same through shared memory, kGatherRows rows at a time (23 us straight from
// global memory at 4096 x 4096).
__global__ void __launch_bounds__(256) pack_kernel(const uint8_t* qb, const int32_t* inv, int64_t rows, int64_t n,
                                                   uint8_t* codes, int* status) {
    extern __shared__ __align__(16) uint8_t gsm[];
    const bool words = (reinterpret_cast<uintptr_t>(codes) & 3) == 0;   // then every row is: n / 2 is a multiple of 8
    for (int64_t r0 = (int64_t)blockIdx.x * kGatherRows; r0 < rows; r0 += (int64_t)gridDim.x * kGatherRows) {
        const int nr = (int)(rows - r0 < kGatherRows ? rows - r0 : kGatherRows);
        __syncthreads();                                                // the last rows are read
        for (int i = threadIdx.x; i < (int)(nr * n / 16); i += 256)
            reinterpret_cast<uint4*>(gsm)[i] = reinterpret_cast<const uint4*>(qb + r0 * n)[i];
        __syncthreads();
        for (int64_t c = 8 * threadIdx.x; c < n; c += 8 * 256) {
            int k[8];
#pragma unroll
            for (int j = 0; j < 8; j++) k[j] = (int)checked_index(inv[c + j], n, status);
#pragma unroll
            for (int i = 0; i < kGatherRows; i++) {
                if (i >= nr) break;
                uint32_t w = 0;
#pragma unroll
                for (int j = 0; j < 8; j++) w |= (uint32_t)(gsm[i * n + k[j]] & 0xFu) << (4 * j);
                uint8_t* d = codes + ((r0 + i) * n + c) / 2;
                if (words) *reinterpret_cast<uint32_t*>(d) = w;
                else
                    for (int b = 0; b < 4; b++) d[b] = (uint8_t)(w >> (8 * b));
            }
        }
    }
}

constexpr int64_t kGatherSmemMax = 200 * 1024;     // dynamic shared memory of the two kernels above

}  // namespace

// diag(H), lambda, Linv; with split, Xtop and the solved panel's TF32 halves.
size_t ldlq_prepare_workspace(int64_t n, bool split) {
    const size_t least = (size_t)((n * 4 + 255) / 256 * 256) + 256 + (size_t)kP * kP * 4;
    return split ? least + (size_t)kP * kP * 4 + (size_t)2 * n * kP * 4 : least;
}

// Stream and events of the factorization's look-ahead, one set per device,
// created on the first prepare call on that device and kept for the process.
// The critical chain (diagonal factor, panel solve, next block column) runs on
// `crit`, created with the device's highest priority so its CTAs are placed
// before the pending tiles of the bulk update on the caller's stream.  The
// mutex serialises enqueueing, so the record/wait pairs of two concurrent calls
// cannot interleave.
struct LookAhead {
    cudaStream_t crit = nullptr;
    cudaEvent_t fork = nullptr, panel_done = nullptr, rest_done = nullptr, crit_done = nullptr, split_done = nullptr;
};

cudaError_t lookahead_for_current_device(LookAhead** out, std::unique_lock<std::mutex>* lock) {
    static std::mutex mu;
    static LookAhead state[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    *lock = std::unique_lock<std::mutex>(mu);
    LookAhead& la = state[dev];
    if (!la.crit) {
        int least = 0, greatest = 0;
        if ((e = cudaDeviceGetStreamPriorityRange(&least, &greatest)) != cudaSuccess) return e;
        if ((e = cudaStreamCreateWithPriority(&la.crit, cudaStreamNonBlocking, greatest)) != cudaSuccess) return e;
        cudaEvent_t* evs[5] = {&la.fork, &la.panel_done, &la.rest_done, &la.crit_done, &la.split_done};
        for (cudaEvent_t* ev : evs)
            if ((e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) return e;
    }
    *out = &la;
    return cudaSuccess;
}

cudaError_t launch_ldlq_prepare(const float* H, int64_t n, float damp, int32_t* perm, float* U, float* D,
                                int* status, void* ws, bool split, int sms, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    char* w = static_cast<char*>(ws);
    float* d = reinterpret_cast<float*>(w);
    float* lam = reinterpret_cast<float*>(w + (n * 4 + 255) / 256 * 256);
    float* Linv = lam + 64;
    const bool vec = n % 4 == 0 && (reinterpret_cast<uintptr_t>(U) & 15) == 0;
    float* Xw = split ? Linv + kP * kP : nullptr;
    float* Lh = split && vec ? Xw + kP * kP : nullptr;          // the solved panel's TF32 halves, [n, 64] each
    float* Ll = Lh ? Lh + n * kP : nullptr;
    diag_kernel<<<1, 1024, 0, s>>>(H, n, damp, d, lam, status);
    rank_kernel<<<(unsigned)((n + 7) / 8), 256, 0, s>>>(d, n, perm);
    const unsigned rg = (unsigned)imin64(n, (int64_t)sms * 8);
    gather_h_kernel<<<rg, 256, 0, s>>>(H, n, perm, lam, U);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // Look-ahead: the trailing update of panel k is split into the next panel's
    // block column (on the high-priority stream, in the kernel that solves the
    // panel, with the diagonal factors) and the rest (on `s`, overlapping them).
    // The two updates of one block column from different panels are ordered by events.
    LookAhead* la = nullptr;
    std::unique_lock<std::mutex> lock;
    e = lookahead_for_current_device(&la, &lock);
    if (e != cudaSuccess) return e;
    cudaStream_t c = la->crit;
    if ((e = cudaEventRecord(la->fork, s)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(c, la->fork, 0)) != cudaSuccess) return e;
    constexpr int kPotrfSmem = 2 * kP * kPad * 4;
    static_assert(kPotrfSmem <= 48 * 1024, "no shared-memory opt-in");
    const auto panel = vec ? panel_kernel<true> : panel_kernel<false>;
    if ((e = cudaFuncSetAttribute(panel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPanelSmem)) != cudaSuccess) return e;
    bool have_rest = false;              // rest_done recorded by this call (waits stay inside a capture)
    for (int64_t k0 = 0; k0 < n; k0 += kP) {
        const int nb = (int)imin64(kP, n - k0);
        // without room of its own Xtop lies transposed above the diagonal, right of the
        // diagonal block, where nothing else is kept until the factor is turned over
        float* Xtop = Xw ? Xw : U + k0 * n + k0 + nb;
        const int64_t xr = Xw ? kP : 1, xc = Xw ? 1 : n;
        // scheduled while the last panel kernel runs, ordered after its writes
        if ((e = launch_dependent_smem(potrf_kernel, 1, kPotrfThreads, kPotrfSmem, c, U, n, k0, nb, Linv, Xtop, xr,
                                       xc, status)) != cudaSuccess)
            return e;
        const int64_t rest = n - k0 - nb;
        if (rest > 0) {
            const int64_t nb2 = imin64(kP, rest);      // width of the next panel
            // the next block column also took the previous panel's rest update
            if (have_rest && (e = cudaStreamWaitEvent(c, la->rest_done, 0)) != cudaSuccess) return e;
            panel<<<(unsigned)((rest + kPanelRows - 1) / kPanelRows), 128, kPanelSmem, c>>>(U, n, k0, Linv, Xtop, xr, xc, Lh,
                                                                                                Ll);
            if (rest > nb2) {
                const int64_t i0 = k0 + nb + nb2, m = rest - nb2;
                float* P = U + i0 * n + k0;            // the solved panel's rows past the next block column
                if ((e = cudaEventRecord(la->panel_done, c)) != cudaSuccess) return e;
                if ((e = cudaStreamWaitEvent(s, la->panel_done, 0)) != cudaSuccess) return e;
                e = cudaErrorNotSupported;
                if (Lh) {
                    const tc::Split L{Lh + i0 * kP, Ll + i0 * kP, kP};
                    e = tc::launch_gemm<true>(U + i0 * n + i0, n, L, L, m, m, nb, -1.0f, status, 0, sms, s);
                }
                if (e == cudaErrorNotSupported)
                    e = launch_gemm<true, true>(U + i0 * n + i0, n, P, n, P, n, m, m, nb, -1.0f, s);
                if (e != cudaSuccess) return e;
                if ((e = cudaEventRecord(la->rest_done, s)) != cudaSuccess) return e;
                have_rest = true;
            }
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if ((e = cudaEventRecord(la->crit_done, c)) != cudaSuccess) return e;          // join
    if ((e = cudaStreamWaitEvent(s, la->crit_done, 0)) != cudaSuccess) return e;
    lock.unlock();
    diag_d_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(U, n, D);
    flip_kernel<<<rg, 256, 0, s>>>(U, n);
    zero_diag_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(U, n);
    return cudaGetLastError();
}

// Workspace: T and Wp [rows, n] f32, qb and sfp [rows, n] bytes, inv [n], and, twice
// (alternating between super-panels), a super-panel's errors [rows, kLdlqPanel], or with
// split the TF32 halves of them and of its rows of U [n, kLdlqPanel].
size_t ldlq_quantize_workspace(int64_t rows, int64_t n, bool split) {
    auto up = [](int64_t b) { return (b + 255) / 256 * 256; };
    const int64_t ep = up((int64_t)kLdlqPanel * rows * 4), up4 = up((int64_t)kLdlqPanel * n * 4);
    return (size_t)(2 * up(rows * n * 4) + 2 * up(rows * n) + (split ? 4 * ep + 4 * up4 : 2 * ep) + up(n * 4));
}

// Columns in super-panels of kLdlqPanel (256), each walked by walk_kernel; after
// the super-panel, GEMMs with K = 256 update every later column, so the targets
// are read and written once per 256 columns.  Look-ahead: that update
// is split into the next super-panel's columns, which run with its panel walks
// on the high-priority stream, and the rest, which runs on `s` concurrently
// with them.  Before the rest of super-panel k, `s` also transposes and splits the rows
// of U that super-panel k + 1 will need.  Without the workspace for that (split false)
// or a driver with tensor maps, the updates run on the FP32 pipe.
cudaError_t launch_ldlq_quantize(LdlqParams p, int dtype, uint8_t* codes, void* ws, bool split, int sms,
                                 cudaStream_t s) {
    if (p.rows <= 0 || p.n <= 0) return cudaSuccess;
    if (tc::encode_fn() == nullptr) split = false;
    auto up = [](int64_t b) { return (b + 255) / 256 * 256; };
    char* w = static_cast<char*>(ws);
    const int64_t mat4 = up(p.rows * p.n * 4), mat1 = up(p.rows * p.n);
    p.T = reinterpret_cast<float*>(w);
    p.Wp = reinterpret_cast<float*>(w + mat4);
    p.qb = reinterpret_cast<uint8_t*>(w + 2 * mat4);
    p.sfp = reinterpret_cast<uint8_t*>(w + 2 * mat4 + mat1);
    const int64_t ep = up((int64_t)kLdlqPanel * p.rows * 4), up4 = up((int64_t)kLdlqPanel * p.n * 4);
    char* q = w + 2 * mat4 + 2 * mat1;
    tc::Split Es[2], Us[2];                        // ld = kLdlqPanel; without split hi is the whole error
    for (int i = 0; i < 2; i++) {
        Es[i] = {reinterpret_cast<float*>(q), split ? reinterpret_cast<float*>(q + ep) : nullptr, kLdlqPanel};
        q += split ? 2 * ep : ep;
        if (split) {
            Us[i] = {reinterpret_cast<float*>(q), reinterpret_cast<float*>(q + up4), kLdlqPanel};
            q += 2 * up4;
        }
    }
    int32_t* inv = reinterpret_cast<int32_t*>(q);
    cudaError_t e = cudaMemsetAsync(inv, 0, (size_t)p.n * 4, s);
    if (e != cudaSuccess) return e;
    invperm_kernel<<<(unsigned)((p.n + 255) / 256), 256, 0, s>>>(p.perm, p.n, inv, p.status);
    const unsigned rg = (unsigned)imin64(p.rows, (int64_t)sms * 8);
    const unsigned rg4 = (unsigned)imin64((p.rows + kGatherRows - 1) / kGatherRows, (int64_t)sms * 8);
    const int64_t gsmem = kGatherRows * ((dtype == 0 ? gather_row_bytes<0>(p.n) : gather_row_bytes<1>(p.n)) + p.kb);
    const int shift = p.block == 16 ? 4 : p.block == 32 ? 5 : 6;
    if (gsmem > kGatherSmemMax) {
        if (dtype == 0) gather_w_long_kernel<0><<<rg, 256, 0, s>>>(p);
        else gather_w_long_kernel<1><<<rg, 256, 0, s>>>(p);
    } else {
        const auto gather = dtype == 0 ? gather_w_kernel<0> : gather_w_kernel<1>;
        if (gsmem > 48 * 1024 &&
            (e = cudaFuncSetAttribute(gather, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGatherSmemMax)) != cudaSuccess)
            return e;
        gather<<<rg4, 256, (size_t)gsmem, s>>>(p, shift);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const bool uvec = (reinterpret_cast<uintptr_t>(p.U) & 15) == 0;
    const auto walk = uvec ? walk_kernel<true> : walk_kernel<false>;
    static std::atomic<bool> attr_set[64];        // per device: the shared-memory opt-in is done
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute(walk_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWalkSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(walk_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWalkSmem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_release);
    }
    const unsigned wg = (unsigned)((p.rows + kWalkRows - 1) / kWalkRows);
    LookAhead* la = nullptr;
    std::unique_lock<std::mutex> lock;
    e = lookahead_for_current_device(&la, &lock);
    if (e != cudaSuccess) return e;
    cudaStream_t c = la->crit;
    if ((e = cudaEventRecord(la->fork, s)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(c, la->fork, 0)) != cudaSuccess) return e;
    bool have_rest = false;              // rest_done recorded by this call (waits stay inside a capture)
    // the second operand of super-panel s0's trailing updates
    auto split_u = [&](int64_t s0, int i) {
        const int64_t c0 = s0 + kLdlqPanel;
        if (!split || c0 >= p.n) return cudaSuccess;
        split_u_kernel<<<dim3((unsigned)((p.n - c0 + 31) / 32), kLdlqPanel / 32), 256, 0, s>>>(
            p.U, p.n, s0, c0, const_cast<float*>(Us[i].hi), const_cast<float*>(Us[i].lo));
        const cudaError_t r = cudaGetLastError();
        return r != cudaSuccess ? r : cudaEventRecord(la->split_done, s);
    };
    // T[:, c0 + d ..] += the errors of super-panel s0 x U, `cols` columns from column d of its trailing ones
    auto update = [&](int64_t s0, int i, int64_t d, int64_t cols, cudaStream_t st) {
        float* C = p.T + s0 + kLdlqPanel + d;
        if (!split)
            return launch_gemm<false, false>(C, p.n, Es[i].hi, kLdlqPanel, p.U + s0 * p.n + s0 + kLdlqPanel + d, p.n,
                                             p.rows, cols, kLdlqPanel, 1.0f, st);
        const tc::Split B{Us[i].hi + d * kLdlqPanel, Us[i].lo + d * kLdlqPanel, kLdlqPanel};
        return tc::launch_gemm<false>(C, p.n, Es[i], B, p.rows, cols, kLdlqPanel, 1.0f, p.status,
                                      (p.starve & kStarveUpdate) != 0, sms, st);
    };
    if ((e = split_u(0, 0)) != cudaSuccess) return e;
    // The walk and the update of its columns (one CTA per SM both) fit the GPU together:
    // then the walk is scheduled beside the update and stages U, the weights and the
    // scales meanwhile (1024 x 4096: 0.601 -> 0.538 ms).  Otherwise its waiting CTAs
    // would only keep SMs from the rest of the update (4096 x 4096: 0.925 -> 0.941 ms).
    // The first walk has no update before it: it goes out the ordinary way, ordered after
    // the gather that writes the weights and scales it reads before its wait.
    const bool early = wg + ((p.rows + 127) / 128) * (kLdlqPanel / 128) <= sms;
    int sp = 0;
    for (int64_t s0 = 0; s0 < p.n; s0 += kLdlqPanel, sp ^= 1) {
        const int64_t span = imin64(kLdlqPanel, p.n - s0);
        float *eh = const_cast<float*>(Es[sp].hi), *el = const_cast<float*>(Es[sp].lo);
        if (early && s0 > 0) {
            e = launch_dependent_smem(walk, wg, kWalkThreads, kWalkSmem, c, p, s0, (int)span, eh, el);
        } else {
            walk<<<wg, kWalkThreads, kWalkSmem, c>>>(p, s0, (int)span, eh, el);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return e;
        const int64_t rest = p.n - (s0 + span);
        if (rest > 0) {
            const int64_t next = imin64(kLdlqPanel, rest);
            if ((e = cudaEventRecord(la->panel_done, c)) != cudaSuccess) return e;
            if (split && (e = cudaStreamWaitEvent(c, la->split_done, 0)) != cudaSuccess) return e;
            // the next super-panel's columns also took the previous rest update, and that
            // update read the buffers the next super-panel overwrites
            if (have_rest && (e = cudaStreamWaitEvent(c, la->rest_done, 0)) != cudaSuccess) return e;
            if ((e = update(s0, sp, 0, next, c)) != cudaSuccess) return e;
            if ((e = cudaStreamWaitEvent(s, la->panel_done, 0)) != cudaSuccess) return e;
            if ((e = split_u(s0 + kLdlqPanel, sp ^ 1)) != cudaSuccess) return e;
            if (rest > next) {
                if ((e = update(s0, sp, next, rest - next, s)) != cudaSuccess) return e;
                if ((e = cudaEventRecord(la->rest_done, s)) != cudaSuccess) return e;
                have_rest = true;
            }
        }
    }
    if ((e = cudaEventRecord(la->crit_done, c)) != cudaSuccess) return e;          // join
    if ((e = cudaStreamWaitEvent(s, la->crit_done, 0)) != cudaSuccess) return e;
    lock.unlock();
    const int64_t psmem = kGatherRows * p.n;
    if (psmem > kGatherSmemMax) {
        pack_long_kernel<<<rg, 256, 0, s>>>(p.qb, inv, p.rows, p.n, codes, p.status);
    } else {
        if (psmem > 48 * 1024 && (e = cudaFuncSetAttribute(pack_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           (int)kGatherSmemMax)) != cudaSuccess)
            return e;
        pack_kernel<<<rg4, 256, (size_t)psmem, s>>>(p.qb, inv, p.rows, p.n, codes, p.status);
    }
    return cudaGetLastError();
}

}  // namespace nvfp4
