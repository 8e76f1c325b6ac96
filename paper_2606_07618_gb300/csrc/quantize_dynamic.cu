// Sweeps with a per-call global scale (the dynamic-activation path).  Tensors of at
// most 4096 segments (a decode batch) with a default window: one launch of one
// thread-block cluster.  Larger ones, and explicit windows: the global scale's
// reduction, then the sweep as its programmatic dependent, whose CTAs fold the
// partial maxima themselves: two ordinary launches, no counter to reset, no wait in
// device code.
#include "quantize_kernel.cuh"

namespace nvfp4 {

// A small tensor in one cluster of up to 16 CTAs, a segment per thread: the input is
// read once and stays in registers while the CTAs exchange their maxima through
// distributed shared memory, then it is swept.  One ordinary launch: no memset, no
// barrier in global memory, no second read.  Bound by latency (the launch, one trip
// to memory, two cluster barriers and one segment's sweep).  Up to 4096 segments
// because 16 CTAs is the largest cluster; more threads per CTA would queue the
// sweeps behind each other on 16 of the 152 SMs.
constexpr int kClusterCtas = 16, kClusterThreads = 256;

template <int DT, int METHOD, int OBJ, int BLOCK>
__global__ void __launch_bounds__(kClusterThreads) quantize_cluster_kernel(QuantParams p) {
    __shared__ Cand tab[kTabN];
    __shared__ uint2 slot[kClusterCtas];             // every CTA's maximum and non-finite flag
    __shared__ uint32_t sm[kClusterThreads / 32], sb[kClusterThreads / 32];
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t g = (int64_t)blockIdx.x * kClusterThreads + tid;
    const bool valid = g < p.nseg;
    Raw cur = {};
    if (valid) load_raw<DT, true>(p.x, g, wide_input(p.x), cur);
    build_table(tab);
    // max |x| with NaN skipped, and whether anything is not finite (as dynamic_scale)
    float m = 0.0f;
    int bad = 0;
    const uint4 v[4] = {cur.a, cur.b, cur.c, cur.d};
#pragma unroll
    for (int q = 0; q < (DT == 0 ? 2 : 4); q++) {
        const uint32_t w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const float a = DT == 0 ? bf16lo(w[j]) : __uint_as_float(w[j]);
            const float b = DT == 0 ? bf16hi(w[j]) : 0.0f;
            bad |= (!isfinite(a)) | (!isfinite(b));
            m = fmaxf(m, fmaxf(fabsf(a), fabsf(b)));
        }
    }
    const uint32_t mw = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    const uint32_t bw = __reduce_or_sync(0xffffffffu, (unsigned)bad);
    if (lane == 0) {
        sm[warp] = mw;
        sb[warp] = bw;
    }
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // every CTA has started
    if (tid < (int)gridDim.x) {                      // this CTA's maximum into CTA tid's slot
        uint32_t a = 0, b = 0;
#pragma unroll
        for (int i = 0; i < kClusterThreads / 32; i++) {
            a = max(a, sm[i]);
            b |= sb[i];
        }
        uint32_t dst;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                     : "=r"(dst)
                     : "r"((uint32_t)__cvta_generic_to_shared(&slot[blockIdx.x])), "r"(tid));
        asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(dst), "r"(a), "r"(b) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    const uint2 o = lane < (int)gridDim.x ? slot[lane] : make_uint2(0u, 0u);
    const uint32_t amax = __reduce_max_sync(0xffffffffu, o.x);
    const uint32_t any = __reduce_or_sync(0xffffffffu, o.y);
    const float S = __fdiv_rn(__uint_as_float(amax), __fmul_rn(6.0f, p.fp8_div));
    if (g == 0) {
        p.S_out[0] = S;
        if (any && p.status_dev) atomicOr(p.status_dev, 1);
    }
    float E = __frcp_rn(S);
    const bool usable = (S > 0.0f) && isfinite(S) && isfinite(E);
    if (!usable) E = 1.0f;
    u64 w2[8];
#pragma unroll
    for (int j = 0; j < 8; j++) w2[j] = 0ull;
    const float* wkey = nullptr;
    quantize_segment<DT, METHOD, OBJ, BLOCK, 1, true>(p, tab, cur, g, valid, pack2(E, E), usable, w2, wkey);
    zero_pads(p.sf_swizzled, p.rows, p.kb, p.kpad4, g, (int64_t)gridDim.x * kClusterThreads);
}

// Launches the cluster kernel; cudaErrorNotSupported (nothing launched) where the
// device cannot hold a cluster of that size, looked up once per device.
template <int DT, int METHOD, int OBJ, int BLOCK>
static cudaError_t launch_cluster(const QuantParams& p, cudaStream_t s) {
    const auto kernel = quantize_cluster_kernel<DT, METHOD, OBJ, BLOCK>;
    int ctas = 1;
    while (ctas * kClusterThreads < p.nseg) ctas *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (ctas > 8) {                                  // beyond the portable size
        static std::atomic<int> state[kOccDevices];  // 0 not looked up, 1 fits, 2 does not
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kOccDevices) return cudaErrorNotSupported;
        int st = state[dev].load(std::memory_order_acquire);
        if (st == 0) {
            int n = 0;
            st = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                         cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0
                     ? 1
                     : 2;
            if (st == 2) (void)cudaGetLastError();
            state[dev].store(st, std::memory_order_release);
        }
        if (st == 2) return cudaErrorNotSupported;
    }
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <int DT, int METHOD, int OBJ, int BLOCK, int FIX>
static cudaError_t launch_dyn(const QuantParams& p_in, int sms, cudaStream_t s) {
    if constexpr (FIX == 1) {
        if (p_in.nseg <= (int64_t)kClusterCtas * kClusterThreads) {
            const cudaError_t e = launch_cluster<DT, METHOD, OBJ, BLOCK>(p_in, s);
            if (e != cudaErrorNotSupported) return e;
        }
    }
    static std::atomic<int> occ_cache[kOccDevices];
    const int occ = occupancy_per_sm(occ_cache, quantize_kernel<DT, METHOD, OBJ, BLOCK, FIX, 1>, 256);
    QuantParams p = p_in;
    const cudaError_t e = launch_amax_partials(p.x, DT, p.nseg * 16, p.part_max, p.part_bad, &p.nparts, sms, s);
    if (e != cudaSuccess) return e;
    int64_t grid = (p.nseg + 255) / 256;
    if (grid > (int64_t)sms * occ) grid = (int64_t)sms * occ;
    return launch_dependent(quantize_kernel<DT, METHOD, OBJ, BLOCK, FIX, 1>, grid, 256, s, p);
}

template <int DT, int METHOD, int OBJ>
static cudaError_t dyn_block(const QuantParams& p, bool fix, int block, int sms, cudaStream_t s) {
    if (METHOD == 0 && !fix) {
        switch (block) {
            case 16: return launch_dyn<DT, METHOD, OBJ, 16, 0>(p, sms, s);
            case 32: return launch_dyn<DT, METHOD, OBJ, 32, 0>(p, sms, s);
            default: return launch_dyn<DT, METHOD, OBJ, 64, 0>(p, sms, s);
        }
    }
    switch (block) {
        case 16: return launch_dyn<DT, METHOD, OBJ, 16, 1>(p, sms, s);
        case 32: return launch_dyn<DT, METHOD, OBJ, 32, 1>(p, sms, s);
        default: return launch_dyn<DT, METHOD, OBJ, 64, 1>(p, sms, s);
    }
}

cudaError_t launch_quantize_dynamic(const QuantParams& p_in, int dtype, int method, int obj, int block, int sms,
                                    cudaStream_t s) {
    QuantParams p = p_in;
    bool fix;
    prepare_quant_params(p, method, obj, block, &fix);
    cudaError_t e;
    if (dtype == 0) {
        if (method == 1) e = dyn_block<0, 1, 0>(p, fix, block, sms, s);
        else if (obj == 1) e = dyn_block<0, 0, 1>(p, fix, block, sms, s);
        else e = dyn_block<0, 0, 0>(p, fix, block, sms, s);
    } else {
        if (method == 1) e = dyn_block<1, 1, 0>(p, fix, block, sms, s);
        else if (obj == 1) e = dyn_block<1, 0, 1>(p, fix, block, sms, s);
        else e = dyn_block<1, 0, 0>(p, fix, block, sms, s);
    }
    return e;
}

}  // namespace nvfp4
