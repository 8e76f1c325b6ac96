// Static-scale launches of the sweep kernel (S read from device memory) and
// the host-side dispatch shared with the dynamic-scale launches.
#include "quantize_kernel.cuh"

namespace nvfp4 {

template <int DT, int METHOD, int OBJ, int BLOCK, int FIX>
static cudaError_t launch_one(const QuantParams& p, int sms, cudaStream_t s) {
    static std::atomic<int> occ_cache[kOccDevices];
    const int occ = occupancy_per_sm(occ_cache, quantize_kernel<DT, METHOD, OBJ, BLOCK, FIX, 0>, 256);
    const int64_t threads_needed = (p.nseg + 31) & ~(int64_t)31;
    int64_t grid = (threads_needed + 255) / 256;
    const int64_t cap = (int64_t)sms * occ;
    if (grid > cap) {
        grid = cap;
        // 4/6 with one weight vector: up to 1/32 fewer CTAs so that a lane keeps its columns
        const int64_t row = p.kb * (BLOCK / 16);
        if (METHOD == 2 && OBJ == 1 && p.w_row_stride == 0)
            for (int64_t g = cap; g >= cap - cap / 32; g--)
                if (g * 256 % row == 0) {
                    grid = g;
                    break;
                }
    }
    return launch_dependent(quantize_kernel<DT, METHOD, OBJ, BLOCK, FIX, 0>, grid, 256, s, p);
}

template <int DT, int METHOD, int OBJ, int BLOCK>
static cudaError_t dispatch_fix(const QuantParams& p, bool fix, int sms, cudaStream_t s) {
    if (METHOD == 0 && !fix) return launch_one<DT, METHOD, OBJ, BLOCK, 0>(p, sms, s);
    return launch_one<DT, METHOD, OBJ, BLOCK, 1>(p, sms, s);
}

template <int DT, int METHOD, int OBJ>
static cudaError_t dispatch_block(const QuantParams& p, bool fix, int block, int sms, cudaStream_t s) {
    switch (block) {
        case 16: return dispatch_fix<DT, METHOD, OBJ, 16>(p, fix, sms, s);
        case 32: return dispatch_fix<DT, METHOD, OBJ, 32>(p, fix, sms, s);
        default: return dispatch_fix<DT, METHOD, OBJ, 64>(p, fix, sms, s);
    }
}

template <int DT, int METHOD>
static cudaError_t dispatch_obj(const QuantParams& p, int obj, bool fix, int block, int sms, cudaStream_t s) {
    if (obj == 1) return dispatch_block<DT, METHOD, 1>(p, fix, block, sms, s);
    return dispatch_block<DT, METHOD, 0>(p, fix, block, sms, s);
}

FastDiv make_fast_div(uint32_t d) {
    FastDiv f;
    uint32_t l = 0;
    while (l < 32 && (1ull << l) < d) l++;
    f.mul = (uint32_t)(((1ull << 32) * ((1ull << l) - d)) / d + 1);
    f.s1 = l < 1 ? l : 1;
    f.s2 = l > 0 ? l - 1 : 0;
    return f;
}

void prepare_quant_params(QuantParams& p, int method, int obj, int block, bool* fix) {
    const int def_lo = (obj == 0 && block == 16) ? -3 : -8;
    *fix = (method != 0) || (p.win_lo == def_lo && p.win_hi == 7 && !p.tight);
    p.need_rowcol = (p.sf_swizzled != nullptr) || (obj == 1);
    if (p.narrow) p.kb_div = make_fast_div((uint32_t)p.kb);
}

cudaError_t launch_quantize(const QuantParams& p_in, int dtype, int method, int obj, int block, int sms,
                            cudaStream_t s) {
    QuantParams p = p_in;
    bool fix;
    prepare_quant_params(p, method, obj, block, &fix);
    if (p.nseg > 0) {
        cudaError_t e;
        if (dtype == 0) {
            if (method == 0) e = dispatch_obj<0, 0>(p, obj, fix, block, sms, s);
            else if (method == 1) e = dispatch_block<0, 1, 0>(p, fix, block, sms, s);
            else e = dispatch_obj<0, 2>(p, obj, fix, block, sms, s);
        } else {
            if (method == 0) e = dispatch_obj<1, 0>(p, obj, fix, block, sms, s);
            else if (method == 1) e = dispatch_block<1, 1, 0>(p, fix, block, sms, s);
            else e = dispatch_obj<1, 2>(p, obj, fix, block, sms, s);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace nvfp4
