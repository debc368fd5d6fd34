// Launch of the fp32 gradient walks (scan_bwd.cuh): a block per unit and eight key dimensions.
#include <atomic>

#include "scan_bwd.cuh"
#include "vig_internal.h"

namespace vig {
namespace {

using namespace scan;

template <typename T, int CN, bool VEC>
__global__ void __launch_bounds__(bwd_max_warps(CN) * 32, CN <= 16 ? 2 : 1) scan_bwd_kernel(const ScanBwdArgs<T> a, const FloatPairs pairs) {
    extern __shared__ __align__(16) float sb_smem[];
    pdl_wait();
    pdl_launch_dependents();
    scan_bwd_slab<T, CN, VEC>(a, pairs, blockIdx.x, blockIdx.y, threadIdx.x >> 5, blockDim.x >> 5, sb_smem);
}

template <typename T, int CN, bool VEC>
cudaError_t launch_scan_bwd_t(ScanBwdArgs<T> a, float2* pairs, long long units, cudaStream_t stream) {
    constexpr int kMaxWarps = bwd_max_warps(CN);
    constexpr size_t kPerWarp = (bwd_stage_floats(CN) + bwd_fold_floats(CN)) * sizeof(float);
    static std::atomic<int> sms_of[64];   // 0: this instance is not configured on the device yet
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int sms = sms_of[dev].load(std::memory_order_acquire);
    if (sms == 0) {
        if ((e = cudaFuncSetAttribute(scan_bwd_kernel<T, CN, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kMaxWarps * kPerWarp))) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        sms_of[dev].store(sms, std::memory_order_release);
    }
    // Segments: about sixteen warps per SM over the whole call, in whole groups of TG tokens; a call that nearly has them
    // without splitting walks whole sequences and skips the first pass, which costs half as much again.
    const int slabs = (a.dk + kRows - 1) / kRows;
    long long want = (16LL * sms + units * slabs / 2) / (units * slabs);
    if (want < 1) want = 1;
    if (want > kMaxWarps) want = kMaxWarps;
    a.seg_len = (int)(((a.L + want - 1) / want + TG - 1) / TG * TG);
    const int nw = (a.L + a.seg_len - 1) / a.seg_len;
    const cudaError_t le = launch_pdl(scan_bwd_kernel<T, CN, VEC>, dim3((unsigned)units, (unsigned)slabs), dim3(nw * 32), nw * kPerWarp, stream, a, FloatPairs{pairs});
    count_launch();
    return le != cudaSuccess ? le : cudaGetLastError();
}

}  // namespace

template <typename T>
cudaError_t launch_scan_bwd(const T* q, const T* k, const T* v, const T* la_f, const T* la_b, const T* d_out, T* dq, T* dk_out, T* dla_f, T* dla_b,
                            void* scratch, long long units, int L, int dk, int dv, cudaStream_t stream) {
    ScanBwdArgs<T> a{q, k, v, la_f, la_b, d_out, dq, dk_out, dla_f, dla_b, L, dk, dv, 0};
    float2* pairs = static_cast<float2*>(scratch);
    const bool vec = dv % 4 == 0;   // rows of whole pieces (the base addresses are 16-byte aligned)
#define VIG_CASE(CN_) \
    if (dv <= 4 * CN_) return vec ? launch_scan_bwd_t<T, CN_, true>(a, pairs, units, stream) : launch_scan_bwd_t<T, CN_, false>(a, pairs, units, stream);
    VIG_CASE(8) VIG_CASE(12) VIG_CASE(16) VIG_CASE(32)
#undef VIG_CASE
    return cudaErrorInvalidValue;
}

template cudaError_t launch_scan_bwd<float>(const float*, const float*, const float*, const float*, const float*, const float*, float*, float*, float*,
                                            float*, void*, long long, int, int, int, cudaStream_t);
template cudaError_t launch_scan_bwd<__nv_bfloat16>(const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*,
                                                    const __nv_bfloat16*, const __nv_bfloat16*, __nv_bfloat16*, __nv_bfloat16*, __nv_bfloat16*,
                                                    __nv_bfloat16*, void*, long long, int, int, int, cudaStream_t);

}  // namespace vig
