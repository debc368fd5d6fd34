// Launches of the fp32 gradient walks (scan_bwd.cuh): a block per unit and eight key dimensions, and, where the gradient with
// respect to v comes by walks as well (scan_fwd.cuh on swapped operands), a block per unit and sixteen value columns beside them.
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

// Both in one launch, the longer walks first.  Either alone leaves SMs idle that hold one block beside SMs that hold two: 48 units
// of 196 tokens, 32 x 64, fp32, 192 blocks each: 31 us and 51 us one after the other, 59 us together.
template <typename T, int CN, int RPL, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, WARPS > 8 ? 1 : 2) scan_grad_kernel(const ScanBwdArgs<T> a, const FloatPairs pairs, const ScanArgs<T> f, int bwd_slabs, int bwd_warps,
                                                           int fwd_warps) {
    extern __shared__ __align__(16) float sg_smem[];
    pdl_wait();
    pdl_launch_dependents();
    const int w = threadIdx.x >> 5, y = blockIdx.y;
    if (y < bwd_slabs) scan_bwd_slab<T, CN, true>(a, pairs, blockIdx.x, y, w, bwd_warps, sg_smem);
    else scan_fwd_slab<T, RPL, true>(f, blockIdx.x, y - bwd_slabs, w, fwd_warps, sg_smem);
}

// Segments: about sixteen warps per SM over the blocks of a call, in whole groups of TG tokens; a call that nearly has them
// without splitting walks whole sequences and skips the first pass, which costs half as much again.
int segment_length(int L, long long blocks, int sms, int most) {
    long long want = (16LL * sms + blocks / 2) / blocks;
    if (want < 1) want = 1;
    if (want > most) want = most;
    return (int)(((L + want - 1) / want + TG - 1) / TG * TG);
}

template <typename T, int CN, int RPL, int WARPS>
cudaError_t launch_scan_grad_t(ScanBwdArgs<T> a, float2* pairs, ScanArgs<T> f, long long units, cudaStream_t stream) {
    constexpr int kMaxWarps = WARPS;
    static_assert(bwd_max_warps(CN) == 8 && scan_max_warps(RPL) == 8, "");
    constexpr size_t kBwd = (bwd_stage_floats(CN) + bwd_fold_floats(CN)) * sizeof(float);
    constexpr size_t kFwd = (scan_stage_floats(RPL) > scan_fold_floats(RPL) ? scan_stage_floats(RPL) : scan_fold_floats(RPL)) * sizeof(float);
    constexpr size_t kPerWarp = kBwd > kFwd ? kBwd : kFwd;
    static std::atomic<int> sms_of[64];   // 0: this instance is not configured on the device yet
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int sms = sms_of[dev].load(std::memory_order_acquire);
    if (sms == 0) {
        if ((e = cudaFuncSetAttribute(scan_grad_kernel<T, CN, RPL, WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kMaxWarps * kPerWarp))) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        sms_of[dev].store(sms, std::memory_order_release);
    }
    const int bs = (a.dk + kRows - 1) / kRows, fs = (f.dv + kCols - 1) / kCols;
    const int most = WARPS > 8 ? many_segments(a.L) : kMaxWarps;
    a.seg_len = segment_length(a.L, units * bs, sms, most);
    f.seg_len = segment_length(f.L, units * fs, sms, most);
    const int nb = (a.L + a.seg_len - 1) / a.seg_len, nf = (f.L + f.seg_len - 1) / f.seg_len, nw = nb > nf ? nb : nf;
    const cudaError_t le = launch_pdl(scan_grad_kernel<T, CN, RPL, WARPS>, dim3((unsigned)units, (unsigned)(bs + fs)), dim3(nw * 32), nw * kPerWarp, stream, a,
                                      FloatPairs{pairs}, f, bs, nb, nf);
    count_launch();
    return le != cudaSuccess ? le : cudaGetLastError();
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
    const int slabs = (a.dk + kRows - 1) / kRows;
    a.seg_len = segment_length(a.L, units * slabs, sms, kMaxWarps);
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

bool scan_grad_supported(int dk, int dv) { return dk <= 32 && dv <= 64 && dk % 4 == 0 && dv % 4 == 0; }
static bool scan_grad_many(long long units, int dk, int dv, int sms) {   // a block an SM at most: sixteen warps each
    return units * ((dk + kRows - 1) / kRows + (dv + kCols - 1) / kCols) <= sms;
}

template <typename T>
cudaError_t launch_scan_grad(const T* q, const T* k, const T* v, const T* la_f, const T* la_b, const T* d_out, T* dq, T* dk_out, T* dv_out, T* dla_f, T* dla_b,
                             void* scratch, long long units, int L, int dk, int dv, cudaStream_t stream) {
    const ScanBwdArgs<T> a{q, k, v, la_f, la_b, d_out, dq, dk_out, dla_f, dla_b, L, dk, dv, 0};
    const ScanArgs<T> f{k, q, d_out, la_b, la_f, dv_out, L, dk, dv, 0, -1, 1};   // the adjoint: operands swapped, gates moved by one token
    float2* pairs = static_cast<float2*>(scratch);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const bool many = scan_grad_many(units, dk, dv, sms);
#define VIG_RPL(CN_, RPL_) \
    return many ? launch_scan_grad_t<T, CN_, RPL_, kManyWarps>(a, pairs, f, units, stream) : launch_scan_grad_t<T, CN_, RPL_, 8>(a, pairs, f, units, stream);
#define VIG_CASE(CN_) \
    if (dv <= 4 * CN_) { \
        if (dk <= 16) VIG_RPL(CN_, 4) else VIG_RPL(CN_, 8) \
    }
    VIG_CASE(8) VIG_CASE(12) VIG_CASE(16)
#undef VIG_CASE
#undef VIG_RPL
    return cudaErrorInvalidValue;
}
template cudaError_t launch_scan_grad<float>(const float*, const float*, const float*, const float*, const float*, const float*, float*, float*, float*,
                                             float*, float*, void*, long long, int, int, int, cudaStream_t);
template cudaError_t launch_scan_grad<__nv_bfloat16>(const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*,
                                                     const __nv_bfloat16*, const __nv_bfloat16*, __nv_bfloat16*, __nv_bfloat16*, __nv_bfloat16*,
                                                     __nv_bfloat16*, __nv_bfloat16*, void*, long long, int, int, int, cudaStream_t);

template cudaError_t launch_scan_bwd<float>(const float*, const float*, const float*, const float*, const float*, const float*, float*, float*, float*,
                                            float*, void*, long long, int, int, int, cudaStream_t);
template cudaError_t launch_scan_bwd<__nv_bfloat16>(const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*,
                                                    const __nv_bfloat16*, const __nv_bfloat16*, __nv_bfloat16*, __nv_bfloat16*, __nv_bfloat16*,
                                                    __nv_bfloat16*, void*, long long, int, int, int, cudaStream_t);

}  // namespace vig
