// Launch of the fp32 forward walks (scan_fwd.cuh): a block per unit and sixteen value columns.
#include <atomic>

#include "scan_fwd.cuh"
#include "vig_internal.h"

namespace vig {
namespace {

using namespace scan;

template <typename T, int RPL, bool VEC, int CPL, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, RPL <= 8 && CPL == 2 && WARPS <= 8 ? 2 : 1) scan_fwd_kernel(const ScanArgs<T> a) {
    extern __shared__ __align__(16) float sc_smem[];
    pdl_wait();
    pdl_launch_dependents();
    scan_fwd_slab<T, RPL, VEC, CPL>(a, blockIdx.x, blockIdx.y, threadIdx.x >> 5, blockDim.x >> 5, sc_smem);
}

template <typename T, int RPL, bool VEC, int CPL, int WARPS = scan_max_warps(RPL)>
cudaError_t launch_scan_t(ScanArgs<T> a, long long units, cudaStream_t stream) {
    constexpr int kMaxWarps = WARPS;
    static std::atomic<int> sms_of[64];   // 0: this instance is not configured on the device yet
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int sms = sms_of[dev].load(std::memory_order_acquire);
    const size_t per_warp = (scan_stage_floats(RPL, CPL) > scan_fold_floats(RPL, CPL) ? scan_stage_floats(RPL, CPL) : scan_fold_floats(RPL, CPL)) * sizeof(float);
    if (sms == 0) {
        if ((e = cudaFuncSetAttribute(scan_fwd_kernel<T, RPL, VEC, CPL, WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kMaxWarps * per_warp))) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        sms_of[dev].store(sms, std::memory_order_release);
    }
    // Segments: about sixteen warps per SM over the whole call (what hides a token's chain of dependent operations), in
    // whole groups of TG tokens.
    const int slabs = (a.dv + 8 * CPL - 1) / (8 * CPL);
    const long long n = form_units(units) * slabs;
    long long want = (16LL * sms + n - 1) / n;
    const int most = WARPS > 8 ? many_segments(a.L) : kMaxWarps;
    if (want > most) want = most;
    a.seg_len = (int)(((a.L + want - 1) / want + TG - 1) / TG * TG);
    const int nw = (a.L + a.seg_len - 1) / a.seg_len;
    const cudaError_t le = launch_pdl(scan_fwd_kernel<T, RPL, VEC, CPL, WARPS>, dim3((unsigned)units, (unsigned)slabs), dim3(nw * 32), nw * per_warp, stream, a);
    count_launch();
    return le != cudaSuccess ? le : cudaGetLastError();
}

}  // namespace

bool scan_supported(int dk, int dv) { return dk >= 1 && dv >= 1 && dk <= 128 && dv <= 256; }

template <typename T>
cudaError_t launch_scan_fwd(const T* q, const T* k, const T* v, const T* la_f, const T* la_b, T* out, long long units, int L, int dk, int dv,
                            bool adjoint, cudaStream_t stream) {
    ScanArgs<T> a{q, k, v, adjoint ? la_b : la_f, adjoint ? la_f : la_b, out, L, dk, dv, 0, adjoint ? -1 : 0, adjoint ? 1 : 0};
    const bool vec = dk % 4 == 0 && dv % 4 == 0;   // rows of whole pieces (the base addresses are 16-byte aligned)
    // Value columns a lane: two, or three or four where that leaves no SM with more blocks than another, since those are waited for and a
    // wider warp costs little more (48 units of 196 tokens, 32 x 64, fp32: 192 blocks of two columns 31 us, 144 of three 25).
    int dev = 0, sms = 0, cpl = 2;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    auto blocks = [&](int x) { return form_units(units) * ((dv + 8 * x - 1) / (8 * x)); };
    if (vec && dk <= 32 && blocks(2) > sms) cpl = blocks(3) <= sms ? 3 : (blocks(4) <= sms ? 4 : 2);
#define VIG_CASE(RPL_) \
    if (dk <= 4 * RPL_) return vec ? launch_scan_t<T, RPL_, true, 2>(a, units, stream) : launch_scan_t<T, RPL_, false, 2>(a, units, stream);
    // Few sequences, blocks with an SM each: sixteen warps (training step of 24 units of 196 tokens, 16 x 64, fp32: 42.1 us, 56.3 with eight).
#define VIG_MANY(RPL_) \
    if (dk <= 4 * RPL_) return launch_scan_t<T, RPL_, true, 2, kManyWarps>(a, units, stream);
    if (vec && dk <= 32 && blocks(2) <= sms && L <= kManyTokens) {
        VIG_MANY(4) VIG_MANY(8)
    }
#undef VIG_MANY
#define VIG_WIDE(RPL_) \
    if (cpl > 2 && dk <= 4 * RPL_) return cpl == 3 ? launch_scan_t<T, RPL_, true, 3>(a, units, stream) : launch_scan_t<T, RPL_, true, 4>(a, units, stream);
    VIG_WIDE(4) VIG_WIDE(8)
    VIG_CASE(4) VIG_CASE(8) VIG_CASE(16) VIG_CASE(32)
#undef VIG_WIDE
#undef VIG_CASE
    return cudaErrorInvalidValue;
}

template cudaError_t launch_scan_fwd<float>(const float*, const float*, const float*, const float*, const float*, float*, long long, int, int, int,
                                            bool, cudaStream_t);
template cudaError_t launch_scan_fwd<__nv_bfloat16>(const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*,
                                                    const __nv_bfloat16*, __nv_bfloat16*, long long, int, int, int, bool, cudaStream_t);

}  // namespace vig
