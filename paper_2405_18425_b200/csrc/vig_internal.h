// Internal declarations shared by the translation units of libvig_bigla (not part of the C ABI).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "vig_bigla.h"

namespace vig {

// Device status word: bit flags set by kernels whose bounded waits expire.
constexpr int kDevStatusTimeout = 1;
constexpr int kDevStatusInternal = 2;   // a kernel found its own set-up inconsistent (reported as VIG_ERR_CUDA)
int* device_status_ptr();            // device address of the status word of the current device (NULL on error);
                                     // one int behind it: the count of units handed to the in-kernel recurrence
int take_expire_next_wait();         // test hook: 1 (2) once after vig_test_expire_next_wait (_exchange), else 0
void count_launch(unsigned n = 1);   // bumps the process-wide launch counter

// ---- Eq. 6 step by step in fp32 on the CUDA cores, any dk <= 128, dv <= 256.  adjoint: with the gates of the two directions
// exchanged and moved by one token, so that on (k, q, d_out) the result is the gradient with respect to v:
//   dv_r = 1/2 sum_{t >= r} (k_r * prod_{m = r+1..t} alpha>_m . q_t) g_t + 1/2 sum_{t <= r} (k_r * prod_{m = t..r-1} alpha<_m . q_t) g_t ----
bool scan_supported(int dk, int dv);
template <typename T>
cudaError_t launch_scan_fwd(const T* q, const T* k, const T* v, const T* la_f, const T* la_b, T* out, long long units, int L, int dk, int dv,
                            bool adjoint, cudaStream_t stream);
// Its gradient with respect to q, k and the log gates, segments of a sequence walked side by side within a block; scratch:
// [units][L][dk] pairs of floats.
template <typename T>
cudaError_t launch_scan_bwd(const T* q, const T* k, const T* v, const T* la_f, const T* la_b, const T* d_out, T* dq, T* dk_out, T* dla_f, T* dla_b,
                            void* scratch, long long units, int L, int dk, int dv, cudaStream_t stream);

// ---- gate preparation ----
template <typename T>
cudaError_t launch_gate_prep(const T* g_f, const T* g_b, T* la_f, T* la_b, long long n, float tau,
                             cudaStream_t stream);
// dg = dlog alpha * sigmoid(-g) / tau, both directions in one launch (the outputs may be the incoming gradients' buffers)
template <typename T>
cudaError_t launch_gate_prep_bwd(const T* g_f, const T* g_b, const T* d_f, const T* d_b, T* o_f, T* o_b, long long n, float tau,
                                 cudaStream_t stream);

// The number of units by which a form is chosen where that depends on it: the call's own, or, for the slices of a host call,
// that of the whole batch, so that a slice has the bits of a device call on the batch.
long long form_units(long long units);

// ---- bf16 tensor-core path: dispatch over the tcgen05 kernels (defined with the entry points) ----
bool tc_supported(int dk, int dv);
// Scratch bytes the tensor-core path needs for this shape; 0 if no launch of it uses scratch.
size_t tc_workspace_bytes(long long units, int L, int dk, int dv);
size_t tc_least_workspace_bytes(long long units, int L, int dk, int dv);   // what the form that needs least takes
// ws_bytes: what there is of it; a form that needs less is taken where the fastest one does not fit.
cudaError_t launch_bigla_tc(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                            const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out,
                            long long units, int L, int dk, int dv, void* ws, size_t ws_bytes, cudaStream_t stream);

// ---- bf16 tcgen05 / TMEM path (units of at most 256 tokens) ----
bool umma_supported(int dk, int dv, int L);
// gate_tau > 0: la_f / la_b hold the gate logits g and the kernel prepares log alpha = logsigmoid(g) / gate_tau itself.
cudaError_t launch_bigla_umma(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                              const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out,
                              long long units, int L, int dk, int dv, float gate_tau, cudaStream_t stream);

// The same on the warp-level tensor-core instructions, a block per unit, a warp per 16 tokens; mma_preferred: the shapes
// (of those of umma_supported) it is the faster of the two for.
bool mma_preferred(long long units, int L, int dk, int dv, bool gates);
cudaError_t launch_bigla_mma(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                             const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out,
                             long long units, int L, int dk, int dv, float gate_tau, cudaStream_t stream);

// Longer sequences on the same instructions: chunks of up to 128 tokens, states through scratch (three launches), the gates
// prepared on the way as well.  mma_chunks_preferred: the shapes it is the faster form for.
bool mma_chunks_supported(long long units, int L, int dk, int dv);
bool mma_chunks_preferred(long long units, int L, int dk, int dv, bool gates);
size_t mma_chunks_workspace_bytes(long long units, int L, int dk, int dv, bool gates);
cudaError_t launch_bigla_mma_chunks(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                    const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out, long long units,
                                    int L, int dk, int dv, float gate_tau, void* ws, cudaStream_t stream);

// Up to eight such chunks as the blocks of a cluster, states through distributed shared memory: one launch, no scratch.
bool mma_cluster_supported(long long units, int L, int dk, int dv);
bool mma_cluster_preferred(long long units, int L, int dk, int dv, bool gates);
cudaError_t launch_bigla_mma_cluster(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                     const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out, long long units,
                                     int L, int dk, int dv, float gate_tau, cudaStream_t stream);

// ---- Eq. 7 around the mixer: depth-wise 3 x 3 convolution (channels last) and the 2-D gate blend ----
bool dwconv_supported(int C, size_t elem);
template <typename T>
cudaError_t launch_dwconv3x3(const T* x, const T* w, const T* bias, T* out, long long images, int Hh, int Ww, int C,
                             cudaStream_t stream);
template <typename T>
cudaError_t launch_gate_blend(const T* o_local, const T* z, const T* o_global, T* out, long long n, cudaStream_t stream);

// ---- the same kernel for sequences of up to 32 x 256 tokens: one block per 256-token segment, the blocks of a unit
// exchange their segment summaries through scratch memory inside one cooperative launch ----
bool umma_seg_supported(int dk, int dv, int L);
size_t umma_seg_workspace_bytes(long long units, int L);
cudaError_t launch_bigla_umma_seg(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                  const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out,
                                  long long units, int L, int dk, int dv, void* ws, cudaStream_t stream);

// ---- bf16 tcgen05 / TMEM path for longer sequences: chunk tasks, states through scratch (three launches) ----
size_t umma_long_workspace_bytes(long long units, int L, int dk, int dv);
cudaError_t launch_bigla_umma_long(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                   const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out,
                                   long long units, int L, int dk, int dv, void* ws, cudaStream_t stream);

// ---- gradient of the forward pass with respect to q, k and the log gates (fp32 recurrences on the CUDA cores):
// launch_scan_bwd, or walks over segments in several launches.  The gates of dv's forward pass on (k, q, d_out), moved by
// one token: launch_shift_gates ----
bool bwd_supported(int dk, int dv);
size_t bwd_scratch_bytes(long long units, int L, int dk, int dv);   // 0: the device could not be queried
bool bwd_in_one_launch(long long units, int L, int dk, int dv);   // launch_scan_grad takes the call: dv among its results
bool scan_grad_supported(int dk, int dv);
template <typename T>
cudaError_t launch_scan_grad(const T* q, const T* k, const T* v, const T* la_f, const T* la_b, const T* d_out, T* dq, T* dk_out, T* dv_out,
                             T* dla_f, T* dla_b, void* scratch, long long units, int L, int dk, int dv, cudaStream_t stream);
template <typename T>
cudaError_t launch_shift_gates(const T* la_f, const T* la_b, T* out_f, T* out_b, long long units, int L, int dk, cudaStream_t stream);
template <typename T>
cudaError_t launch_bigla_bwd(const T* q, const T* k, const T* v, const T* la_f, const T* la_b, const T* d_out, T* dq, T* dk_out, T* dla_f,
                             T* dla_b, float* scratch, long long units, int L, int dk, int dv, cudaStream_t stream);

// ---- the whole gradient of the bf16 forward pass on the tensor cores (head sizes of the paper's models, 16 tokens or more) ----
bool grad_supported(long long units, int L, int dk, int dv);
size_t grad_scratch_bytes(long long units, int L, int dk, int dv);   // 0: the call uses no scratch
cudaError_t launch_bigla_grad(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v, const __nv_bfloat16* la_f,
                              const __nv_bfloat16* la_b, const __nv_bfloat16* d_out, __nv_bfloat16* dq, __nv_bfloat16* dk_out,
                              __nv_bfloat16* dv_out, __nv_bfloat16* dla_f, __nv_bfloat16* dla_b, void* scratch, long long units, int L, int dk,
                              int dv, cudaStream_t stream);

// ---- copies between pinned host memory and the device by a kernel ----
constexpr int kHostCopies = 5;   // per launch
struct HostCopy {
    const void* src;
    void* dst;
    size_t bytes;   // a multiple of 16; both addresses 16-byte aligned
};
bool host_copy_usable(const void* host, size_t bytes);   // all of it pinned and mapped, aligned
cudaError_t launch_host_copy(const HostCopy* copies, int n, int max_blocks, cudaStream_t stream);

// Launch with programmatic stream serialization: the kernel's prologue (everything before its pdl_wait) may overlap
// the tail of the kernel before it in the stream.  cluster: blocks of a cluster (along x; the grid is a multiple of it).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, int cluster, cudaStream_t stream,
                                      Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              Args&&... args) {
    return launch_pdl_cluster(kernel, grid, block, smem, 1, stream, static_cast<KArgs>(args)...);
}

// Kernel family the bf16 entry points use (a vig_test_kernel value; test_hooks.h): the default unless a test changed it.
int kernel_preference();

}  // namespace vig
