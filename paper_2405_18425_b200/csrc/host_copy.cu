// Copies between pinned host memory and the device by a kernel instead of a copy engine.  Reading the host link this way
// runs at 51 GB/s where the engine reaches 55, but one launch moves several buffers and starts at once (an engine copy has a
// fixed cost of about 5 us, more while the other direction is busy); and results that travel back beside copies to the device
// can be paced: at full rate either way the link carries about 70 GB/s in both directions together, and the writes out,
// which share their lane with the requests of the copies in, hold those back more than their share (57.8 MB in, 19.3 MB out
// in three slices: 1.38 ms at full rate, 1.33 ms from one or two blocks).
#include <cuda.h>

#include <cstring>

#include "ptx.cuh"
#include "vig_internal.h"

namespace vig {
namespace {

struct CopySet {
    HostCopy c[kHostCopies];
};

__global__ void __launch_bounds__(512) host_copy_kernel(const CopySet s) {
    const size_t stride = (size_t)gridDim.x * blockDim.x, first = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
#pragma unroll 1
    for (int i = 0; i < kHostCopies; ++i) {
        const uint4* src = static_cast<const uint4*>(s.c[i].src);
        uint4* dst = static_cast<uint4*>(s.c[i].dst);
        const size_t n = s.c[i].bytes / 16;
        size_t x = first;
        for (; x + 3 * stride < n; x += 4 * stride) {   // four loads in flight: a round trip over the link takes microseconds
            const uint4 a = src[x], b = src[x + stride], c = src[x + 2 * stride], d = src[x + 3 * stride];
            dst[x] = a;
            dst[x + stride] = b;
            dst[x + 2 * stride] = c;
            dst[x + 3 * stride] = d;
        }
        for (; x < n; x += stride) dst[x] = src[x];
    }
}

}  // namespace

// Every byte has to be mapped: a kernel that runs past the end of a registered range faults, where an engine copy returns an
// error.  Ranges that follow one another without a gap (memory registered piece by piece) will do.
bool host_copy_usable(const void* host, size_t bytes) {
    if ((reinterpret_cast<uintptr_t>(host) & 15) != 0 || bytes == 0 || bytes % 16 != 0) return false;
    using AttributeFn = CUresult (*)(void*, CUpointer_attribute, CUdeviceptr);
    static const AttributeFn attribute = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPoint("cuPointerGetAttribute", &f, cudaEnableDefault, &found) != cudaSuccess || found != cudaDriverEntryPointSuccess) f = nullptr;
        return reinterpret_cast<AttributeFn>(f);
    }();
    if (!attribute) return false;
    uintptr_t p = reinterpret_cast<uintptr_t>(host);
    const uintptr_t end = p + bytes;
    for (int ranges = 0; p < end; ++ranges) {
        cudaPointerAttributes at;
        if (ranges == 64 || cudaPointerGetAttributes(&at, reinterpret_cast<void*>(p)) != cudaSuccess) {
            cudaGetLastError();   // (nothing of the failed query is left behind)
            return false;
        }
        if (at.type != cudaMemoryTypeHost || reinterpret_cast<uintptr_t>(at.devicePointer) != p) return false;   // pinned, and mapped at its own address
        CUdeviceptr start = 0;
        size_t size = 0;
        if (attribute(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, (CUdeviceptr)p) != CUDA_SUCCESS ||
            attribute(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, (CUdeviceptr)p) != CUDA_SUCCESS || start + size <= p)
            return false;
        p = start + size;
    }
    return true;
}

cudaError_t launch_host_copy(const HostCopy* copies, int n, int max_blocks, cudaStream_t stream) {
    CopySet s;
    memset(&s, 0, sizeof s);
    size_t most = 0;
    for (int i = 0; i < n && i < kHostCopies; ++i) {
        s.c[i] = copies[i];
        if (copies[i].bytes > most) most = copies[i].bytes;
    }
    // As many threads as there are pieces for small copies, so that a single round trip moves them; the link is full with eight
    // blocks of 256 threads and more.
    size_t blocks = (most / 16 + 511) / 512;
    if (blocks < 1) blocks = 1;
    if (blocks > (size_t)max_blocks) blocks = max_blocks;
    host_copy_kernel<<<(unsigned)blocks, 512, 0, stream>>>(s);
    count_launch();
    return cudaGetLastError();
}

}  // namespace vig
