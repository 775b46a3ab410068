// launch.cuh -- grid sizing for the persistent grid-stride kernels: as many
// resident blocks (256 threads unless said otherwise) as the SMs hold (a
// multiple of the SM count), never more blocks than tiles of as many tracks.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace geonav {

// Resident blocks per SM of a kernel (at least 1).  The occupancy query costs
// about as much host time as a launch, and its answer depends on the kernel, the block
// and the device alone, so each thread keeps the answers it has had.
static inline int resident_blocks(const void* kernel, int threads, int smem) {
    struct Entry {
        const void* kernel;
        int threads, smem, device, blocks;
    };
    constexpr int kEntries = 64;
    static thread_local Entry cache[kEntries];
    static thread_local int used = 0;
    int device = -1, per_sm = 0;
    const bool known = cudaGetDevice(&device) == cudaSuccess;
    for (int k = 0; known && k < used; ++k) {
        const Entry& e = cache[k];
        if (e.kernel == kernel && e.threads == threads && e.smem == smem && e.device == device) return e.blocks;
    }
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return 1;
    }
    if (known && used < kEntries) cache[used++] = {kernel, threads, smem, device, per_sm};
    return per_sm;
}

template <typename K>
static inline int blocks_for(K kernel, int64_t n, int smem, int num_sms, int threads = 256) {
    const int per_sm = resident_blocks(reinterpret_cast<const void*>(kernel), threads, smem);
    const int64_t need = (n + threads - 1) / threads;
    const int64_t cap = int64_t(per_sm) * num_sms;
    return int(need < cap ? need : cap);
}

// Lets a kernel take `smem` bytes of dynamic shared memory.  The limit that
// holds without this (48 KB) counts the kernel's static shared memory too, of
// which the callers' kernels have up to 16 KB.  The limit is set to all that the device
// gives, never to this call's size: it belongs to the kernel, and another thread
// could lower it to its own size before this one launches.  Each thread keeps the
// limits it has set.
static inline cudaError_t raise_smem(const void* kernel, int smem) {
    struct Entry {
        const void* kernel;
        int device, most;
    };
    constexpr int kEntries = 64;
    static thread_local Entry cache[kEntries];
    static thread_local int used = 0;
    int device = 0, most = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    for (int k = 0; k < used; ++k)
        if (cache[k].kernel == kernel && cache[k].device == device)
            return smem <= cache[k].most ? cudaSuccess : cudaErrorInvalidValue;
    cudaFuncAttributes a;
    if ((e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device)) != cudaSuccess ||
        (e = cudaFuncGetAttributes(&a, kernel)) != cudaSuccess)
        return e;
    most -= int(a.sharedSizeBytes);
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return e;
    if (used < kEntries) cache[used++] = {kernel, device, most};
    return smem <= most ? cudaSuccess : cudaErrorInvalidValue;
}
template <typename K>
static inline cudaError_t prep(K kernel, int smem) {
    return smem > 32 * 1024 ? raise_smem(reinterpret_cast<const void*>(kernel), smem) : cudaSuccess;
}

}  // namespace geonav
