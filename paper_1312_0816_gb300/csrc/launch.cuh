// launch.cuh -- grid sizing for the persistent grid-stride kernels: as many
// resident blocks (256 threads unless said otherwise) as the SMs hold (a
// multiple of the SM count), never more blocks than tiles of as many tracks.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace geonav {

template <typename K>
static inline int blocks_for(K kernel, int64_t n, int smem, int num_sms, int threads = 256) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    const int64_t need = (n + threads - 1) / threads;
    const int64_t cap = int64_t(per_sm) * num_sms;
    return int(need < cap ? need : cap);
}

// Lets a kernel take `smem` bytes of dynamic shared memory.  The limit that
// holds without this (48 KB) counts the kernel's static shared memory too, of
// which the callers' kernels have up to 16 KB.
template <typename K>
static inline cudaError_t prep(K kernel, int smem) {
    if (smem > 32 * 1024) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return cudaSuccess;
}

}  // namespace geonav
