// nav_refine_grid.cu -- the filter step (GEO_FP32_REFINE) of a volume with the
// uniform grid (no tube segments, polycones or apex cones among its solids).
//
// Baskets of more than one wave of tracks: each warp takes up to 128 tracks
// through the FP32 pass before their FP64 (k_grid_sheets, sheet.cuh), with the
// grid's short form and the filter's records staged in shared memory where
// they fit.  Smaller baskets: one thread per track, everything read through L1.
#include <cuda_runtime.h>

#include "geo_internal.h"
#include "launch.cuh"
#include "nav_common.cuh"
#include "nav_refine.cuh"
#include "sheet.cuh"
#include "stage.cuh"

namespace geonav {

constexpr int kGrid = 256, kGridBlocks = 4;   // k_dist_grid: threads per block, resident blocks per SM

__global__ void __launch_bounds__(kGrid, kGridBlocks)
    k_dist_grid(const __grid_constant__ VolView v, Basket b, double* __restrict__ step, int32_t* __restrict__ hit,
                double* __restrict__ bpoint, int32_t* __restrict__ nref) {
    __shared__ ShapeRec64 m64;
    __shared__ double pd[6][kGrid];   // each thread's track, so that it does not live in registers
    const int t = threadIdx.x;
    if (t < int(sizeof(ShapeRec64) / sizeof(double)))
        reinterpret_cast<double*>(&m64)[t] = reinterpret_cast<const double*>(&v.m64)[t];
    __syncthreads();
    const int64_t stride = int64_t(gridDim.x) * kGrid;
    for (int64_t i = int64_t(blockIdx.x) * kGrid + t; i < b.n; i += stride) {
        RefineState rs;
        double best = 0.0;
        int h = -2, nev = 0;
        {
            const double px = b.x[i], py = b.y[i], pz = b.z[i];
            const double qx = b.dx[i], qy = b.dy[i], qz = b.dz[i];
            pd[0][t] = px; pd[1][t] = py; pd[2][t] = pz;
            pd[3][t] = qx; pd[4][t] = qy; pd[5][t] = qz;
            asm volatile("" ::: "memory");   // read again below
            refine_pass1<kTravGrid, false>(v, FiltTab{}, GridTab{}, v.d64, px, py, pz, qx, qy, qz, [&](int c) { return pd[c][t]; },
                                           rs, best, h, nev);
        }
        const double px = pd[0][t], py = pd[1][t], pz = pd[2][t], qx = pd[3][t], qy = pd[4][t], qz = pd[5][t];
        finish_direct(v, v.d64, m64, rs, px, py, pz, qx, qy, qz, best, h, nev);
        store_result(i, b.n, best, h, px, py, pz, qx, qy, qz, step, hit, bpoint);
        if (nref) nref[i] = nev;
    }
}

// What bounds it: issue slots (80 %) at 9 of 32 lanes, since a warp walks as long
// as its longest track (22 cells, the mean is 7); FP64 41 warp instructions per
// 32 tracks (70 with one thread per track, whose unit was 67 % busy).  512
// daughters, 2^22 tracks: 1745 us with the walk to the mother's exit in the
// pipelined kernel, 754 with one thread per track, 698 here.
constexpr int kStaged = 1024;   // threads: one block per SM, its tables staged once
constexpr int kOnSheet = 128;   // tracks that a warp takes at a time

template <bool STAGED>
__global__ void __launch_bounds__(kStaged, 1)
    k_grid_sheets(const __grid_constant__ VolView v, Basket b, double* __restrict__ step, int32_t* __restrict__ hit,
                  double* __restrict__ bpoint, int32_t* __restrict__ nref) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    __shared__ ShapeRec64 m64;
    const int t = threadIdx.x;
    if (t < int(sizeof(ShapeRec64) / sizeof(double)))
        reinterpret_cast<double*>(&m64)[t] = reinterpret_cast<const double*>(&v.m64)[t];
    Sheet<kOnSheet>& w = reinterpret_cast<Sheet<kOnSheet>*>(smem_raw)[t >> 5];
    GridTab g = grid_lists(v);
    if (STAGED) {
        unsigned char* tab = smem_raw + sizeof(Sheet<kOnSheet>) * (kStaged / 32);
        const uint32_t bh = uint32_t(v.nf) * uint32_t(sizeof(FiltHvy));
        if (!stage_tables(tab, v.fhvy, bh, tab + bh, v.vox_small, v.vox_small_bytes, &bar, v.status)) return;
        g.hvy = reinterpret_cast<const FiltHvy*>(tab);
        g.cells = reinterpret_cast<const uint32_t*>(tab + bh);
        g.ids16 = reinterpret_cast<const uint16_t*>(tab + bh + v.vox_small_cells);
    }
    __syncthreads();
    // an equal share of the basket, in whole groups of 32 tracks, for every warp
    const int64_t warp = int64_t(blockIdx.x) * (kStaged / 32) + (t >> 5), warps = int64_t(gridDim.x) * (kStaged / 32);
    const int64_t groups = (b.n + 31) >> 5, end = min((groups * (warp + 1) / warps) << 5, b.n);
    for (int64_t first = (groups * warp / warps) << 5; first < end; first += kOnSheet) {
        const int count = int(min(end - first, int64_t(kOnSheet)));
        step_sheet<STAGED ? kTravGridSmall : kTravGrid, kTravGrid>(v, FiltTab{}, g, m64, w, count, b,
                                                                   [&](int k) { return first + k; }, step, hit, bpoint, nref);
    }
}

template <bool STAGED>
static cudaError_t launch_sheets(const VolView& v, const Basket& b, double* step, int32_t* hit, double* bpoint,
                               int32_t* nref, int smem, cudaStream_t s, int num_sms) {
    auto kernel = k_grid_sheets<STAGED>;
    cudaError_t e = prep(kernel, smem);
    if (e != cudaSuccess) return e;
    kernel<<<blocks_for(kernel, b.n, smem, num_sms, kStaged), kStaged, smem, s>>>(v, b, step, hit, bpoint, nref);
    return cudaGetLastError();
}

// k_grid_sheets from 1.25 waves of its tracks on, with the tables in shared memory
// if they fit (us, k_dist_grid against it: 155648 tracks, a wave, 48.8 / 60.6, 200000
// 73.9 / 65.7, 311000 85.4 / 87.6, 500000 133 / 125, 2^20 244 / 210).  Not over
// host memory: it reads a track twice.
cudaError_t launch_dist_grid(const VolView& v, const Basket& b, double* step, int32_t* hit, double* bpoint, int32_t* nref,
                             cudaStream_t s, int num_sms) {
    if (!b.link && 4 * b.n >= int64_t(num_sms) * kStaged * 5) {
        const int64_t own = int64_t(sizeof(Sheet<kOnSheet>)) * (kStaged / 32);
        const int64_t staged = own + int64_t(v.nf) * int64_t(sizeof(FiltHvy)) + int64_t(v.vox_small_bytes);
        int dev = 0, most = 0;
        if (v.vox_small && cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
            staged + 1024 <= most)
            return launch_sheets<true>(v, b, step, hit, bpoint, nref, int(staged), s, num_sms);
        return launch_sheets<false>(v, b, step, hit, bpoint, nref, int(own), s, num_sms);
    }
    k_dist_grid<<<blocks_for(k_dist_grid, b.n, 0, num_sms, kGrid), kGrid, 0, s>>>(v, b, step, hit, bpoint, nref);
    return cudaGetLastError();
}

}  // namespace geonav
