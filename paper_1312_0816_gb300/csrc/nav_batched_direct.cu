// nav_batched_direct.cu -- the batched persistent launch for volumes of boxes,
// tubes and cones: tiles of many logical volumes, claimed in order from a
// device counter (largest estimated cost first when the host sorted them so).
//
// A warp claims a part of a tile, runs the FP32 pass on its tracks and then their
// FP64 in groups of one sort (sheet.cuh): no warp ever waits for another.  The volume's view and
// tables are read through L1.
//
// What bounds it: latency of the lanes' record gathers through L1 (a third of
// the warps' time) with issue slots at 62 % and the FP64 unit at 51 %.  64
// volumes of 4 to 200 daughters, 2^22 tracks: 675 us with producer and consumer warps over
// tables staged per tile, 617 us here (parts of 192 tracks 630, of 64 644).  Tracks that
// start on a daughter's surface, where FP32 is certain of nothing, are the exception:
// 524288 of them in the toy detector 276 us with the producers' lists, 405 here, where
// about half of them take the FP32 pass twice (refine_again).
#include <cuda_runtime.h>

#include "geo_internal.h"
#include "launch.cuh"
#include "nav_common.cuh"
#include "nav_refine.cuh"
#include "sheet.cuh"

namespace geonav {

constexpr int kPart = 128;                            // tracks of a sheet
constexpr int kBatchThreads = 128, kBatchBlocks = 7;   // 72 registers

// VOX: a volume of the batch has a uniform grid, which is walked.
template <bool VOX>
__global__ void __launch_bounds__(kBatchThreads, kBatchBlocks)
    k_batched_direct(BatchView bv, Basket b, double* __restrict__ step, int32_t* __restrict__ hit, unsigned parts,
                     int size) {
    __shared__ Sheet<kPart> sheets[kBatchThreads / 32];
    const int lane = threadIdx.x & 31;
    Sheet<kPart>& w = sheets[threadIdx.x >> 5];
    for (;;) {
        unsigned claim = 0;
        if (lane == 0) claim = atomicAdd(bv.counter, 1u);
        claim = __shfl_sync(0xffffffffu, claim, 0);
        const unsigned q = claim / parts;
        if (int64_t(q) >= bv.ntiles) break;
        const BatchTile tl = bv.tiles[q];
        const int skip = int(claim - q * parts) * size;
        const bool packed = tl.count < 0;
        const int count = min((packed ? -tl.count : tl.count) - skip, size);
        const int64_t base = tl.base + skip;
        const VolView& v = bv.vols[tl.vol];
        const FiltTab f = {v.fsph, v.fhvy, v.nq1, v.nq, v.nf};
        constexpr int kTrav = VOX ? kTravEither : kTravAll;
        step_sheet<kTrav, kTrav>(
            v, f, GridTab{}, v.m64, w, count, b,
            [&](int k) -> int64_t {
                const int64_t i = packed ? bv.idx[base + k] : base + k;
                if (i >= 0 && i < b.n) return i;
                atomicOr(bv.status, ST_BAD_INDEX);   // a stale or corrupt tile list: skip, and say so
                atomicOr(v.status, ST_BAD_INDEX);
                return -1;
            },
            step, hit, nullptr, nullptr);
    }
}

template <bool VOX>
static cudaError_t launch(const BatchView& bv, const Basket& b, double* step, int32_t* hit, int blocks_per_sm, int tile_tracks,
                          cudaStream_t s, int num_sms) {
    const int most = resident_blocks(reinterpret_cast<const void*>(k_batched_direct<VOX>), kBatchThreads, 0);
    // the caller's limit counts blocks of 512 threads (k_dist_batched's): four of
    // these each, so that two are the whole SM for either kernel
    const int per_sm = (blocks_per_sm <= 0 || 4 * int64_t(blocks_per_sm) > most) ? most : 4 * blocks_per_sm;
    // Parts of 128 tracks sort best, but a warp takes 80 us for one: while there are
    // fewer than two for each warp, smaller ones (us for parts of 32 / 64 / 128, 64 volumes:
    // 4096 tracks 45 / 60 / 83, 300000 85 / 89 / 117, 600000 124 / 118 / 138,
    // 1.2e6 218 / 207 / 198).
    const int64_t warps = int64_t(per_sm) * num_sms * (kBatchThreads / 32), tracks = bv.ntiles * tile_tracks;
    const int size = tracks >= warps * 2 * kPart ? kPart : (tracks >= warps * kPart ? kPart / 2 : 32);
    k_batched_direct<VOX><<<per_sm * num_sms, kBatchThreads, 0, s>>>(bv, b, step, hit,
                                                                     unsigned((tile_tracks + size - 1) / size), size);
    return cudaGetLastError();
}

cudaError_t launch_batched_direct(const BatchView& bv, const Basket& b, double* step, int32_t* hit, int blocks_per_sm,
                                  int tile_tracks, cudaStream_t s, int num_sms) {
    return bv.vox ? launch<true>(bv, b, step, hit, blocks_per_sm, tile_tracks, s, num_sms)
                  : launch<false>(bv, b, step, hit, blocks_per_sm, tile_tracks, s, num_sms);
}

}  // namespace geonav
