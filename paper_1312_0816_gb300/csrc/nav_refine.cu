// nav_refine.cu -- the navigator step of Fig. 1b with an FP32 filter and FP64
// refinement (GEO_FP32_REFINE): dispatch, the batched launch.
//
// Pass 1 (FP32, every daughter; filter_pass.cuh): a LOWER bound L_j of
// DistFromOutside from each daughter's inflated FP32 copy that the track comes
// near before the mother's exit (upper bound U), and where it is certain the
// surface the track enters through.  The kCand = 2 smallest bounds are kept in
// registers, sorted.
// Pass 2 (FP64, one surface or few solids): candidates are refined in ascending
// order of their bounds, the mother (bound L_m of its exit) taking its place in
// that order, with the operations of the plain kernel's routines; refinement
// stops as soon as the next bound exceeds the best FP64 step.  Ties resolve as
// in the sequential algorithm of Fig. 1a (mother, then lowest index).  If a
// bound that had to be dropped from the list could still win, the track falls
// back to the full FP64 loop.  Every track therefore gets exactly the plain
// FP64 kernel's answer.
#include <cuda_runtime.h>

#include <algorithm>

#include "geo_internal.h"
#include "launch.cuh"
#include "nav_common.cuh"
#include "nav_refine.cuh"
#include "stage.cuh"
#include "refine_kernel.cuh"

namespace geonav {

size_t refine_stage_bytes() { return 2 * (sizeof(Stage<kProd>) + sizeof(Answers<kProd>)); }

// ---------------------------------------------------------------------------
// Batched persistent launch of volumes with a tube segment, a polycone or a cone
// with an apex among them: tiles of many logical volumes, claimed in order
// from a device counter (largest estimated cost first when the host sorted
// them so), with the same producer / consumer pipeline.  The tile header of a
// stage carries a copy of the tile's volume view.  The filter's tables of a
// tile's volume are copied to shared memory (bulk copy): the lanes gather
// records of different solids from them, which through L1 costs a tag lookup
// for each (64 volumes, 4 to 200 daughters, 2^22 tracks: 1277 us with the tables
// read through L1 and every bound run for the union of a warp's lanes, 675 us
// so).  The
// tables of even tiles sit at the bottom of the table area, those of odd tiles
// at its top; the next tile is claimed, and its tables are copied, while the
// current one is bounded when both fit side by side, and otherwise once every
// producer is done with the current tables.  The FP64 records are read through
// L1 (each track reads one).  A packed tile (negative count) lists its
// tracks' indices in bv.idx from its base on (the ragged tails of a volume's
// baskets gathered into full tiles).
//
// A wait that runs out is recorded and never followed by a read of what it waited
// for: tracks whose tables did not arrive take the whole FP64 routines, as do those
// of the block's later tiles, and a stage whose consumers did not finish is left
// to them (the block ends).
struct __align__(16) TileHdr {
    VolView vol;
    int64_t base;
    int count;
    int tile;   // -1: the queue is empty
    int vol_index;
    int staged;          // the tile's tables were sent to the table area
    int pad[2];
};

// the next tile, as claimed by producer thread 0 (which alone uses it)
struct NextTile {
    int64_t base;
    int tile, count, vol_index;
    int staged;          // its tables go to the table area
    uint32_t bytes;      // of its filter tables
    int pending;         // 1: their copy is not issued yet
    const void* src;
    int staging;         // tiles' tables are still copied
    uint32_t owed;       // bit p: a copy on tabs[p] that was not seen to end (bit 2 + p: its parity)
};

// GLOB = false: no volume has a uniform grid and every volume's filter tables
// fit the table area (`room` bytes); the kernel carries only the all-daughter
// FP32 pass over staged tables (10 % faster on the 64-volume batch than with
// the grid walk's code beside it).  GLOB = true: the tables are read from
// global memory, a volume's grid is walked where it has one.  P producer
// threads (one track each of a tile of P) and C consumer threads.
template <bool GLOB, int P, int C>
__global__ void __launch_bounds__(P + C, 2) k_dist_batched(BatchView bv, Basket b, double* __restrict__ step,
                                                              int32_t* __restrict__ hit, uint32_t room) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t full[2], done[2], tabs[2];
    __shared__ NextTile N;
    Stage<P>* S = reinterpret_cast<Stage<P>*>(smem_raw);
    TileHdr* H = reinterpret_cast<TileHdr*>(smem_raw + 2 * sizeof(Stage<P>));
    unsigned char* area = smem_raw + 2 * (sizeof(Stage<P>) + sizeof(TileHdr));
    const int t = threadIdx.x;
    const int lane = t & 31;
    bool healthy = true;
    if (t == 0) {
        N.staging = !GLOB;
        N.owed = 0;
        mbar_init(&full[0], P / 32);
        mbar_init(&full[1], P / 32);
        mbar_init(&done[0], C / 32);
        mbar_init(&done[1], C / 32);
        mbar_init(&tabs[0], 1);
        mbar_init(&tabs[1], 1);
    }
    __syncthreads();
    constexpr int kWords = int(sizeof(VolView) / sizeof(int4));

    if (t < P) {
        // ------------------------------------------------------ producers --
        // thread 0: copy of N's tables for tile k of this block
        auto copy_tables = [&](int k) {
            unsigned char* dst = (k & 1) ? area + (room - N.bytes) : area;
            if (N.bytes == 0) {
                mbar_arrive(&tabs[k & 1]);
            } else {
                mbar_expect_tx(&tabs[k & 1], N.bytes);
                for (uint32_t off = 0; off < N.bytes; off += kChunk)
                    bulk_g2s(dst + off, static_cast<const unsigned char*>(N.src) + off, min(kChunk, N.bytes - off),
                             &tabs[k & 1]);
            }
            N.pending = 0;
        };
        // thread 0: claims this block's tile k; its tables are copied now when
        // they fit beside the `used` bytes of the tile before
        auto claim = [&](int k, uint32_t used) {
            const unsigned q = atomicAdd(bv.counter, 1u);
            N.pending = 0;
            N.staged = 0;
            N.bytes = 0;
            if (int64_t(q) < bv.ntiles) {
                const BatchTile tl = bv.tiles[q];
                N.tile = int(q);
                N.base = tl.base;
                N.count = tl.count;
                N.vol_index = tl.vol;
                if (!GLOB && N.staging) {
                    N.staged = 1;
                    const VolView& nv = bv.vols[tl.vol];
                    N.bytes = uint32_t(nv.nf) * uint32_t(sizeof(FiltSph) + sizeof(FiltHvy));
                    N.src = nv.fsph;
                    if (used + N.bytes <= room) copy_tables(k);
                    else N.pending = 1;
                }
            } else {
                N.tile = -1;
            }
        };
        if (t == 0) claim(0, 0);
        for (int k = 0;; ++k) {
            Stage<P>& st_ = S[k & 1];
            TileHdr& hd = H[k & 1];
            // the stage and its header held tile k-2, which its consumers must
            // have finished
            if (k >= 2) mbar_wait_bounded(&done[k & 1], uint32_t(((k - 2) >> 1) & 1), bv.status, healthy);
            if (t == 0) {
                hd.tile = healthy ? N.tile : -1;
                if (healthy) {
                    hd.base = N.base;
                    hd.count = N.count;
                    hd.vol_index = N.vol_index;
                    hd.staged = N.staged;
#pragma unroll
                    for (int q = 0; q < kTaskBins; ++q) st_.cnt[q] = 0;
                    st_.next = 0;
                } else if (N.staged) {
                    N.owed |= (1u | uint32_t((k >> 1) & 1) << 2) << (k & 1);
                }
            }
            producer_barrier<P>();
            const int tile = hd.tile;
            if (tile >= 0) {
                if (t < kWords)
                    reinterpret_cast<int4*>(&hd.vol)[t] = reinterpret_cast<const int4*>(bv.vols + hd.vol_index)[t];
                const int64_t base = hd.base;
                const bool packed = hd.count < 0;
                const int count = packed ? -hd.count : hd.count;
                if (t == 0) claim(k + 1, N.bytes);
                producer_barrier<P>();
                const VolView& v = hd.vol;
                FiltTab f = {v.fsph, v.fhvy, v.nq1, v.nq, v.nf};
                if (!GLOB) {
                    // every tile's copy is waited for, so none is in flight when the block ends
                    if (!hd.staged) {
                        hd.vol.dd_min = f_inf();   // no direction is long enough for the FP32 pass
                    } else if (!mbar_wait_limited(&tabs[k & 1], uint32_t((k >> 1) & 1), bv.table_polls)) {
                        hd.vol.dd_min = f_inf();
                        atomicOr(bv.status, ST_TMA_TIMEOUT);
                        atomicOr(v.status, ST_TMA_TIMEOUT);
                        if (t == 0) {
                            N.staging = 0;
                            N.owed |= (1u | uint32_t((k >> 1) & 1) << 2) << (k & 1);
                        }
                    }
                    const unsigned char* tab =
                        (k & 1) ? area + (room - uint32_t(v.nf) * uint32_t(sizeof(FiltSph) + sizeof(FiltHvy))) : area;
                    f.sph = reinterpret_cast<const FiltSph*>(tab);
                    f.hvy = reinterpret_cast<const FiltHvy*>(tab + size_t(v.nf) * sizeof(FiltSph));
                }
                bool live = t < count;
                int64_t i = live ? (packed ? bv.idx[base + t] : base + t) : 0;
                if (live && (i < 0 || i >= b.n)) {   // a stale or corrupt tile list: skip, and say so
                    atomicOr(bv.status, ST_BAD_INDEX);
                    atomicOr(v.status, ST_BAD_INDEX);
                    live = false;
                    i = 0;
                }
                double px = 0, py = 0, pz = 0, qx = 1, qy = 0, qz = 0;
                if (live) {
                    px = b.x[i]; py = b.y[i]; pz = b.z[i];
                    qx = b.dx[i]; qy = b.dy[i]; qz = b.dz[i];
                }
                st_.pd[0][t] = px; st_.pd[1][t] = py; st_.pd[2][t] = pz;
                st_.pd[3][t] = qx; st_.pd[4][t] = qy; st_.pd[5][t] = qz;
                asm volatile("" ::: "memory");   // the FP64 paths of the FP32 pass read the stage again
                RefineState rs;
                double best = 0.0;
                int h = -2, nev = 0;
                rs.status = 1;
                if (live)
                    refine_pass1<GLOB ? kTravEither : kTravAll>(v, f, GridTab{}, v.d64, px, py, pz, qx, qy, qz,
                                                                [&](int c) { return st_.pd[c][t]; }, rs, best, h, nev);
                int task = 0, bin = -1;
                if (rs.status == 0) {
                    task = first_task(rs);
                    bin = task_bin(rs.tag, task, v.d64);
                }
                const int slot = bin >= 0 ? atomicAdd(&st_.cnt[bin], 1) : 0;
                producer_barrier<P>();
                if (!GLOB && t == 0 && N.pending) {   // nobody reads the current tables any more
                    if (N.staging) copy_tables(k + 1);
                    else N.staged = 0;
                }
                if (bin >= 0) st_.task[bin_start(st_.cnt, bin) + slot] = t | ((task + 1) << kOwnerBits);
                pad_bins<P>(st_, t);
                if (rs.status == 0) {
#pragma unroll
                    for (int q = 0; q < kCand; ++q) {
                        st_.L[q][t] = rs.c.L[q];
                        st_.j[q][t] = rs.c.j[q];
                    }
                    st_.Lm[t] = rs.Lm;
                    st_.dropped[t] = rs.c.dropped;
                    st_.n[t] = rs.c.n | rs.tag << 8;
                } else if (live) {
                    store_result(i, b.n, best, h, px, py, pz, qx, qy, qz, step, hit, nullptr);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[k & 1]);
            if (tile < 0) break;
        }
        if (t == 0 && N.owed) {
            for (int q = 0; q < bv.nvols; ++q) atomicOr(bv.vols[q].status, ST_TMA_TIMEOUT);
            // do not leave while a late copy may still write this block's memory
            for (int p = 0; p < 2; ++p)
                if (N.owed >> p & 1u) mbar_wait_limited(&tabs[p], N.owed >> (2 + p) & 1u, kWaitLimit);
        }
    } else {
        // ------------------------------------------------------ consumers --
        for (int k = 0;; ++k) {
            Stage<P>& st_ = S[k & 1];
            TileHdr& hd = H[k & 1];
            mbar_wait_bounded(&full[k & 1], uint32_t((k >> 1) & 1), bv.status, healthy);
            // warp-uniform; all consumer warps see the same tile
            if (!__all_sync(0xffffffffu, healthy) || hd.tile < 0) break;
            const VolView& v = hd.vol;
            const int64_t base = hd.base;
            const bool packed = hd.count < 0;
            const int64_t* idx = bv.idx;
            // the outputs are in device memory: each track is stored as it is
            // finished (staging the tile's answers was 4 % slower here)
            drain_tasks<P, false>(v, v.d64, v.m64, st_, nullptr, [=](int o) { return packed ? idx[base + o] : base + o; },
                                        b.n, step, hit);
            __syncwarp();
            if (lane == 0) mbar_arrive(&done[k & 1]);
        }
    }
    // a wait that ran out is also reported in every volume's status word,
    // which geo_check_device_status reads
    if (!healthy)
        for (int q = 0; q < bv.nvols; ++q) atomicOr(bv.vols[q].status, ST_SYNC_TIMEOUT);
}

// A bounded wait that runs out: one warp waits, with `polls` polls of the
// pipeline's own wait (mbar_wait_limited), on an mbarrier that no thread
// arrives at, then records ST_SYNC_TIMEOUT in the status word and returns
// (the failure path of every wait of the pipeline, exercised on purpose by
// the tests).
__global__ void k_wait_selftest(unsigned int* status, uint32_t polls) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) mbar_init(&bar, 1);
    __syncthreads();
    if (mbar_wait_limited(&bar, 0, polls)) return;
    if (threadIdx.x == 0) atomicOr(status, ST_SYNC_TIMEOUT);
}

cudaError_t launch_wait_selftest(unsigned int* status, uint32_t polls, cudaStream_t s) {
    k_wait_selftest<<<1, 32, 0, s>>>(status, polls);
    return cudaGetLastError();
}

// shared memory of one SM and of one block
static void smem_limits(int* per_sm, int* per_block) {
    int dev = 0, a = 0, c = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&a, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&c, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        a = c = 48 * 1024;
    }
    *per_sm = a;
    *per_block = c;
}

// The table area of a batch: two tables of its largest volume, or what half an
// SM's shared memory leaves beside the stages (two blocks per SM); 0 when that
// does not hold the largest volume's.
template <int P>
static uint32_t table_room(int max_nf) {
    const int fixed = 2 * int(sizeof(Stage<P>) + sizeof(TileHdr));
    int per_sm, per_block;
    smem_limits(&per_sm, &per_block);
    const int64_t avail = std::min(per_sm / 2 - 2048, per_block - 1024) - fixed;
    const int64_t one = int64_t(max_nf) * int64_t(sizeof(FiltSph) + sizeof(FiltHvy));
    if (one > avail) return 0;
    return uint32_t(std::max<int64_t>(std::min(2 * one, avail) & ~int64_t(15), 16));
}

template <bool GLOB, int P, int C>
static cudaError_t launch_batched(const BatchView& bv, const Basket& b, double* step, int32_t* hit, int blocks_per_sm,
                                  uint32_t room, cudaStream_t s, int num_sms) {
    const int smem = 2 * int(sizeof(Stage<P>) + sizeof(TileHdr)) + (GLOB ? 0 : int(room));
    cudaError_t e = prep(k_dist_batched<GLOB, P, C>, smem);
    if (e != cudaSuccess) return e;
    const int maxb = resident_blocks(reinterpret_cast<const void*>(k_dist_batched<GLOB, P, C>), P + C, smem);
    const int per_sm = (blocks_per_sm <= 0 || blocks_per_sm > maxb) ? maxb : blocks_per_sm;
    k_dist_batched<GLOB, P, C><<<per_sm * num_sms, P + C, smem, s>>>(bv, b, step, hit, room);
    return cudaGetLastError();
}

template <int P, int C>
static cudaError_t launch_batched_shape(const BatchView& bv, const Basket& b, double* step, int32_t* hit,
                                        int blocks_per_sm, cudaStream_t s, int num_sms) {
    const uint32_t room = bv.vox ? 0 : table_room<P>(bv.max_nf);
    return room == 0 ? launch_batched<true, P, C>(bv, b, step, hit, blocks_per_sm, room, s, num_sms)
                     : launch_batched<false, P, C>(bv, b, step, hit, blocks_per_sm, room, s, num_sms);
}

// Volumes of boxes, tubes and cones take the kernel without producers and
// consumers (nav_batched_direct.cu).  For the others two tile shapes, the autotuner's choice per batch: tiles of kTileTracks =
// 384 tracks with 12 producer + 4 consumer warps, or tiles of 256 with 8 + 4.
cudaError_t launch_dist_batched(const BatchView& bv, const Basket& b, double* step, int32_t* hit, int blocks_per_sm,
                                int tile_tracks, cudaStream_t s, int num_sms) {
    static_assert(sizeof(TileHdr) % 16 == 0 && sizeof(VolView) % 16 == 0, "16-byte copies");
    if (!bv.segs) return launch_batched_direct(bv, b, step, hit, blocks_per_sm, tile_tracks, s, num_sms);
    if (tile_tracks == kLatProd)
        return launch_batched_shape<kLatProd, kLatCons>(bv, b, step, hit, blocks_per_sm, s, num_sms);
    return launch_batched_shape<kProd, kCons>(bv, b, step, hit, blocks_per_sm, s, num_sms);
}

// A small basket in a volume of many daughters takes the split kernel
// (split_basket()); otherwise volumes of boxes, tubes and cones without a grid
// take the direct kernel whatever the size (against the pipelined kernel: toy
// detector 19457 tracks 29.1 -> 21.8 us, 2^20 218 -> 138 us; with a
// grid nav_refine_grid.cu), and
// the others the pipelined one: its latency configuration for a basket of at
// most two tiles of 256 tracks per resident block (two blocks per SM), else its
// throughput configuration (measured on the toy detector, when it took this
// kernel: 65536 tracks 43.8 us instead of 59.1 us, from 196608 tracks on equal).
cudaError_t launch_dist_refine_stats(const VolView& v, const Basket& b, double* step, int32_t* hit,
                                     double* bpoint, int32_t* nref, cudaStream_t s, int num_sms) {
    if (split_basket(v, b.n, num_sms)) return launch_dist_refine_split(v, b, step, hit, bpoint, nref, s);
    if (!v.segs) return launch_dist_direct(v, b, step, hit, bpoint, nref, s, num_sms);
    if (b.n <= int64_t(4) * num_sms * kLatProd)
        return launch_dist_refine_latency(v, b, step, hit, bpoint, nref, s, num_sms);
    return launch_refine_cfg<kProd, kCons>(v, b, step, hit, bpoint, nref, s, num_sms);
}

// Small baskets take the warp-per-track FP64 kernel (the same answers: both
// modes return the plain FP64 bits); the filter pays off only when its
// threads are many.
cudaError_t launch_dist_refine(const VolView& v, const Basket& b, double* step, int32_t* hit, double* bpoint,
                               cudaStream_t s, int num_sms) {
    if (small_basket(v, b.n, num_sms)) return launch_dist_warp(v, b, step, hit, bpoint, s, num_sms);
    return launch_dist_refine_stats(v, b, step, hit, bpoint, nullptr, s, num_sms);
}

}  // namespace geonav
