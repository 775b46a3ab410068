// queries.cu -- kernels of the FP32-filtered Contains and Safety (the
// per-point routines and the argument for their exactness are in
// queries.cuh).  One thread per point, grid-stride; the FP32 daughter table
// is staged in shared memory with the bulk-copy engine when it fits.
#include <cuda_runtime.h>

#include "launch.cuh"
#include "point_pass.cuh"
#include "queries.cuh"
#include "stage.cuh"

namespace geonav {

constexpr int kQueryTable32Max = 96 * 1024;   // bytes of FP32 records staged per block
constexpr int kQueryListsMax = 110 * 1024;    // bytes per block of the kernels over the filter's tables

// Volumes with tube segments or polycones (the others: k_contains_lists and
// k_safety_zones below; small baskets in small volumes: launch_safety_filter).
//
// Contains: per tile of 256 points, the FP32 tests run per thread and give
// each point its first candidate (the first daughter whose inflated copy
// holds it); the FP64 decisions for those candidates are binned by solid
// kind and taken by whole warps over the binned list, as in the Safety
// kernel below (the FP64 pipe charges a warp instruction whatever its active
// lanes, and a thread-per-point loop runs the FP64 test once for every
// daughter that any lane of the warp stops at).  A point whose candidate
// fails goes on with the remaining candidates on its own thread (rare).
template <bool SMEM>
__global__ void __launch_bounds__(256) k_contains32(VolView v, Basket b, int32_t* __restrict__ where) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    __shared__ double s_p[3][256];
    __shared__ int s_task[256];
    __shared__ int s_list[256];
    __shared__ unsigned char s_in[256];
    __shared__ int s_cnt[5];
    const ShapeRec32* t32 = v.d32;
    if (SMEM) {
        if (!stage_table(smem_raw, v.d32, uint32_t(v.nd) * sizeof(ShapeRec32), &bar, v.status)) return;
        t32 = reinterpret_cast<const ShapeRec32*>(smem_raw);
    }
    const int t = threadIdx.x;
    const int64_t ntiles = (b.n + 255) / 256;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t i = tile * 256 + t;
        const bool live = i < b.n;
        double p[3] = {0.0, 0.0, 0.0};
        float p32[3] = {0.f, 0.f, 0.f};
        if (live) point32(b, i, p, p32);
        int w = -2, j1 = -1;
        if (live && mother_contains<true>(v, p, p32)) {
            w = -1;
            j1 = contains_next(v, t32, p32, 0);
        }
        const int kd = j1 >= 0 ? v.d64[j1].kind : -1;
        const int bin = (kd >= 0 && kd < 5) ? kd : -1;
        s_p[0][t] = p[0];
        s_p[1][t] = p[1];
        s_p[2][t] = p[2];
        s_task[t] = j1;
        if (t < 5) s_cnt[t] = 0;
        __syncthreads();
        const int slot = bin >= 0 ? atomicAdd(&s_cnt[bin], 1) : 0;
        __syncthreads();
        int start = 0;
#pragma unroll
        for (int q = 0; q < 5; ++q)
            if (q < bin) start += s_cnt[q];
        if (bin >= 0) s_list[start + slot] = t;
        const int total = s_cnt[0] + s_cnt[1] + s_cnt[2] + s_cnt[3] + s_cnt[4];
        __syncthreads();
        for (int q = t; q < total; q += 256) {
            const int o = s_list[q];
            const double po[3] = {s_p[0][o], s_p[1][o], s_p[2][o]};
            s_in[o] = contains_daughter64<true>(v, s_task[o], po) ? 1 : 0;
        }
        __syncthreads();
        if (live) {
            if (bin >= 0) w = s_in[t] ? j1 : contains_rest<true>(v, t32, p, p32, j1);
            else if (j1 >= 0) w = contains_filter<true>(v, t32, p, p32);   // a kind outside the bins
            where[i] = w;
        }
        __syncthreads();   // the tile's shared arrays are rewritten next
    }
}

// Safety: per tile of 256 points, the FP32 pass runs per thread; the first
// FP64 evaluation of every point (its smallest-bound candidate) is then
// binned by solid kind (mother, box, tube, cone) and evaluated by whole warps
// over the binned list, so a warp mostly runs one kind's code (a warp pays
// for every code path its lanes take, and the FP64 pipe charges a warp
// instruction whatever the number of active lanes).  Each point then
// finishes on its own thread (rarely with more FP64 work).  Which warp
// evaluates a task does not change its value, so results are deterministic.
// (Two blocks per SM without spills with the segments' and polycones' code, six
// without it.)
template <bool SMEM, bool SEGS>
__global__ void __launch_bounds__(256, SEGS ? 2 : 6) k_safety32(VolView v, Basket b, double* __restrict__ saf) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    __shared__ double s_p[3][256];
    __shared__ double s_res[256];
    __shared__ int s_task[256];
    __shared__ int s_list[256];
    __shared__ int s_cnt[4];
    const ShapeRec32* t32 = v.d32;
    if (SMEM) {
        if (!stage_table(smem_raw, v.d32, uint32_t(v.nd) * sizeof(ShapeRec32), &bar, v.status)) return;
        t32 = reinterpret_cast<const ShapeRec32*>(smem_raw);
    }
    const float tau = safety_tau(v);
    const int t = threadIdx.x;
    const int64_t ntiles = (b.n + 255) / 256;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t i = tile * 256 + t;
        const bool live = i < b.n;
        double p[3] = {0.0, 0.0, 0.0};
        float p32[3] = {0.f, 0.f, 0.f};
        if (live) point32(b, i, p, p32);
        SafetyState st;
        st.Lm = st.L2 = 0.f;
        st.j1 = -1;
        const bool in = live && safety_pass1<SEGS>(v, t32, p, p32, st);
        const int bin = in ? (st.j1 < 0 ? 0 : 1 + t32[st.j1].kind) : -1;
        s_p[0][t] = p[0];
        s_p[1][t] = p[1];
        s_p[2][t] = p[2];
        s_task[t] = st.j1;
        if (t < 4) s_cnt[t] = 0;
        __syncthreads();
        const int slot = bin >= 0 ? atomicAdd(&s_cnt[bin], 1) : 0;
        __syncthreads();
        int start = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q < bin) start += s_cnt[q];
        if (bin >= 0) s_list[start + slot] = t;
        const int total = s_cnt[0] + s_cnt[1] + s_cnt[2] + s_cnt[3];
        __syncthreads();
        for (int q = t; q < total; q += 256) {
            const int o = s_list[q];
            const double po[3] = {s_p[0][o], s_p[1][o], s_p[2][o]};
            s_res[o] = safety_of<SEGS>(v, s_task[o], po);
        }
        __syncthreads();
        if (live) {
            double s = 0.0;
            if (in) {
                int nev;
                s = safety_finish<SEGS>(v, t32, p, p32, st, s_res[t], tau, &nev);
            }
            saf[i] = s;
        }
        __syncthreads();   // the tile's shared arrays are rewritten next
    }
}

// The under-estimating safety (GEO_SAFETY_ESTIMATE): the FP32 pass alone.
// Every solid's bound is its inflated (mother: deflated) FP32 copy's
// distance lowered by a relative 2^-18: box and tube the exact distance to
// the copy, cone the largest supporting half-plane distance, tube segment
// and polycone their enclosing tube, segment and polycone mothers 0; a
// daughter's bound is raised to the distance to its copy's bounding sphere
// where that is larger, so the sphere cull cannot change the minimum.  The
// minimum is a lower bound of the exact safety; no FP64 work but the
// mother's containment test where its FP32 copies cannot decide.
template <bool SMEM, bool SEGS>
__global__ void __launch_bounds__(256) k_safety_est(VolView v, Basket b, double* __restrict__ saf) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    const ShapeRec32* t32 = v.d32;
    if (SMEM) {
        if (!stage_table(smem_raw, v.d32, uint32_t(v.nd) * sizeof(ShapeRec32), &bar, v.status)) return;
        t32 = reinterpret_cast<const ShapeRec32*>(smem_raw);
    }
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < b.n; i += stride) {
        double p[3];
        float p32[3];
        point32(b, i, p, p32);
        float L = 0.f;
        if (mother_contains<SEGS>(v, p, p32)) {
            L = safety_in_lb32(v.m32, p32);
            for (int j = 0; j < v.nd && L > 0.f; ++j) {
                const ShapeRec32& r = t32[j];
                float o[3], x[3];
                const float c2 = offset32(r, p32, o);
                if (beyond(r, c2, L)) continue;   // the whole copy is farther than L
                local32(r, o, x);
                L = fminf(L, fmaxf(safety_out_lb32(r, x), sphere_lb32(r, c2)));
            }
        }
        saf[i] = double(L);
    }
}

// Volumes of boxes, tubes and cones: the lists of point_pass.cuh.  One thread
// per point, no barrier; the point's FP64 coordinates are read again in the
// rare case that FP64 has to decide.
//
// What bounds it: issue slots (75 %; 780 warp instructions per 32 points of the
// toy detector, 30 of 32 lanes active, FP64 idle).  2^22 points: 115 us, 1.0 TB/s; the
// thread-per-point walk to the first copy that holds the point with
// binned FP64 tests (k_contains32) took 271 us and 1920 instructions.
static __device__ __noinline__ bool contains_mother_cold(const VolView& v, const Basket& b, int64_t i) {
    const double p[3] = {b.x[i], b.y[i], b.z[i]};
    return contains64<false>(v.m64, p);
}
static __device__ __noinline__ bool contains_cold(const VolView& v, const Basket& b, int64_t i, int j) {
    const double p[3] = {b.x[i], b.y[i], b.z[i]};
    return contains_daughter64<false>(v, j, p);
}

// the filter's tables of the volume, staged or in global memory (false: a wait ran out)
template <bool SMEM>
__device__ __forceinline__ bool stage_filter(const VolView& v, unsigned char* smem, uint64_t* bar, FiltTab& f) {
    f = {v.fsph, v.fhvy, v.nq1, v.nq, v.nf};
    if (SMEM) {
        if (!stage_table(smem, v.fsph, uint32_t(v.nf) * uint32_t(sizeof(FiltSph) + sizeof(FiltHvy)), bar, v.status))
            return false;
        f.sph = reinterpret_cast<const FiltSph*>(smem);
        f.hvy = reinterpret_cast<const FiltHvy*>(smem + size_t(v.nf) * sizeof(FiltSph));
    }
    return true;
}

template <bool SMEM>
__global__ void __launch_bounds__(256) k_contains_lists(const __grid_constant__ VolView v, const __grid_constant__ Basket b,
                                                        int32_t* __restrict__ where) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    FiltTab f;
    if (!stage_filter<SMEM>(v, smem_raw, &bar, f)) return;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < b.n; i += stride) {
        const float p[3] = {f64_to_f32_trunc(b.x[i]), f64_to_f32_trunc(b.y[i]), f64_to_f32_trunc(b.z[i])};
        int w = -2;
        if (contains32(v.m32, p) || (contains32(v.m32u, p) && contains_mother_cold(v, b, i)))
            w = point_contains(f, p, [&](int j) { return contains_cold(v, b, i, j); });
        where[i] = w;
    }
}

// Safety: the basket is shared equally by all resident warps (toy detector, 524288
// points: 98 us with whole batches of 128 dealt in turn, 88 so; 203 and 176 for points
// on the daughters' surfaces).  Each takes up to 128 points at a time; the FP32 pass
// runs 32 of them at a time and sorts them by their FP64 work (zone_sort), which then
// runs 32 points of one sort at a time (an FP64 instruction holds its unit for 64 cycles
// however few lanes take part).  Everything is the warp's own, so there is no barrier.
//
// What bounds it: issue slots (59 %) and the FP64 unit (54 %): 2290 warp
// instructions and 38 FP64 instructions per 32 points of the toy detector.  2^21 +
// 77 points: 238 us; k_safety32, whole solids binned by kind with block barriers,
// took 514 us with 3950 and 101.
constexpr int kSafWarps = 8;
constexpr int kSafBatch = 128;
struct __align__(16) SafetyBatch {   // one warp's
    double p[3][kSafBatch];
    int task[kSafBatch];             // daughter (-1 the mother) + 1 | zone << kTagShift
    float L2[kSafBatch], L3[kSafBatch];
    int k2[kSafBatch];
    unsigned char list[kZoneSorts][kSafBatch];
};

static __device__ __noinline__ double safety_cold(const VolView& v, int j, double px, double py, double pz) {
    const double p[3] = {px, py, pz};
    return safety_of<false>(v, j, p);
}
// The points of a batch that their two nearest candidates do not settle (marked in
// k2; L2: the bound above which no candidate matters), one after the other by the whole
// warp: the least value of every candidate up to that bound, the mother or a daughter for
// each lane.  They are rare (a few in 10^5), but one lane alone took 17 us over the 40
// daughters of the toy detector, and its basket waited for it (60013 points 49 us, 27
// without such a point).
constexpr int kSafRest = -2;
static __device__ __noinline__ void safety_rest(const VolView& v, SafetyBatch& B, int per, double* saf) {
    const int lane = threadIdx.x & 31;
    for (int base = 0; base < per; base += 32) {
        const bool mine = base + lane < per && B.k2[base + lane] == kSafRest;
        for (unsigned m = __ballot_sync(0xffffffffu, mine); m; m &= m - 1) {
            const int q = base + __ffs(m) - 1;
            const double p[3] = {B.p[0][q], B.p[1][q], B.p[2][q]};
            const float p32[3] = {f64_to_f32_trunc(p[0]), f64_to_f32_trunc(p[1]), f64_to_f32_trunc(p[2])};
            const float th = B.L2[q];
            double s = d_inf();
            for (int j = lane - 1; j < v.nd; j += 32) {
                if (j >= 0) {
                    const ShapeRec32& r = v.d32[j];
                    float o[3], x[3];
                    const float c2 = offset32(r, p32, o);
                    if (beyond(r, c2, th)) continue;
                    local32(r, o, x);
                    if (safety_out_lb32(r, x) > th) continue;
                }
                s = fmin(s, safety_of<false>(v, j, p));
            }
            __syncwarp();
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s = fmin(s, __shfl_xor_sync(0xffffffffu, s, off));
            if (lane == 0) {
                saf[q] = s;
                B.k2[q] = -1;
            }
        }
    }
    __syncwarp();
}

template <bool SMEM>
__global__ void __launch_bounds__(kSafWarps * 32, 4)
    k_safety_zones(const __grid_constant__ VolView v, const __grid_constant__ Basket b, double* __restrict__ saf) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    __shared__ ShapeRec64 m64;
    FiltTab f;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t < int(sizeof(ShapeRec64) / sizeof(double)))
        reinterpret_cast<double*>(&m64)[t] = reinterpret_cast<const double*>(&v.m64)[t];
    if (!stage_filter<SMEM>(v, smem_raw + kSafWarps * sizeof(SafetyBatch), &bar, f)) return;
    __syncthreads();
    SafetyBatch& B = reinterpret_cast<SafetyBatch*>(smem_raw)[warp];
    const float tau = safety_tau(v);
    // an equal share of the basket, in whole groups of 32 points, for every warp
    const int64_t share = int64_t(blockIdx.x) * kSafWarps + warp, shares = int64_t(gridDim.x) * kSafWarps;
    const int64_t groups = (b.n + 31) >> 5, end = min((groups * (share + 1) / shares) << 5, b.n);
    for (int64_t first = (groups * share / shares) << 5; first < end; first += kSafBatch) {
        const int per = int(min(end - first, int64_t(kSafBatch)));
        int cnt[kZoneSorts] = {0, 0, 0, 0};
        for (int o = lane; o - lane < per; o += 32) {
            const int64_t i = first + o;
            int sort = -1;
            if (o < per) {
                const double px = b.x[i], py = b.y[i], pz = b.z[i];
                const float p[3] = {f64_to_f32_trunc(px), f64_to_f32_trunc(py), f64_to_f32_trunc(pz)};
                const bool surely = contains32(v.m32, p);
                int zone = kZoneInside;   // (outside the mother: 0 as well)
                if (surely || (contains32(v.m32u, p) && contains_mother_cold(v, b, i))) {
                    Nearest n;
                    n.L1 = surely ? safety_in_lb32(v.m32, p) : 0.f;
                    n.k1 = n.k2 = -1;
                    n.L2 = n.L3 = f_inf();
                    point_nearest(f, p, n);
                    const FiltHvy* h = f.hvy + max(n.k1, 0);
                    zone = n.k1 >= 0 ? entry_zone(h, p) : (surely ? mother_zone(v, p) : kZoneNone);
                    if (zone != kZoneInside) {
                        B.p[0][o] = px; B.p[1][o] = py; B.p[2][o] = pz;
                        B.task[o] = (n.k1 >= 0 ? h->id + 1 : 0) | (zone << kTagShift);
                        B.L2[o] = n.L2;
                        B.L3[o] = n.L3;
                        B.k2[o] = n.k2;
                        // (32 points are not worth several runs)
                        sort = per > 32 || zone == kZoneNone ? zone_sort(zone) : 0;
                    }
                }
                if (zone == kZoneInside) {
                    saf[i] = 0.0;
                    B.k2[o] = -1;
                }
            }
#pragma unroll
            for (int s = 0; s < kZoneSorts; ++s) {
                const unsigned same = __ballot_sync(0xffffffffu, sort == s);
                if (sort == s) B.list[s][cnt[s] + __popc(same & ((1u << lane) - 1u))] = (unsigned char)o;
                cnt[s] += __popc(same);
            }
        }
        __syncwarp();
        bool rest = false;
        // 32 points of one sort at a time (one copy of the code: c counts up through the sorts)
        for (int sort = 0, c = 0; sort < kZoneSorts;) {
            const int n = sort == 0 ? cnt[0] : (sort == 1 ? cnt[1] : (sort == 2 ? cnt[2] : cnt[3]));
            if (c >= n) {
                ++sort;
                c = 0;
                continue;
            }
            if (c + lane < n) {
                const int o = B.list[sort][c + lane];
                const int w = B.task[o], j = (w & kIdMask) - 1, zone = w >> kTagShift;
                const double px = B.p[0][o], py = B.p[1][o], pz = B.p[2][o];
                double r;
                if (zone != kZoneNone) r = zone64(j < 0 ? m64 : v.d64[j], zone, j < 0, px, py, pz);
                else r = safety_cold(v, j, px, py, pz);
                if (!(B.L2[o] > above(r, tau))) {
                    const int k2 = B.k2[o];
                    r = fmin(r, safety_cold(v, k2 < 0 ? -1 : f.hvy[k2].id, px, py, pz));
                    if (!(B.L3[o] > above(r, tau))) {
                        B.k2[o] = kSafRest;
                        B.L2[o] = above(r, tau);
                        rest = true;
                    }
                }
                saf[first + o] = r;
            }
            __syncwarp();
            c += 32;
        }
        if (__any_sync(0xffffffffu, rest)) safety_rest(v, B, per, saf + first);
    }
}

template <typename K1, typename K0, typename... A>
static cudaError_t launch_lists(K1 staged, K0 global, int fixed, const VolView& v, const Basket& b, cudaStream_t s,
                                int num_sms, A... args) {
    const int64_t bytes = int64_t(v.nf) * int64_t(sizeof(FiltSph) + sizeof(FiltHvy));
    // two blocks' tables per SM at least
    if (bytes + fixed <= kQueryListsMax) {
        const int smem = fixed + int(bytes);
        cudaError_t e = prep(staged, smem);
        if (e != cudaSuccess) return e;
        staged<<<blocks_for(staged, b.n, smem, num_sms), 256, smem, s>>>(v, b, args...);
    } else {
        cudaError_t e = prep(global, fixed);
        if (e != cudaSuccess) return e;
        global<<<blocks_for(global, b.n, fixed, num_sms), 256, fixed, s>>>(v, b, args...);
    }
    return cudaGetLastError();
}

// the FP32 table staged when it fits; the polycone's code only for volumes
// holding segments or polycones
template <typename K1, typename K0, typename... A>
static cudaError_t launch32(K1 staged, K0 global, const VolView& v, const Basket& b, cudaStream_t s, int num_sms,
                            A... args) {
    const int bytes = v.nd * int(sizeof(ShapeRec32));
    if (bytes <= kQueryTable32Max) {
        cudaError_t e = prep(staged, bytes);
        if (e != cudaSuccess) return e;
        staged<<<blocks_for(staged, b.n, bytes, num_sms), 256, bytes, s>>>(v, b, args...);
    } else {
        global<<<blocks_for(global, b.n, 0, num_sms), 256, 0, s>>>(v, b, args...);
    }
    return cudaGetLastError();
}

cudaError_t launch_contains_filter(const VolView& v, const Basket& b, int32_t* where, cudaStream_t s,
                                   int num_sms) {
    if (v.segs) return launch32(k_contains32<true>, k_contains32<false>, v, b, s, num_sms, where);
    return launch_lists(k_contains_lists<true>, k_contains_lists<false>, 0, v, b, s, num_sms, where);
}

cudaError_t launch_safety_estimate(const VolView& v, const Basket& b, double* saf, cudaStream_t s, int num_sms) {
    if (v.segs) return launch32(k_safety_est<true, true>, k_safety_est<false, true>, v, b, s, num_sms, saf);
    return launch32(k_safety_est<true, false>, k_safety_est<false, false>, v, b, s, num_sms, saf);
}

cudaError_t launch_safety_filter(const VolView& v, const Basket& b, double* saf, cudaStream_t s, int num_sms) {
    if (v.segs) return launch32(k_safety32<true, true>, k_safety32<false, true>, v, b, s, num_sms, saf);
    // few points near few solids: a block's warps take one kind of solid each,
    // which is the shorter chain (16384 points: four boxes 5.9 us against 7.1
    // with k_safety_zones, eight solids of the toy detector 16.0 against 17.3;
    // from 100000 points on 10.7 / 10.8 and 27.6 / 24.2; 40 solids 36.8 / 20.5)
    if (v.nd <= 8 && b.n <= 32768) return launch32(k_safety32<true, false>, k_safety32<false, false>, v, b, s, num_sms, saf);
    return launch_lists(k_safety_zones<true>, k_safety_zones<false>, kSafWarps * int(sizeof(SafetyBatch)), v, b, s, num_sms,
                        saf);
}

}  // namespace geonav
