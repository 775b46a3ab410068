// sheet.cuh -- the filter step of a warp's tracks, with FP64 in groups of one
// sort.
//
// An FP64 instruction holds its unit for 64 cycles however few lanes take
// part, and a plane needs 20 of them, a rotated quadric 60: a warp whose 32
// tracks are of both sorts pays for both.  So a warp runs the FP32 pass on up
// to Q tracks first, keeps each track's first task and the least bound beside
// it (8 bytes), and then evaluates them 32 at a time, the quadrics first, then
// the planes (512 rotated solids: 41 FP64 instructions per 32 tracks instead of
// 70).  All of it is the warp's own: no barrier of the block.  The FP64 track is read
// again from the basket (it is still in L2, and its latency is small beside
// the FP32 pass).  Where nearly all surfaces are quadrics there is nothing to
// gain: the toy detector keeps one thread per track (141 us; 146 us so).
#pragma once
#include "nav_refine.cuh"

namespace geonav {

template <int Q>
struct Sheet {
    static_assert(Q % 32 == 0 && Q <= 256, "the order's entries are bytes");
    int task[Q];        // index + 1 (0: the mother) | tag << kTagShift; kTaskNone: nothing (left) to do
    float rest[Q];      // the least bound beside the task's
    uint8_t order[Q];   // quadrics from the front, planes and uncertain tracks from the back
};
constexpr int kTaskNone = -1;

// A track that its first task (solid h, value s) does not settle (0.02 %, out of
// line): the FP32 pass again, for its whole list of candidates.  This copy of the
// pass may round a bound differently (the compiler contracts each copy's expressions
// by itself) and name another first task; the loop over every daughter then
// decides.  (Two more candidates kept per track instead: the grid 709 us for 700.)
template <int TRAV>
static __device__ __noinline__ void refine_again(const VolView& v, double& s, double px, double py, double pz, double qx,
                                                 double qy, double qz, int& h, int& nev) {
    const double pd[6] = {px, py, pz, qx, qy, qz};
    const int first = h;
    const double s_first = s;
    RefineState rs;
    refine_pass1<TRAV, false>(v, FiltTab{v.fsph, v.fhvy, v.nq1, v.nq, v.nf}, GridTab{}, v.d64, px, py, pz, qx, qy, qz,
                              [&](int c) { return pd[c]; }, rs, s, h, nev);
    if (rs.status != 0) return;
    if (first_task(rs) != first) rs.c.dropped = 0.f;   // below any value
    refine_rest<false>(v, v.d64, rs, s_first, px, py, pz, qx, qy, qz, s, h, nev);
}

// The step of the tracks at(0) .. at(count - 1), count <= Q, by one warp.  at(k) < 0: no
// track.  TRAV: the FP32 pass (f, g: its tables); AGAIN: the same over the tables in global memory.
template <int TRAV, int AGAIN, int Q, class At>
__device__ __forceinline__ void step_sheet(const VolView& v, const FiltTab& f, const GridTab& g, const ShapeRec64& m64,
                                           Sheet<Q>& w, int count, const Basket& b, At at, double* step, int32_t* hit,
                                           double* bpoint, int32_t* nref) {
    const int lane = threadIdx.x & 31;
    const unsigned all = 0xffffffffu, below = (1u << lane) - 1u;
#pragma unroll 1
    for (int k = lane; k - lane < count; k += 32) {
        w.task[k] = kTaskNone;
        const int64_t i = k < count ? at(k) : -1;
        if (i >= 0) {
            RefineState rs;
            double best = 0.0;
            int h = -2, nev = 0;
            refine_pass1<TRAV, false>(
                v, f, g, v.d64, b.x[i], b.y[i], b.z[i], b.dx[i], b.dy[i], b.dz[i],
                [&](int c) { return (c == 0 ? b.x : c == 1 ? b.y : c == 2 ? b.z : c == 3 ? b.dx : c == 4 ? b.dy : b.dz)[i]; },
                rs, best, h, nev);
            if (rs.status == 0) {
                const int j = first_task(rs);
                w.task[k] = (j + 1) | rs.tag << kTagShift;
                w.rest[k] = fminf(rs.c.dropped, fminf(rs.c.L[1], j < 0 ? rs.c.L[0] : rs.Lm));
            } else {
                store_result(i, b.n, best, h, b.x[i], b.y[i], b.z[i], b.dx[i], b.dy[i], b.dz[i], step, hit, bpoint);
                if (nref) nref[i] = nev;
            }
        }
    }
    __syncwarp();
    int quads = 0, planes = 0;
#pragma unroll 1
    for (int k = lane; k - lane < count; k += 32) {
        const int tk = w.task[k], tag = tk >> kTagShift;
        const bool quad = tk >= 0 && (tag == kTagOuter || tag == kTagInner), plane = tk >= 0 && !quad;
        const unsigned mq = __ballot_sync(all, quad), mp = __ballot_sync(all, plane);
        if (quad) w.order[quads + __popc(mq & below)] = uint8_t(k);
        if (plane) w.order[Q - 1 - planes - __popc(mp & below)] = uint8_t(k);
        quads += __popc(mq);
        planes += __popc(mp);
    }
    __syncwarp();
    // one sequence: the group in which the quadrics end is filled up with planes
#pragma unroll 1
    for (int e = lane; e < quads + planes; e += 32) {
        const int k = w.order[e < quads ? e : Q - 1 - (e - quads)], tk = w.task[k];
        const int j = (tk & kIdMask) - 1, tag = tk >> kTagShift;
        const int64_t i = at(k);
        const double px = b.x[i], py = b.y[i], pz = b.z[i];
        const double qx = b.dx[i], qy = b.dy[i], qz = b.dz[i];
        double s = tag != kTagNone ? surface64(j < 0 ? m64 : v.d64[j], tag, j < 0, px, py, pz, qx, qy, qz)
                                   : eval64_cold(v, v.d64, j, px, py, pz, qx, qy, qz);
        int h = j, nev = 1;
        // refine_fast()'s rule
        if (!(LT(s, d_inf()) && w.rest[k] > f64_to_f32_up(s))) refine_again<AGAIN>(v, s, px, py, pz, qx, qy, qz, h, nev);
        store_result(i, b.n, s, h, px, py, pz, qx, qy, qz, step, hit, bpoint);
        if (nref) nref[i] = nev;
    }
    __syncwarp();
}

}  // namespace geonav
