// What the wavefront kernels over 4 x 3-line tiles share (the FP64 sweeps and
// the factorisation): the barriers that open a level and the counters between
// the warps of a CTA.
#pragma once
#include "tiles.cuh"

namespace bo {

constexpr int LINES = TSJ * TSK;          // x-lines of a tile
constexpr int RING = 8;                   // levels of the shared-memory rings (power of two)
constexpr int FACE_WARPS = 4;             // warps that open the levels, each every fourth
constexpr int WAIT_LIMIT = 1 << 26;       // polls of a level counter (several seconds)
constexpr int FACE_LIMIT = 1 << 22;       // polls of a face slot, a trip to L2 each (several seconds)
constexpr int OPEN = 32 * (TSJ + 1);      // threads that open a level
static_assert(TSJ == 4 && TSK == 3, "one warp per j-line of the tile, three lines a warp");

__device__ __forceinline__ unsigned sa(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
// Level counters in shared memory.  Plain volatile accesses: such a counter only
// says that a place may be overwritten.  Its store follows a barrier that every
// reader of the place has passed (the reads are performed by then), and the writer
// of the place has the counter's value before it issues its stores.  A release
// would also wait for the warp's global stores under way (several hundred cycles a
// level).
__device__ __forceinline__ int ld_level(const int* p) {
    int v;
    asm volatile("ld.volatile.shared.b32 %0, [%1];" : "=r"(v) : "r"(sa(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_level(int* p, int v) {
    asm volatile("st.volatile.shared.b32 [%0], %1;" ::"r"(sa(p)), "r"(v) : "memory");
}
// A counter that announces data: the writes that came before it (with a
// __syncwarp, those of the whole warp) are seen by whoever reads the new value.
__device__ __forceinline__ int ld_level_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.cta.shared.b32 %0, [%1];" : "=r"(v) : "r"(sa(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_level_release(int* p, int v) {
    asm volatile("st.release.cta.shared.b32 [%0], %1;" ::"r"(sa(p)), "r"(v) : "memory");
}
// Opening of a level, on one of RING barriers in turn: its face warp arrives
// (possibly several levels early), the compute warps wait.  The forms that
// count threads: a warp that has come apart at a branch must not arrive twice.
__device__ __forceinline__ void level_sync(int place) {
    asm volatile("barrier.cta.sync %0, %1;" ::"r"(1 + place), "n"(OPEN) : "memory");
}
__device__ __forceinline__ void level_arrive(int place) {
    asm volatile("barrier.cta.arrive %0, %1;" ::"r"(1 + place), "n"(OPEN) : "memory");
}
// This CTA's next tile; every CTA of a launch draws exactly one ticket past the
// last tile, so a launch takes T + gridDim.x of them.
__device__ __forceinline__ unsigned draw_tile(const SweepArgs& a) {
    return (unsigned)(atomicAdd(a.ticket, 1ull) % (unsigned long long)(a.T + gridDim.x));
}
// A warp's wait until a level counter has come to `least`, SLEEP ns between the polls.
// Gives up after the bound.  Returns the counter.
template <int SLEEP>
__device__ __forceinline__ int await_level(const int* counter, int least, int lane, int* err,
                                           int limit = WAIT_LIMIT) {
    int v, q = 0;
    while ((v = ld_level(counter)) < least && ++q < limit) __nanosleep(SLEEP);
    if (q >= limit && lane == 0) atomicExch(err, 1);
    return v;
}
// The same without a pause for a counter that announces data, until it is past `last`.
__device__ __forceinline__ void await_data(const int* counter, int last, int lane, int* err,
                                           int limit = WAIT_LIMIT) {
    int q = 0;
    while (ld_level_acquire(counter) <= last && ++q < limit) {}
    if (q >= limit && lane == 0) atomicExch(err, 1);
}
// A face warp's wait before it writes the ring place of level l, read last at
// level l - RING (done: levels begun by the compute warps).
__device__ __forceinline__ void await_place(const int* done, int l, int lane, int* err) {
    await_level<32>(done, l - RING + 1, lane, err);
}

// One of a face warp's values of a level: *at once it is written (need), else 0.
// Polls until every lane has its N values; gives up (zeros) after the bound or
// when another wait of the launch has given up.
template <int N>
__device__ __forceinline__ void poll_faces(double* const (&at)[N], const bool (&need)[N],
                                           double (&v)[N], bool& abort, int lane, int* err,
                                           int limit = FACE_LIMIT) {
    bool all = true;
#pragma unroll
    for (int u = 0; u < N; ++u) {
        v[u] = need[u] ? ld_relaxed(at[u]) : 0.0;
        all = all && !is_sentinel(v[u]);
    }
    for (int q = 1; !__all_sync(FULL, all) && !abort; ++q) {
        all = true;
#pragma unroll
        for (int u = 0; u < N; ++u) {
            if (need[u]) v[u] = ld_relaxed(at[u]);
            all = all && !is_sentinel(v[u]);
        }
        if ((q & 1023) == 0) {
            const bool late = q >= limit;
            if (late && lane == 0) atomicExch(err, 1);
            abort = __any_sync(FULL, late || ld_relaxed_i(err) != 0);
        }
    }
#pragma unroll
    for (int u = 0; u < N; ++u)
        if (is_sentinel(v[u])) v[u] = 0.0;
}

}  // namespace bo
