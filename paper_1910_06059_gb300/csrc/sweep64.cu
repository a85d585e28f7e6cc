// FP64 triangular sweeps of the block ILU(0) preconditioner (arXiv
// 1910.06059, Section 2.3.1: ILU0 is BiCGStab's default preconditioner and
// takes most of the solve time).
//
//   forward  y_c = D_c^-1 r_c - sum_lower (D_c^-1 A_ck) y_k
//   backward z_c = y_c       - sum_upper (D_c^-1 A_cj) z_j
//
// The backward sweep is the forward sweep of the mirrored grid (i, j, k ->
// nx-1-i, ny-1-j, nz-1-k), so one kernel does both: cell (i, j, k) takes its
// three neighbours i-1, j-1, k-1 of its own direction.
//
// What bounds it.  The recurrence runs over nx + ny + nz - 2 wavefront levels
// (363 on the 60x220x85 model).  An FP64 warp instruction takes 64 cycles, in
// throughput of its sub-partition and in latency, and an SM issues one in 19
// cycles, so a level costs its longest chain of FP64 operations, plus what is
// lost between levels.  Bytes do not bind: the 350 MB a sweep moves on that
// model take 51 us.
//   * A cell's row is u + (v + w): three chains of three products, one per
//     neighbour.  Each chain has its own lane (9 lanes a cell, 3 cells a
//     warp), so a level is 3 dependent products and 2 additions, 5 x 77 cycles
//     with four warps; three chains in one lane would be 11 operations.
//   * A CTA has four such warps (one per sub-partition) and a tile of 4 x 3
//     x-lines (TSJ x TSK), of one box or of several boxes side by side; at tile level
//     l, line (jj, kk) handles cell i = l - jj - kk.  Results pass through a small plane in shared memory, one barrier a
//     level; a level of a tile on its own takes 600 cycles, 304 ns.
//   * The factors are stored lane by lane, a level's 3 KB in one piece: a copy
//     warp brings them and the right-hand side into a ring in shared memory with
//     16-byte asynchronous copies, up to RING levels ahead, and announces the
//     levels that are in (304 ns a level; the copies issued by the compute warps:
//     343, loads by the face warps through registers: 327, plain loads by the
//     compute warps six levels ahead: 400).
//   * Values of the neighbouring tiles come through write-once slots in global
//     memory that hold a NaN sentinel until written.  Four face warps poll them,
//     each every fourth level, write them to a ring in shared memory and arrive
//     at the barrier that opens their level, so a round trip to L2 (0.47 us one
//     way between two SMs) is paid once per tile crossing, 0.73 us in all, and
//     not once per level.
//   * CTAs take tiles from a ticket counter in topological order (sorted by the
//     level at which a tile can start).  A tile waits only for tiles with smaller
//     tickets, which CTAs already running hold, so every wait ends whatever else
//     shares the GPU and no launch has to be resident as a whole.
// Measured, a sweep: 60x220x85 267 us (405 before, with one warp per row of an
// 8 x 4 tile and a handoff per level), 33x27x9 31 us (52.6 before).
// Waits are bounded; one that runs out sets the error flag and the sweep ends
// with zeros for the missing values.
#include <algorithm>
#include <tuple>
#include <vector>

#include "wavefront.cuh"

namespace bo {

constexpr int SWEEP_THREADS = 32 * (TSJ + FACE_WARPS + 1);   // compute, face and copy warps
constexpr int SLOT = 3 * LINES;           // doubles of one level in shared memory
constexpr int STAGE = 96 * TSJ + SLOT;    // doubles of a level: factors, right-hand side
constexpr int STAGE_LOADS = 96 * TSJ / 64 + 1;   // 16-byte loads of a lane for a level
static_assert(96 * TSJ % 64 == 0 && SLOT % 2 == 0 && SLOT / 2 <= 32, "a level in whole loads");
constexpr int FACE_LANES = 3 * (TSK + TSJ);   // face values of one level: j-face, k-face
static_assert(TSJ + TSK <= LINES && FACE_LANES <= FACE_W, "a level's face values fit a slot");

// ---------------------------------------------------------------------------
// q = D^-1 r in the forward sweep's order: its right-hand side, formed by all
// SMs before the wavefront (9 products a cell, bound by bytes: 72 + 24 in, 24
// out).  Idle slots keep the zeros they were allocated with.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_sweep_rhs(int n, int nx, const unsigned* __restrict__ lb, const double* __restrict__ Dn,
            const double* __restrict__ r, double* __restrict__ Q,
            const KrylovScalars* __restrict__ ks) {
    if (ks_skip_t(ks)) return;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        const int jk = c / nx, i = c - jk * nx;
        const double r0 = r[c], r1 = r[(size_t)n + c], r2 = r[2 * (size_t)n + c];
        double* q = Q + lb[jk] + (size_t)i * SLOT;
#pragma unroll
        for (int row = 0; row < 3; ++row) {
            double v = Dn[(size_t)(3 * row) * n + c] * r0;
            v = fma(Dn[(size_t)(3 * row + 1) * n + c], r1, v);
            v = fma(Dn[(size_t)(3 * row + 2) * n + c], r2, v);
            q[row] = v;
        }
    }
}

__device__ __forceinline__ void copy16(unsigned dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// ---------------------------------------------------------------------------
// a8: one sweep.  Compute warp w owns the lines jj = w, lane 9 kk + 3 row + d
// the chain of row `row` towards neighbour d (0: i-1, 1: j-1, 2: k-1).
// FWD writes y in the backward sweep's order, else z in natural order.
// ---------------------------------------------------------------------------
template <bool FWD>
__global__ void __launch_bounds__(SWEEP_THREADS, 2)
k_sweep(SweepArgs a, const double* __restrict__ S, const double* __restrict__ Q,
        const unsigned* __restrict__ lbout, double* __restrict__ out,
        const KrylovScalars* __restrict__ ks) {
    if (ks_skip_t(ks)) return;
    // PLANE: results of the last two levels [comp][kk TSJ + jj]; HALO: face
    // values of RING levels [comp][kk | TSK + jj]; ZERO: no neighbour
    constexpr int PLANE = 0, HALO = 2 * SLOT, ZERO = HALO + RING * SLOT;
    __shared__ double ex[ZERO + SLOT];
    __shared__ __align__(16) double ring[RING][STAGE];   // a level's factors and right-hand side
    __shared__ unsigned s_rank;
    __shared__ int s_copied;                  // levels whose entries have come to the ring
    __shared__ int s_done, s_begun;           // levels begun by the compute warps; level 0 is in
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int NL = a.NL, nx = a.g.nx, n = a.g.n;

    for (;;) {
        if (threadIdx.x == 0) {
            s_rank = draw_tile(a);
            s_done = s_begun = s_copied = 0;
        }
        for (int q = threadIdx.x; q < 2 * SLOT; q += SWEEP_THREADS) ex[PLANE + q] = 0.0;
        for (int q = threadIdx.x; q < SLOT; q += SWEEP_THREADS) ex[ZERO + q] = 0.0;
        __syncthreads();
        const unsigned rank = s_rank;
        if (rank >= (unsigned)a.T) return;
        const SweepTile t = a.tiles[rank];
        if (warp == TSJ + FACE_WARPS) {
            // ---- copy warp: a level's factors and right-hand side into its place,
            // once the level that held it before has begun (its entries are read
            // one level earlier); levels under way are waited for when no place is
            // free, and announced ------------------------------------------------
            const char* Sp = reinterpret_cast<const char*>(S + (size_t)rank * NL * (TSJ * 96)) + 16 * lane;
            const char* Qp = reinterpret_cast<const char*>(Q + (size_t)rank * NL * SLOT) + 16 * lane;
            auto begun = [&] { return __shfl_sync(FULL, ld_level(&s_done), 0); };   // as one warp
            int known = 0, told = 0;   // levels seen begun, levels announced
            for (int l = 0;; ++l) {
                if (l == NL || (known + RING <= l && (known = begun()) + RING <= l)) {
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    __syncwarp();
                    if (told != l && lane == 0) st_level_release(&s_copied, l);
                    told = l;
                    if (l == NL) break;
                    known = __shfl_sync(FULL, await_level<20>(&s_done, l - RING + 1, lane, a.err), 0);
                }
                const unsigned dst = sa(ring[l & (RING - 1)]) + 16 * lane;
                const char* f = Sp + (size_t)l * (TSJ * 96 * 8);
#pragma unroll
                for (int u = 0; u < STAGE_LOADS - 1; ++u) copy16(dst + 512 * u, f + 512 * u);
                if (lane < SLOT / 2) copy16(dst + TSJ * 96 * 8, Qp + (size_t)l * (SLOT * 8));
            }
        } else if (warp >= TSJ) {
            // ---- face warps: levels warp - TSJ, + FACE_WARPS, ... ------------
            const bool jf = lane < 3 * TSK;
            const int e = jf ? lane : lane - 3 * TSK;
            const int line = e / 3, comp = e % 3;
            const bool has = lane < FACE_LANES && (jf ? t.depJ && line < t.nk : (t.takeK & 1) && line < t.nj);
            double* in = a.inbox + (size_t)rank * NL * FACE_W + lane;
            const int to = HALO + comp * LINES + (jf ? line : TSK + line);
            const double sent = __longlong_as_double((long long)SENTINEL_BITS);
            bool abort = false;
            // the later levels are polled once the first has come
            if (warp > TSJ) await_level<32>(&s_begun, 1, lane, a.err);
            for (int l = warp - TSJ; l < NL; l += FACE_WARPS) {
                await_place(&s_done, l, lane, a.err);
                const int i = l - line;
                const bool need[1] = {has && i >= 0 && i < nx};
                double* const at[1] = {in + (size_t)l * FACE_W};
                double v[1];
                poll_faces(at, need, v, abort, lane, a.err);
                if (lane < FACE_LANES) ex[to + ((l + 1) & (RING - 1)) * SLOT] = v[0];
                if (l == 0 && lane == 0) st_level(&s_begun, 1);
                // the next level's entries (the first one's too) are in
                await_data(&s_copied, min(l + 1, NL - 1), lane, a.err);
                __syncwarp();
                level_arrive(l & (RING - 1));
                if (need[0]) st_relaxed(at[0], sent);
            }
        } else {
            // ---- compute warps ----------------------------------------------
            const bool work = lane < 27;
            const int kk = work ? lane / 9 : TSK - 1, row = (lane % 9) / 3, d = lane % 3, jj = warp;
            const bool valid = work && jj < t.nj && kk < t.nk;
            const bool head = valid && d == 0;         // the lane that ends with the result
            const bool rhs = work && d == 0;
            // neighbour source at level l: src + ((l + 1) & mask) SLOT, components LINES apart
            int src, mask;
            if (d == 0) {
                src = PLANE + kk * TSJ + jj;
                mask = 1;
            } else if (d == 1) {
                src = jj > 0 ? PLANE + kk * TSJ + jj - 1 : t.depJ ? HALO + kk : ZERO;
                mask = jj > 0 ? 1 : t.depJ ? RING - 1 : 0;
            } else {
                const bool takes = t.takeK >> kk & 1;
                src = !takes ? ZERO : kk > 0 ? PLANE + (kk - 1) * TSJ + jj : HALO + TSK + jj;
                mask = !takes ? 0 : kk > 0 ? 1 : RING - 1;
            }
            double L[3], q;                   // the current level's entries
            const int mine = jj * 96 + lane, rhs_at = TSJ * 96 + (jj * TSK + kk) * 3 + row;
            // where results go
            const int l0 = jj + kk;
            const int res = PLANE + row * LINES + kk * TSJ + jj;
            double* outp = out;
            long long ostep = 0;
            double *pj = a.inbox, *pk = a.inbox;       // the neighbours' inboxes
            bool toJ = false, toK = false;
            if (head) {
                if (FWD) {
                    const int jk = (t.j0 + jj) + a.g.ny * (t.k0 + kk);
                    ostep = -(long long)SLOT;
                    outp = out + (size_t)lbout[jk] + row - (long long)(l0 + 1) * ostep;
                } else {
                    const int j = a.g.ny - 1 - (t.j0 + jj), k = a.g.nz - 1 - (t.k0 + kk);
                    ostep = -1;
                    outp = out + (size_t)row * n + (size_t)nx * (j + (size_t)a.g.ny * k) + (nx - 1) + l0 + 1;
                }
                toJ = t.nextJ >= 0 && jj == TSJ - 1;
                toK = t.nextK >= 0 && kk == TSK - 1;
                if (toJ) pj = a.inbox + ((long long)t.nextJ * NL - (TSJ - 1)) * FACE_W + kk * 3 + row;
                if (toK) pk = a.inbox + ((long long)t.nextK * NL - (TSK - 1)) * FACE_W + 3 * TSK + jj * 3 + row;
            }
            double acc = 0.0;                 // the last level's result, not yet written out
            bool act = false;
            int ya = src + (1 & mask) * SLOT;
            unsigned i = (unsigned)-l0;       // this level's cell of the line
            for (int lb = 0; lb < NL; lb += RING) {
#pragma unroll
                for (int u = 0; u < RING; ++u) {
                    const int l = lb + u;
                    if (l >= NL) break;
                    level_sync(u);
                    const double y0 = ex[ya], y1 = ex[ya + LINES], y2 = ex[ya + 2 * LINES];
                    if (u == 0 && l == 0) {
#pragma unroll
                        for (int s = 0; s < 3; ++s) L[s] = ring[0][mine + s * 32];
                        q = rhs ? ring[0][rhs_at] : -0.0;   // the other chains start from nothing
                    }
                    double v = fma(-L[0], y0, q);
                    v = fma(-L[1], y1, v);
                    v = fma(-L[2], y2, v);
                    // in the shadow of the chain: the last level's result, the next
                    // level's entries
                    if (act) *outp = acc;
                    outp += ostep;
                    if (threadIdx.x == 0) st_level(&s_done, l);
#pragma unroll
                    for (int s = 0; s < 3; ++s) L[s] = ring[(u + 1) % RING][mine + s * 32];
                    q = rhs ? ring[(u + 1) % RING][rhs_at] : -0.0;
                    const bool in = i < (unsigned)nx;
                    act = in && head;
                    ++i;
                    ya = src + ((l + 2) & mask) * SLOT;
                    // u + (v + w): the j-1 lane adds the k-1 chain, the i-1 lane the sum
                    const double vw = v + __shfl_down_sync(FULL, v, 1);
                    acc = v + __shfl_down_sync(FULL, vw, 1);
                    if (!(in && valid)) acc = 0.0;
                    if (rhs) ex[res + (u & 1) * SLOT] = acc;
                    if (in && toJ) st_relaxed(pj, acc);
                    if (in && toK) st_relaxed(pk, acc);
                    pj += FACE_W;
                    pk += FACE_W;
                }
            }
            if (act) *outp = acc;
        }
        __syncthreads();   // the plane, the rings and the ticket are free again
    }
}

// ---------------------------------------------------------------------------
// Host side: tiles of both directions
// ---------------------------------------------------------------------------
namespace {
// The tiles of one axis: boxes of `sub` lines (0: one box) counted from the low end
// of the grid, cut into tiles of up to `ext` lines in the sweep's direction; with
// `across` a tile may hold lines of several boxes.
struct AxisTile {
    int start, count;
    int group;   // first line of the run of tiles that it belongs to, each waiting for the last
    int takes;   // bit m: line m takes the line before it (it is not the first of its box)
};
std::vector<AxisTile> axis_tiles(int n, int sub, int ext, bool mirrored, bool across) {
    std::vector<char> first(n, 0);   // first lines of the boxes
    const int step = sub > 0 ? sub : n;
    for (int b = 0; b < n; b += step) first[mirrored ? n - std::min(n, b + step) : b] = 1;
    std::vector<AxisTile> t;
    for (int s = 0, group = 0; s < n;) {
        int e = s + 1, takes = !first[s];
        while (e < n && e - s < ext && (across || !first[e])) {
            takes |= !first[e] << (e - s);
            ++e;
        }
        if (first[s]) group = s;
        t.push_back({s, e - s, group, takes});
        s = e;
    }
    return t;
}
}  // namespace

SweepOrder sweep_order(const Geom& g, int ysub, int zsub, bool mirrored) {
    // Boxes that fill their tiles badly share tiles instead, at the price of runs of
    // tiles that wait for one another up to the next common edge.  Boxes of 4 layers
    // (3 + 1: half as many tiles again) gain, a backward sweep on 60x220x85 with boxes
    // (8, 4) 185 us for 247; boxes of 8 (3 + 3 + 2) and more lose, on 60x110x44 with
    // boxes (0, 8) 121 us for 111, (0, 16) 127 for 119.
    const bool across = zsub > 0 && 4 * ((zsub + TSK - 1) / TSK * TSK) > 5 * zsub;
    const std::vector<AxisTile> tj = axis_tiles(g.ny, ysub, TSJ, mirrored, false);
    const std::vector<AxisTile> tk = axis_tiles(g.nz, zsub, TSK, mirrored, across);
    const int NJ = (int)tj.size(), NK = (int)tk.size(), T = NJ * NK, NL = g.nx + TSJ + TSK - 2;
    // topological order: the level at which a tile can start within its run
    std::vector<int> ids(T), rank(T);
    for (int q = 0; q < T; ++q) ids[q] = q;
    auto key = [&](int q) {
        const AxisTile &a = tj[q % NJ], &b = tk[q / NJ];
        return std::make_tuple((a.start - a.group) + (b.start - b.group), q);
    };
    std::sort(ids.begin(), ids.end(), [&](int x, int y) { return key(x) < key(y); });
    for (int q = 0; q < T; ++q) rank[ids[q]] = q;
    SweepOrder o;
    o.T = T;
    o.tiles.resize(T);
    o.line.assign((size_t)g.ny * g.nz, 0);
    for (int J = 0; J < NJ; ++J)
        for (int K = 0; K < NK; ++K) {
            const int r = rank[J + NJ * K];
            SweepTile& t = o.tiles[r];
            t.j0 = tj[J].start;
            t.k0 = tk[K].start;
            t.nj = (short)tj[J].count;
            t.nk = (short)tk[K].count;
            t.depJ = tj[J].takes & 1;
            t.takeK = tk[K].takes;
            t.nextJ = J + 1 < NJ && (tj[J + 1].takes & 1) ? rank[J + 1 + NJ * K] : -1;
            t.nextK = K + 1 < NK && (tk[K + 1].takes & 1) ? rank[J + NJ * (K + 1)] : -1;
            for (int jj = 0; jj < t.nj; ++jj)
                for (int kk = 0; kk < t.nk; ++kk) {
                    const int j = mirrored ? g.ny - 1 - (t.j0 + jj) : t.j0 + jj;
                    const int k = mirrored ? g.nz - 1 - (t.k0 + kk) : t.k0 + kk;
                    const size_t lev = (size_t)r * NL + jj + kk + (mirrored ? g.nx - 1 : 0);
                    o.line[j + (size_t)g.ny * k] = (unsigned)(lev * SLOT + (jj * TSK + kk) * 3);
                }
        }
    return o;
}

SweepArgs sweep_args(const bo_sim* s, int dir) {
    const SweepPlan& p = s->sweep;
    SweepArgs a;
    a.g = s->geo;
    a.T = p.T;
    a.NL = p.NL;
    a.tiles = p.tiles[dir];
    a.inbox = p.inbox;
    a.ticket = p.ticket + dir;
    a.err = s->d_sweep_sync + 2;
    return a;
}

SweepFactors sweep_factors(const bo_sim* s) {
    const SweepPlan& p = s->sweep;
    return SweepFactors{p.line[0], p.line[1], p.S[0], p.S[1], p.Dn};
}

// CTAs of a sweep per SM: sweep_ctas_per_sm (two by default).  Up to 470 tiles
// (3 an SM) could be under way in the middle of the 60x220x85 model's
// wavefront, but tiles on one SM share its FP64 pipes (one warp instruction in
// 19 cycles, 20 a tile level): 2, 3 and 4 CTAs per SM took 265, 276 and 288 us.
int sweep_grid(const bo_sim* s) {
    int dev, sms;
    BO_CUDA(cudaGetDevice(&dev));
    BO_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    return std::min(s->sweep.T, s->sweep_ctas_per_sm * sms);
}

static void free_plan(SweepPlan& p) {
    void* ptrs[] = {p.tiles[0], p.tiles[1], p.line[0], p.line[1], p.S[0], p.S[1],
                    p.Q[0],     p.Q[1],     p.inbox,   p.inbox9,  p.ticket, p.Dn};
    for (void* q : ptrs)
        if (q) cudaFree(q);
    p = SweepPlan();
}
void free_sweeps64(bo_sim* s) { free_plan(s->sweep); }

__global__ void k_fill_inbox(double* __restrict__ p, size_t count) {
    const double sent = __longlong_as_double((long long)SENTINEL_BITS);
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < count;
         q += (size_t)gridDim.x * blockDim.x)
        p[q] = sent;
}
void reset_inbox(bo_sim* s, cudaStream_t st) {
    const SweepPlan& p = s->sweep;
    k_fill_inbox<<<304, 256, 0, st>>>(p.inbox, (size_t)p.T * p.NL * FACE_W);
    count_launch(s, st);
    k_fill_inbox<<<304, 256, 0, st>>>(p.inbox9, (size_t)p.T * p.NL * FACE9_W);
    count_launch(s, st);
    BO_LAUNCH_CHECK("k_fill_inbox");
}

// The tickets of a launch are counted from the last launch's with the same grid.
// On the simulator's stream: the legacy stream has no order with a non-blocking one.
void reset_tickets(bo_sim* s) {
    BO_CUDA(cudaMemsetAsync(s->sweep.ticket, 0, 3 * sizeof(unsigned long long), s->stream));
}

// Plan of both sweeps for the current block-Jacobi boxes, filled on the
// simulator's stream.  The old plan goes first, so a change of boxes needs no room for
// two; on failure there is none (T = 0).
void setup_sweeps64(bo_sim* s) {
    const Geom& g = s->geo;
    free_plan(s->sweep);
    SweepPlan p;
    try {
        p.NL = g.nx + TSJ + TSK - 2;
        for (int d = 0; d < 2; ++d) {
            const SweepOrder o = sweep_order(g, s->ysub, s->zsub, d == 1);
            p.T = o.T;
            const size_t lev = (size_t)o.T * p.NL;
            if (lev * SLOT >= (1ull << 32))
                fail(BO_ERR_INVALID_ARG, "grid too large for the sweeps' 32-bit positions");
            auto alloc = [&](auto** q, size_t count) {
                BO_CUDA(cudaMalloc(reinterpret_cast<void**>(q), sizeof(**q) * count));
                BO_CUDA(cudaMemsetAsync(*q, 0, sizeof(**q) * count, s->stream));   // idle slots stay zero
            };
            alloc(&p.tiles[d], o.tiles.size());
            alloc(&p.line[d], o.line.size());
            alloc(&p.S[d], lev * TSJ * 96);
            alloc(&p.Q[d], lev * SLOT);
            BO_CUDA(cudaMemcpyAsync(p.tiles[d], o.tiles.data(), sizeof(SweepTile) * o.tiles.size(),
                                    cudaMemcpyHostToDevice, s->stream));
            BO_CUDA(cudaMemcpyAsync(p.line[d], o.line.data(), sizeof(unsigned) * o.line.size(),
                                    cudaMemcpyHostToDevice, s->stream));
            if (d == 0) {
                alloc(&p.inbox, lev * FACE_W);
                alloc(&p.inbox9, lev * FACE9_W);
                alloc(&p.ticket, 3);
                alloc(&p.Dn, 9 * (size_t)g.n);
            }
            BO_CUDA(cudaStreamSynchronize(s->stream));   // the host arrays end here
        }
    } catch (...) {
        free_plan(p);
        throw;
    }
    s->sweep = p;
    s->tile_valid = false;
    // two CTAs on an SM hold about 60 KB of shared memory (a ring of 27 KB each)
    for (const void* k : {(const void*)k_sweep<true>, (const void*)k_sweep<false>})
        BO_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared));
    reset_inbox(s, s->stream);
    BO_CUDA(cudaStreamSynchronize(s->stream));
}

void enqueue_fwd64(bo_sim* s, cudaStream_t st, const double* r, const KrylovScalars* ks) {
    const SweepPlan& p = s->sweep;
    k_sweep_rhs<<<152 * 8, 256, 0, st>>>(s->geo.n, s->geo.nx, p.line[0], p.Dn, r, p.Q[0], ks);
    count_launch(s, st);
    k_sweep<true><<<sweep_grid(s), SWEEP_THREADS, 0, st>>>(sweep_args(s, 0), p.S[0], p.Q[0],
                                                           p.line[1], p.Q[1], ks);
    count_launch(s, st);
    BO_LAUNCH_CHECK("k_sweep forward");
}

void enqueue_bwd64(bo_sim* s, cudaStream_t st, double* z, const KrylovScalars* ks) {
    const SweepPlan& p = s->sweep;
    k_sweep<false><<<sweep_grid(s), SWEEP_THREADS, 0, st>>>(sweep_args(s, 1), p.S[1], p.Q[1],
                                                            nullptr, z, ks);
    count_launch(s, st);
    BO_LAUNCH_CHECK("k_sweep backward");
}

}  // namespace bo
