// Block ILU(0) factorisation of the 7-point pattern (arXiv 1910.06059, Section
// 2.3.1: ILU0 is BiCGStab's default preconditioner).
//
// ILU(0) on this pattern changes only the diagonal blocks (the grid graph is
// bipartite, so no fill position lies in the pattern):
//     D_c = A_cc - sum_{k in {-x,-y,-z}} A_ck D_k^-1 A_kc,
//     M   = (L_A + D) D^-1 (D + U_A).
//
// k_factor_wave    D, D^-1 and the scaled upper blocks U = D^-1 A_{c,+x/+y/+z}
//                  along the wavefront: D^-1 in natural order, U in the
//                  backward sweep's lane order.
// k_scaled_blocks  the scaled lower blocks D^-1 A_{c,-x/-y/-z} in the forward
//                  sweep's lane order, off the wavefront.
//
// What bounds the wavefront.  A cell costs about 200 FP64 operations, and a level
// of the recurrence runs through all of them; with one lane a cell that was 10
// us a level (an FP64 warp instruction takes 64 cycles).  Here the nine entries
// of a cell's blocks have a lane each (27 of a warp's lanes, three cells): nine
// products for D, six operations and a reciprocal for D^-1, nine products for U,
// about 29 FP64 warp instructions a level.  Tiles, levels, tickets and the face
// warps are the sweeps' (sweep64.cu); a face carries a 3x3 block a line.
// Measured, k_factor_wave: 1.29 ms on 60x220x85 (4.27 ms with one lane a cell),
// 115 us on 33x27x9 (696), 1.67 us a level of a tile on its own; the FP64 pipes
// bind it where several tiles share an SM (29 x 4 warp instructions a tile level,
// one in 19 cycles).
#include <cmath>

#include "wavefront.cuh"

namespace bo {

constexpr int FACTOR_THREADS = 32 * (TSJ + FACE_WARPS);
constexpr int BLOCKS_W = 27;                       // Ux, Uy, Uz of a line
constexpr int BPLANE = LINES * BLOCKS_W;           // one level's blocks of the tile
constexpr int BFACES = 9 * (TSK + TSJ);            // face values of one level
static_assert(BFACES <= FACE9_W && FACE9_W == 64, "two face values a lane");

// row . column of a block product; one order of operations for every caller
__device__ __forceinline__ double dot3(double a0, double b0, double a1, double b1, double a2,
                                       double b2) {
    return fma(a2, b2, fma(a0, b0, __dmul_rn(a1, b1)));
}

__global__ void __launch_bounds__(FACTOR_THREADS, 2)
k_factor_wave(SweepArgs a, const double* __restrict__ A, const unsigned* __restrict__ bline,
              double* __restrict__ Dn, double* __restrict__ B, int* __restrict__ bad) {
    // PLANE: U of the last two levels [line][27]; HALO: RING levels of face
    // blocks [9 kk + e | 27 + 9 jj + e]; ZERO: no neighbour
    constexpr int PLANE = 0, HALO = 2 * BPLANE, ZERO = HALO + RING * FACE9_W;
    __shared__ double ex[ZERO + 9];
    __shared__ double nbr[2][LINES][6][9];    // a level's off-diagonal blocks of A
    __shared__ double xd[LINES][9], xc[LINES][9];   // D, D^-1 and cofactors between nine lanes
    __shared__ unsigned s_rank;
    __shared__ int s_done, s_begun;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int NL = a.NL, nx = a.g.nx, n = a.g.n;

    for (;;) {
        if (threadIdx.x == 0) {
            s_rank = draw_tile(a);
            s_done = s_begun = 0;
        }
        for (int q = threadIdx.x; q < 2 * BPLANE; q += FACTOR_THREADS) ex[PLANE + q] = 0.0;
        if (threadIdx.x < 9) ex[ZERO + threadIdx.x] = 0.0;
        __syncthreads();
        const unsigned rank = s_rank;
        if (rank >= (unsigned)a.T) return;
        const SweepTile t = a.tiles[rank];

        if (warp >= TSJ) {
            // ---- face warps -------------------------------------------------
            int line[2];
            bool has[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int v = lane + 32 * u;
                const bool jf = v < 9 * TSK;
                line[u] = jf ? v / 9 : (v - 9 * TSK) / 9;
                has[u] = v < BFACES && (jf ? t.depJ && line[u] < t.nk : (t.takeK & 1) && line[u] < t.nj);
            }
            double* in = a.inbox + (size_t)rank * NL * FACE9_W + lane;
            const double sent = __longlong_as_double((long long)SENTINEL_BITS);
            bool abort = false;
            if (warp > TSJ) await_level<32>(&s_begun, 1, lane, a.err);
            for (int l = warp - TSJ; l < NL; l += FACE_WARPS) {
                await_place(&s_done, l, lane, a.err);
                bool need[2];
                double* at[2];
                double v[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int i = l - line[u];
                    need[u] = has[u] && i >= 0 && i < nx;
                    at[u] = in + (size_t)l * FACE9_W + 32 * u;
                }
                poll_faces(at, need, v, abort, lane, a.err);
                double* to = ex + HALO + ((l + 1) & (RING - 1)) * FACE9_W + lane;
                to[0] = v[0];
                to[32] = v[1];
                if (l == 0 && lane == 0) st_level(&s_begun, 1);
                __syncwarp();
                level_arrive(l & (RING - 1));
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (need[u]) st_relaxed(at[u], sent);
            }
        } else {
            // ---- compute warps: lane 9 kk + 3 r + s has entry (r, s) of the
            // blocks of line (jj = warp, kk) -----------------------------------
            const bool work = lane < 27;
            const int kk = work ? lane / 9 : TSK - 1, e = lane % 9, r = e / 3, s = e % 3, jj = warp;
            const int ln = kk * TSJ + jj;
            const bool valid = work && jj < t.nj && kk < t.nk;
            // couplings that leave the box are left out
            const bool takeK = t.takeK >> kk & 1;
            const bool keep[6] = {true, jj > 0 || t.depJ, takeK, true, jj + 1 < t.nj || t.nextJ >= 0,
                                  kk + 1 < t.nk ? (t.takeK >> (kk + 1) & 1) != 0 : t.nextK >= 0};
            constexpr int from[6] = {NB_MX, NB_MY, NB_MZ, NB_PX, NB_PY, NB_PZ};
            // the neighbours' blocks: source, ring mask and place size
            const int sx = PLANE + ln * BLOCKS_W;
            const int sy = jj > 0 ? PLANE + (ln - 1) * BLOCKS_W + 9 : t.depJ ? HALO + 9 * kk : ZERO;
            const int my = jj > 0 ? 1 : t.depJ ? RING - 1 : 0, wy = jj > 0 ? BPLANE : FACE9_W;
            const int sz = !takeK ? ZERO : kk > 0 ? PLANE + (ln - TSJ) * BLOCKS_W + 18
                                                  : HALO + 9 * TSK + 9 * jj;
            const int mz = !takeK ? 0 : kk > 0 ? 1 : RING - 1, wz = kk > 0 ? BPLANE : FACE9_W;
            const int l0 = jj + kk, j = t.j0 + jj, k = t.k0 + kk;
            const long long cbase = (long long)nx * (j + (long long)a.g.ny * k) - l0;   // cell: + l
            const double* Ae = A + (size_t)e * n;
            double* Bo = B;                       // backward factors of the cell: - l stages
            if (valid) {
                const unsigned p = bline[j + (size_t)a.g.ny * k], q = p % (3 * LINES) / 3;
                Bo = B + ((long long)(p / (3 * LINES) + l0) * TSJ + q / TSK) * 96 + q % TSK * 9 + 3 * r;
            }
            const bool toJ = valid && t.nextJ >= 0 && jj == TSJ - 1;
            const bool toK = valid && t.nextK >= 0 && kk == TSK - 1;
            double* pj = a.inbox + ((long long)t.nextJ * NL - (TSJ - 1)) * FACE9_W + 9 * kk + e;
            double* pk = a.inbox + ((long long)t.nextK * NL - (TSK - 1)) * FACE9_W + 9 * TSK + 9 * jj + e;
            // cofactor (s, r) of a block: rows s + 1, s + 2, columns r + 1, r + 2
            const int s1 = (s + 1) % 3, s2 = (s + 2) % 3, r1 = (r + 1) % 3, r2 = (r + 2) % 3;
            double diag = 0.0, off[6];            // this lane's entries of the next level's cell
            auto load = [&](int l) {
                const int i = l - l0;
                const bool act = valid && i >= 0 && i < nx;
                const double* p = Ae + (cbase + l);
                diag = r == s ? 1.0 : 0.0;
                if (act) diag = p[0];
#pragma unroll
                for (int b = 0; b < 6; ++b) {
                    off[b] = 0.0;
                    if (act && keep[b]) off[b] = p[(size_t)from[b] * 9 * n];
                }
            };
            load(0);
            for (int l = 0; l < NL; ++l) {
                const int par = l & 1, i = l - l0;
                const bool act = valid && i >= 0 && i < nx;
                double D = diag;
                double(*N)[9] = nbr[par][ln];
                if (work) {
#pragma unroll
                    for (int b = 0; b < 6; ++b) N[b][e] = off[b];
                }
                if (l + 1 < NL) load(l + 1);      // in the shadow of this level
                level_sync(l & (RING - 1));
                if (threadIdx.x == 0) st_level(&s_done, l);
                // D -= A_-x Ux + A_-y Uy + A_-z Uz, one chain in this order
                const double* ux = ex + sx + (par ^ 1) * BPLANE + s;
                const double* uy = ex + sy + ((l + 1) & my) * wy + s;
                const double* uz = ex + sz + ((l + 1) & mz) * wz + s;
#pragma unroll
                for (int m = 0; m < 3; ++m) D = fma(-N[0][3 * r + m], ux[3 * m], D);
#pragma unroll
                for (int m = 0; m < 3; ++m) D = fma(-N[1][3 * r + m], uy[3 * m], D);
#pragma unroll
                for (int m = 0; m < 3; ++m) D = fma(-N[2][3 * r + m], uz[3 * m], D);
                // D^-1: cofactors over the determinant
                double *X = xd[ln], *C = xc[ln];
                if (work) X[e] = D;
                __syncwarp();
                const double cof = fma(X[3 * s1 + r1], X[3 * s2 + r2],
                                       -__dmul_rn(X[3 * s1 + r2], X[3 * s2 + r1]));
                const double x0 = X[0], x1 = X[1], x2 = X[2];
                if (work) C[e] = cof;
                __syncwarp();
                const double Di = cof * (1.0 / dot3(x0, C[0], x1, C[3], x2, C[6]));
                if (work) X[e] = Di;
                __syncwarp();
                // U = D^-1 A_+: the data the next cells wait for
                const double d0 = X[3 * r], d1 = X[3 * r + 1], d2 = X[3 * r + 2];
                double U[3];
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    U[d] = dot3(d0, N[3 + d][s], d1, N[3 + d][3 + s], d2, N[3 + d][6 + s]);
                    if (!act) U[d] = 0.0;
                    if (work) ex[PLANE + par * BPLANE + ln * BLOCKS_W + 9 * d + e] = U[d];
                }
                if (act) {
                    if (toJ) st_relaxed(pj + (long long)l * FACE9_W, U[1]);
                    if (toK) st_relaxed(pk + (long long)l * FACE9_W, U[2]);
                    Dn[(size_t)e * n + cbase + l] = Di;
                    double* b = Bo - (long long)l * (TSJ * 96) + s * 32;
#pragma unroll
                    for (int d = 0; d < 3; ++d) b[d] = U[d];
                    if (!isfinite(Di)) atomicAdd(bad, 1);
                }
            }
        }
        __syncthreads();
    }
}

// Scaled blocks D^-1 A towards the three neighbours of one sweep direction (DIR 0:
// -x, -y, -z; 1: +x, +y, +z) in its lane order: a warp a line of tiles' jj and
// CHUNK levels (a 32-byte sector of A holds four cells of a line, so the levels
// of a chunk share them), 27 lanes (kk, row, d), three entries a lane.  Idle
// places keep the zeros they were allocated with.  Couplings that leave a box of the
// plan, or of cy x cz lines (0: no cut), are left out.
constexpr int CHUNK = 8;
template <int DIR>
__global__ void __launch_bounds__(256)
k_scaled_blocks(SweepArgs a, const double* __restrict__ A, const double* __restrict__ Dn,
                double* __restrict__ S, int cy, int cz) {
    const int lane = threadIdx.x & 31, chunks = (a.NL + CHUNK - 1) / CHUNK;
    const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int jj = (int)(w % TSJ), ch = (int)(w / TSJ % chunks);
    const long long rank = w / TSJ / chunks;
    if (rank >= a.T || lane >= 27) return;
    const SweepTile t = a.tiles[rank];
    const int kk = lane / 9, row = lane % 9 / 3, d = lane % 3, n = a.g.n, nx = a.g.nx;
    if (jj >= t.nj || kk >= t.nk) return;
    const int js = t.j0 + jj, ks = t.k0 + kk;
    const int j = DIR ? a.g.ny - 1 - js : js, k = DIR ? a.g.nz - 1 - ks : ks;
    const int cut = d == 1 ? cy : cz;
    const bool keep = d == 0 || ((d == 1 ? jj > 0 || t.depJ : t.takeK >> kk & 1) &&
                                 (cut == 0 || ((d == 1 ? j : k) + DIR) % cut != 0));
    const int blk = 1 + 2 * d + DIR;   // NB_MX, NB_PX, NB_MY, ... in turn
    static_assert(NB_MX == 1 && NB_PX == 2 && NB_MY == 3 && NB_PY == 4 && NB_MZ == 5 && NB_PZ == 6,
                  "block numbers");
    const double *Ab = A + (size_t)blk * 9 * n, *Dr = Dn + (size_t)3 * row * n;
    double* out = S + ((size_t)rank * a.NL * TSJ + jj) * 96 + lane;
    for (int l = ch * CHUNK; l < min(a.NL, (ch + 1) * CHUNK); ++l) {
        const int is = l - jj - kk;
        if (is < 0 || is >= nx) continue;
        const size_t c = (DIR ? nx - 1 - is : is) + (size_t)nx * (j + (size_t)a.g.ny * k);
        const double d0 = Dr[c], d1 = Dr[(size_t)n + c], d2 = Dr[2 * (size_t)n + c];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            double b[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) b[m] = keep ? Ab[(size_t)(3 * m + s) * n + c] : 0.0;
            out[(size_t)l * (TSJ * 96) + s * 32] = dot3(d0, b[0], d1, b[1], d2, b[2]);
        }
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
template <int DIR>
static void enqueue_scaled(bo_sim* s, cudaStream_t st, int cy = 0, int cz = 0) {
    const SweepPlan& p = s->sweep;
    const long long warps = (long long)p.T * TSJ * ((p.NL + CHUNK - 1) / CHUNK);
    k_scaled_blocks<DIR><<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(sweep_args(s, DIR), s->d_A,
                                                                     p.Dn, p.S[DIR], cy, cz);
    count_launch(s, st);
    BO_LAUNCH_CHECK("k_scaled_blocks");
}

void enqueue_factor(bo_sim* s, cudaStream_t st, int* bad) {
    const SweepPlan& p = s->sweep;
    SweepArgs a = sweep_args(s, 0);
    a.inbox = p.inbox9;
    a.ticket = p.ticket + 2;
    k_factor_wave<<<sweep_grid(s), FACTOR_THREADS, 0, st>>>(a, s->d_A, p.line[1], p.Dn, p.S[1], bad);
    count_launch(s, st);
    BO_LAUNCH_CHECK("k_factor_wave");
    enqueue_scaled<0>(s, st);
    if (s->mixed) convert_factors32(s, st);
}

void enqueue_scaled_factors(bo_sim* s, cudaStream_t st, int ysub, int zsub) {
    s->tile_valid = false;
    enqueue_scaled<0>(s, st, ysub, zsub);
    enqueue_scaled<1>(s, st, ysub, zsub);
}

// D^-1 of every cell, [n][9].
void export_dinv(bo_sim* s, double* dinv) {
    const size_t n = s->geo.n;
    std::vector<double> D(9 * n);
    BO_CUDA(cudaMemcpy(D.data(), s->sweep.Dn, sizeof(double) * D.size(), cudaMemcpyDeviceToHost));
    for (size_t c = 0; c < n; ++c)
        for (int e = 0; e < 9; ++e) dinv[9 * c + e] = D[e * n + c];
}

}  // namespace bo
