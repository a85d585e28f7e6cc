// Tile geometry of the FP32 sweeps and the one-CTA solve (8 x 4 x-lines) and of
// the FP64 wavefront kernels (4 x 3), face slots, the sentinel protocol of the
// face buffers and relaxed global accesses.
#pragma once
#include "common.cuh"

namespace bo {

constexpr int TJ = 8, TK = 4;          // tile of x-lines per warp (lane = jj + TJ kk)
constexpr unsigned long long SENTINEL_BITS = 0x7FF4DEADBEEF0001ull;  // a NaN no arithmetic yields
constexpr long long POLL_LIMIT = 1LL << 20;   // unit of the FP32 sweeps' bounded waits
constexpr unsigned FULL = 0xffffffffu;

// ILU(0) data in tile order: slot s = t NL + l (tile t, level l) holds NPE
// entries x 32 lanes contiguously, P[(s NPE + q) 32 + lane]; q = 9 b + e with
// b 0: D^-1, 1..3: D^-1 A_{c,-x/-y/-z}, 4..6: D^-1 A_{c,+x/+y/+z}.  Entries
// 0..35 of a slot are the forward sweep's data, 36..62 the backward sweep's.
constexpr int NPE = 63;
__host__ __device__ __forceinline__ size_t pidx(size_t slot, int q, int lane) {
    return (slot * NPE + q) * 32 + lane;
}

struct TileArgs {
    Geom g;
    int NJ, NK, T, NL;
    size_t NP;
    int* err;
    int ysub;   // block-Jacobi slabs of ysub cell rows in y (a multiple of TJ), 0: no cut in y
    int zsub;   // and of zsub cell layers in z (a multiple of TK), 0: no cut in z
};

// j is the first cell row of a block-Jacobi slab (not the first of the grid):
// the -y coupling of row j and the +y coupling of row j - 1 are left out of
// the factors, and no face crosses the cut.  Cuts fall on tile boundaries.
__device__ __forceinline__ bool ycut(const TileArgs& a, int j) {
    return a.ysub > 0 && j > 0 && j % a.ysub == 0;
}
// The same in z: layer k starts a slab, the -z coupling of layer k and the +z
// coupling of layer k - 1 are left out.
__device__ __forceinline__ bool zcut(const TileArgs& a, int k) {
    return a.zsub > 0 && k > 0 && k % a.zsub == 0;
}

__device__ __forceinline__ double ld_relaxed(const double* p) {
    double v;
    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(double* p, double v) {
    asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ int ld_relaxed_i(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ bool is_sentinel(double v) {
    return (unsigned long long)__double_as_longlong(v) == SENTINEL_BITS;
}
// FP32 faces of the mixed-precision sweeps: a NaN payload no arithmetic yields
constexpr unsigned SENTINEL_BITS32 = 0x7FA5DEADu;
__device__ __forceinline__ float ld_relaxed(const float* p) {
    float v;
    asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(float* p, float v) {
    asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ bool is_sentinel(float v) {
    return (unsigned)__float_as_uint(v) == SENTINEL_BITS32;
}

// Face slots: j-face of tile t for lane row kk at x index i; k-face for jj.
__device__ __forceinline__ size_t jslot(const TileArgs& a, int t, int i, int kk, int K) {
    return (((size_t)t * a.g.nx + i) * TK + kk) * K;
}
__device__ __forceinline__ size_t kslot(const TileArgs& a, int t, int i, int jj, int K) {
    return (((size_t)t * a.g.nx + i) * TJ + jj) * K;
}

__device__ __forceinline__ bool ks_skip_t(const KrylovScalars* ks) {
    return ks != nullptr && ks->state != KS_RUN;
}

// Host side: tile geometry of a model, face buffers, cooperative launches.
TileArgs tile_args(const bo_sim* s);
double* faceJ3(bo_sim* s);   // 3-value face buffers of the sweeps
double* faceK3(bo_sim* s);

template <class... Args>
void launch_coop(cudaStream_t st, int grid, int block, void (*kern)(Args...), Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    BO_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
}

// FP64 sweeps (sweep64.cu): a CTA owns a tile of TSJ x TSK x-lines.  Tiles are
// numbered in the order a sweep takes them (per direction), a tile has NL =
// nx + TSJ + TSK - 2 levels, and position (tile NL + level) 36 + 3 (TSK jj + kk)
// + row of Q holds a right-hand side entry.  S[((tile NL + level) TSJ + jj) 96
// + 32 s + 9 kk + 3 row + d] is entry (row, s) of the scaled block towards
// neighbour d.  line[j + ny k] is the Q position of cell (0, j, k); a step in i
// is one level up (forward) or down (backward).
constexpr int FACE_W = 24;   // doubles of a level in a tile's inbox: 9 j-face, 12 k-face
constexpr int FACE9_W = 64;  // the same for the factorisation's blocks: 27 j-face, 36 k-face
struct SweepArgs {
    Geom g;
    int T, NL;
    const SweepTile* tiles;
    double* inbox;                // [T][NL][FACE_W] neighbours' values, sentinel until written
    unsigned long long* ticket;   // tiles handed out; a launch takes T + grid of them
    int* err;
};
struct SweepFactors {
    const unsigned *fline, *bline;
    double *F, *B, *Dn;           // S of both directions, D^-1 [9][n] in natural order
};
// The scaled lower (-x, -y, -z) and upper blocks of cell (i, j, k), jk = j + ny k:
// entry (row, s) towards neighbour d at [lane_entry(row, s, d)].
__device__ __forceinline__ const double* lower_blocks(const SweepFactors& f, size_t jk, int i) {
    const unsigned p = f.fline[jk], line = p % 36 / 3;
    return f.F + ((size_t)(p / 36 + i) * TSJ + line / TSK) * 96 + line % TSK * 9;
}
__device__ __forceinline__ const double* upper_blocks(const SweepFactors& f, size_t jk, int i) {
    const unsigned p = f.bline[jk], line = p % 36 / 3;
    return f.B + ((size_t)(p / 36 - i) * TSJ + line / TSK) * 96 + line % TSK * 9;
}
__host__ __device__ constexpr int lane_entry(int row, int s, int d) { return 32 * s + 3 * row + d; }
struct SweepOrder {
    int T;
    std::vector<SweepTile> tiles;
    std::vector<unsigned> line;
};
SweepOrder sweep_order(const Geom& g, int ysub, int zsub, bool mirrored);
SweepArgs sweep_args(const bo_sim* s, int dir);
SweepFactors sweep_factors(const bo_sim* s);
int sweep_grid(const bo_sim* s);                             // CTAs of a wavefront launch
void setup_sweeps64(bo_sim* s);                              // plan for the current boxes
void reset_inbox(bo_sim* s, cudaStream_t st);
void enqueue_fwd64(bo_sim* s, cudaStream_t st, const double* r, const KrylovScalars* ks);
void enqueue_bwd64(bo_sim* s, cudaStream_t st, double* z, const KrylovScalars* ks);

// FP32 sweeps of the mixed-precision solver (ilu_sweep32.cu)
void setup_sweeps32(bo_sim* s);                              // attributes, residency check
void convert_factors32(bo_sim* s, cudaStream_t st);          // factorisation -> FP32 sweep layout
void enqueue_fwd32(bo_sim* s, cudaStream_t st, const double* r, const KrylovScalars* ks);
void enqueue_bwd32(bo_sim* s, cudaStream_t st, double* z, const KrylovScalars* ks);
void reset_faces32(bo_sim* s, cudaStream_t st);

}  // namespace bo
