// ILU(0) data in the 8 x 4-line tile order that the one-CTA solve (block_solve.cu)
// reads, gathered from the factorisation at its launch; the dispatch of the sweeps
// by precision; the bounded wait's self-test.
#include <algorithm>
#include <cmath>
#include <vector>

#include "wavefront.cuh"

namespace bo {

// P[(slot 63 + q) 32 + lane]: D^-1, the scaled lower and the scaled upper blocks
// of every cell (pidx in tiles.cuh).  Idle places stay zero.
__global__ void __launch_bounds__(256)
k_tile_factors(TileArgs a, SweepFactors f, double* __restrict__ P) {
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < a.NP;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int lane = (int)(idx & 31);
        const size_t tl = idx >> 5;
        const int t = (int)(tl / a.NL), l = (int)(tl % a.NL);
        const int jj = lane % TJ, kk = lane / TJ;
        const int j = t % a.NJ * TJ + jj, k = t / a.NJ * TK + kk, i = l - jj - kk;
        if (j >= a.g.ny || k >= a.g.nz || i < 0 || i >= a.g.nx) continue;
        const size_t jk = j + (size_t)a.g.ny * k, c = i + (size_t)a.g.nx * jk;
        const double *lo = lower_blocks(f, jk, i), *up = upper_blocks(f, jk, i);
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            P[pidx(tl, e, lane)] = f.Dn[(size_t)e * a.g.n + c];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                P[pidx(tl, 9 + 9 * d + e, lane)] = lo[lane_entry(e / 3, e % 3, d)];
                P[pidx(tl, 36 + 9 * d + e, lane)] = up[lane_entry(e / 3, e % 3, d)];
            }
        }
    }
}

// Self-test of the sweeps' bounded waits with shorter bounds: a face slot that nothing
// writes, then a level counter that nothing advances, in both its forms.  out: the time,
// and 1 (the slot's wait set the flag and gave zeros) + 2 + 4 (the counter's waits set it).
__global__ void k_wait_selftest(double* slot, int* err, long long* out) {
    __shared__ int counter;
    unsigned long long t0, t1;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    const int lane = threadIdx.x;
    if (lane == 0) counter = 0;
    __syncwarp();
    double* const at[1] = {slot + lane};
    const bool need[1] = {true};
    double v[1];
    bool abort = false;
    poll_faces(at, need, v, abort, lane, err, FACE_LIMIT / 4);
    const bool polled = __all_sync(FULL, abort && v[0] == 0.0 && (lane > 0 || ld_relaxed_i(err) == 1));
    int seen = polled ? 1 : 0;
    if (lane == 0) atomicExch(err, 0);
    __syncwarp();
    await_level<32>(&counter, 1, lane, err, WAIT_LIMIT / 16);
    __syncwarp();
    if (lane == 0) {
        if (ld_relaxed_i(err) == 1) seen += 2;
        atomicExch(err, 0);
    }
    __syncwarp();
    await_data(&counter, 0, lane, err, WAIT_LIMIT / 16);
    __syncwarp();
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
    if (lane == 0) {
        if (ld_relaxed_i(err) == 1) seen += 4;
        out[0] = (long long)(t1 - t0);
        out[1] = seen;
    }
}
__global__ void k_fill_sentinel(double* __restrict__ p, size_t count) {
    const double sent = __longlong_as_double((long long)SENTINEL_BITS);
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < count;
         q += (size_t)gridDim.x * blockDim.x)
        p[q] = sent;
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
TileArgs tile_args(const bo_sim* s) {
    TileArgs a;
    a.g = s->geo;
    a.NJ = (s->geo.ny + TJ - 1) / TJ;
    a.NK = (s->geo.nz + TK - 1) / TK;
    a.T = a.NJ * a.NK;
    a.NL = s->geo.nx + TJ + TK - 2;
    a.NP = (size_t)a.T * a.NL * 32;
    a.err = s->d_sweep_sync + 2;
    a.ysub = s->ysub;
    a.zsub = s->zsub;
    return a;
}

// face buffers of the FP32 sweeps (3 values per slot)
size_t face_storage(const bo_sim* s) {
    const TileArgs a = tile_args(s);
    return (size_t)a.T * s->geo.nx * (TK + TJ) * 3;
}
double* faceJ3(bo_sim* s) { return s->d_face; }
double* faceK3(bo_sim* s) {
    TileArgs a = tile_args(s);
    return faceJ3(s) + (size_t)a.T * s->geo.nx * TK * 3;
}

void setup_sweeps(bo_sim* s) {
    BO_CUDA(cudaMemsetAsync(s->d_sweep_sync, 0, sizeof(int) * 4, s->stream));
    setup_sweeps64(s);
    setup_sweeps32(s);
}

// For the one-CTA solve, at its launch: what it reads is gathered once for every
// factorisation that it is used with, and for none that it is not.
void current_tile_factors(bo_sim* s) {
    if (s->tile_valid) return;
    const TileArgs a = tile_args(s);
    if (!s->d_P) {
        const size_t bytes = sizeof(double) * NPE * a.NP;
        BO_CUDA(cudaMalloc(reinterpret_cast<void**>(&s->d_P), bytes));
        BO_CUDA(cudaMemsetAsync(s->d_P, 0, bytes, s->stream));   // idle places
    }
    k_tile_factors<<<152 * 8, 256, 0, s->stream>>>(a, sweep_factors(s), s->d_P);
    count_launch(s, s->stream);
    BO_LAUNCH_CHECK("k_tile_factors");
    s->tile_valid = true;
}

// Sentinels of the current precision's sweeps (after a precision switch or an
// abandoned sweep).
void reset_sweep_faces(bo_sim* s) {
    fill_sweep_faces(s, s->mixed);
    if (s->mixed) reset_inbox(s, s->stream);   // the factorisation is FP64 in both
}

void fill_sweep_faces(bo_sim* s, bool fp32) {
    if (fp32)
        reset_faces32(s, s->stream);
    else
        reset_inbox(s, s->stream);
    BO_LAUNCH_CHECK("fill_sweep_faces");
}

// The forward sweep leaves y in the backward sweep's order (a work vector of its
// own in either precision) and the backward sweep writes z in natural order; the
// two always run as a pair (y is not needed in natural order).
void enqueue_fwd(bo_sim* s, cudaStream_t st, const double* r, double* y, const KrylovScalars* ks) {
    (void)y;
    if (s->mixed) {
        enqueue_fwd32(s, st, r, ks);
        return;
    }
    enqueue_fwd64(s, st, r, ks);
}

void enqueue_bwd(bo_sim* s, cudaStream_t st, double* z, const KrylovScalars* ks) {
    if (s->mixed) {
        enqueue_bwd32(s, st, z, ks);
        return;
    }
    enqueue_bwd64(s, st, z, ks);
}

void read_flags_async(bo_sim* s) {
    BO_CUDA(cudaMemcpyAsync(&s->h_flags->sweep_timeout, s->d_sweep_sync + 2, sizeof(int),
                            cudaMemcpyDeviceToHost, s->stream));
    s->h_flags->cpr_singular = 0;
    if (s->precond == BO_PRECOND_CPR)
        BO_CUDA(cudaMemcpyAsync(&s->h_flags->cpr_singular, cpr_status_ptr(s), sizeof(int),
                                cudaMemcpyDeviceToHost, s->stream));
}

// Runs waits that can only time out; returns the time they took.
double wait_selftest(bo_sim* s) {
    int* err = s->d_sweep_sync + 3;   // a flag of its own: the sweeps' flag stays clear
    long long* out = nullptr;
    double* slot = nullptr;           // a face slot of its own that nothing writes
    BO_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s->stream));
    BO_CUDA(cudaMalloc(&out, 2 * sizeof(long long)));
    BO_CUDA(cudaMalloc(&slot, 32 * sizeof(double)));
    k_fill_sentinel<<<1, 32, 0, s->stream>>>(slot, 32);
    count_launch(s, s->stream);
    k_wait_selftest<<<1, 32, 0, s->stream>>>(slot, err, out);
    count_launch(s, s->stream);
    BO_LAUNCH_CHECK("k_wait_selftest");
    long long h[2] = {0, 0};
    BO_CUDA(cudaMemcpyAsync(h, out, sizeof(h), cudaMemcpyDeviceToHost, s->stream));
    BO_CUDA(cudaStreamSynchronize(s->stream));
    cudaFree(out);
    cudaFree(slot);
    BO_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s->stream));
    if (h[1] != 7) fail(BO_ERR_STATE, "bounded-wait self-test: a wait did not run out as it should");
    return h[0] * 1e-9;
}

}  // namespace bo
