// Device-side state and deterministic reductions shared by the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "host_common.h"

namespace fftg {

constexpr int kThreads = 256;

// Device material table: per phase K, G, sigma_0, H, n, eps_0, t_0, model
// (the fields of fftg_phase, the model id as a double), and 1 / (3G + H), the
// slope's reciprocal of the linear return.
constexpr int kMatStride = 9;
enum : int { MODEL_J2 = 0, MODEL_NLELASTIC = 1, MODEL_VISCO = 2 };

// Roundoff floor (relative to the norm of the projected field) below which a
// CG residual is treated as FFT roundoff; see the CG readings.
constexpr double kRoundoffRel = 1e-13;

// CG status values in CGState::done. CG_STAGNATED ends an inner (FP32)
// solve that has stopped improving: no new minimum of <r, r> for
// `stag_window` iterations, or a finite <p, q> <= 0 (rounding noise has
// overtaken the search direction). The iterate is kept and the FP64 Newton
// iteration refines it. CG_BREAKDOWN is a NaN or Inf.
enum : int { CG_RUNNING = 0, CG_CONVERGED = 1, CG_MAXIT = 2, CG_BREAKDOWN = 3, CG_STAGNATED = 4 };

// State of one CG solve (one right-hand side), resident on the device so
// that the iteration needs no host round trip. The last block of each
// reducing kernel updates it.
struct CGState {
    double rr;       // <r, r> of the current residual
    double rr0;      // <r0, r0>
    double gs2;      // ||G sigma||^2 of the right-hand side before rounding
    double tol2;     // relative tolerance squared (set by the host)
    double floor2;   // absolute roundoff floor squared
    double stop2;    // max(tol2 * rr0, floor2)
    double pq;       // <p, q>
    double alpha;
    double beta;
    double omega;    // > 0: Richardson iteration with this fixed step (the
                     // basic scheme, Section 3.2) instead of CG; 0: CG
    double rr_min;   // smallest <r, r> so far
    int it_min;      // iteration of rr_min
    int stag_window; // > 0: stagnation test window (set by the host)
    int it;          // iterations done
    int max_it;      // cap (set by the host)
    int fixed_it;    // > 0: exactly this many iterations (set by the host)
    int done;        // CG_* status
    unsigned int ticket;  // last-block counter (always 0 between kernels)
    int pend;        // 1: x still lacks alpha p of the last update (the next
                     // P1 or the finishing kernel adds it)
};

// Scalars of one Newton iteration / one constitutive evaluation.
struct NewtonDev {
    double sig2;      // ||sigma||^2 (Frobenius, summed over voxels)
    double sum[6];    // sum of sigma over voxels, per component
    double de2;       // ||d eps||^2 of the last Newton update
    double extra[8];  // reductions of auxiliary kernels (tangent averages)
    unsigned int ticket;
    int nplastic;     // unused slot kept for alignment
};

// Transitions of a CGState, taken by thread 0 of the last block of a
// reducing kernel once the block totals are in.
//
// Start of a solve, after the right-hand side pass: rr = <r0, r0> in the
// inner precision, gs2 = ||G sigma||^2 before rounding to it.
__device__ __forceinline__ void cg_start(CGState* cg, double rr, double gs2) {
    cg->rr = rr;
    cg->rr0 = rr;
    cg->rr_min = rr;
    cg->it_min = 0;
    cg->gs2 = gs2;
    cg->it = 0;
    cg->beta = 0.0;
    cg->alpha = 0.0;
    const double stop2 = fmax(cg->tol2 * rr, cg->floor2);
    cg->stop2 = stop2;
    if (!isfinite(rr) || !isfinite(gs2)) {
        cg->done = CG_BREAKDOWN;
    } else if (gs2 <= cg->floor2 || rr == 0.0) {
        cg->done = CG_CONVERGED;
    } else if (cg->fixed_it <= 0 && rr <= stop2) {
        cg->done = CG_CONVERGED;
    } else {
        cg->done = CG_RUNNING;
    }
}

// Sets a solve's state from a kernel argument: no host memory has to stay
// unchanged until the stream gets here.
static __global__ void k_set_cg(CGState* cg, CGState value) { *cg = value; }

// After the matvec of an iteration: alpha = <r, r>/<p, q>, or the fixed
// Richardson step.
__device__ __forceinline__ void cg_after_dot(CGState* cg, double pq) {
    cg->pq = pq;
    cg->pend = 0;  // P1 of this iteration has added the previous step
    if (!isfinite(pq)) {
        cg->done = CG_BREAKDOWN;
    } else if (cg->omega > 0.0) {
        cg->alpha = cg->omega;  // Richardson: fixed step, <p, q> unused
    } else if (!(pq > 0.0)) {
        cg->done = cg->stag_window > 0 ? CG_STAGNATED : CG_BREAKDOWN;
    } else {
        cg->alpha = cg->rr / pq;
    }
}

// After r -= alpha q: rr = <r, r>; beta and the stopping tests. The step
// x += alpha p is left pending.
__device__ __forceinline__ void cg_after_update(CGState* cg, double rr) {
    const int it = cg->it + 1;
    cg->it = it;
    cg->pend = 1;
    cg->beta = cg->omega > 0.0 ? 0.0 : rr / cg->rr;  // Richardson: p = r
    cg->rr = rr;
    if (!isfinite(rr)) {
        cg->done = CG_BREAKDOWN;
    } else if (cg->fixed_it > 0) {
        if (it >= cg->fixed_it) cg->done = CG_CONVERGED;
    } else if (rr <= cg->stop2) {
        cg->done = CG_CONVERGED;
    } else if (it >= cg->max_it) {
        cg->done = CG_MAXIT;
    } else if (cg->stag_window > 0) {
        if (rr < cg->rr_min) {
            cg->rr_min = rr;
            cg->it_min = it;
        } else if (it - cg->it_min >= cg->stag_window) {
            cg->done = CG_STAGNATED;
        }
    }
}

// Frobenius product of symmetric tensors stored as 6 components
template <typename T>
__device__ __forceinline__ T frob(const T* a, const T* b) {
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2] + T(2) * (a[3] * b[3] + a[4] * b[4] + a[5] * b[5]);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over a block of kThreads threads (1D); result valid in every thread.
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double red[kThreads / 32];
    __shared__ double total;
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    if (wid == 0) {
        double s = (lane < kThreads / 32) ? red[lane] : 0.0;
        s = warp_sum(s);
        if (lane == 0) total = s;
    }
    __syncthreads();
    return total;
}

// Sum over a block of any size up to 1024 threads (1D), in a fixed order
// (lanes by shuffles, then the warps in index order); result in thread 0.
__device__ __forceinline__ double block_sum_any(double v) {
    __shared__ double red_any[32];
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) red_any[wid] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < nw; ++w) s += red_any[w];
    return s;
}

// Sum of the partials in[0 .. nb) at stride `st` in a fixed order over the
// block; valid in thread 0.
__device__ __forceinline__ double sum_partials(const double* in, int nb, int st) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) acc += in[(size_t)b * st];
    return block_sum_any(acc);
}

// Start of the solves of a right-hand side from its pass's block partials
// ([nf][nb][2]: <r, r> and the squared norm before rounding), one block per
// field.
static __global__ void __launch_bounds__(1024) k_cg_begin(const double* partials, int nb, CGState* cg,
                                                          const int* active) {
    const int f = blockIdx.x;
    if (active && !active[f]) return;
    const double* in = partials + (size_t)f * nb * 2;
    const double rr = sum_partials(in, nb, 2);
    const double gs2 = sum_partials(in + 1, nb, 2);
    if (threadIdx.x == 0) cg_start(cg + f, rr, gs2);
}

// <r, r> of a CG iteration from the block partials of its last pass
// ([nf][nb], one per block): one block per field sums them in a fixed order
// and takes the CG state's update step (beta and the stopping tests).
__device__ __forceinline__ void cg_rr_block(const double* partials, int nb, CGState* cg) {
    const int f = blockIdx.x;
    if (cg[f].done) return;
    const double acc = sum_partials(partials + (size_t)f * nb, nb, 1);
    if (threadIdx.x == 0) cg_after_update(cg + f, acc);
}
static __global__ void __launch_bounds__(1024) k_cg_rr(const double* partials, int nb, CGState* cg) {
    cg_rr_block(partials, nb, cg);
}

// Store this block's NV partial sums and report whether this block is the
// last one of `nblocks` to do so. Partials of the other blocks are then
// visible to it (fence before the ticket).
template <int NV>
__device__ __forceinline__ bool publish_partials(const double (&v)[NV], double* partials, int bid,
                                                 int nblocks, unsigned int* ticket) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int j = 0; j < NV; ++j) partials[(size_t)bid * NV + j] = v[j];
        __threadfence();
        unsigned int prev = atomicAdd(ticket, 1u);
        last = (prev == (unsigned int)(nblocks - 1));
    }
    __syncthreads();
    return last;
}

// In the last block: totals over all blocks in a fixed order (thread i takes
// blocks i, i + kThreads, ...; then a fixed tree), so the result does not
// depend on which block finished last. Resets the ticket.
template <int NV>
__device__ __forceinline__ void reduce_partials(const double* partials, int nblocks, unsigned int* ticket,
                                                double (&tot)[NV]) {
    __threadfence();
    double acc[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) acc[j] = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kThreads) {
#pragma unroll
        for (int j = 0; j < NV; ++j) acc[j] += __ldcg(partials + (size_t)b * NV + j);
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) tot[j] = block_sum(acc[j]);
    if (threadIdx.x == 0) *ticket = 0u;
}

// The allocation that a caller's buffer starts in (host_common.h), as the
// driver reports it. The range is the driver API's to give; its entry point is
// looked up once.
inline BufferRange buffer_range(const void* p) {
    using GetRange = int (*)(unsigned long long*, size_t*, unsigned long long);
    static const GetRange get = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return (GetRange)f;
    }();
    BufferRange r;
    cudaPointerAttributes at{};
    int dev = -1;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return r;
    }
    r.here = at.type == cudaMemoryTypeManaged || (at.type == cudaMemoryTypeDevice && at.device == dev);
    unsigned long long base = 0;
    if (r.here && get && get(&base, &r.size, (unsigned long long)(uintptr_t)p) == 0)
        r.base = (uintptr_t)base;
    else
        r.size = 0;
    return r;
}
inline bool in_place(const void* p, size_t bytes, size_t es) { return usable_in_place(buffer_range(p), p, bytes, es); }

}  // namespace fftg
