// Deterministic block reductions shared by the FGMRES kernels.
#pragma once

#include "common.cuh"

namespace abilu {

constexpr int RED_THREADS = 256;
constexpr int RED_WARPS = RED_THREADS / 32;

// Block-wide sum of K values per thread; result in sh_out[k], k < kn (valid
// after the call's final barrier).  sh_w holds K * TH doubles, TH the CTA's
// threads.  The
// values are staged in shared memory and warp k sums value k: each lane adds
// its TH / 32 values (threads lane, lane + 32, ...) in order, then a 5-level
// shuffle tree.  A fixed order, so deterministic.  This GPU has two FP64 lanes
// per SM, so a warp-wide FP64 add occupies its FP64 pipe for 16 cycles
// whatever the lanes do: per value this form issues 12 warp-wide FP64 adds
// where a shuffle tree in every warp and a cross-warp stage issued 43-48,
// which was most of the gap between the dot kernels and their FMA floor.
template <int K, int TH = RED_THREADS>
__device__ __forceinline__ void block_sum(double (&v)[K], double *sh_w, double *sh_out, int kn) {
#pragma unroll
    for (int k = 0; k < K; k++) sh_w[k * TH + threadIdx.x] = v[k];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < kn; k += TH / 32) {
        const double *p = sh_w + k * TH + lane;
        double s = p[0];
#pragma unroll
        for (int r = 1; r < TH / 32; r++) s += p[32 * r];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) sh_out[k] = s;
    }
    __syncthreads();
}

// Whether this CTA is the last of `total` to arrive at *counter with its
// partials stored; every thread of the CTA calls it.  (A fence by the first
// warp alone, which stores the partials, was slower: fused product and dots of
// the 2.6 M-row batch 348 against 331 us.)
__device__ __forceinline__ bool last_arrival(unsigned *counter, unsigned total) {
    __shared__ bool am_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) am_last = atomicAdd(counter, 1u) == total - 1;
    __syncthreads();
    if (am_last) __threadfence();
    return am_last;
}

// ---- the Givens update of a single-reduction Arnoldi step
//
// What it reads of a solve's state besides the new column, staged in shared
// memory by the last CTA of a reduction while it reduces the partials, so that
// the serial FP64 chain reads no global memory (an FP64 operation takes 64
// cycles on this GPU and an L2 load several hundred).
constexpr int GIVENS_MAX = 64;
struct GivensIn {
    double cs[GIVENS_MAX], sn[GIVENS_MAX], gj, bnorm;
    int iters;
    double h[GIVENS_MAX + 1];   // the column's coefficients, h[0..j], by the caller
    double ww;                  // ||w||^2, by the caller
    double a, t, hn;            // between the two warps
};
template <typename State>
__device__ __forceinline__ void givens_stage(const State *S, int j, GivensIn *G) {
    for (int i = threadIdx.x; i < j; i += blockDim.x) {
        G->cs[i] = S->cs[i];
        G->sn[i] = S->sn[i];
    }
    switch (threadIdx.x) {
    case 0: G->gj = S->g[j]; break;
    case 1: G->bnorm = S->bnorm; break;
    case 2: G->iters = S->iters; break;
    default: break;
    }
}

// h_{j+1,j} = sqrt(||w||^2 - sum_k h_k^2) (Pythagoras: w - V h is orthogonal to
// V_0..V_j when they are orthonormal, so the norm needs neither a pass over the
// updated w nor a second reduction), the update of column j, the residual
// estimate and the end-of-cycle test.  Every thread of the CTA calls it, with
// *G staged and a barrier behind it; returns done in thread 0.  A difference below
// 1e-12 ||w||^2 (more than twelve digits cancelled, or negative) is taken as a
// breakdown: the cycle ends at this column and the explicit FP64 residual at its
// end decides whether it restarts.
//
// The chain is what a small solve waits for (an FP64 square root takes about
// 660 cycles, a division 420), so its parts run side by side: the second warp
// carries the column through the earlier rotations while the first forms h_{j+1,j};
// the rotation's length comes from h_{j+1,j}^2 (no second root in sequence); the
// four divisions are one instruction sequence in four lanes.
template <typename State>
__device__ __forceinline__ int givens_update(State *S, int j, GivensIn *G, double rtol, int max_iters,
                                             int m) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        double hh = 0.0;
        for (int k = lane; k <= j; k += 32) hh = fma(G->h[k], G->h[k], hh);
        for (int o = 16; o > 0; o >>= 1) hh += __shfl_down_sync(0xffffffffu, hh, o);
        if (lane == 0) {
            const double ww = G->ww, d = ww - hh;
            const double t = d > 1e-12 * ww ? d : 0.0;
            const double hn = sqrt(t);
            G->t = t;
            G->hn = hn;
        }
    } else if (warp == 1 && lane == 0) {
        // the previous rotations, i = 0 .. j-1, each mixing entries i and i+1 of
        // the new column: one carried value
        double a = G->h[0];
        for (int i = 0; i < j; i++) {
            const double c = G->h[i + 1];
            S->H[i * GIVENS_MAX + j] = G->cs[i] * a + G->sn[i] * c;
            a = -G->sn[i] * a + G->cs[i] * c;
        }
        G->a = a;
    }
    __syncthreads();
    if (warp != 0) return 0;
    const double a = G->a, hn = G->hn, gj = G->gj;
    const double d = sqrt(fma(a, a, G->t));
    const double num = lane == 0 ? a : lane == 1 ? hn : lane == 2 ? gj : 1.0;
    const double den = lane < 2 ? d : lane == 2 ? G->bnorm : hn;
    const double r = den != 0.0 ? num / den : (lane == 0 ? 1.0 : 0.0);
    if (lane == 3) S->hn_inv = r;
    const double cs = __shfl_sync(0xffffffffu, r, 0), sn = __shfl_sync(0xffffffffu, r, 1);
    const double rel = __shfl_sync(0xffffffffu, r, 2);   // g_j / ||b||
    if (lane != 0) return 0;
    const double g1 = -sn * gj;
    S->cs[j] = cs;
    S->sn[j] = sn;
    S->H[j * GIVENS_MAX + j] = cs * a + sn * hn;
    S->g[j + 1] = g1;
    S->g[j] = cs * gj;
    const int iters = G->iters + 1;
    S->iters = iters;
    S->kdim = j + 1;
    S->est = fabs(sn * rel);
    S->breakdown = hn == 0.0 ? 1 : 0;
    const int done = (fabs(g1) <= rtol * G->bnorm || hn == 0.0 || iters >= max_iters || j + 1 >= m) ? 1 : 0;
    S->done = done;
    S->counter = 0;
    return done;
}

}  // namespace abilu
