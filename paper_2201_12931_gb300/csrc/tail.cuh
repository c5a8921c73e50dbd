// Scalar steps of CG (Algorithm 1) and the reduction that feeds them, run by
// the last block of the kernel that wrote the partial sums.
#pragma once

#include "common.cuh"

namespace topo {

// alpha = rz / p.q, beta = rz_new / rz, or r.r from a finished sum; aux = 1 is
// the breakdown flag that the host reads
__device__ __forceinline__ void cg_scalar(int kind, double s, Scalars* sc, double* hist) {
    if (kind == TAIL_ALPHA) {
        sc->pq = s;
        if (s > 0.0 && isfinite(s) && isfinite(sc->rz)) {
            sc->alpha = sc->rz / s;
        } else {
            sc->alpha = 0.0;
            sc->aux = 1.0;
        }
        if (hist) *hist = sc->alpha;
    } else if (kind == TAIL_BETA) {
        const double old = sc->rz;
        sc->rz_old = old;
        sc->rz_new = s;
        sc->beta = (old != 0.0 && isfinite(s)) ? s / old : 0.0;
        if (!isfinite(s)) sc->aux = 1.0;
        sc->rz = s;
    } else {
        sc->rr = s;
    }
}

// Called by all THREADS threads of every block after thread 0 has written its
// block's partial sum: the last block to arrive sums them in a fixed order
// and runs the scalar step.  Replaces a launch of one block (3 of about 25
// launches of an iteration on a small grid).
template <int THREADS>
__device__ __forceinline__ void dot_tail(const DotTail& t, const double* partials, unsigned blocks, int tid) {
    if (t.kind == TAIL_NONE) return;
    __shared__ unsigned last;
    __shared__ double red[THREADS / 32];
    if (tid == 0) {
        __threadfence();
        last = atomicAdd(t.ticket, 1u) == blocks - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s = 0.0;
    for (unsigned i = tid; i < blocks; i += THREADS) s += __ldcg(partials + i);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((tid & 31) == 0) red[tid >> 5] = s;
    __syncthreads();
    if (tid >= 32) return;
    static_assert(THREADS / 32 <= 16, "one half-warp holds the warps' sums");
    s = tid < THREADS / 32 ? red[tid] : 0.0;
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (tid == 0) {
        cg_scalar(t.kind, s, t.sc, t.hist);
        *t.ticket = 0;
    }
}

}  // namespace topo
