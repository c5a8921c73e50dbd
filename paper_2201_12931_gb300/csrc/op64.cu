// FP64 operator by elements: every element once, then a gather per node.
//
// What bounds the FP64 operator: FP64 instructions run at 2 lanes per clock
// and SM on this part, about 150 of them per element.  The tile kernel of
// stencil.cu (k_op) recomputes a halo of elements per tile and a layer per
// z chunk, and a CTA of 8 warps needs 8.7 us of the SM's FP64 pipe per layer,
// so that a grid of a few tiles keeps most SMs idle: 70 us per operator on
// 48x24x24 elements and still on 24x12x12.  Here a thread computes a short
// column of elements (cz layers, chosen by op64_plan) from its nodes with
// the modal arithmetic of operator.cuh and writes the contributions of its
// faces to a scratch array (no shared memory, no barrier, blocks of one
// warp: the work spreads over all SMs in units of 32 columns); a second
// kernel sums the contributions at every node in a fixed order and applies
// the epilogue, with the stored D^-1 in place of 1 / (kdiag sum E), a
// division of about 10 FP64 instructions.  Measured: a state step on 48x24x24
// elements (3 levels, 19 iterations) 16.6 -> 10.2 ms by this alone (5.4 with the
// later coarsest factorization and reductions), the compliance gradient on
// 96x48x48 48.7 -> 26.0 (19.8) ms, K.u over 128x64x64 elements 258 -> 189 us.
#include <algorithm>

#include "common.cuh"
#include "operator.cuh"
#include "tail.cuh"

namespace topo {

namespace {

enum InMode { IN_U, IN_P, IN_F };

// What the elements read at a node: u (IN_U), p = u + beta f (IN_P: u = z, f =
// the old direction, no beta: u), or u1 = omega D^-1 f (IN_F); 0 at fixed DOFs
template <int IN>
__device__ __forceinline__ void node_value(const double* __restrict__ u, const double* __restrict__ f,
                                           const double* __restrict__ Dinv, const uint8_t* __restrict__ mask, int n,
                                           double omega, double beta, bool has_beta, double* v) {
    const unsigned m = mask[n];
    if constexpr (IN == IN_F) {
        const double s = omega * Dinv[n];
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] = ((m >> c) & 1u) ? 0.0 : f[3 * n + c] * s;
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double t = u[3 * n + c];
            if constexpr (IN == IN_P)
                if (has_beta) t = fma(beta, f[3 * n + c], t);
            v[c] = ((m >> c) & 1u) ? 0.0 : t;
        }
    }
}

template <int IN>
__global__ void __launch_bounds__(32) k_el64(const ModalK<double> mk, const double* __restrict__ E,
                                             const uint8_t* __restrict__ mask, const double* __restrict__ u,
                                             const double* __restrict__ f, const double* __restrict__ Dinv, int nx,
                                             int ny, int nz, int cz, double omega, const double* __restrict__ beta,
                                             double* __restrict__ scratch) {
    const int ncol = nx * ny, nt = ncol * ((nz + cz - 1) / cz);
    const int t = blockIdx.x * 32 + threadIdx.x;
    if (t >= nt) return;
    const int col = t % ncol, i = col % nx, j = col / nx;
    const int k0 = t / ncol * cz, k1 = min(k0 + cz, nz);
    const int NX = nx + 1, plane = NX * (ny + 1), n0 = i + NX * j;
    const double b = IN == IN_P && beta ? *beta : 0.0;
    const bool hb = IN == IN_P && beta;
    auto face = [&](int k, double* F) {
        double c00[3], c10[3], c01[3], c11[3];
        const int n = n0 + plane * k;
        node_value<IN>(u, f, Dinv, mask, n, omega, b, hb, c00);
        node_value<IN>(u, f, Dinv, mask, n + 1, omega, b, hb, c10);
        node_value<IN>(u, f, Dinv, mask, n + NX, omega, b, hb, c01);
        node_value<IN>(u, f, Dinv, mask, n + NX + 1, omega, b, hb, c11);
        face_forward<double>(c00, c10, c01, c11, F);
    };
    auto put = [&](int fc, const double* A) {
        double c[4][3];
        face_inverse<double>(A, c[0], c[1], c[2], c[3]);
        double* s = scratch + (long long)fc * 12 * nt + t;
#pragma unroll
        for (int q = 0; q < 12; ++q) s[(long long)q * nt] = c[q / 3][q % 3];
    };
    double lo[12], hi[12], top[12], Bo[12], To[12];
    face(k0, lo);
#pragma unroll
    for (int q = 0; q < 12; ++q) top[q] = 0.0;
    for (int k = k0; k < k1; ++k) {
        face(k + 1, hi);
        element_modal<double>(mk, E[col + (long long)ncol * k], lo, hi, Bo, To);
        if (k > k0) {
#pragma unroll
            for (int q = 0; q < 12; ++q) Bo[q] += top[q];
        }
        put(k - k0, Bo);
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            top[q] = To[q];
            lo[q] = hi[q];
        }
    }
    put(k1 - k0, top);
}

// Node gather and epilogue (the modes of k_op).  The contributions of column
// (i - ax, j - ay) at its corner ax + 2 ay: one face where both layers around
// the node are in one chunk, else the top face of the lower chunk and the
// bottom face of the upper one.
template <int MODE, bool DOT>
__global__ void __launch_bounds__(128) k_node64(const double* __restrict__ scratch, const uint8_t* __restrict__ mask,
                                                const double* __restrict__ u, const double* __restrict__ f,
                                                const double* __restrict__ Dinv, double* __restrict__ out, int nx,
                                                int ny, int nz, int cz, double omega, double* __restrict__ partials,
                                                double* __restrict__ pout, const double* __restrict__ beta,
                                                const DotTail tail) {
    __shared__ double sred[4];
    const int NX = nx + 1, NY = ny + 1, nn = NX * NY * (nz + 1);
    const int ncol = nx * ny, nt = ncol * ((nz + cz - 1) / cz);
    const int n = blockIdx.x * 128 + threadIdx.x;
    double dot = 0.0;
    if (n < nn) {
        const int i = n % NX, j = (n / NX) % NY, k = n / (NX * NY);
        const int qu = k / cz, ql = k > 0 ? (k - 1) / cz : -1;
        const bool up = k < nz && qu != ql;   // a bottom face of its own chunk
        double y[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int ay = 0; ay < 2; ++ay)
#pragma unroll
            for (int ax = 0; ax < 2; ++ax) {
                const int ci = i - ax, cj = j - ay;
                if (ci < 0 || ci >= nx || cj < 0 || cj >= ny) continue;
                const int col = ci + nx * cj, a = ax + 2 * ay;
                if (ql >= 0) {
                    const double* s = scratch + (long long)((k - ql * cz) * 12 + 3 * a) * nt + col + ncol * ql;
#pragma unroll
                    for (int c = 0; c < 3; ++c) y[c] += s[(long long)c * nt];
                }
                if (up) {
                    const double* s = scratch + (long long)(3 * a) * nt + col + ncol * qu;
#pragma unroll
                    for (int c = 0; c < 3; ++c) y[c] += s[(long long)c * nt];
                }
            }
        const unsigned m = mask[n];
        double d = (MODE == ST_JACOBI || MODE == ST_JACOBI2) ? omega * Dinv[n] : 0.0;
        // a node without stiffness has no diagonal: the sweep is not finite there
        if constexpr (MODE == ST_JACOBI)
            if (__double2hiint(d) == 0) d = __longlong_as_double(0x7ff0000000000000ll);
        const double b = MODE == ST_APPLY_P && beta ? *beta : 0.0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const bool fixed = (m >> c) & 1u;
            const double fo = MODE == ST_APPLY || MODE == ST_APPLY_P ? 0.0 : f[3 * n + c];
            double uo = 0.0, r;
            if constexpr (MODE != ST_JACOBI2) uo = u[3 * n + c];
            if constexpr (MODE == ST_APPLY_P) {
                if (beta) uo = fma(b, f[3 * n + c], uo);
                pout[3 * n + c] = uo;
            }
            if constexpr (MODE == ST_APPLY || MODE == ST_APPLY_P) {
                r = fixed ? uo : y[c];
                if (DOT) dot = fma(uo, r, dot);
            } else if constexpr (MODE == ST_RESID) {
                r = fo - (fixed ? uo : y[c]);
                if (DOT) dot = fma(r, r, dot);
            } else if constexpr (MODE == ST_JACOBI2) {
                const double u1 = fixed ? omega * fo : fo * d;
                r = fixed ? u1 + omega * (fo - u1) : fma(fo - y[c], d, u1);
            } else {
                r = fixed ? uo + omega * (fo - uo) : fma(fo - y[c], d, uo);
                if (DOT) dot = fma(fo, r, dot);
            }
            out[3 * n + c] = r;
        }
    }
    if constexpr (DOT) {
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        if ((threadIdx.x & 31) == 0) sred[threadIdx.x >> 5] = dot;
        __syncthreads();
        if (threadIdx.x == 0) partials[blockIdx.x] = (sred[0] + sred[1]) + (sred[2] + sred[3]);
        dot_tail<128>(tail, partials, gridDim.x, threadIdx.x);
    }
}

}  // namespace

// Layers per thread: the time of the fullest scheduler in both kernels.  Each of
// the four schedulers of an SM takes 64 clocks per FP64 warp instruction (half
// a lane per clock; a lone warp measured 78), so a grid wants at least four
// warps per SM: 48x24x24 elements in 144 warps of 6 layers took 36 us.  A
// thread of cz layers costs 48 (cz + 1) + 80 cz + 12 (cz - 1) instructions, a
// node 15 + 12 / cz.
Op64Plan op64_plan(const Geom& g, int nsm) {
    Op64Plan p;
    double best = -1.0;
    const long long units = 4ll * nsm;
    for (int cz = 1; cz <= 8 && cz <= g.nz; ++cz) {
        const long long warps = ((long long)g.nx * g.ny * ((g.nz + cz - 1) / cz) + 31) / 32;
        const double el = (double)((warps + units - 1) / units) * (48.0 * (cz + 1) + 80.0 * cz + 12.0 * (cz - 1));
        const double nd = (double)((g.nn + 32 * units - 1) / (32 * units)) * (15.0 + 12.0 / cz);
        if (best < 0.0 || el + nd < best) {
            best = el + nd;
            p.cz = cz;
        }
    }
    p.nt = (long long)g.nx * g.ny * ((g.nz + p.cz - 1) / p.cz);
    p.blocks = (int)((g.nn + 127) / 128);
    return p;
}

int op64_apply(const Ctx& c, int mode, const Geom& g, const Op64Plan& p, const ModalK<double>& mk, const double* E,
               const uint8_t* mask, const double* u, const double* f, double* out, double omega, double* dot,
               const double* Dinv, double* pout, const double* beta, double* scratch, const DotTail& tail) {
    const unsigned ge = (unsigned)((p.nt + 31) / 32), gn = (unsigned)p.blocks;
#define EL(IN) \
    k_el64<IN><<<ge, 32, 0, c.s>>>(mk, E, mask, u, f, Dinv, g.nx, g.ny, g.nz, p.cz, omega, beta, scratch)
#define ND(MODE, DOT)                                                                                               \
    k_node64<MODE, DOT><<<gn, 128, 0, c.s>>>(scratch, mask, u, f, Dinv, out, g.nx, g.ny, g.nz, p.cz, omega, dot, pout, \
                                             beta, tail)
    if (mode == ST_APPLY_P) EL(IN_P);
    else if (mode == ST_JACOBI2) EL(IN_F);
    else EL(IN_U);
    TOPO_LAUNCH_CHECK(c);
    switch (mode) {
        case ST_APPLY: ND(ST_APPLY, false); break;
        case ST_APPLY_P: ND(ST_APPLY_P, true); break;   // CG only: always with p.q
        case ST_JACOBI:
            if (dot) ND(ST_JACOBI, true);
            else ND(ST_JACOBI, false);
            break;
        case ST_JACOBI2: ND(ST_JACOBI2, false); break;
        default:
            if (dot) ND(ST_RESID, true);
            else ND(ST_RESID, false);
            break;
    }
    TOPO_LAUNCH_CHECK(c);
#undef EL
#undef ND
    return mode == ST_JACOBI2 || mode == ST_APPLY || !dot ? 0 : (tail.kind != TAIL_NONE ? -1 : p.blocks);
}

}  // namespace topo
