// FP32 operators on small grids, brick by brick.
//
// What bounds a small grid: latency.  The tile kernel of stencil.cu marches
// along z, one barrier and one exposed load latency per plane, 8 to 12 planes
// per chunk even at its shortest chunk, while most of the GPU is idle.  Here
// a CTA owns a brick of 16 x 4 x 4 nodes and works in three steps with two
// barriers: the brick's nodes with a halo of one into shared memory (all
// loads in flight at once), one element per thread and turn with its 24
// contributions to shared memory, and the sum of the 8 contributions with
// the epilogue at every node.  The elements on the brick's surface are
// computed by two to eight CTAs (1.66 elements per node), which costs
// arithmetic that an idle GPU has to spare and is why large grids keep the
// z-march (shared memory traffic: 16 128-bit accesses per element here).
// The correction of the coarse grid can be added while loading, which saves
// the prolongation's launch and its pass over the iterate.
#include "common.cuh"
#include "operator.cuh"
#include "opio.cuh"
#include "tail.cuh"

namespace topo {

namespace {

constexpr int BX = 16, BY = 4, BZ = 4, kThreads = BX * BY * BZ;   // (448 threads, every element in one turn, were 2 % slower)
constexpr int PX = BX + 2, PY = BY + 2, PZ = BZ + 2, kNodes = PX * PY * PZ;
constexpr int EX = BX + 1, EY = BY + 1, EZ = BZ + 1, kElems = EX * EY * EZ;
constexpr size_t kSmem = sizeof(float4) * (kNodes + 8 * kElems);

struct Coarser {          // correction of the next coarser level (P e)
    const float* e;
    const uint8_t* mask;
};

// trilinear interpolation of the masked coarse correction at fine node (i, j, k):
// in the plane first, then between planes, as k_prolong_z
__device__ __forceinline__ void interpolate(const Coarser& cr, int nx, int ny, int i, int j, int k, float* v) {
    const int NXc = nx / 2 + 1, NYc = ny / 2 + 1;
    const float w = ((i & 1) ? 0.5f : 1.0f) * ((j & 1) ? 0.5f : 1.0f);
    auto plane = [&](int K, float* s) {
        s[0] = s[1] = s[2] = 0.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int dx = q & 1, dy = q >> 1;
            if ((dx && !(i & 1)) || (dy && !(j & 1))) continue;
            const int N = (i >> 1) + dx + NXc * ((j >> 1) + dy + NYc * K);
            const unsigned m = cr.mask[N];
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (!((m >> c) & 1u)) s[c] += w * cr.e[3 * N + c];
        }
    };
    plane(k >> 1, v);
    if (k & 1) {
        float t[3];
        plane((k >> 1) + 1, t);
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] = 0.5f * (v[c] + t[c]);
    }
}

template <int MODE, bool DOT, bool PROLONG>
__global__ void __launch_bounds__(kThreads) k_brick(const ModalK<float> mk, const float* __restrict__ E,
                                                    const uint8_t* __restrict__ mask, const float* __restrict__ u,
                                                    const float* __restrict__ f, float* __restrict__ out, const int nx,
                                                    const int ny, const int nz, const float omega,
                                                    double* __restrict__ partials, float* __restrict__ pout,
                                                    const double* __restrict__ beta, const float* __restrict__ Dinv,
                                                    const Coarser cr, const DotTail tail) {
    extern __shared__ float4 smem[];
    float4* const val = smem;                 // node values, 0 at fixed DOFs and outside the grid
    float4* const con = smem + kNodes;        // con[a * kElems + e]: contribution of element e to its corner a
    __shared__ double sred[kThreads / 32];
    const int tid = threadIdx.x;
    const int NX = nx + 1, NY = ny + 1, NZ = nz + 1;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY, z0 = blockIdx.z * BZ;
    const float bet = MODE == ST_APPLY_P && beta ? (float)*beta : 0.0f;
    for (int t = tid; t < kNodes; t += kThreads) {
        const int i = x0 - 1 + t % PX, j = y0 - 1 + t / PX % PY, k = z0 - 1 + t / (PX * PY);
        float v[3] = {0.0f, 0.0f, 0.0f};
        if (i >= 0 && i < NX && j >= 0 && j < NY && k >= 0 && k < NZ) {
            const int n = i + NX * (j + NY * k);
            const unsigned m = mask[n];
            if constexpr (MODE == ST_JACOBI2) {   // u1 = omega D^-1 f
                const float d = Dinv[n];
#pragma unroll
                for (int c = 0; c < 3; ++c) v[c] = omega * f[3 * n + c] * d;
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) v[c] = u[3 * n + c];
                if constexpr (MODE == ST_APPLY_P)
                    if (beta) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) v[c] = v[c] + bet * f[3 * n + c];
                    }
                if constexpr (PROLONG) {
                    float e[3];
                    interpolate(cr, nx, ny, i, j, k, e);
#pragma unroll
                    for (int c = 0; c < 3; ++c) v[c] += e[c];
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if ((m >> c) & 1u) v[c] = 0.0f;
        }
        val[t] = make_float4(v[0], v[1], v[2], 0.0f);
    }
    __syncthreads();
    for (int e = tid; e < kElems; e += kThreads) {
        const int ex = e % EX, ey = e / EX % EY, ez = e / (EX * EY);
        const int i = x0 - 1 + ex, j = y0 - 1 + ey, k = z0 - 1 + ez;
        const bool ok = i >= 0 && i < nx && j >= 0 && j < ny && k >= 0 && k < nz;
        float c[8][3] = {};
        if (ok) {
            const float* s = reinterpret_cast<const float*>(val + ex + PX * (ey + PY * ez));
            float FB[12], FT[12], Bo[12], To[12];
#pragma unroll
            for (int a = 0; a < 8; ++a) ld3(s + 4 * ((a & 1) + PX * ((a >> 1 & 1) + PY * (a >> 2))), c[a]);
            face_forward<float>(c[0], c[1], c[2], c[3], FB);
            face_forward<float>(c[4], c[5], c[6], c[7], FT);
            element_modal<float>(mk, E[i + nx * (j + ny * k)], FB, FT, Bo, To);
            face_inverse<float>(Bo, c[0], c[1], c[2], c[3]);
            face_inverse<float>(To, c[4], c[5], c[6], c[7]);
        }
#pragma unroll
        for (int a = 0; a < 8; ++a) con[a * kElems + e] = make_float4(c[a][0], c[a][1], c[a][2], 0.0f);
    }
    __syncthreads();
    const int tx = tid % BX, ty = tid / BX % BY, tz = tid / (BX * BY);
    const int i = x0 + tx, j = y0 + ty, k = z0 + tz;
    float dot = 0.0f;
    if (i < NX && j < NY && k < NZ) {
        const int n = i + NX * (j + NY * k);
        float y[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            float v[3];
            ld3(reinterpret_cast<const float*>(
                    con + a * kElems + (tx + 1 - (a & 1)) + EX * ((ty + 1 - (a >> 1 & 1)) + EY * (tz + 1 - (a >> 2)))),
                v);
#pragma unroll
            for (int c = 0; c < 3; ++c) y[c] += v[c];
        }
        const unsigned m = mask[n];
        float uo[3];
        ld3(reinterpret_cast<const float*>(val + (tx + 1) + PX * ((ty + 1) + PY * (tz + 1))), uo);
        [[maybe_unused]] float d = 0.0f;
        if constexpr (MODE == ST_JACOBI || MODE == ST_JACOBI2) d = Dinv[n];
        // a node without stiffness has no diagonal: the sweep is not finite there
        if constexpr (MODE == ST_JACOBI)
            if (d == 0.0f) d = __int_as_float(0x7f800000);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const bool fixed = (m >> c) & 1u;
            const float fo = MODE == ST_APPLY || MODE == ST_APPLY_P ? 0.0f : f[3 * n + c];
            if (fixed) {   // val holds 0 there
                if constexpr (MODE == ST_JACOBI2) {
                    uo[c] = omega * fo;
                } else {
                    uo[c] = u[3 * n + c];
                    if constexpr (MODE == ST_APPLY_P)
                        if (beta) uo[c] = uo[c] + bet * f[3 * n + c];
                }
            }
            float r;
            if constexpr (MODE == ST_APPLY || MODE == ST_APPLY_P) {
                r = fixed ? uo[c] : y[c];
                if (DOT) dot += uo[c] * r;
                if constexpr (MODE == ST_APPLY_P) pout[3 * n + c] = uo[c];
            } else if constexpr (MODE == ST_RESID) {
                r = fo - (fixed ? uo[c] : y[c]);
                if (DOT) dot += r * r;
            } else {
                r = fixed ? uo[c] + omega * (fo - uo[c]) : uo[c] + omega * (fo - y[c]) * d;
                if (DOT) dot += fo * r;
            }
            out[3 * n + c] = r;
        }
    }
    if constexpr (DOT) {
        double v = (double)dot;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0) sred[tid >> 5] = v;
        __syncthreads();
        if (tid < 32) {
            double s = tid < kThreads / 32 ? sred[tid] : 0.0;
            for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (tid == 0) partials[blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)] = s;
        }
        dot_tail<kThreads>(tail, partials, gridDim.x * gridDim.y * gridDim.z, tid);
    }
}

// Residual and its restriction in one launch: a CTA owns 8 x 2 x 2 coarse nodes,
// computes the residual at the 17 x 5 x 5 fine nodes around them (1.66 times
// the nodes of a brick, from 648 elements) into shared memory and sums it with
// the weights of k_restrict_z.  Saves a launch and the residual's way through
// memory; only where launches count.  State step on 64x32x32 elements 15.3 ->
// 13.8 ms, V-cycle on 128x64x64 229 -> 212 us.
constexpr int RX = BX + 1, RY = BY + 1, RZ = BZ + 1, kResNodes = RX * RY * RZ;
constexpr int FX = BX + 2, FY = BY + 2, FZ = BZ + 2, kResElems = FX * FY * FZ;
constexpr int QX = BX + 3, QY = BY + 3, QZ = BZ + 3, kResHalo = QX * QY * QZ;
constexpr int kResThreads = 448;   // every residual in one turn (672, every element too, 1 % slower)
constexpr size_t kResSmem = sizeof(float4) * (kResHalo + 8 * kResElems);

__global__ void __launch_bounds__(kResThreads) k_brick_restrict(const ModalK<float> mk, const float* __restrict__ E,
                                                                const uint8_t* __restrict__ mask,
                                                                const float* __restrict__ u, const float* __restrict__ f,
                                                                const int nx, const int ny, const int nz,
                                                                const uint8_t* __restrict__ maskc,
                                                                float* __restrict__ fc) {
    extern __shared__ float4 smem[];
    float4* const val = smem;                  // node values from (x0 - 2, ..), then the residual from (x0 - 1, ..)
    float4* const con = smem + kResHalo;
    const int tid = threadIdx.x;
    const int NX = nx + 1, NY = ny + 1, NZ = nz + 1;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY, z0 = blockIdx.z * BZ;
    for (int t = tid; t < kResHalo; t += kResThreads) {
        const int i = x0 - 2 + t % QX, j = y0 - 2 + t / QX % QY, k = z0 - 2 + t / (QX * QY);
        float v[3] = {0.0f, 0.0f, 0.0f};
        if (i >= 0 && i < NX && j >= 0 && j < NY && k >= 0 && k < NZ) {
            const int n = i + NX * (j + NY * k);
            const unsigned m = mask[n];
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] = u[3 * n + c];
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if ((m >> c) & 1u) v[c] = 0.0f;
        }
        val[t] = make_float4(v[0], v[1], v[2], 0.0f);
    }
    // (the residual's own loads, in flight meanwhile; fixed DOFs restrict as 0)
    const int rx = tid % RX, ry = tid / RX % RY, rz = tid / (RX * RY);
    const int i = x0 - 1 + rx, j = y0 - 1 + ry, k = z0 - 1 + rz;
    const bool node = tid < kResNodes && i >= 0 && i < NX && j >= 0 && j < NY && k >= 0 && k < NZ;
    float r[3] = {0.0f, 0.0f, 0.0f};
    unsigned m = 7u;
    if (node) {
        const int n = i + NX * (j + NY * k);
        m = mask[n];
#pragma unroll
        for (int c = 0; c < 3; ++c) r[c] = f[3 * n + c];
    }
    __syncthreads();
    for (int e = tid; e < kResElems; e += kResThreads) {
        const int ex = e % FX, ey = e / FX % FY, ez = e / (FX * FY);
        const int ei = x0 - 2 + ex, ej = y0 - 2 + ey, ek = z0 - 2 + ez;
        float c[8][3] = {};
        if (ei >= 0 && ei < nx && ej >= 0 && ej < ny && ek >= 0 && ek < nz) {
            const float* s = reinterpret_cast<const float*>(val + ex + QX * (ey + QY * ez));
            float FB[12], FT[12], Bo[12], To[12];
#pragma unroll
            for (int a = 0; a < 8; ++a) ld3(s + 4 * ((a & 1) + QX * ((a >> 1 & 1) + QY * (a >> 2))), c[a]);
            face_forward<float>(c[0], c[1], c[2], c[3], FB);
            face_forward<float>(c[4], c[5], c[6], c[7], FT);
            element_modal<float>(mk, E[ei + nx * (ej + ny * ek)], FB, FT, Bo, To);
            face_inverse<float>(Bo, c[0], c[1], c[2], c[3]);
            face_inverse<float>(To, c[4], c[5], c[6], c[7]);
        }
#pragma unroll
        for (int a = 0; a < 8; ++a) con[a * kResElems + e] = make_float4(c[a][0], c[a][1], c[a][2], 0.0f);
    }
    __syncthreads();
    if (node) {
        float y[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            float v[3];
            ld3(reinterpret_cast<const float*>(
                    con + a * kResElems + (rx + 1 - (a & 1)) + FX * ((ry + 1 - (a >> 1 & 1)) + FY * (rz + 1 - (a >> 2)))),
                v);
#pragma unroll
            for (int c = 0; c < 3; ++c) y[c] += v[c];
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) r[c] = (m >> c) & 1u ? 0.0f : r[c] - y[c];
    }
    if (tid < kResNodes) val[tid] = make_float4(r[0], r[1], r[2], 0.0f);   // (val was last read before the barrier)
    __syncthreads();
    // coarse nodes, one thread per component
    if (tid >= 3 * (BX / 2) * (BY / 2) * (BZ / 2)) return;
    const int c = tid % 3, q = tid / 3, I = q % (BX / 2), J = q / (BX / 2) % (BY / 2), K = q / (BX / 2 * (BY / 2));
    const int Ig = x0 / 2 + I, Jg = y0 / 2 + J, Kg = z0 / 2 + K, NXc = nx / 2 + 1, NYc = ny / 2 + 1;
    if (Ig >= NXc || Jg >= NYc || Kg > nz / 2) return;
    const int N = Ig + NXc * (Jg + NYc * Kg);
    const float* w = reinterpret_cast<const float*>(val + 2 * I + RX * (2 * J + RY * 2 * K)) + c;
    float p[3];   // in-plane sums of the three fine planes
#pragma unroll
    for (int dz = 0; dz < 3; ++dz) {
        p[dz] = 0.0f;
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
                p[dz] += (dx == 1 ? 1.0f : 0.5f) * (dy == 1 ? 1.0f : 0.5f) * w[4 * (dx + RX * (dy + RY * dz))];
    }
    fc[3 * N + c] = (maskc[N] >> c) & 1u ? 0.0f : 0.5f * p[0] + p[1] + 0.5f * p[2];
}

dim3 brick_grid(const Geom& g) {
    return dim3((g.nx + BX) / BX, (g.ny + BY) / BY, (g.nz + BZ) / BZ);   // nodes: one more than elements
}

template <int MODE, bool DOT, bool PROLONG>
void launch(const Ctx& c, const Geom& g, const ModalK<float>& mk, const float* E, const uint8_t* mask, const float* u,
            const float* f, float* out, float omega, double* dot, const float* Dinv, float* pout, const double* beta,
            const Coarser& cr, const DotTail& tail) {
    k_brick<MODE, DOT, PROLONG><<<brick_grid(g), kThreads, kSmem, c.s>>>(mk, E, mask, u, f, out, g.nx, g.ny, g.nz, omega,
                                                                       dot, pout, beta, Dinv, cr, tail);
    TOPO_LAUNCH_CHECK(c);
}

}  // namespace

cudaError_t brick_init() {
    cudaError_t e = cudaSuccess;
    auto set = [&](auto k) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    };
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_brick_restrict, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem);
    set(k_brick<ST_APPLY_P, true, false>);
    set(k_brick<ST_APPLY, false, false>);
    set(k_brick<ST_JACOBI, true, true>);
    set(k_brick<ST_JACOBI, false, true>);
    set(k_brick<ST_JACOBI, true, false>);
    set(k_brick<ST_JACOBI, false, false>);
    set(k_brick<ST_JACOBI2, false, false>);
    set(k_brick<ST_RESID, false, false>);
    return e;
}

long long brick_ctas(const Geom& g) {
    const dim3 d = brick_grid(g);
    return (long long)d.x * d.y * d.z;
}

int brick_apply(const Ctx& c, int mode, const Geom& g, const ModalK<float>& mk, const float* E, const uint8_t* mask,
                const float* u, const float* f, float* out, float omega, double* dot, const float* Dinv, float* pout,
                const double* beta, const float* ec, const uint8_t* maskc, const DotTail& tail) {
    const Coarser cr{ec, maskc};
#define GO(MODE, DOT, PRO) launch<MODE, DOT, PRO>(c, g, mk, E, mask, u, f, out, omega, dot, Dinv, pout, beta, cr, tail)
    switch (mode) {
        case ST_APPLY_P: GO(ST_APPLY_P, true, false); break;   // CG only: always with p.q
        case ST_APPLY: GO(ST_APPLY, false, false); return 0;
        case ST_JACOBI:
            if (ec && dot) GO(ST_JACOBI, true, true);
            else if (ec) GO(ST_JACOBI, false, true);
            else if (dot) GO(ST_JACOBI, true, false);
            else GO(ST_JACOBI, false, false);
            break;
        case ST_JACOBI2: GO(ST_JACOBI2, false, false); return 0;
        default: GO(ST_RESID, false, false); return 0;
    }
#undef GO
    return dot ? (tail.kind != TAIL_NONE ? -1 : (int)brick_ctas(g)) : 0;
}

void brick_restrict(const Ctx& c, const Geom& g, const ModalK<float>& mk, const float* E, const uint8_t* mask,
                    const float* u, const float* f, const uint8_t* maskc, float* fc) {
    // bricks of coarse nodes: nx / 2 + 1 of them per axis
    const dim3 grid((g.nx / 2 + BX / 2) / (BX / 2), (g.ny / 2 + BY / 2) / (BY / 2), (g.nz / 2 + BZ / 2) / (BZ / 2));
    k_brick_restrict<<<grid, kResThreads, kResSmem, c.s>>>(mk, E, mask, u, f, g.nx, g.ny, g.nz, maskc, fc);
    TOPO_LAUNCH_CHECK(c);
}

}  // namespace topo
