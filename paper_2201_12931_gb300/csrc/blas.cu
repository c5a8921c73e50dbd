// Vector kernels of the CG loop (Algorithm 1: dots, alpha/beta, x/r/p updates;
// all on the device, no host round trip per iteration) and the dense direct
// solve on the coarsest grid (Algorithm 3 "Solve the problem directly"):
// blocked right-looking Cholesky K_c = L L^T, explicit W = L^-1, and per
// application u = W^T (W r) as two triangular matrix-vector products.
// Reductions add their blocks' partial sums in a fixed order, in a second pass
// (k_reduce_to, k_cg_scalar) or in the last block to finish (tail.cuh), over
// grids that are fixed per handle, so results are bitwise
// reproducible run to run.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fp64.cuh"
#include "tail.cuh"

namespace topo {

namespace {

constexpr int TB = 32;   // dense tile

inline unsigned grid_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    if (b > 2147483647LL) b = 2147483647LL;
    return (unsigned)(b < 1 ? 1 : b);
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
    if (w == 0) {
        t = (l < (int)(blockDim.x >> 5)) ? sh[l] : 0.0;
        t = warp_sum(t);
    }
    return t;
}

template <typename A, typename B>
__global__ void __launch_bounds__(256) k_dot(long long n, const A* __restrict__ a, const B* __restrict__ b,
                                             double* __restrict__ partials) {
    __shared__ double sh[32];
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        s += (double)a[i] * (double)b[i];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

__device__ __forceinline__ double sum_partials(const double* __restrict__ p, int n, double* sh) {
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += p[i];
    return block_sum(s, sh);
}

__global__ void __launch_bounds__(1024) k_reduce_to(const double* __restrict__ p, int n, double* dst) {
    __shared__ double sh[32];
    const double s = sum_partials(p, n, sh);
    if (threadIdx.x == 0) *dst = s;
}

__global__ void __launch_bounds__(1024) k_cg_scalar(int kind, const double* __restrict__ p, int n, Scalars* sc,
                                                    double* __restrict__ hist) {
    __shared__ double sh[32];
    const double s = sum_partials(p, n, sh);
    if (threadIdx.x == 0) cg_scalar(kind, s, sc, hist);
}

__global__ void __launch_bounds__(1024) k_cg_beta_flexible(const double* __restrict__ p, int n, Scalars* sc) {
    __shared__ double sh[32];
    const double zq = sum_partials(p, n, sh);
    if (threadIdx.x == 0) {
        const double old = sc->rz_old;
        sc->beta = (old != 0.0 && isfinite(zq)) ? -sc->alpha * zq / old : 0.0;
        if (!isfinite(zq)) sc->aux = 1.0;
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_update_xr(long long n, const Scalars* __restrict__ sc, const T* __restrict__ p,
                                                   const T* __restrict__ q, T* __restrict__ x, T* __restrict__ r,
                                                   double* __restrict__ partials) {
    __shared__ double sh[32];
    const T a = (T)sc->alpha;
    double s = 0.0;
    long long i0 = 0;
    if constexpr (std::is_same<T, float>::value) {
        // 128-bit accesses; r.r (used only for the stopping test) as FP32
        // sums of 4 squares added in FP64: one FP64 add per 4 entries
        // instead of a conversion and an FP64 FMA per entry
        const long long n4 = n / 4;
        const float4* p4 = reinterpret_cast<const float4*>(p);
        const float4* q4 = reinterpret_cast<const float4*>(q);
        float4* x4 = reinterpret_cast<float4*>(x);
        float4* r4 = reinterpret_cast<float4*>(r);
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n4;
             i += (long long)gridDim.x * blockDim.x) {
            const float4 pv = p4[i], qv = q4[i];
            float4 xv = x4[i], rv = r4[i];
            xv.x += a * pv.x;
            xv.y += a * pv.y;
            xv.z += a * pv.z;
            xv.w += a * pv.w;
            rv.x -= a * qv.x;
            rv.y -= a * qv.y;
            rv.z -= a * qv.z;
            rv.w -= a * qv.w;
            x4[i] = xv;
            r4[i] = rv;
            s += (double)(rv.x * rv.x + rv.y * rv.y + rv.z * rv.z + rv.w * rv.w);
        }
        i0 = 4 * n4;
    }
    for (long long i = i0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        x[i] += a * p[i];
        const T ri = r[i] - a * q[i];
        r[i] = ri;
        s += (double)ri * (double)ri;
    }
    s = block_sum(s, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

// r -= alpha q and r.r (as k_update_xr without x; the last block reduces)
template <typename T>
__global__ void __launch_bounds__(256) k_update_r(long long n, const Scalars* sc, const T* __restrict__ q,
                                                  T* __restrict__ r, double* __restrict__ partials,
                                                  const DotTail tail) {
    __shared__ double sh[32];
    const T a = (T)sc->alpha;
    double s = 0.0;
    long long i0 = 0;
    if constexpr (std::is_same<T, float>::value) {
        const long long n4 = n / 4;
        const float4* q4 = reinterpret_cast<const float4*>(q);
        float4* r4 = reinterpret_cast<float4*>(r);
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n4;
             i += (long long)gridDim.x * blockDim.x) {
            const float4 qv = q4[i];
            float4 rv = r4[i];
            rv.x -= a * qv.x;
            rv.y -= a * qv.y;
            rv.z -= a * qv.z;
            rv.w -= a * qv.w;
            r4[i] = rv;
            s += (double)(rv.x * rv.x + rv.y * rv.y + rv.z * rv.z + rv.w * rv.w);
        }
        i0 = 4 * n4;
    }
    for (long long i = i0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const T ri = r[i] - a * q[i];
        r[i] = ri;
        s += (double)ri * (double)ri;
    }
    s = block_sum(s, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
    dot_tail<256>(tail, partials, gridDim.x, threadIdx.x);
}

// x += alpha_j p_j, j = 0 .. count-1 in order: per entry the same fused
// multiply-adds as count successive x += alpha p updates, with x read and
// written once
template <typename T>
struct DirRing {
    const T* p[kDirRing];
};
template <typename T>
__global__ void __launch_bounds__(256) k_flush_x(long long n, DirRing<T> ring, const double* __restrict__ alpha,
                                                 int count, T* __restrict__ x) {
    T a[kDirRing];
#pragma unroll
    for (int j = 0; j < kDirRing; ++j) a[j] = j < count ? (T)alpha[j] : T(0);
    long long i0 = 0;
    if constexpr (std::is_same<T, float>::value) {
        const long long n4 = n / 4;
        float4* x4 = reinterpret_cast<float4*>(x);
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n4;
             i += (long long)gridDim.x * blockDim.x) {
            float4 xv = x4[i];
#pragma unroll
            for (int j = 0; j < kDirRing; ++j) {
                if (j < count) {
                    const float4 pv = reinterpret_cast<const float4*>(ring.p[j])[i];
                    xv.x += a[j] * pv.x;
                    xv.y += a[j] * pv.y;
                    xv.z += a[j] * pv.z;
                    xv.w += a[j] * pv.w;
                }
            }
            x4[i] = xv;
        }
        i0 = 4 * n4;
    }
    for (long long i = i0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        T xi = x[i];
#pragma unroll
        for (int j = 0; j < kDirRing; ++j)
            if (j < count) xi += a[j] * ring.p[j][i];
        x[i] = xi;
    }
}

template <typename T>
__global__ void k_update_p(long long n, const Scalars* __restrict__ sc, const T* __restrict__ z, T* __restrict__ p) {
    const T b = (T)sc->beta;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        p[i] = z[i] + b * p[i];
}

// FP64 <-> FP32 conversion instructions run at the FP64 rate, which bounds a
// pass of 12 bytes per value (12.8M values: 26 us); narrow() and widen() are
// the same values from integer instructions
template <typename S, typename D>
__global__ void __launch_bounds__(256) k_convert(long long n, const S* __restrict__ s, D* __restrict__ d) {
    auto conv = [](S v) -> D {
        if constexpr (std::is_same<S, double>::value && std::is_same<D, float>::value) return narrow(v);
        else if constexpr (std::is_same<S, float>::value && std::is_same<D, double>::value) return widen(v);
        else return (D)v;
    };
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {   // four loads in flight
        S v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = s[i + q * stride];
#pragma unroll
        for (int q = 0; q < 4; ++q) d[i + q * stride] = conv(v[q]);
    }
    for (; i < n; i += stride) d[i] = conv(s[i]);
}

__global__ void k_axpy_f32(long long n, const float* __restrict__ d, double* __restrict__ x) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] += (double)d[i];
}

// ---- dense coarse solve --------------------------------------------------

// The dense coarse factorization is a chain of small steps, and FP64
// arithmetic runs on a narrow pipe (1/64 of the FP32 rate on this GPU): the
// kernels below spread each step's FP64 work over as many SMs as it allows,
// in strips of kStrip rows (or columns) of a 32 x 32 tile per CTA of 128
// threads, instead of one tile per CTA.
constexpr int kStrip = 4;

// One step of the factorization: the diagonal blocks kb of one or two chains
// that do not touch each other, and the block rows below each that are not
// zero: m1 of its own chain, then (up to m) separator rows from s0 on.  W has
// columns c0 .. kb in block row kb.
struct Front {
    int chains, kb[2], c0[2], m1[2], s0[2], m[2];
    __device__ int row(int q, int t) const { return t < m1[q] ? kb[q] + 1 + t : s0[q] + t - m1[q]; }
    __device__ bool sep(int q, int b) const { return b >= s0[q] && b < s0[q] + m[q] - m1[q]; }
};

// Cholesky factor of diagonal block kb and its inverse by one CTA, as
// A = U D U^T (U unit lower) with W = U^-1 carried along, so that a pivot step
// is a reciprocal, one rank-one update and one barrier.  FP64 instructions
// bound it, 64 clocks each on the pipe of one of the four warp schedulers.
//
// The chain of 32 pivots has a scheduler of its own: warp 0 holds the pivot
// column, brings the next one up to date, publishes it (as it is, and divided
// by the pivot: U's column), and nothing else runs beside it.  The warps of
// the other three schedulers hold the rest of A and W in registers, folded:
// lanes c..31 of register c are rows c..31 of column c, lanes 0..c-1 rows
// 32-c..31 of column 32-c, so that the triangles take 17 registers each and
// not 32.  A column is handed to warp 0 through shared memory one step before
// its turn.  Square roots come at the end, all 32 at once: L = U D^(1/2),
// L^-1 = D^(-1/2) W.  A block takes 20.8 us, 1150 clocks a pivot (24.5 with
// the columns spread evenly over 16 warps, one a register, and the warp of the
// next pivot's column doing that first).
//
// One CTA per chain: a step of two chains takes as long as one of one.
// L goes back to the block (zeros above the diagonal), L^-1 to Dk (block kb:
// TB x TB row-major at Dk + kb TB^2).  After a non-positive or non-finite pivot
// the factorization continues with pivot 1; info ends as n minus the smallest
// DOF (order: of each row) whose pivot failed, whichever block finds it first.
__global__ void __launch_bounds__(512) k_potrf_diag(double* __restrict__ A, int n, int npad, Front f, int* info,
                                                    const int* __restrict__ order, double* __restrict__ Dk) {
    static_assert(TB == 32, "a lane per row");
    __shared__ double col[TB][TB + 1], ucol[TB][TB + 1];   // pivot columns and U's (rows below the diagonal)
    __shared__ double next[2][TB], piv[TB], root[TB];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long base = (long long)f.kb[blockIdx.x] * TB;
    const bool worker = w & 3;
    // registers c = cs, cs + 12 of A and W (up to 16; column 0 of A is never
    // updated), this lane's row and column of each
    const int cs = (w & 3) - 1 + 3 * (w >> 2);
    double a[2], x[2];
    int row[2], cl[2];
    double v = 0.0, vn = 0.0, u = 0.0;   // warp 0: the pivot column, the next one, U's column
    if (worker) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int c = cs + 12 * e;
            const bool own = lane >= c;   // (c = 16: both halves are column 16)
            cl[e] = own ? c : TB - c;
            row[e] = own ? lane : TB - c + lane;
            if (c > 16) cl[e] = row[e] = 0;
            a[e] = c <= 16 ? A[(base + row[e]) * npad + base + cl[e]] : 0.0;
            x[e] = row[e] == cl[e] ? 1.0 : 0.0;
        }
    } else if (w == 0) {
        v = A[(base + lane) * npad + base];
        if (lane >= 1) vn = A[(base + lane) * npad + base + 1];
    }
    unsigned failed = 0u;                // warp 0: rows whose pivot is not positive and finite
    auto publish = [&](int j) {   // warp 0: v is column j, up to date
        double d = __shfl_sync(0xffffffffu, v, j);
        const int hi = __double2hiint(d), lo = __double2loint(d);
        if (!((hi > 0 || (hi == 0 && lo != 0)) && hi < 0x7ff00000)) {   // not positive and finite
            failed |= 1u << j;
            d = 1.0;
        }
        // v / d = v y0 (1 + e + e^2) with e = 1 - d y0: v y0 is off the chain
        double y0, e = 0.0;
        if (seed_range(d)) {
            y0 = recip_seed(d);
            e = fma(-d, y0, 1.0);
            e = fma(e, e, e);
        } else {
            y0 = 1.0 / d;
        }
        const double u0 = v * y0;
        u = fma(u0, e, u0);
        if (lane > j) {
            col[j][lane] = v;
            ucol[j][lane] = u;
        }
        if (lane == j) piv[j] = d;
    };
    if (w == 0) publish(0);
#pragma unroll 1
    for (int j = 0; j < TB - 1; ++j) {
        __syncthreads();
        if (w == 0) {
            if (j > 0) vn = lane > j ? next[(j + 1) & 1][lane] : 0.0;
            v = fma(-u, __shfl_sync(0xffffffffu, v, j + 1), vn);
            publish(j + 1);
        } else if (worker) {
            const int cn = min(j + 2, TB - (j + 2));   // register of column j + 2
            auto updateA = [&](int e) {
                if (cl[e] > j) a[e] = fma(-ucol[j][row[e]], col[j][cl[e]], a[e]);
            };
            const int en = cn == cs ? 0 : cn == cs + 12 ? 1 : 2;
            if (en < 2 && j + 2 < TB) {   // the column that warp 0 takes next
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (e == en) {
                        updateA(e);
                        if (cl[e] == j + 2) next[j & 1][row[e]] = a[e];
                    }
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int c = cs + 12 * e;
                if (c > 16) continue;
                if (c > 0 && TB - c > j && !(e == en && j + 2 < TB)) updateA(e);
                if (c <= j) {   // rows below j of the columns up to j
                    const double r = __shfl_sync(0xffffffffu, x[e], lane >= c ? j : j - (TB - c));
                    if (cl[e] <= j && row[e] > j) x[e] = fma(-ucol[j][row[e]], r, x[e]);
                }
            }
        }
    }
    __syncthreads();
    if (w == 0) {
        root[lane] = rsqrt(piv[lane]);
        // (noted after the chain of pivots: an order lookup in it took 1 us a block)
        if ((failed >> lane) & 1u) atomicMax(info, n - (base + lane < n ? order[base + lane] : n - 1));
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int i = w + 16 * e, c = lane;
        A[(base + i) * npad + base + c] = i < c ? 0.0 : (i == c ? piv[c] : col[c][i]) * root[c];
        if (i < c) Dk[base * TB + i * TB + c] = 0.0;
        if (worker && cs + 12 * e <= 16) Dk[base * TB + row[e] * TB + cl[e]] = x[e] * root[row[e]];
    }
}

// L_ib,kb = A_ib,kb L_kk^-T: block row ib = row blockIdx.y of chain
// blockIdx.z, its rows kStrip*blockIdx.x .. +kStrip (threads: 32 columns x
// kStrip rows)
__global__ void __launch_bounds__(128) k_trsm_panel(double* __restrict__ A, int npad, Front f,
                                                    const double* __restrict__ Dk) {
    __shared__ double sI[TB][TB + 1];
    __shared__ double sA[kStrip][TB + 1];
    const int q = blockIdx.z;
    if (blockIdx.y >= f.m[q]) return;
    const int kb = f.kb[q], ib = f.row(q, blockIdx.y), r0 = kStrip * blockIdx.x;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TB + tx;
    const long long rb = (long long)ib * TB + r0, cb = (long long)kb * TB;
    for (int e = tid; e < TB * TB; e += 128) sI[e / TB][e % TB] = Dk[cb * TB + e];
    sA[ty][tx] = A[(rb + ty) * npad + cb + tx];
    __syncthreads();
    double s = 0.0;
#pragma unroll 8
    for (int t = 0; t < TB; ++t) s += sA[ty][t] * sI[tx][t];
    A[(rb + ty) * npad + cb + tx] = s;
}

// A_ib,jb -= L_ib,kb L_jb,kb^T for the pairs jb <= ib of a chain's rows (pair
// blockIdx.y), rows kStrip*blockIdx.x .. +kStrip of the tile.  blockIdx.z: the
// chain; with two chains, whose separator rows overlap, their pairs of
// separator rows are left to blockIdx.z = 2, which subtracts both (pairs of
// the ns rows from sep0 on).
__global__ void __launch_bounds__(128) k_syrk(double* __restrict__ A, int npad, Front f, int sep0, int ns) {
    __shared__ double sI[kStrip][TB + 1];
    __shared__ double sJ[TB][TB + 1];
    const int t = blockIdx.y, z = blockIdx.z;
    int ii = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
    while ((ii + 1) * (ii + 2) / 2 <= t) ++ii;
    while (ii * (ii + 1) / 2 > t) --ii;
    const int jj = t - ii * (ii + 1) / 2;
    if (ii >= (z < 2 ? f.m[z] : ns) || (z < 2 && f.chains == 2 && jj >= f.m1[z])) return;
    const int ib = z < 2 ? f.row(z, ii) : sep0 + ii, jb = z < 2 ? f.row(z, jj) : sep0 + jj, r0 = kStrip * blockIdx.x;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TB + tx;
    const long long rb = (long long)ib * TB + r0, jr = (long long)jb * TB;
    double v = A[(rb + ty) * npad + jr + tx];
    for (int q = z < 2 ? z : 0; q < (z < 2 ? z + 1 : 2); ++q) {
        if (z == 2 && !(f.sep(q, ib) && f.sep(q, jb))) continue;   // (the same for the whole block)
        const long long cb = (long long)f.kb[q] * TB;
        __syncthreads();
        sI[ty][tx] = A[(rb + ty) * npad + cb + tx];
        for (int e = tid; e < TB * TB; e += 128) sJ[e / TB][e % TB] = A[(jr + e / TB) * npad + cb + e % TB];
        __syncthreads();
        double s = 0.0;
#pragma unroll 8
        for (int c = 0; c < TB; ++c) s += sI[ty][c] * sJ[tx][c];
        v -= s;
    }
    A[(rb + ty) * npad + jr + tx] = v;
}

__global__ void k_identity(double* __restrict__ W, int npad) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long n2 = (long long)npad * npad;
    if (i >= n2) return;
    W[i] = ((i / npad) == (i % npad)) ? 1.0 : 0.0;
}

// W_kb,jb = L_kk^-1 B_kb,jb for jb = c0 + blockIdx.y <= kb of chain
// blockIdx.z, its columns kStrip*blockIdx.x .. +kStrip (threads: kStrip columns
// x 32 rows)
__global__ void __launch_bounds__(128) k_trsm_rows(double* __restrict__ W, int npad, Front f,
                                                   const double* __restrict__ Dk) {
    __shared__ double sI[TB][TB + 1];
    __shared__ double sB[TB][kStrip + 1];
    const int kb = f.kb[blockIdx.z], jb = f.c0[blockIdx.z] + blockIdx.y, c0 = kStrip * blockIdx.x;
    if (jb > kb) return;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kStrip + tx;
    const long long rb = (long long)kb * TB, cb = (long long)jb * TB + c0;
    for (int e = tid; e < TB * TB; e += 128) sI[e / TB][e % TB] = Dk[rb * TB + e];
    sB[ty][tx] = W[(rb + ty) * npad + cb + tx];
    __syncthreads();
    double s = 0.0;
#pragma unroll 8
    for (int t = 0; t < TB; ++t) s += sI[ty][t] * sB[t][tx];
    W[(rb + ty) * npad + cb + tx] = s;
}

// B_ib,jb -= L_ib,kb W_kb,jb for jb = c0 + blockIdx.y <= kb and the rows ib of
// a chain (blockIdx.z: mm rows of the first chain, then the second's; their
// columns differ), rows kStrip*blockIdx.x .. +kStrip of the tile
__global__ void __launch_bounds__(128) k_gemm_update(const double* __restrict__ L, double* __restrict__ W, int npad,
                                                     Front f, int mm) {
    __shared__ double sL[kStrip][TB + 1];
    __shared__ double sW[TB][TB + 1];
    const int q = blockIdx.z >= mm, i = blockIdx.z - q * mm, kb = f.kb[q], jb = f.c0[q] + blockIdx.y;
    if (i >= f.m[q] || jb > kb) return;
    const int ib = f.row(q, i), r0 = kStrip * blockIdx.x;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TB + tx;
    const long long kbase = (long long)kb * TB, rb = (long long)ib * TB + r0, cb = (long long)jb * TB;
    sL[ty][tx] = L[(rb + ty) * npad + kbase + tx];
    for (int e = tid; e < TB * TB; e += 128) sW[e / TB][e % TB] = W[(kbase + e / TB) * npad + cb + e % TB];
    __syncthreads();
    double s = 0.0;
#pragma unroll 8
    for (int c = 0; c < TB; ++c) s += sL[ty][c] * sW[c][tx];
    W[(rb + ty) * npad + cb + tx] -= s;
}

__global__ void k_transpose(const double* __restrict__ W, double* __restrict__ WT, int npad) {
    __shared__ double s[TB][TB + 1];
    const int bx = blockIdx.x, by = blockIdx.y, tx = threadIdx.x, ty = threadIdx.y;
    s[ty][tx] = W[((long long)by * TB + ty) * npad + (long long)bx * TB + tx];
    __syncthreads();
    WT[((long long)bx * TB + ty) * npad + (long long)by * TB + tx] = s[tx][ty];
}

// y_i = sum_{j<=i} W_ij r_order(j) (lower) or u_order(i) = sum_{j>=i} W^T_ij y_j
// (upper); a block of 128 threads per row.  What bounds it is the latency of a
// row's loads: with a warp per row, a row of 1911 was a chain of up to 8
// batches of loads (and of the order behind them: 22 us), now of two.
// FP64 matrices: FP64 sums.  FP32 matrices: every product and sum with its
// exact rounding error carried in a second FP32 word (TwoProduct by fused
// multiply-add, Knuth's TwoSum): 12 FP32 instructions per entry where two
// conversions and an FP64 multiply-add take 48 issue cycles of the SM.
// Against exact sums of the same entries (rows of 1 to 1911, with and without
// cancellation) the two words are off by at most 2^-46.4 of the sum of the
// terms' sizes, FP64 sums by 2^-51.2, and both round to the same FP32 number;
// the entries themselves are rounded to 2^-24.  The second word needs the
// exponents between: with every term below 2^-80 (its errors would underflow)
// or one at 2^100 or more (a sum could overflow before it cancels) the row is
// summed in FP64, unless all its terms are exactly 0 (fixed DOFs).
__device__ __forceinline__ void two_sum_into(float& s, float& c, float p) {
    const float t = __fadd_rn(s, p), b = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(p, b)));
    s = t;
}
constexpr int kGemv = 128;
template <typename T, bool LOWER>
__global__ void __launch_bounds__(kGemv) k_trigemv(int n, int npad, const T* __restrict__ M, const T* __restrict__ v,
                                                   T* __restrict__ y, const int* __restrict__ order) {
    __shared__ T red[3][kGemv / 32];
    const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int j1 = LOWER ? row + 1 : n;
    const T* mr = M + (long long)row * npad;
    T s = T(0);
    [[maybe_unused]] float c = 0.0f, largest = 0.0f, factor = 0.0f;   // factor: > 0 once a term is not 0
    auto add = [&](T a, T b) {
        if constexpr (std::is_same<T, float>::value) {
            const float p = __fmul_rn(a, b);
            largest = fmaxf(largest, fabsf(p));
            factor = fmaxf(factor, fminf(fabsf(a), fabsf(b)));
            c = __fadd_rn(c, __fmaf_rn(a, b, -p));
            two_sum_into(s, c, p);
        } else {
            s = fma(a, b, s);
        }
    };
    constexpr int U = 8;   // loads of each array in flight
    for (int j = (LOWER ? 0 : row) + tid; j < j1; j += U * kGemv) {
        T a[U], b[U];
        int at[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int jq = j + q * kGemv;
            a[q] = jq < j1 ? mr[jq] : T(0);
            at[q] = jq < j1 ? (LOWER ? order[jq] : jq) : -1;
        }
#pragma unroll
        for (int q = 0; q < U; ++q) b[q] = at[q] >= 0 ? v[at[q]] : T(0);
#pragma unroll
        for (int q = 0; q < U; ++q)
            if (at[q] >= 0) add(a[q], b[q]);
    }
    auto merge = [&](T so, [[maybe_unused]] float co) {
        if constexpr (std::is_same<T, float>::value) {
            c += co;
            two_sum_into(s, c, so);
        } else {
            s += so;
        }
    };
    for (int o = 16; o > 0; o >>= 1) {
        const T so = __shfl_xor_sync(0xffffffffu, s, o);
        float co = 0.0f;
        if constexpr (std::is_same<T, float>::value) co = __shfl_xor_sync(0xffffffffu, c, o);
        merge(so, co);
    }
    if constexpr (std::is_same<T, float>::value) {
        largest = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(largest)));
        if (largest == 0.0f && !__any_sync(0xffffffffu, factor > 0.0f)) largest = -1.0f;
    }
    if (lane == 0) {
        red[0][w] = s;
        red[1][w] = (T)c;
        red[2][w] = (T)largest;
    }
    __syncthreads();
    if constexpr (std::is_same<T, float>::value) {
#pragma unroll
        for (int q = 0; q < kGemv / 32; ++q) largest = fmaxf(largest, red[2][q]);
        if (largest >= 0.0f && !(largest >= 0x1p-80f && largest < 0x1p100f)) {   // (the same for the whole block)
            __shared__ double sums[kGemv / 32];
            double d = 0.0;
            for (int j = (LOWER ? 0 : row) + tid; j < j1; j += kGemv) d = fma((double)mr[j], (double)v[LOWER ? order[j] : j], d);
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if (lane == 0) sums[w] = d;
            __syncthreads();
            if (tid == 0) y[LOWER ? row : order[row]] = (float)((sums[0] + sums[1]) + (sums[2] + sums[3]));
            return;
        }
    }
    if (tid == 0) {
#pragma unroll
        for (int q = 1; q < kGemv / 32; ++q) merge(red[0][q], (float)red[1][q]);
        y[LOWER ? row : order[row]] = s + (T)c;
    }
}

}  // namespace

template <typename A, typename B>
void dot_partials(const Ctx& c, long long n, const A* a, const B* b, double* partials) {
    k_dot<A, B><<<kRedBlocks, 256, 0, c.s>>>(n, a, b, partials);
    TOPO_LAUNCH_CHECK(c);
}
template void dot_partials<double, double>(const Ctx&, long long, const double*, const double*, double*);
template void dot_partials<float, float>(const Ctx&, long long, const float*, const float*, double*);
template void dot_partials<double, float>(const Ctx&, long long, const double*, const float*, double*);

void reduce_to(const Ctx& c, const double* partials, int n, double* dst) {
    k_reduce_to<<<1, 1024, 0, c.s>>>(partials, n, dst);
    TOPO_LAUNCH_CHECK(c);
}
void cg_alpha(const Ctx& c, const double* partials, int n, Scalars* sc, double* hist) {
    k_cg_scalar<<<1, 1024, 0, c.s>>>(TAIL_ALPHA, partials, n, sc, hist);
    TOPO_LAUNCH_CHECK(c);
}
void cg_beta(const Ctx& c, const double* partials, int n, Scalars* sc) {
    k_cg_scalar<<<1, 1024, 0, c.s>>>(TAIL_BETA, partials, n, sc, nullptr);
    TOPO_LAUNCH_CHECK(c);
}
void cg_beta_flexible(const Ctx& c, const double* partials, int n, Scalars* sc) {
    k_cg_beta_flexible<<<1, 1024, 0, c.s>>>(partials, n, sc);
    TOPO_LAUNCH_CHECK(c);
}

template <typename T>
void cg_update_xr(const Ctx& c, long long n, const Scalars* sc, const T* p, const T* q, T* x, T* r,
                  double* partials) {
    k_update_xr<T><<<kRedBlocks, 256, 0, c.s>>>(n, sc, p, q, x, r, partials);
    TOPO_LAUNCH_CHECK(c);
}
template void cg_update_xr<double>(const Ctx&, long long, const Scalars*, const double*, const double*, double*,
                                   double*, double*);
template void cg_update_xr<float>(const Ctx&, long long, const Scalars*, const float*, const float*, float*, float*,
                                  double*);

template <typename T>
void cg_update_p(const Ctx& c, long long n, const Scalars* sc, const T* z, T* p) {
    k_update_p<T><<<grid_for(n, 256) > 8192 ? 8192 : grid_for(n, 256), 256, 0, c.s>>>(n, sc, z, p);
    TOPO_LAUNCH_CHECK(c);
}
template void cg_update_p<double>(const Ctx&, long long, const Scalars*, const double*, double*);
template void cg_update_p<float>(const Ctx&, long long, const Scalars*, const float*, float*);

template <typename T>
void cg_update_r(const Ctx& c, long long n, Scalars* sc, const T* q, T* r, double* partials, unsigned* ticket) {
    const unsigned g = grid_for(n, 1024);   // four entries per thread until the GPU is full
    k_update_r<T><<<g > kUpdateBlocks ? kUpdateBlocks : g, 256, 0, c.s>>>(n, sc, q, r, partials,
                                                                       DotTail{TAIL_RR, sc, nullptr, ticket});
    TOPO_LAUNCH_CHECK(c);
}
template void cg_update_r<double>(const Ctx&, long long, Scalars*, const double*, double*, double*, unsigned*);
template void cg_update_r<float>(const Ctx&, long long, Scalars*, const float*, float*, double*, unsigned*);

template <typename T>
void cg_flush_x(const Ctx& c, long long n, T* const* ring, const double* alpha, int count, T* x) {
    DirRing<T> dr;
    for (int j = 0; j < kDirRing; ++j) dr.p[j] = ring[j];
    k_flush_x<T><<<grid_for(n, 256) > 8192 ? 8192 : grid_for(n, 256), 256, 0, c.s>>>(n, dr, alpha, count, x);
    TOPO_LAUNCH_CHECK(c);
}
template void cg_flush_x<double>(const Ctx&, long long, double* const*, const double*, int, double*);
template void cg_flush_x<float>(const Ctx&, long long, float* const*, const double*, int, float*);

template <typename S, typename D>
void convert(const Ctx& c, long long n, const S* src, D* dst) {
    const unsigned g = grid_for(n, 1024);
    k_convert<S, D><<<g > kUpdateBlocks ? kUpdateBlocks : g, 256, 0, c.s>>>(n, src, dst);
    TOPO_LAUNCH_CHECK(c);
}
template void convert<double, float>(const Ctx&, long long, const double*, float*);
template void convert<float, double>(const Ctx&, long long, const float*, double*);
template void convert<bf16, float>(const Ctx&, long long, const bf16*, float*);

void axpy_f32_into_f64(const Ctx& c, long long n, const float* d, double* x) {
    k_axpy_f32<<<grid_for(n, 256) > 8192 ? 8192 : grid_for(n, 256), 256, 0, c.s>>>(n, d, x);
    TOPO_LAUNCH_CHECK(c);
}

template <typename T>
void zero(const Ctx& c, long long n, T* v) {
    cudaMemsetAsync(v, 0, sizeof(T) * (size_t)n, c.s);
}
template void zero<double>(const Ctx&, long long, double*);
template void zero<float>(const Ctx&, long long, float*);

// Blocks of a banded matrix (A_ij = 0 for |i - j| > band) that can be nonzero
// below the diagonal block of block column kb: block rows kb+1 .. kb+bb.
inline int band_blocks(int band) { return (band + TB - 1) / TB; }

void chol_inverse(const Ctx& c, cudaStream_t side, cudaEvent_t ready, double* A, double* W, int n, int npad, int band,
                  int* info, const int* order, double* Dk) {
    // The Cholesky factor of a banded matrix keeps its band, so the panel and
    // the trailing update of a step touch only the bb block rows below it; the
    // blocks left out are zero in A and L alike.  Two chains of `a` blocks run
    // to the separator in the same launches (60 steps of 13 x 7 x 7 nodes
    // become 33: the factorization and inverse of a density update take 1.0 ms
    // less), then the separator, whose rows keep their order and so their
    // band.  W = L^-1 is lower triangular with a zero block between the chains;
    // L_ib,kb vanishes outside a step's rows, so the update after block row kb
    // reaches only those.
    const int nb = npad / TB, bb = band_blocks(band), a = coarse_chain(n, band), sep0 = 2 * a, ns = nb - sep0;
    const int nsep = n - 2 * TB * a;   // rows of the separator
    const long long n2 = (long long)npad * npad;
    const Ctx cs{side, c.launches};
    auto follow = [&](cudaStream_t from, cudaStream_t to) {   // to waits for what from has been given so far
        if (side == c.s) return;
        cudaEventRecord(ready, from);
        cudaStreamWaitEvent(to, ready, 0);
    };
    cudaMemsetAsync(info, 0, sizeof(int), c.s);
    follow(c.s, side);
    k_identity<<<grid_for(n2, 256), 256, 0, cs.s>>>(W, npad);
    TOPO_LAUNCH_CHECK(cs);
    for (int step = 0; step < a + ns; ++step) {
        Front f{};
        f.chains = step < a ? 2 : 1;
        if (f.chains == 2) {
            for (int q = 0; q < 2; ++q) {
                f.kb[q] = q * a + step;
                f.c0[q] = q * a;
                f.m1[q] = std::min(a - 1 - step, bb);
            }
            // separator rows in reach: blocks from the front for the first
            // chain, rows from the back for the second
            const int front = std::max(0, std::min(ns, step + bb - (a - 1)));
            const int back = std::max(0, std::min(nsep, TB * (step + 1 - a) + band));
            f.s0[0] = sep0;
            f.m[0] = f.m1[0] + front;
            f.s0[1] = sep0 + (nsep - back) / TB;
            f.m[1] = f.m1[1] + (back > 0 ? ns - (nsep - back) / TB : 0);
        } else {
            f.kb[0] = sep0 + step - a;
            f.m1[0] = f.m[0] = std::min(nb - f.kb[0] - 1, bb);
        }
        const int m = std::max(f.m[0], f.m[1]), cols = f.kb[0] - f.c0[0] + 1, nz = f.chains;
        const bool sep = f.m[0] > f.m1[0] || f.m[1] > f.m1[1];
        k_potrf_diag<<<nz, 512, 0, c.s>>>(A, n, npad, f, info, order, Dk);
        TOPO_LAUNCH_CHECK(c);
        if (m > 0) {
            k_trsm_panel<<<dim3(TB / kStrip, m, nz), dim3(TB, kStrip), 0, c.s>>>(A, npad, f, Dk);
            TOPO_LAUNCH_CHECK(c);
        }
        follow(c.s, side);   // block column kb of L and its Dk are final
        k_trsm_rows<<<dim3(TB / kStrip, cols, nz), dim3(kStrip, TB), 0, cs.s>>>(W, npad, f, Dk);
        TOPO_LAUNCH_CHECK(cs);
        if (m > 0) {
            k_gemm_update<<<dim3(TB / kStrip, cols, m * nz), dim3(TB, kStrip), 0, cs.s>>>(A, W, npad, f, m);
            TOPO_LAUNCH_CHECK(cs);
            const int pairs = std::max(m * (m + 1) / 2, sep ? ns * (ns + 1) / 2 : 0);
            k_syrk<<<dim3(TB / kStrip, pairs, sep ? 3 : nz), dim3(TB, kStrip), 0, c.s>>>(A, npad, f, sep0, ns);
            TOPO_LAUNCH_CHECK(c);
        }
    }
    follow(side, c.s);
}

void transpose_dense(const Ctx& c, const double* W, double* WT, int npad) {
    const int nb = npad / TB;
    k_transpose<<<dim3(nb, nb), dim3(TB, TB), 0, c.s>>>(W, WT, npad);
    TOPO_LAUNCH_CHECK(c);
}

template <typename T>
void coarse_apply(const Ctx& c, const Coarse& cs, const T* W, const T* WT, const T* rhs, T* y, T* out) {
    const int n = cs.n, npad = cs.npad;
    k_trigemv<T, true><<<n, kGemv, 0, c.s>>>(n, npad, W, rhs, y, cs.order);
    TOPO_LAUNCH_CHECK(c);
    k_trigemv<T, false><<<n, kGemv, 0, c.s>>>(n, npad, WT, y, out, cs.order);
    TOPO_LAUNCH_CHECK(c);
}
template void coarse_apply<double>(const Ctx&, const Coarse&, const double*, const double*, const double*, double*,
                                   double*);
template void coarse_apply<float>(const Ctx&, const Coarse&, const float*, const float*, const float*, float*, float*);

}  // namespace topo
