// Density filter (weights of Eqs. Neighbourhood / NB_dist, normalised by the
// in-domain weight sum S_e), its transpose, and the paper's sensitivity filter.
//
// What bounds it: FP64 instructions run at 2 lanes per clock and SM on this
// part (1/64 of the FP32 rate), so a neighbour-by-neighbour sum costs one
// FP64 multiply-add per neighbour and element (93 at r = 3, 905 at r = 6)
// while memory and the other pipes idle.  The weight depends on
// dx^2 + dy^2 + dz^2 only, so the values are summed by symmetry first and
// multiplied once per class:
//   Y_b(i, j)  = v(i, j - b) + v(i, j + b)                  (shared by the row)
//   G_ab(i, j) = sum of the 4 or 8 values at (+-a, +-b), (+-b, +-a), a >= b
//   F_c(i, j)  = sum over the classes of w(a, b, c) G_ab
//   out(k)     = F_0(k) + sum over c of F_c(k - c) + F_c(k + c)
// marching along z with 2R + 1 running sums per column: 30 FP64
// instructions per element instead of 93 at r = 3, 146 instead of 905 at
// r = 6.  S_e depends only on the distances to the six faces, so it is a
// table of (2R + 1)^3 entries, with reciprocals for the division.
// Thin, odd and small grids, whose tiles and chunks are mostly halo, are summed
// neighbour by neighbour instead (k_filter_near, chosen by filter_plan).
//
// Measured, forward + transpose of 256x128x128 elements: r = 3, 2149 -> 725
// us; the first call with a new radius 3690 -> 775 us.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace topo {

namespace {

// class of index i along an axis of n elements: everything that the cut
// neighbourhood depends on
__host__ __device__ inline int face_class(int i, int n, int R) {
    if (n <= 2 * R) return i;
    return i < R ? i : (i >= n - R ? 2 * R - (n - 1 - i) : R);
}
__host__ __device__ constexpr int pair_class(int a, int b) { return a >= b ? a * (a + 1) / 2 + b : b * (b + 1) / 2 + a; }

// S of every class triple and 1 / S, for k_filter and for k_filter_near.  S is
// formed by the very operations of each kernel on in-domain values of 1 (the
// counts G are exact), so that H of values in [0, 1] stays in [0, 1] and H 1 = 1
// exactly: every operation is monotone in the values.
__global__ void k_filter_weights(const __grid_constant__ FilterW W, int R, int nx, int ny, int nz, bool march, bool near,
                                 double* __restrict__ stab) {
    const int nc = 2 * R + 1, t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nc * nc * nc) return;
    const int cl[3] = {t % nc, (t / nc) % nc, t / (nc * nc)}, n[3] = {nx, ny, nz};
    int lo[3], hi[3];
    for (int q = 0; q < 3; ++q) {
        if (n[q] <= 2 * R && cl[q] >= n[q]) return;   // no such element
        lo[q] = -min(cl[q], R);
        hi[q] = min(n[q] <= 2 * R ? n[q] - 1 - cl[q] : 2 * R - cl[q], R);
    }
    if (march) {
        // in-domain values among the distinct (+-a, +-b)
        auto count = [&](int a, int b) {
            const int ca = a == 0 ? 1 : (-a >= lo[0]) + (a <= hi[0]), cb = b == 0 ? 1 : (-b >= lo[1]) + (b <= hi[1]);
            return ca * cb;
        };
        double s = 0.0;
        for (int dz = lo[2]; dz <= hi[2]; ++dz) {
            const int c = abs(dz);
            double F = 0.0;
            for (int a = 0; a <= R; ++a)
                for (int b = 0; b <= a; ++b) {
                    const int p = pair_class(a, b);
                    if ((W.bits[p] >> c) & 1u) F = fma(W.w[c][p], (double)(count(a, b) + (a != b ? count(b, a) : 0)), F);
                }
            s += F;
        }
        stab[t] = s;
        stab[kFilterTab + t] = 1.0 / s;
    }
    if (near) {
        double s = 0.0;
        for (int dz = lo[2]; dz <= hi[2]; ++dz)
            for (int dy = lo[1]; dy <= hi[1]; ++dy) {
                const int c = abs(dz), b = abs(dy), x = W.reach[c][b], d0 = max(lo[0], -x), d1 = min(hi[0], x);
#pragma unroll
                for (int dx = -5; dx <= 5; ++dx)
                    if (dx >= d0 && dx <= d1) s += W.w[c][pair_class(abs(dx), b)];
            }
        stab[2 * kFilterTab + t] = s;
        stab[3 * kFilterTab + t] = 1.0 / s;
    }
}

// a / s with rs = fl(1 / s): product, exact remainder, correction (Markstein) --
// 3 FP64 instructions instead of about 10.  Zeros, values near the ends of
// the exponent range, infinities and NaN take the plain division; the tests
// are on integer words.
__device__ __forceinline__ double div_by(double a, double s, double rs) {
    const int hi = __double2hiint(a);
    if (((hi & 0x7fffffff) | __double2loint(a)) == 0) return a;
    if ((unsigned)(((hi >> 20) & 0x7ff) - 128) >= 1792u) return a / s;
    const double q = a * rs;
    return fma(fma(-q, s, a), rs, q);
}

// MODE 0: out = H in; MODE 1: out = H^T in (in null: H^T 1); MODE 2: the
// sensitivity filter H(rho in) / max(gamma, rho).
// One CTA: TX x (128 / TX) element columns and a chunk of cz planes.  Per
// plane: the tile with its halo goes to shared memory (loaded one plane
// ahead into registers), Y, then G and F per thread.  128 threads, one warp
// per scheduler; several CTAs per SM hide the two barriers per plane.
// Weights that are zero inside the class list (r not an integer) are skipped
// by the class's bit mask, not multiplied, so that an infinity or NaN
// spreads to exactly the elements whose neighbourhood holds it.
template <int R, int TX, int MODE>
__global__ void __launch_bounds__(128) k_filter(const __grid_constant__ FilterW W, const int nx, const int ny,
                                                const int nz, const int cz, const double* __restrict__ in,
                                                const double* __restrict__ rho, const double gamma,
                                                const double* __restrict__ stab, double* __restrict__ out) {
    constexpr int TY = 128 / TX, PW = TX + 2 * R, PH = TY + 2 * R, NT = PW * PH, NL = (NT + 127) / 128;
    constexpr int nc = 2 * R + 1;
    __shared__ double v[2][PH][PW];
    __shared__ double Y[R > 0 ? R : 1][TY][PW];
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    // one-dimensional grid (x tiles fastest): long thin grids exceed the y and z limits
    const int gx = (nx + TX - 1) / TX, gy = (ny + TY - 1) / TY;
    const int bxy = blockIdx.x % (gx * gy);
    const int i0 = bxy % gx * TX, j0 = bxy / gx * TY;
    const int k0 = blockIdx.x / (gx * gy) * cz, k1 = min(k0 + cz, nz);
    const int nxy = nx * ny;
    int off[NL];
    [[maybe_unused]] int cxy[NL];
    double raw[NL];
    [[maybe_unused]] double raw2[NL];
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        const int pos = tid + 128 * l, gi = i0 - R + pos % PW, gj = j0 - R + pos / PW;
        const bool ok = pos < NT && gi >= 0 && gi < nx && gj >= 0 && gj < ny;
        off[l] = ok ? gi + nx * gj : -1;
        if constexpr (MODE == 1) cxy[l] = ok ? face_class(gj, ny, R) * nc + face_class(gi, nx, R) : 0;
        raw[l] = 0.0;
    }
    // H^T of a block whose values all have the same weight sum: one division
    // per output instead of one per staged value (2.25 of them at R = 2)
    bool uniform = false;
    if constexpr (MODE == 1)
        uniform = in && i0 >= 2 * R && i0 + TX + 2 * R <= nx && j0 >= 2 * R && j0 + TY + 2 * R <= ny && k0 >= 2 * R &&
                  k1 + 2 * R <= nz;
    auto fetch = [&](int k) {
#pragma unroll
        for (int l = 0; l < NL; ++l)
            if (off[l] >= 0) {
                if (MODE != 1 || in) raw[l] = in[off[l] + nxy * k];
                if constexpr (MODE == 2) raw2[l] = rho[off[l] + nxy * k];
            }
    };
    const int i = i0 + tx, j = j0 + ty;
    const bool act = i < nx && j < ny;
    const int ccol = act ? face_class(j, ny, R) * nc + face_class(i, nx, R) : 0;
    double acc[2 * R + 1];
#pragma unroll
    for (int d = 0; d <= 2 * R; ++d) acc[d] = 0.0;
    const int kb = max(k0 - R, 0), ke = min(k1 - 1 + R, nz - 1);
    fetch(kb);
    for (int k = kb; k <= k1 - 1 + R; ++k) {
        if (k <= ke) {
            double(*vb)[PW] = v[k & 1];
#pragma unroll
            for (int l = 0; l < NL; ++l) {
                const int pos = tid + 128 * l;
                if (pos < NT) {
                    double t = raw[l];
                    if constexpr (MODE == 1) {
                        const int ct = face_class(k, nz, R) * nc * nc + cxy[l];
                        if (off[l] >= 0 && !uniform) t = in ? div_by(t, stab[ct], stab[kFilterTab + ct]) : stab[kFilterTab + ct];
                    }
                    if constexpr (MODE == 2)
                        if (off[l] >= 0) t *= raw2[l];
                    vb[pos / PW][pos % PW] = t;
                }
            }
            if (k < ke) fetch(k + 1);
            __syncthreads();
            if constexpr (R > 0) {
                for (int t = tid; t < TY * PW; t += 128) {
                    const int row = t / PW, col = t % PW;
#pragma unroll
                    for (int b = 1; b <= R; ++b) Y[b - 1][row][col] = vb[row + R - b][col] + vb[row + R + b][col];
                }
                __syncthreads();
            }
            if (act) {
                // planes k - c and k + c that this chunk outputs
                unsigned need = 0;
#pragma unroll
                for (int c = 0; c <= R; ++c)
                    if ((k - c >= k0 && k - c < k1) || (k + c >= k0 && k + c < k1)) need |= 1u << c;
                double F[R + 1];
#pragma unroll
                for (int c = 0; c <= R; ++c) F[c] = 0.0;
                const double* vr = &vb[ty + R][tx + R];
#pragma unroll
                for (int a = 0; a <= R; ++a)
#pragma unroll
                    for (int b = 0; b <= a; ++b) {
                        const int p = pair_class(a, b);
                        const unsigned m = W.bits[p] & need;
                        if (m == 0) continue;
                        double G;
                        if (a == 0) {
                            G = vr[0];
                        } else if (b == 0) {
                            G = (vr[-a] + vr[a]) + Y[a - 1][ty][tx + R];
                        } else if (a == b) {
                            G = Y[a - 1][ty][tx + R - a] + Y[a - 1][ty][tx + R + a];
                        } else {
                            const double* ya = Y[a - 1][ty] + tx + R;
                            const double* yb = Y[b - 1][ty] + tx + R;
                            G = (ya[-b] + ya[b]) + (yb[-a] + yb[a]);
                        }
#pragma unroll
                        for (int c = 0; c <= R; ++c)
                            if ((m >> c) & 1u) F[c] = fma(W.w[c][p], G, F[c]);
                    }
#pragma unroll
                for (int d = 0; d <= 2 * R; ++d) {
                    const int ko = k - R + d;
                    if (ko >= k0 && ko < k1) acc[d] += F[d < R ? R - d : d - R];
                }
            }
        }
        const int ko = k - R;
        if (act && ko >= k0) {
            const int e = i + nx * j + nxy * ko;
            double o = acc[0];
            if constexpr (MODE != 1) {
                const int ct = face_class(ko, nz, R) * nc * nc + ccol;
                o = div_by(o, stab[ct], stab[kFilterTab + ct]);
                if constexpr (MODE == 2) o = o / fmax(gamma, rho[e]);
            } else if (uniform) {
                constexpr int ct = (nc * nc + nc + 1) * R;
                o = div_by(o, stab[ct], stab[kFilterTab + ct]);
            }
            out[e] = o;
        }
#pragma unroll
        for (int d = 0; d < 2 * R; ++d) acc[d] = acc[d + 1];
        acc[2 * R] = 0.0;
    }
}

// The same sums neighbour by neighbour, a thread per element: one FP64
// multiply-add per neighbour, whatever the grid's shape.  It is the better side
// where the march has little to share: thin or odd grids, whose tiles are
// mostly idle lanes, and small ones, where a chunk's halo planes outnumber its
// own (filter_plan).  Values of a row are loaded together; then 2 X + 1
// multiply-adds, each in the lanes that have the neighbour: the FP64 pipe takes
// its time per active lane, and for instructions that are only predicated off.
// MODE as k_filter.  FORM: the summed values are formed where they are read (H^T:
// in / S, in null: 1 / S; sensitivity filter: rho in), else `in` holds them
// (k_filter_values).
// Measured, march -> this: 1x512x512 elements at r = 1.5, H 152 -> 10 us and H^T
// 171 -> 13; 2x2x100000 at r = 3, 515 -> 39 and 523 -> 43; 75x26x33 at r = 2.5,
// 20.5 -> 16.4 and 24.7 -> 20.2; 259x105x159 at r = 1, 47 -> 35 and 47 -> 37.
template <int R, int MODE, bool FORM>
__global__ void __launch_bounds__(256) k_filter_near(const __grid_constant__ FilterW W, const int nx, const int ny,
                                                     const int nz, const double* __restrict__ in,
                                                     const double* __restrict__ rho, const double gamma,
                                                     const double* __restrict__ stab, double* __restrict__ out) {
    constexpr int nc = 2 * R + 1;
    const int e = blockIdx.x * 256 + threadIdx.x, ne = nx * ny * nz;
    const bool act = e < ne;
    const int i = e % nx, j = e / nx % ny, k = e / (nx * ny);
    double acc = 0.0;
    const int Rz = min(R, nz - 1), Ry = min(R, ny - 1);
#pragma unroll 1
    for (int dz = -Rz; dz <= Rz; ++dz) {
        const int kk = k + dz, c = abs(dz);
        const bool okz = act && (unsigned)kk < (unsigned)nz;
#pragma unroll 1
        for (int dy = -Ry; dy <= Ry; ++dy) {
            const int jj = j + dy, b = abs(dy), x = min((int)W.reach[c][b], nx - 1);
            const bool okr = okz && (unsigned)jj < (unsigned)ny;
            if (x < 0 || !__any_sync(0xffffffffu, okr)) continue;
            const int row = nx * (jj + ny * kk) + i;
            [[maybe_unused]] int ct = 0;
            if constexpr (FORM && MODE == 1)
                if (okr) ct = (face_class(kk, nz, R) * nc + face_class(jj, ny, R)) * nc;
            auto sum_row = [&](auto reach) {
                constexpr int X = decltype(reach)::value;
                double v[2 * X + 1];
#pragma unroll
                for (int dx = -X; dx <= X; ++dx) {
                    const int ii = i + dx;
                    double t = 0.0;   // (set in every lane: the loads stay together, ahead of the sums)
                    if (okr && (unsigned)ii < (unsigned)nx) {
                        if constexpr (FORM && MODE == 1) {
                            const int f = ct + face_class(ii, nx, R);
                            t = in ? div_by(in[row + dx], stab[f], stab[kFilterTab + f]) : stab[kFilterTab + f];
                        } else {
                            t = in[row + dx];
                            if constexpr (FORM) t *= rho[row + dx];
                        }
                    }
                    v[dx + X] = t;
                }
#pragma unroll
                for (int dx = -X; dx <= X; ++dx)
                    if (okr && (unsigned)(i + dx) < (unsigned)nx)
                        acc = fma(W.w[c][pair_class(abs(dx), b)], v[dx + X], acc);
            };
            if (x == 0) sum_row(std::integral_constant<int, 0>{});
            else if (R == 1 || x == 1) sum_row(std::integral_constant<int, R < 1 ? R : 1>{});
            else if (R == 2 || x == 2) sum_row(std::integral_constant<int, R < 2 ? R : 2>{});
            else if (R == 3 || x == 3) sum_row(std::integral_constant<int, R < 3 ? R : 3>{});
            else if (R == 4 || x == 4) sum_row(std::integral_constant<int, R < 4 ? R : 4>{});
            else sum_row(std::integral_constant<int, R < 5 ? R : 5>{});
        }
    }
    if (!act) return;
    if constexpr (MODE != 1) {
        const int f = (face_class(k, nz, R) * nc + face_class(j, ny, R)) * nc + face_class(i, nx, R);
        acc = div_by(acc, stab[f], stab[kFilterTab + f]);
        if constexpr (MODE == 2) acc = acc / fmax(gamma, rho[e]);
    }
    out[e] = acc;
}

// what k_filter_near sums: in / S for the transpose (MODE 1), rho in for the
// sensitivity filter (MODE 2)
template <int R, int MODE>
__global__ void __launch_bounds__(256) k_filter_values(int nx, int ny, int nz, const double* __restrict__ in,
                                                       const double* __restrict__ rho, const double* __restrict__ stab,
                                                       double* __restrict__ v) {
    constexpr int nc = 2 * R + 1;
    const int e = blockIdx.x * 256 + threadIdx.x;
    if (e >= nx * ny * nz) return;
    if constexpr (MODE == 1) {
        const int f = (face_class(e / (nx * ny), nz, R) * nc + face_class(e / nx % ny, ny, R)) * nc + face_class(e % nx, nx, R);
        v[e] = div_by(in[e], stab[f], stab[kFilterTab + f]);
    } else {
        v[e] = rho[e] * in[e];
    }
}

// without scratch (H^T), for H^T 1 and with no neighbours (R = 0) the values
// are formed where they are read: one launch
template <int R>
void launch_near(const Ctx& c, const Geom& g, const FilterPlan& p, int mode, const double* in, const double* rho,
                 double gamma, const double* stab, double* scratch, double* out) {
    const unsigned grid = (unsigned)((g.ne + 255) / 256);
#define NEAR(MODE, FORM, IN) \
    k_filter_near<R, MODE, FORM><<<grid, 256, 0, c.s>>>(p.w, g.nx, g.ny, g.nz, IN, rho, gamma, stab, out)
#define VALUES(MODE)                                                                                   \
    k_filter_values<R, MODE><<<grid, 256, 0, c.s>>>(g.nx, g.ny, g.nz, in, rho, stab, scratch); \
    TOPO_LAUNCH_CHECK(c);                                                                              \
    NEAR(MODE, false, scratch)
    if (mode == 0) {
        NEAR(0, false, in);
    } else if constexpr (R == 0) {
        if (mode == 1) NEAR(1, true, in);
        else NEAR(2, true, in);
    } else if (mode == 1 && (!scratch || !in)) {
        NEAR(1, true, in);
    } else if (mode == 1) {
        VALUES(1);
    } else {
        VALUES(2);
    }
#undef VALUES
#undef NEAR
    TOPO_LAUNCH_CHECK(c);
}

template <int R, int TX>
void launch(const Ctx& c, const Geom& g, const FilterPlan& p, int mode, const double* in, const double* rho,
            double gamma, const double* stab, double* out) {
    constexpr int TY = 128 / TX;
    const unsigned grid = (unsigned)((g.nx + TX - 1) / TX) * ((g.ny + TY - 1) / TY) * ((g.nz + p.cz - 1) / p.cz);
    if (mode == 0)
        k_filter<R, TX, 0><<<grid, 128, 0, c.s>>>(p.w, g.nx, g.ny, g.nz, p.cz, in, nullptr, 0.0, stab, out);
    else if (mode == 1)
        k_filter<R, TX, 1><<<grid, 128, 0, c.s>>>(p.w, g.nx, g.ny, g.nz, p.cz, in, nullptr, 0.0, stab, out);
    else
        k_filter<R, TX, 2><<<grid, 128, 0, c.s>>>(p.w, g.nx, g.ny, g.nz, p.cz, in, rho, gamma, stab, out);
    TOPO_LAUNCH_CHECK(c);
}

template <int R>
void launch_tx(const Ctx& c, const Geom& g, const FilterPlan& p, int mode, const double* in, const double* rho,
               double gamma, const double* stab, double* scratch, double* out) {
    if (p.near[mode])
        launch_near<R>(c, g, p, mode, in, rho, gamma, stab + 2 * kFilterTab, scratch, out);
    else if (p.tx == 16) launch<R, 16>(c, g, p, mode, in, rho, gamma, stab, out);
    else launch<R, 32>(c, g, p, mode, in, rho, gamma, stab, out);
}

}  // namespace

// Estimates in clocks of both kernels (filter_plan), fitted to 1224 timings of H,
// H^T and the sensitivity filter: 51 grids of 512 elements to 5 million, cubes,
// rods, plates and odd sizes, r = 1 to 6.  FP64 instructions take 64 clocks on
// each of an SM's four schedulers.
namespace {

// planes of a chunk in turn, each with the classes that its outputs need; what
// counts is how many CTAs share an SM, the lanes of a tile inside the grid, the
// chain of one CTA and the staged values
double march_clocks(const Geom& g, const FilterPlan& p, int mode, int nsm, int adds) {
    const int R = p.R, cz = std::min(p.cz, g.nz), tx = p.tx, ty = 128 / tx;
    int classes[6] = {};
    for (int c = 0; c <= R; ++c)
        for (int q = 0; q < (R + 1) * (R + 2) / 2; ++q) classes[c] += (p.w.bits[q] >> c) & 1u;
    const double staged = (tx + 2 * R) * (ty + 2 * R) / 128.0, rows = R * ty * (tx + 2 * R) / 128.0;
    double own = cz * (mode == 0 ? 3.0 : mode == 1 ? 0.0 : 13.0), shared = 0.0;   // per thread over a chunk
    for (int t = -R; t < cz + R; ++t) {
        const int c0 = t < 0 ? -t : t >= cz ? t - cz + 1 : 0, c1 = std::min(R, std::max(t, cz - 1 - t));
        for (int c = c0; c <= c1; ++c) own += classes[c];
        own += adds + std::min(cz - 1, t + R) - std::max(0, t - R) + 1;
        shared += rows + staged * (mode == 0 ? 0.0 : mode == 1 ? 3.0 : 1.0);
    }
    const double tiles = (double)((g.nx + tx - 1) / tx) * ((g.ny + ty - 1) / ty);
    const double ctas = std::max(1.0, tiles * ((g.nz + cz - 1) / cz) / nsm), lanes = (double)g.nx * g.ny / (128.0 * tiles);
    return 8300.0 + 64.0 * (0.46 * ctas * own * lanes + 1.85 * (own + shared)) +
           290.0 * ctas * std::min(cz + 2 * R, g.nz + R) * staged;
}

// the neighbours that the grid has room for, per warp and as the chain of one
// thread; a launch more where the values are formed first, four FP64
// instructions a neighbour where the transpose divides as it reads
double near_clocks(const Geom& g, const FilterPlan& p, int mode, int nsm, bool scratch) {
    int n = 0;
    for (int c = 0; c <= std::min(p.R, g.nz - 1); ++c)
        for (int b = 0; b <= std::min(p.R, g.ny - 1); ++b)
            if (p.w.reach[c][b] >= 0) n += (2 * std::min((int)p.w.reach[c][b], g.nx - 1) + 1) * (b ? 2 : 1) * (c ? 2 : 1);
    const double per = mode == 1 && !scratch ? 4.0 : 1.0, warps = std::max(1.0, g.ne / (128.0 * nsm));
    // (without scratch the table of weight sums is formed in every call)
    return 8900.0 + (scratch ? (mode > 0 ? 9700.0 : 0.0) : 100.0 * n) +
           64.0 * (per * warps * (n + 3) + 1.5 * n * (per > 1.0 ? 2.0 : 1.0));
}

}  // namespace

void filter_plan(const Geom& g, double r, int nsm, bool scratch, FilterPlan* p) {
    p->R = (int)ceil(r) - 1;   // largest offset along an axis with a positive weight
    const int R = p->R;
    int adds = 0, fmas = 2 * R;
    for (int a = 0; a <= R; ++a)
        for (int b = 0; b <= a; ++b) {
            const int q = pair_class(a, b);
            p->w.bits[q] = 0;
            for (int c = 0; c <= R; ++c) {
                const double w = r - sqrt((double)(a * a + b * b + c * c));
                p->w.w[c][q] = w > 0.0 ? w : 0.0;
                if (w > 0.0) {
                    p->w.bits[q] |= 1u << c;
                    ++fmas;
                }
            }
            if (p->w.bits[q]) adds += a == 0 ? 0 : (b == 0 ? 2 : (a == b ? 1 : 3));
        }
    for (int c = 0; c <= 5; ++c)
        for (int b = 0; b <= 5; ++b) {
            p->w.reach[c][b] = -1;
            if (c <= R && b <= R)
                for (int a = 0; a <= R; ++a)
                    if ((p->w.bits[pair_class(a, b)] >> c) & 1u) p->w.reach[c][b] = (signed char)a;
        }
    // Tile width and planes per CTA that minimise the FP64 time of the
    // fullest SM (16 clocks per warp instruction and SM, 4 warps per CTA)
    // plus the latency of the march (about 600 clocks a plane).  A chunk of
    // cz planes sums cz + 2R of them; narrow grids waste fewer lanes on tiles
    // of 16.
    double best = -1.0;
    for (int tx = 16; tx <= 32; tx *= 2) {
        const double per_plane = adds + (double)R * (tx + 2 * R) / tx;
        const long long xy = (long long)((g.nx + tx - 1) / tx) * ((g.ny + 128 / tx - 1) / (128 / tx));
        for (int gz = 1, cz; gz <= g.nz && gz <= 1024; gz = cz > 1 ? (g.nz - 1) / (cz - 1) + 1 : g.nz + 1) {
            cz = (g.nz + gz - 1) / gz;   // (then on to the next shorter chunk)
            const long long ctas = xy * ((g.nz + cz - 1) / cz);
            const double dp = 64.0 * ((cz + 2 * R) * per_plane + cz * (fmas + 3.0));
            const double t = (double)((ctas + nsm - 1) / nsm) * dp + 600.0 * (cz + 2 * R);
            if (best < 0.0 || t < best) {
                best = t;
                p->tx = tx;
                p->cz = cz;
            }
        }
    }
    // Neighbour by neighbour where the estimates say so, by a margin that keeps
    // the wrong choices cheap (the chosen side is 2 % slower than the better one
    // in the mean; H^T is estimated low on the march's side); always without
    // neighbours, where it is one load per output.
    const double margin[3] = {0.9, 1.1, 0.8}, m = scratch ? 1.0 : 0.6;
    for (int mode = 0; mode < 3; ++mode)
        p->near[mode] = R == 0 || near_clocks(g, *p, mode, nsm, scratch) < m * margin[mode] * march_clocks(g, *p, mode, nsm, adds);
}

void filter_weights(const Ctx& c, const Geom& g, const FilterPlan& p, double* stab) {
    const int nc = 2 * p.R + 1;
    // (the tables that the plan's modes read)
    const bool near = p.near[0] || p.near[1] || p.near[2], march = !(p.near[0] && p.near[1] && p.near[2]);
    k_filter_weights<<<(nc * nc * nc + 31) / 32, 32, 0, c.s>>>(p.w, p.R, g.nx, g.ny, g.nz, march, near, stab);
    TOPO_LAUNCH_CHECK(c);
}

void filter_launch(const Ctx& c, const Geom& g, const FilterPlan& p, int mode, const double* in, const double* rho,
                   double gamma, const double* stab, double* scratch, double* out) {
    switch (p.R) {
        case 0: launch_tx<0>(c, g, p, mode, in, rho, gamma, stab, scratch, out); break;
        case 1: launch_tx<1>(c, g, p, mode, in, rho, gamma, stab, scratch, out); break;
        case 2: launch_tx<2>(c, g, p, mode, in, rho, gamma, stab, scratch, out); break;
        case 3: launch_tx<3>(c, g, p, mode, in, rho, gamma, stab, scratch, out); break;
        case 4: launch_tx<4>(c, g, p, mode, in, rho, gamma, stab, scratch, out); break;
        default: launch_tx<5>(c, g, p, mode, in, rho, gamma, stab, scratch, out); break;
    }
}

}  // namespace topo
