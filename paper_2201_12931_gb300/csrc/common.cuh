// Internal declarations of the GB300 topology-optimisation library.
// Layout in HBM (all device arrays, natural x-fastest indexing):
//   nodal vectors  : interleaved 3*nn scalars, dof = 3*n + c
//   element arrays : ne scalars, e = i + nx*(j + ny*k)
//   Dirichlet mask : one byte per node, bit c set = DOF c fixed
//   per level      : modulus E_l (FP64 and FP32 copies) with the element
//                    scale 2^l folded in, homogenized density, mask, and the
//                    V-cycle work vectors of each precision.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "dfloat.cuh"
#include "modal.cuh"
#include "topo.h"

namespace topo {

using bf16 = __nv_bfloat16;

struct Ctx {
    cudaStream_t s;
    long long* launches;
};

struct Geom {
    int nx, ny, nz;       // elements per axis
    long long nn, ne;     // nodes, elements
    int NX() const { return nx + 1; }
    int NY() const { return ny + 1; }
    int NZ() const { return nz + 1; }
};

struct OpLaunch {          // launch geometry of the operator kernel on one level
    Geom g;
    int gx = 1, gy = 1, gz = 1, cz = 1;
    long long ctas() const { return (long long)gx * gy * gz; }
};

struct Op64Plan {          // FP64 operator by elements (op64.cu)
    int cz = 0;            // layers per thread; 0: the level uses the tile kernel
    int blocks = 0;        // blocks of the node kernel (dot partials)
    long long nt = 0;      // element threads
    size_t scratch() const { return (size_t)(cz + 1) * 12 * nt; }   // doubles
};

template <typename T>
struct ModalK;

template <typename T>
struct VBuf {             // V-cycle work vectors of one level in one precision
    T* a = nullptr;
    T* b = nullptr;
    T* f = nullptr;       // right-hand side (levels > 0)
};

struct Level {
    Geom g;
    bf16* ha = nullptr;       // BF16 V-cycle iterates (TOPO_MIXED_BF16, levels < L-1)
    bf16* hb = nullptr;
    double* Ke64 = nullptr;   // stored Galerkin element matrices (homogenize = 2, levels >= 1)
    float* Ke32 = nullptr;
    OpLaunch op32, op64, opdf;   // operator launch geometry per precision
    OpLaunch optc;            // tensor-core FP32 operator (tc_op.cu)
    Op64Plan p64;             // FP64 operator by elements (op64.cu)
    bool brick = false;       // FP32 operators by bricks (op_brick.cu)
    double scale = 1.0;       // 2^l
    double* rho = nullptr;    // homogenized density
    double* E64 = nullptr;    // 2^l * (Emin + rho^p (E0 - Emin))
    float* E32 = nullptr;
    double* Dinv64 = nullptr; // per node 1 / (kdiag * sum of E over the <= 8 elements around it)
    float* Dinv32 = nullptr;
    uint8_t* mask = nullptr;
    VBuf<double> v64;
    VBuf<float> v32;
};

struct Coarse {           // dense coarsest-grid solve: K_c^-1 = W^T W, W = L^-1
    int n = 0, npad = 0;
    double* A = nullptr;      // npad^2 work matrix (assembly, Cholesky factor)
    double* W64 = nullptr;    // L^-1 (lower, row-major npad^2)
    double* WT64 = nullptr;   // (L^-1)^T (upper, row-major)
    float* W32 = nullptr;
    float* WT32 = nullptr;
    double* y64 = nullptr;    // temporaries of length npad
    float* y32 = nullptr;
    int* info = nullptr;      // device: n - smallest DOF with a non-positive pivot (0 = ok)
    int* order = nullptr;     // DOF of the level's node order at each row: nodes along the shortest axis first, then two-ended
    double* Dk = nullptr;     // inverses of the 32 x 32 diagonal blocks of L (npad x 32)
};

constexpr int kDirRing = 8;   // CG direction buffers of the fused iterations

struct PcgGraph {             // a captured launch sequence (a PCG iteration, or the coarsest factorization)
    cudaGraphExec_t exec = nullptr;
    long long launches = 0;   // kernel launches per replay
    bool failed = false;      // capture not possible: direct launches
};

// Filter weights by class: w[c][pair_class(a, b)] = max(0, r - |(a, b, c)|) for
// offsets 0 <= b <= a <= R in a plane and c planes apart (R <= 5); bit c of
// bits = that weight is positive
struct FilterW {
    double w[6][21];
    unsigned bits[21];
    signed char reach[6][6];      // [c][b]: the largest a with a positive weight, -1: none
};
struct FilterPlan {
    FilterW w;
    int R = 0, tx = 32, cz = 1;   // largest offset; tile width and planes per CTA of the march
    bool near[3] = {};            // by mode: neighbour by neighbour instead of the march
};
// weight sums S by distance to the faces, 1 / S; the same for k_filter_near
constexpr int kFilterTab = 11 * 11 * 11, kFilterTables = 4 * kFilterTab;

struct Scalars {              // device-resident CG scalars
    double rz, rz_new, pq, rr, alpha, beta, ff, aux;
    double rz_old;            // z.r of the previous iteration (flexible beta)
};

// What the last block of a kernel with partial sums does with them (tail.cuh)
enum TailKind { TAIL_NONE, TAIL_ALPHA, TAIL_BETA, TAIL_RR };
struct DotTail {
    int kind = TAIL_NONE;
    Scalars* sc = nullptr;
    double* hist = nullptr;       // TAIL_ALPHA: alpha of the direction's ring slot, may be null
    unsigned* ticket = nullptr;   // device counter, 0 between kernels
};

}  // namespace topo

struct topo_grid {
    topo_params prm{};
    cudaStream_t stream = nullptr;
    int device = 0;
    int L = 1;
    std::vector<topo::Level> lev;
    topo::Coarse cs;
    // fine-level vectors (interleaved, 3*nn)
    double *x = nullptr, *f = nullptr, *r = nullptr, *z = nullptr, *p = nullptr, *q = nullptr;
    float *r32 = nullptr, *z32 = nullptr, *p32 = nullptr, *q32 = nullptr, *d32 = nullptr;
    double* K0d = nullptr;          // reference element matrix (E = 1, h = 1), 24x24
    float* K0f = nullptr;
    topo::ModalCoef modal{};
    topo::ModalK<double>* mk64 = nullptr;   // host copies of the operator coefficients
    topo::ModalK<float>* mk32 = nullptr;
    topo::ModalK<topo::dfl>* mkdf = nullptr;  // double-FP32 split of mk64
    uint32_t* tcB = nullptr;        // B operand image of the tensor-core operator (tc_b_image)
    int* tc_err = nullptr;          // device: a tensor-core MMA wait ran out (0 = ok)
    long long npartials = 0;                // size of the partials buffer
    double* dc_work = nullptr;      // element work arrays (filter / OC)
    double* xnew_work = nullptr;
    double* oc_hi = nullptr;        // OC upper move-limit bounds
    double* G64 = nullptr;          // Galerkin child matrices P_o^T K0 P_o (homogenize = 2)
    double* oc_dv = nullptr;        // active-element indicator of a passive OC step (lazy)
    topo::FilterPlan filt{};        // weights and launch geometry of the filter for S_radius
    double* stab = nullptr;         // its tables of weight sums (kFilterTables)
    double* dv_cache = nullptr;     // H^T 1 for dv_radius
    double* rdv_cache = nullptr;    // its reciprocal (on first use)
    double S_radius = -1.0, dv_radius = -1.0;
    int nsm = 152;                  // multiprocessors of the device
    double* lam = nullptr;          // OC bisection state (device)
    char* oc_ws = nullptr;          // search for the OC multiplier (oc_search_bytes, on first use)
    double* dtmp = nullptr;         // device scratch scalars
    int* dflag = nullptr;           // device: density out of [0,1] seen
    bool coarse_dirty = true;
    bool dinv64_dirty = true;       // FP64 D^-1 of the levels: formed when an FP64 V-cycle first needs it
    bool x_zero = true;             // warm start is u = 0 (initial residual is f)
    // launch timing of fine-level operator kernels (topo_profile_enable)
    bool prof_on = false;
    std::vector<cudaEvent_t> prof_ev;     // 2 per record
    std::vector<int> prof_kind;           // mode * 2 + (float ? 1 : 0)
    int prof_n = 0;
    double* partials = nullptr;     // reduction partials
    topo::Scalars* sc = nullptr;    // device scalars
    double* host_sc = nullptr;      // pinned host mirror
    bool have_density = false, have_bc = false, fp64_ready = false, fp32_ready = false, bf16_ready = false;
    long long launches = 0;
    // CG directions of the fused iterations: a ring of kDirRing buffers (p,
    // level 0's v.b, and these), so that x += alpha p runs once per ring
    // (cg_flush_x) instead of once per iteration
    double* dring64[topo::kDirRing - 2] = {};
    float* dring32[topo::kDirRing - 2] = {};
    double* alpha_hist = nullptr;   // device: alpha of each ring slot
    unsigned* ticket = nullptr;     // device: blocks that have finished (DotTail)
    double* el64 = nullptr;         // face contributions of the FP64 operator by elements (op64.cu)
    topo::PcgGraph graph64[topo::kDirRing], graph32[topo::kDirRing];   // captured PCG iterations per ring slot
    topo::PcgGraph coarse_graph;            // captured coarsest-grid assembly, factorization and inverse
    cudaStream_t cap_stream = nullptr;  // private stream the graphs are captured on
    cudaStream_t side_stream = nullptr; // second branch of a captured graph
    cudaEvent_t side_event = nullptr;
    topo_solve_stats stats{};
    std::string err;
    topo::Ctx ctx() { return topo::Ctx{stream, &launches}; }
};

namespace topo {

constexpr int kUpdateBlocks = 8 * 152;   // largest grid of cg_update_r: 2048 threads on every SM
constexpr int kRedBlocks = 1024;   // fixed grid of reduction kernels (deterministic order)
constexpr int kProfMax = 65536;    // launch records of topo_profile_enable

// ---- stencil.cu ----------------------------------------------------------
// ST_APPLY_P: K.p of CG with the direction update fused in: p = u + beta p_old
// (u = z, f = p_old, beta from the device scalars or 0 when null), q = K p
// written to out and p to pout
// ST_JACOBI2: the first two damped-Jacobi sweeps from u = 0 in one pass:
// u1 = omega D^-1 f formed per node from f and D^-1, then u2 = u1 + omega
// D^-1 (f - K u1) (u unused)
enum StencilMode { ST_APPLY = 0, ST_JACOBI = 1, ST_RESID = 2, ST_JACOBI0 = 3, ST_APPLY_P = 4, ST_JACOBI2 = 5 };
// out = op(u, f); with dot != nullptr also writes per-CTA partial sums of
//   APPLY: u.out   JACOBI/JACOBI0: f.out   RESID: out.out
// and returns the number of partials written.
// nsm: multiprocessors of the device (wave-aware z chunking)
OpLaunch op_launch32(const Geom& g, int nsm);
OpLaunch op_launch64(const Geom& g, int nsm);
OpLaunch op_launch_df(const Geom& g, int nsm);
template <typename T>
int stencil(const Ctx& c, int mode, const OpLaunch& L, const ModalK<T>& mk, const T* E, const uint8_t* mask,
            const T* u, const T* f, T* out, T omega, double* dot_partials, const T* Dinv, T* pout = nullptr,
            const double* beta = nullptr);
// V-cycle operators with BF16 iterates and FP32 arithmetic: u BF16, f FP32,
// output BF16 (out_h) or FP32 (out_f).  Instantiated: JACOBI0 -> BF16,
// JACOBI -> BF16, JACOBI -> FP32 (with or without dot), RESID -> FP32;
// returns -1 for any other combination, else as stencil().
int stencil_bf16(const Ctx& c, int mode, const OpLaunch& L, const ModalK<float>& mk, const float* E,
                 const uint8_t* mask, const bf16* u, const float* f, bf16* out_h, float* out_f, float omega,
                 double* dot_partials, const float* Dinv);
// Operator in double-FP32 arithmetic (dfloat.cuh) on FP64 storage: u, f and
// the modulus E are FP64, split into FP32 pairs on load; launch geometry of
// the FP64 kernel.  Instantiated: APPLY -> FP64 out; RESID -> FP64 out; RESID
// -> FP32 out with r.r partials (the outer residual of the mixed solve).
// Returns -1 for any other combination, else as stencil().
int stencil_df(const Ctx& c, int mode, const OpLaunch& L, const ModalK<dfl>& mk, const double* E, const uint8_t* mask,
               const double* u, const double* f, double* out64, float* out32, double* dot_partials);
// ---- op64.cu: FP64 operators by elements -----------------------------------
// Levels of at most this many elements take op64_apply for every mode but
// JACOBI0.  What sets the line is memory, not time: the scratch takes 12 (cz + 1)
// / cz values per element, at most 200 MB up to here.  The z-march is the slower
// side throughout: K.u over 0.46M elements 160 us by elements and 227 by the
// march, 1.05M 361 / 511, 1.07M 362 / 437, 1.23M 411 / 562, 4.2M 1355 / 1728.
constexpr long long kOp64Max = 1LL << 20;
Op64Plan op64_plan(const Geom& g, int nsm);
// as stencil(); Dinv is read by JACOBI and JACOBI2; scratch: p.scratch() doubles
int op64_apply(const Ctx& c, int mode, const Geom& g, const Op64Plan& p, const ModalK<double>& mk, const double* E,
               const uint8_t* mask, const double* u, const double* f, double* out, double omega, double* dot_partials,
               const double* Dinv, double* pout, const double* beta, double* scratch, const DotTail& tail);
// ---- op_brick.cu: FP32 operators of small levels ---------------------------
// Levels of at most this many nodes take brick_apply for every mode but JACOBI0.
// The two sides cross here: 48 CG iterations with bricks / the z-march on the
// finest level take 5.11 / 5.27 ms at 71k nodes, 5.58 / 5.80 at 76k, 6.72 / 6.51
// at 83k, 4.84 / 4.72 at 88k, 5.37 / 4.85 at 109k, 5.73 / 4.85 at 137k and
// 6.55 / 5.58 at 204k (grids of several shapes).  A V-cycle alone crosses between
// 99k and 109k: it has no K.p, whose march gains most from a full GPU.
constexpr long long kBrickMax = 80000;
cudaError_t brick_init();   // per device, before the first launch
long long brick_ctas(const Geom& g);
// as stencil(); Dinv is read by JACOBI and JACOBI2; ec (JACOBI only, may be
// null): the iterate is u + P~ ec, ec and its mask maskc on the next coarser level
int brick_apply(const Ctx& c, int mode, const Geom& g, const ModalK<float>& mk, const float* E, const uint8_t* mask,
                const float* u, const float* f, float* out, float omega, double* dot_partials, const float* Dinv,
                float* pout, const double* beta, const float* ec, const uint8_t* maskc, const DotTail& tail);
// fc = diag(free_c) P^T diag(free) (f - K u), on the next coarser level
void brick_restrict(const Ctx& c, const Geom& g, const ModalK<float>& mk, const float* E, const uint8_t* mask,
                    const float* u, const float* f, const uint8_t* maskc, float* fc);
// ---- tc_op.cu: FP32 operators with the element products on tcgen05 tensor cores
OpLaunch op_launch(const Geom& g, int ty, int resident_ctas, bool fp64 = false);
OpLaunch op_launch_tc(const Geom& g, int nsm);
constexpr int kTcBWords = 2304;
// host: shared-memory image of B = [K0_hi | K0_lo | K0_hi] (TF32), kTcBWords words
void tc_b_image(const double* K0, uint32_t* img);
// APPLY / JACOBI / RESID (with or without dot partials) as stencil(); -1 for
// JACOBI0.  *err is set if a bounded wait on the tensor cores ran out.
int stencil_tc(const Ctx& c, int mode, const OpLaunch& L, float kdiag, const float* E, const uint8_t* mask,
               const float* u, const float* f, float* out, float omega, const uint32_t* Bimg, double* dot_partials,
               int* err);
// dense coarsest operator from E_e K0, or from stored element matrices Ke (non-null);
// order (3 * nodes) receives the DOF of each row (two-ended, see coarse_chain)
void assemble_coarse(const Ctx& c, const Geom& g, const double* K0, const double* E, const double* Ke,
                     const uint8_t* mask, double* A, int npad, int* order);
// Half-bandwidth of that operator: rows follow the node order with the
// shortest axis running fastest and the longest slowest, which makes it
// 3 (1 + N0 + N0 N1) + 2 for the two smaller node counts N0 <= N1
int coarse_band(const Geom& g);
// The factorization is a chain of 32 x 32 diagonal blocks.  A matrix of n rows
// and half-bandwidth band is eliminated from both ends at once: the first and
// the last coarse_chain blocks of rows do not touch each other as long as the
// rows between them are band or more.  Rows are stored in that order: the first
// t = 32 coarse_chain rows, the last t backwards, then those between.
inline int coarse_chain(int n, int band) { return n > band ? (n - band) / 64 : 0; }
// ---- galerkin.cu: stored Galerkin coarse element matrices ------------------
void galerkin_init_constants();
// host: the 8 child matrices G_o = P_o^T K0 P_o (8 x 576, o-major)
void galerkin_child_matrices(const double* K0, double* G);
// Kc (coarse elements of the level below gf) = sum_o P_o^T Kchild P_o; the
// children are Ef[e] K0 (Kf null: scaled sum of G) or Kf[e] (576 per
// element, element-major)
void galerkin_build(const Ctx& c, const Geom& gf, const double* K0, const double* G, const double* Ef, const double* Kf,
                    double* Kc);
// the operator modes of stencil() on a level given by element matrices (no dot)
template <typename T>
void elem_op(const Ctx& c, int mode, const Geom& g, const T* Ke, const uint8_t* mask, const T* u, const T* f, T* out,
             T omega);
// low = true: FP32 modal contraction of FP64-relative displacements (mixed modes)
void element_energy_sens(const Ctx& c, const Geom& g, const ModalCoef& mc, const double* u, const double* rho,
                         double E0, double Emin, double penal, double* dc_out, double* partials, bool low);

// ---- transfer.cu ---------------------------------------------------------
template <typename T>
void restrict_residual(const Ctx& c, const Geom& gf, const uint8_t* maskf, const uint8_t* maskc,
                       const T* rf, T* rc);
template <typename T>
void prolong_add(const Ctx& c, const Geom& gf, const uint8_t* maskf, const uint8_t* maskc,
                 const T* ec, T* uf);
// uf (BF16) += P~ ec with FP32 arithmetic; ec FP32 (coarsest solve) or BF16
template <typename TE>
void prolong_add_bf16(const Ctx& c, const Geom& gf, const uint8_t* maskf, const uint8_t* maskc, const TE* ec,
                      bf16* uf);
// coarse = scale * mean of the 8 children (densities: scale 1; moduli: scale 2)
void homogenize(const Ctx& c, const Geom& gf, const double* rho_f, double* rho_c, double scale);
// per node D^-1 = 1 / (kdiag * sum of E over the <= 8 elements around it),
// in the precision of E (indices in 32 bits: the grid limit of create_grid)
template <typename T>
void diag_inverse(const Ctx& c, const Geom& g, const T* E, T kdiag, T* Dinv);
void simp_moduli(const Ctx& c, long long ne, const double* rho, double scale, double E0,
                 double Emin, double penal, double* E64, float* E32, int* bad_flag);
void mask_from_dofs(const Ctx& c, long long nn, const uint8_t* fixed_dofs, uint8_t* mask);
void inject_mask(const Ctx& c, const Geom& gf, const uint8_t* maskf, uint8_t* maskc);
void masked_copy_load(const Ctx& c, long long nn, const uint8_t* mask, const double* fin, double* fout);

// ---- blas.cu -------------------------------------------------------------
template <typename A, typename B>
void dot_partials(const Ctx& c, long long n, const A* a, const B* b, double* partials);
// reduces n partials into *dst (device double), fixed order
void reduce_to(const Ctx& c, const double* partials, int n, double* dst);
// CG scalar steps, all on device: alpha = rz/pq ; beta = rz_new/rz, rz = rz_new
// hist != nullptr: alpha is also stored there (the direction ring's slot)
void cg_alpha(const Ctx& c, const double* partials, int n, Scalars* sc, double* hist = nullptr);
void cg_beta(const Ctx& c, const double* partials, int n, Scalars* sc);
// flexible (Polak-Ribiere) beta for a preconditioner that varies between
// applications: beta = z_new.(r_new - r_old) / z_old.r_old = -alpha z_new.q / rz_old,
// from the partial sums of z_new.q; run after cg_beta
void cg_beta_flexible(const Ctx& c, const double* partials_zq, int n, Scalars* sc);
template <typename T>
void cg_update_xr(const Ctx& c, long long n, const Scalars* sc, const T* p, const T* q, T* x, T* r,
                  double* partials);
template <typename T>
void cg_update_p(const Ctx& c, long long n, const Scalars* sc, const T* z, T* p);
// r -= alpha q and sc->rr = r.r (x updated later by cg_flush_x)
template <typename T>
void cg_update_r(const Ctx& c, long long n, Scalars* sc, const T* q, T* r, double* partials, unsigned* ticket);
// x += alpha_j p_j for j = 0 .. count-1 in that order (the same operations as
// count successive x += alpha p steps); p_j = ring[j], alpha_j = alpha[j]
template <typename T>
void cg_flush_x(const Ctx& c, long long n, T* const* ring, const double* alpha, int count, T* x);
template <typename S, typename D>
void convert(const Ctx& c, long long n, const S* src, D* dst);
void axpy_f32_into_f64(const Ctx& c, long long n, const float* d, double* x);
template <typename T>
void zero(const Ctx& c, long long n, T* v);
// dense coarse solve
// A = L L^T in place and W = L^-1 for n rows in two-ended order (see
// coarse_chain).  band: half-bandwidth of A in entries before the reordering
// (npad for a dense matrix); order: the DOF of each row; Dk (npad x 32 doubles)
// receives the inverses of the 32 x 32 diagonal blocks of L; info: n minus the
// smallest DOF whose pivot is not positive, 0 if there is none.  The inverse of a block row needs the factor
// up to its block column only: with side != c.s (stream capture) its launches
// go to that stream, ordered by the event, beside the chain of diagonal
// blocks, and are joined at the end.
void chol_inverse(const Ctx& c, cudaStream_t side, cudaEvent_t ready, double* A, double* W, int n, int npad, int band,
                  int* info, const int* order, double* Dk);
void transpose_dense(const Ctx& c, const double* W, double* WT, int npad);
template <typename T>
void coarse_apply(const Ctx& c, const Coarse& cs, const T* W, const T* WT, const T* rhs, T* y, T* out);

// message returned by topo_last_error(NULL)
void set_global_error(const std::string& msg);
// ---- filter.cu -----------------------------------------------------------
// weights and launch geometry for radius r (0 < r <= 6); scratch: whether
// filter_launch gets it
void filter_plan(const Geom& g, double r, int nsm, bool scratch, FilterPlan* p);
// fills stab (kFilterTables doubles) with the weight sums of the plan's radius
void filter_weights(const Ctx& c, const Geom& g, const FilterPlan& p, double* stab);
// mode 0: out = H in; 1: out = H^T in (in null: H^T 1); 2: the sensitivity
// filter out = H(rho in) / max(gamma, rho).  scratch: one value per element, or
// null (not for the sensitivity filter; H^T then divides where it reads)
void filter_launch(const Ctx& c, const Geom& g, const FilterPlan& p, int mode, const double* in, const double* rho,
                   double gamma, const double* stab, double* scratch, double* out);
// ---- oc.cu ---------------------------------------------------------------
// OC update: q = x sqrt(max(-dc~, 1e-30) / dv~) (in place over dc~ allowed),
// move-limit bounds lo / hi, and FP32 copies of (q, lo, hi, dv) in pack (16 B
// per element).  dv null: 1 (the volume of x itself), else rdv = 1 / dv; passive (0 active, 1
// solid, 2 void): lo = hi = 1 / 0, q = 0, and dv is written (0; active: 1).
void oc_prepare(const Ctx& c, long long ne, const double* x, const double* dct, double* q, double* dv,
                const double* rdv, const uint8_t* passive, double move, double* lo, double* hi, void* pack, void* search);
void reciprocal(const Ctx& c, long long n, const double* v, double* r);
// the multiplier with sum dv clamp(q lambda^(-1/2), lo, hi) = target: screening
// passes in FP32, then the bisection on [0, 1e9] with exact volumes; result
// and success in the search state (oc_search_bytes of device memory)
size_t oc_search_bytes();
void oc_search(const Ctx& c, long long ne, const double* lo, const double* hi, const double* q, const double* dv,
               const void* pack, void* search, double target, double tol);
// x_new of a successful search (x untouched else), then the change and
// whether the search failed (synchronises)
void oc_search_write(const Ctx& c, long long ne, double* x, const double* lo, const double* hi, const double* q,
                     void* search, double* partials);
cudaError_t oc_search_read(const Ctx& c, const void* search, double* change, bool* bad);
// self-weight load f_out = f_ext (null: 0) - (w/8) sum of rho over the elements at each node, in z
void gravity_load(const Ctx& c, const Geom& g, const double* rho, const double* f_ext, double* f_out, double w);
// dc_e += -(w/4) sum of u_z over the corners of e
void gravity_sensitivity(const Ctx& c, const Geom& g, const double* u, double* dc, double w);
void oc_bisect_step(const Ctx& c, long long ne, const double* lo, const double* hi, const double* num,
                    const double* dv, double* partials, double* lam_state);
void oc_bisect_finalize(const Ctx& c, const double* partials, double* lam_state, double volfrac_ne,
                        double tol);
void oc_write(const Ctx& c, long long ne, double* x, const double* lo, const double* hi, const double* q,
              const double* lam_state, void* search, double* partials);

}  // namespace topo

#define TOPO_LAUNCH_CHECK(ctx)                 \
    do {                                       \
        ++*(ctx).launches;                     \
    } while (0)
