// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include "fastdiv.h"
#include "pic_poisson.h"

namespace pp {

// ------------------------------------------------------------------ errors
void set_error(const char *fmt, ...);
void clear_error();

#define PP_CUDA(call)                                                                   \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess) {                                                        \
            ::pp::set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_),     \
                            __FILE__, __LINE__);                                        \
            return PIC_POISSON_ECUDA;                                                   \
        }                                                                               \
    } while (0)

// ------------------------------------------------------------------ complex vector types
template <class T> struct V2t;
template <> struct V2t<double> { using type = double2; };
template <> struct V2t<float> { using type = float2; };
template <class T> using V2 = typename V2t<T>::type;

constexpr int kMaxBatch = PIC_POISSON_MAX_BATCH;
constexpr int kSMs = 152;                 // of this GPU: what launches are sized for (any number runs them)

// ------------------------------------------------------------------ one multigrid level
// Coefficients of A_m on a uniform level (appendix Eqs. interior_face_conductances,
// dirichlet_face_conductances), separated by direction:
//   (A_m u)_(i,k) = (D0r_i + tz_k cz_i + lambda_m mu_i) u_(i,k)
//                   - cw_i u_(i-1,k) - ce_i u_(i+1,k) - cz_i (u_(i,k-1) + u_(i,k+1))
// with cw_0 = ce_(nr-1) = 0 (Dirichlet r faces fold into D0r) and the axial
// neighbour terms dropped on the wall rows, whose tz is 3 (one interior face plus
// a half-distance Dirichlet face of conductance 2 cz) instead of 2.
struct LevelHost {
    int nr = 0, nz = 0;
    double dr = 0, dz = 0;        // dr: the mean radial width (the spacing itself on a uniform mesh)
    std::vector<double> rf;       // [nr + 1] radial faces
    std::vector<double> rc, drc;  // [nr] cell centres (face midpoints) and widths
    int ncls = 0;                 // distinct axial row classes: min(nz, 3)
    std::vector<double> cw, ce, cz, d0r, mu;   // per radial index
    std::vector<double> tz;       // per class
    std::vector<double> invd, diag;             // [ncls][nr][nm]
    std::vector<double> hw, he, hz;             // [ncls][nr][nm]: cw, ce, cz divided by diag
    // composite domain (empty otherwise): active flags [nz][nr], the coefficient
    // class of every row [nz] (rows with the same active pattern in themselves
    // and both neighbours share one), and each class's sum of face conductances
    // D0 [ncls][nr] (zero for inactive cells)
    std::vector<unsigned char> act;
    std::vector<int> rcls;
    std::vector<double> d0c;
    // non-uniform axial mesh (empty otherwise): faces [nz+1], centres and widths [nz]
    std::vector<double> zf, zc, dzc;
    // per-row tables (composite domain or non-uniform axial mesh): north
    // coupling hn [ncls][nr][nm] (hz then holds the south one) and the four
    // face conductances toward active neighbours [ncls][nr] (0 across a
    // Dirichlet face) for the residual
    std::vector<double> hn, ccw, cce, ccs, ccn;
};

// One level of one problem, as the kernels see it.
template <class T> struct LevelDev {
    int nr, nz, nm, ncls;
    unsigned rnm, rnr, rhr;       // floor((2^32 - 1) / d) for d = nm, nr, nr / 2 (fdiv, fastdiv.h)
    int nt;                       // azimuthal cells (Parseval weights of the norms)
    int init;                     // what a restriction into the next level writes (see launch_residual_restrict)
    int strip;                    // smoother: rows of one parity updated per thread (1, 2 or 4; 0: one entry)
    T relax;                      // 1 - omega (over-relaxed smoother; the h tables and invd carry omega)
    const T *cw, *ce, *cz;        // [nr]
    const T *invd, *diag;         // [ncls][nr][nm]: omega / diag, diag
    const T *hw, *he, *hz;        // [ncls][nr][nm] omega * off-diagonal conductances / diag
    const int4 *hzw;              // FP64 levels: the h tables in limbs (fixed.h), (hz, hw), [ncls][nr][nm]; null with
    const int2 *hev;              // per-row tables of many classes.  he beside it without per-row tables; else null.
                                  // (Made for any omega; the over-relaxed smoother does not read them)
    const int4 *rzw;              // FP64 levels without per-row tables: cz, cw [nr], ce [nr] and
    const int2 *rev, *rdg;        // diag [ncls][nr][nm] times 2^rq in limbs; with per-row tables: hen, ren below
    int rq;
    const int4 *hen, *ren;        // FP64 levels with per-row tables of few classes: (he, hn) in limbs beside hzw, which
                                  // then holds (hz, hw), and (cce, ccn) beside rzw, (ccs, ccw), [ncls][nr]; else null
    const int *rcls;              // per-row tables (composite domain or non-uniform axial mesh): coefficient
                                  // class of each row [nz]; null: rows 0 and nz-1 are classes 0 and
                                  // ncls-1, the others class 1.  An inactive cell has zero diag, invd and
                                  // h entries, holds u = 0 and has no residual
    int holes;                    // the level has cells outside a composite domain's patches
    const T *hn;                  // per-row tables: omega * north conductance / diag (hz: the south one)
    const T *ccw, *cce, *ccs, *ccn;   // per-row tables: face conductances [ncls][nr] for the residual
    V2<T> *u;                     // iterate / correction, [nz][nr][nm]
    V2<T> *b;                     // right-hand side, [nz][nr][nm]
    V2<T> *bh;                    // right-hand side / diag, [nz][nr][nm]
};

// Coarsest level: separable direct solve (z eigenbasis, tridiagonal in r).
template <class T> struct CoarseDev {
    int nr, nz, nm;
    const T *V;                   // [nz][nz] orthonormal eigenvectors of the axial operator, V[k*nz+j]
    const int2 *Vl;               // FP64: the same as limbs of V 2^61 (fixed.h); else null
    const T *e;                   // [nr] off-diagonal -ce_i of the radial operator
    const T *piv;                 // [nm][nz][nr] inverse pivots of the Thomas factorisation
    const T *cpr;                 // [nm][nz][nr] upper multipliers of the Thomas factorisation
    const T *f, *fq;              // [nm][nz][nr], [nm][nz][TRI_Q]: its factors as tri_rows (coarse.h) takes them
    // composite domain (nact > 0): dense solve over the nact active cells,
    // A_m = A_0 + lambda_m diag(mu) = M^(-1/2) Q (Lambda + lambda_m) Q^T M^(-1/2) with M = diag(mu)
    int nact;
    const int *aidx;              // [nact] cell index k nr + i of each active cell
    const int *amap;              // [nz][nr] active index of a cell, -1 when inactive
    // (applied in FP32 for both precisions: a coarse-grid correction)
    const float *Q;               // [nact][nact] eigenvectors, Q[a nact + j]
    const float *QT;              // [nact][nact] the transpose
    const float *lam;             // [nact] eigenvalues of M^(-1/2) A_0 M^(-1/2)
    const float *isq;             // [nact] 1 / sqrt(mu) of each active cell
    const float *lamm;            // [nm] lambda_m
    float *Y, *Z;                 // [2 nm][nact] scratch of the dense solve: y = M^(-1/2) b scaled, then
                                  // z = (Lambda + lambda_m)^(-1) Q^T y, one column per (mode, part)
    double *up;                   // [2 nm] the power of two each column was scaled down by
};

// Work of one launch over a batch of problems: problem p owns the blocks
// [start[p], start[p+1]) of the grid; f / c are its fine / coarse level views.
// done: the convergence loop's per-problem stop flags (Ctrl::done) or null;
// blocks of a problem that has stopped return at once, so its iterate stays
// the one whose residual was reported while other problems of the batch go on.
template <class T> struct LaunchTab {
    int n;
    const int *done;
    int pid[kMaxBatch];           // problem index of each entry (entries list only the problems that take part)
    unsigned start[kMaxBatch + 1];
    int chunk;                    // consecutive pieces of a block's size that each block works on
    LevelDev<T> f[kMaxBatch];
    LevelDev<T> c[kMaxBatch];
};
// A block of a batch looks its problem up and copies its level views, a chain of
// some ten dependent loads, before it has work: it then works on `chunk` pieces,
// as many as leave the launch four times the blocks that the chip holds.
inline int batch_chunk(size_t blocks) {
    const size_t c = blocks / (kSMs * 6 * 4);
    return (int)(c < 1 ? 1 : c > 8 ? 8 : c);
}

// What a launch over a table gets: the table and, for a plan of one problem,
// its entry by value.  The kernel then reads the level views from its own
// parameters (constant bank) instead of through three dependent loads, and
// keeps none of them in registers: the restriction of every cell on a stretched
// axial mesh needs 48 registers instead of 80 (4.0 -> 2.0 ms per mixed solve at
// 512 x 128 x 400, the whole solve 11.7 -> 9.1 ms).
template <class T> struct LevelArg {
    const LaunchTab<T> *tab;
    LevelDev<T> f, c;
};
template <class T> struct TabRef {
    LaunchTab<T> *tab = nullptr;  // device (null when no problem takes part)
    bool one = false;             // plan of one problem: f and c below are its entry
    LevelDev<T> f{}, c{};
    explicit operator bool() const { return tab != nullptr; }
    LevelArg<T> arg() const { return {tab, f, c}; }
};

template <class T> struct CoarseTab {
    int n;
    const int *done;
    int pid[kMaxBatch];           // problem index of each entry (entries list only the problems that take part)
    unsigned start[kMaxBatch + 1];
    LevelDev<T> f[kMaxBatch];
    CoarseDev<T> c[kMaxBatch];
    size_t smem;                  // dynamic shared memory of the largest problem
};

// The dense coarsest solves of a batch (csrc/dense.cu): problem p owns the
// blocks [start[p], start[p+1]) of the preparation launch (one per mode and
// part) and [gstart[p], gstart[p+1]) of each GEMM launch (one per tile).
template <class T> struct DenseTab {
    int n;
    const int *done;
    int pid[kMaxBatch];
    unsigned start[kMaxBatch + 1];
    unsigned gstart[kMaxBatch + 1];
    LevelDev<T> f[kMaxBatch];     // the coarsest level (b in, u out)
    CoarseDev<T> c[kMaxBatch];
};

struct DefectTab {                // mixed precision: FP64 level 0 and FP32 level 0 of each problem
    int n;
    const int *done;
    int pid[kMaxBatch];           // problem index of each entry (entries list only the problems that take part)
    unsigned start[kMaxBatch + 1];
    LevelDev<double> d[kMaxBatch];
    LevelDev<float> s[kMaxBatch];
    int init_red[kMaxBatch];
};

// Azimuthal transforms of one problem's finest level.
struct FFTProb {
    int nr, nt, nz, nm, ncls, log2M;
    const int4 *tw;               // [M+1][2] e^{-2 pi i m / nt}, M = nt / 2: limbs (fixed.h) of cos, -sin; +sin, 0
    double half_inv_n;            // 1 / (2 nt)
    const double *s;              // [nr] s_i (Eq. mode_rhs), [nz][nr] when s_rows; null: plain 1/N transform
    int s_rows;                   // composite domain: s per cell, 0 outside the patches
    const int *rcls;              // composite domain: level-0 coefficient class per row (b_hat)
    const double *bD;             // [nz][nr] Dirichlet right-hand side; may be null
    const double *invd;           // level-0 inverse diagonal [ncls][nr][nm]; null: no b_hat
    double2 *b;                   // mode-layout output of the forward transform
    double2 *bh;                  // b / diag (may be null)
    const double2 *uhat;          // mode-layout input of the inverse transform
    const double *rho;            // (nz, nt, nr) input of the forward transform
    double *phi;                  // (nz, nt, nr) output of the inverse transform
    const double2 *guess;         // mode-layout initial iterate copied into b (mode-space guesses)
};

struct FFTTab {
    int n;
    unsigned start[kMaxBatch + 1];
    FFTProb p[kMaxBatch];
    size_t smem;
};

// Device-side state of the convergence loop (one per plan).
// tol <= 0 (solve to the rounding floor): the loop stops once the relative
// residual has not fallen below half of its last reference value (the value
// at the last halving) in this many consecutive convergence tests.  Six
// tolerates a contraction of up to 0.89 per test, as on strongly stretched
// meshes where the point smoother loses much of its effect.
constexpr int kFloorWindow = 6;

struct Ctrl {
    double tol;                   // per solve
    int max_cycles;               // per solve
    int inc;                      // cycles added by one pass of the loop body
    int inc_first;                // cycles added by the first pass (mixed: inner_first)
    int cycles;                   // V-cycles applied so far
    int cont;                     // 1 while some problem is still iterating
    int n;                        // problems
    int scaled;                   // residual partials are of the sigma-scaled residual (mixed)
    double bnorm2[kMaxBatch];     // Parseval-weighted ||b||^2
    double rel[kMaxBatch];        // latest relative residual
    double best[kMaxBatch];       // reference relative residual: the value at the last halving (floor detection)
    double sigma_used[kMaxBatch]; // mixed: scale of the correction problem being solved
    double inv_sigma_used[kMaxBatch];
    double sigma_next[kMaxBatch]; // mixed: scale for the next defect
    double count[kMaxBatch];      // cells of the 3-D grid (scale normalisation)
    double rel_first[kMaxBatch];  // relative residual at the first convergence test
    int stall[kMaxBatch];
    int status[kMaxBatch];
    int done[kMaxBatch];
    int done_cycles[kMaxBatch];
    unsigned rbegin[kMaxBatch];   // residual-norm partials of problem p: [rbegin, rend)
    unsigned rend[kMaxBatch];
    unsigned arrived;             // blocks that have come to a test of launch_deep_solve
    int polls;                    // per solve: reads of `arrived` after which a test's wait gives up
};

// First stage of the residual-norm reduction: each block sums PSUM_CHUNK
// consecutive block partials of one problem, so the convergence test (one
// block) adds a few dozen numbers instead of tens of thousands -- on one SM
// the FP64 additions alone took longer than the rest of the test.
constexpr int PSUM_CHUNK = 2048;
// Up to PSUM_MIN partials the test adds them itself, which saves the launch of k_psum (a batch: plan.cu).  Solves
// without that launch over solves with it, by partials: FP64 1,000 0.984, 2,100 0.988, 4,200
// 0.993, 6,200 0.999, 8,300 1.000; mixed 1,600 0.965, 4,200 0.991, 8,300 0.990, 10,400 0.995,
// 12,500 1.000, 16,600 1.003, 25,000 1.009.
constexpr unsigned PSUM_MIN = 10000;
struct PsumTab {
    int n;
    unsigned start[kMaxBatch + 1];    // blocks (chunks) of problem p: [start[p], start[p+1])
    unsigned in_begin[kMaxBatch];     // its first-level partials
    unsigned in_end[kMaxBatch];
};

// ------------------------------------------------------------------ overlapped launches
// The solve's kernels are launched so that a kernel's blocks may start while
// the one before still runs (programmatic dependent launch): they read their
// launch table and level view -- written at plan time -- and work out their
// indices; pdl_wait() then blocks until the kernel before has completed and
// its writes are visible.  Nothing a kernel of the solve writes is read before
// that.  pdl_go(), after the wait, lets the next kernel start likewise.  Most
// kernels below level 0 run for 2 to 4 us, of which launch, table reads and
// index arithmetic were more than half.  With the level views by value (LevelArg)
// and overlapped launches: 32 x 16 x 32 in one graph 632 -> 534 us, 152 x 32 x 90
// from the host 1,393 -> 1,002 us, channel-plume 256 x 64 x 192 3,170 -> 2,700 us;
// of these the views alone give 592, 1,308 and 2,812 us.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
constexpr size_t PDL_MAX_THREADS = size_t(kSMs) * 2048;
template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    // a launch of several waves hides its own start, and blocks that wait early
    // only take room from the ones at work
    const bool overlap = (size_t)grid * block <= (size_t)PDL_MAX_THREADS;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// ------------------------------------------------------------------ dynamic shared memory
// A kernel's limit of dynamic shared memory belongs to the process, not to a
// launch: the launchers set it to the kernel's ceiling below, never to the size
// of their own launch, which a plan with smaller arrays on another thread would
// lower between the call and the launch ("too many resources requested").
constexpr int kMaxNtheta = 256;           // azimuthal cells
constexpr int kMaxCoarseCells = 4096;     // cells and rows of an exactly solved coarsest level
constexpr int kMaxCoarseNz = 64;
constexpr int TRI_Q = 48;         // products of factors per row of the tridiagonal solves (coarse.h)
// Elements that k_coarse holds of an nr x nz level: b, then four padded arrays, the
// rows of V that it reads, the products of the factors, the columns' exponents.
constexpr size_t coarse_smem_elems(int nr, int nz) {
    return (size_t)nr * nz + 4 * (size_t)(nr + 1) * nz + (size_t)(nz - nz / 2) * nz + (size_t)nz * TRI_Q + (size_t)nr;
}
// (5 nr nz + nr + 52 nz + nz ceil(nz / 2): with nr nz given it is largest at one end of the range of nz)
constexpr size_t COARSE_MAX_ELEMS =
    coarse_smem_elems(kMaxCoarseCells / kMaxCoarseNz, kMaxCoarseNz) > coarse_smem_elems(kMaxCoarseCells, 1)
        ? coarse_smem_elems(kMaxCoarseCells / kMaxCoarseNz, kMaxCoarseNz)
        : coarse_smem_elems(kMaxCoarseCells, 1);
static_assert(COARSE_MAX_ELEMS * sizeof(double) <= 227 * 1024, "the largest exact solve fits one block");

// ------------------------------------------------------------------ launchers
// All launchers enqueue on `st` and return cudaGetLastError().  `grid` is the
// table's total block count (start[n]); tables live in device memory.
cudaError_t launch_forward(const FFTTab *tab, unsigned grid, size_t smem, double *partials, cudaStream_t st);
cudaError_t launch_inverse(const FFTTab *tab, unsigned grid, size_t smem, cudaStream_t st);
// b = guess for every problem of the table (mode-layout initial iterates).
cudaError_t launch_copy_guess(const FFTTab *tab, unsigned grid, cudaStream_t st);

// threads: block size of the smoother (64, 128, 256 or 512; the table's block
// ranges must have been computed with the same size).
// strip: see pic_poisson_desc.smooth_strip; sor: over-relaxed update (omega != 1).
template <class T>
cudaError_t launch_smooth(const TabRef<T> &tab, unsigned grid, int color, int threads, int strip, bool sor,
                          cudaStream_t st, bool rowwise = false);
// red_only: residual of the red fine cells only (valid right after a black half-sweep).
// Per problem, f.init selects what is written into the coarse level c: 0 = b only
// (coarsest, solved directly); 1 = also b_hat and u = 0; 2 = also b_hat and
// u = (red ? b_hat : 0), the first red half-sweep from zero.
// masked: the plan holds per-row tables -- a composite domain or a
// non-uniform axial mesh (class tables per row, no residual or correction
// outside the patches); false runs the plain kernels.
template <class T>
cudaError_t launch_residual_restrict(const TabRef<T> &tab, unsigned grid, bool red_only, double *partials,
                                     cudaStream_t st, bool masked = false);
// r = b - A_m u on level f of every problem (r_out: optional per-problem output
// in c[p].u), Parseval-weighted norms of r and b into partials[block] and
// partials[partial_stride + block].
template <class T>
cudaError_t launch_residual(const LaunchTab<T> *tab, unsigned grid, bool write_r, double *partials,
                            unsigned partial_stride, cudaStream_t st, bool masked = false);
template <class T>
cudaError_t launch_prolong(const TabRef<T> &tab, unsigned grid, bool black_only, cudaStream_t st,
                           bool masked = false);
template <class T>
cudaError_t launch_coarse(const CoarseTab<T> *tab, unsigned grid, size_t smem, cudaStream_t st);
// Dense coarsest solves, in stage order: 0 preparation (g_prep blocks), 1 and 2 the two GEMMs (g_gemm blocks);
// nmax: active cells of the largest.
template <class T>
cudaError_t launch_dense(const DenseTab<T> *tab, int stage, unsigned g_prep, unsigned g_gemm, int nmax, cudaStream_t st);
unsigned dense_gemm_blocks(int nact, int nm);   // GEMM blocks of one problem
// Full-multigrid start: u_f = P u_c on every fine cell (black_only: on the
// black ones, for a red Gauss-Seidel half-sweep to follow); coarse b =
// restricted fine b.
template <class T>
cudaError_t launch_interp(const TabRef<T> &tab, unsigned grid, cudaStream_t st, bool masked = false,
                          bool black_only = false);
template <class T>
cudaError_t launch_rhs_restrict(const TabRef<T> &tab, unsigned grid, cudaStream_t st, bool masked = false);

// f and Q of a coarsest level from its factorisation.
template <class T> cudaError_t launch_tri_factors(const CoarseDev<T> &D, cudaStream_t st);
// V 2^61 of n entries in limbs (CoarseDev::Vl).
cudaError_t launch_limbs_v(const double *V, int2 *Vl, int n, cudaStream_t st);
// The limb tables of levels from their binary64 ones (ntab entries of [ncls][nr][nm] each).
struct LimbSet {
    static constexpr int MAX = 12;
    int n = 0;
    size_t ntab[MAX];
    LevelDev<double> L[MAX];
};
cudaError_t launch_limbs(const LimbSet &set, cudaStream_t st);

// zero_x: the FP64 iterate is zero (r = b; the kernel also writes x = 0).
cudaError_t launch_defect(const DefectTab *tab, unsigned grid, const Ctrl *ctrl, double *partials, bool zero_x,
                          cudaStream_t st, bool masked = false);
cudaError_t launch_update(const DefectTab *tab, unsigned grid, const Ctrl *ctrl, cudaStream_t st);

// Sums of the forward transform's partials per problem -> ctrl->bnorm2; initial
// scale of the mixed correction problem.
cudaError_t launch_bnorm(Ctrl *ctrl, const FFTTab *fft, const double *partials, cudaStream_t st);
// Convergence test: per-problem residual norms from partials, stop rule,
// cycle count (+inc when counting == 1, +inc_first when 2), graph
// conditionals (use_handle bit 0: handle, bit 1: handle2).
// out[start[p] + c] = sum of chunk c of problem p's partials (fixed order).
cudaError_t launch_psum(const PsumTab *tab, unsigned grid, const double *partials, double *out, cudaStream_t st);
cudaError_t launch_check(Ctrl *ctrl, const double *partials, int counting, cudaGraphConditionalHandle handle,
                         cudaGraphConditionalHandle handle2, int use_handle, cudaStream_t st);
// Plain sum of n partials into *out (single problem helpers).
cudaError_t launch_sum(const double *partials, int n, double *out, cudaStream_t st);

cudaError_t measure_fma(cudaStream_t st, double *fp64_gflops, double *fp32_gflops);

// Threads per block of the multigrid kernels and the block count a launch
// over `entries` work items of one problem needs.
constexpr int MG_THREADS = 256;
inline unsigned mg_blocks(size_t entries, int threads = MG_THREADS) {
    return (unsigned)((entries + threads - 1) / threads);
}
// Blocks of one smoother launch over a level (see k_smooth): rows of each
// parity in strips of `strip`, and per strip the (nr/2) * nm entries of one
// colour of a row.
inline unsigned smooth_blocks(int nr, int nz, int nm, int strip, int threads) {
    const size_t w = (size_t)(nr / 2) * nm;
    const unsigned bx = (unsigned)((w + threads - 1) / threads);
    const unsigned s0 = (unsigned)(((nz + 1) / 2 + strip - 1) / strip), s1 = (unsigned)((nz / 2 + strip - 1) / strip);
    return (s0 + s1) * bx;
}
// Fused multi-sweep smoother of one FP32 level of one problem (fused.cu).
struct FusedProb {
    LevelDev<float> L;            // the level (coefficient tables, b_hat; L.u is not used)
    LevelDev<float> C;            // the next coarser level (restriction fused into pre-smoothing)
    int init;                     // what the fused restriction writes into C (as LevelDev::init)
    const float2 *in;             // iterate before the half-sweeps
    float2 *out;                  // iterate after them (another buffer)
    int G, ngroups;               // modes per block, mode groups
    int P, ntiles;                // column pairs per block (halo included), column tiles
    int R, nkr;                   // output rows per block, row ranges
};
struct FusedTab {
    int n;
    const int *done;
    int pid[kMaxBatch];           // problem index of each entry (entries list only the problems that take part)
    unsigned start[kMaxBatch + 1];
    FusedProb p[kMaxBatch];
};
constexpr int FUSED_THREADS = 256;
// nh = 2 or 4 half-sweeps, red first; res: also the red-cell residual and
// its restriction into FusedProb::C (levels coarsened 2:1 in r and z).
// rw: per-row coefficient classes (composite domains; plain problems of the
// batch keep the three-class path).
cudaError_t launch_smooth_fused(const FusedTab *tab, unsigned grid, int nh, bool res, cudaStream_t st, bool rw);
// Block shape and count for an nr x nz level with nm modes (about target_blocks blocks).
void fused_shape(int nr, int nz, int nm, int nh, bool res, int target_blocks, FusedProb &f, unsigned &blocks);

// Mode-local bottom of the V-cycle (bottom.cu): the level above the coarsest
// (U) and the coarsest level's solve, one block per (problem, mode, part).
template <class T> struct BottomProb {
    LevelDev<T> U;
    CoarseDev<T> D;
    int pre, post;                // sweeps
    int red_only, black_only;     // restriction of the red cells, prolongation to the black cells
};
template <class T> struct BottomTab {
    int n;
    const int *done;
    int pid[kMaxBatch];           // problem index of each entry (entries list only the problems that take part)
    unsigned start[kMaxBatch + 1];
    BottomProb<T> p[kMaxBatch];
};
constexpr int BOTTOM_THREADS = 1024;
constexpr size_t BOTTOM_MAX_SMEM = 200 * 1024;
template <class T> size_t bottom_smem_bytes(int nr, int nz, int ncls, int ncr, int ncz);
template <class T> cudaError_t launch_bottom(const BottomTab<T> *tab, unsigned grid, size_t smem, cudaStream_t st);

// V-cycles of the lower levels in the shared memory of one cluster per mode
// (deep.cu): levels l .. L-2 smoothed, level L-1 solved exactly.
constexpr int DEEP_THREADS = 512;
constexpr int DEEP_LEVELS = 8;
constexpr size_t DEEP_MAX_SMEM = 225 * 1024;
constexpr int DEEP_MAX_NZ = kMaxCoarseNz;   // rows of the coarsest level
constexpr int DEEP_POLLS = 1 << 22;      // default of Ctrl::polls: seconds, where a test's wait takes microseconds
// Entries (cells x modes) of the first level up to which it takes that way.  Whole
// hierarchies: whatever the shared memory of 8 blocks per mode holds is faster (deep.cu;
// of 40 sizes of 230 thousand to 2.4 million entries none above 626 thousand fits).
// Lower levels: above, the level kernels fill the chip and are as fast or faster --
// solves with launches / in shared memory from a level of 139 k entries 981 / 916 us,
// 208 k 5,060 / 5,077, 832 k 5,060 / 5,280 (FP64 9,600 / 10,470).
constexpr size_t DEEP_MAX_WHOLE = 640000, DEEP_MAX_LOWER = 160000;
template <class T> struct DeepLevel {
    LevelDev<T> L;
    int fz, fr, zmul;             // coarsening to the next level; rows per row of the coarsest level
    unsigned u, bh, b, tab;       // shared-memory offsets
};
template <class T> struct DeepArg {
    int nl = 0;                   // smoothed levels (0: not available)
    int C = 1;                    // blocks per cluster; the coarsest level has at least as many rows
    int pre = 0, post = 0, red_only = 0, black_only = 0;
    int top_b = 0;                // the first level's b is held in shared memory too
    int bottom = 0;               // a full-multigrid start solves the two coarsest levels together
    unsigned bc = 0, fo = 0, ws = 0, V = 0, ps = 0, fs = 0, cs = 0, Q = 0, ecol = 0, smem = 0;
    CoarseDev<T> D{};
    DeepLevel<T> lv[DEEP_LEVELS]{};
};
template <class T> size_t deep_layout(DeepArg<T> &A, int C);   // sets C and the offsets, returns the bytes
template <class T> int deep_resident(const DeepArg<T> &A);      // clusters of A that the device holds at a time
template <class T> cudaError_t launch_deep(const DeepArg<T> &A, bool from_zero, int cycles, cudaStream_t st);
// The whole solve in one cooperative launch; every cluster must be resident.
// start: 0 from the level's iterate, 1 from zero, 2 a full-multigrid start; partials: two per block.
cudaError_t launch_deep_solve(const DeepArg<double> &A, int start, Ctrl *ctrl, double *partials, cudaStream_t st);

// Pieces of the separable coarsest-level solve shared by k_coarse (mg.cu) and
// k_bottom (bottom.cu).
//
// One element copied from global to shared memory by cp.async (4 or 8
// bytes, no register round trip): a block issues every load of its problem
// before it waits once, instead of one L2 round trip per loop step.
template <class T> __device__ __forceinline__ void cp_async_elem(T *smem, const T *gmem) {
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "4- or 8-byte elements");
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"((int)sizeof(T)) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// Close the thread's current group of copies; wait until at most N groups are in flight.
__device__ __forceinline__ void cp_async_group_close() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_group_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

constexpr int FFT_TI = 32;        // radial columns per transform CTA
constexpr int FFT_THREADS = 256;
size_t fft_smem_bytes(int nt);

// 3x3 convolution on the tcgen05 tensor cores (conv_tc.cu): 0 on success, 1
// when the shape or alignment is not taken (run the mma.sync kernel), else a
// PIC_POISSON_* error.  up: see pic_nn_conv3x3_cat (null: one input); pool:
// see pic_nn_conv3x3_pool (null: none).
int launch_conv3x3_tc(const void *up, int cu, const void *in, int cin, const void *w, const float *bias, void *out,
                      float *out32, void *pool, int cout, int n, int h, int wd, int relu, cudaStream_t st);

// Weight and bias gradients of a 3x3 convolution on mma.sync (wgrad.cu):
// whether it takes these tensors, and the two launches (at most max_parts
// partials of 9 cin cout + cout floats in scratch).
// up: see pic_nn_conv3x3_cat (null: one input).
bool wgrad_mma_takes(const void *up, int cu, const void *in, int cin, const void *dout, int cout);
cudaError_t launch_wgrad_mma(const void *up, int cu, const void *in, int cin, const void *dout, int cout, int n, int h, int wd, float *dw,
                             float *dbias, float *scratch, int max_parts, cudaStream_t st);

}  // namespace pp
