// Internal declarations shared by the translation units of libfvm.
// Host-side launchers are declared here; kernels live in fvm_stage.cu
// (one forward-Euler stage: smoothing, interface geometry, scalar transport,
// momentum predictor, projection right-hand side, correction) and fvm_mg.cu
// (geometric multigrid, reductions); the reverse-mode kernels are declared in
// fvm_adjoint.h.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/fvm.h"

namespace fvm {

enum { PER = 0, WALL = 1 };

// Geometry of one grid level.
struct Geo {
  int n[3];          // cells per axis x, y, z
  int bc[3];         // PER or WALL per axis
  double h;          // cell edge of the finest level (fine kernels)
  double ih;         // 1 / h
  double hd[3];      // cell edge per axis on this level (multigrid)
  double w[3];       // 1 / hd^2 (0 for an axis of one cell: no coupling)
  long long sy, sz;  // strides of y and z
  long long N;       // cell count (< 2^31, checked at create)
};

// Dirichlet temperature walls (at most one axis carries them).
struct TBC {
  int axis;           // -1: no Dirichlet side
  int dir[2];         // 1 if the low / high side of `axis` is Dirichlet
  double T0[2], amp[2];
  int s_axis;         // tangential coordinate of the cosine
  double Ls;          // domain length along s_axis
};

// Material and source parameters (in the form the kernels use).
struct Phys {
  double rho[2], mu[2], lam[2], rcp[2];   // rcp = rho * cp per phase
  double sigma0, dsdT, T0;
  double g[3];
  double q_power, q_radius, q_x0, q_y0, q_speed;
  double eps_a, eps_T, eps_u;             // WENO eps per field
  double eps_n;                           // normal regulariser 1e-8 / h
  double L[3];                            // domain lengths
  double dsdc, c0;                        // sigma += dsdc (c - c0) with a concentration
  double diff_c[2];                       // diffusivity of c per phase
  double eps_c;                           // WENO eps of c
};

// Pointers of one state (u, v, w, alpha, T and the concentration c, null
// when there is none) in the working precision R.
template <typename R>
struct Fields {
  R* u[3];
  R* alpha;
  R* T;
  R* c;
};

// One multigrid level in precision T.
template <typename T>
struct MGLevel {
  Geo geo;
  T* x;
  T* x2 = nullptr;   // the sweeps go in pairs from x to here and swap the two (null: in place)
  T* b;
  T* beta[3];
  T w[3];            // 1 / hd^2 in the level's precision (0: no coupling)
  T wu;              // the one weight of every coupled axis, 0 when they differ
  T* inv;            // reciprocal diagonal per cell (null: the sweeps divide)
  int f[3];          // coarsening factor to the next level
};

constexpr int kMaxLevels = 24;
// thread-block tile of the stage kernels (x fastest)
constexpr int kBX = 32, kBY = 4, kBZ = 4;
constexpr int kRedBlocks = 1024;   // partial-sum slots of the two-pass reductions

// ----- launches that overlap their predecessor's end --------------------------
// A kernel launched with overlap_launch() may be scheduled while the kernel
// before it on the stream still runs; it calls dependency_wait() before it
// touches memory, which returns once that kernel has completed and its writes
// are visible, and so keeps the stream's order (of kernels before that one as
// well: each waits for its own predecessor).  Such a kernel reads what earlier
// ones wrote with plain loads only: a pointer to const __restrict__ or __ldg
// allows the read-only path, whose data must not change while the kernel runs,
// and it is running before its predecessor has finished.
template <typename... P, typename... A>
inline void overlap_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                           A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Offset of the cell above one at offset o, in planes of nxy cells, n in all; the
// last plane wraps to the first.  n may be as large as 2^31 - 1, so that o + nxy is
// formed without a sign.
#ifdef __CUDACC__
__host__ __device__
#endif
inline int plane_above(int o, int nxy, int n) {
  const unsigned a = (unsigned)o + (unsigned)nxy;
  return (int)(a >= (unsigned)n ? a - (unsigned)n : a);
}

#ifdef __CUDACC__
// wait for the predecessor, and let the successor be scheduled
__device__ __forceinline__ void dependency_wait() {
  asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}
#endif

// Work of a pass whose threads walk columns upward and whose blocks each leave
// a partial sum: 32 x 8 columns and a run of kz planes per item; the blocks loop
// over the items.  kRunBlocks fills the chip once (152 SMs x 6 blocks of 256
// threads at 40 registers): 1008 blocks of 64 planes left a second wave of 96,
// 0.27 ms against 0.19 ms for the residual update at 256^3.  Runs of 8 planes
// keep the items even among the blocks (one z-face more per run); small grids
// take shorter runs, down to 2 planes, so that every SM has a block: the right-hand
// side of 88 x 72 x 40 took 28 us with runs of 16 and takes 13.5 us.
constexpr int kRunBlocks = 912;
static_assert(kRunBlocks <= kRedBlocks, "a partial sum per block");
struct ColumnRuns {
  int tx, ty, chunks, kz, blocks;
};
inline ColumnRuns column_runs(const Geo& g) {
  ColumnRuns r;
  r.tx = (g.n[0] + 31) / 32;
  r.ty = (g.n[1] + 7) / 8;
  const long long tiles = (long long)r.tx * r.ty;
  const long long kz = tiles * g.n[2] / kRunBlocks;
  r.kz = (int)(kz < 2 ? 2 : (kz > 8 ? 8 : kz));
  r.chunks = (g.n[2] + r.kz - 1) / r.kz;
  const long long work = tiles * r.chunks;
  r.blocks = (int)(work < kRunBlocks ? work : kRunBlocks);
  return r;
}

// ----- stage launchers (fvm_stage.cu) --------------------------------------
template <typename R>
void launch_smooth(const Geo& g, const R* in, R* out, cudaStream_t s);
// smoothing (passes 0..2), face normals, curvature and Marangoni vector
template <typename R>
void launch_interface(const Geo& g, const Phys& ph, const TBC& tb, int passes, const R* alpha,
                      const R* T, const R* c, R* kappa, R* M0, R* M1, R* M2, cudaStream_t s);
// fct_p / fct_m: limiter ratios of the bounded alpha transport (null: WENO5)
template <typename R>
void launch_scalars(const Geo& g, const Phys& ph, const TBC& tb, Fields<R> X, Fields<R> Sn,
                    Fields<R> Y, const double* dt, double a, double b, double xc_shift,
                    const R* fct_p, const R* fct_m, cudaStream_t s);
// limiter ratios R+, R- of the bounded alpha transport (flux-corrected
// blend of upwind and WENO5 fluxes with the bounds 0 and 1)
template <typename R>
void launch_fct_ratios(const Geo& g, const Phys& ph, Fields<R> X, const double* dt, R* Rp, R* Rm,
                       cudaStream_t s);
// transport of the concentration c (WENO5 advection, diffusion) and its stage
// update Y.c = a Sn.c + b (X.c + dt R_c)
template <typename R>
void launch_concentration(const Geo& g, const Phys& ph, Fields<R> X, Fields<R> Sn, Fields<R> Y,
                          const double* dt, double a, double b, cudaStream_t s);
// phi (optional): the force sum V + f_n + f_M of every face before 1/rho_f
template <typename R>
void launch_momentum(const Geo& g, const Phys& ph, const TBC& tb, Fields<R> X, const R* kappa,
                     const R* M0, const R* M1, const R* M2, R* us0, R* us1, R* us2,
                     const double* dt, cudaStream_t s, R* const* phi = nullptr);
// (returns the number of partial sums it leaves)
template <typename R>
int launch_div_rhs(const Geo& g, R* const* us, const double* dt, double* b, double* partial,
                   cudaStream_t s);
template <typename R, typename B>
void launch_beta(const Geo& g, const Phys& ph, const R* alpha, B* b0, B* b1, B* b2,
                 cudaStream_t s);
template <typename R, typename B>
void launch_correct(const Geo& g, Fields<R> Sn, Fields<R> Y, R* const* us, const double* p,
                    B* const* beta, const double* dt, double a, double b, cudaStream_t s);
template <typename R>
void launch_dt_reduce(const Geo& g, const Phys& ph, Fields<R> X, unsigned long long* maxbits,
                      int* nanflag, cudaStream_t s);
void launch_dt_final(const Geo& g, const Phys& ph, double cfl, double c_cap, double c_visc,
                     double c_therm, double dt_max, const unsigned long long* maxbits,
                     double* dt, int* limiter, cudaStream_t s);
void launch_set_scalar(double* dst, double v, cudaStream_t s);
template <typename R>
void launch_diagnostics(const Geo& g, const Phys& ph, Fields<R> X, const double* p,
                        const double* dt, double* partial, unsigned long long* maxbits,
                        int* nanflag, cudaStream_t s);

// ----- reductions and multigrid (fvm_mg.cu) ----------------------------------
// Deterministic two-pass sums: per-block partial sums in `partial`, then one
// block adds them in a fixed order into *out.
void launch_sum_partials(const double* partial, int nparts, double* out, cudaStream_t s,
                         const int* gate = nullptr);
template <typename T>
void launch_sum_field(const T* a, long long n, bool squares, double* partial, double* out,
                      cudaStream_t s);
void launch_sub_mean(double* a, long long n, const double* sum, cudaStream_t s);
template <typename T>
void launch_zero(T* a, long long n, cudaStream_t s);

// gate (optional): the sweep does nothing once *gate >= gate_min
// xin (optional): the array the neighbours are read from instead of L.x
template <typename T>
void launch_gs(const MGLevel<T>& L, int colour, cudaStream_t s, const int* gate = nullptr,
               int gate_min = 0, const T* xin = nullptr);


// half: the last sweep was of colour 1, whose cells' residuals are taken as 0
template <typename T>
void launch_residual_restrict(const MGLevel<T>& F, const MGLevel<T>& C, cudaStream_t s,
                              bool sweep = false, bool half = false);
// L.inv from the betas
template <typename T>
void launch_inv_diag(const MGLevel<T>& L, cudaStream_t s);
template <typename T>
void launch_prolong(const MGLevel<T>& F, const MGLevel<T>& C, cudaStream_t s);
// a sweep of `colour` on F reading the other colour plus the coarse
// correction C.x of its parent cells (the prolongation folded into the sweep)
template <typename T>
void launch_gs_prolong(const MGLevel<T>& F, const MGLevel<T>& C, int colour, cudaStream_t s);
// a sweep of `colour` from x = 0 that also zeroes the other colour
template <typename T>
void launch_gs_zero(const MGLevel<T>& L, int colour, cudaStream_t s);
// Sweeps of colours `first` and 1 - first in one pass from L.x to L.x2 (see
// k_gs_pair); C: apply the coarse correction first; p: add the result to it, and
// store x2 only with `keep`.  pairs_fit: the grids it takes.
bool pairs_fit(const Geo& g, int fx);
void launch_gs_pair(const MGLevel<float>& L, const MGLevel<float>* C, int first, double* p,
                    bool keep, cudaStream_t s);
// a float sweep of `colour` that adds the new values of its cells and the
// values of the other colour to the double p (p += x after the sweep); store:
// the new values are written to x as well
void launch_gs_addp(const MGLevel<float>& L, int colour, double* p, bool store, cudaStream_t s);
template <typename T>
void launch_beta_coarsen(const MGLevel<T>& F, const MGLevel<T>& C, cudaStream_t s);
// state of a pressure solve's stopping test on the device
struct SolveCtl {
  int iters;      // cycles (F64) or refinements (MIXED) done
  int status;     // 0, FVM_ENOCONV or FVM_EUNSTABLE
  int zero;       // 1: ||b|| = 0, the solution is set to 0
  int verify;     // 1: the updated residual would stop the solve; form it from p
  double rel;     // last relative residual
};

// The coarse tail of a V-cycle (fvm_tail.cu): the levels from the first one
// that fits down to the coarsest, in one launch of one cluster of kTailCTAs
// CTAs.
constexpr int kTailCTAs = 16;
constexpr int kTailLevels = 16;
constexpr int kTailMaxCells = 32768;        // of the tail's first level
constexpr int kTailTopCells = 16384;        // of a double grid solved in the tail as a whole
constexpr int kTailSmem = 220 * 1024;       // shared memory of a CTA
constexpr int kTailCells32 = 512, kTailCells64 = 256;   // cells a CTA should have (float, double)
constexpr int kTailCgCells = 64, kTailCgSingle = 400;    // the same for the coarsest level's CG
constexpr int kTailInvCells = 32;           // the same for the coarsest level by a float inverse
// Cells of a coarsest level solved with a float inverse.  It replaces only conjugate
// gradients that the caller's iteration cap (1000 by default) does not cut short,
// so that a larger limit changes nothing by default.  With a cap of 4000, six cycles
// in double: 961 cells 0.96 ms; 1089 cells 12.0 ms by conjugate gradients, 1.36 with
// the limit at 2048; 2025 cells 15.9 and 3.4 ms.
constexpr int kTailInvMax = 1000;
template <typename T>
struct TailLevel {
  int n[3], f[3];              // cells per axis, coarsening factor to the next level
  int hx, pitch, rows;         // column pairs of a row, stored row length, rows (ny nz)
  int rpc, nact, cap;          // rows per CTA, CTAs with rows, stored cells per CTA
  int ox, ob, oa, otab;        // byte offsets in shared memory: x, b, coefficients, row table
  int cb;                      // bytes of a CTA's coefficients
  bool wall[3];
  T w[3];                      // 1 / hd^2
  const T* beta[3];
  const T* b;                  // the first level's right-hand side and solution
  T* x;
  size_t opack;                // byte offset of the level's blocks in the packed coefficients
};
// With ctl the launch is a whole solve of L[0] (the finest level, x its start):
// cycles until ||b - L x|| <= tol ||b||, b's squared norm in *bn2; otherwise
// it is one cycle from x = 0.
template <typename T>
struct TailArgs {
  int nl;                      // levels, the last one the coarsest
  TailLevel<T> L[kTailLevels];
  int oscr, ocg, ored, ovec;   // byte offsets: fine residuals, CG vectors, reductions, float residual
  int np;                      // order of the float inverse (a multiple of 64; 0: none)
  const float* G;              // the inverse of the coarsest operator / *gscale (null: CG)
  const double* gscale;
  SolveCtl* ctl;
  const double* bn2;
  double tol;
  int maxcycles, fixed;
  const void* pack;            // coefficients of launch_tail_pack (null: formed from beta)
  double rtol;
  int maxit, pre, post;
  int pre0, post0;             // sweeps of the first level
  bool direct;                 // the coarsest level by its packed inverse instead of CG
};
// lay out levels Ls[0 .. nl-1]; false when they do not fit.  smem: bytes per
// CTA, pack: bytes of the packed coefficients
// (inverse: the coarsest level is solved with a float inverse, A.np set)
template <typename T>
bool tail_layout(const MGLevel<T>* Ls, int nl, bool inverse, TailArgs<T>& A, size_t* smem,
                 size_t* pack);
// the float inverse takes one launch per block of 32 pivots and ends in W0 when
// their number is even, else in W1
template <typename T>
int inverse_blocks(const TailArgs<T>& A) {
  const TailLevel<T>& L = A.L[A.nl - 1];
  return (L.rows * L.n[0] + 31) / 32;
}
template <typename T>
void launch_tail_inverse(const TailArgs<T>& A, float* W0, float* W1, double* gscale,
                         cudaStream_t s);
template <typename T>
void launch_tail_pack(const TailArgs<T>& A, cudaStream_t s);
template <typename T>
void launch_tail(const TailArgs<T>& A, size_t smem, cudaStream_t s);
// false where the device cannot hold the cluster: the levels then run one by one
template <typename T>
bool tail_schedulable();
// CG on a coarsest level too large for the tail, vectors in global memory
// (double in both precisions)
template <typename T>
void launch_coarse_cg(const MGLevel<T>& L, double* r, double* d, double* Ad, double rtol,
                      int maxit, cudaStream_t s);
// ||b - L x||^2 into *out (double), x, b, beta in precision T
template <typename T>
void launch_residual_norm2(const MGLevel<T>& L, double* partial, double* out, cudaStream_t s);
// Mixed form: r = b - L p in double with float beta; writes r32, with rd the
// double r too, and ||r||^2.  e32, w32: also the first sweep of the next
// inner solve.  gate (optional): nothing is done unless *gate.
void launch_residual64(const Geo& g, const double* p, const double* b, float* const* beta,
                       float* r32, double* partial, double* out, cudaStream_t s,
                       float* e32 = nullptr, const float* w32 = nullptr, double* rd = nullptr,
                       const int* gate = nullptr);
// rd -= L e (L.x) and the same outputs: r32 (L.b), ||r||^2, and with y the next
// inner solve's first sweep (colour 0; colour 1 is set to 0)
void launch_residual_update(const MGLevel<float>& L, double* rd, float* y, double* partial,
                            double* out, cudaStream_t s);
void launch_add_correction(long long n, double* p, const float* e, cudaStream_t s);

// ----- device-side control of the pressure solve (fvm_mg.cu) -----------------
// The stopping test of a solve runs on the device, inside a CUDA graph with
// a conditional WHILE node: after every cycle (refinement) the controller
// kernel forms ||b - L p|| / ||b|| from the two reduction slots and sets the
// node's condition, so the host never waits for a residual.
void launch_ctl_reset(SolveCtl* ctl, cudaStream_t s);
// bn2 = ||b||^2 and r2 = ||b - L p||^2 (device); fixed > 0: exactly `fixed`
// cycles; runs_total counts the cycles of every solve (launch bookkeeping)
void launch_ctl_step(cudaGraphConditionalHandle h, SolveCtl* ctl, const double* bn2,
                     const double* r2, double rtol, int maxit, int fixed,
                     unsigned long long* runs_total, cudaStream_t s);
// verify = whether the updated residual r2 would stop the solve after this cycle
void launch_ctl_check(SolveCtl* ctl, const double* bn2, const double* r2, double rtol, int maxit,
                      int fixed, cudaStream_t s);
void launch_zero_if_rhs_zero(const SolveCtl* ctl, double* p, long long n, cudaStream_t s);
// copy the controller into a per-stage record and raise the sticky status
void launch_ctl_store(const SolveCtl* ctl, SolveCtl* rec, int* sticky, cudaStream_t s);

}  // namespace fvm
