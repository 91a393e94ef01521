// Host-side launchers of the RMT kernels (explicitly instantiated for float and double).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "rmt_common.cuh"

// streaming multiprocessors of the current device (its attribute, read once per device); launch
// widths are multiples of it
int sm_count();

// Launches in a chain of dependent kernels on one stream.  An ordinary launch behind another kernel costs
// 4.1 us of the stream's time on a GB300 however short the kernels are, one with programmatic
// serialization 1.4 us (and 1.05 against 1.22 us as a node of a captured graph): the solves outside
// step graphs, some 800 launches per timestep, are bound by this.  The kernel may start before its
// predecessor has ended, so it must call wait_prior() before it touches memory; the predecessor gives no
// early trigger (a trigger at its start let the waiting blocks take SMs from the running ones: 17.5
// against 9.5 us on 16384 blocks).
__device__ __forceinline__ void wait_prior() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... P, typename... A>
inline void launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  lc.gridDim = grid;
  lc.blockDim = block;
  lc.dynamicSmemBytes = smem;
  lc.stream = s;
  lc.attrs = &at;
  lc.numAttrs = 1;
  cudaLaunchKernelEx(&lc, kernel, P(args)...);
}

// Planes per thread column of a column-marching kernel over `units` points (cap at most): one
// plane on small grids, where a column's planes would only follow one another, and more once
// the columns alone give every SM a full set of resident threads.
inline int column_chunk(long units, int cap) {
  const long c = units / ((long)sm_count() * 2048);
  return c < 1 ? 1 : (c > cap ? cap : (int)c);
}

// A multigrid right-hand side or solution as the step kernels see it.  FP64 mode: the FP64
// array d.  FP32 mode: two-float pairs, value = h + l (d is null), so that no FP64 arithmetic
// runs in the FP32 step.
struct MGVec {
  double* d;
  float* h;
  float* l;
};

// face-array bundle: vector value at every d-face (3 comps) for d = 0..2
template <typename T>
struct Faces3 {
  T* v[3][3];  // v[d][a]
};

// ---- flow (rmt_flow.cu) -------------------------------------------------------------
// scratch for the cells that some band reaches: their list, the bodies at each, their count, and whether
// a cell is listed
struct StressList {
  int* cell;       // N
  uint64_t* mask;  // N
  int8_t* listed;  // N
  int* count;
};
// bbs: band boxes of the bodies (6 ints each, stride ints apart) of the time level of views;
// rows: nine cell arrays of scratch for the face rows of the listed cells (the Godunov slope arrays,
// free at both stress passes)
// t: device pointer to the simulated time; the stress is evaluated at *t + toff
template <typename T>
cudaError_t launch_stress_div(const Geo& g, const T* u, const Body* bodies, const BodyView<T>* views, int nb,
                              const int* bbs, int bstride, const double* t, double toff, T* out, const StressList& L,
                              T* const rows[9], cudaStream_t s);
void launch_tick(double* t, double dt, cudaStream_t s);
// advecting velocities of the bar states and the upwinded face states of the velocity; bodies / views / nb: the
// bodies at step n, for the wall-repulsion term of the forcing.  slopes and wcell (nine cell arrays each) are
// scratch of the FP64 form; the FP32 form needs none
template <typename T>
cudaError_t launch_godunov(const Geo& g, const T* u, const T* p, const T* rho, const T* divtau, const Body* bodies,
                           const BodyView<T>* views, int nb, T* const vadv[3], T* const uf[3][3], T* const slopes[9],
                           T* const wcell[9], cudaStream_t s);
template <typename T>
void launch_mac_setup(const Geo& g, T* const uf[3][3], MGVec b, cudaStream_t s);
template <typename T>
void launch_mac_correct(const Geo& g, T* const uf[3][3], const T* rho, MGVec q, T* const umac[3],
                        cudaStream_t s);
template <typename T>
void launch_advect(const Geo& g, T* const uf[3][3], T* const umac[3], T* adv, cudaStream_t s);
template <typename T>
void launch_density(const Geo& g, const Body* bodies, const BodyView<T>* views, int nb, const int* bbs, int bstride,
                    T* rho, cudaStream_t s);
template <typename T>
// bodies / views / nb: the bodies at step n+1/2, for the wall-repulsion term
void launch_ustar(const Geo& g, const T* u, const T* adv, const T* p, const T* rho_h, const T* divtau_h,
                  T* ustar, const Body* bodies, const BodyView<T>* views, int nb, cudaStream_t s);
// the wall-repulsion acceleration of every cell from the given bodies' phi, as FP64 (3 N)
template <typename T>
void launch_rep_field(const Geo& g, const Body* bodies, const BodyView<T>* views, int nb, double* out, cudaStream_t s);

// ---- swimmer diagnostics (rmt_diag.cu) ----------------------------------------------
// one body's sums [w u (3), w, w sigma_a : grad u, w Phi_elas, w over cells with F, w (J-1)^2]
// into scratch[0..8) (FP64); scratch holds body_stats_scratch_bytes(); t: device time
size_t body_stats_scratch_bytes();
template <typename T>
void launch_body_stats(const Geo& g, const T* u, const Body& b, const BodyView<T>& v, const double* t, double* scratch,
                       cudaStream_t s);
template <typename T>
void launch_fe_setup(const Geo& g, const T* u, const T* ustar, MGVec b, cudaStream_t s);
template <typename T>
void launch_fe_update(const Geo& g, const T* ustar, const T* rho_h, MGVec psi, T* u, T* p,
                      T* psi_out, cudaStream_t s);
template <typename T>
void launch_fill(T* a, T v, long n, cudaStream_t s);

// ---- extrapolation (rmt_extrap.cu) ------------------------------------------------
// One body's arrays.  list: the band's cells sorted by layer (capacity: the grid), written by the layer
// passes and read by the fits and the corrector of the same step; cnt: BAND_COUNTERS ints,
// cnt[l] the cells of layer l (l = 1..8), cnt[BAND_TICKET] the finished blocks of the last pass; bb: the
// band's bounding boxes of the two parities (6 ints each)
constexpr int BAND_COUNTERS = 10, BAND_TICKET = 9;
template <typename T>
struct Band {
  T *X[2], *PHI[2];
  int8_t* LAY[2];
  T *XH, *PHIH;
  int *list, *cnt, *bb;
};
// The bodies that a launch works on, one per grid row y: bodies m0, m0 + 1, ... of the device arrays, or
// (bodies null) the one given here.  out: the parity that is written; in: the parity whose box bounds the
// windows and whose map the corrector starts from (-1: the windows are the grid)
template <typename T>
struct BandSet {
  const Body* bodies;
  const Band<T>* bands;
  int m0, count, out, in;
  Body one;
  Band<T> oneb;
};
template <typename T>
void launch_init_xi(const Geo& g, const Body& b, T* x, cudaStream_t s);
// predictor of every body's map at layers 0 and 1, from the map at in to the map at out; tiles: launch width for
// a body's tiles (the kernel strides over the whole window)
template <typename T>
cudaError_t launch_xi_predict(const Geo& g, const T* u, T* const vadv[3], T* const uf[3][3], T* const umac[3],
                              const BandSet<T>& S, int tiles, cudaStream_t s);
// blocks: launch width for a body's window (kernels stride over the whole window); wls_blocks: launch
// width of the fits.  err[0] counts degenerate fits, err[1] (FP32 storage) band cells near the seam of
// their body's image window
template <typename T>
void launch_extrapolate(const Geo& g, const BandSet<T>& S, int blocks, int wls_blocks, int* err, cudaStream_t s);
// the same for the map at out, followed by the corrector: xi^{n+1/2} from the maps at in and out
template <typename T>
void launch_extrapolate_correct(const Geo& g, const BandSet<T>& S, int blocks, int wls_blocks, int* err,
                                cudaStream_t s);

// ---- multigrid (rmt_mg.cu) ----------------------------------------------------------
struct MGSolver;  // opaque
// kind 0: cell-centred 7-point (MAC), kind 1: nodal trilinear FE (27-point)
MGSolver* mg_create(const Geo& g, int kind, int prec_fp32, cudaError_t* err);
size_t mg_footprint(const Geo& g, int kind, int prec_fp32);  // device bytes mg_create would request
size_t mg_device_bytes(const MGSolver* m);                   // device bytes it did request
// device bytes charged for one allocation of `bytes` (allocations are 256-byte granular, at least 16 bytes asked)
inline size_t dev_bytes(size_t bytes) { return ((bytes < 16 ? 16 : bytes) + 255) / 256 * 256; }
void mg_destroy(MGSolver* m);
// Level-0 right-hand side (filled before a solve) and solution, as MGVec.
MGVec mg_rhs(MGSolver* m);
MGVec mg_solution(MGSolver* m);
// FP64 copy of the solution for read-back (FP32 mode: converted on s first)
const double* mg_solution64(MGSolver* m, cudaStream_t s);
// the cell density the operator is built from on the finest level (the caller's array, type T)
void mg_set_density(MGSolver* m, const void* rho);
// smoother sweeps before/after the coarse correction and the Jacobi weight (negative: keep)
void mg_set_smoother(MGSolver* m, int pre, int post, double omega);
// sweeps on the levels below the finest (negative: the finest level's counts)
void mg_set_coarse_smoother(MGSolver* m, int pre, int post);
// V-cycles on the correction equation between FP64 residual evaluations (>= 1)
void mg_set_inner(MGSolver* m, int inner);
// block height (1, 2, 4 or 8 rows of 32 threads) of the level kernels
void mg_set_block(MGSolver* m, int by);
// start each solve from the previous solution (zero before the first) instead of from zero
void mg_set_warm(MGSolver* m, int warm);
// device int set to 1 when a solve's right-hand-side mean, solution mean or residual norm is
// not finite (null: not checked)
void mg_set_nonfinite_flag(MGSolver* m, int* flag);
// z-chunk length (planes a block marches) of the finest level's stencil tiles: the fused
// red-black sweep (MAC; ignored where the level does not take it) or the FE tile kernels;
// 0 restores the wave-filling heuristic.  mg_zchunk returns the length in use.
void mg_set_zchunk(MGSolver* m, int zchunk);
int mg_zchunk(const MGSolver* m);
// MAC in FP32: one fused red-black pass per sweep (1: on the large levels that allow it, the
// default; 2: on every level that allows it; 0: never), else one pass per colour
void mg_set_sweep(MGSolver* m, int fused);
// Optional timing hook around the finest-level smoother and FP64-residual launches:
// hook(ctx, which, begin, stream) with which = 0 (smoother colour, or all sweeps of a smoothing call where
// mg_block_sweeps), 1 (FP64 residual) or 2 (fused red-black sweep).
typedef void (*mg_hook_fn)(void* ctx, int which, int begin, cudaStream_t s);
void mg_set_hook(MGSolver* m, mg_hook_fn fn, void* ctx);
// whether the finest level (MAC) is small enough that one launch makes all sweeps of a smoothing call
bool mg_block_sweeps(const MGSolver* m);
// Solves to rtol (or a fixed cycle count); returns cycles used, -1 on non-convergence.
int mg_solve(MGSolver* m, double rtol, int max_cycles, int fixed_cycles, cudaStream_t s, cudaError_t* err);
