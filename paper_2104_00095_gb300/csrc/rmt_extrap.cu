// Parallel layer-wise extrapolation of the reference map (arXiv 2104.00095, main text
// "Extrapolation of xi(x,t)"; SI "Weighting scheme for weighted least squares-based
// extrapolation"): classification of the interior (phi_0(xi) < 0), layer marking over
// face neighbours, and one weighted least-squares fit per band cell, layer after layer.
//
// This translation unit is compiled with --fmad=false: the fits are evaluated operation
// by operation in a fixed order, so that the integer outcomes (layer labels, which fits
// are degenerate, which weights are positive) are reproducible.  FP64 storage fits in FP64;
// FP32 storage holds displacements S = xi - x0 (rmt_common.cuh) and fits them in FP32, redone
// in FP64 when ill-conditioned.
#include "rmt_band.cuh"

namespace {

constexpr int TPB = 128;
inline int nblocks(long n) {
  long b = (n + TPB - 1) / TPB;
  if (b > (long)sm_count() * 128) b = (long)sm_count() * 128;
  return (int)(b < 1 ? 1 : b);
}

// xi^0 = x at every cell; on a periodic axis the image of x nearest the body centre (FP32
// storage: the displacement from the cell's image, zero)
template <typename T>
__global__ void k_init_xi(Geo g, Body b, T* __restrict__ x) {
  wait_prior();
  GRID_LOOP(c, g.N) {
    if constexpr (disp_storage<T>()) {
      x[c] = x[g.N + c] = x[2 * g.N + c] = T(0);
      continue;
    }
    int ii[3];
    decode(c, g.n[0], g.n[1], ii[0], ii[1], ii[2]);
#pragma unroll
    for (int d = 0; d < 3; d++) {
      double v = g.lo[d] + (ii[d] + 0.5) * g.h;
      if (g.per[d]) v += g.len[d] * floor((b.c[d] - v) / g.len[d] + 0.5);
      x[d * g.N + c] = (T)v;
    }
  }
}

// layer 0 = candidates (finite xi) with phi_0(xi) < 0; everything else unmarked; the counters and the new
// band's box start empty
template <typename T>
__global__ void __launch_bounds__(TPB) k_classify(Geo g, const __grid_constant__ BandSet<T> S) {
  wait_prior();
  __shared__ BandCtx<T> ctx;
  load_ctx(S, ctx);
  const Body& b = ctx.b;
  const T* __restrict__ x = ctx.a.X[S.out];
  int8_t* __restrict__ lay = ctx.a.LAY[S.out];
  if (blockIdx.x == 0) {
    if (threadIdx.x < BAND_COUNTERS) ctx.a.cnt[threadIdx.x] = 0;
    if (threadIdx.x < 6) ctx.a.bb[6 * S.out + threadIdx.x] = threadIdx.x < 3 ? 0x7fffffff : -0x7fffffff;
  }
  const Win w = band_win(g, S, ctx);
  WIN_ROWS(w, row) {
    const WinRow r(g, w, row);
    ROW_CELLS(w, a) {
      const int i = r.x(a);
      const long c = r.base + i;
      const T x0 = x[c], x1 = x[g.N + c], x2 = x[2 * g.N + c];
      int8_t l = -1;
      if (finite_bits(x0) && finite_bits(x1) && finite_bits(x2) && phi_stored_neg(g, b, i, r.j, r.k, x0, x1, x2)) l = 0;
      lay[c] = l;
    }
  }
}

// The band list is sorted by layer: cnt[l] (l = 1..L) counts the cells of layer l, and they sit
// at list[base_l ...], base_l = cnt[1] + ... + cnt[l-1] (the earlier passes have finished).
__device__ __forceinline__ int layer_base(const int* __restrict__ cnt, int l) {
  int b = 0;
  for (int q = 1; q < l; q++) b += cnt[q];
  return b;
}

// unmarked face neighbours of layer l-1 become layer l (walls stop, periodic axes wrap) and are
// appended to layer l's segment of the band list; in place is race-free: only -1 -> l writes,
// and only l-1 is tested
template <typename T>
__global__ void __launch_bounds__(TPB) k_bfs(Geo g, const __grid_constant__ BandSet<T> S, int l) {
  wait_prior();
  __shared__ BandCtx<T> ctx;
  load_ctx(S, ctx);
  int8_t* __restrict__ lay = ctx.a.LAY[S.out];
  int* __restrict__ list = ctx.a.list;
  int* __restrict__ cnt = ctx.a.cnt;
  const Win w = band_win(g, S, ctx);
  const int base = layer_base(cnt, l);
  const int lane = threadIdx.x & 31, plane = g.n[0] * g.n[1];
  WIN_ROWS(w, row) {
    const WinRow r(g, w, row);
    // the four neighbouring rows (-1: beyond a wall)
    const int ym = r.j > 0 ? r.base - g.n[0] : (g.per[1] ? r.base + plane - g.n[0] : -1);
    const int yp = r.j + 1 < g.n[1] ? r.base + g.n[0] : (g.per[1] ? r.base - plane + g.n[0] : -1);
    const int zm = r.k > 0 ? r.base - plane : (g.per[2] ? r.base + (g.n[2] - 1) * plane : -1);
    const int zp = r.k + 1 < g.n[2] ? r.base + plane : (g.per[2] ? r.base - (g.n[2] - 1) * plane : -1);
    for (int a0 = 0; a0 < w.ext[0]; a0 += 32) {
      const int a = a0 + lane;
      bool hit = false;
      int c = 0;
      if (a < w.ext[0]) {
        const int i = r.x(a);
        c = r.base + i;
        if (lay[c] == -1) {
          const int im = i > 0 ? i - 1 : (g.per[0] ? g.n[0] - 1 : -1), ip = i + 1 < g.n[0] ? i + 1 : (g.per[0] ? 0 : -1);
          const int v0 = im >= 0 ? lay[r.base + im] : -1, v1 = ip >= 0 ? lay[r.base + ip] : -1;
          const int v2 = ym >= 0 ? lay[ym + i] : -1, v3 = yp >= 0 ? lay[yp + i] : -1;
          const int v4 = zm >= 0 ? lay[zm + i] : -1, v5 = zp >= 0 ? lay[zp + i] : -1;
          const int m = l - 1;
          hit = v0 == m || v1 == m || v2 == m || v3 == m || v4 == m || v5 == m;
        }
      }
      const unsigned want = __ballot_sync(0xffffffffu, hit);
      if (!want) continue;
      int at = 0;
      if (lane == 0) at = atomicAdd(&cnt[l], __popc(want));  // one counter update per warp and 32 cells
      at = base + __shfl_sync(0xffffffffu, at, 0);
      if (hit) {
        lay[c] = (int8_t)l;
        list[at + __popc(want & ((1u << lane) - 1u))] = c;
      }
    }
  }
}

// LDL^T solve of the 4x4 normal equations, three right-hand sides, in AT; fails (degenerate)
// when a pivot is not above tolfac * trace(A)/4 (tolfac = 1e-12 in FP64)
template <typename AT>
__device__ bool solve4(AT A[4][4], AT B[4][3], AT X[4][3], AT tolfac) {
  AT L[4][4], D[4], iD[4];
  for (int r = 0; r < 4; r++)
    for (int q = 0; q < 4; q++) L[r][q] = AT(0);
  const AT tr = A[0][0] + A[1][1] + A[2][2] + A[3][3];
  const AT tol = tolfac * tr / AT(4);
  for (int k = 0; k < 4; k++) {
    AT s = A[k][k];
    for (int j = 0; j < k; j++) s -= L[k][j] * L[k][j] * D[j];
    D[k] = s;
    if (!(s > tol)) return false;
    iD[k] = AT(1) / s;  // one division per pivot: each is some ten instructions; the rest are quot()s
    L[k][k] = AT(1);
    for (int i = k + 1; i < 4; i++) {
      AT t = A[i][k];
      for (int j = 0; j < k; j++) t -= L[i][j] * L[k][j] * D[j];
      L[i][k] = quot(t, s, iD[k]);
    }
  }
  for (int c = 0; c < 3; c++) {
    AT y[4];
    for (int i = 0; i < 4; i++) {
      AT t = B[i][c];
      for (int j = 0; j < i; j++) t -= L[i][j] * y[j];
      y[i] = t;
    }
    for (int i = 0; i < 4; i++) y[i] = quot(y[i], D[i], iD[i]);
    for (int i = 3; i >= 0; i--) {
      AT t = y[i];
      for (int j = i + 1; j < 4; j++) t -= L[j][i] * X[j][c];
      X[i][c] = t;
    }
  }
  return true;
}

// The candidate cells of the radius-2 search box around one cell, loaded once per cell for
// both fits that use that box (the kernel-only and the normal-weighted one):
// lane L holds the candidates t = L + 32 q (q < 4) of the 5^3 box, a bit per slot that says
// whether the candidate is a cell of a lower layer, and its stored values.  The layer bytes of
// the four slots are read first and the values of the usable ones after them, so a cell costs
// two dependent memory round trips instead of two per slot and fit.
constexpr int RS0 = 2, NC0 = (2 * RS0 + 1) * (2 * RS0 + 1) * (2 * RS0 + 1), NQ0 = (NC0 + 31) / 32;
template <typename T>
struct Cand {
  unsigned ok;
  T v[NQ0][3];
};

template <typename T>
__device__ __forceinline__ void load_cand(const Geo& g, const T* __restrict__ x, const int8_t* __restrict__ lay,
                                          int i, int j, int k, int le, Cand<T>& cd) {
  const int lane = threadIdx.x & 31;
  long cc[NQ0];
  int ld[NQ0];
#pragma unroll
  for (int q = 0; q < NQ0; q++) {
    const int t = lane + 32 * q, w = 2 * RS0 + 1;
    ld[q] = -1;
    cc[q] = 0;
    long c;
    if (t < NC0 && cell_at(g, i + t % w - RS0, j + (t / w) % w - RS0, k + t / (w * w) - RS0, c)) {
      cc[q] = c;
      ld[q] = lay[c];
    }
  }
  cd.ok = 0u;
#pragma unroll
  for (int q = 0; q < NQ0; q++) {
    cd.v[q][0] = cd.v[q][1] = cd.v[q][2] = T(0);
    if (ld[q] >= 0 && ld[q] < le) {
      cd.ok |= 1u << q;
      cd.v[q][0] = x[cc[q]];
      cd.v[q][1] = x[g.N + cc[q]];
      cd.v[q][2] = x[2 * g.N + cc[q]];
    }
  }
}

// One affine WLS fit centred at cell (i,j,k) of layer le with search radius rs, computed by a
// whole warp: the lanes split the (2 rs + 1)^3 candidate cells and the normal-equation sums are
// combined by a butterfly (every lane ends with the same totals, in a fixed order).
// mode 0: kernel 2^-(|di|+|dj|+|dk|); mode 1: times max(0, cos) against the normal n_e.
// The data are the stored values: xi_d (FP64 storage), or the displacements S_d (FP32 storage),
// which the affine model fits exactly as it fits xi (the identity is affine): the fitted values
// are then small, so the solve's error, which scales with the data, carries no O(1) positions
// into the extrapolated maps.  With cd (rs = 2 only) the candidates come from the registers that
// load_cand filled, in the same order, so the sums are the same to the last bit.
template <typename T>
__device__ bool wls_fit_warp(const Geo& g, const T* __restrict__ x, const int8_t* __restrict__ lay, int i, int j,
                             int k, int le, int rs, int mode, const double nrm[3], double sol[4][3],
                             const Cand<T>* cd = nullptr) {
  const int lane = threadIdx.x & 31;
  double a[10], bsum[12];
#pragma unroll
  for (int q = 0; q < 10; q++) a[q] = 0.0;
#pragma unroll
  for (int q = 0; q < 12; q++) bsum[q] = 0.0;
  int npos = 0;
  const int w = 2 * rs + 1, nc = w * w * w;
  // one candidate's contribution; false when its weight is not positive
  auto add = [&](int di, int dj, int dk, T x0, T x1, T x2) {
    const int sr = abs(di) + abs(dj) + abs(dk);
    double wt = ldexp(1.0, -sr);
    if (mode == 1) {
      const double len = sqrt((double)(di * di + dj * dj + dk * dk));
      const double cs = -((double)di * nrm[0] + (double)dj * nrm[1] + (double)dk * nrm[2]) / len;
      wt = cs * wt;
      if (!(wt > 0.0)) return;
    }
    const double v[4] = {1.0, (double)di, (double)dj, (double)dk};
    const double xv[3] = {(double)x0, (double)x1, (double)x2};
    int q = 0;
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
      for (int cc = r; cc < 4; cc++) a[q++] += wt * v[r] * v[cc];
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
      for (int d = 0; d < 3; d++) bsum[3 * r + d] += wt * v[r] * xv[d];
    npos++;
  };
  if (cd) {
#pragma unroll
    for (int q = 0; q < NQ0; q++) {
      if (!(cd->ok >> q & 1u)) continue;
      const int t = lane + 32 * q;
      add(t % w - rs, (t / w) % w - rs, t / (w * w) - rs, cd->v[q][0], cd->v[q][1], cd->v[q][2]);
    }
  } else {
    for (int t = lane; t < nc; t += 32) {
      const int di = t % w - rs, dj = (t / w) % w - rs, dk = t / (w * w) - rs;
      long c;
      if (!cell_at(g, i + di, j + dj, k + dk, c)) continue;
      const int ld = lay[c];
      if (ld < 0 || ld >= le) continue;
      add(di, dj, dk, x[c], x[g.N + c], x[2 * g.N + c]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int q = 0; q < 10; q++) a[q] += __shfl_xor_sync(0xffffffffu, a[q], o);
#pragma unroll
    for (int q = 0; q < 12; q++) bsum[q] += __shfl_xor_sync(0xffffffffu, bsum[q], o);
    npos += __shfl_xor_sync(0xffffffffu, npos, o);
  }
  if (npos < 4) return false;
  double A[4][4], B[4][3];
  int q = 0;
  for (int r = 0; r < 4; r++)
    for (int cc = r; cc < 4; cc++) {
      A[r][cc] = a[q];
      A[cc][r] = a[q];
      q++;
    }
  for (int r = 0; r < 4; r++)
    for (int d = 0; d < 3; d++) B[r][d] = bsum[3 * r + d];
  return solve4<double>(A, B, sol, 1e-12);
}

// A cell whose batched fit failed, fitted again by the whole warp in FP64: the kernel-only fit, then (layers 1 and 2)
// the fit weighted by the normal n_e = normalised (grad xi)^T grad_X phi_0(xi_e) of that first fit; the search radius
// grows up to 4 while the system stays degenerate.  FP32 storage comes here when a system was too ill-conditioned
// for FP32.  Rare, so it is kept out of the callers' registers.  The failed cells of a batch follow one another in their
// warp: with a disk of 0.9 to 4 cells' half-thickness across the grid (64^3 .. 128^3, fits of radius 2 failing along its
// edge or all over it) every extrapolation that succeeds takes 0.3 to 0.7 of its time with a list of failed cells spread
// over all SMs (96^3, tilted, 1.2 cells: 1.77 -> 0.83 ms); one that ends degenerate takes up to 1.55 times as long.
// Returns 1 with the map at the cell in lane 0's out, 0 when degenerate.
template <typename T>
__device__ __noinline__ int wls_again(const Geo& g, const Body& b, const T* x, const int8_t* lay, long c, int le,
                                      double out[3]) {
  int i, j, k;
  decode(c, g.n[0], g.n[1], i, j, k);
  Cand<T> cd;
  load_cand(g, x, lay, i, j, k, le, cd);
  // FP32 storage fits displacements: the identity's slope per cell offset is added back to the
  // fitted gradient, and the cell's x0 - c to the fitted value, where the normal needs xi
  const double hid = disp_storage<T>() ? g.h : 0.0;
  int ok = 0;
  for (int rs = RS0; rs <= 4 && !ok; rs++) {
    const Cand<T>* cp = rs == RS0 ? &cd : nullptr;
    double s1[4][3];
    if (!wls_fit_warp(g, x, lay, i, j, k, le, rs, 0, nullptr, s1, cp)) continue;
    if (le <= 2) {
      double gX[3], v[3];
      if constexpr (disp_storage<T>()) {
        const double r0[3] = {cell_rel<double>(g, b, 0, i) + s1[0][0], cell_rel<double>(g, b, 1, j) + s1[0][1],
                              cell_rel<double>(g, b, 2, k) + s1[0][2]};
        phi0_dir_r<double>(b, r0, gX);
      } else {
        const double c0[3] = {s1[0][0], s1[0][1], s1[0][2]};
        phi0_dir<double>(b, c0, gX);
      }
      for (int q = 0; q < 3; q++)
        v[q] = (s1[1 + q][0] + (q == 0 ? hid : 0.0)) * gX[0] + (s1[1 + q][1] + (q == 1 ? hid : 0.0)) * gX[1] +
               (s1[1 + q][2] + (q == 2 ? hid : 0.0)) * gX[2];
      const double nv = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
      if (!(nv > 0.0)) continue;
      const double nrm[3] = {v[0] / nv, v[1] / nv, v[2] / nv};
      double s2[4][3];
      if (!wls_fit_warp(g, x, lay, i, j, k, le, rs, 1, nrm, s2, cp)) continue;
      for (int d = 0; d < 3; d++) out[d] = s2[0][d];
    } else {
      for (int d = 0; d < 3; d++) out[d] = s1[0][d];
    }
    ok = 1;
  }
  __syncwarp();
  return ok;
}

// ---- batches of cells ------------------------------------------------------------------
// A warp fits up to 32 cells together: cell after cell the lanes sum the normal equations over the 125
// candidates of the radius-2 box, and then every lane solves the 4 x 4 system of a cell of its own, so
// that the solves (some 200 dependent operations each) cost a warp once per batch instead of once
// per cell and fit.  What bounds it is the FP64 pipe (two lanes per SM: a warp instruction takes 16
// cycles) in the FP64 form and instruction issue in the FP32 form, so the sums are cut to what cannot
// be avoided:
//  * the kernel-only fit's weights 2^-(|di|+|dj|+|dk|) and its products with the offsets are exact
//    multiples of 2^-6: its normal matrix is summed in integers (one redux per entry), and the
//    right-hand sides take one FMA per candidate and entry (the weight times the value is exact);
//  * the normal-weighted fit's sums take one FMA each;
//  * sums over the lanes are transposed: at every step a lane hands over half of its partial sums,
//    16 + 8 + 4 + 2 + 1 additions for 22 totals instead of 110, added in the same tree.
// One warp per cell with 66 multiplications and additions per candidate and fit and a solve by all
// lanes took 136 us per layer and body of the 128^3 settling mixture in FP64, and 1.50 ms per
// extrapolation of one body on 96^3 (0.60 now); with it a step of the mixture took 5.5 ms longer.
constexpr int WB = 32;                 // cells of a batch at most
constexpr int NSUM = 22, NPAD = 23;    // totals of a fit, padded against bank conflicts
// 1 / sqrt(s), s = 0 .. 12 (the squared lengths of the 5^3 box's offsets)
__constant__ double INV_SQRT[13] = {0.0,
                                    1.0,
                                    0.70710678118654752440,
                                    0.57735026918962576451,
                                    0.5,
                                    0.44721359549995793928,
                                    0.40824829046386301637,
                                    0.37796447300922722721,
                                    0.35355339059327376220,
                                    0.33333333333333333333,
                                    0.31622776601683793320,
                                    0.30151134457776362265,
                                    0.28867513459481288225};
template <typename AT>
struct WlsShared {
  AT v[TPB / 32][WB][NPAD];
  // per candidate: 2^-sr, and times di, dj, dk; di, dj, dk; 2^-sr / |d| (an integer converted to FP64 per
  // use would occupy the FP64 pipe)
  AT k[NQ0][4][32], d[NQ0][3][32], kl[NQ0][32];
  __device__ void fill() {
    for (int t = threadIdx.x; t < 32 * NQ0; t += blockDim.x) {
      const int q = t >> 5, lane = t & 31, w = 2 * RS0 + 1;
      const int o[3] = {t % w - RS0, (t / w) % w - RS0, t / (w * w) - RS0};
      const float wt = (float)(64 >> min(abs(o[0]) + abs(o[1]) + abs(o[2]), 6)) * (1.0f / 64.0f);
      const int s2 = o[0] * o[0] + o[1] * o[1] + o[2] * o[2];
      k[q][0][lane] = (AT)wt;
      for (int d3 = 0; d3 < 3; d3++) {
        k[q][1 + d3][lane] = (AT)(wt * (float)o[d3]);
        d[q][d3][lane] = (AT)(float)o[d3];
      }
      kl[q][lane] = (AT)wt * (AT)INV_SQRT[s2 <= 12 ? s2 : 0];  // past the box's end: unused
    }
    __syncthreads();
  }
};

// this lane's candidates t = lane + 32 q of the 5^3 box
struct Slots {
  int off[NQ0];        // linear offset from the cell
  signed char d[NQ0][3];
  bool in[NQ0];
};
__device__ __forceinline__ Slots wls_slots(const Geo& g) {
  Slots s;
  const int lane = threadIdx.x & 31, w = 2 * RS0 + 1;
#pragma unroll
  for (int q = 0; q < NQ0; q++) {
    const int t = lane + 32 * q;
    const int di = t % w - RS0, dj = (t / w) % w - RS0, dk = t / (w * w) - RS0;
    s.in[q] = t < NC0;
    s.d[q][0] = (signed char)di;
    s.d[q][1] = (signed char)dj;
    s.d[q][2] = (signed char)dk;
    s.off[q] = di + g.n[0] * (dj + g.n[1] * dk);
  }
  return s;
}
template <typename T>
__device__ __forceinline__ void slot_cand(const Geo& g, const Slots& s, const T* __restrict__ x,
                                          const int8_t* __restrict__ lay, long c, int i, int j, int k, int le,
                                          Cand<T>& cd) {
  long cc[NQ0];
  int ld[NQ0];
  const bool inner = i >= RS0 && i + RS0 < g.n[0] && j >= RS0 && j + RS0 < g.n[1] && k >= RS0 && k + RS0 < g.n[2];
#pragma unroll
  for (int q = 0; q < NQ0; q++) {
    ld[q] = -1;
    cc[q] = c;
    bool in = s.in[q];
    if (inner) cc[q] = c + s.off[q];
    else if (in) in = cell_at(g, i + s.d[q][0], j + s.d[q][1], k + s.d[q][2], cc[q]);
    if (in) ld[q] = lay[cc[q]];
  }
  cd.ok = 0u;
#pragma unroll
  for (int q = 0; q < NQ0; q++) {
    cd.v[q][0] = cd.v[q][1] = cd.v[q][2] = T(0);
    if (ld[q] >= 0 && ld[q] < le) {
      cd.ok |= 1u << q;
      cd.v[q][0] = x[cc[q]];
      cd.v[q][1] = x[g.N + cc[q]];
      cd.v[q][2] = x[2 * g.N + cc[q]];
    }
  }
}

// lane totals: v[q] summed over the warp ends in lane q (32 values) -- or, HALF (16 values), in lanes
// 2 q and 2 q + 1
template <typename AT, bool HALF>
__device__ __forceinline__ AT warp_transpose_sum(AT* v) {
  const int lane = threadIdx.x & 31;
  constexpr int N = HALF ? 8 : 16;
#pragma unroll
  for (int h = N, o = 16; h >= 1; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int q = 0; q < h; q++) {
      const AT give = up ? v[q] : v[q + h];
      const AT keep = up ? v[q + h] : v[q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  if (HALF) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  return v[0];
}

template <typename AT>
__device__ __forceinline__ bool solve_totals(const AT* t, int npos, AT tolfac, AT sol[4][3]) {
  if (npos < 4) return false;
  AT A[4][4], B[4][3];
  int q = 0;
#pragma unroll
  for (int r = 0; r < 4; r++)
#pragma unroll
    for (int c = r; c < 4; c++) {
      A[r][c] = t[q];
      A[c][r] = t[q];
      q++;
    }
#pragma unroll
  for (int r = 0; r < 4; r++)
#pragma unroll
    for (int d = 0; d < 3; d++) B[r][d] = t[10 + 3 * r + d];
  return solve4<AT>(A, B, sol, tolfac);
}

// Fits this lane's cell c (none: c < 0) of layer le together with the other lanes' cells.  Returns 1 with
// out, 0 when the radius-2 system is degenerate or (FP32) too ill-conditioned to trust.
template <typename AT, typename T>
__device__ int wls_batch(const Geo& g, const Body& b, const Slots& sl, WlsShared<AT>& sh, const T* __restrict__ x,
                         const int8_t* __restrict__ lay, long c, int le, AT out[3]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // FP64: the degeneracy threshold; FP32: also the point below which the fit is redone in FP64
  const AT tolfac = sizeof(AT) == 8 ? AT(1e-12) : AT(1e-4);
  const AT hid = disp_storage<T>() ? cv<AT>(g.h, g.f.h) : AT(0);
  int i = 0, j = 0, k = 0;
  if (c >= 0) decode(c, g.n[0], g.n[1], i, j, k);
  const unsigned todo = __ballot_sync(0xffffffffu, c >= 0);
  int npos = 0;
  // kernel-only fit: normal matrix in units of 2^-6
  for (unsigned m = todo; m; m &= m - 1) {
    const int src = __ffs(m) - 1;
    const long cc = __shfl_sync(0xffffffffu, c, src);
    const int ci = __shfl_sync(0xffffffffu, i, src), cj = __shfl_sync(0xffffffffu, j, src), ck = __shfl_sync(0xffffffffu, k, src);
    Cand<T> cd;
    slot_cand(g, sl, x, lay, cc, ci, cj, ck, le, cd);
    int a[10];
    AT bs[16];
#pragma unroll
    for (int q = 0; q < 10; q++) a[q] = 0;
#pragma unroll
    for (int q = 0; q < 16; q++) bs[q] = AT(0);
#pragma unroll
    for (int q = 0; q < NQ0; q++) {
      if (!(cd.ok >> q & 1u)) continue;
      const int di = sl.d[q][0], dj = sl.d[q][1], dk = sl.d[q][2];
      const int w = 64 >> (abs(di) + abs(dj) + abs(dk));
      const int v[4] = {1, di, dj, dk};
      int e = 0;
#pragma unroll
      for (int r = 0; r < 4; r++)
#pragma unroll
        for (int s = r; s < 4; s++) a[e++] += w * v[r] * v[s];
#pragma unroll
      for (int r = 0; r < 4; r++) {
        const AT wv = sh.k[q][r][lane];
#pragma unroll
        for (int d = 0; d < 3; d++) bs[3 * r + d] = fma_any(wv, (AT)cd.v[q][d], bs[3 * r + d]);
      }
    }
    const int np = __reduce_add_sync(0xffffffffu, __popc(cd.ok));
    if (lane == src) npos = np;
#pragma unroll
    for (int q = 0; q < 10; q++) a[q] = __reduce_add_sync(0xffffffffu, a[q]);
    const AT tot = warp_transpose_sum<AT, true>(bs);
    if (lane < 24 && !(lane & 1)) sh.v[warp][src][10 + (lane >> 1)] = tot;
    if (lane == 0) {
#pragma unroll
      for (int q = 0; q < 10; q++) sh.v[warp][src][q] = (AT)((float)a[q] * (1.0f / 64.0f));
    }
  }
  __syncwarp();
  int ok = 0;
  AT s1[4][3], nrm[3] = {AT(0), AT(0), AT(0)};
  if (c >= 0 && solve_totals<AT>(sh.v[warp][lane], npos, tolfac, s1)) {
    ok = 1;
#pragma unroll
    for (int d = 0; d < 3; d++) out[d] = s1[0][d];
    if (le <= 2) {
      // n_e = normalised (grad xi)^T grad_X phi_0(xi_e); FP32 storage: the identity's part added back
      AT gX[3], v[3];
      if constexpr (disp_storage<T>()) {
        const AT r0[3] = {cell_rel<AT>(g, b, 0, i) + s1[0][0], cell_rel<AT>(g, b, 1, j) + s1[0][1],
                          cell_rel<AT>(g, b, 2, k) + s1[0][2]};
        phi0_dir_r<AT>(b, r0, gX);
      } else {
        const AT c0[3] = {s1[0][0], s1[0][1], s1[0][2]};
        phi0_dir<AT>(b, c0, gX);
      }
#pragma unroll
      for (int q = 0; q < 3; q++)
        v[q] = (s1[1 + q][0] + (q == 0 ? hid : AT(0))) * gX[0] + (s1[1 + q][1] + (q == 1 ? hid : AT(0))) * gX[1] +
               (s1[1 + q][2] + (q == 2 ? hid : AT(0))) * gX[2];
      const AT nv = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
      if (nv > AT(0)) {
        const AT in = AT(1) / nv;
#pragma unroll
        for (int q = 0; q < 3; q++) nrm[q] = quot(v[q], nv, in);
      } else {
        ok = 0;
      }
    }
  }
  __syncwarp();  // the totals have been read
  if (le > 2) return ok;
  // the fit weighted by max(0, cos) of the angle to the normal
  for (unsigned m = __ballot_sync(0xffffffffu, ok != 0); m; m &= m - 1) {
    const int src = __ffs(m) - 1;
    const long cc = __shfl_sync(0xffffffffu, c, src);
    const int ci = __shfl_sync(0xffffffffu, i, src), cj = __shfl_sync(0xffffffffu, j, src), ck = __shfl_sync(0xffffffffu, k, src);
    AT n[3];
#pragma unroll
    for (int d = 0; d < 3; d++) n[d] = __shfl_sync(0xffffffffu, nrm[d], src);
    Cand<T> cd;
    slot_cand(g, sl, x, lay, cc, ci, cj, ck, le, cd);
    AT sum[32];
#pragma unroll
    for (int q = 0; q < 32; q++) sum[q] = AT(0);
    int pos = 0;
#pragma unroll
    for (int q = 0; q < NQ0; q++) {
      if (!(cd.ok >> q & 1u)) continue;
      const AT di = sh.d[q][0][lane], dj = sh.d[q][1][lane], dk = sh.d[q][2][lane];
      const AT wt = -(di * n[0] + dj * n[1] + dk * n[2]) * sh.kl[q][lane];
      if (!(wt > AT(0))) continue;
      pos++;
      const AT wv[4] = {wt, wt * di, wt * dj, wt * dk}, v[4] = {AT(1), di, dj, dk};
      int e = 0;
#pragma unroll
      for (int r = 0; r < 4; r++)
#pragma unroll
        for (int s = r; s < 4; s++, e++) sum[e] = s == 0 ? sum[e] + wt : fma_any(wv[r], v[s], sum[e]);
#pragma unroll
      for (int r = 0; r < 4; r++)
#pragma unroll
        for (int d = 0; d < 3; d++) sum[10 + 3 * r + d] = fma_any(wv[r], (AT)cd.v[q][d], sum[10 + 3 * r + d]);
    }
    const int np = __reduce_add_sync(0xffffffffu, pos);
    if (lane == src) npos = np;
    const AT tot = warp_transpose_sum<AT, false>(sum);
    if (lane < NSUM) sh.v[warp][src][lane] = tot;
  }
  __syncwarp();
  if (ok && solve_totals<AT>(sh.v[warp][lane], npos, tolfac, s1)) {
#pragma unroll
    for (int d = 0; d < 3; d++) out[d] = s1[0][d];
  } else {
    ok = 0;
  }
  __syncwarp();  // the totals have been read: the next batch may write
  return ok;
}

// Cells per batch for n cells on the launch's warps.  FP64 fits want fuller batches, since the pipe is
// busy with a few warps an SM: a quarter of the warps (a half: 19.3 ms per step of the 128^3 mixture, a
// quarter 18.9, an eighth 18.7, but 0.62, 0.66 and 0.81 ms per 96^3 extrapolation).  FP32 fits want the
// warps in flight (batches of at least 1, 2, 4, 8: 7.99, 8.11, 8.22, 8.33 ms per 4 steps at 112^3).
template <typename AT>
__device__ __forceinline__ int batch_size(int n, int warps) {
  const int want = sizeof(AT) == 8 ? (warps + 3) / 4 : warps;
  const int g = (n + want - 1) / want;
  return g < 1 ? 1 : (g > WB ? WB : g);
}

// The cells of layer l (its segment of the band list) in the storage type, batch by batch
template <typename T>
__global__ void __launch_bounds__(TPB, sizeof(T) == 4 ? 4 : 2) k_wls(Geo g, const __grid_constant__ BandSet<T> S, int l,
                                                                     int* __restrict__ err) {
  wait_prior();
  __shared__ WlsShared<T> sh;
  __shared__ BandCtx<T> ctx;
  load_ctx(S, ctx);
  const Body& b = ctx.b;
  T* x = ctx.a.X[S.out];
  int8_t* lay = ctx.a.LAY[S.out];
  const int lane = threadIdx.x & 31;
  const int base = layer_base(ctx.a.cnt, l), n = ctx.a.cnt[l];
  const int* list = ctx.a.list + base;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int G = batch_size<T>(n, warps);
  if ((int)blockIdx.x * (TPB / 32) * G >= n) return;
  sh.fill();
  const Slots sl = wls_slots(g);
  for (int e0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * G; e0 < n; e0 += warps * G) {
    const long c = lane < G && e0 + lane < n ? list[e0 + lane] : -1;
    T out[3];
    const int r = wls_batch<T>(g, b, sl, sh, x, lay, c, l, out);
    if (c >= 0 && r) {
      x[c] = out[0];
      x[g.N + c] = out[1];
      x[2 * g.N + c] = out[2];
    }
    for (unsigned m = __ballot_sync(0xffffffffu, c >= 0 && !r); m; m &= m - 1) {
      const long cc = __shfl_sync(0xffffffffu, c, __ffs(m) - 1);
      double o[3];
      const int q = wls_again(g, b, x, lay, cc, l, o);
      if (lane == 0) {
        if (q == 1) {
          x[cc] = (T)o[0];
          x[g.N + cc] = (T)o[1];
          x[2 * g.N + cc] = (T)o[2];
        } else {
          lay[cc] = -1;
          atomicAdd(err, 1);
        }
      }
    }
  }
}

// The end of the extrapolation: phi of the band cells, NaN elsewhere, the band's box (reduced per warp and
// block before it reaches the six global words; shifted so that its minimum lies in [0, n) on a periodic axis
// by the last block); FP32 storage: band cells near the seam of the body's image window are counted in *seam.
// CORR: the corrector xi^{n+1/2} = (xi^n + xi^{n+1})/2 where both exist.
template <typename T, bool CORR>
__global__ void __launch_bounds__(TPB) k_finalize(Geo g, const __grid_constant__ BandSet<T> S, int* __restrict__ seam) {
  wait_prior();
  __shared__ BandCtx<T> ctx;
  __shared__ int box[6];
  if (threadIdx.x < 6) box[threadIdx.x] = threadIdx.x < 3 ? 0x7fffffff : -0x7fffffff;
  load_ctx(S, ctx);
  const Body& b = ctx.b;
  T* __restrict__ x = ctx.a.X[S.out];
  T* __restrict__ phi = ctx.a.PHI[S.out];
  const int8_t* __restrict__ lay = ctx.a.LAY[S.out];
  const T* __restrict__ xo = ctx.a.X[CORR ? S.in : 0];
  const int8_t* __restrict__ layo = ctx.a.LAY[CORR ? S.in : 0];
  T* __restrict__ xh = ctx.a.XH;
  const T nanv = T(__longlong_as_double(0x7ff8000000000000ll));
  int lo[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, hi[3] = {-0x7fffffff, -0x7fffffff, -0x7fffffff};
  const Win w = band_win(g, S, ctx);
  WIN_ROWS(w, row) {
    const WinRow r(g, w, row);
    ROW_CELLS(w, a) {
      const int i = r.x(a);
      const long c = r.base + i;
      if (lay[c] >= 0) {
        lo[0] = min(lo[0], w.lo[0] + a);
        hi[0] = max(hi[0], w.lo[0] + a);
        lo[1] = min(lo[1], r.u1);
        hi[1] = max(hi[1], r.u1);
        lo[2] = min(lo[2], r.u2);
        hi[2] = max(hi[2], r.u2);
        const T x0 = x[c], x1 = x[g.N + c], x2 = x[2 * g.N + c];
        phi[c] = phi_stored(g, b, i, r.j, r.k, x0, x1, x2);
        if (disp_storage<T>() && near_seam(g, b, i, r.j, r.k)) atomicAdd(seam, 1);
        if (CORR) {
          if (layo[c] >= 0) {
            xh[c] = T(0.5) * (xo[c] + x0);
            xh[g.N + c] = T(0.5) * (xo[g.N + c] + x1);
            xh[2 * g.N + c] = T(0.5) * (xo[2 * g.N + c] + x2);
          } else {
            xh[c] = xh[g.N + c] = xh[2 * g.N + c] = nanv;
          }
        }
      } else {
        x[c] = x[g.N + c] = x[2 * g.N + c] = nanv;
        phi[c] = nanv;
        if (CORR) xh[c] = xh[g.N + c] = xh[2 * g.N + c] = nanv;
      }
    }
  }
#pragma unroll
  for (int d = 0; d < 3; d++) {
    lo[d] = __reduce_min_sync(0xffffffffu, lo[d]);
    hi[d] = __reduce_max_sync(0xffffffffu, hi[d]);
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&box[d], lo[d]);
      atomicMax(&box[3 + d], hi[d]);
    }
  }
  __syncthreads();
  int* const bb = ctx.a.bb + 6 * S.out;
  if (threadIdx.x < 3) atomicMin(&bb[threadIdx.x], box[threadIdx.x]);
  else if (threadIdx.x < 6) atomicMax(&bb[threadIdx.x], box[threadIdx.x]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(&ctx.a.cnt[BAND_TICKET], 1) == (int)gridDim.x - 1) {
    __threadfence();
    for (int d = 0; d < 3; d++) {
      const int l0 = ((volatile int*)bb)[d], h0 = ((volatile int*)bb)[3 + d];
      if (!g.per[d] || l0 > h0) continue;
      int q = l0 / g.n[d];
      if (l0 < 0 && l0 % g.n[d]) q -= 1;
      bb[d] = l0 - q * g.n[d];
      bb[3 + d] = h0 - q * g.n[d];
    }
  }
}

// cells new to the band: xi^{n+1/2} by the same WLS from the corrected lower layers (layer l's segment of
// the new band's list).  Few of a segment's cells are new: a warp looks at 32 of them and fits those in
// one batch; where a fit stays degenerate xi^{n+1/2} = xi^{n+1}
template <typename T>
__global__ void __launch_bounds__(TPB, sizeof(T) == 4 ? 4 : 2) k_wls_half(Geo g, const __grid_constant__ BandSet<T> S,
                                                                          int l, int* __restrict__ err) {
  wait_prior();
  __shared__ WlsShared<T> sh;
  __shared__ BandCtx<T> ctx;
  load_ctx(S, ctx);
  const Body& b = ctx.b;
  const int8_t *lay = ctx.a.LAY[S.in], *layn = ctx.a.LAY[S.out];
  const T* xn = ctx.a.X[S.out];
  T* xh = ctx.a.XH;
  const int lane = threadIdx.x & 31;
  const int base = layer_base(ctx.a.cnt, l), n = ctx.a.cnt[l];
  const int* list = ctx.a.list + base;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  if ((int)blockIdx.x * TPB >= n) return;
  sh.fill();
  const Slots sl = wls_slots(g);
  for (int e0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; e0 < n; e0 += warps * 32) {
    long c = e0 + lane < n ? list[e0 + lane] : -1;
    if (c >= 0 && (layn[c] != l || lay[c] >= 0)) c = -1;
    if (!__any_sync(0xffffffffu, c >= 0)) continue;
    T out[3];
    const int r = wls_batch<T>(g, b, sl, sh, xh, layn, c, l, out);
    if (c >= 0 && r) {
      xh[c] = out[0];
      xh[g.N + c] = out[1];
      xh[2 * g.N + c] = out[2];
    }
    for (unsigned m = __ballot_sync(0xffffffffu, c >= 0 && !r); m; m &= m - 1) {
      const long cc = __shfl_sync(0xffffffffu, c, __ffs(m) - 1);
      double o[3];
      const int q = wls_again(g, b, xh, layn, cc, l, o);
      if (lane == 0) {
        if (q == 1) {
          xh[cc] = (T)o[0];
          xh[g.N + cc] = (T)o[1];
          xh[2 * g.N + cc] = (T)o[2];
        } else {
          xh[cc] = xn[cc];
          xh[g.N + cc] = xn[g.N + cc];
          xh[2 * g.N + cc] = xn[2 * g.N + cc];
          atomicAdd(err, 1);
        }
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(TPB) k_phi_half(Geo g, const __grid_constant__ BandSet<T> S) {
  wait_prior();
  __shared__ BandCtx<T> ctx;
  load_ctx(S, ctx);
  const T* __restrict__ xh = ctx.a.XH;
  const int8_t* __restrict__ layn = ctx.a.LAY[S.out];
  T* __restrict__ phih = ctx.a.PHIH;
  const T nanv = T(__longlong_as_double(0x7ff8000000000000ll));
  const Win w = band_win(g, S, ctx);
  WIN_ROWS(w, row) {
    const WinRow r(g, w, row);
    ROW_CELLS(w, a) {
      const int i = r.x(a);
      const long c = r.base + i;
      phih[c] = layn[c] >= 0 ? phi_stored(g, ctx.b, i, r.j, r.k, xh[c], xh[g.N + c], xh[2 * g.N + c]) : nanv;
    }
  }
}

}  // namespace

template <typename T>
void launch_init_xi(const Geo& g, const Body& b, T* x, cudaStream_t s) {
  launch_after(k_init_xi<T>, nblocks(g.N), TPB, 0, s, g, b, x); rmt_count_launches(1);
}

namespace {
template <typename T, bool CORR>
void extrapolate(const Geo& g, const BandSet<T>& S, int blocks, int wls_blocks, int* err, cudaStream_t s) {
  const dim3 gw(blocks, S.count), gf(wls_blocks, S.count);
  launch_after(k_classify<T>, gw, TPB, 0, s, g, S);
  for (int l = 1; l <= g.layers; l++) launch_after(k_bfs<T>, gw, TPB, 0, s, g, S, l);
  for (int l = 1; l <= g.layers; l++) launch_after(k_wls<T>, gf, TPB, 0, s, g, S, l, err);
  launch_after(k_finalize<T, CORR>, gw, TPB, 0, s, g, S, err + 1);
  rmt_count_launches(2 + 2 * g.layers);
}
}  // namespace

template <typename T>
void launch_extrapolate(const Geo& g, const BandSet<T>& S, int blocks, int wls_blocks, int* err, cudaStream_t s) {
  extrapolate<T, false>(g, S, blocks, wls_blocks, err, s);
}

template <typename T>
void launch_extrapolate_correct(const Geo& g, const BandSet<T>& S, int blocks, int wls_blocks, int* err,
                                cudaStream_t s) {
  extrapolate<T, true>(g, S, blocks, wls_blocks, err, s);
  for (int l = 1; l <= g.layers; l++) launch_after(k_wls_half<T>, dim3(wls_blocks, S.count), TPB, 0, s, g, S, l, err);
  launch_after(k_phi_half<T>, dim3(blocks, S.count), TPB, 0, s, g, S);
  rmt_count_launches(1 + g.layers);
}

#define INST(T)                                                                                           \
  template void launch_init_xi<T>(const Geo&, const Body&, T*, cudaStream_t);                              \
  template void launch_extrapolate<T>(const Geo&, const BandSet<T>&, int, int, int*, cudaStream_t);        \
  template void launch_extrapolate_correct<T>(const Geo&, const BandSet<T>&, int, int, int*, cudaStream_t);
INST(float)
INST(double)
