// Predictor of the reference map (arXiv 2104.00095, eq. dis_xi_adv with the Godunov face
// states of eq. xi_taylor_final and the tangential terms of SI "Tangential derivatives"):
// limited slopes of xi, transverse bar states on faces, face states, then the predictor at the
// cells of layers 0 and 1 -- for all bodies in one launch, without scratch.
//
// FP32 storage holds S = xi - x0 (rmt_common.cuh).  The slopes are those of xi (the limiter sees
// differences of xi: h + dS along the component's own axis, dS across it); every face state
// is stored as the displacement from the face centre's image, so where the FP64 form adds a
// Taylor term (h/2) s to xi, the FP32 form adds (h/2)(s - 1) for the component along the
// face's axis, and a difference of face states across a cell gains h on that component.
//
// A block takes tiles of 8^3 cells of a body's window and one component of xi (the components
// meet only in the velocities): it stages the component and the layers with a halo of three
// cells, and slopes, bar states and face states stay in shared memory, 45 KB (FP64 87 KB).
// Kept in memory instead, these 21 words per window cell bound the three passes that each
// body needs, and a body's window leaves most of the chip idle.  The halo repeats about twice
// the slopes of a full tile; the choice of the upwind side before the state is formed, and a
// face's state formed once for both its cells, take half of the states away.  All bodies of a step, three
// passes for each and this: 20 bodies in 128^3 501 -> 170 us (FP64 1333 -> 644 us, bound by its arithmetic),
// 3 in 48^3 81 -> 31 us, 8 in 256^3 327 -> 230 us.
#include "rmt_band.cuh"

namespace {

constexpr int XT = 8;                  // tile width in cells
constexpr int XL = XT + 6;             // with the halo of the staged map and layers
constexpr int XR = XT + 2;             // with one cell around: slopes and bar states
constexpr int XF = (XT + 1) * XT * XT; // faces of one direction
constexpr int XTPB = 256;

struct XiPredPtrs {
  const void* vadv[3];
  const void* unpre[3];
  const void* umac[3];
};

// Shared arrays of a block: s[e], bar[e] at q = x + 1 + XR (y + 1 + XR (z + 1)) the limited slope along e and the
// upwinded bar state on the e-face below tile cell (x, y, z); f[d] the state on the d-faces of the tile; x, lay the
// staged component and layers (-1 beyond a wall).
template <typename T>
struct XiTile {
  T x[XL * XL * XL], s[3][XR * XR * XR], bar[3][XR * XR * XR], f[3][XF];
  int8_t lay[XL * XL * XL];
};
__device__ __forceinline__ int stage_at(int x, int y, int z) { return x + 3 + XL * (y + 3 + XL * (z + 3)); }
__device__ __forceinline__ int ring_at(int x, int y, int z) { return x + 1 + XR * (y + 1 + XR * (z + 1)); }
__device__ __forceinline__ int stage_step(int d) { return d == 0 ? 1 : (d == 1 ? XL : XL * XL); }
__device__ __forceinline__ int ring_step(int d) { return d == 0 ? 1 : (d == 1 ? XR : XR * XR); }

// Taylor state of component a from tile cell v toward its d-face (eq. xi_taylor_final): side 0 the face above
// the cell (L state), side 1 the face below (R state)
template <typename T>
__device__ __forceinline__ T xi_state(const Geo& g, const T* __restrict__ u, const XiPredPtrs& pp, const XiTile<T>& t,
                                      const int org[3], int a, int d, int side, int vx, int vy, int vz) {
  const T h = cv<T>(g.h, g.f.h), dt = cv<T>(g.dt, g.f.dt), ih = cv<T>(g.ih, g.f.ih);
  int i = org[0] + vx, j = org[1] + vy, k = org[2] + vz;
  wrap_axis(g, 0, i);
  wrap_axis(g, 1, j);
  wrap_axis(g, 2, k);
  const int p = stage_at(vx, vy, vz), q = ring_at(vx, vy, vz);
  const T ud = u[d * g.N + cidx(g, i, j, k)];
  T tr = T(0);
#pragma unroll
  for (int e = 0; e < 3; e++) {
    // bar states on the e-faces below and above the cell, where both are formed
    if (e == d || t.lay[p - stage_step(e)] < 0 || t.lay[p + stage_step(e)] < 0) continue;
    const T* va = (const T*)pp.vadv[e];
    const long lo = fidx(g, e, i, j, k), up = fidx(g, e, i + (e == 0), j + (e == 1), k + (e == 2));
    const T vav = T(0.5) * (va[lo] + va[up]);
    tr += vav * (t.bar[e][q + ring_step(e)] - t.bar[e][q]) * ih;
    // FP32 storage: the two bar states are displacements from face centres h apart along e
    if constexpr (disp_storage<T>()) {
      if (a == e) tr += vav;
    }
  }
  const T s = t.s[d][q];
  if constexpr (disp_storage<T>()) {
    // displacement from the face centre's image x0_c +- (h/2) e_d
    const T sg = side == 0 ? T(0.5) * h : -T(0.5) * h;
    return t.x[p] + sg * (s - (a == d ? T(1) : T(0))) - T(0.5) * dt * ud * s - T(0.5) * dt * tr;
  } else {
    const T coef = side == 0 ? (T(0.5) * h - T(0.5) * dt * ud) : -(T(0.5) * h + T(0.5) * dt * ud);
    return t.x[p] + coef * s - T(0.5) * dt * tr;
  }
}

// grid (tiles of a window, bodies, components).  A band cell's neighbours are at most one layer further out, so
// the cells of layers 0 and 1 read states of layers up to 2 and bar states and slopes of layers up to 3.
template <typename T>
__global__ void __launch_bounds__(XTPB) k_xi_predict(Geo g, const T* __restrict__ u,
                                                     const __grid_constant__ XiPredPtrs pp,
                                                     const __grid_constant__ BandSet<T> S) {
  wait_prior();
  extern __shared__ double xi_smem[];
  XiTile<T>& t = *reinterpret_cast<XiTile<T>*>(xi_smem);
  const int m = S.m0 + blockIdx.y, a = blockIdx.z, tid = threadIdx.x;
  const Band<T>& band = S.bands[m];
  const T* __restrict__ x = band.X[S.in] + a * g.N;
  const int8_t* __restrict__ lay = band.LAY[S.in];
  T* __restrict__ xn = band.X[S.out] + a * g.N;
  const Win w = make_win(g, band.bb + 6 * S.in, 2);
  const T h = cv<T>(g.h, g.f.h), dt = cv<T>(g.dt, g.f.dt), ih = cv<T>(g.ih, g.f.ih), tol = cv<T>(g.utol, g.f.utol);
  const T nanv = T(__longlong_as_double(0x7ff8000000000000ll));
  const int n0 = (w.ext[0] + XT - 1) / XT, n1 = (w.ext[1] + XT - 1) / XT, n2 = (w.ext[2] + XT - 1) / XT;
  const int tiles = w.vol > 0 ? n0 * n1 * n2 : 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int o0 = tile % n0 * XT, o1 = tile / n0 % n1 * XT, o2 = tile / (n0 * n1) * XT;
    const int org[3] = {w.lo[0] + o0, w.lo[1] + o1, w.lo[2] + o2};
    // a tile without cells of layers 0 and 1 only gets its NaNs
    bool live = false;
    for (int q = tid; q < XT * XT * XT; q += XTPB) {
      const int vx = q % XT, vy = q / XT % XT, vz = q / (XT * XT);
      if (o0 + vx >= w.ext[0] || o1 + vy >= w.ext[1] || o2 + vz >= w.ext[2]) continue;
      int i = org[0] + vx, j = org[1] + vy, k = org[2] + vz;
      wrap_axis(g, 0, i);
      wrap_axis(g, 1, j);
      wrap_axis(g, 2, k);
      const long c = cidx(g, i, j, k);
      if ((unsigned)lay[c] <= 1u) live = true;
      else xn[c] = nanv;
    }
    if (!__syncthreads_or(live)) continue;  // also: the last tile's reads are done

    for (int r = tid / 16; r < XL * XL; r += XTPB / 16) {
      const int tx = tid % 16;
      if (tx < XL) {
        int i = org[0] + tx - 3, j = org[1] + r % XL - 3, k = org[2] + r / XL - 3;
        int l = -1;
        T v = T(0);
        if (wrap_axis(g, 0, i) && wrap_axis(g, 1, j) && wrap_axis(g, 2, k)) {
          const long c = cidx(g, i, j, k);
          l = lay[c];
          v = x[c];
        }
        t.lay[tx + XL * r] = (int8_t)l;
        t.x[tx + XL * r] = l >= 0 ? v : T(0);
      }
    }
    __syncthreads();

    // limited slopes
    for (int q = tid; q < XR * XR * XR; q += XTPB) {
      const int p = stage_at(q % XR - 1, q / XR % XR - 1, q / (XR * XR) - 1);
      if ((unsigned)t.lay[p] > 3u) continue;
#pragma unroll
      for (int e = 0; e < 3; e++) {
        T v[5];
        unsigned ok = 0;
#pragma unroll
        for (int b = -2; b <= 2; b++) {
          const int pb = p + b * stage_step(e);
          if (t.lay[pb] >= 0) ok |= 1u << (b + 2);
          v[b + 2] = t.x[pb];
          // FP32 storage: the identity's part of xi_e along axis e, relative to the centre cell (the
          // band never pairs cells across the seam of the body's image window)
          if constexpr (disp_storage<T>()) v[b + 2] += a == e ? T(b) * h : T(0);
        }
        t.s[e][q] = lim_slope(v, ok, ih);
      }
    }
    __syncthreads();

    // transverse bar states (SI "Tangential derivatives"), upwinded with the velocity's advecting bar velocity;
    // unavailable on walls and where either cell lacks xi
    for (int q = tid; q < XR * XR * XR; q += XTPB) {
      const int v[3] = {q % XR - 1, q / XR % XR - 1, q / (XR * XR) - 1};
      const int p = stage_at(v[0], v[1], v[2]);
      if ((unsigned)t.lay[p] > 3u) continue;
      int cc[3] = {org[0] + v[0], org[1] + v[1], org[2] + v[2]};
#pragma unroll
      for (int d = 0; d < 3; d++) wrap_axis(g, d, cc[d]);
#pragma unroll
      for (int e = 0; e < 3; e++) {
        const int pD = p - stage_step(e), qD = q - ring_step(e);
        if (v[e] < 0 || (unsigned)t.lay[pD] > 3u) continue;
        int lo[3] = {cc[0], cc[1], cc[2]};
        lo[e] = cc[e] > 0 ? cc[e] - 1 : g.n[e] - 1;
        const T va = ((const T*)pp.vadv[e])[fidx(g, e, cc[0], cc[1], cc[2])];
        T L = T(0), R = T(0);
        if (!(va < -tol)) {
          const T uD = u[e * g.N + cidx(g, lo[0], lo[1], lo[2])], sD = t.s[e][qD];
          if constexpr (disp_storage<T>())  // displacement from the face centre's image x0_D + (h/2) e_e
            L = t.x[pD] + T(0.5) * h * (sD - (a == e ? T(1) : T(0))) - T(0.5) * dt * uD * sD;
          else
            L = t.x[pD] + (T(0.5) * h - T(0.5) * dt * uD) * sD;
        }
        if (!(va > tol)) {
          const T uU = u[e * g.N + cidx(g, cc[0], cc[1], cc[2])], sU = t.s[e][q];
          if constexpr (disp_storage<T>())  // x0_U - (h/2) e_e, the same point
            R = t.x[p] - T(0.5) * h * (sU - (a == e ? T(1) : T(0))) - T(0.5) * dt * uU * sU;
          else
            R = t.x[p] - (T(0.5) * h + T(0.5) * dt * uU) * sU;
        }
        t.bar[e][q] = upwind(L, R, va, tol);
      }
    }
    __syncthreads();

    // face states next to cells of layers 0 and 1
    for (int r = tid; r < 3 * XF; r += XTPB) {
      const int d = r / XF, q = r - d * XF;
      const int m0 = d == 0 ? XT + 1 : XT, m1 = d == 1 ? XT + 1 : XT;
      const int vx = q % m0, vy = q / m0 % m1, vz = q / (m0 * m1);
      const int pU = stage_at(vx, vy, vz), pD = pU - stage_step(d);
      const int lU = t.lay[pU], lD = t.lay[pD];
      if ((unsigned)lU > 1u && (unsigned)lD > 1u) continue;
      const bool both = lU >= 0 && lD >= 0;
      bool needL = lD >= 0, needR = lU >= 0;
      T un = T(0);
      if (both) {
        int i = org[0] + vx, j = org[1] + vy, k = org[2] + vz;
        wrap_axis(g, 0, i);
        wrap_axis(g, 1, j);
        wrap_axis(g, 2, k);
        un = ((const T*)pp.unpre[d])[fidx(g, d, i, j, k)];
        needL = !(un < -tol);
        needR = !(un > tol);
      }
      T L = T(0), R = T(0);
      // one state in the common case, from the cell on its side
      const int side = needL ? 0 : 1;
      const T first = xi_state(g, u, pp, t, org, a, d, side, vx - (side == 0 && d == 0), vy - (side == 0 && d == 1),
                               vz - (side == 0 && d == 2));
      if (needL) L = first;
      else R = first;
      if (needL && needR) R = xi_state(g, u, pp, t, org, a, d, 1, vx, vy, vz);
      t.f[d][q] = both ? upwind(L, R, un, tol) : (lD >= 0 ? L : R);
    }
    __syncthreads();

    // xi^{n+1} = xi^n - dt [(u.grad) xi]^{n+1/2}
    for (int q = tid; q < XT * XT * XT; q += XTPB) {
      const int vx = q % XT, vy = q / XT % XT, vz = q / (XT * XT);
      const int p = stage_at(vx, vy, vz);
      if ((unsigned)t.lay[p] > 1u || o0 + vx >= w.ext[0] || o1 + vy >= w.ext[1] || o2 + vz >= w.ext[2]) continue;
      int i = org[0] + vx, j = org[1] + vy, k = org[2] + vz;
      wrap_axis(g, 0, i);
      wrap_axis(g, 1, j);
      wrap_axis(g, 2, k);
      T acc = T(0);
#pragma unroll
      for (int d = 0; d < 3; d++) {
        const T* U = (const T*)pp.umac[d];
        const long lo = fidx(g, d, i, j, k), up = fidx(g, d, i + (d == 0), j + (d == 1), k + (d == 2));
        const T va = T(0.5) * (U[lo] + U[up]);
        const int f = d == 0 ? vx + (XT + 1) * (vy + XT * vz) : vx + XT * (vy + (d == 1 ? XT + 1 : XT) * vz);
        const int fs = d == 0 ? 1 : (d == 1 ? XT : XT * XT);
        acc += va * (t.f[d][f + fs] - t.f[d][f]) * ih;
        // FP32 storage: the face states are displacements from face centres h apart along d
        if constexpr (disp_storage<T>()) {
          if (a == d) acc += va;
        }
      }
      xn[cidx(g, i, j, k)] = t.x[p] - dt * acc;
    }
  }
}

}  // namespace

template <typename T>
cudaError_t launch_xi_predict(const Geo& g, const T* u, T* const vadv[3], T* const uf[3][3], T* const umac[3],
                              const BandSet<T>& S, int tiles, cudaStream_t s) {
  XiPredPtrs pp;
  for (int d = 0; d < 3; d++) {
    pp.vadv[d] = vadv[d];
    pp.unpre[d] = uf[d][d];
    pp.umac[d] = umac[d];
  }
  const size_t smem = sizeof(XiTile<T>);
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_xi_predict<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  launch_after(k_xi_predict<T>, dim3(tiles, S.count, 3), XTPB, smem, s, g, u, pp, S);
  rmt_count_launches(1);
  return cudaSuccess;
}

#define INST(T)                                                                                                 \
  template cudaError_t launch_xi_predict<T>(const Geo&, const T*, T* const[3], T* const[3][3], T* const[3],     \
                                            const BandSet<T>&, int, cudaStream_t);
INST(float)
INST(double)
