// Godunov face states of the velocity (arXiv 2104.00095, SI "Evaluating the advective term"): limited slopes,
// transverse bar states, cell states and the upwinded normal-face states -- in one pass in FP32, in eight in FP64.
//
// FP32.  Kept in memory, the 36 words per cell between the passes (and their halos) bound the eight kernels.  Here
// a block takes a tile of columns and marches up z: u comes through a ring of five planes in shared memory, what
// is needed across x goes through shuffles (a warp is a row), across y through shared memory, across z through
// registers.  A ring of one column around the tile is computed twice; with it 930 instructions per cell and plane
// bound the kernel (69% of the issue slots, DRAM 11%).  Time of the stage, eight passes and this: 256^3 1419 ->
// 843 us, 128^3 214 -> 141 us (walls 282 -> 149), 48^3 49 -> 23 us.  Blocks of 32 x 8 threads, two to an SM; 32 x 10
// and 32 x 12 (fewer registers) took 3 and 13% longer at 128^3, leaving out what the ring's rows do not need 9%
// (branches in place of one straight run).
#include "rmt_kernels.h"

namespace {

constexpr int GX = 32, GY = 8;             // threads of a block: columns (x, y) with a ring of one around the tile
constexpr int GTX = GX - 2, GTY = GY - 2;  // its own columns
constexpr int GSX = GX + 4, GSY = GY + 4;  // the staged planes of u: two more columns on each side
constexpr int GRING = 5;                   // planes k-1 .. k+3
constexpr int GPC = GSX * GSY, GPL = 3 * GPC;  // a staged plane's component, a staged plane

struct GodOut {
  float* vadv[3];
  float* uf[3][3];
};
struct GodSmem {
  float ring[GRING * GPL];
  float qy[3][GY][GX], ly[3][GY][GX], by[4][GY][GX];
};

// cell coordinate v of axis d folded into the grid: wrapped, mirrored across a wall (face = 1 + 2 d or 2 + 2 d,
// else 0), or, further out than any stencil, clamped
__device__ __forceinline__ int fold(const Geo& g, int d, int v, int& face) {
  const int n = g.n[d];
  face = 0;
  if (v >= 0 && v < n) return v;
  if (g.per[d]) {
    v %= n;
    return v < 0 ? v + n : v;
  }
  face = v < 0 ? 1 + 2 * d : 2 + 2 * d;
  v = v < 0 ? -1 - v : 2 * n - 1 - v;
  return v < 0 ? 0 : (v >= n ? n - 1 : v);
}
__device__ __forceinline__ bool wall_face(const Geo& g, int d, int f) { return !g.per[d] && (f == 0 || f == g.n[d]); }

__global__ void __launch_bounds__(GX* GY, 2)
    k_godunov(Geo g, const float* __restrict__ u, const float* __restrict__ p, const float* __restrict__ rho,
              const float* __restrict__ divtau, const __grid_constant__ GodOut out, const Body* __restrict__ bodies,
              const BodyView<float>* __restrict__ views, int nb, int zc) {
  wait_prior();
  extern __shared__ float god_smem[];
  GodSmem& sm = *reinterpret_cast<GodSmem*>(god_smem);
  const float hh = 0.5f * g.f.h, hdt = 0.5f * g.f.dt, ih = g.f.ih, tol = g.f.utol;
  const int lane = threadIdx.x, ty = threadIdx.y, tid = lane + GX * ty;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2], plane = n0 * n1;
  const long N = g.N;
  const int i = blockIdx.x * GTX - 1 + lane, j = blockIdx.y * GTY - 1 + ty;
  const int k0 = blockIdx.z * zc, k1 = min(k0 + zc, n2 + 1);
  const bool own = lane >= 1 && lane <= GTX && ty >= 1 && ty <= GTY && i <= n0 && j <= n1;
  const bool own_x = own && j < n1, own_y = own && i < n0, own_z = own && i < n0 && j < n1;
  int fc;
  const int ic = fold(g, 0, i, fc), jc = fold(g, 1, j, fc), col = ic + n0 * jc;
  const bool wx = wall_face(g, 0, i), wy = wall_face(g, 1, j);

  // this thread's columns of a staged plane
  constexpr int NS = (GPC + GX * GY - 1) / (GX * GY);
  int scol[NS], sface[NS];
#pragma unroll
  for (int q = 0; q < NS; q++) {
    const int e = tid + q * GX * GY;
    int fx, fy;
    const int vx = fold(g, 0, (int)blockIdx.x * GTX - 3 + e % GSX, fx), vy = fold(g, 1, (int)blockIdx.y * GTY - 3 + e / GSX, fy);
    scol[q] = vx + n0 * vy;
    sface[q] = fx | fy << 4;
  }
  auto load_plane = [&](int k, float v[NS][3]) {
    int fz;
    const int kc = fold(g, 2, k, fz);
#pragma unroll
    for (int q = 0; q < NS; q++) {
      if (tid + q * GX * GY >= GPC) continue;
#pragma unroll
      for (int a = 0; a < 3; a++) v[q][a] = u[a * N + scol[q] + plane * kc];
      const int f = sface[q] | fz << 8;
      if (f) {
        // mirrored ghosts 2 u_wall - u, axis by axis
#pragma unroll
        for (int a = 0; a < 3; a++) {
          float add = 0.f, s = 1.f;
#pragma unroll
          for (int d = 0; d < 3; d++) {
            const int w = (f >> (4 * d) & 15) - 1;
            if (w >= 0) {
              add += s * (2.f * g.f.wall[w][a]);
              s = -s;
            }
          }
          v[q][a] = add + s * v[q][a];
        }
      }
    }
  };
  auto stage = [&](int slot, const float v[NS][3]) {
#pragma unroll
    for (int q = 0; q < NS; q++) {
      const int e = tid + q * GX * GY;
      if (e < GPC) {
#pragma unroll
        for (int a = 0; a < 3; a++) sm.ring[slot + a * GPC + e] = v[q][a];
      }
    }
  };
  // the four pressure nodes of node plane k around this column
  auto nodes = [&](int k, float v[4]) {
    const int kn = g.per[2] ? (k < 0 ? k + n2 : k % n2) : min(max(k, 0), n2);
#pragma unroll
    for (int q = 0; q < 4; q++) v[q] = p[node_at(g, ic + (q & 1), jc + (q >> 1), kn)];
  };
  const int at = lane + 2 + GSX * (ty + 2);
#pragma unroll
  for (int b = 0; b < GRING; b++) {
    float v[NS][3];
    load_plane(k0 - 3 + b, v);
    stage(b * GPL, v);
  }
  float nx[NS][3];
  load_plane(k0 + 2, nx);
  float pn[4];
  nodes(k0 - 1, pn);
  __syncthreads();
  int sl[GRING] = {0, GPL, 2 * GPL, 3 * GPL, 4 * GPL};  // where planes k-2 .. k+2 lie
  // carried from plane to plane: the slopes along z and the limited differences of planes k and k + 1, the z-bar
  // below, the state below along z, the y-state
  float Sz[3], dz[2][3], bz[3] = {}, vz = 0.f, lz[3] = {}, ry[3] = {};
#pragma unroll
  for (int a = 0; a < 3; a++) {
    float q[5];
#pragma unroll
    for (int b = 0; b < 5; b++) q[b] = sm.ring[sl[b] + a * GPC + at];
    const float dm = dflim2(q[0], q[1], q[2]);
    dz[0][a] = dflim2(q[1], q[2], q[3]);
    dz[1][a] = dflim2(q[2], q[3], q[4]);
    Sz[a] = lim_slope4(q[1], q[2], q[3], dm, dz[1][a]) * ih;
  }
  __syncthreads();
  stage(0, nx);
  __syncthreads();

  // faces along y of a plane, from the states below (shared) and above (kept)
  auto faces_y = [&](int m) {
    if (!own_y || m < k0 || m >= n2) return;
    const int f = (int)fidx(g, 1, i, j, m);
    float L[3];
#pragma unroll
    for (int a = 0; a < 3; a++) L[a] = sm.ly[a][ty - 1][lane];
    const float vf = god_normal(L[1], ry[1], tol);
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const float v = a == 1 ? vf : upwind(L[a], ry[a], vf, tol);
      out.uf[1][a][f] = wy ? g.f.wall[j == 0 ? 2 : 3][a] : v;
    }
  };

  for (int k = k0 - 1; k < k1; k++) {
    const int oldest = sl[0];  // its plane, k - 2, was replaced by k + 3
#pragma unroll
    for (int b = 0; b < 4; b++) sl[b] = sl[b + 1];
    sl[4] = oldest;
    if (k + 1 < k1) load_plane(k + 4, nx);
    int fz;
    const int kc = fold(g, 2, k, fz);
    const int c = col + plane * kc;
    float pu[4], F[3], un[3], S[6], cD[3], cU[3], t0[3], t2[3], qU[3], by[3], vy;
    nodes(k + 1, pu);
    const float r = rho[c];
#pragma unroll
    for (int a = 0; a < 3; a++) F[a] = divtau[a * N + c];
    // slopes along x and y of plane k, along z of plane k + 1
    float Szn[3], up[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const float* __restrict__ q0 = sm.ring + sl[1] + a * GPC + at;
      const int o = a * GPC + at;
      const float v0 = q0[0];
      un[a] = v0;
      const float qx[5] = {q0[-2], q0[-1], v0, q0[1], q0[2]};
      S[a] = lim_slope(qx, 0x1Fu, ih);
      const float qy[5] = {q0[-2 * GSX], q0[-GSX], v0, q0[GSX], q0[2 * GSX]};
      S[3 + a] = lim_slope(qy, 0x1Fu, ih);
      const float z1 = sm.ring[sl[2] + o], z2 = sm.ring[sl[3] + o], dn = dflim2(z1, z2, sm.ring[sl[4] + o]);
      Szn[a] = lim_slope4(v0, z1, z2, dz[0][a], dn) * ih;
      dz[0][a] = dz[1][a];
      dz[1][a] = dn;
      up[a] = z1;
    }
#pragma unroll
    for (int d = 0; d < 3; d++) {
      cD[d] = hh - hdt * un[d];
      cU[d] = hh + hdt * un[d];
    }
#pragma unroll
    for (int a = 0; a < 3; a++) sm.qy[a][ty][lane] = un[a] + cD[1] * S[3 + a];
    // z-bar state above the cell, and the term along z
    {
      float bn[3], vn;
      const float cz = hh + hdt * up[2];
      if (wall_face(g, 2, k + 1)) {
        const int w = k + 1 == 0 ? 4 : 5;
#pragma unroll
        for (int a = 0; a < 3; a++) bn[a] = g.f.wall[w][a];
        vn = bn[2];
      } else {
        float qD[3];
#pragma unroll
        for (int a = 0; a < 3; a++) {
          qD[a] = un[a] + cD[2] * Sz[a];
          qU[a] = up[a] - cz * Szn[a];
        }
        vn = god_normal(qD[2], qU[2], tol);
#pragma unroll
        for (int a = 0; a < 3; a++) bn[a] = upwind(qD[a], qU[a], vn, tol);
      }
      if (own_z && k >= k0) out.vadv[2][fidx(g, 2, i, j, k)] = vz;
      const float va = 0.5f * (vz + vn);
#pragma unroll
      for (int a = 0; a < 3; a++) {
        t2[a] = va * (bn[a] - bz[a]) * ih;
        bz[a] = bn[a];
      }
      vz = vn;
    }
    // bar on the x-face below the cell, and the term along x
    {
      float bx[3], vx, qD[3];
#pragma unroll
      for (int a = 0; a < 3; a++) {
        qD[a] = __shfl_up_sync(0xffffffffu, un[a] + cD[0] * S[a], 1);
        qU[a] = un[a] - cU[0] * S[a];
      }
      vx = god_normal(qD[0], qU[0], tol);
#pragma unroll
      for (int a = 0; a < 3; a++) bx[a] = upwind(qD[a], qU[a], vx, tol);
      if (wx) {
        const int w = i == 0 ? 0 : 1;
#pragma unroll
        for (int a = 0; a < 3; a++) bx[a] = g.f.wall[w][a];
        vx = bx[0];
      }
      if (own_x && k >= k0 && k < n2) out.vadv[0][fidx(g, 0, i, j, k)] = vx;
      const float va = 0.5f * (vx + __shfl_down_sync(0xffffffffu, vx, 1));
#pragma unroll
      for (int a = 0; a < 3; a++) t0[a] = va * (__shfl_down_sync(0xffffffffu, bx[a], 1) - bx[a]) * ih;
    }
    __syncthreads();

    faces_y(k - 1);
    // bar on the y-face below the cell
    {
      float qD[3];
#pragma unroll
      for (int a = 0; a < 3; a++) {
        qD[a] = sm.qy[a][ty > 0 ? ty - 1 : 0][lane];
        qU[a] = un[a] - cU[1] * S[3 + a];
      }
      vy = god_normal(qD[1], qU[1], tol);
#pragma unroll
      for (int a = 0; a < 3; a++) by[a] = upwind(qD[a], qU[a], vy, tol);
      if (wy) {
        const int w = j == 0 ? 2 : 3;
#pragma unroll
        for (int a = 0; a < 3; a++) by[a] = g.f.wall[w][a];
        vy = by[1];
      }
#pragma unroll
      for (int a = 0; a < 3; a++) sm.by[a][ty][lane] = by[a];
      sm.by[3][ty][lane] = vy;
      if (own_y && k >= k0 && k < n2) out.vadv[1][fidx(g, 1, i, j, k)] = vy;
    }
    if (k + 1 < k1) stage(sl[0], nx);  // plane k - 1 has been read by all
    __syncthreads();

    // u + dt/(2 rho) F with F = -grad p + div tau + (rho - rho_f) g, the term along y, and the faces
    const int tu = ty < GY - 1 ? ty + 1 : ty;
    const float va = 0.5f * (vy + sm.by[3][tu][lane]);
    float rep[3];
    const bool has_rep = g.any_rep && rep_accel(g, bodies, views, nb, ic, jc, kc, (long)c, rep);
    float gp[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const float pv = q < 4 ? pn[q] : pu[q - 4];
      gp[0] += q & 1 ? pv : -pv;
      gp[1] += q & 2 ? pv : -pv;
      gp[2] += q & 4 ? pv : -pv;
    }
    const float hr = hdt / r;
    float L0[3], R0[3], L2[3], R2[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
      float f = -gp[a] * (0.25f * ih) + F[a] + (r - g.f.rho_f) * g.f.grav[a];
      if (has_rep) f = f + r * rep[a];
      const float t1 = va * (sm.by[a][tu][lane] - by[a]) * ih;
      const float base = un[a] + hr * f;
      const float W0 = base - hdt * (t1 + t2[a]), W1 = base - hdt * (t0[a] + t2[a]), W2 = base - hdt * (t0[a] + t1);
      sm.ly[a][ty][lane] = W1 + cD[1] * S[3 + a];
      ry[a] = W1 - cU[1] * S[3 + a];
      L0[a] = __shfl_up_sync(0xffffffffu, W0 + cD[0] * S[a], 1);
      R0[a] = W0 - cU[0] * S[a];
      L2[a] = lz[a];
      R2[a] = W2 - cU[2] * Sz[a];
      lz[a] = W2 + cD[2] * Sz[a];
      Sz[a] = Szn[a];
    }
    if (own_x && k >= k0 && k < n2) {
      const int f = (int)fidx(g, 0, i, j, k);
      const float vf = god_normal(L0[0], R0[0], tol);
#pragma unroll
      for (int a = 0; a < 3; a++) {
        const float v = a == 0 ? vf : upwind(L0[a], R0[a], vf, tol);
        out.uf[0][a][f] = wx ? g.f.wall[i == 0 ? 0 : 1][a] : v;
      }
    }
    if (own_z && k >= k0) {
      const int f = (int)fidx(g, 2, i, j, k);
      const bool wz = wall_face(g, 2, k);
      const float vf = god_normal(L2[2], R2[2], tol);
#pragma unroll
      for (int a = 0; a < 3; a++) {
        const float v = a == 2 ? vf : upwind(L2[a], R2[a], vf, tol);
        out.uf[2][a][f] = wz ? g.f.wall[k == 0 ? 4 : 5][a] : v;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; q++) pn[q] = pu[q];
  }
  __syncthreads();
  faces_y(k1 - 1);
}

// ---------------------------------------------------------------------------------
// FP64: separate passes.  The FP64 units bound these kernels, and the ring of columns around a tile of the fused
// kernel above costs more there than the passes over memory it saves (walls,
// 128^3: fused 3.69 ms, separate 1.68 ms).

// Limited slopes of the three velocity components along the three axes at every cell
// (SI "Normal derivatives"); S[3 * d + a] = d u_a / d x_d.
struct Slopes9 {
  void* s[9];
};
// One component to a block (grid z: component, chunk of planes).  A thread marches up a column: along z each
// inner limited difference is formed once and serves three slopes.  Ghosts across walls are folded into the
// loads, so that the warps at a wall take the path of the others (128^3 with walls: 0.80 ms, a thread to a cell
// with a separate path at the walls 1.5 ms with the limiters of the time).
__global__ void __launch_bounds__(TILE_X* TILE_Y) k_slopes64(Geo g, const double* __restrict__ u,
                                                             const __grid_constant__ Slopes9 S, int zc, int chunks) {
  wait_prior();
  const int i = blockIdx.x * TILE_X + threadIdx.x, j = blockIdx.y * TILE_Y + threadIdx.y;
  if (i >= g.n[0] || j >= g.n[1]) return;
  const int a = blockIdx.z / chunks, k0 = blockIdx.z % chunks * zc, k1 = min(k0 + zc, g.n[2]);
  const double ih = g.ih;
  const int n0 = g.n[0], plane = n0 * g.n[1], col = i + n0 * j;
  const double* __restrict__ ua = u + a * g.N;
  // the columns of the neighbours -2, -1, 1, 2 along x and y, and the walls they mirror across
  int cx[4], cy[4], fx[4], fy[4];
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int sft = q < 2 ? q - 2 : q - 1;
    cx[q] = fold(g, 0, i + sft, fx[q]) + n0 * j;
    cy[q] = i + n0 * fold(g, 1, j + sft, fy[q]);
  }
  auto ghost = [&](double v, int f) { return f ? 2.0 * g.wall[f - 1][a] - v : v; };
  auto at = [&](int k) {
    int fz;
    const int kc = fold(g, 2, k, fz);
    return ghost(ua[col + (long)plane * kc], fz);
  };
  double zm = at(k0 - 1), z0 = at(k0), zp = at(k0 + 1);
  double dm = dflim2(at(k0 - 2), zm, z0), d0 = dflim2(zm, z0, zp);
  for (int k = k0; k < k1; k++) {
    const long c = col + (long)plane * k;
    const double zpp = at(k + 2);
    const double dp = dflim2(z0, zp, zpp);
    ((double*)S.s[6 + a])[c] = lim_slope4(zm, z0, zp, dm, dp) * ih;
    double q[5];
    q[2] = z0;
#pragma unroll
    for (int b = 0; b < 4; b++) q[b < 2 ? b : b + 1] = ghost(ua[cx[b] + (long)plane * k], fx[b]);
    ((double*)S.s[a])[c] = lim_slope(q, 0x1Fu, ih);
#pragma unroll
    for (int b = 0; b < 4; b++) q[b < 2 ? b : b + 1] = ghost(ua[cy[b] + (long)plane * k], fy[b]);
    ((double*)S.s[3 + a])[c] = lim_slope(q, 0x1Fu, ih);
    zm = z0;
    z0 = zp;
    zp = zpp;
    dm = d0;
    d0 = dp;
  }
}

__device__ __forceinline__ void cell_faces(const Geo& g, int e, int i, int j, int k, long& lo, long& hi) {
  lo = fidx(g, e, i, j, k);
  int ii[3] = {i, j, k};
  ii[e] += 1;
  hi = fidx(g, e, ii[0], ii[1], ii[2]);
}

// transverse bar states at every e-face (SI "Tangential derivatives")
template <int e>
__global__ void __launch_bounds__(TILE_X* TILE_Y) k_bar(Geo g, const double* __restrict__ u, Slopes9 S,
                                                         double* __restrict__ ub0, double* __restrict__ ub1, double* __restrict__ ub2,
                                                         double* __restrict__ vadv) {
  wait_prior();
  const int ex = g.n[0] + (e == 0), ey = g.n[1] + (e == 1), ez = g.n[2] + (e == 2);
  const double h = g.h, dt = g.dt;
  double* ub[3] = {ub0, ub1, ub2};
  THREAD_XYZ(i, j, k);
  if (i >= ex || j >= ey || k >= ez) return;
  const long f = (long)(i + ex * (j + ey * k));
  const int fi = e == 0 ? i : (e == 1 ? j : k);
  if (wall_face(g, e, fi)) {
    const int face = fi == 0 ? 2 * e : 2 * e + 1;
#pragma unroll
    for (int a = 0; a < 3; a++) ub[a][f] = g.wall[face][a];
    vadv[f] = g.wall[face][e];
    return;
  }
  // the two cells of an interior (or periodic) face: D below, U above
  int lo[3] = {i, j, k}, hi[3] = {i, j, k};
  lo[e] -= 1;
  if (lo[e] < 0) lo[e] += g.n[e];
  if (hi[e] >= g.n[e]) hi[e] -= g.n[e];
  const long cD = cidx(g, lo[0], lo[1], lo[2]), cU = cidx(g, hi[0], hi[1], hi[2]);
  const double uD = u[e * g.N + cD], uU = u[e * g.N + cU];
  double qD[3], qU[3];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const double* Sa = (const double*)S.s[3 * e + a];
    qD[a] = u[a * g.N + cD] + (0.5 * h - 0.5 * dt * uD) * Sa[cD];
    qU[a] = u[a * g.N + cU] - (0.5 * h + 0.5 * dt * uU) * Sa[cU];
  }
  const double va = god_normal(qD[e], qU[e], g.utol);
  vadv[f] = va;
#pragma unroll
  for (int a = 0; a < 3; a++) ub[a][f] = upwind(qD[a], qU[a], va, g.utol);
}

struct BarPtrs {
  const void* ub[3][3];
  const void* vadv[3];
  void* uf[3];
};

// Side-independent part of the face states of every cell (eqs. left_final, right_final):
// W[3d+a] = u_a - (dt/2) T_d(u_a) + dt/(2 rho) F_a, with T_d the tangential terms along the two
// axes other than d (SI "Tangential derivatives") and F = -grad p^{n-1/2} + div tau^n + b^n,
// b = (rho - rho_f) g.  A face state is then W + (+-h/2 - dt/2 u_d) * slope.
__global__ void __launch_bounds__(TILE_X* TILE_Y) k_cellw(Geo g, const double* __restrict__ u, const double* __restrict__ p,
                                                           const double* __restrict__ rho, const double* __restrict__ divtau,
                                                           BarPtrs bp, Slopes9 W, const Body* __restrict__ bodies,
                                                           const BodyView<double>* __restrict__ views, int nb) {
  wait_prior();
  THREAD_XYZ(i, j, k);
  if (i >= g.n[0] || j >= g.n[1]) return;
  const double dt = g.dt, ih = g.ih;
  const long c = cidx(g, i, j, k);
  double gp[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int q = 0; q < 8; q++) {
    const int sa = q & 1, sb = (q >> 1) & 1, sc = (q >> 2) & 1;
    const double pv = p[node_at(g, i + sa, j + sb, k + sc)];
    gp[0] += sa ? pv : -pv;
    gp[1] += sb ? pv : -pv;
    gp[2] += sc ? pv : -pv;
  }
  const double r = rho[c];
  // wall repulsion joins b (SI "Contact with a wall"), from phi^n
  double rep[3];
  const bool has_rep = g.any_rep && rep_accel(g, bodies, views, nb, i, j, k, c, rep);
  double vavg[3];
  long lo[3], hi[3];
#pragma unroll
  for (int e = 0; e < 3; e++) {
    cell_faces(g, e, i, j, k, lo[e], hi[e]);
    const double* vad = (const double*)bp.vadv[e];
    vavg[e] = 0.5 * (vad[lo[e]] + vad[hi[e]]);
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    double F = -gp[a] * (0.25 * ih) + divtau[a * g.N + c] + (r - g.rho_f) * g.grav[a];
    if (has_rep) F = F + r * rep[a];
    double term[3];
#pragma unroll
    for (int e = 0; e < 3; e++) {
      const double* ube = (const double*)bp.ub[e][a];
      term[e] = vavg[e] * (ube[hi[e]] - ube[lo[e]]) * ih;
    }
    const double base = u[a * g.N + c] + 0.5 * dt / r * F;
    ((double*)W.s[a])[c] = base - 0.5 * dt * (term[1] + term[2]);
    ((double*)W.s[3 + a])[c] = base - 0.5 * dt * (term[0] + term[2]);
    ((double*)W.s[6 + a])[c] = base - 0.5 * dt * (term[0] + term[1]);
  }
}

// normal-face states of the velocity and the Godunov choice (SI "Godunov-type upwinding")
template <int d>
__global__ void __launch_bounds__(TILE_X* TILE_Y) k_face(Geo g, const double* __restrict__ u, Slopes9 S, Slopes9 W,
                                                          BarPtrs bp) {
  wait_prior();
  const int ex = g.n[0] + (d == 0), ey = g.n[1] + (d == 1), ez = g.n[2] + (d == 2);
  const double h = g.h, dt = g.dt;
  double* uf[3] = {(double*)bp.uf[0], (double*)bp.uf[1], (double*)bp.uf[2]};
  THREAD_XYZ(i, j, k);
  if (i >= ex || j >= ey || k >= ez) return;
  const long f = (long)(i + ex * (j + ey * k));
  const int fi = d == 0 ? i : (d == 1 ? j : k);
  if (wall_face(g, d, fi)) {
    const int face = fi == 0 ? 2 * d : 2 * d + 1;
#pragma unroll
    for (int a = 0; a < 3; a++) uf[a][f] = g.wall[face][a];
    return;
  }
  int lo[3] = {i, j, k}, hi[3] = {i, j, k};
  lo[d] -= 1;
  if (lo[d] < 0) lo[d] += g.n[d];
  if (hi[d] >= g.n[d]) hi[d] -= g.n[d];
  const long cc[2] = {cidx(g, lo[0], lo[1], lo[2]), cidx(g, hi[0], hi[1], hi[2])};
  double st[2][3];
#pragma unroll
  for (int side = 0; side < 2; side++) {
    const long c = cc[side];
    const double ud = u[d * g.N + c];
    const double coef = side == 0 ? (0.5 * h - 0.5 * dt * ud) : -(0.5 * h + 0.5 * dt * ud);
#pragma unroll
    for (int a = 0; a < 3; a++) st[side][a] = ((const double*)W.s[3 * d + a])[c] + coef * ((const double*)S.s[3 * d + a])[c];
  }
  const double un = god_normal(st[0][d], st[1][d], g.utol);
#pragma unroll
  for (int a = 0; a < 3; a++) uf[a][f] = (a == d) ? un : upwind(st[0][a], st[1][a], un, g.utol);
}

}  // namespace

template <>
cudaError_t launch_godunov<float>(const Geo& g, const float* u, const float* p, const float* rho, const float* divtau,
                                  const Body* bodies, const BodyView<float>* views, int nb, float* const vadv[3],
                                  float* const uf[3][3], float* const[9], float* const[9], cudaStream_t s) {
  GodOut o;
  for (int d = 0; d < 3; d++) {
    o.vadv[d] = vadv[d];
    for (int a = 0; a < 3; a++) o.uf[d][a] = uf[d][a];
  }
  const size_t smem = sizeof(GodSmem);
  const cudaError_t e = cudaFuncSetAttribute(k_godunov, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // the number of chunks along z that leaves the least work to the fullest SM: two blocks of an SM at a time,
  // a chunk's planes and about four more to begin and end it
  const int bx = (g.n[0] + GTX) / GTX, by = (g.n[1] + GTY) / GTY, nz = g.n[2] + 1;
  const long slots = 2l * sm_count();
  long best = -1;
  int zc = nz;
  for (int ch = 1; ch <= (nz + 1) / 2; ch++) {
    const int len = (nz + ch - 1) / ch;
    const long blocks = (long)bx * by * ((nz + len - 1) / len), cost = (blocks + slots - 1) / slots * (len + 4);
    if (best < 0 || cost < best) {
      best = cost;
      zc = len;
    }
  }
  launch_after(k_godunov, dim3(bx, by, (nz + zc - 1) / zc), dim3(GX, GY), smem, s, g, u, p, rho, divtau, o, bodies, views, nb, zc);
  rmt_count_launches(1);
  return cudaSuccess;
}

template <>
cudaError_t launch_godunov<double>(const Geo& g, const double* u, const double* p, const double* rho,
                                   const double* divtau, const Body* bodies, const BodyView<double>* views, int nb,
                                   double* const vadv[3], double* const uf[3][3], double* const slopes[9],
                                   double* const wcell[9], cudaStream_t s) {
  Slopes9 S, W;
  BarPtrs bp;
  for (int q = 0; q < 9; q++) {
    S.s[q] = slopes[q];
    W.s[q] = wcell[q];
  }
  const dim3 tile(TILE_X, TILE_Y), gc((g.n[0] + TILE_X - 1) / TILE_X, (g.n[1] + TILE_Y - 1) / TILE_Y, g.n[2]);
  // about 16 blocks to an SM, and no less than eight planes to a chunk where the grid has them
  const int want = (16 * sm_count() + 3 * (int)(gc.x * gc.y) - 1) / (3 * (int)(gc.x * gc.y));
  const int most = (g.n[2] + 7) / 8, chunks = want < most ? want : most, zc = (g.n[2] + chunks - 1) / chunks;
  launch_after(k_slopes64, dim3(gc.x, gc.y, 3 * chunks), tile, 0, s, g, u, S, zc, chunks);
  rmt_count_launches(1);
  auto grid = [&](int d) {
    return dim3((g.n[0] + (d == 0) + TILE_X - 1) / TILE_X, (g.n[1] + (d == 1) + TILE_Y - 1) / TILE_Y, g.n[2] + (d == 2));
  };
  for (int e = 0; e < 3; e++) {
    // the direction is a template argument: a runtime index into the pointer bundles would
    // copy them to local memory in every thread
    auto kb = e == 0 ? k_bar<0> : (e == 1 ? k_bar<1> : k_bar<2>);
    launch_after(kb, grid(e), tile, 0, s, g, u, S, uf[e][0], uf[e][1], uf[e][2], vadv[e]);
    rmt_count_launches(1);
    for (int a = 0; a < 3; a++) bp.ub[e][a] = uf[e][a];  // the bar states give way to the face states
    bp.vadv[e] = vadv[e];
  }
  launch_after(k_cellw, gc, tile, 0, s, g, u, p, rho, divtau, bp, W, bodies, views, nb);
  rmt_count_launches(1);
  for (int d = 0; d < 3; d++) {
    for (int a = 0; a < 3; a++) bp.uf[a] = uf[d][a];
    auto kf = d == 0 ? k_face<0> : (d == 1 ? k_face<1> : k_face<2>);
    launch_after(kf, grid(d), tile, 0, s, g, u, S, W, bp);
    rmt_count_launches(1);
  }
  return cudaGetLastError();
}
