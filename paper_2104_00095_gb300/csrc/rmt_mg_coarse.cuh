// The coarsest multigrid level solved on chip by one thread-block cluster (included by rmt_mg.cu).
//
// Conjugate gradients in FP32 with one reduction per iteration (Chronopoulos & Gear 1989: the two
// inner products r.r and r.Ar are summed together, and A p follows from A r by the same
// recurrence as p), so an iteration is one halo exchange, one operator and one reduction.  A level
// of up to COARSE_ONE unknowns is one block; a larger one is split into slabs of z-planes over a
// cluster of up to 8 blocks, whose boundary planes and partial sums travel through distributed
// shared memory.  Each thread keeps its unknowns' x, r, p and A p in registers; the published
// vector, the face coefficients (7-point; formed once instead of by a division per face and
// iteration) or the cell coefficients (27-point, padded so that the stencil has no branches) sit in
// shared memory.
//
// FP64 levels: FP32 solves inside FP64 refinement.  The FP64 residual of the solution is updated
// as r -= A e with FP64 coefficients and sums until it is 1e-10 of the right-hand side, the
// criterion of an FP64 CG (it ends at 1e-11 to 3e-11, the CG at 3e-11 to 1e-10); three refinements
// replace 20 to 200 FP64 iterations, and GB300 has 2 FP64 lanes per SM against 128 FP32 ones,
// which the one-block FP64 CG was bound by.  A level whose FP32 solves stall on rounding, or that needs
// more iterations than the launch allows, is left above the criterion, as the CG left it at its
// iteration limit; the outer solve measures its own residual.
//
// Bound: the latency chain of an iteration (shared loads, butterfly, barriers; about 0.3 us in one
// block, 1 us in a cluster).  Against the one-block CG that formed its coefficients in every
// iteration, a whole timestep: 32^3 cavity FP64 (4^3 cells, 5^3 nodes) 16.0 -> 9.8 ms, 136 x 120 x
// 128 FP32 (17 x 15 x 16, 18 x 16 x 17) 15.2 -> 8.7 ms, 112^3 FP32 (7^3) 2.9 -> 2.2 ms, 128^3
// settling FP64 36.1 -> 32.2 ms.
#pragma once

constexpr int COARSE_CL = 8;         // largest cluster (the portable limit)
constexpr int COARSE_ONE = 1024;     // unknowns of a single-block solve (FP32)
constexpr int COARSE_ONE64 = 256;    // ... FP64: its operator is bound by one SM's FP64 lanes
constexpr int COARSE_UPT = 8;        // unknowns per thread at most
constexpr int COARSE_WORK = 8;       // FP64: FP32 iterations of all passes together, in units of max_it
// threads of a block: one unknown each up to 1024 (64 registers), else 4 or 8 on 512 (128 registers; the 27-point
// forms of 8 are given 64 and spill some 1.2 KB a thread)
constexpr int COARSE_MAXT = 1024, COARSE_MULTT = 512;

// split of a coarsest level over a cluster
struct CoarseCfg {
  int cs = 0;       // blocks (0: the level is too large for this kernel)
  int planes = 0;   // z-planes of unknowns
  int ps = 0;       // unknowns per plane
  int mcap = 0;     // unknowns of the largest slab
  int tpb = 0, upt = 0;
  size_t smem = 0;
};
__host__ __device__ inline int coarse_k0(int planes, int cs, int rank) { return (int)((long)planes * rank / cs); }

struct CoarseRed {
  double part[2][COARSE_CL][2];  // [parity][block][value]
  double warp[COARSE_MAXT / 32][2];
};

// shared-memory words after CoarseRed: the published float vector with a halo plane on each side,
// then the coefficients as float and (FP64) as double
inline size_t coarse_smem_bytes(int kind, const Lv& L, int ps, int mplanes, size_t esz) {
  const size_t m = (size_t)mplanes * ps;
  const size_t coef = kind == 0 ? 6 * m : (size_t)(mplanes + 1) * (L.n[0] + 2) * (L.n[1] + 2);
  const size_t vec = ((size_t)(mplanes + 2) * ps + 1) & ~(size_t)1;
  return sizeof(CoarseRed) + (vec + ((coef + 1) & ~(size_t)1)) * sizeof(float) + (esz == 8 ? coef * sizeof(double) : 0);
}
inline CoarseCfg coarse_cfg(int kind, const Lv& L, size_t esz) {
  CoarseCfg c;
  const int* ext = kind == 0 ? L.n : L.nn;
  if (L.nunk > (long)COARSE_CL * COARSE_UPT * COARSE_MULTT) return c;
  c.planes = ext[2];
  c.ps = ext[0] * ext[1];
  int cs = 1;
  if (L.nunk > (esz == 8 ? COARSE_ONE64 : COARSE_ONE))
    while (cs < COARSE_CL && 2 * cs <= c.planes) cs *= 2;
  const int mplanes = (c.planes + cs - 1) / cs;
  c.mcap = mplanes * c.ps;
  c.tpb = c.mcap > COARSE_MAXT ? COARSE_MULTT : (c.mcap + 31) / 32 * 32;
  c.upt = (c.mcap + c.tpb - 1) / c.tpb;
  c.smem = coarse_smem_bytes(kind, L, c.ps, mplanes, esz);
  if (c.upt > COARSE_UPT || c.smem > 227 * 1024) return c;  // cs stays 0
  c.upt = c.upt <= 1 ? 1 : (c.upt <= 4 ? 4 : 8);
  c.cs = cs;
  return c;
}

template <typename T, int KIND, int UPT>
__global__ void __launch_bounds__(UPT == 1 ? COARSE_MAXT : COARSE_MULTT)
    k_coarse_solve(Lv L, int cs, int mplanes, int max_it, float tol,
                                                              double tol64, T* __restrict__ gx,
                                                              const T* __restrict__ gb, const T* __restrict__ grho) {
  wait_prior();
  namespace cg = cooperative_groups;
  constexpr bool F64 = sizeof(T) == 8;
  extern __shared__ __align__(16) unsigned char coarse_sm[];
  CoarseRed& red = *reinterpret_cast<CoarseRed*>(coarse_sm);
  const int ex = KIND == 0 ? L.n[0] : L.nn[0], ey = KIND == 0 ? L.n[1] : L.nn[1], ez = KIND == 0 ? L.n[2] : L.nn[2];
  const int ps = ex * ey, t = threadIdx.x, nt = blockDim.x;
  const int rank = blockIdx.x;  // the grid is one cluster
  const int k0 = coarse_k0(ez, cs, rank), np = coarse_k0(ez, cs, rank + 1) - k0, m = np * ps;
  const int mcap = mplanes * ps;
  // 27-point: cell coefficients of cells (i-1, j-1) at (i, j) of an (n0+2) x (n1+2) plane
  const int bw = L.n[0] + 2, bp = bw * (L.n[1] + 2);
  const int ncoef = KIND == 0 ? 6 * mcap : (mplanes + 1) * bp;
  float* const vec = reinterpret_cast<float*>(coarse_sm + sizeof(CoarseRed));
  float* const cf = vec + (((mplanes + 2) * ps + 1) & ~1);
  double* const cd = reinterpret_cast<double*>(cf + ((ncoef + 1) & ~1));
  auto sync_all = [&]() {
    if (cs == 1) __syncthreads();
    else cg::this_cluster().sync();
  };
  // the neighbours' halo planes: the first own plane goes to the block below, the last one above
  float *dlo = nullptr, *dhi = nullptr;
  {
    const int lo = rank > 0 ? rank - 1 : (L.per[2] ? cs - 1 : -1), hi = rank + 1 < cs ? rank + 1 : (L.per[2] ? 0 : -1);
    if (lo >= 0) {
      const int nlo = coarse_k0(ez, cs, lo + 1) - coarse_k0(ez, cs, lo);
      float* v = cs == 1 ? vec : cg::this_cluster().map_shared_rank(vec, lo);
      dlo = v + (nlo + 1) * ps;
    }
    if (hi >= 0) dhi = cs == 1 ? vec : cg::this_cluster().map_shared_rank(vec, hi);
  }
  // zero halo planes (they stay zero beyond a wall) and the coefficients
  for (int q = t; q < ps; q += nt) vec[q] = vec[(np + 1) * ps + q] = 0.f;
  if (KIND == 1) {
    for (int q = t; q < (np + 1) * bp; q += nt) {
      const int i = q % bw, j = (q / bw) % (L.n[1] + 2), k = q / bp;
      const int ci = cnb(L, 0, i - 1), cj = cnb(L, 1, j - 1), ck = cnb(L, 2, k0 + k - 1);
      const T v = ci >= 0 && cj >= 0 && ck >= 0 ? grho[cix(L, ci, cj, ck)] : T(0);
      cf[q] = (float)v;
      if (F64) cd[q] = (double)v;
    }
  }
  // this thread's unknowns: position in vec, in-plane neighbour offsets, coefficient position
  int pos[UPT], xm[UPT], xp[UPT], ym[UPT], yp[UPT], cpos[UPT];
  bool own[UPT], first[UPT], last[UPT];
#pragma unroll
  for (int q = 0; q < UPT; q++) {
    const int e = t + q * nt;
    own[q] = e < m;
    const int ee = own[q] ? e : 0;
    const int lk = ee / ps, rem = ee - lk * ps, j = rem / ex, i = rem - j * ex;
    pos[q] = ee + ps;
    first[q] = own[q] && lk == 0 && dlo;
    last[q] = own[q] && lk == np - 1 && dhi;
    xm[q] = i > 0 ? -1 : (L.per[0] ? ex - 1 : 0);
    xp[q] = i + 1 < ex ? 1 : (L.per[0] ? 1 - ex : 0);
    ym[q] = j > 0 ? -ex : (L.per[1] ? ps - ex : 0);
    yp[q] = j + 1 < ey ? ex : (L.per[1] ? ex - ps : 0);
    cpos[q] = KIND == 0 ? ee : i + bw * j + bp * lk;
    if (KIND == 0 && own[q]) {
      const int k = k0 + lk;
      const T rc = grho[cix(L, i, j, k)];
      const int nb[6][3] = {{i - 1, j, k}, {i + 1, j, k}, {i, j - 1, k}, {i, j + 1, k}, {i, j, k - 1}, {i, j, k + 1}};
#pragma unroll
      for (int f = 0; f < 6; f++) {
        int n3[3] = {i, j, k};
        const int d = f >> 1, v = cnb(L, d, nb[f][d]);
        T beta = T(0);
        if (v >= 0) {
          n3[d] = v;
          beta = face_beta<false>(rc, grho[cix(L, n3[0], n3[1], n3[2])]);
        }
        cf[f * mcap + ee] = (float)beta;
        if (F64) cd[f * mcap + ee] = (double)beta;
      }
    }
  }
  sync_all();  // every block runs, its coefficients and zero halo are in place
  // A v at unknown q of the published vector, coefficients c (float or double)
  auto apply = [&](int q, auto c, auto ctag) {
    using R = decltype(ctag);
    const float* v = vec + pos[q];
    if constexpr (KIND == 0) {
      const R b0 = c[cpos[q]], b1 = c[mcap + cpos[q]], b2 = c[2 * mcap + cpos[q]], b3 = c[3 * mcap + cpos[q]],
              b4 = c[4 * mcap + cpos[q]], b5 = c[5 * mcap + cpos[q]];
      const R off = b0 * (R)v[xm[q]] + b1 * (R)v[xp[q]] + b2 * (R)v[ym[q]] + b3 * (R)v[yp[q]] + b4 * (R)v[-ps] +
                    b5 * (R)v[ps];
      const R dg = ((b0 + b1) + (b2 + b3)) + (b4 + b5);
      return (dg * (R)v[0] - off) * cv<R>(L.ih2, L.f_ih2);
    } else {
      R b[2][2][2];
#pragma unroll
      for (int z = 0; z < 2; z++)
#pragma unroll
        for (int y = 0; y < 2; y++)
#pragma unroll
          for (int x = 0; x < 2; x++) b[x][y][z] = c[cpos[q] + x + y * bw + z * bp];
      const int dx[2] = {xm[q], xp[q]}, dy[2] = {ym[q], yp[q]};
      R s0 = R(0), s1 = R(0), s2 = R(0), s3 = R(0);
#pragma unroll
      for (int z = 0; z < 2; z++) {
        const float* vz = v + (z ? ps : -ps);
#pragma unroll
        for (int y = 0; y < 2; y++) {
          const float* vy = vz + dy[y];
          s0 += b[0][y][z] * (R)vy[dx[0]];
          s1 += b[1][y][z] * (R)vy[dx[1]];
          s2 += (b[0][y][z] + b[1][y][z]) * (R)vy[0];
        }
#pragma unroll
        for (int x = 0; x < 2; x++) s3 += (b[x][0][z] + b[x][1][z]) * (R)vz[dx[x]];
      }
#pragma unroll
      for (int y = 0; y < 2; y++)
#pragma unroll
        for (int x = 0; x < 2; x++) s2 += (b[x][y][0] + b[x][y][1]) * (R)v[dy[y] + dx[x]];
      const R bs = ((b[0][0][0] + b[1][0][0]) + (b[0][1][0] + b[1][1][0])) +
                   ((b[0][0][1] + b[1][0][1]) + (b[0][1][1] + b[1][1][1]));
      return (R(4) * bs * (R)v[0] - ((s0 + s1) + (s2 + s3))) * cv<R>(L.s12, L.f_s12);
    }
  };
  int parity = 0;
  // sums of a and b over the whole cluster, the same bits in every thread: warps in order, then
  // blocks in order
  auto sum2 = [&](auto& a, auto& b) {
    using R = typename std::remove_reference<decltype(a)>::type;
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    const int nw = nt >> 5;
    if (nw == 1 && cs == 1) return;
    R* wr = reinterpret_cast<R*>(&red.warp[0][0]);
    if ((t & 31) == 0) {
      wr[2 * (t >> 5)] = a;
      wr[2 * (t >> 5) + 1] = b;
    }
    __syncthreads();
    // every warp adds the warps' sums the same way
    R x = R(0), y = R(0);
    if ((t & 31) < nw) {
      x = wr[2 * (t & 31)];
      y = wr[2 * (t & 31) + 1];
    }
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if (cs > 1) {
      if (t < cs) {
        double* d = cg::this_cluster().map_shared_rank(&red.part[parity][rank][0], t);
        reinterpret_cast<R*>(d)[0] = x;
        reinterpret_cast<R*>(d)[1] = y;
      }
      cg::this_cluster().sync();
      x = y = R(0);
      for (int c = 0; c < cs; c++) {
        const R* d = reinterpret_cast<const R*>(&red.part[parity][c][0]);
        x += d[0];
        y += d[1];
      }
      parity ^= 1;
    } else {
      __syncthreads();  // the warps' sums are read before the next call writes them
    }
    a = x;
    b = y;
  };
  auto publish = [&](int q, float v) {
    if (!own[q]) return;
    vec[pos[q]] = v;
    const int in = pos[q] - ps;  // first own plane: position in the plane
    if (first[q]) dlo[in] = v;
    if (last[q]) dhi[in - (np - 1) * ps] = v;
  };
  float x[UPT], r[UPT], p[UPT], s[UPT];
  // Scalars' quotients: two of them lie in an iteration's chain.  FP64 levels solve for a residual of norm 1, so the
  // reciprocal neither overflows nor vanishes and the corrected product rounds as a division does (32^3 cavity FP64: 9.55
  // against 9.66 ms); FP32 levels divide, down to the smallest right-hand sides
  auto over = [](float a, float b) { return F64 ? quot(a, b, rcp_approx(b)) : a / b; };
  // FP32 CG of A x = r from x = 0 to the relative residual tol, in at most left iterations; r is used up.  Returns
  // the iterations taken
  auto solve32 = [&](int left) {
    float g = 0.f, dummy = 0.f;
#pragma unroll
    for (int q = 0; q < UPT; q++) {
      x[q] = p[q] = s[q] = 0.f;
      g += r[q] * r[q];
      publish(q, r[q]);
    }
    sum2(g, dummy);
    const float stop = tol * tol * g;
    float gamma = g, alpha = 0.f;
    int it = 0;
    for (; it < left && gamma > stop; it++) {
      if (it > 0) {
#pragma unroll
        for (int q = 0; q < UPT; q++) publish(q, r[q]);
      }
      sync_all();
      float w[UPT], rr = 0.f, rw = 0.f;
#pragma unroll
      for (int q = 0; q < UPT; q++) {
        w[q] = 0.f;
        if (own[q]) w[q] = apply(q, (const float*)cf, 0.f);
        rr += r[q] * r[q];
        rw += r[q] * w[q];
      }
      sum2(rr, rw);
      if (it > 0 && !(rr > stop)) break;
      const float beta = it > 0 ? over(rr, gamma) : 0.f, back = it > 0 ? over(rr, alpha) : 0.f;
      const float den = rw - beta * back;
      if (!(den > 0.f)) break;
      gamma = rr;
      alpha = over(rr, den);
#pragma unroll
      for (int q = 0; q < UPT; q++) {
        p[q] = r[q] + beta * p[q];
        s[q] = w[q] + beta * s[q];
        x[q] += alpha * p[q];
        r[q] -= alpha * s[q];
      }
    }
    return it;
  };
  const long u0 = (long)k0 * ps;
  const double inv_n = 1.0 / (double)L.nunk;
  if constexpr (!F64) {
    float mean = 0.f, xm_ = 0.f, dummy = 0.f;
#pragma unroll
    for (int q = 0; q < UPT; q++) {
      r[q] = own[q] ? gb[u0 + pos[q] - ps] : 0.f;
      mean += r[q];
    }
    sum2(mean, dummy);
    mean *= (float)inv_n;
#pragma unroll
    for (int q = 0; q < UPT; q++) r[q] = own[q] ? r[q] - mean : 0.f;
    solve32(max_it);
    dummy = 0.f;
#pragma unroll
    for (int q = 0; q < UPT; q++) xm_ += x[q];
    sum2(xm_, dummy);
    xm_ *= (float)inv_n;
#pragma unroll
    for (int q = 0; q < UPT; q++)
      if (own[q]) gx[u0 + pos[q] - ps] = x[q] - xm_;
  } else {
    double rd[UPT], xd[UPT], mean = 0.0, dummy = 0.0;
#pragma unroll
    for (int q = 0; q < UPT; q++) {
      rd[q] = own[q] ? gb[u0 + pos[q] - ps] : 0.0;
      xd[q] = 0.0;
      mean += rd[q];
    }
    sum2(mean, dummy);
    mean *= inv_n;
    double rr = 0.0;
    dummy = 0.0;
#pragma unroll
    for (int q = 0; q < UPT; q++) {
      rd[q] = own[q] ? rd[q] - mean : 0.0;
      rr += rd[q] * rd[q];
    }
    sum2(rr, dummy);
    const double stop = tol64 * tol64 * rr;
    // Each pass gains the FP32 solve's factor tol, or what rounding leaves of it: on to the next one while a pass takes
    // a tenth off the residual.  A pass that does not lower the residual is dropped.  COARSE_WORK max_it iterations in
    // all bound the launch.  With a body of 1/1000 to 1000 times the fluid's density, levels of 4^3 to 27^3 cells or
    // nodes (restated on the CPU): the residual is at or below that of an FP64 CG of max_it iterations everywhere, and
    // 1e-10 of the right-hand side up to a ratio of 100 either way on 17 x 15 x 16; 1/1000 ends at 1e-4 .. 3e-3
    // (the FP64 CG at 0.1 .. 0.6).
    for (int left = COARSE_WORK * max_it; left > 0 && rr > stop;) {
      const double nrm = sqrt(rr), inv = 1.0 / nrm;
#pragma unroll
      for (int q = 0; q < UPT; q++) r[q] = (float)(rd[q] * inv);
      left -= max(solve32(left), 1);
      sync_all();  // the last operator has read the published vector
#pragma unroll
      for (int q = 0; q < UPT; q++) publish(q, x[q]);
      sync_all();
      double rn = 0.0;
      dummy = 0.0;
#pragma unroll
      for (int q = 0; q < UPT; q++) {
        if (own[q]) rd[q] -= nrm * apply(q, (const double*)cd, 0.0);
        rn += rd[q] * rd[q];
      }
      sum2(rn, dummy);
      if (!(rn < rr)) break;
#pragma unroll
      for (int q = 0; q < UPT; q++) xd[q] += nrm * (double)x[q];
      if (!(rn < 0.81 * rr)) break;
      rr = rn;
    }
    double xs = 0.0;
    dummy = 0.0;
#pragma unroll
    for (int q = 0; q < UPT; q++) xs += xd[q];
    sum2(xs, dummy);
    xs *= inv_n;
#pragma unroll
    for (int q = 0; q < UPT; q++)
      if (own[q]) gx[u0 + pos[q] - ps] = xd[q] - xs;
  }
  if (cs > 1) cg::this_cluster().sync();  // no block leaves while another may write its memory
}

template <typename T, int KIND>
const void* coarse_fn(int upt) {
  return upt == 1 ? (const void*)k_coarse_solve<T, KIND, 1>
                  : (upt == 4 ? (const void*)k_coarse_solve<T, KIND, 4> : (const void*)k_coarse_solve<T, KIND, 8>);
}
inline const void* coarse_fn(int kind, bool f64, int upt) {
  if (f64) return kind == 0 ? coarse_fn<double, 0>(upt) : coarse_fn<double, 1>(upt);
  return kind == 0 ? coarse_fn<float, 0>(upt) : coarse_fn<float, 1>(upt);
}

template <typename T>
cudaError_t launch_coarse_solve(const CoarseCfg& c, int kind, const Lv& L, int max_it, double tol, T* x, const T* b,
                                const T* rho, cudaStream_t s) {
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at[2];
  lc.gridDim = dim3(c.cs);
  lc.blockDim = dim3(c.tpb);
  lc.dynamicSmemBytes = c.smem;
  lc.stream = s;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_after
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = c.cs;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = c.cs > 1 ? 2 : 1;
  Lv Lk = L;
  int cs = c.cs, mplanes = c.mcap / c.ps, mi = max_it;
  // FP64: FP32 passes of 3e-4; three reach 1e-10 where none of them runs out of iterations
  float tf = sizeof(T) == 8 ? 3e-4f : (float)tol;
  double td = tol;
  void* args[] = {&Lk, &cs, &mplanes, &mi, &tf, &td, &x, (void*)&b, (void*)&rho};
  return cudaLaunchKernelExC(&lc, coarse_fn(kind, sizeof(T) == 8, c.upt), args);
}
