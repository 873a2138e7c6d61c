// ssd_viscous.cuh -- viscous chain of the sliding-mesh SD residual (Sec. 2.1
// viscous fluxes; Sec. 3.1 common solution / common viscous flux on cell
// faces; Sec. 3.2 viscous mortar procedure).  Included by ssd_engine.cuh.
//
// Per stage, after the stage clock and mortar merge:
//   k_faces_cq                 common solution Q_c on conforming faces (average)
//                              and boundaries (the state on the boundary)
//   k_mortar_flux<MORTAR_AVG_Q>  Q_c on the interface: both sides projected
//                              to the mortars, averaged, projected back (summed
//                              into each face by the gradient kernel)
//   k_grad_trace               gradients of the conservative variables at the
//                              SPs (derivative of the degree-N polynomial through
//                              the FP values with Q_c at the end FPs, chain rule
//                              with the SP metrics), stored for k_volume_visc and
//                              interpolated to the faces
//   k_faces_visc               Rusanov + average of both sides' viscous normal
//                              flux evaluated with Q_c (boundaries: boundary state,
//                              interior gradient)
//   k_mortar_flux<MORTAR_RUSANOV_FV>: traces and the viscous normal flux of
//                              both sides projected to the mortars in one pass,
//                              Rusanov + average of the viscous fluxes, projected
//                              back as one sum (summed into each face by the
//                              viscous volume kernel)
//   k_volume_visc              inviscid + viscous fluxes at interior FPs (with
//                              the stored SP gradients), divergence, Runge-Kutta
//                              update, traces; persistent, tiles fed by 1-D
//                              bulk copies one tile ahead
//
// Layout.  On this path the values of a point lie together: the state is
// [E][N^2][4], traces, common solution and common fluxes [E][4 faces][N][4], SP
// gradients [E][2][N^2][4] and gradient traces [E][4][N][8] (x then y).  A point's
// state is one 16-byte access (two in FP64) and two packed FP32x2 operands, where
// one variable at a time took four loads and four FMAs; the kernels here were
// bound by instructions and latency with their tiles in L2, not by bytes.  The
// state crosses the ABI as [E][4][N][N] and is converted with the double-float
// split.  us a step, one variable at a time ->
// points (FP32): 14,752 cells N = 4, five stages 192 -> 152; 20,096 cells N = 5
// 181 -> 164 (the volume kernel's warp instructions 18.2 -> 12.3 million, now
// barrier and shared-load latency with 20 warps per SM).
#pragma once

namespace ssd {

// viscous fluxes of Sec. 2.1 (with the paper's leading minus sign) from Q and
// the physical gradients of the conservative variables; conduct = false drops
// the heat conduction (adiabatic walls)
template <typename T>
__device__ __forceinline__ void viscous_flux(const T *q, const T *qx, const T *qy, const MeshDev &md, T *F, T *G,
                                             bool conduct = true) {
  const T gm1 = pick<T>(md.gm1, md.gm1_f), mu = pick<T>(md.mu, md.mu_f);
  const T kr = conduct ? pick<T>(md.kcR, md.kcR_f) : T(0);  // conductivity / R
  const T ir = recip(q[0]);
  const T u = q[1] * ir, v = q[2] * ir;
  // velocity gradients rounded as products (mul_rn): they are summed with each
  // other below, where an FMA could otherwise take either one
  const T ux = mul_rn(qx[1] - u * qx[0], ir), uy = mul_rn(qy[1] - u * qy[0], ir);
  const T vx = mul_rn(qx[2] - v * qx[0], ir), vy = mul_rn(qy[2] - v * qy[0], ir);
  const T ke = T(0.5) * mul_add(u, u, v, v);
  const T p = gm1 * (q[3] - ke * q[0]);
  const T pr = p * ir;  // R T
  const T px = mul_rn(gm1, qx[3] - fma(u, qx[1], mul_sub(v, qx[2], ke, qx[0])));
  const T py = mul_rn(gm1, qy[3] - fma(u, qy[1], mul_sub(v, qy[2], ke, qy[0])));
  // R grad T = (grad p - R T grad rho) / rho; the heat flux takes k / R
  const T Tx = fma(-pr, qx[0], px) * ir, Ty = fma(-pr, qy[0], py) * ir;
  const T lam = T(-2) / T(3) * mu, dv = ux + vy;
  const T txx = mul_add(T(2) * mu, ux, lam, dv), tyy = mul_add(T(2) * mu, vy, lam, dv), txy = mu * (uy + vx);
  F[0] = 0;
  F[1] = -txx;
  F[2] = -txy;
  F[3] = -fma(u, txx, mul_add(v, txy, kr, Tx));
  G[0] = 0;
  G[1] = -txy;
  G[2] = -tyy;
  G[3] = -fma(u, txy, mul_add(v, tyy, kr, Ty));
}

// The FP64 pipe's way to the same fluxes through a vector (nx, ny): one
// reciprocal, the stress and heat flux taken along the vector first (three
// products where F and G are formed in full: six), no zero component.  Adds the
// viscous flux to f; u, v, ke, pr as viscous_flux forms them.
__device__ __forceinline__ void add_viscous_along(const double *qx, const double *qy, double ir, double u, double v,
                                                  double ke, double pr, const MeshDev &md, double nx, double ny,
                                                  double kr, double *f) {
  const double ux = fma(-u, qx[0], qx[1]) * ir, uy = fma(-u, qy[0], qy[1]) * ir;
  const double vx = fma(-v, qx[0], qx[2]) * ir, vy = fma(-v, qy[0], qy[2]) * ir;
  const double px = md.gm1 * fma(ke, qx[0], fma(-v, qx[2], fma(-u, qx[1], qx[3])));
  const double py = md.gm1 * fma(ke, qy[0], fma(-v, qy[2], fma(-u, qy[1], qy[3])));
  const double Tx = fma(-pr, qx[0], px) * ir, Ty = fma(-pr, qy[0], py) * ir;
  const double l = (-2.0 / 3.0 * md.mu) * (ux + vy), m2 = 2.0 * md.mu;
  const double txx = fma(m2, ux, l), tyy = fma(m2, vy, l), txy = md.mu * (uy + vx);
  const double tx = fma(txx, nx, txy * ny), ty = fma(txy, nx, tyy * ny), qn = fma(Tx, nx, Ty * ny);
  f[1] -= tx;
  f[2] -= ty;
  f[3] = fma(-u, tx, fma(-v, ty, fma(-kr, qn, f[3])));
}

// inviscid ALE and viscous flux through (nx, ny) with vgn = V_g . (nx, ny)
__device__ __forceinline__ void total_flux(const double *q, const double *g8, const MeshDev &md, double nx, double ny,
                                           double vgn, double *f) {
  const double ir = recip(q[0]), u = q[1] * ir, v = q[2] * ir, ke = 0.5 * fma(u, u, v * v);
  const double p = md.gm1 * fma(-ke, q[0], q[3]), un = fma(u, nx, v * ny), w = un - vgn;
  f[0] = q[0] * w;
  f[1] = fma(q[1], w, p * nx);
  f[2] = fma(q[2], w, p * ny);
  f[3] = fma(q[3], w, p * un);
  add_viscous_along(g8, g8 + 4, ir, u, v, ke, p * ir, md, nx, ny, md.kcR, f);
}

// ---- state conversion and traces ----------------------------------------------

// FP64 state [E][4][N^2] -> the points layout (a double-float pair, a float or a
// double per value); thread = one SP
template <typename T, int NN>
__global__ void k_split_points(const double *__restrict__ Q, T *hi, T *lo, int n) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int t = (blockIdx.x * 2 + u) * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const size_t g = (size_t)(t / NN) * 4 * NN + t % NN;
    T h[4], l[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const double x = Q[g + v * NN];
      h[v] = (T)x;
      l[v] = (T)(x - (double)h[v]);
    }
    st4(hi + (size_t)t * 4, h);
    if (lo) st4(lo + (size_t)t * 4, l);
  }
}

template <typename T, int NN>
__global__ void k_join_points(const T *__restrict__ hi, const T *__restrict__ lo, double *Q, int n) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int t = (blockIdx.x * 2 + u) * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const size_t g = (size_t)(t / NN) * 4 * NN + t % NN;
    T h[4], l[4] = {0, 0, 0, 0};
    ld4(hi + (size_t)t * 4, h);
    if (lo) ld4(lo + (size_t)t * 4, l);
#pragma unroll
    for (int v = 0; v < 4; ++v) Q[g + v * NN] = lo ? (double)h[v] + (double)l[v] : (double)h[v];
  }
}

// face traces of a state; thread = one face point
template <typename T, int N>
__global__ void k_trace_points(MeshDev md, const T *__restrict__ Q) {
  pdl_enter();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= md.E * 4 * N) return;
  const int e = t / (4 * N), r = t - e * 4 * N, f = r / N, j = r - f * N;
  const VolBasis<T, N> &B = cVB<T, N>;
  const T *q = Q + (size_t)e * 4 * N * N;
  T acc[4] = {0, 0, 0, 0};
#pragma unroll
  for (int k = 0; k < N; ++k) {
    T v[4];
    ld4(q + 4 * ((f == 0 || f == 2) ? k * N + j : j * N + k), v);
    fma4(acc, (f == 1 || f == 2) ? B.H1[k] : B.H0[k], v);
  }
  st4((T *)md.TR + (size_t)t * 4, acc);
}

// ---- common solution -------------------------------------------------------

template <typename T, int N>
__device__ __forceinline__ void k_face_cq_point(const MeshDev &md, int t) {
  const int fi = t / N, j = t - fi * N;
  const int4 fc = md.faces[fi];
  const int efA = fc.x, efB = fc.y, jB = fc.z ? N - 1 - j : j;
  const T *TR = (const T *)md.TR;
  T *CQ = (T *)md.CQ;
  T a[4], b[4], c[4];
  ld4(TR + ((size_t)efA * N + j) * 4, a);
  ld4(TR + ((size_t)efB * N + jB) * 4, b);
#pragma unroll
  for (int v = 0; v < 4; ++v) c[v] = T(0.5) * (a[v] + b[v]);
  st4(CQ + ((size_t)efA * N + j) * 4, c);
  st4(CQ + ((size_t)efB * N + jB) * 4, c);
}

// boundary faces: the common solution is the state on the boundary
template <typename T, int N, bool OTF>
__device__ __forceinline__ void k_bface_cq_point(const MeshDev &md, int t) {
  const int b = t / N, j = t - b * N;
  const int4 bf = md.bfaces[b];
  const int ef = bf.x;
  const T *TR = (const T *)md.TR;
  T q[4], qg[4], qb[4];
  ld4(TR + ((size_t)ef * N + j) * 4, q);
  T nx, ny, sS, vgn, ug, vg;
  bface_geom<T, N, OTF>(md, b, j, nx, ny, sS, vgn, ug, vg);
  boundary_states(md, bf.y, q, ug, vg, nx, ny, qg, qb);
  st4((T *)md.CQ + ((size_t)ef * N + j) * 4, qb);
}

// common solution at all face points of a stage (conforming, then boundary)
template <typename T, int N, bool OTF>
__global__ void k_faces_cq(MeshDev md) {
  pdl_enter();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < md.nF * N) k_face_cq_point<T, N>(md, t);
  else if (t < (md.nF + md.nB) * N) k_bface_cq_point<T, N, OTF>(md, t - md.nF * N);
}

// ---- gradients ---------------------------------------------------------------

// Elements per block of the viscous kernels (two threads per SP line pair:
// 2 N threads per element).  FP32 N = 5: 161 us a step with 4, 163 with 8 and 16
// (20,096 cells: about one and a half tiles per CTA slot, so small tiles end together).
template <typename T, int N>
struct VisCfg {
  static constexpr bool F = sizeof(T) == 4;
  static constexpr int EPB = N == 3 ? 16 : (N == 4 ? 8 : (N == 5 ? (F ? 4 : 8) : (F ? 8 : 4)));
  static constexpr int THREADS = EPB * 2 * N;
};

// Gradients at the SPs of a tile (thread per SP line, then per SP): on
// return sDx / sDe hold Q_x / Q_y [element][SP][4], and gsp (the tile's rows of
// GSP, [element][2][SP][4]) the same.  The caller synchronises before and after.
template <typename T, int N, bool OTF>
__device__ __forceinline__ void tile_gradients(const MeshDev &md, int e0, int ne, const T *sQ, const T *sCQ, T *sDx,
                                               T *sDe, const T *zt, const int *sEF, const T *sEG, const T *sXs,
                                               T *gsp) {
  constexpr int NN = N * N, NT = VisCfg<T, N>::THREADS;
  const VolBasis<T, N> &B = cVB<T, N>;
  const int le = threadIdx.x / (2 * N);
  const int r = threadIdx.x - le * 2 * N;
  const int d = r / N, m = r - d * N;
  if (le < ne) {
    // the line's N + 1 flux-point values, the common solution at its ends
    T val[N + 1][4], qv[N][4];
    ld4(sCQ + (le * 4 + (d == 0 ? 3 : 0)) * 4 * N + 4 * m, val[0]);
    ld4(sCQ + (le * 4 + (d == 0 ? 1 : 2)) * 4 * N + 4 * m, val[N]);
#pragma unroll
    for (int k = 0; k < N; ++k) ld4(sQ + 4 * (le * NN + (d == 0 ? m * N + k : k * N + m)), qv[k]);
#pragma unroll
    for (int i = 1; i < N; ++i) {
#pragma unroll
      for (int v = 0; v < 4; ++v) val[i][v] = 0;
#pragma unroll
      for (int k = 0; k < N; ++k) fma4(val[i], B.Hf[i * N + k], qv[k]);
    }
    T *o = d == 0 ? sDx : sDe;  // d/dxi at SP (k, m), or d/deta at SP (m, k)
#pragma unroll
    for (int k = 0; k < N; ++k) {
      T acc[4] = {0, 0, 0, 0};
#pragma unroll
      for (int i = 0; i <= N; ++i) fma4(acc, B.Dm[k * (N + 1) + i], val[i]);
      st4(o + 4 * (le * NN + (d == 0 ? m * N + k : k * N + m)), acc);
    }
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < ne * NN; idx += NT) {
    const int l2 = idx / NN, sp = idx - l2 * NN;
    ElemGeo<T, N, OTF> G;
    G.load_rec(md, e0 + l2, sEF[l2], sEG + l2 * 8, zt);
    T xix, xiy, etx, ety, a[4], b[4], gx[4], gy[4];
    G.sp_grad_at(sp, sXs[sp % N], sXs[sp / N], xix, xiy, etx, ety);
    ld4(sDx + 4 * idx, a);
    ld4(sDe + 4 * idx, b);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      gx[v] = mul_add(xix, a[v], etx, b[v]);
      gy[v] = mul_add(xiy, a[v], ety, b[v]);
    }
    st4(sDx + 4 * idx, gx);
    st4(sDe + 4 * idx, gy);
    st4(gsp + (size_t)(l2 * 2 * NN + sp) * 4, gx);
    st4(gsp + (size_t)(l2 * 2 * NN + NN + sp) * 4, gy);
  }
}

// Shared-memory layout of the persistent gradient kernel: two stages of a
// tile's state (4 N^2 values per element) and common solution (16 N), one
// contiguous run each as in global memory; then the gradient arrays.
template <typename T, int N>
struct GradCfg {
  static constexpr int EPB = VisCfg<T, N>::EPB, THREADS = VisCfg<T, N>::THREADS, NN = N * N;
  static constexpr int QE = 4 * NN * (int)sizeof(T), CE = 16 * N * (int)sizeof(T);
  static constexpr int GEE = 8 * (int)sizeof(T);  // bilinear cell record
  static constexpr int O_Q = 0, O_C = O_Q + EPB * QE, O_EG = O_C + EPB * CE, O_EF = O_EG + EPB * GEE;
  static constexpr int STAGE = ((O_EF + EPB * 4) + 127) / 128 * 128;
  static constexpr int O_DX = 2 * STAGE, O_DE = O_DX + EPB * QE;
  static constexpr int O_BAR = ((O_DE + EPB * QE) + 15) / 16 * 16;
  static constexpr int O_XS = O_BAR + 2 * 8;  // the solution points
  static constexpr int SMEM = O_XS + N * (int)sizeof(T);
  static_assert(QE % 16 == 0 && CE % 16 == 0, "bulk-copy sizes and alignment");
  static_assert(SMEM <= 227 * 1024, "dynamic shared memory of one CTA");
};

// SP gradients GSP [E][2][N^2][4] and gradient traces GTR [E][4 faces][N][8]
// (component v = dQ_v/dx, 4 + v = dQ_v/dy).  Persistent: each CTA walks
// tiles; thread 0 issues the next tile's state and common solution (two 1-D
// bulk copies) into the other stage while the CTA computes the current one.
template <typename T, int N, bool OTF, class Src>
__global__ void __launch_bounds__(GradCfg<T, N>::THREADS) k_grad_trace(Src src, int nitems) {
  pdl_enter();
  using C = GradCfg<T, N>;
  constexpr int EPB = C::EPB, NT = C::THREADS, NN = N * N;
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t *bar = (uint64_t *)(smem + C::O_BAR);
  T *sDx = (T *)(smem + C::O_DX), *sDe = (T *)(smem + C::O_DE), *sXs = (T *)(smem + C::O_XS);
  // the state of the stage (the item's case's input state), the common
  // solution, the cell records (on-the-fly path) and flags; the flags are
  // copied in whole groups of 4 (16 bytes), within the tile-padded array
  auto issue = [&](int item, int st) {
    int cn, tl;
    src.item(item, cn, tl);
    const MeshDev &mn = src.mesh(cn);
    const T *Q = (const T *)src.args(cn).in.hi;
    unsigned char *sb = smem + st * C::STAGE;
    if (!batch_check(mn, tl >= 0 && tl * EPB < mn.E)) {
      mbar_expect_tx(&bar[st], 0);  // a work item outside its case: nothing copied
      return;
    }
    const size_t e0 = (size_t)tl * EPB;
    const uint32_t ne = (uint32_t)min(EPB, mn.E - (int)e0), nf = (ne + 3u) & ~3u;
    mbar_expect_tx(&bar[st], ne * (C::QE + C::CE + (OTF ? C::GEE : 0)) + nf * 4u);
    bulk_g2s(sb + C::O_Q, Q + e0 * 4 * NN, ne * C::QE, &bar[st]);
    bulk_g2s(sb + C::O_C, (const T *)mn.CQ + e0 * 16 * N, ne * C::CE, &bar[st]);
    if (OTF) bulk_g2s(sb + C::O_EG, (const T *)mn.egeo + e0 * 8, ne * C::GEE, &bar[st]);
    bulk_g2s(sb + C::O_EF, mn.eflag + e0, nf * 4u, &bar[st]);
  };
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_mbar_init();
  }
  __syncthreads();
  int item = blockIdx.x;
  if (threadIdx.x == 0 && item < nitems) issue(item, 0);
  const VolBasis<T, N> &B = cVB<T, N>;
  if (threadIdx.x < N) sXs[threadIdx.x] = B.Xs[threadIdx.x];  // (read after the first barrier below)
  const int le = threadIdx.x / (2 * N);
  const int r = threadIdx.x - le * 2 * N;
  const int d = r / N, m = r - d * N;
  int it = 0;
  for (; item < nitems; item += gridDim.x, ++it) {
    const int st = it & 1;
    const int next = item + gridDim.x;
    int cs, tile;
    src.item(item, cs, tile);
    const MeshDev &md = src.mesh(cs);
    const T *zt = zone_tab<T>(md.clk);
    if (threadIdx.x == 0 && next < nitems) {
      fence_proxy_async_smem();
      issue(next, st ^ 1);
    }
    if (!cta_wait(&bar[st], (uint32_t)((it >> 1) & 1))) {
      if (threadIdx.x == 0) {
        atomicOr(&md.clk->flags, 4);
        if (next < nitems) mbar_wait_bounded(&bar[st ^ 1], (uint32_t)(((it + 1) >> 1) & 1));
      }
      return;
    }
    unsigned char *sb = smem + st * C::STAGE;
    const T *sQ = (const T *)(sb + C::O_Q), *sCQ = (const T *)(sb + C::O_C);
    const T *sEG = (const T *)(sb + C::O_EG);
    const int *sEF = (const int *)(sb + C::O_EF);
    const int e0 = tile * EPB;
    const int ne = min(EPB, md.E - e0);
    // the tile's interface faces: their common solution from the mortar
    // contributions, also into CQ for the viscous mortar pass that follows
    if (gather_tile<T, N, GATHER_Q, LAY_POINTS>(md, e0, ne, sEF, (T *)(sb + C::O_C), 16 * N, true, NT)) __syncthreads();
    // the SP gradients, also stored for the volume kernel of this stage
    tile_gradients<T, N, OTF>(md, e0, ne, sQ, sCQ, sDx, sDe, zt, sEF, sEG, sXs, (T *)md.GSP + (size_t)e0 * 8 * NN);
    __syncthreads();
    if (le < ne) {
      T *g = (T *)md.GTR + (size_t)(e0 + le) * 32 * N + 8 * m;
      const int fa = d == 0 ? 3 : 0, fb = d == 0 ? 1 : 2;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        T a0[4] = {0, 0, 0, 0}, a1[4] = {0, 0, 0, 0};
#pragma unroll
        for (int k = 0; k < N; ++k) {
          T val[4];
          ld4((c ? sDe : sDx) + 4 * (le * NN + (d == 0 ? m * N + k : k * N + m)), val);
          fma4(a0, B.H0[k], val);
          fma4(a1, B.H1[k], val);
        }
        st4(g + fa * 8 * N + 4 * c, a0);
        st4(g + fb * 8 * N + 4 * c, a1);
      }
    }
    // every read of this tile's stage and of the gradient arrays is done
    // before they are refilled
    __syncthreads();
  }
}

// ---- common fluxes -------------------------------------------------------------

// normal viscous flux F_vis . n from Q and the 8 gradient components
template <typename T>
__device__ __forceinline__ void viscous_normal(const T *q, const T *g8, T nx, T ny, const MeshDev &md, T *fn,
                                               bool conduct = true) {
  if constexpr (std::is_same<T, double>::value) {
    const T ir = recip(q[0]), u = q[1] * ir, v = q[2] * ir, ke = T(0.5) * fma(u, u, v * v);
    const T pr = md.gm1 * fma(-ke, q[0], q[3]) * ir;
    fn[0] = fn[1] = fn[2] = fn[3] = T(0);
    add_viscous_along(g8, g8 + 4, ir, u, v, ke, pr, md, nx, ny, conduct ? md.kcR : 0.0, fn);
  } else {
    T F[4], G[4];
    viscous_flux(q, g8, g8 + 4, md, F, G, conduct);
#pragma unroll
    for (int v = 0; v < 4; ++v) fn[v] = mul_add(F[v], nx, G[v], ny);
  }
}

template <typename T, int N>
__device__ __forceinline__ void k_face_visc_point(const MeshDev &md, int t) {
  const int fi = t / N, j = t - fi * N;
  const int4 fc = md.faces[fi];
  const int efA = fc.x, efB = fc.y, jB = fc.z ? N - 1 - j : j;
  const T *TR = (const T *)md.TR, *CQ = (const T *)md.CQ, *GT = (const T *)md.GTR;
  T qA[4], qB[4], qc[4], gA[8], gB[8];
  const size_t pA = (size_t)efA * N + j, pB = (size_t)efB * N + jB;
  ld4(TR + pA * 4, qA);
  ld4(TR + pB * 4, qB);
  ld4(CQ + pA * 4, qc);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    ld4(GT + pA * 8 + 4 * h, gA + 4 * h);
    ld4(GT + pB * 8 + 4 * h, gB + 4 * h);
  }
  const T *g = (const T *)md.fgeo + (size_t)fi * 5 * N;
  T nx = g[j], ny = g[N + j];
  const T sA = g[2 * N + j], sB = g[3 * N + j], vgn = g[4 * N + j];
  const int z = md.eflag[efA >> 2] & kZoneMask;
  if (z) {
    const T *zt = zone_tab<T>(md.clk);
    const T c = zt[z], s = zt[kZT + z];
    const T rx = mul_sub(c, nx, s, ny), ry = mul_add(s, nx, c, ny);
    nx = rx;
    ny = ry;
  }
  T Fn[4], va[4], vb[4];
  rusanov(qA, qB, nx, ny, vgn, pick<T>(md.gamma, md.gamma_f), Fn);
  viscous_normal(qc, gA, nx, ny, md, va);
  viscous_normal(qc, gB, nx, ny, md, vb);
  T *CF = (T *)md.CF;
  T fA[4], fB[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const T f = Fn[v] + T(0.5) * (va[v] + vb[v]);
    fA[v] = sA * f;
    fB[v] = -sB * f;
  }
  st4(CF + pA * 4, fA);
  st4(CF + pB * 4, fB);
}

// boundary faces: Rusanov through the ghost state plus the viscous flux of the
// boundary state with the interior gradient
template <typename T, int N, bool OTF>
__device__ __forceinline__ void k_bface_visc_point(const MeshDev &md, int t) {
  const int b = t / N, j = t - b * N;
  const int4 bf = md.bfaces[b];
  const int ef = bf.x;
  const T *TR = (const T *)md.TR, *GT = (const T *)md.GTR;
  T q[4], qg[4], qb[4], g8[8];
  ld4(TR + ((size_t)ef * N + j) * 4, q);
#pragma unroll
  for (int h = 0; h < 2; ++h) ld4(GT + ((size_t)ef * N + j) * 8 + 4 * h, g8 + 4 * h);
  T nx, ny, sS, vgn, ug, vg;
  bface_geom<T, N, OTF>(md, b, j, nx, ny, sS, vgn, ug, vg);
  boundary_states(md, bf.y, q, ug, vg, nx, ny, qg, qb);
  T Fn[4], fv[4];
  rusanov(q, qg, nx, ny, vgn, pick<T>(md.gamma, md.gamma_f), Fn);
  viscous_normal(qb, g8, nx, ny, md, fv, bf.y != SD_BC_ADIABATIC);
  T *CF = (T *)md.CF;
#pragma unroll
  for (int v = 0; v < 4; ++v) Fn[v] = sS * (Fn[v] + fv[v]);
  st4(CF + ((size_t)ef * N + j) * 4, Fn);
}

// common inviscid + viscous fluxes at all face points of a stage
template <typename T, int N, bool OTF>
__global__ void k_faces_visc(MeshDev md) {
  pdl_enter();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < md.nF * N) k_face_visc_point<T, N>(md, t);
  else if (t < (md.nF + md.nB) * N) k_bface_visc_point<T, N, OTF>(md, t - md.nF * N);
}

// ---- volume ------------------------------------------------------------------

// Shared-memory layout of the persistent viscous volume kernel: two stages of
// a tile's state (4 N^2 values per element), SP gradients (8 N^2: x then y)
// and common fluxes (16 N), each one contiguous run as in global memory, so a
// tile arrives by three 1-D bulk copies; then the tile's transformed fluxes at
// the interior flux points and the interpolation / derivative weights.  One
// thread per interior flux point of every SP line of the tile: 2 N (N - 1)
// threads per element, so that a CTA holds few elements and many threads.
template <typename T, int N>
struct VisVolCfg {
  // elements per tile (FP32 N = 4: 149 us a step with 4, 151 with 8, 163 with 16
  // on 14,752 cells, five stages; N = 5: 163 with 4, 172 with 8 on 20,096 cells)
  static constexpr int EPB = N == 3 ? 16 : (N == 4 && sizeof(T) == 8 ? 8 : 4);
  static constexpr int NN = N * N, LINES = EPB * 2 * N, THREADS = LINES * (N - 1);
  static constexpr int QE = 4 * NN * (int)sizeof(T), GE = 8 * NN * (int)sizeof(T), CE = 16 * N * (int)sizeof(T);
  static constexpr int GEE = 8 * (int)sizeof(T);  // bilinear cell record
  static constexpr int O_Q = 0, O_G = O_Q + EPB * QE, O_C = O_G + EPB * GE, O_EG = O_C + EPB * CE;
  static constexpr int O_EF = O_EG + EPB * GEE;
  static constexpr int STAGE = ((O_EF + EPB * 4) + 127) / 128 * 128;
  // fluxes [EPB][2 directions][N lines][LS]: a line's N - 1 interior points,
  // 4 values each; a stride of an odd number of points puts eight neighbouring
  // lines in different banks
  static constexpr int LS = 4 * ((N - 1) | 1);
  static constexpr int O_FL = 2 * STAGE;
  static constexpr int O_W = O_FL + (EPB * 2 * N * LS * (int)sizeof(T) + 15) / 16 * 16;  // Hf, Dm, Xs, Xf
  static constexpr int O_BAR = (O_W + (2 * N * (N + 1) + 2 * N + 1) * (int)sizeof(T) + 15) / 16 * 16;
  static constexpr int SMEM = O_BAR + 2 * 8;
  static_assert(QE % 16 == 0 && GE % 16 == 0 && CE % 16 == 0, "bulk-copy sizes and alignment");
  static_assert(SMEM <= 227 * 1024 && THREADS <= 1024, "one CTA");
  // resident CTAs per SM the register budget is set for (warps per SM), or what
  // the shared memory admits.  us for 16 / 20 / 25 / 32 warps, FP32, three steps of
  // the 20,096-cell ellipse: N = 3 304 / 285 / 282 / 283, N = 4 358 / 352 / 344 / 336,
  // N = 5 546 / 518 / 518 / 550, N = 6 767 / 767 / 708 / 745; of a 10,368-cell
  // Couette gap N = 3 241 / 229 / 236 / 236, N = 6 474 / 474 / 448 / 484; two
  // five-stage steps of the 14,752-cell tank at N = 4 352 / 336 / 320 / 322; 288
  // cells at N = 3, one step 55.7 / 55.8 / 56.4 / 60.0.  FP64, one step of the
  // ellipse: within 0.6 % of each other at every N.
  static constexpr int WARPS = (THREADS + 31) / 32;
  static constexpr int BUDGET = sizeof(T) == 4 ? (N == 4 || N == 6 ? 25 : 20) : 16;
  static constexpr int BY_WARPS = BUDGET / WARPS > 0 ? BUDGET / WARPS : 1;
  static constexpr int BY_SMEM = 228 * 1024 / (SMEM + 1024);
  static constexpr int MINB = BY_WARPS < BY_SMEM ? BY_WARPS : (BY_SMEM > 0 ? BY_SMEM : 1);
};

// Inviscid + viscous fluxes at the interior FPs with the stored SP gradients,
// common fluxes at the end FPs, divergence, Runge-Kutta stage, traces.
// Persistent: each CTA walks tiles of EPB elements; thread 0 issues the next
// tile's three bulk copies into the other stage while the CTA computes the
// current one.  Every wait is bounded (device flag bit 2 on timeout).
template <typename T, int N, int MODE, bool OTF, bool LO, class Src>
__global__ void __launch_bounds__(VisVolCfg<T, N>::THREADS, VisVolCfg<T, N>::MINB)
    k_volume_visc(Src src, int nitems) {
  pdl_enter();
  using C = VisVolCfg<T, N>;
  constexpr int EPB = C::EPB, NT = C::THREADS, NN = N * N;
  constexpr bool FF = std::is_same<T, float>::value;
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t *bar = (uint64_t *)(smem + C::O_BAR);
  T *sFl = (T *)(smem + C::O_FL);
  T *sHf = (T *)(smem + C::O_W), *sDm = sHf + (N + 1) * N, *sXs = sDm + (N + 1) * N, *sXf = sXs + N;
  const VolBasis<T, N> &B = cVB<T, N>;
  // the state, the SP gradients that k_grad_trace formed from it in this
  // stage, and the common fluxes of tile tl into stage st
  // with the cell records (on-the-fly path) and flags, the flags in whole
  // groups of 4 (16 bytes), within the tile-padded array
  auto issue = [&](int item, int st) {
    int cn, tl;
    src.item(item, cn, tl);
    const MeshDev &mn = src.mesh(cn);
    unsigned char *sb = smem + st * C::STAGE;
    if (!batch_check(mn, tl >= 0 && tl * EPB < mn.E)) {
      mbar_expect_tx(&bar[st], 0);  // a work item outside its case: nothing copied
      return;
    }
    const size_t e0 = (size_t)tl * EPB;
    const uint32_t ne = (uint32_t)min(EPB, mn.E - (int)e0), nf = (ne + 3u) & ~3u;
    mbar_expect_tx(&bar[st], ne * (C::QE + C::GE + C::CE + (OTF ? C::GEE : 0)) + nf * 4u);
    bulk_g2s(sb + C::O_Q, (const T *)src.args(cn).in.hi + e0 * 4 * NN, ne * C::QE, &bar[st]);
    bulk_g2s(sb + C::O_G, (const T *)mn.GSP + e0 * 8 * NN, ne * C::GE, &bar[st]);
    bulk_g2s(sb + C::O_C, (const T *)mn.CF + e0 * 16 * N, ne * C::CE, &bar[st]);
    if (OTF) bulk_g2s(sb + C::O_EG, (const T *)mn.egeo + e0 * 8, ne * C::GEE, &bar[st]);
    bulk_g2s(sb + C::O_EF, mn.eflag + e0, nf * 4u, &bar[st]);
  };
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_mbar_init();
  }
  // the interpolation and derivative weights, read per thread at different points
  for (int k = threadIdx.x; k < (N + 1) * N; k += NT) {
    sHf[k] = B.Hf[k];
    sDm[k] = B.Dm[k];
    if (k < N) sXs[k] = B.Xs[k];
    if (k <= N) sXf[k] = B.Xf[k];
  }
  __syncthreads();
  int item = blockIdx.x;
  if (threadIdx.x == 0 && item < nitems) issue(item, 0);
  // phase-1 thread: interior flux point fi of SP line m in direction d of
  // tile element le; the threads with fi = 1 also take the line's traces
  const int fi = 1 + (int)threadIdx.x / C::LINES;
  const int t1 = (int)threadIdx.x - (fi - 1) * C::LINES;
  const int le = t1 / (2 * N);
  const int r = t1 - le * 2 * N;
  const int d = r / N, m = r - d * N;
  bool bad = false;
  int it = 0;
  for (; item < nitems; item += gridDim.x, ++it) {
    const int st = it & 1;
    const int next = item + gridDim.x;
    int cs, tile;
    src.item(item, cs, tile);
    const MeshDev &md = src.mesh(cs);
    const VolArgs<T> &va = src.args(cs);
    const StatePtr in = va.in, base = va.base, out = va.out;
    const RkCoef<T> rk = va.rk;
    const int has_base = va.has_base;
    T *const w_out = va.w_out;
    const T *const w_in = va.w_in;
    double *const Rout = va.R;
    const T *zt = zone_tab<T>(md.clk);
    const T gm1 = pick<T>(md.gm1, md.gm1_f);
    if (threadIdx.x == 0 && next < nitems) {
      // the other stage was last read before the previous iteration's closing
      // barrier; order those generic reads before the async writes
      fence_proxy_async_smem();
      issue(next, st ^ 1);
    }
    if (!cta_wait(&bar[st], (uint32_t)((it >> 1) & 1))) {
      if (threadIdx.x == 0) {
        atomicOr(&md.clk->flags, 4);
        // let the copy in flight land before the CTA exits
        if (next < nitems) mbar_wait_bounded(&bar[st ^ 1], (uint32_t)(((it + 1) >> 1) & 1));
      }
      return;
    }
    unsigned char *sb = smem + st * C::STAGE;
    T *sQ = (T *)(sb + C::O_Q);                                                     // [EPB][NN][4]
    const T *sG = (const T *)(sb + C::O_G), *sCF = (const T *)(sb + C::O_C);        // [EPB][2][NN][4], [EPB][4][N][4]
    const T *sEG = (const T *)(sb + C::O_EG);
    const int *sEF = (const int *)(sb + C::O_EF);
    const int e0 = tile * EPB;
    const int ne = min(EPB, md.E - e0);
    // the tile's interface faces: their common fluxes from the mortar contributions
    if (gather_tile<T, N, GATHER_FLUX, LAY_POINTS>(md, e0, ne, sEF, (T *)(sb + C::O_C), 16 * N, false, NT)) __syncthreads();
    // ---- phase 1: one thread per interior flux point: Q and its gradients
    // interpolated to the point (Eq. Qt), the inviscid ALE flux and the
    // viscous flux (Sec. 2.1) transformed with the point's metric vector,
    // into the tile's flux array ----
    if (le < ne) {
      ElemGeo<T, N, OTF> G;
      G.load_rec(md, e0 + le, sEF[le], sEG + le * 8, zt);
      const T *h = sHf + fi * N;
      T qf[4] = {0, 0, 0, 0}, g8[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int sp = d == 0 ? m * N + k : k * N + m;
        T q[4], gx[4], gy[4];
        ld4(sQ + 4 * (le * NN + sp), q);
        ld4(sG + 4 * (le * 2 * NN + sp), gx);
        ld4(sG + 4 * (le * 2 * NN + NN + sp), gy);
        fma4(qf, h[k], q);
        fma4(g8, h[k], gx);
        fma4(g8 + 4, h[k], gy);
      }
      T vx, vy, vg;
      G.fp_at(d, fi, m, sXf[fi], sXs[m], vx, vy, vg);
      T f[4];
      if constexpr (std::is_same<T, double>::value) {
        total_flux(qf, g8, md, vx, vy, vg, f);
      } else {
        const T p = pressure_of(qf, gm1);
        T Fv[4], Gv[4];
        normal_flux(qf, p, vx, vy, vg, f);
        viscous_flux(qf, g8, g8 + 4, md, Fv, Gv);
#pragma unroll
        for (int v = 0; v < 4; ++v) f[v] = fma(vx, Fv[v], fma(vy, Gv[v], f[v]));
      }
      st4(sFl + ((le * 2 + d) * N + m) * C::LS + (fi - 1) * 4, f);
    }
    __syncthreads();
    // (RF + RG)[v] at SP sp = (i, j) of element l2: each direction's
    // divergence over its line's flux points 0..N in order (Eqs. Ft, Gt), the
    // end points from the common fluxes
    auto divergence = [&](int l2, int sp, T *dsum) {
      const int i = sp % N, j = sp / N;
      const T *fx = sFl + ((l2 * 2 + 0) * N + j) * C::LS, *fe = sFl + ((l2 * 2 + 1) * N + i) * C::LS;
      const T *wx = sDm + i * (N + 1), *we = sDm + j * (N + 1);
      const T *cf = sCF + l2 * 16 * N;
      T a[4] = {0, 0, 0, 0}, b[4] = {0, 0, 0, 0}, t[4];
      ld4(cf + (3 * N + j) * 4, t);
      fma4(a, wx[0], t);
      ld4(cf + (0 * N + i) * 4, t);
      fma4(b, we[0], t);
#pragma unroll
      for (int l = 1; l < N; ++l) {
        ld4(fx + (l - 1) * 4, t);
        fma4(a, wx[l], t);
        ld4(fe + (l - 1) * 4, t);
        fma4(b, we[l], t);
      }
      ld4(cf + (1 * N + j) * 4, t);
      fma4(a, wx[N], t);
      ld4(cf + (2 * N + i) * 4, t);
      fma4(b, we[N], t);
#pragma unroll
      for (int v = 0; v < 4; ++v) dsum[v] = a[v] + b[v];
    };
    // ---- phase 2: dQ/dt at the SPs and the Runge-Kutta stage; an SP's base
    // state and lo planes come from global memory, the next SP's loads issued
    // before this SP's stores (later stages update the state in place, so the
    // compiler keeps loads behind earlier stores unless the program orders them
    // first) ----
    auto fetch = [&](int idx, T *bh, T *kl, T *bl) {
      const size_t gi = ((size_t)e0 * NN + idx) * 4;
#pragma unroll
      for (int v = 0; v < 4; ++v) bh[v] = kl[v] = bl[v] = 0;
      if (has_base) ld4((const T *)base.hi + gi, bh);
      if constexpr (FF && LO) {
        ld4((const T *)in.lo + gi, kl);
        if (has_base) ld4((const T *)base.lo + gi, bl);
      }
    };
    T bh[4], kl[4], bl[4];
    if (MODE == MODE_RK && (int)threadIdx.x < ne * NN) fetch(threadIdx.x, bh, kl, bl);
    for (int idx = threadIdx.x; idx < ne * NN; idx += NT) {
      T nbh[4], nkl[4], nbl[4];
      if (MODE == MODE_RK && idx + NT < ne * NN) fetch(idx + NT, nbh, nkl, nbl);
      const int l2 = idx / NN, sp = idx - l2 * NN;
      const T iJ = ElemGeo<T, N, OTF>::inv_jac_at(md, sEF[l2], sEG + l2 * 8, sp, sXs[sp % N], sXs[sp / N]);
      T dsum[4];
      divergence(l2, sp, dsum);
      if constexpr (MODE == MODE_RESIDUAL) {
        const size_t gi = ((size_t)(e0 + l2) * 4) * NN + sp;
#pragma unroll
        for (int v = 0; v < 4; ++v) Rout[gi + v * NN] = -(double)(dsum[v] * iJ);
      } else {
        const size_t gi = ((size_t)e0 * NN + idx) * 4;
        T h[4], w[4], hn[4], ln[4];
        ld4(sQ + 4 * idx, h);
        if (w_in) ld4(w_in + gi, w);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const T R = -(dsum[v] * iJ);
          T inc = mul_rn(rk.bdt, R);
          if constexpr (FF && LO) {
            // double-float state: the increment added exactly (two-sum)
            if (has_base) inc = fma(rk.a0, (bh[v] - h[v]) + (bl[v] - kl[v]), inc);
            if (w_in) inc += w[v];
            float sum, err;
            two_sum(h[v], inc, sum, err);
            err += kl[v];
            hn[v] = sum + err;
            ln[v] = err - (hn[v] - sum);
          } else {
            // FP64, or a single-float state rounded to float once
            if (has_base) inc = fma(rk.a0, bh[v] - h[v], inc);
            if (w_in) inc += w[v];
            hn[v] = h[v] + inc;
          }
          w[v] = FF ? fma(-rk.g, inc, rk.ddt * R) : mul_sub(rk.ddt, R, rk.g, inc);
        }
        st4((T *)out.hi + gi, hn);
        if constexpr (FF && LO) st4((T *)out.lo + gi, ln);
        if (w_out) st4(w_out + gi, w);
        bad |= !physical(hn);
        st4(sQ + 4 * idx, hn);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          bh[v] = nbh[v];
          kl[v] = nkl[v];
          bl[v] = nbl[v];
        }
      }
    }
    if (MODE == MODE_RK) {
      __syncthreads();
      // ---- phase 3: face traces of the new state, one thread per end of an SP line ----
      for (int q = threadIdx.x; q < 2 * C::LINES; q += NT) {
        const int end = q / C::LINES, ln = q - end * C::LINES;
        const int l3 = ln / (2 * N), r3 = ln - l3 * 2 * N;
        const int d3 = r3 / N, m3 = r3 - d3 * N;
        if (l3 < ne) {
          T a0[4] = {0, 0, 0, 0};
#pragma unroll
          for (int k = 0; k < N; ++k) {
            T v[4];
            ld4(sQ + 4 * (l3 * NN + (d3 == 0 ? m3 * N + k : k * N + m3)), v);
            fma4(a0, end ? B.H1[k] : B.H0[k], v);
          }
          const int f3 = d3 == 0 ? (end ? 1 : 3) : (end ? 2 : 0);
          st4((T *)md.TR + ((size_t)(e0 + l3) * 4 + f3) * 4 * N + 4 * m3, a0);
        }
      }
    }
    // every read of this tile's stage is done before it is refilled (a batch
    // raises the non-physical flag on the tile's own case here)
    if constexpr (Src::kMulti) {
      if (__syncthreads_or(bad) && threadIdx.x == 0 && MODE == MODE_RK) atomicOr(&md.clk->flags, 1);
      bad = false;
    } else {
      __syncthreads();
    }
  }
  if constexpr (!Src::kMulti) {
    if (MODE == MODE_RK && __syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&src.mesh(0).clk->flags, 1);
  }
}

}  // namespace ssd
