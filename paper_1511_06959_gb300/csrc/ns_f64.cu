// FP64 stage kernels of the central scheme on 3D boxes: the residual and its transpose of
// ns_rhs.cu and ns_adj.cu, with the Runge-Kutta epilogues, arranged for few FP64
// operations.
//
// GB300 issues an FP64 instruction at 1/64 of the FP32 rate (1.05 TFLOP/s measured), so an
// FP64 stage is bound by their number, and loads, shared memory and integer work are next
// to free.  Against the kernels that the mixed path shares with it, this form
//   - takes the convective flux per cell, once, and differences it between the two
//     neighbours (the sum over a cell's faces of the two-cell means is that difference)
//     instead of forming both cells' fluxes at every face;
//   - forms the central differences of the velocity once per cell and adds the two cells'
//     values at a face, and keeps the constants of each term multiplied out;
//   - divides once per position (the transpose keeps 1/rho).
// A CTA owns TX x TY columns and marches its piece of planes (March); TY = 4 lets two
// CTAs of 128 threads share an SM, one computing while the other waits at a barrier.
// 128x64x64, per launch: residual 386 us before and 224 us now (at the FP64 pipe's full rate
// for 82% of the time), transpose with the added viscosity 650 us before and 422 to 442 us now;
// a step of four stages 1538 us before and 889 us now, an adjoint step 3720 and 2409 us.
#include "ns_common.cuh"
#include "ns_kernels.h"

namespace ns {
namespace f64k {

constexpr int TY = 4;
constexpr int NT = TX * TY;
constexpr int SY = TY + 2;
constexpr int SP = SX * SY;
constexpr int RND = 2;                         // load rounds of a plane
static_assert(SP > NT && SP <= 2 * NT - 32, "positions of the second round");
constexpr int DX = TY * SX;                    // own rows x shared columns
constexpr int DY = SY * TX;                    // shared rows x own columns
constexpr int FX = TY * (TX + 1);
constexpr int FY = (TY + 1) * TX;

// The work beyond one cell per thread goes to fixed warps so that the four schedulers'
// FP64 units get equal shares: warps 1 to 3 load, convert and (transpose) take the z-faces
// of the SP - NT positions after the first NT, warp 0 takes the tile's last faces, warps 2
// and 3 (residual) or 0 (transpose) the halo rows' terms.  Handed out from thread 0 up, all
// of it fell on the same scheduler.
__device__ __forceinline__ int shared_pos(int it) { return it == 0 ? (int)threadIdx.x : NT + (int)threadIdx.x - 32; }
__device__ __forceinline__ bool has_pos(int it) { return it == 0 || (threadIdx.x >= 32 && shared_pos(it) < SP); }

// In-plane offsets, periodic wrap resolved, of this thread's shared positions.
struct Halo {
  int o[RND];
};
__device__ __forceinline__ Halo halo_of(const GridDesc& g, int x0, int y0) {
  Halo h;
#pragma unroll
  for (int it = 0; it < RND; ++it) {
    const int t = shared_pos(it);
    const int ly = t / SX, lx = t - ly * SX;
    h.o[it] = has_pos(it) ? wrap(y0 + ly - 1, g.ny) * g.nx + wrap(x0 + lx - 1, g.nx) : 0;
  }
  return h;
}

struct Plane {
  double v[RND][5];
};
__device__ __forceinline__ void plane_load(Plane& r, const GridDesc& g, size_t box, int k, const Halo& h,
                                           const double* __restrict__ W) {
  const size_t pb = box + (size_t)wrap(k, g.nz) * g.plane;
  const long long n5 = 5 * g.cells * g.batch;   // field extent (debug bounds checks)
  (void)n5;
#pragma unroll
  for (int it = 0; it < RND; ++it)
    if (has_pos(it)) {
#pragma unroll
      for (int v = 0; v < 5; ++v) r.v[it][v] = NS_LD(g, W, pb + v * (size_t)g.cells, h.o[it], n5);
    }
}

// Constants of the terms below, multiplied out on the host and read from the parameter
// bank: a product of constants formed in the kernel would take an FP64 instruction per
// cell or a register pair.
struct Consts {
  double gm1, idx[3], hidx[3];
  double c[3], t[3];      // mu / (4 dx_d), -2/3 mu / (4 dx_d)
  double k[3], k43[3];    // mu / dx_d, 4/3 mu / dx_d
  double a[3];            // alpha / dx_d
  // transpose: 2 alpha / dx_d^2; mu / dx_d^2 (4/3 of it where the row j is d); the
  // tangential parts mu / (4 dx_f dx_l) and -2/3 of it, f the faces' direction, l the
  // difference's; 1 / (2 dx_d^2)
  double e2[3], n[3][3], m[3][3], m23[3][3], w[3];
};
Consts consts_of(const Coef<double>& c) {
  Consts k;
  k.gm1 = c.gm1;
  for (int d = 0; d < 3; ++d) {
    k.idx[d] = c.idx[d];
    k.hidx[d] = c.hidx[d];
    k.c[d] = c.mu * c.i4dx[d];
    k.t[d] = -2.0 / 3.0 * k.c[d];
    k.k[d] = c.mu * c.idx[d];
    k.k43[d] = 4.0 / 3.0 * k.k[d];
    k.a[d] = c.alpha * c.idx[d];
    k.e2[d] = 2.0 * k.a[d] * c.idx[d];
    k.w[d] = 0.5 * c.idx[d] * c.idx[d];
    for (int j = 0; j < 3; ++j) {
      k.n[d][j] = (j == d ? k.k43[d] : k.k[d]) * c.idx[d];
      k.m[d][j] = c.mu * c.idx[d] * c.i4dx[j];
      k.m23[d][j] = -2.0 / 3.0 * k.m[d][j];
    }
  }
  return k;
}

// What several places of a kernel evaluate (a face may be a tile's own, a neighbour's or the
// first of a range) is written with explicit roundings, so that its value does not depend on
// the place, nor the result on how the planes are cut into pieces.
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }

// x-face terms of shared position i (own row): a1 = d u_x / dy, a2 = d u_x / dz, d1 = the
// divergence's y and z parts.  U0, Um, Up: velocity (stride SP) of planes k, k-1, k+1.
__device__ __forceinline__ void x_terms(const Consts& K, const double* U0, const double* Um, const double* Up, int i,
                                        double o[3]) {
  o[0] = mul(K.c[1], U0[i + SX] - U0[i - SX]);
  o[1] = mul(K.c[2], Up[i] - Um[i]);
  o[2] = fma(K.t[2], Up[2 * SP + i] - Um[2 * SP + i], mul(K.t[1], U0[SP + i + SX] - U0[SP + i - SX]));
}
// y-face terms: d u_y / dx, d u_y / dz, the divergence's x and z parts
__device__ __forceinline__ void y_terms(const Consts& K, const double* U0, const double* Um, const double* Up, int i,
                                        double o[3]) {
  o[0] = mul(K.c[0], U0[SP + i + 1] - U0[SP + i - 1]);
  o[1] = mul(K.c[2], Up[SP + i] - Um[SP + i]);
  o[2] = fma(K.t[2], Up[2 * SP + i] - Um[2 * SP + i], mul(K.t[0], U0[i + 1] - U0[i - 1]));
}
// in-plane differences of one plane at the own cell: d u_z / dx, d u_z / dy (z-face terms)
// and the divergence's x and y parts
__device__ __forceinline__ void plane_terms(const Consts& K, const double* U0, int i, double o[4]) {
  o[0] = mul(K.c[0], U0[2 * SP + i + 1] - U0[2 * SP + i - 1]);
  o[1] = mul(K.c[1], U0[2 * SP + i + SX] - U0[2 * SP + i - SX]);
  o[2] = mul(K.t[0], U0[i + 1] - U0[i - 1]);
  o[3] = mul(K.t[1], U0[SP + i + SX] - U0[SP + i - SX]);
}

// The transverse terms of plane k: the own cell's (from the carried in-plane differences
// pt of plane k) and those of the halo cells next to the tile.
template <bool RHS>
__device__ __forceinline__ void fill_terms(const Consts& K, const double* U0, const double* Um, const double* Up,
                                           const double pt[4], int tx, int ty, int ic, double* __restrict__ sDX,
                                           double* __restrict__ sDY) {
  const double dz = Up[2 * SP + ic] - Um[2 * SP + ic];
  const int ix = ty * SX + tx + 1, iy = (ty + 1) * TX + tx;
  sDX[ix] = mul(K.c[1], U0[ic + SX] - U0[ic - SX]);
  sDX[DX + ix] = mul(K.c[2], Up[ic] - Um[ic]);
  sDX[2 * DX + ix] = fma(K.t[2], dz, pt[3]);
  sDY[iy] = mul(K.c[0], U0[SP + ic + 1] - U0[SP + ic - 1]);
  sDY[DY + iy] = mul(K.c[2], Up[SP + ic] - Um[SP + ic]);
  sDY[2 * DY + iy] = fma(K.t[2], dz, pt[2]);
  // the halo rows (0 and SY-1, one per warp) and columns (0 and SX-1)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double o[3];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    if (warp == (RHS ? 2 + r : 0)) {
      const int row = r == 0 ? 0 : SY - 1;
      y_terms(K, U0, Um, Up, row * SX + lane + 1, o);
#pragma unroll
      for (int j = 0; j < 3; ++j) sDY[j * DY + row * TX + lane] = o[j];
    }
  }
  if (warp == 1 && lane < 2 * TY) {
    const int row = lane >> 1, col = (lane & 1) ? SX - 1 : 0;
    x_terms(K, U0, Um, Up, (row + 1) * SX + col, o);
#pragma unroll
    for (int j = 0; j < 3; ++j) sDX[j * DX + row * SX + col] = o[j];
  }
}

// ---------------------------------------------------------------------------------
// residual and Runge-Kutta stage
// ---------------------------------------------------------------------------------
// viscous face values: stress row (3) and the energy flux, between cells iL and iR of U
// (values u1, u2, u3, e); t[j]: the two cells' transverse terms of row entry j, added
__device__ __forceinline__ void stress_face(double kn, double kd, double ka, int D, const double uL[4],
                                            const double uR[4], const double t[3], double o[4]) {
  double en = 0.0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    o[j] = fma(j == D ? kd : kn, uR[j] - uL[j], t[j]);
    en = j == 0 ? mul(uL[j] + uR[j], o[j]) : fma(uL[j] + uR[j], o[j], en);
  }
  o[3] = fma(0.5, en, mul(ka, uR[3] - uL[3]));
}

constexpr int NG = 12;   // m (3), Fxx, Fxy, Fxz, Fyy, Fyz, Fzz, (E + p) u (3)
constexpr size_t RHS_SMEM = sizeof(double) * (3 * 4 * SP + 2 * NG * SP + 3 * (DX + DY) + 4 * (FX + FY));

__device__ __forceinline__ void rhs_store(const Plane& r, double gm1, double* __restrict__ U, double* __restrict__ G) {
#pragma unroll
  for (int it = 0; it < RND; ++it) {
    const int t = shared_pos(it);
    if (has_pos(it)) {
      const double* w = r.v[it];
      const double ir = recip(w[0]);
      const double u[3] = {mul(w[1], ir), mul(w[2], ir), mul(w[3], ir)};
      const double ei = fma(-0.5, fma(w[3], u[2], fma(w[2], u[1], mul(w[1], u[0]))), w[4]);   // rho e
      const double p = mul(gm1, ei), H = w[4] + p;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        U[j * SP + t] = u[j];
        G[j * SP + t] = w[1 + j];
        G[(9 + j) * SP + t] = H * u[j];
      }
      U[3 * SP + t] = ei * ir;
      G[3 * SP + t] = fma(w[1], u[0], p);
      G[4 * SP + t] = w[1] * u[1];
      G[5 * SP + t] = w[1] * u[2];
      G[6 * SP + t] = fma(w[2], u[1], p);
      G[7 * SP + t] = w[2] * u[2];
      G[8 * SP + t] = fma(w[3], u[2], p);
    }
  }
}

__global__ void __launch_bounds__(NT, 2) k_rhs_f64(GridDesc g, const __grid_constant__ Consts K, StageArgs<double, double> a) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sU = reinterpret_cast<double*>(smem_raw);   // [3][4][SP] u1, u2, u3, e
  double* sG = sU + 3 * 4 * SP;                        // [2][NG][SP] convective fluxes
  double* sDX = sG + 2 * NG * SP;                      // [3][TY][SX]
  double* sDY = sDX + 3 * DX;                          // [3][SY][TX]
  double* sFX = sDY + 3 * DY;                          // [4][TY][TX+1]
  double* sFY = sFX + 4 * FX;                          // [4][TY+1][TX]
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  int b, x0, y0, kz0, kz1;
  March<TX, TY> march;
#pragma unroll 1
  while (march.next(g, b, x0, y0, kz0, kz1)) {
  const int gx = x0 + tx, gy = y0 + ty;
  const bool valid = gx < g.nx && gy < g.ny;
  const int cp = valid ? gy * g.nx + gx : 0;
  const size_t box = (size_t)b * 5 * g.cells, fc = (size_t)g.cells;
  const long long n5 = 5 * g.cells * g.batch;   // field extent (debug bounds checks)
  (void)n5;
  const Halo h = halo_of(g, x0, y0);
  auto slot = [&](int k) { return sU + ((k - kz0 + 1) % 3) * 4 * SP; };
  auto gslot = [&](int k) { return sG + ((k - kz0 + 1) & 1) * NG * SP; };
  const int ic = (ty + 1) * SX + tx + 1;
  // z-fluxes of the own column in planes k-1 and k, carried along the march
  constexpr int GZ[5] = {2, 5, 7, 8, 11};
  double gzm[5], gz0[5];
  {
    Plane p0, p1, p2;
    plane_load(p0, g, box, kz0 - 1, h, a.W);
    plane_load(p1, g, box, kz0, h, a.W);
    plane_load(p2, g, box, kz0 + 1, h, a.W);
    rhs_store(p0, K.gm1, slot(kz0 - 1), gslot(kz0 - 1));
    rhs_store(p1, K.gm1, slot(kz0), gslot(kz0));
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      gzm[v] = gslot(kz0 - 1)[GZ[v] * SP + ic];
      gz0[v] = gslot(kz0)[GZ[v] * SP + ic];
    }
    __syncthreads();   // plane kz0-1's fluxes are replaced by those of plane kz0+1
    rhs_store(p2, K.gm1, slot(kz0 + 1), gslot(kz0 + 1));
  }
  __syncthreads();
  double pt[4], zlo[4];
  plane_terms(K, slot(kz0), ic, pt);
  {
    double pm[4], uL[4], uR[4], t[3];
    plane_terms(K, slot(kz0 - 1), ic, pm);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uL[j] = slot(kz0 - 1)[j * SP + ic];
      uR[j] = slot(kz0)[j * SP + ic];
    }
    t[0] = pm[0] + pt[0];
    t[1] = pm[1] + pt[1];
    t[2] = (pm[2] + pm[3]) + (pt[2] + pt[3]);
    stress_face(K.k[2], K.k43[2], K.a[2], 2, uL, uR, t, zlo);
  }
  for (int k = kz0; k < kz1; ++k) {
    const bool more = k + 1 < kz1;
    const double *U0 = slot(k), *Um = slot(k - 1), *Up = slot(k + 1);
    Plane pf;
    if (more) plane_load(pf, g, box, k + 2, h, a.W);
    const size_t pb = box + (size_t)k * g.plane;
    double e_src[5], e_dacc[5], e_base[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      e_src[v] = 0.0;
      e_dacc[v] = 0.0;
      e_base[v] = 0.0;
    }
    if (valid) {
      if (a.src) {
#pragma unroll
        for (int v = 0; v < 5; ++v) e_src[v] = NS_LD(g, a.src, pb + v * fc, cp, n5);
      }
      if (a.dacc && !a.dacc_init) {
#pragma unroll
        for (int v = 0; v < 5; ++v) e_dacc[v] = NS_LD(g, a.dacc, pb + v * fc, cp, n5);
      }
      if (a.Wout) {
#pragma unroll
        for (int v = 0; v < 5; ++v) e_base[v] = NS_LD(g, a.base, pb + v * fc, cp, n5);
      } else if (a.wout && a.wbase) {
#pragma unroll
        for (int v = 0; v < 5; ++v) e_base[v] = NS_LD(g, a.wbase, pb + v * fc, cp, n5);
      }
    }
    fill_terms<true>(K, U0, Um, Up, pt, tx, ty, ic, sDX, sDY);
    // convective part: central differences of the cell fluxes
    double R[5];
    {
      const double *G0 = gslot(k), *Gp = gslot(k + 1);
      constexpr int GX[5] = {0, 3, 4, 5, 9}, GY[5] = {1, 4, 6, 7, 10};
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const double gzp = Gp[GZ[v] * SP + ic];
        R[v] = (G0[GX[v] * SP + ic - 1] - G0[GX[v] * SP + ic + 1]) * K.hidx[0];
        R[v] += (G0[GY[v] * SP + ic - SX] - G0[GY[v] * SP + ic + SX]) * K.hidx[1];
        R[v] += (gzm[v] - gzp) * K.hidx[2];
        gzm[v] = gz0[v];
        gz0[v] = gzp;
      }
    }
    __syncthreads();
    // plane k+2 replaces plane k-1 (and plane k's fluxes): nothing reads those any more
    if (more) rhs_store(pf, K.gm1, slot(k + 2), gslot(k + 2));
    double xs[4], ys[4], zhi[4];
    {
      double uC[4], uN[4], t[3];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uC[j] = U0[j * SP + ic];
        uN[j] = U0[j * SP + ic - 1];
      }
      const int ix = ty * SX + tx;
      t[0] = sDX[2 * DX + ix] + sDX[2 * DX + ix + 1];
      t[1] = sDX[ix] + sDX[ix + 1];
      t[2] = sDX[DX + ix] + sDX[DX + ix + 1];
      stress_face(K.k[0], K.k43[0], K.a[0], 0, uN, uC, t, xs);
      const int iy = ty * TX + tx;
#pragma unroll
      for (int j = 0; j < 4; ++j) uN[j] = U0[j * SP + ic - SX];
      t[0] = sDY[iy] + sDY[iy + TX];
      t[1] = sDY[2 * DY + iy] + sDY[2 * DY + iy + TX];
      t[2] = sDY[DY + iy] + sDY[DY + iy + TX];
      stress_face(K.k[1], K.k43[1], K.a[1], 1, uN, uC, t, ys);
      double pn[4];
      plane_terms(K, Up, ic, pn);
#pragma unroll
      for (int j = 0; j < 4; ++j) uN[j] = Up[j * SP + ic];
      t[0] = pt[0] + pn[0];
      t[1] = pt[1] + pn[1];
      t[2] = (pt[2] + pt[3]) + (pn[2] + pn[3]);
      stress_face(K.k[2], K.k43[2], K.a[2], 2, uC, uN, t, zhi);
#pragma unroll
      for (int j = 0; j < 4; ++j) pt[j] = pn[j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      sFX[j * FX + ty * (TX + 1) + tx] = xs[j];
      sFY[j * FY + ty * TX + tx] = ys[j];
    }
    // the tile's last x-faces and y-faces
    if (tid < TX) {
      double uL[4], uR[4], t[3], o[4];
      {
        const int iL = TY * SX + tid + 1, iy = TY * TX + tid;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uL[j] = U0[j * SP + iL];
          uR[j] = U0[j * SP + iL + SX];
        }
        t[0] = sDY[iy] + sDY[iy + TX];
        t[1] = sDY[2 * DY + iy] + sDY[2 * DY + iy + TX];
        t[2] = sDY[DY + iy] + sDY[DY + iy + TX];
        stress_face(K.k[1], K.k43[1], K.a[1], 1, uL, uR, t, o);
#pragma unroll
        for (int j = 0; j < 4; ++j) sFY[j * FY + TY * TX + tid] = o[j];
      }
      if (tid < TY) {
        const int r = tid, iL = (r + 1) * SX + TX, ix = r * SX + TX;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uL[j] = U0[j * SP + iL];
          uR[j] = U0[j * SP + iL + 1];
        }
        t[0] = sDX[2 * DX + ix] + sDX[2 * DX + ix + 1];
        t[1] = sDX[ix] + sDX[ix + 1];
        t[2] = sDX[DX + ix] + sDX[DX + ix + 1];
        stress_face(K.k[0], K.k43[0], K.a[0], 0, uL, uR, t, o);
#pragma unroll
        for (int j = 0; j < 4; ++j) sFX[j * FX + r * (TX + 1) + TX] = o[j];
      }
    }
    __syncthreads();
    if (valid) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        R[1 + j] += (sFX[j * FX + ty * (TX + 1) + tx + 1] - xs[j]) * K.idx[0];
        R[1 + j] += (sFY[j * FY + (ty + 1) * TX + tx] - ys[j]) * K.idx[1];
        R[1 + j] += (zhi[j] - zlo[j]) * K.idx[2];
      }
      if (a.src) {
#pragma unroll
        for (int v = 0; v < 5; ++v) R[v] += e_src[v];
      }
      double dv[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) dv[v] = e_dacc[v] + a.cacc * R[v];
      if (a.wout) {
        double e_wb[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) e_wb[v] = e_base[v];
        if (a.Wout && a.wbase) {
#pragma unroll
          for (int v = 0; v < 5; ++v) e_wb[v] = NS_LD(g, a.wbase, pb + v * fc, cp, n5);
        } else if (a.Wout) {
#pragma unroll
          for (int v = 0; v < 5; ++v) e_wb[v] = 0.0;
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          const double wv = e_wb[v] + dv[v];
          NS_ST(g, a.wout, pb + v * fc, cp, n5, wv);
          if (a.wout_mirror) NS_ST(g, a.wout_mirror, pb + v * fc, cp, n5, wv);
        }
      } else if (a.dacc) {
#pragma unroll
        for (int v = 0; v < 5; ++v) NS_ST(g, a.dacc, pb + v * fc, cp, n5, dv[v]);
      }
      if (a.Wout) {
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          double wv = e_base[v] + a.cout * R[v];
          if (a.cd != 0.0) wv += a.cd * dv[v];
          NS_ST(g, a.Wout, pb + v * fc, cp, n5, wv);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) zlo[j] = zhi[j];
  }
  }
}

// ---------------------------------------------------------------------------------
// transposed product and adjoint stage
// ---------------------------------------------------------------------------------
constexpr int NFX = SY * (SX - 1), NFY = (SY - 1) * SX, NF = NFX + NFY;   // in-plane faces of a plane
constexpr size_t ADJ_SMEM = sizeof(double) * (3 * 6 * SP + 3 * 5 * SP + 3 * SP + 2 * 4 * NF + 2 * 3 * SP +
                                              3 * (DX + DY) + 3 * (FX + FY));

struct AdjPlane {
  Plane q, a;
  double n[RND];
};
__device__ __forceinline__ void adj_load(AdjPlane& r, const GridDesc& g, size_t box, int b, int k, const Halo& h,
                                         const AdjArgs<double, double, double>& a) {
  plane_load(r.q, g, box, k, h, a.W);
  plane_load(r.a, g, box, k, h, a.A);
  const long long n1 = g.cells * g.batch;
  (void)n1;
  const size_t nb = (size_t)b * g.cells + (size_t)wrap(k, g.nz) * g.plane;
  if (a.nu) {
#pragma unroll
    for (int it = 0; it < RND; ++it)
      if (has_pos(it)) r.n[it] = widen_exact(NS_LD(g, a.nu, nb, h.o[it], n1));
  } else if (a.nud) {
#pragma unroll
    for (int it = 0; it < RND; ++it)
      if (has_pos(it)) r.n[it] = NS_LD(g, a.nud, nb, h.o[it], n1);
  }
}
// U: u1, u2, u3, rho, 1/rho, e (stride SP); A: the stage's seed ca A
__device__ __forceinline__ void adj_store(const AdjPlane& r, double ca, double* __restrict__ U, double* __restrict__ A,
                                          double* __restrict__ N, bool with_nu) {
#pragma unroll
  for (int it = 0; it < RND; ++it) {
    const int t = shared_pos(it);
    if (has_pos(it)) {
      const double* w = r.q.v[it];
      const double ir = recip(w[0]);
      const double u[3] = {mul(w[1], ir), mul(w[2], ir), mul(w[3], ir)};
#pragma unroll
      for (int j = 0; j < 3; ++j) U[j * SP + t] = u[j];
      U[3 * SP + t] = w[0];
      U[4 * SP + t] = ir;
      U[5 * SP + t] = fma(-0.5, fma(u[2], u[2], fma(u[1], u[1], mul(u[0], u[0]))), mul(w[4], ir));
#pragma unroll
      for (int v = 0; v < 5; ++v) A[v * SP + t] = ca == 1.0 ? r.a.v[it][v] : ca * r.a.v[it][v];
      if (with_nu) N[t] = r.n[it];
    }
  }
}

// face s-vector without its 1/dx: s_j = (a_L - a_R)_{1+j} + h (u_L + u_R)_j, and
// h = (a_L - a_R)_4 / 2
__device__ __forceinline__ void face_s(const double* UL, const double* AL, int iL, const double* UR, const double* AR,
                                       int iR, double s[3], double& hf) {
  hf = 0.5 * (AL[4 * SP + iL] - AR[4 * SP + iR]);
#pragma unroll
  for (int j = 0; j < 3; ++j)
    s[j] = fma(hf, UL[j * SP + iL] + UR[j * SP + iR], AL[(1 + j) * SP + iL] - AR[(1 + j) * SP + iR]);
}

// s-vectors of every x-face and y-face of a plane
__device__ __forceinline__ void fill_faces(double* __restrict__ F, const double* U, const double* A) {
#pragma unroll 1
  for (int t = threadIdx.x; t < NF; t += NT) {
    double s[3], hf;
    int iL, iR;
    if (t < NFX) {
      const int row = t / (SX - 1);
      iL = row * SX + (t - row * (SX - 1));
      iR = iL + 1;
    } else {
      iL = t - NFX;
      iR = iL + SX;
    }
    face_s(U, A, iL, U, A, iR, s, hf);
#pragma unroll
    for (int j = 0; j < 3; ++j) F[j * NF + t] = s[j];
    F[3 * NF + t] = hf;
  }
}
// z-face s-vectors between two planes: every shared position; the own cell's returned
__device__ __forceinline__ void fill_z(double* __restrict__ Z, const double* UL, const double* AL, const double* UR,
                                       const double* AR, int ic, double so[3], double& ho) {
  face_s(UL, AL, ic, UR, AR, ic, so, ho);
#pragma unroll
  for (int j = 0; j < 3; ++j) Z[j * SP + ic] = so[j];
  const int t = (int)threadIdx.x - 32;   // halo positions, by warps 1 to 3
  if (t >= 0 && t < 2 * SX + 2 * TY) {
    int i;
    if (t < SX) i = t;
    else if (t < 2 * SX) i = (SY - 1) * SX + (t - SX);
    else {
      const int r = t - 2 * SX;
      i = (1 + (r >> 1)) * SX + ((r & 1) ? SX - 1 : 0);
    }
    double s[3], hf;
    face_s(UL, AL, i, UR, AR, i, s, hf);
#pragma unroll
    for (int j = 0; j < 3; ++j) Z[j * SP + i] = s[j];
  }
}
static_assert(2 * SX + 2 * TY <= NT - 32, "halo z-faces of warps 1 to 3");

// primal stress row of a face (no energy flux)
__device__ __forceinline__ void sigma_face(double kn, double kd, int D, const double uL[3], const double uR[3],
                                           const double t[3], double o[3]) {
#pragma unroll
  for (int j = 0; j < 3; ++j) o[j] = fma(j == D ? kd : kn, uR[j] - uL[j], t[j]);
}

__global__ void __launch_bounds__(NT, 2) k_adj_f64(GridDesc g, const __grid_constant__ Consts K,
                                                   AdjArgs<double, double, double> a) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sU = reinterpret_cast<double*>(smem_raw);   // [3][6][SP]
  double* sA = sU + 3 * 6 * SP;                        // [3][5][SP]
  double* sN = sA + 3 * 5 * SP;                        // [3][SP]
  double* sF = sN + 3 * SP;                            // [2][4][NF]
  double* sZ = sF + 2 * 4 * NF;                        // [2][3][SP]
  double* sDX = sZ + 2 * 3 * SP;                       // [3][TY][SX]
  double* sDY = sDX + 3 * DX;                          // [3][SY][TX]
  double* sGX = sDY + 3 * DY;                          // [3][TY][TX+1] stress of the x-faces
  double* sGY = sGX + 3 * FX;                          // [3][TY+1][TX]
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  int b, x0, y0, kz0, kz1;
  March<TX, TY> march;
#pragma unroll 1
  while (march.next(g, b, x0, y0, kz0, kz1)) {
  const int gx = x0 + tx, gy = y0 + ty;
  const bool valid = gx < g.nx && gy < g.ny;
  const int cp = valid ? gy * g.nx + gx : 0;
  const size_t box = (size_t)b * 5 * g.cells, fc = (size_t)g.cells;
  const long long n5 = 5 * g.cells * g.batch;   // field extent (debug bounds checks)
  (void)n5;
  const Halo h = halo_of(g, x0, y0);
  const bool with_nu = a.nu != nullptr || a.nud != nullptr;
  auto sl = [&](int k) { return (k - kz0 + 1) % 3; };
  auto U_of = [&](int k) { return sU + sl(k) * 6 * SP; };
  auto A_of = [&](int k) { return sA + sl(k) * 5 * SP; };
  auto F_of = [&](int k) { return sF + ((k - kz0 + 1) & 1) * 4 * NF; };
  auto Z_of = [&](int k) { return sZ + ((k - kz0 + 1) & 1) * 3 * SP; };   // z-face k + 1/2
  const int ic = (ty + 1) * SX + tx + 1;
  {
    AdjPlane p;
#pragma unroll 1
    for (int q = kz0 - 1; q <= kz0 + 1; ++q) {
      adj_load(p, g, box, b, q, h, a);
      adj_store(p, a.ca, U_of(q), A_of(q), sN + sl(q) * SP, with_nu);
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int q = kz0 - 1; q <= kz0; ++q) fill_faces(F_of(q), U_of(q), A_of(q));
  double zsl[3], zhl, zgl[3], pt[4];   // lower z-face: s-vector, h, stress; in-plane terms of plane k
  fill_z(Z_of(kz0 - 1), U_of(kz0 - 1), A_of(kz0 - 1), U_of(kz0), A_of(kz0), ic, zsl, zhl);
  plane_terms(K, U_of(kz0), ic, pt);
  {
    double pm[4], uL[3], uR[3], t[3];
    plane_terms(K, U_of(kz0 - 1), ic, pm);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      uL[j] = U_of(kz0 - 1)[j * SP + ic];
      uR[j] = U_of(kz0)[j * SP + ic];
    }
    t[0] = pm[0] + pt[0];
    t[1] = pm[1] + pt[1];
    t[2] = (pm[2] + pm[3]) + (pt[2] + pt[3]);
    sigma_face(K.k[2], K.k43[2], 2, uL, uR, t, zgl);
  }
  // S_x[2], S_y[2] and the z-difference's diagonal part S_x[0] / dx + S_y[1] / dy (scaled)
  // of a plane at the own cell
  auto own_S = [&](const double* F, double o[3]) {
    const int xl = (ty + 1) * (SX - 1) + tx, yl = NFX + ty * SX + tx + 1;
    o[0] = F[2 * NF + xl] + F[2 * NF + xl + 1];
    o[1] = F[2 * NF + yl] + F[2 * NF + yl + SX];
    o[2] = fma(K.m23[0][2], F[xl] + F[xl + 1], mul(K.m23[1][2], F[NF + yl] + F[NF + yl + SX]));
  };
  __syncthreads();
  double own_m[3], own_0[3];
  own_S(F_of(kz0 - 1), own_m);
  own_S(F_of(kz0), own_0);
  __syncthreads();
  for (int k = kz0; k < kz1; ++k) {
    const bool more = k + 1 < kz1;
    const double *U0 = U_of(k), *Um = U_of(k - 1), *Up = U_of(k + 1);
    const double *A0 = A_of(k), *Ap = A_of(k + 1);
    const double* F0 = F_of(k);
    const size_t pb = box + (size_t)k * g.plane;
    AdjPlane pf;
    if (more) adj_load(pf, g, box, b, k + 2, h, a);
    double gin[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, lfv[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (valid) {
      if (a.Gin) {
#pragma unroll
        for (int v = 0; v < 5; ++v) gin[v] = NS_LD(g, a.Gin, pb + v * fc, cp, n5);
      }
      if (a.Anext) {
#pragma unroll
        for (int v = 0; v < 5; ++v) lfv[v] = NS_LD(g, a.lamf, pb + v * fc, cp, n5);
      }
    }
    fill_terms<false>(K, U0, Um, Up, pt, tx, ty, ic, sDX, sDY);
    fill_faces(F_of(k + 1), Up, Ap);
    double zsh[3], zhh, zgh[3], pn[4];
    fill_z(Z_of(k), U0, A0, Up, Ap, ic, zsh, zhh);
    plane_terms(K, Up, ic, pn);
    double uC[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) uC[j] = U0[j * SP + ic];
    {
      double uN[3], t[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) uN[j] = Up[j * SP + ic];
      t[0] = pt[0] + pn[0];
      t[1] = pt[1] + pn[1];
      t[2] = (pt[2] + pt[3]) + (pn[2] + pn[3]);
      sigma_face(K.k[2], K.k43[2], 2, uC, uN, t, zgh);
#pragma unroll
      for (int j = 0; j < 4; ++j) pt[j] = pn[j];
    }
    // plane k-1 is read below at the own cell only
    double am[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) am[v] = A_of(k - 1)[v * SP + ic];
    const double nzm = with_nu ? sN[sl(k - 1) * SP + ic] : 0.0;
    __syncthreads();
    if (more) adj_store(pf, a.ca, U_of(k + 2), A_of(k + 2), sN + sl(k + 2) * SP, with_nu);
    double xg[3], yg[3];
    {
      double uN[3], t[3];
      const int ix = ty * SX + tx, iy = ty * TX + tx;
#pragma unroll
      for (int j = 0; j < 3; ++j) uN[j] = U0[j * SP + ic - 1];
      t[0] = sDX[2 * DX + ix] + sDX[2 * DX + ix + 1];
      t[1] = sDX[ix] + sDX[ix + 1];
      t[2] = sDX[DX + ix] + sDX[DX + ix + 1];
      sigma_face(K.k[0], K.k43[0], 0, uN, uC, t, xg);
#pragma unroll
      for (int j = 0; j < 3; ++j) uN[j] = U0[j * SP + ic - SX];
      t[0] = sDY[iy] + sDY[iy + TX];
      t[1] = sDY[2 * DY + iy] + sDY[2 * DY + iy + TX];
      t[2] = sDY[DY + iy] + sDY[DY + iy + TX];
      sigma_face(K.k[1], K.k43[1], 1, uN, uC, t, yg);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        sGX[j * FX + ty * (TX + 1) + tx] = xg[j];
        sGY[j * FY + ty * TX + tx] = yg[j];
      }
    }
    if (tid < TX) {
      double uL[3], uR[3], t[3], o[3];
      {
        const int iL = TY * SX + tid + 1, iy = TY * TX + tid;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          uL[j] = U0[j * SP + iL];
          uR[j] = U0[j * SP + iL + SX];
        }
        t[0] = sDY[iy] + sDY[iy + TX];
        t[1] = sDY[2 * DY + iy] + sDY[2 * DY + iy + TX];
        t[2] = sDY[DY + iy] + sDY[DY + iy + TX];
        sigma_face(K.k[1], K.k43[1], 1, uL, uR, t, o);
#pragma unroll
        for (int j = 0; j < 3; ++j) sGY[j * FY + TY * TX + tid] = o[j];
      }
      if (tid < TY) {
        const int r = tid, iL = (r + 1) * SX + TX, ix = r * SX + TX;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          uL[j] = U0[j * SP + iL];
          uR[j] = U0[j * SP + iL + 1];
        }
        t[0] = sDX[2 * DX + ix] + sDX[2 * DX + ix + 1];
        t[1] = sDX[ix] + sDX[ix + 1];
        t[2] = sDX[DX + ix] + sDX[DX + ix + 1];
        sigma_face(K.k[0], K.k43[0], 0, uL, uR, t, o);
#pragma unroll
        for (int j = 0; j < 3; ++j) sGX[j * FX + r * (TX + 1) + TX] = o[j];
      }
    }
    __syncthreads();
    double own_p[3] = {0.0, 0.0, 0.0};
    if (valid) {
      const int xl = (ty + 1) * (SX - 1) + tx, yl = NFX + ty * SX + tx + 1;   // own lower faces in F
      const double *Zl = Z_of(k - 1), *Zh = Z_of(k);
      // viscous primitive adjoints: the normal gradients' part and, in u, the faces'
      // velocities' (1/dx h sigma)
      double ub[3], eb;
      const double hx = F0[3 * NF + xl], hx1 = F0[3 * NF + xl + 1], hy = F0[3 * NF + yl], hy1 = F0[3 * NF + yl + SX];
      eb = K.e2[0] * (hx - hx1);
      eb += K.e2[1] * (hy - hy1);
      eb += K.e2[2] * (zhl - zhh);
      const double ex = K.idx[0] * hx, ex1 = K.idx[0] * hx1, ey = K.idx[1] * hy, ey1 = K.idx[1] * hy1,
                   ez = K.idx[2] * zhl, ez1 = K.idx[2] * zhh;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        double q = K.n[0][j] * (F0[j * NF + xl] - F0[j * NF + xl + 1]);
        q += K.n[1][j] * (F0[j * NF + yl] - F0[j * NF + yl + SX]);
        q += K.n[2][j] * (zsl[j] - zsh[j]);
        q += ex * xg[j];
        q += ex1 * sGX[j * FX + ty * (TX + 1) + tx + 1];
        q += ey * yg[j];
        q += ey1 * sGY[j * FY + (ty + 1) * TX + tx];
        q += ez * zgl[j];
        q += ez1 * zgh[j];
        ub[j] = q;
      }
      {
        // tangential parts (see ns_adj.cu), the faces' 1/dx in the constants
        const int il = ic - 1, ir = ic + 1, idn = ic - SX, iup = ic + SX;
        const double* Y0 = F0 + NFX + ty * SX + tx;   // lower y-face of the cell at column tx (= own - 1)
        auto Sy = [&](int j, int dc) { return Y0[j * NF + dc] + Y0[j * NF + SX + dc]; };
        const double* X0 = F0 + ty * (SX - 1) + tx;   // lower x-face of the cell a row below
        auto Sx = [&](int j, int dr) { return X0[j * NF + dr * (SX - 1)] + X0[j * NF + dr * (SX - 1) + 1]; };
        auto Sz = [&](int j, int i) { return Zl[j * SP + i] + Zh[j * SP + i]; };
        ub[0] += K.m23[1][0] * (Sy(1, 0) - Sy(1, 2));
        ub[0] += K.m23[2][0] * (Sz(2, il) - Sz(2, ir));
        ub[1] += K.m[1][0] * (Sy(0, 0) - Sy(0, 2));
        ub[2] += K.m[2][0] * (Sz(0, il) - Sz(0, ir));
        ub[0] += K.m[0][1] * (Sx(1, 0) - Sx(1, 2));
        ub[1] += K.m23[0][1] * (Sx(0, 0) - Sx(0, 2));
        ub[1] += K.m23[2][1] * (Sz(2, idn) - Sz(2, iup));
        ub[2] += K.m[2][1] * (Sz(1, idn) - Sz(1, iup));
        own_S(F_of(k + 1), own_p);
        ub[0] += K.m[0][2] * (own_m[0] - own_p[0]);
        ub[1] += K.m[1][2] * (own_m[1] - own_p[1]);
        ub[2] += own_m[2] - own_p[2];
      }
      // convective part and pull-back
      const double rho = U0[3 * SP + ic], ir = U0[4 * SP + ic], e = U0[5 * SP + ic];
      const double Esp = e + 0.5 * (uC[0] * uC[0] + uC[1] * uC[1] + uC[2] * uC[2]);
      const double gr = K.gm1 * rho, H = rho * Esp + gr * e;
      double mb[3], Eb = 0.0, pbar = 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        double D[5];
#pragma unroll
        for (int v = 0; v < 5; ++v)
          D[v] = d == 2 ? Ap[v * SP + ic] - am[v]
                        : A0[v * SP + ic + (d == 0 ? 1 : SX)] - A0[v * SP + ic - (d == 0 ? 1 : SX)];
        const double hd = K.hidx[d];
        mb[d] = hd * (D[0] + D[1] * uC[0] + D[2] * uC[1] + D[3] * uC[2]);
        const double hm = hd * rho * uC[d], D4 = hd * D[4];
#pragma unroll
        for (int j = 0; j < 3; ++j) ub[j] += D[1 + j] * hm;
        const double t = D4 * uC[d];
        pbar += hd * D[1 + d] + t;
        Eb += t;
        ub[d] += D4 * H;
      }
      eb += gr * pbar;
      const double ei = eb * ir;
      double gout[5];
      gout[0] = K.gm1 * e * pbar - ei * Esp;
      gout[4] = Eb + ei;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double ui = (ub[j] - eb * uC[j]) * ir;
        gout[1 + j] = mb[j] + ui;
        gout[0] -= ui * uC[j];
      }
      // added adjoint viscosity: the six neighbours' differences with the weights
      // (nu + nu_q) / (2 dx^2) (a weighted sum less the weights' total would take five
      // operations fewer, but loses digits where a is smooth)
      if (with_nu) {
        const double *N0 = sN + sl(k) * SP, nc = N0[ic];
        const double f[6] = {(nc + N0[ic - 1]) * K.w[0],  (nc + N0[ic + 1]) * K.w[0], (nc + N0[ic - SX]) * K.w[1],
                             (nc + N0[ic + SX]) * K.w[1], (nc + nzm) * K.w[2], (nc + sN[sl(k + 1) * SP + ic]) * K.w[2]};
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          const double* Av = A0 + v * SP + ic;
          const double ac = Av[0];
          double L = f[0] * (Av[-1] - ac);
          L += f[1] * (Av[1] - ac);
          L += f[2] * (Av[-SX] - ac);
          L += f[3] * (Av[SX] - ac);
          L += f[4] * (am[v] - ac);
          L += f[5] * (Ap[v * SP + ic] - ac);
          gout[v] += a.nus[v == 0 ? 0 : (v == 4 ? 2 : 1)] * L;
        }
      }
      // epilogue
      double gs[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) gs[v] = gout[v];
      if (a.Gin) {
#pragma unroll
        for (int v = 0; v < 5; ++v) gs[v] += gin[v];
      }
      if (a.Gout) {
#pragma unroll
        for (int v = 0; v < 5; ++v) NS_ST(g, a.Gout, pb + v * fc, cp, n5, gs[v]);
      }
      if (a.lam_out) {
        double lv[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) lv[v] = gs[v];
        if (a.lam_in) {
#pragma unroll
          for (int v = 0; v < 5; ++v) lv[v] += NS_LD(g, a.lam_in, pb + v * fc, cp, n5);
        }
        if (a.obj_ndsc && (gx == a.obj_iL || gx == a.obj_iR)) {
          // the objective source of this step on the plane's two columns
          const int nf = g.ny * g.nz;
          const double* Af = a.obj_aface + ((size_t)b * nf + (size_t)k * g.ny + gy) * 5;
          const double NoD = a.obj_ndsc[2 * b], sc = a.obj_ndsc[2 * b + 1];
          const int reps = (gx == a.obj_iL ? 1 : 0) + (gx == a.obj_iR ? 1 : 0);
          for (int q = 0; q < reps; ++q) {
#pragma unroll
            for (int v = 0; v < 5; ++v) lv[v] += sc * (Af[v] - (v == 0 ? NoD : 0.0));
          }
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) NS_ST(g, a.lam_out, pb + v * fc, cp, n5, lv[v]);
        if (a.lam_out_mirror) {
#pragma unroll
          for (int v = 0; v < 5; ++v) NS_ST(g, a.lam_out_mirror, pb + v * fc, cp, n5, lv[v]);
        }
      }
      if (a.Anext) {
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          double an = a.cl * lfv[v] + a.cg * gout[v];
          if (a.cs != 0.0) an += a.cs * gs[v];
          NS_ST(g, a.Anext, pb + v * fc, cp, n5, an);
        }
      }
      if (a.SBout || a.sbar) {
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          double ss = A0[v * SP + ic];
          if (a.SBin) ss += NS_LD(g, a.SBin, pb + v * fc, cp, n5);
          if (a.SBout) NS_ST(g, a.SBout, pb + v * fc, cp, n5, ss);
          if (a.sbar) NS_ST(g, a.sbar, pb + v * fc, cp, n5, NS_LD(g, a.sbar, pb + v * fc, cp, n5) + ss);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      zsl[j] = zsh[j];
      zgl[j] = zgh[j];
      own_m[j] = own_0[j];
      own_0[j] = own_p[j];
    }
    zhl = zhh;
    __syncthreads();   // faces, z-faces and terms free; plane k+2 visible
  }
  }
}

}  // namespace f64k

cudaError_t launch_rhs_f64(const GridDesc& g, const Coef<double>& c, const StageArgs<double, double>& a,
                           cudaStream_t st) {
  static MarchShape<TX, f64k::TY> shape;
  int ctas = 0;
  cudaError_t e = shape.get(f64k::k_rhs_f64, f64k::RHS_SMEM, g, "NS_RHS_CTAS", ctas);
  if (e != cudaSuccess) return e;
  count_launch();
  return launch_pdl(f64k::k_rhs_f64, dim3(ctas), dim3(f64k::NT), f64k::RHS_SMEM, st, g, f64k::consts_of(c), a);
}

cudaError_t launch_adj_f64(const GridDesc& g, const Coef<double>& c, const AdjArgs<double, double, double>& a,
                           cudaStream_t st) {
  static MarchShape<TX, f64k::TY> shape;
  int ctas = 0;
  cudaError_t e = shape.get(f64k::k_adj_f64, f64k::ADJ_SMEM, g, "NS_ADJ_CTAS", ctas);
  if (e != cudaSuccess) return e;
  count_launch();
  return launch_pdl(f64k::k_adj_f64, dim3(ctas), dim3(f64k::NT), f64k::ADJ_SMEM, st, g, f64k::consts_of(c), a);
}

}  // namespace ns
