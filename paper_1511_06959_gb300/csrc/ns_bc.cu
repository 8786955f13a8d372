// Boundaries of a bounded box: characteristic (non-reflecting) inflow at x = 0 and
// outflow at x = L_x (section "Numerical methods"; the incoming characteristics are
// set there, section "Energy analysis"), and isothermal no-slip walls at y = 0 and
// y = L_y (the vane surface is isothermal, section "Problem setup"); z stays periodic.
//
// A bounded context works on the box padded by one ghost layer: ghost columns at
// x = -1 and x = nx (inflow, outflow), ghost rows at y = -1 and y = ny (walls), the
// rows built over the columns so that a corner is the wall's ghost of the inflow or
// outflow ghost.  The residual is the periodic residual of the padded box, cropped:
// the periodic stage kernels run unchanged on the padded box once its ghosts are
// filled (k_bc_ghosts).  The adjoint is the exact transpose of that map: the periodic
// transposed product runs on the padded box with a zero adjoint in the ghosts, and
// k_bc_adj_epilogue pulls each ghost's output back to the cell the ghost was built from
// through the transposed 5 x 5 ghost Jacobian (reversed by hand), rows first, then
// columns (the reverse of the padding's order).  The added adjoint viscosity
// passes no flux through the boundary faces, which keeps it symmetric and
// non-positive; the epilogue applies it on the unpadded box with those faces closed.
//
// Ghost states.  Inflow and outflow hold the boundary state of the x-direction Riemann
// invariants R+- = u1 +- 2c/(gamma-1): at the outflow R+, the entropy p/rho^gamma and
// the tangential velocity come from the adjacent cell and R- from the far field; at the
// inflow R- comes from the adjacent cell and the rest from the far field (subsonic flow
// along +x).  A wall ghost has the adjacent cell's density, its momentum reversed and
// the internal energy 2 e_w - e, so that the face velocity is zero and the face
// temperature is the wall's.
#include <cuda_runtime.h>

#include <type_traits>

#include "ns_common.cuh"
#include "ns_kernels.h"

namespace ns {

namespace {

__device__ __forceinline__ double dsqrt(double a) { return sqrt(a); }
__device__ __forceinline__ double dpow(double a, double e) { return pow(a, e); }
__device__ __forceinline__ float dsqrt(float a) { return sqrtf(a); }
__device__ __forceinline__ float dpow(float a, double e) { return powf(a, (float)e); }

// boundary state of a characteristic inflow (side 0) or outflow (side 1) ghost from the
// adjacent cell's conservative state wc
template <class T>
__device__ void char_state(const T wc[5], int side, const BcDesc& bc, T out[5]) {
  const double g = bc.gamma, k = 2.0 / (g - 1.0);
  const T rho = wc[0];
  const T u0 = wc[1] / rho, u1 = wc[2] / rho, u2 = wc[3] / rho;
  const T p = T(g - 1.0) * (wc[4] - T(0.5) * rho * (u0 * u0 + u1 * u1 + u2 * u2));
  const T c = dsqrt(T(g) * p / rho);
  const double uf1 = bc.far[1], uf2 = bc.far[2], uf3 = bc.far[3], cf = bc.cf;
  T Rp, Rm, ent, ut2, ut3;
  if (side == 1) {
    Rp = u0 + T(k) * c;
    Rm = T(uf1 - k * cf);
    ent = p / dpow(rho, g);
    ut2 = u1;
    ut3 = u2;
  } else {
    Rp = T(uf1 + k * cf);
    Rm = u0 - T(k) * c;
    ent = T(bc.ent);
    ut2 = T(uf2);
    ut3 = T(uf3);
  }
  const T ub = T(0.5) * (Rp + Rm);
  const T cb = T(0.25 * (g - 1.0)) * (Rp - Rm);
  const T rhob = dpow(cb * cb / (T(g) * ent), 1.0 / (g - 1.0));
  const T pb = rhob * cb * cb / T(g);
  out[0] = rhob;
  out[1] = rhob * ub;
  out[2] = rhob * ut2;
  out[3] = rhob * ut3;
  out[4] = pb / T(g - 1.0) + T(0.5) * rhob * (ub * ub + ut2 * ut2 + ut3 * ut3);
}

// isothermal no-slip wall ghost, bottom (side 0) or top (side 1)
template <class T>
__device__ void wall_state(const T wc[5], int side, const BcDesc& bc, T out[5]) {
  const T rho = wc[0];
  const T u0 = wc[1] / rho, u1 = wc[2] / rho, u2 = wc[3] / rho;
  const T k2 = T(0.5) * (u0 * u0 + u1 * u1 + u2 * u2);
  const T e = wc[4] / rho - k2;
  const T eg = T(2.0 * bc.wall_e[side]) - e;
  out[0] = rho;
  out[1] = -wc[1];
  out[2] = -wc[2];
  out[3] = -wc[3];
  out[4] = rho * (eg + k2);
}

struct Pad {
  int ix, iy;          // ghost widths in x and y (0 or 1)
  int nxp, nyp;        // padded sizes
  long long planep, cellsp;
};

__device__ __forceinline__ Pad pad_of(const GridDesc& g, const BcDesc& bc) {
  Pad p;
  p.ix = bc.inout;
  p.iy = bc.walls;
  p.nxp = g.nx + 2 * p.ix;
  p.nyp = g.ny + 2 * p.iy;
  p.planep = (long long)p.nxp * p.nyp;
  p.cellsp = p.planep * g.nz;
  return p;
}

// Row kernels: a warp takes a row (a component's y-row of one plane), so that the row's place
// is worked out once and lanes move along x.  (A thread per element spent most of its time on
// the 64-bit divisions that split its index: 10.3 us for the field of a 96x48x48 duct.)  Of
// rows up to 16 long it takes as many as its lanes hold.
constexpr int BR = 8;   // warps per CTA
__host__ __device__ __forceinline__ int rows_per_warp(int width) { return width > 16 ? 1 : 32 / width; }
// this lane's place in a warp's rows: which one (rows_per_warp for the lanes left over) and x
struct RowLane {
  int row, x;
};
__device__ __forceinline__ RowLane row_lane(int width, int rpw) {
  const int lane = threadIdx.x & 31;
  RowLane l;
  l.row = rpw == 1 ? 0 : lane / width;
  l.x = lane - l.row * width;
  return l;
}

// padded fields (interior copied and converted, ghosts zero), ncomp components per box:
// dst = cvt(scale src); dst2 (may be null) = src unscaled in FP64
template <class TO, class TI>
__global__ void __launch_bounds__(32 * BR) k_bc_embed(GridDesc g, BcDesc bc, int ncomp, double scale,
                                                      const TI* __restrict__ src, TO* __restrict__ dst,
                                                      double* __restrict__ dst2) {
  pdl_enter();
  const Pad P = pad_of(g, bc);
  const long long rows = (long long)P.nyp * g.nz * ncomp * g.batch;
  const int rpw = rows_per_warp(P.nxp);
  const RowLane l = row_lane(P.nxp, rpw);
  if (l.row >= rpw) return;
  for (long long r = ((long long)blockIdx.x * BR + (threadIdx.x >> 5)) * rpw + l.row; r < rows;
       r += (long long)gridDim.x * BR * rpw) {
    const long long q = r / P.nyp;                       // (box, component, plane)
    const int y = (int)(r - q * P.nyp) - P.iy;
    const bool in = y >= 0 && y < g.ny;
    const TI* s = src + q * g.plane + (long long)(in ? y : 0) * g.nx;
    TO* d = dst + r * P.nxp;
    for (int xp = l.x; xp < P.nxp; xp += 32) {
      const int x = xp - P.ix;
      const double v = in && x >= 0 && x < g.nx ? (double)s[x] : 0.0;
      d[xp] = cvt<TO>(scale * v);
      if (dst2) dst2[r * P.nxp + xp] = v;
    }
  }
}

// interior of a padded field
template <class TO, class TI>
__global__ void __launch_bounds__(32 * BR) k_bc_crop(GridDesc g, BcDesc bc, int ncomp, const TI* __restrict__ src,
                                                     TO* __restrict__ dst) {
  pdl_enter();
  const Pad P = pad_of(g, bc);
  const long long rows = (long long)g.ny * g.nz * ncomp * g.batch;
  const int rpw = rows_per_warp(g.nx);
  const RowLane l = row_lane(g.nx, rpw);
  if (l.row >= rpw) return;
  for (long long r = ((long long)blockIdx.x * BR + (threadIdx.x >> 5)) * rpw + l.row; r < rows;
       r += (long long)gridDim.x * BR * rpw) {
    const long long q = r / g.ny;
    const int y = (int)(r - q * g.ny);
    const TI* s = src + q * P.planep + (long long)(y + P.iy) * P.nxp + P.ix;
    for (int x = l.x; x < g.nx; x += 32) dst[r * g.nx + x] = (TO)s[x];
  }
}

template <class T>
__device__ __forceinline__ void load5(const T* f, long long o, long long stride, T v[5]) {
#pragma unroll
  for (int k = 0; k < 5; ++k) v[k] = f[o + k * stride];
}

// the ghost layer of a padded state field, from its interior boundary cells
template <class T>
__global__ void k_bc_ghosts(GridDesc g, BcDesc bc, T* __restrict__ W) {
  pdl_enter();
  const Pad P = pad_of(g, bc);
  // ghost cells per plane: the x columns' interior rows, then the y rows' full width
  const int nxg = P.ix ? 2 * g.ny : 0, nyg = P.iy ? 2 * P.nxp : 0;
  const long long per = (long long)(nxg + nyg) * g.nz;
  const long long n = per * g.batch;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long b = i / per, r = i - b * per;
    const int z = (int)(r / (nxg + nyg));
    int j = (int)(r - (long long)z * (nxg + nyg));
    const long long box = b * 5 * P.cellsp + (long long)z * P.planep;
    auto at = [&](int xp, int yp) { return box + (long long)yp * P.nxp + xp; };
    T wc[5], gs[5];
    long long dst;
    if (j < nxg) {
      // inflow (side 0) or outflow (side 1) column at interior row y
      const int side = j / g.ny, y = j - side * g.ny;
      const int xc = side == 0 ? P.ix : P.ix + g.nx - 1;
      load5(W, at(xc, y + P.iy), P.cellsp, wc);
      char_state<T>(wc, side, bc, gs);
      dst = at(side == 0 ? 0 : P.nxp - 1, y + P.iy);
    } else {
      // wall rows over the full padded width; at a corner, the wall ghost of the
      // inflow or outflow ghost of the corner cell
      j -= nxg;
      const int side = j / P.nxp, xp = j - side * P.nxp;
      const int yc = side == 0 ? P.iy : P.iy + g.ny - 1;
      const int x = xp - P.ix;
      if (x >= 0 && x < g.nx) {
        load5(W, at(xp, yc), P.cellsp, wc);
      } else {
        T wi[5];
        load5(W, at(x < 0 ? P.ix : P.ix + g.nx - 1, yc), P.cellsp, wi);
        char_state<T>(wi, x < 0 ? 0 : 1, bc, wc);
      }
      wall_state<T>(wc, side, bc, gs);
      dst = at(xp, side == 0 ? 0 : P.nyp - 1);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) W[dst + k * P.cellsp] = gs[k];
  }
}

// d = J^T h, J the Jacobian of a wall ghost with respect to the cell wc it was built from:
// the ghost is (rho, -m, 2 e_w rho - rho E + |m|^2 / rho).
__device__ __forceinline__ void wall_pullback(const double wc[5], int side, const BcDesc& bc, const double h[5],
                                              double d[5]) {
  const double ir = 1.0 / wc[0];
  const double u[3] = {wc[1] * ir, wc[2] * ir, wc[3] * ir};
  d[0] = h[0] + h[4] * (2.0 * bc.wall_e[side] - (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));
#pragma unroll
  for (int k = 0; k < 3; ++k) d[1 + k] = 2.0 * u[k] * h[4] - h[1 + k];
  d[4] = -h[4];
}

// d = J^T h, J the Jacobian of a characteristic ghost with respect to the cell wc it was
// built from: char_state reversed step by step.  The ghost's density is written
// rho_b = rho_0 (c_b / c_0)^(2/(gamma-1)), its entropy being that of (rho_0, c_0): the
// cell's at the outflow, the far field's at the inflow.
__device__ __forceinline__ void char_pullback(const double wc[5], int side, const BcDesc& bc, const double h[5],
                                              double d[5]) {
  const double g = bc.gamma, gm1 = g - 1.0, k = 2.0 / gm1;
  const double rho = wc[0], ir = 1.0 / rho;
  const double u[3] = {wc[1] * ir, wc[2] * ir, wc[3] * ir};
  const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const double p = gm1 * (wc[4] - 0.5 * rho * uu);
  const double c = sqrt(g * p * ir);
  const bool out = side == 1;
  const double Rp = out ? u[0] + k * c : bc.far[1] + k * bc.cf;
  const double Rm = out ? bc.far[1] - k * bc.cf : u[0] - k * c;
  const double ub = 0.5 * (Rp + Rm), cb = 0.25 * gm1 * (Rp - Rm);
  const double t2 = out ? u[1] : bc.far[2], t3 = out ? u[2] : bc.far[3];
  const double r0 = out ? rho : bc.far[0], c0 = out ? c : bc.cf;
  const double x = cb / c0, x2 = x * x;
  // (x^2)^(1/(gamma-1)); gamma = 1.4 gives |x|^5
  const double rb = r0 * (fabs(k - 5.0) < 1e-12 ? x2 * x2 * fabs(x) : pow(x2, 0.5 * k));
  const double igg = 1.0 / (g * gm1);
  const double rbb = h[0] + h[1] * ub + h[2] * t2 + h[3] * t3 +
                     h[4] * (cb * cb * igg + 0.5 * (ub * ub + t2 * t2 + t3 * t3));
  const double ubb = rb * (h[1] + h[4] * ub);
  const double krb = k * rb * rbb;
  const double cbb = 2.0 * h[4] * rb * cb * igg + krb / cb;
  const double Rb = out ? 0.5 * ubb + 0.25 * gm1 * cbb : 0.5 * ubb - 0.25 * gm1 * cbb;
  double us[3] = {Rb, 0.0, 0.0}, rs = 0.0;
  double cs = out ? k * Rb : -k * Rb;
  if (out) {
    us[1] = rb * (h[2] + h[4] * t2);
    us[2] = rb * (h[3] + h[4] * t3);
    rs = rbb * rb * ir;
    cs -= krb / c;
  }
  // c^2 = gamma p / rho, then (rho, u, p) to conservative variables
  const double ps = cs * c / (2.0 * p);
  rs -= 0.5 * cs * c * ir;
  d[0] = rs - (us[0] * u[0] + us[1] * u[1] + us[2] * u[2]) * ir + 0.5 * gm1 * uu * ps;
#pragma unroll
  for (int j = 0; j < 3; ++j) d[1 + j] = us[j] * ir - gm1 * u[j] * ps;
  d[4] = gm1 * ps;
}

// The boundary epilogue of one transposed stage on a bounded box, per interior cell:
//   g   = gp(c) + the ghosts' outputs pulled back + L_nu a (boundary faces closed)
// then, as the periodic adjoint stage does:
//   mode 0 (transposed residual only):  out = g
//   mode 1 (a Runge-Kutta stage):        Gs = (first ? 0 : G) + g; G = Gs (not last);
//       a_next = cl lam + cg g + cs Gs (not last); lam_out = lam + Gs (last);
//       sbar += a (when sbar != null); seed = a_next in the padded stage type, the next
//       stage's input (its ghosts stay zero)
// gp: the transposed product on the padded box (FP64); W: the padded stage state
// (ghost inputs); A, sa: the stage's seed a = sa A (unpadded FP64).
//
// The pull-backs take a few hundred FP64 instructions, which GB300 issues at 1/64 of the
// FP32 rate, and only the cells next to a boundary need them: the first nbb CTAs take
// those cells, packed so that all 32 lanes of a warp have one, and the other CTAs the
// cells of whole rows, leaving out the packed ones.  With every cell in one grid, each
// row's end cells held two of its three warps for the whole pull-back: 931 us per stage of
// a 96x48x48 duct (a primal and an adjoint step: 4070 us, 505 us with this split and the Laplacian below).
struct EpiArgs {
  const double* gp;
  const double* A;
  double sa, snus[3], hi2[3];   // sa, sa nu factors (rho, rho u, rho E), 1 / (2 dx^2)
  int mode, first, last;
  const double* lam;
  double* G;
  double cl, cg, cs;
  double* a_next;
  double* out;
  double* sbar;
};

template <class CT, class NU>
__device__ __forceinline__ void epilogue_cell(const GridDesc& g, const Pad& P, const EpiArgs& e,
                                              const NU* __restrict__ nu, CT* __restrict__ seed, int b, int x, int y,
                                              int z, double gc[5]) {
  const long long r = (long long)z * g.plane + (long long)y * g.nx + x;
  const long long o = (long long)b * 5 * g.cells + r;
  const double sa = e.sa;
  double A[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) A[k] = e.A[o + k * g.cells];
  if (nu) {
    // L_nu a = sa sum_q F_q (A_q - A), F_q = (nu + nu_q) / (2 dx_q^2), zero at closed faces:
    // FP64 operations bind this kernel, so the weights are formed once per cell and the
    // seed's scale is applied once per component
    const NU* nb = nu + (long long)b * g.cells;
    long long q[6] = {r + (x == 0 ? g.nx - 1 : -1), r + (x == g.nx - 1 ? 1 - g.nx : 1),
                      r + (long long)(y == 0 ? g.ny - 1 : -1) * g.nx, r + (long long)(y == g.ny - 1 ? 1 - g.ny : 1) * g.nx,
                      r + (z == 0 ? g.nz - 1 : -1) * g.plane, r + (z == g.nz - 1 ? 1 - g.nz : 1) * g.plane};
    const bool closed[6] = {P.ix && x == 0, P.ix && x == g.nx - 1, P.iy && y == 0, P.iy && y == g.ny - 1, false, false};
    const NU nc = nb[r];
    NU nq[6];
    bool sub = subnormal(nc);   // one test for all seven
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      nq[d] = nb[q[d]];
      sub = sub || subnormal(nq[d]);
    }
    double F[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) F[d] = closed[d] ? 0.0 : (widen(nc) + widen(nq[d])) * e.hi2[d >> 1];
    if (sub) {
#pragma unroll
      for (int d = 0; d < 6; ++d) F[d] = closed[d] ? 0.0 : ((double)nc + (double)nq[d]) * e.hi2[d >> 1];
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const double* Ak = e.A + (long long)b * 5 * g.cells + (long long)k * g.cells;
      double L = 0.0;
#pragma unroll
      for (int d = 0; d < 6; ++d) L += F[d] * (Ak[q[d]] - A[k]);
      gc[k] += e.snus[k == 0 ? 0 : (k == 4 ? 2 : 1)] * L;
    }
  }
  const long long op = (long long)b * 5 * P.cellsp + (long long)z * P.planep + (long long)(y + P.iy) * P.nxp + x + P.ix;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const long long ok = o + (long long)k * g.cells;
    if (e.mode == 0) {
      e.out[ok] = gc[k];
      continue;
    }
    const double Gs = (e.first ? 0.0 : e.G[ok]) + gc[k];
    if (e.last) {
      e.out[ok] = e.lam[ok] + Gs;
    } else {
      e.G[ok] = Gs;
      double an = e.cl * e.lam[ok] + e.cg * gc[k];
      if (e.cs != 0.0) an += e.cs * Gs;
      e.a_next[ok] = an;
      seed[op + (long long)k * P.cellsp] = cvt<CT>(an);
    }
    if (e.sbar) e.sbar[ok] += sa * A[k];
  }
}

constexpr int BBT = 64;   // packed boundary cells per CTA: two of its warps, so that they spread over the SMs

template <class CT, class NU>
__global__ void __launch_bounds__(32 * BR) k_bc_adj_epilogue(GridDesc g, BcDesc bc, EpiArgs e,
                                                             const CT* __restrict__ W, const NU* __restrict__ nu,
                                                             CT* __restrict__ seed, int nbb) {
  pdl_enter();
  const Pad P = pad_of(g, bc);
  if ((int)blockIdx.x >= nbb) {
    // 32-cell pieces of rows, one per warp (of rows up to 16 long several), without the cells
    // next to a boundary
    const int pieces = (g.nx + 31) / 32, rpw = rows_per_warp(g.nx);
    const RowLane l = row_lane(g.nx, rpw);
    if (l.row >= rpw) return;
    const long long jobs = (long long)pieces * g.ny * g.nz * g.batch, step = (long long)(gridDim.x - nbb) * BR * rpw;
    for (long long j = ((long long)(blockIdx.x - nbb) * BR + (threadIdx.x >> 5)) * rpw + l.row; j < jobs; j += step) {
      const long long r = j / pieces;
      const int x = (int)(j - r * pieces) * 32 + l.x;
      const long long q = r / g.ny;
      const int y = (int)(r - q * g.ny);
      const int z = (int)(q % g.nz), b = (int)(q / g.nz);
      if (x >= g.nx || (P.iy && (y == 0 || y == g.ny - 1)) || (P.ix && (x == 0 || x == g.nx - 1))) continue;
      const double* gr = e.gp + (long long)b * 5 * P.cellsp + (long long)z * P.planep +
                         (long long)(y + P.iy) * P.nxp + P.ix;
      double gc[5];
      load5(gr, x, P.cellsp, gc);
      epilogue_cell<CT, NU>(g, P, e, nu, seed, b, x, y, z, gc);
    }
    return;
  }
  if (threadIdx.x >= BBT) return;
  // cells next to a boundary of one plane: the inflow and outflow columns (an only column
  // is both), then the wall rows without the columns' cells
  const int ncol = P.ix ? (g.nx > 1 ? 2 : 1) : 0, nrow = P.iy ? (g.ny > 1 ? 2 : 1) : 0;
  const int rw = g.nx - ncol;                            // cells of a wall row outside the columns
  const int per = ncol * g.ny + nrow * rw;
  const long long i = (long long)blockIdx.x * BBT + threadIdx.x;
  if (i >= (long long)per * g.nz * g.batch) return;
  const long long q = i / per;
  const int z = (int)(q % g.nz), b = (int)(q / g.nz);
  int j = (int)(i - q * per), x, y;
  if (j < ncol * g.ny) {
    x = j < g.ny ? 0 : g.nx - 1;
    y = j < g.ny ? j : j - g.ny;
  } else {
    j -= ncol * g.ny;
    y = j < rw ? 0 : g.ny - 1;
    x = (j < rw ? j : j - rw) + (P.ix ? 1 : 0);
  }
  const long long boxp = (long long)b * 5 * P.cellsp + (long long)z * P.planep;
  auto atp = [&](int xp, int yp) { return boxp + (long long)yp * P.nxp + xp; };
  auto wget = [&](long long o, double v[5]) {
#pragma unroll
    for (int k = 0; k < 5; ++k) v[k] = (double)W[o + k * P.cellsp];
  };
  const int xp = x + P.ix, yp = y + P.iy;
  double gc[5], h[5], d[5], wc[5];
  load5(e.gp, atp(xp, yp), P.cellsp, gc);
  wget(atp(xp, yp), wc);
  // wall rows first: a ghost row's output goes to the row it was built from
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    if (!P.iy || y != (side == 0 ? 0 : g.ny - 1)) continue;
    load5(e.gp, atp(xp, side == 0 ? 0 : P.nyp - 1), P.cellsp, h);
    wall_pullback(wc, side, bc, h, d);
#pragma unroll
    for (int k = 0; k < 5; ++k) gc[k] += d[k];
  }
  // then the inflow and outflow columns: each column ghost's output, with its wall
  // ghosts' outputs pulled back onto it at the first and last rows
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    if (!P.ix || x != (side == 0 ? 0 : g.nx - 1)) continue;
    const int xg = side == 0 ? 0 : P.nxp - 1;
    load5(e.gp, atp(xg, yp), P.cellsp, h);
#pragma unroll 1
    for (int ws = 0; ws < 2; ++ws) {
      if (!P.iy || y != (ws == 0 ? 0 : g.ny - 1)) continue;
      double hc[5], wg[5];
      load5(e.gp, atp(xg, ws == 0 ? 0 : P.nyp - 1), P.cellsp, hc);
      wget(atp(xg, yp), wg);   // the column ghost the corner was built from
      wall_pullback(wg, ws, bc, hc, d);
#pragma unroll
      for (int k = 0; k < 5; ++k) h[k] += d[k];
    }
    char_pullback(wc, side, bc, h, d);
#pragma unroll
    for (int k = 0; k < 5; ++k) gc[k] += d[k];
  }
  epilogue_cell<CT, NU>(g, P, e, nu, seed, b, x, y, z, gc);
}

constexpr int BB = 64;   // ghost cells per CTA: few, so that they spread over the SMs

unsigned blocks_for(long long n) {
  long long b = (n + BB - 1) / BB;
  if (b > 152 * 16) b = 152 * 16;
  return (unsigned)(b > 0 ? b : 1);
}

}  // namespace

long long bc_padded_cells(const GridDesc& g, const BcDesc& bc) {
  return (long long)(g.nx + 2 * bc.inout) * (g.ny + 2 * bc.walls) * g.nz;
}

// CTAs of the row kernels: BR warps' rows of this width each, at most sixteen per SM (the rest
// by the stride)
static unsigned blocks_for_rows(long long rows, int width) {
  const long long per = (long long)BR * rows_per_warp(width), b = (rows + per - 1) / per;
  return (unsigned)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

template <class TO, class TI>
cudaError_t launch_bc_embed(const GridDesc& g, const BcDesc& bc, int ncomp, double scale, const TI* src, TO* dst,
                            cudaStream_t st, double* dst2) {
  const long long rows = (long long)(g.ny + 2 * bc.walls) * g.nz * ncomp * g.batch;
  count_launch();
  return launch_pdl(k_bc_embed<TO, TI>, dim3(blocks_for_rows(rows, g.nx + 2 * bc.inout)), dim3(32 * BR), 0, st, g, bc, ncomp, scale, src, dst,
                    dst2);
}

template <class TO, class TI>
cudaError_t launch_bc_crop(const GridDesc& g, const BcDesc& bc, int ncomp, const TI* src, TO* dst, cudaStream_t st) {
  const long long rows = (long long)g.ny * g.nz * ncomp * g.batch;
  count_launch();
  return launch_pdl(k_bc_crop<TO, TI>, dim3(blocks_for_rows(rows, g.nx)), dim3(32 * BR), 0, st, g, bc, ncomp, src, dst);
}

template <class T>
cudaError_t launch_bc_ghosts(const GridDesc& g, const BcDesc& bc, T* W, cudaStream_t st) {
  const long long per = (long long)((bc.inout ? 2 * g.ny : 0) + (bc.walls ? 2 * (g.nx + 2 * bc.inout) : 0)) * g.nz;
  count_launch();
  // FP64 ghosts are some hundred FP64 instructions a cell, so the CTAs have to spread evenly over
  // the SMs.  As a dependent launch they are placed while the stage kernel before them, whose two
  // CTAs fill an SM's registers, is draining: on the SMs that fall free first, four and more
  // together.  A primal step of 96x48x48 cells with inflow, outflow and walls took 859 us so, of
  // 20x64x64 cells 666 us; 707 and 413 us launched after it.  (The 2D stage kernels leave room:
  // 128x128 146 us as a dependent launch, 154 us after it.)
  if (sizeof(T) == 8 && g.nz > 1) {
    k_bc_ghosts<T><<<blocks_for(per * g.batch), BB, 0, st>>>(g, bc, W);
    return cudaGetLastError();
  }
  return launch_pdl(k_bc_ghosts<T>, dim3(blocks_for(per * g.batch)), dim3(BB), 0, st, g, bc, W);
}

template <class CT, class NU>
cudaError_t launch_bc_adj_epilogue(const GridDesc& g, const BcDesc& bc, const BcEpilogue& e, const double* gp,
                                   const CT* W, const NU* nu, CT* seed, cudaStream_t st) {
  EpiArgs a;
  a.gp = gp; a.A = e.A; a.sa = e.sa;
  for (int k = 0; k < 3; ++k) { a.snus[k] = e.sa * e.nus[k]; a.hi2[k] = 0.5 * e.i2[k]; }
  a.mode = e.mode; a.first = e.first; a.last = e.last;
  a.lam = e.lam; a.G = e.G; a.cl = e.cl; a.cg = e.cg; a.cs = e.cs;
  a.a_next = e.a_next; a.out = e.out; a.sbar = e.sbar;
  const long long ncol = bc.inout ? (g.nx > 1 ? 2 : 1) : 0, nrow = bc.walls ? (g.ny > 1 ? 2 : 1) : 0;
  const long long cells = (ncol * g.ny + nrow * (g.nx - ncol)) * g.nz * g.batch;   // next to a boundary
  const long long nbb = (cells + BBT - 1) / BBT;
  if (nbb > (1LL << 30)) return cudaErrorInvalidConfiguration;
  const unsigned rows = blocks_for_rows((long long)((g.nx + 31) / 32) * g.ny * g.nz * g.batch, g.nx);
  count_launch();
  return launch_pdl(k_bc_adj_epilogue<CT, NU>, dim3((unsigned)nbb + rows), dim3(32 * BR), 0, st, g, bc, a, W, nu, seed,
                    (int)nbb);
}

template cudaError_t launch_bc_embed<double, double>(const GridDesc&, const BcDesc&, int, double, const double*,
                                                     double*, cudaStream_t, double*);
template cudaError_t launch_bc_embed<float, double>(const GridDesc&, const BcDesc&, int, double, const double*,
                                                    float*, cudaStream_t, double*);
template cudaError_t launch_bc_crop<double, double>(const GridDesc&, const BcDesc&, int, const double*, double*,
                                                    cudaStream_t);
template cudaError_t launch_bc_crop<float, float>(const GridDesc&, const BcDesc&, int, const float*, float*,
                                                  cudaStream_t);
template cudaError_t launch_bc_ghosts<double>(const GridDesc&, const BcDesc&, double*, cudaStream_t);
template cudaError_t launch_bc_ghosts<float>(const GridDesc&, const BcDesc&, float*, cudaStream_t);
template cudaError_t launch_bc_adj_epilogue<double, float>(const GridDesc&, const BcDesc&, const BcEpilogue&,
                                                           const double*, const double*, const float*, double*, cudaStream_t);
template cudaError_t launch_bc_adj_epilogue<double, double>(const GridDesc&, const BcDesc&, const BcEpilogue&,
                                                            const double*, const double*, const double*, double*, cudaStream_t);
template cudaError_t launch_bc_adj_epilogue<float, float>(const GridDesc&, const BcDesc&, const BcEpilogue&,
                                                          const double*, const float*, const float*, float*, cudaStream_t);

}  // namespace ns
