// Learned adjoint-viscosity closure: per-cell features, BF16 tensor-core inference and
// a BF16 training step with an FP32 Adam master copy.
//
// The stabilised adjoint of section "Energy analysis" adds div(lambda sigma_1 grad w_hat)
// with a hand-tuned constant lambda (its automatic estimation is left open in the
// conclusion).  Here lambda(x) = dx^2 softplus(MLP(f(x))) per cell, so that
//   nu(x) = kappa dx^2 sigma_1(x) softplus(MLP(f(x)))
// with a global factor kappa.  Network: 14 -> 64 -> 64 -> 1, GELU, softplus; weights
// BF16, accumulation FP32, hidden activations rounded to BF16 between the two tensor-core
// layers, the last layer an FP32 dot product.
//
// Features f (14 per cell, stored padded to 16 floats): v = S(q_bar)(q - q_bar) / c_bar
// (symmetrised variables about the box-mean primitive state, section "Symmetrization")
// and the 9 central-difference entries of grad u times L / c_bar (L = 1).
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "ns_common.cuh"
#include "ns_kernels.h"
#include "ns_mlp.h"

namespace ns {

namespace cg = cooperative_groups;

namespace {

constexpr int RB = 256;
constexpr int RGM = 296;

// a state value as float: the FP64 state rounded (d2f), or the float mirror as it is
// (the mirror holds exactly d2f of the state, so both give the same bits)
__device__ __forceinline__ float ldf(const double* p, size_t o) { return d2f(p[o]); }
__device__ __forceinline__ float ldf(const float* p, size_t o) { return p[o]; }

// ------------------------------------------------------------------------------------
// box means of (rho, u1, u2, u3, p): FP32 per cell, sums of FP64's precision or better,
// deterministic
// ------------------------------------------------------------------------------------
template <class TIN>
__device__ __forceinline__ void mean_terms(const TIN* __restrict__ w, size_t o, long long cells, float gamma, float x[5]) {
  const float r = ldf(w, o);
  const float ir = 1.0f / r;
  const float u0 = ldf(w, o + cells) * ir, u1 = ldf(w, o + 2 * cells) * ir, u2 = ldf(w, o + 3 * cells) * ir;
  x[0] = r;
  x[1] = u0;
  x[2] = u1;
  x[3] = u2;
  x[4] = (gamma - 1.0f) * (ldf(w, o + 4 * cells) - 0.5f * r * (u0 * u0 + u1 * u1 + u2 * u2));
}

// s = a + b and its rounding error (Knuth's two-sum, exact while nothing overflows)
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}
// A float sum with the errors of its additions summed apart, and theirs again (cascaded
// summation: Rump, Ogita and Oishi's SumK with K = 3): the rounding of lo, below 2^-70 of the
// terms' magnitude, is all that is lost.
struct Sum3 {
  float hi = 0.0f, mid = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float x) {
    float e, f;
    hi = two_sum(hi, x, e);
    mid = two_sum(mid, e, f);
    lo = __fadd_rn(lo, f);
  }
  __device__ __forceinline__ void add(const Sum3& x) {
    float f;
    add(x.hi);
    mid = two_sum(mid, x.mid, f);
    lo = __fadd_rn(lo, __fadd_rn(x.lo, f));
  }
};
// own += the other half's value, of the two a lane holds: the lanes without the bit o of
// their number keep a, the others b
__device__ __forceinline__ Sum3 halve(const Sum3& a, const Sum3& b, int o) {
  const bool up = (threadIdx.x & o) != 0;
  Sum3 own = up ? b : a, away = up ? a : b, in;
  in.hi = __shfl_xor_sync(0xffffffffu, away.hi, o);
  in.mid = __shfl_xor_sync(0xffffffffu, away.mid, o);
  in.lo = __shfl_xor_sync(0xffffffffu, away.lo, o);
  own.add(in);
  return own;
}

// The block's sums of the terms in FP64, for values beyond what float sums hold
template <class TIN>
__device__ __noinline__ void box_sums_f64(const TIN* __restrict__ w, size_t box, long long cells, float gamma,
                                          double (*sh)[RB / 32]) {
  double acc[5] = {0, 0, 0, 0, 0};
  for (long long i = (long long)blockIdx.x * RB + threadIdx.x; i < cells; i += (long long)gridDim.x * RB) {
    float x[5];
    mean_terms(w, box + i, cells, gamma, x);
    for (int q = 0; q < 5; ++q) acc[q] += (double)x[q];
  }
  for (int q = 0; q < 5; ++q) {
    for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    if ((threadIdx.x & 31) == 0) sh[q][threadIdx.x >> 5] = acc[q];
  }
}

// GB300 issues FP64 additions at 1/64 of the FP32 rate, and a thread has some three cells, so
// the sums stay in floats (Sum3) until a warp has one value per term: the butterfly across the
// warp halves the terms a lane keeps (3, 2, 1, then 1 and 1 for lanes of the same term: eight
// additions in place of 25), and each term's lane makes the FP64 value.  The block falls back
// to FP64 where a float sum is not finite.  Means and features of 1.77 M cells in eight boxes
// take 66.5 us, of 256x128x128 cells 183 us, at five CTAs per SM (48 registers: a cell's five
// loads at once); 70.0 and 217 us at six; 66.3 and 191 us with sums in float pairs, which hold
// 2^-44 of the terms' magnitude.
template <class TIN>
__global__ void __launch_bounds__(RB, 5) k_box_means(GridDesc g, float gamma, const TIN* __restrict__ w,
                                                  double* partial) {
  pdl_enter();
  __shared__ double sh[5][RB / 32];
  const int b = blockIdx.y;
  const size_t box = (size_t)b * 5 * g.cells;
  Sum3 s[5];
  for (long long i = (long long)blockIdx.x * RB + threadIdx.x; i < g.cells; i += (long long)gridDim.x * RB) {
    float x[5];
    mean_terms(w, box + i, g.cells, gamma, x);
#pragma unroll
    for (int q = 0; q < 5; ++q) s[q].add(x[q]);
  }
  const Sum3 z;
  const Sum3 t0 = halve(s[0], s[3], 16), t1 = halve(s[1], s[4], 16), t2 = halve(s[2], z, 16);
  const Sum3 v0 = halve(t0, t2, 8), v1 = halve(t1, z, 8);
  Sum3 r = halve(v0, v1, 4);
  r = halve(r, r, 2);
  r = halve(r, r, 1);
  // the term of this lane's sum: the first keeps above had (0, 1, 2) or (3, 4, -), then
  // (0, 1) or (2, -) of those, then one
  const int q = ((threadIdx.x & 16) ? 3 : 0) + ((threadIdx.x & 8) ? 2 : 0) + ((threadIdx.x & 4) ? 1 : 0);
  const bool term = (threadIdx.x & 3) == 0 && (threadIdx.x & 12) != 12 && q < 5;
  if (term) sh[q][threadIdx.x >> 5] = f2d(r.hi) + (f2d(r.mid) + f2d(r.lo));
  if (__syncthreads_or(term && !(fabsf(r.hi) < INFINITY && fabsf(r.mid) < INFINITY && fabsf(r.lo) < INFINITY))) {
    box_sums_f64(w, box, g.cells, gamma, sh);
    __syncthreads();
  }
  if (threadIdx.x < 5) {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < RB / 32; ++i) t += sh[threadIdx.x][i];
    partial[((size_t)b * 5 + threadIdx.x) * gridDim.x + blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(RB) k_box_means_final(int nblk, double inv_cells, const double* partial,
                                                        double* qbar) {
  pdl_enter();
  __shared__ double sh[RB];
  const int b = blockIdx.x / 5, q = blockIdx.x % 5;
  double s = 0.0;
  for (int i = threadIdx.x; i < nblk; i += RB) s += partial[((size_t)b * 5 + q) * nblk + i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int k = RB / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) sh[threadIdx.x] += sh[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) qbar[b * 5 + q] = sh[0] * inv_cells;
}

// ------------------------------------------------------------------------------------
// features
// ------------------------------------------------------------------------------------
// One CTA takes TX x FY columns and a range of planes (march_range) and keeps 1/rho and
// rho u of three planes with a one-cell halo in a shared-memory ring, so each cell's state is loaded
// and divided once per tile instead of seven times; a warp's 32 x 16 features go out
// through shared memory as whole lines.  1.77 M cells in eight boxes: 115 us with a thread
// per cell reading its six neighbours, 42 us now (27 us at the memory's rate).
namespace fk {
constexpr int FY = 8;
constexpr int NT = TX * FY;
constexpr int SY = FY + 2;
constexpr int SP = SX * SY;
constexpr int OS = 20;   // padded row of the output staging (16 floats and a bank shift)
static_assert(SP <= 2 * NT, "a plane must fit two load rounds");
constexpr size_t smem = sizeof(float) * (3 * 4 * SP + NT * OS);
}  // namespace fk

template <class TIN>
__global__ void __launch_bounds__(fk::NT) k_features(GridDesc g, Coef<float> c, const TIN* __restrict__ w,
                                                     const double* qbar, float* __restrict__ feat) {
  pdl_enter();
  using namespace fk;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* sQ = reinterpret_cast<float*>(smem_raw);   // [3][4][SP]: 1/rho, rho u1, rho u2, rho u3
  float* sO = sQ + 3 * 4 * SP;                       // [NT][OS]
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX, lane = tid & 31;
  int b, x0, y0, kz0, kz1;
  if (!march_range<TX, FY>(g, b, x0, y0, kz0, kz1)) return;
  const int gx = x0 + tx, gy = y0 + ty;
  const bool valid = gx < g.nx && gy < g.ny;
  const int cp = valid ? gy * g.nx + gx : 0;
  const size_t box = (size_t)b * 5 * g.cells, fc = (size_t)g.cells;
  int ho[2];
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int t = tid + it * NT, ly = t / SX, lx = t - ly * SX;
    ho[it] = t < SP ? wrap(y0 + ly - 1, g.ny) * g.nx + wrap(x0 + lx - 1, g.nx) : 0;
  }
  auto load = [&](float (&q)[2][4], int k) {
    const size_t pb = box + (size_t)wrap(k, g.nz) * g.plane;
#pragma unroll
    for (int it = 0; it < 2; ++it)
      if (tid + it * NT < SP) {
#pragma unroll
        for (int v = 0; v < 4; ++v) q[it][v] = ldf(w, pb + v * fc + ho[it]);
      }
  };
  auto store = [&](const float (&q)[2][4], int slot) {
    float* P = sQ + slot * 4 * SP;
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int t = tid + it * NT;
      if (t < SP) {
        P[t] = 1.0f / q[it][0];
        P[SP + t] = q[it][1];
        P[2 * SP + t] = q[it][2];
        P[3 * SP + t] = q[it][3];
      }
    }
  };
  auto slot = [&](int k) { return (k - kz0 + 1) % 3; };
  {
    float q0[2][4], q1[2][4], q2[2][4];
    load(q0, kz0 - 1);
    load(q1, kz0);
    load(q2, kz0 + 1);
    store(q0, slot(kz0 - 1));
    store(q1, slot(kz0));
    store(q2, slot(kz0 + 1));
  }
  const float gam = c.gamma, gm1 = c.gm1;
  const float rb = (float)qbar[b * 5 + 0], pb = (float)qbar[b * 5 + 4];
  float ub[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) ub[k] = (float)qbar[b * 5 + 1 + k];
  const float cb = sqrtf(gam * pb / rb);
  const float icb = rsqrtf(gam * pb / rb);
  const float f0r = cb / (sqrtf(gam) * rb);
  const float f4r = -cb / (rb * sqrtf(gam * gm1)), f4p = sqrtf(gam / gm1) / (rb * cb);
  __syncthreads();
  const int ic = (ty + 1) * SX + tx + 1;
  for (int k = kz0; k < kz1; ++k) {
    const bool more = k + 1 < kz1;
    float qf[2][4];
    if (more) load(qf, k + 2);
    const size_t o = box + (size_t)k * g.plane + cp;
    const float rho = ldf(w, o), E = ldf(w, o + 4 * fc);
    const float* P0 = sQ + slot(k) * 4 * SP;
    const float* Pm = sQ + slot(k - 1) * 4 * SP;
    const float* Pp = sQ + slot(k + 1) * 4 * SP;
    const float ir = P0[ic], mo[3] = {P0[SP + ic], P0[2 * SP + ic], P0[3 * SP + ic]};
    const float u[3] = {mo[0] * ir, mo[1] * ir, mo[2] * ir};
    // p - p_bar; the roundings of these sums are written out (so that the features do not
    // change with the code around them)
    const float uu = __fmaf_rn(u[2], u[2], __fmaf_rn(u[0], u[0], __fmul_rn(u[1], u[1])));
    const float dp = __fmaf_rn(gm1, __fmaf_rn(-__fmul_rn(0.5f, rho), uu, E), -pb);
    float f[16];
    f[0] = f0r * (rho - rb) * icb;
#pragma unroll
    for (int q = 0; q < 3; ++q) f[1 + q] = __fsub_rn(u[q], ub[q]) * icb;
    f[4] = __fmaf_rn(f4p, dp, __fmul_rn(f4r, rho - rb)) * icb;
    // velocity differences u+ - u-, the upper one's product fused into the subtraction
    auto du = [&](const float* Ph, int ih, const float* Pl, int il, int q) {
      return __fmaf_rn(Ph[q * SP + ih], Ph[ih], -__fmul_rn(Pl[q * SP + il], Pl[il]));
    };
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      f[5 + 3 * q] = du(P0, ic + 1, P0, ic - 1, 1 + q) * c.hidx[0] * icb;
      f[6 + 3 * q] = du(P0, ic + SX, P0, ic - SX, 1 + q) * c.hidx[1] * icb;
      f[7 + 3 * q] = du(Pp, ic, Pm, ic, 1 + q) * c.hidx[2] * icb;
    }
    f[14] = 0.0f;
    f[15] = 0.0f;
    float4* so = reinterpret_cast<float4*>(sO + tid * OS);
#pragma unroll
    for (int q = 0; q < 4; ++q) so[q] = make_float4(f[4 * q], f[4 * q + 1], f[4 * q + 2], f[4 * q + 3]);
    __syncwarp();
    // the warp's row: cell lane / 4 + 8 i, quarter lane % 4
    if (gy < g.ny) {
      float4* out = reinterpret_cast<float4*>(feat + ((size_t)b * fc + (size_t)k * g.plane + (size_t)gy * g.nx + x0) * 16);
      const int nrow = g.nx - x0 < TX ? g.nx - x0 : TX;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int cell = (lane >> 2) + 8 * i;
        if (cell < nrow) out[cell * 4 + (lane & 3)] = reinterpret_cast<const float4*>(sO + (ty * TX + cell) * OS)[lane & 3];
      }
    }
    __syncthreads();   // plane k-1 no longer read
    if (more) store(qf, slot(k - 1));
    __syncthreads();   // plane k+2 visible
  }
}

// ------------------------------------------------------------------------------------
// activations
// ------------------------------------------------------------------------------------
// erf by the rational approximation of Abramowitz & Stegun, formula 7.1.26
// (|error| <= 1.5e-7, below the BF16 resolution of the activations it feeds):
// erf(x) = 1 - (a1 t + a2 t^2 + a3 t^3 + a4 t^4 + a5 t^5) exp(-x^2), t = 1 / (1 + p x), x >= 0
// (reciprocal and exponential flush subnormals, which 1 + p x >= 1 never is and beside
// which the exponential counts for nothing; without that they take several instructions
// more each)
__device__ __forceinline__ float rcp_ftz(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float ex2_ftz(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float exp_ftz(float x) { return ex2_ftz(x * 1.4426950408889634f); }
__device__ __forceinline__ float erf_as(float x) {
  const float ax = fabsf(x);
  const float t = rcp_ftz(fmaf(0.3275911f, ax, 1.0f));
  float q = fmaf(1.061405429f, t, -1.453152027f);
  q = fmaf(q, t, 1.421413741f);
  q = fmaf(q, t, -0.284496736f);
  q = fmaf(q, t, 0.254829592f);
  const float y = fmaf(-q * t, exp_ftz(-ax * ax), 1.0f);
  return copysignf(y, x);
}
__device__ __forceinline__ float softplus(float y) { return fmaxf(y, 0.0f) + log1pf(expf(-fabsf(y))); }
__device__ __forceinline__ float sigmoid(float y) { return 1.0f / (1.0f + expf(-y)); }
__device__ __forceinline__ float bfr(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<unsigned*>(&v);
}

// D = A (16x16 bf16, row) * B (16x8 bf16, col) + C, FP32 accumulate
__device__ __forceinline__ void mma_bf16(float d[4], const unsigned a[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// gelu(z) = z (1 + erf(z / sqrt 2)) / 2 of two values, erf_as() in paired FP32 instructions.
// The factor 1/2 is in the polynomial's coefficients: scaling by a power of two commutes with
// every rounding, so the bits are those of erf_as() and a product fewer is issued.
__device__ __forceinline__ float2 gelu2(float2 z) {
  const float2 x = __fmul2_rn(z, f2(0.70710678118654752f, 0.70710678118654752f));
  const float2 ax = f2(fabsf(x.x), fabsf(x.y));
  const float2 den = __ffma2_rn(f2(0.3275911f, 0.3275911f), ax, f2(1.0f, 1.0f));
  const float2 t = f2(rcp_ftz(den.x), rcp_ftz(den.y));
  float2 q = __ffma2_rn(f2(0.5f * 1.061405429f, 0.5f * 1.061405429f), t, f2(-0.5f * 1.453152027f, -0.5f * 1.453152027f));
  q = __ffma2_rn(q, t, f2(0.5f * 1.421413741f, 0.5f * 1.421413741f));
  q = __ffma2_rn(q, t, f2(-0.5f * 0.284496736f, -0.5f * 0.284496736f));
  q = __ffma2_rn(q, t, f2(0.5f * 0.254829592f, 0.5f * 0.254829592f));
  const float2 qt = __fmul2_rn(q, t);
  const float2 ex = __fmul2_rn(__fmul2_rn(ax, ax), f2(-1.4426950408889634f, -1.4426950408889634f));
  const float2 y = __ffma2_rn(f2(-qt.x, -qt.y), f2(ex2_ftz(ex.x), ex2_ftz(ex.y)), f2(0.5f, 0.5f));
  return __fmul2_rn(z, __fadd2_rn(f2(0.5f, 0.5f), f2(copysignf(y.x, x.x), copysignf(y.y, x.y))));
}

// ------------------------------------------------------------------------------------
// tensor-core inference: one warp per 32 cells (two 16-row tiles, which share every
// weight fragment read); the weights are staged once per CTA in shared memory in the
// order of the fragments, so that a lane reads a 16-wide slice of W1 as one 64-bit word
// pair and two such slices of W2 as one 128-bit word (row strides free of bank
// conflicts).  The 128 GELUs per cell bound the kernel: their FP32 arithmetic, two values
// per instruction, some 85 us of the FMA units for 1.77 M cells, and two special-function
// operations each.  146 us for those cells: 228 us with 16 cells per warp and scalar GELUs,
// 154 us with the factor 1/2 of the GELU a product of its own.  (Three CTAs per SM, 80
// registers: 151 us.  Tiles drawn from a counter: 147 us.)
// ------------------------------------------------------------------------------------
constexpr int W1S = 8;    // 32-bit words per row of W1t (16 bf16)
constexpr int W2S = 36;   // padded row stride of W2t: 64 bf16 = 32 words

// WIDE: the features are read in pairs, which want 8-byte alignment; a caller's array that has
// only a float's is read one by one.
template <bool WIDE>
__global__ void __launch_bounds__(256, 2) k_mlp_infer(long long n, MlpView net, const float* __restrict__ feat,
                                                      const float* __restrict__ sigma1, float scale, float limit_nu,
                                                      float* __restrict__ nu, unsigned* err, bool cap) {
  pdl_enter();
  __shared__ __align__(16) unsigned sW1[NH * W1S];
  __shared__ __align__(16) unsigned sW2[NH * W2S];
  __shared__ __align__(16) float sb1[NH], sb2[NH], sw3[NH];
  {
    const unsigned* w1 = reinterpret_cast<const unsigned*>(net.W1t);
    const unsigned* w2 = reinterpret_cast<const unsigned*>(net.W2t);
    // word (kk, half h, t) of a row (8 kk + 4 h + t) goes to place t, slice kk, half h
    for (int i = threadIdx.x; i < NH * 8; i += blockDim.x) {
      const int w = i & 7;
      sW1[(i >> 3) * W1S + (w & 3) * 2 + (w >> 2)] = w1[i];
    }
    for (int i = threadIdx.x; i < NH * 32; i += blockDim.x) {
      const int w = i & 31;
      sW2[(i >> 5) * W2S + (w & 3) * 8 + (w >> 3) * 2 + ((w >> 2) & 1)] = w2[i];
    }
    for (int i = threadIdx.x; i < NH; i += blockDim.x) {
      sb1[i] = net.b1[i];
      sb2[i] = net.b2[i];
      sw3[i] = net.w3q[i];
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int gq = lane >> 2, tq = lane & 3;
  const float b3 = net.b3[0];
  const long long ntiles = (n + 31) / 32;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long tile = warp; tile < ntiles; tile += nwarps) {
    // rows r + 8 i, i = 0..3: tile m has i = 2 m, 2 m + 1
    const long long r = tile * 32 + gq;
    unsigned a[2][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const bool in = r + 8 * i < n;
      const float* f = feat + (size_t)(r + 8 * i) * 16;
      auto pair = [&](int k) {
        if constexpr (WIDE) return reinterpret_cast<const float2*>(f)[k];
        else return f2(f[2 * k], f[2 * k + 1]);
      };
      const float2 lo = in ? pair(tq) : f2(0.0f, 0.0f), hi = in ? pair(tq + 4) : f2(0.0f, 0.0f);
      a[i >> 1][i & 1] = pack_bf16(lo.x, lo.y);
      a[i >> 1][2 + (i & 1)] = pack_bf16(hi.x, hi.y);
    }
    unsigned a2[2][4][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint2 w = *reinterpret_cast<const uint2*>(&sW1[(8 * j + gq) * W1S + 2 * tq]);
      const float2 c = *reinterpret_cast<const float2*>(&sb1[8 * j + 2 * tq]);
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        float h[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        mma_bf16(h, a[m], w.x, w.y);
        const float2 g0 = gelu2(__fadd2_rn(f2(h[0], h[1]), c)), g1 = gelu2(__fadd2_rn(f2(h[2], h[3]), c));
        a2[m][j >> 1][2 * (j & 1)] = pack_bf16(g0.x, g0.y);
        a2[m][j >> 1][2 * (j & 1) + 1] = pack_bf16(g1.x, g1.y);
      }
    }
    float y[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint4* wp = reinterpret_cast<const uint4*>(&sW2[(8 * j + gq) * W2S + 8 * tq]);
      const uint4 w0 = wp[0], w1 = wp[1];
      const float2 c = *reinterpret_cast<const float2*>(&sb2[8 * j + 2 * tq]);
      const float2 v = *reinterpret_cast<const float2*>(&sw3[8 * j + 2 * tq]);
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        float z[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        mma_bf16(z, a2[m][0], w0.x, w0.y);
        mma_bf16(z, a2[m][1], w0.z, w0.w);
        mma_bf16(z, a2[m][2], w1.x, w1.y);
        mma_bf16(z, a2[m][3], w1.z, w1.w);
        const float2 g0 = gelu2(__fadd2_rn(f2(z[0], z[1]), c)), g1 = gelu2(__fadd2_rn(f2(z[2], z[3]), c));
        y[2 * m] += g0.x * v.x + g0.y * v.y;
        y[2 * m + 1] += g1.x * v.x + g1.y * v.y;
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      y[i] += __shfl_xor_sync(0xffffffffu, y[i], 1);
      y[i] += __shfl_xor_sync(0xffffffffu, y[i], 2);
    }
    // lane tq of a row group writes row r + 8 tq
    const float yo = tq == 0 ? y[0] : (tq == 1 ? y[1] : (tq == 2 ? y[2] : y[3]));
    const long long ro = r + 8 * tq;
    if (ro < n) nu[ro] = nu_checked(scale * sigma1[ro] * softplus(yo + b3), limit_nu, cap, err);
  }
}

// ------------------------------------------------------------------------------------
// training: forward + backward of one minibatch chunk of TS samples per CTA, with the
// quantisation points of the inference path; per-CTA gradient partials, then one kernel
// that adds them in a fixed order, makes the FP32 Adam update and rewrites the inference
// copies.  Every matrix product (the two layers, the backward through layer 2 and the two
// weight gradients) runs on the tensor cores as BF16 m16n8k16 products with FP32
// accumulation; their operands are the BF16 values of the inference path (inputs,
// weights, hidden activations) and, in the backward pass, the BF16-rounded gradients
// dZ2 and dZ1 of the pre-activations (the bias gradients sum the FP32 ones).
//
// A minibatch is a few thousand samples: the step is a chain of short phases, so what
// counts is the number of SMs and threads that share each one.  Chunks of 32 samples give
// a 4096-sample minibatch 128 CTAs; operands are kept in shared memory as BF16 and read
// by ldmatrix (transposed where a product sums over samples or needs W2^T); each GELU and
// its derivative are formed once, by the thread that holds the pre-activation; the column
// sums are spread over all threads.  With 64-sample chunks, float operands rounded at
// every use and 64 threads forming the column sums, a 4096-sample step took 32 us in this
// kernel and 14 us in the loss, Adam and publishing kernels after it; 18 and 5 us now.
// ------------------------------------------------------------------------------------
constexpr int TS = 32;       // samples per CTA
constexpr int TT = 256;      // threads per CTA (8 warps)
constexpr int LD = NH + 1;   // padded row of the FP32 activations
constexpr int LB = NH + 8;   // padded row of the BF16 operands (16-byte rows, no ldmatrix bank conflicts)
constexpr int LX = 24;       // the same for the 16 inputs

struct TrainSmem {
  __nv_bfloat16 W1[NF][LB];   // [k][j], rows 14, 15 zero
  __nv_bfloat16 W2[NH][LB];   // [k][j]
  __nv_bfloat16 X[TS][LX];
  __nv_bfloat16 H1[TS][LB];   // gelu(Z1)
  __nv_bfloat16 D2b[TS][LB];  // dZ2
  __nv_bfloat16 D1b[TS][LB];  // dZ1
  float D1[TS][LD];           // gelu'(Z1), then dZ1
  float H2[TS][LD];           // gelu(Z2)
  float D2[TS][LD];           // gelu'(Z2), then dZ2
  float b1[NH], b2[NH], w3[NH];
  float dy[TS];
  float sum[3][4][NH];        // column sums by quarter of the samples
  float G[NPAR];              // the CTA's gradient
};
constexpr int TC = 4;         // CTAs per cluster: their gradients are added before they go out

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// A fragment (16 x 16 at (m0, k0)) of S[m][k], row stride ld
__device__ __forceinline__ void frag_a(unsigned a[4], const __nv_bfloat16* S, int ld, int m0, int k0) {
  const int l = threadIdx.x & 31;
  const unsigned p = smem_addr(S + (m0 + (l & 15)) * ld + k0 + (l >> 4) * 8);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(p));
}
// the same of the transpose of S[k][m]
__device__ __forceinline__ void frag_at(unsigned a[4], const __nv_bfloat16* S, int ld, int m0, int k0) {
  const int l = threadIdx.x & 31;
  const unsigned p = smem_addr(S + (k0 + (l & 7) + (l >> 4) * 8) * ld + m0 + ((l >> 3) & 1) * 8);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(p));
}
// B fragment (16 x 8 at (k0, n0)) of S[k][n]
__device__ __forceinline__ void frag_b(unsigned b[2], const __nv_bfloat16* S, int ld, int k0, int n0) {
  const int l = threadIdx.x & 15;
  const unsigned p = smem_addr(S + (k0 + l) * ld + n0);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(b[0]), "=r"(b[1]) : "r"(p));
}
// the same of the transpose of S[n][k]
__device__ __forceinline__ void frag_bt(unsigned b[2], const __nv_bfloat16* S, int ld, int k0, int n0) {
  const int l = threadIdx.x & 15;
  const unsigned p = smem_addr(S + (n0 + (l & 7)) * ld + k0 + (l >> 3) * 8);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(b[0]), "=r"(b[1]) : "r"(p));
}

// the (m, n) accumulator element of fragment slot q (0..3) of this lane
__device__ __forceinline__ void acc_at(int m0, int n0, int q, int& m, int& n) {
  const int lane = threadIdx.x & 31, gq = lane >> 2, tq = lane & 3;
  m = m0 + gq + (q >= 2 ? 8 : 0);
  n = n0 + 2 * tq + (q & 1);
}

// gelu(z) and its derivative from one erf.  The derivative's exponential keeps its subnormal
// values (|z| above 13.2): they reach the gradients beside a large dL/dy.
__device__ __forceinline__ void gelu_both(float z, float& h, float& d) {
  const float w = 1.0f + erf_as(z * 0.70710678118654752f);
  h = 0.5f * z * w;
  d = 0.5f * w + z * __expf(-0.5f * z * z) * 0.39894228040143268f;
}

__global__ void __cluster_dims__(TC, 1, 1) __launch_bounds__(TT) k_mlp_train_partial(MlpView net, const float* __restrict__ feat,
                                                          const float* __restrict__ target,
                                                          const int* __restrict__ idx, int n,
                                                          float* __restrict__ partial, float* loss_partial) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smraw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(smraw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float* P = net.master;
  const int s0 = blockIdx.x * TS;
  for (int q = tid; q < TS * NF; q += TT) {
    const int s = q / NF, k = q % NF, gs = s0 + s;
    S.X[s][k] = __float2bfloat16_rn((gs < n && k < NIN) ? feat[(size_t)idx[gs] * 16 + k] : 0.0f);
  }
  for (int q = tid; q < NF * NH; q += TT) {
    const int k = q / NH, j = q % NH;
    S.W1[k][j] = __float2bfloat16_rn(k < NIN ? P[OFF_W1 + k * NH + j] : 0.0f);
  }
  for (int q = tid; q < NH * NH; q += TT) S.W2[q / NH][q % NH] = __float2bfloat16_rn(P[OFF_W2 + q]);
  if (tid < NH) {
    S.b1[tid] = P[OFF_B1 + tid];
    S.b2[tid] = P[OFF_B2 + tid];
    S.w3[tid] = bfr(P[OFF_W3 + tid]);
  }
  __syncthreads();
  constexpr int MT = TS / 16, JT = MT * (NH / 8);   // row tiles, tiles of a TS x 64 result
  // layer 1: Z1 = X W1 + b1, H1 = bf16(gelu(Z1))
#pragma unroll
  for (int t = warp; t < JT; t += TT / 32) {
    const int m0 = (t % MT) * 16, n0 = (t / MT) * 8;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    unsigned a[4], b[2];
    frag_a(a, &S.X[0][0], LX, m0, 0);
    frag_b(b, &S.W1[0][0], LB, 0, n0);
    mma_bf16(acc, a, b[0], b[1]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int m, nn;
      acc_at(m0, n0, q, m, nn);
      float h, d;
      gelu_both(acc[q] + S.b1[nn], h, d);
      S.H1[m][nn] = __float2bfloat16_rn(h);
      S.D1[m][nn] = d;
    }
  }
  __syncthreads();
  // layer 2: Z2 = H1 W2 + b2
#pragma unroll
  for (int t = warp; t < JT; t += TT / 32) {
    const int m0 = (t % MT) * 16, n0 = (t / MT) * 8;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k0 = 0; k0 < NH; k0 += 16) {
      unsigned a[4], b[2];
      frag_a(a, &S.H1[0][0], LB, m0, k0);
      frag_b(b, &S.W2[0][0], LB, k0, n0);
      mma_bf16(acc, a, b[0], b[1]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int m, nn;
      acc_at(m0, n0, q, m, nn);
      gelu_both(acc[q] + S.b2[nn], S.H2[m][nn], S.D2[m][nn]);
    }
  }
  __syncthreads();
  // output, loss and dL/dy, one sample per lane of the first warp
  if (tid < TS) {
    const int gs = s0 + tid;
    float y = P[OFF_B3];
#pragma unroll 16
    for (int k = 0; k < NH; ++k) y += S.H2[tid][k] * S.w3[k];
    float d = 0.0f, l = 0.0f;
    if (gs < n) {
      const float r = softplus(y) - target[idx[gs]];
      l = r * r;
      d = 2.0f * r / (float)n * sigmoid(y);
    }
    S.dy[tid] = d;
    loss_partial[(size_t)blockIdx.x * TS + tid] = l;
  }
  __syncthreads();
  // dZ2 = dy w3 gelu'(Z2)
  for (int q = tid; q < TS * NH; q += TT) {
    const int m = q / NH, j = q % NH;
    const float dz = S.dy[m] * S.w3[j] * S.D2[m][j];
    S.D2[m][j] = dz;
    S.D2b[m][j] = __float2bfloat16_rn(dz);
  }
  __syncthreads();
  // dZ1 = (bf16(dZ2) W2^T) gelu'(Z1)
#pragma unroll
  for (int t = warp; t < JT; t += TT / 32) {
    const int m0 = (t % MT) * 16, n0 = (t / MT) * 8;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k0 = 0; k0 < NH; k0 += 16) {
      unsigned a[4], b[2];
      frag_a(a, &S.D2b[0][0], LB, m0, k0);
      frag_bt(b, &S.W2[0][0], LB, k0, n0);
      mma_bf16(acc, a, b[0], b[1]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int m, kk;
      acc_at(m0, n0, q, m, kk);
      const float dz = acc[q] * S.D1[m][kk];
      S.D1[m][kk] = dz;
      S.D1b[m][kk] = __float2bfloat16_rn(dz);
    }
  }
  __syncthreads();
  // weight gradients of this CTA, in parameter order:
  //   dW2[k][j] = sum_s H1[s][k] bf16(dZ2[s][j]),  dW1[k][j] = sum_s X[s][k] bf16(dZ1[s][j])
  float* G = S.G;
#pragma unroll
  for (int t = warp; t < (NH / 16) * (NH / 8); t += TT / 32) {
    const int m0 = (t % (NH / 16)) * 16, n0 = (t / (NH / 16)) * 8;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k0 = 0; k0 < TS; k0 += 16) {
      unsigned a[4], b[2];
      frag_at(a, &S.H1[0][0], LB, m0, k0);
      frag_b(b, &S.D2b[0][0], LB, k0, n0);
      mma_bf16(acc, a, b[0], b[1]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int k, j;
      acc_at(m0, n0, q, k, j);
      G[OFF_W2 + k * NH + j] = acc[q];
    }
  }
  {
    const int n0 = warp * 8;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k0 = 0; k0 < TS; k0 += 16) {
      unsigned a[4], b[2];
      frag_at(a, &S.X[0][0], LX, 0, k0);
      frag_b(b, &S.D1b[0][0], LB, k0, n0);
      mma_bf16(acc, a, b[0], b[1]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int k, j;
      acc_at(0, n0, q, k, j);
      if (k < NIN) G[OFF_W1 + k * NH + j] = acc[q];
    }
  }
  {
    const int j = tid & (NH - 1), part = tid >> 6;
    float a1 = 0.0f, a2 = 0.0f, a3 = 0.0f;
#pragma unroll
    for (int s = part * (TS / 4); s < (part + 1) * (TS / 4); ++s) {
      a1 += S.D1[s][j];
      a2 += S.D2[s][j];
      a3 += S.H2[s][j] * S.dy[s];
    }
    S.sum[0][part][j] = a1;
    S.sum[1][part][j] = a2;
    S.sum[2][part][j] = a3;
  }
  __syncthreads();
  if (tid < 3 * NH) {
    const int w = tid / NH, j = tid % NH;
    const float v = (S.sum[w][0][j] + S.sum[w][1][j]) + (S.sum[w][2][j] + S.sum[w][3][j]);
    G[(w == 0 ? OFF_B1 : (w == 1 ? OFF_B2 : OFF_W3)) + j] = v;
  } else if (warp == TT / 32 - 1) {
    float a = S.dy[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) G[OFF_B3] = a;
  }
  // the cluster's gradients, added in rank order through distributed shared memory: one
  // partial per cluster (a quarter of the traffic and of the scratch)
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  const int rank = (int)cl.block_rank();
  const float* Gc[TC];
#pragma unroll
  for (int i = 0; i < TC; ++i) Gc[i] = cl.map_shared_rank(S.G, i);
  float* out = partial + (size_t)(blockIdx.x / TC) * NPAR;
  for (int q = rank * TT + tid; q < NPAR; q += TC * TT) {
    float v = Gc[0][q];
#pragma unroll
    for (int i = 1; i < TC; ++i) v += Gc[i][q];
    out[q] = v;
  }
  cl.sync();   // no CTA leaves while others read its gradient
}
static_assert(TS == 32 && TT == 4 * NH, "the last sums of k_mlp_train_partial");

// the inference copy of master parameter q: transposed BF16 weights, FP32 biases,
// BF16-rounded output weights
__device__ __forceinline__ void publish_param(const MlpView& net, int q, float v) {
  if (q < OFF_B1) {
    const int k = (q - OFF_W1) / NH, j = (q - OFF_W1) % NH;
    net.W1t[j * 16 + k] = __float2bfloat16_rn(v);
  } else if (q < OFF_W2) {
    net.b1[q - OFF_B1] = v;
  } else if (q < OFF_B2) {
    const int k = (q - OFF_W2) / NH, j = (q - OFF_W2) % NH;
    net.W2t[j * NH + k] = __float2bfloat16_rn(v);
  } else if (q < OFF_W3) {
    net.b2[q - OFF_B2] = v;
  } else if (q < OFF_B3) {
    net.w3q[q - OFF_W3] = bfr(v);
  } else {
    net.b3[0] = v;
  }
}

// The clusters' gradient partials added in a fixed order (eight strided slices, then the
// slices), the Adam update and the inference copies of 32 parameters per CTA; the CTA
// after the last parameter's adds the per-sample losses (padding samples hold 0).
constexpr int AP = 32, ASL = 8;   // parameters and slices per CTA
__global__ void __launch_bounds__(AP * ASL) k_mlp_adam(int nblk, int nloss, int n, MlpView net, const float* __restrict__ partial,
                                                       const float* __restrict__ lp, float* __restrict__ loss,
                                                       int step, float lr, float beta1, float beta2, float eps) {
  pdl_enter();
  __shared__ float sh[AP * ASL];
  const int tid = threadIdx.x;
  if (blockIdx.x * AP >= NPAR) {
    float s = 0.0f;
    for (int i = tid; i < nloss; i += AP * ASL) s += lp[i];
    sh[tid] = s;
    __syncthreads();
    for (int k = AP * ASL / 2; k > 0; k >>= 1) {
      if (tid < k) sh[tid] += sh[tid + k];
      __syncthreads();
    }
    if (tid == 0) loss[0] = sh[0] / (float)n;
    return;
  }
  const int q = blockIdx.x * AP + tid % AP, sl = tid / AP;
  float g = 0.0f;
  if (q < NPAR) {
#pragma unroll 4
    for (int b = sl; b < nblk; b += ASL) g += partial[(size_t)b * NPAR + q];
  }
  sh[tid] = g;
  __syncthreads();
  if (tid >= AP || q >= NPAR) return;
  g = 0.0f;
#pragma unroll
  for (int i = 0; i < ASL; ++i) g += sh[i * AP + tid];
  const float m = net.m[q] = beta1 * net.m[q] + (1.0f - beta1) * g;
  const float v = net.v[q] = beta2 * net.v[q] + (1.0f - beta2) * g * g;
  const float mh = m / (1.0f - powf(beta1, (float)step));
  const float vh = v / (1.0f - powf(beta2, (float)step));
  const float w = net.master[q] - lr * mh / (sqrtf(vh) + eps);
  net.master[q] = w;
  publish_param(net, q, w);
}

__global__ void k_mlp_reset(MlpView net, const float* __restrict__ params) {
  pdl_enter();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < NH) {   // the two padding inputs' weights
    net.W1t[q * 16 + NIN] = __float2bfloat16_rn(0.0f);
    net.W1t[q * 16 + NIN + 1] = __float2bfloat16_rn(0.0f);
  }
  if (q >= NPAR) return;
  const float v = params[q];
  net.master[q] = v;
  net.m[q] = 0.0f;
  net.v[q] = 0.0f;
  publish_param(net, q, v);
}

__global__ void k_label_target(long long n, const float* __restrict__ acc, const float* __restrict__ sig,
                               float dx2, float tmax, float* __restrict__ t) {
  pdl_enter();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float v = acc[i] / (dx2 * sig[i] + 1e-30f);
  t[i] = v < tmax ? v : tmax;
}

}  // namespace

cudaError_t launch_label_target(long long n, const float* acc, const float* sig, double dx2, double tmax,
                                float* t, cudaStream_t st) {
  count_launch();
  return launch_pdl(k_label_target, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, n, acc, sig, (float)dx2, (float)tmax, t);
}

MlpView mlp_view(void* blob) {
  char* p = (char*)blob;
  MlpView v;
  v.master = (float*)(p + MLP_OFF_MASTER);
  v.m = (float*)(p + MLP_OFF_M);
  v.v = (float*)(p + MLP_OFF_V);
  v.W1t = (__nv_bfloat16*)(p + MLP_OFF_W1T);
  v.W2t = (__nv_bfloat16*)(p + MLP_OFF_W2T);
  v.b1 = (float*)(p + MLP_OFF_VEC);
  v.b2 = v.b1 + NH;
  v.w3q = v.b2 + NH;
  v.b3 = v.w3q + NH;
  return v;
}

template <class TIN>
cudaError_t launch_box_means(const GridDesc& g, double gamma, const TIN* w, double* qbar, double* scratch,
                             cudaStream_t st) {
  count_launch();
  cudaError_t e = launch_pdl(k_box_means<TIN>, dim3(dim3(RGM, g.batch)), dim3(RB), 0, st, g, (float)gamma, w, scratch);
  if (e != cudaSuccess) return e;
  count_launch();
  return launch_pdl(k_box_means_final, dim3(g.batch * 5), dim3(RB), 0, st, RGM, 1.0 / (double)g.cells, scratch, qbar);
}

size_t box_means_scratch_doubles(const GridDesc& g) { return (size_t)5 * RGM * g.batch; }

template <class TIN>
cudaError_t launch_features(const GridDesc& g, const Coef<float>& c, const TIN* w, const double* qbar,
                            float* feat, cudaStream_t st) {
  static MarchShape<TX, fk::FY> shape;
  int ctas = 0;
  GridDesc gm = g;
  cudaError_t e = shape.get_ranges(k_features<TIN>, fk::smem, gm, nullptr, ctas);
  if (e != cudaSuccess) return e;
  count_launch();
  return launch_pdl(k_features<TIN>, dim3(ctas), dim3(fk::NT), fk::smem, st, gm, c, w, qbar, feat);
}
template cudaError_t launch_box_means<double>(const GridDesc&, double, const double*, double*, double*, cudaStream_t);
template cudaError_t launch_box_means<float>(const GridDesc&, double, const float*, double*, double*, cudaStream_t);
template cudaError_t launch_features<double>(const GridDesc&, const Coef<float>&, const double*, const double*,
                                             float*, cudaStream_t);
template cudaError_t launch_features<float>(const GridDesc&, const Coef<float>&, const float*, const double*,
                                            float*, cudaStream_t);

cudaError_t launch_mlp_infer(long long n, void* blob, const float* feat, const float* sigma1, double scale,
                             double limit_nu, float* nu, unsigned* err, cudaStream_t st, bool cap) {
  const long long tiles = (n + 31) / 32;
  long long blocks = (tiles + 7) / 8;
  if (blocks > 2 * 152) blocks = 2 * 152;   // one wave at two resident CTAs per SM
  if (blocks < 1) blocks = 1;
  count_launch();
  const bool wide = ((uintptr_t)feat & 7) == 0;
  return launch_pdl(wide ? k_mlp_infer<true> : k_mlp_infer<false>, dim3((unsigned)blocks), dim3(256), 0, st, n,
                    mlp_view(blob), feat, sigma1, (float)scale, (float)limit_nu, nu, err, cap);
}

// CTAs of a minibatch: whole clusters (the last ones may have no samples)
static int train_ctas(int n) { return ((n + TS - 1) / TS + TC - 1) / TC * TC; }

size_t mlp_train_scratch_floats(int n) {
  const int nblk = train_ctas(n);
  return (size_t)(nblk / TC) * NPAR + (size_t)nblk * TS + 16;
}

cudaError_t launch_mlp_train_step(void* blob, const float* feat, const float* target, const int* idx, int n,
                                  int step, double lr, float* scratch, float* loss, cudaStream_t st) {
  const int nblk = train_ctas(n);
  MlpView v = mlp_view(blob);
  float* partial = scratch;
  float* lp = scratch + (size_t)(nblk / TC) * NPAR;
  const size_t smem = sizeof(TrainSmem);
  cudaError_t e = cudaFuncSetAttribute(k_mlp_train_partial, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = launch_pdl(k_mlp_train_partial, dim3(nblk), dim3(TT), smem, st, v, feat, target, idx, n, partial, lp);
  count_launch();
  if (e != cudaSuccess) return e;
  const int pb = (NPAR + AP - 1) / AP;
  e = launch_pdl(k_mlp_adam, dim3(pb + (loss ? 1 : 0)), dim3(AP * ASL), 0, st, nblk / TC, nblk * TS, n, v,
                 (const float*)partial,
                 (const float*)lp, loss, step, (float)lr, 0.9f, 0.999f, 1e-8f);
  count_launch();
  return e;
}

cudaError_t launch_mlp_set(void* blob, const float* params, cudaStream_t st) {
  MlpView v = mlp_view(blob);
  count_launch();
  return launch_pdl(k_mlp_reset, dim3((NPAR + 255) / 256), dim3(256), 0, st, v, params);
}

}  // namespace ns
