// Shared device-side definitions of the NS stencil kernels (sm_103a).
//
// Tile geometry: a CTA owns TX x TY cell columns of one box (TX = 32 below; TY is set in each
// kernel's file: 8 in the stage kernels of ns_rhs.cu and ns_adj.cu, sigma_1 and the features, 4
// in the FP64 stage kernels of ns_f64.cu) and marches a range of
// z-planes, keeping a ring of three planes (k-1, k, k+1) of primitive variables with
// a one-cell halo in x and y in shared memory.  Every face flux of the range is
// computed once; periodic wrap is resolved when a plane is loaded, so every shared
// position holds a valid cell even when the box is smaller than the tile.
//
// Work split (MarchShape): a launch shares the planes of all tile columns among the kernel's
// resident slots on the device (occupancy calculator x SMs).  The FP64 stage kernels, which
// have registers to spare, launch one CTA per slot: they lay the columns end to end, with
// MARCH_GAP units between two columns for the cost of starting one, and cut that into equal
// pieces; a CTA marches its piece, range by range where it spans the end of a column (March).
// In the FP32 kernels that outer loop costs registers they do not have (the adjoint stage
// spilled and took 15% longer): there a CTA marches one range (march_range), and get_ranges
// chooses among three launches: the same pieces with the part of each beyond a column's end as
// a CTA of its own (slots + columns - 1 CTAs), one wave of even ranges (as many CTAs as slots),
// or several whole waves of equal ranges where the columns outnumber the slots.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>

#include <atomic>
#include <type_traits>
#include <utility>

namespace ns {

// Process-wide count of this library's kernel launches (read by ns_launch_count).
inline std::atomic<unsigned long long> g_launches{0};
inline void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

constexpr int TX = 32;
constexpr int SX = TX + 2;    // shared plane width incl. halo

struct GridDesc {
  int nx, ny, nz, batch;
  long long plane;     // nx * ny
  long long cells;     // nx * ny * nz  (one box)
  unsigned* dbg_err;   // sticky error word for the bounds checks of debug builds (may be null)
  int split;           // split of a one-range-per-CTA march (set for each launch)
};

constexpr int MARCH_SPLIT = 8;  // most ranges per column in whole waves
constexpr int MARCH_GAP = 2;    // planes' worth of starting a range: priming its three planes

// The ranges of this CTA's piece, one tile column after the other, for tiles of TXK x TYK
// columns (see the file comment).  The state is the last column alone: a march keeps one
// register for it, and the piece's ends are formed again at each column.  128x64x64, FP64
// primal step: 1021 us with each column cut into whole ranges (up to 16 planes, the mean
// being 13.5), 915 us in pieces.
template <int TXK, int TYK>
struct March {
  int col = -1;
  // the next range: box b, tile origin, planes [kz0, kz1); false when the piece is done
  __device__ __forceinline__ bool next(const GridDesc& g, int& b, int& x0, int& y0, int& kz0, int& kz1) {
    const int ncx = (g.nx + TXK - 1) / TXK, ncy = (g.ny + TYK - 1) / TYK, len = g.nz + MARCH_GAP;
    const long long T = (long long)ncx * ncy * g.batch * len - MARCH_GAP;
    const long long u0 = T * blockIdx.x / gridDim.x, u1 = T * (blockIdx.x + 1) / gridDim.x;
    if (col < 0) {
      col = (int)(u0 / len);
      if (u0 - (long long)col * len >= g.nz) ++col;   // the piece begins in a gap
    } else {
      ++col;
    }
    const long long start = (long long)col * len;
    if (start >= u1) return false;
    kz0 = u0 > start ? (int)(u0 - start) : 0;
    kz1 = u1 - start < g.nz ? (int)(u1 - start) : g.nz;
    x0 = (col % ncx) * TXK;
    const int r = col / ncx;
    y0 = (r % ncy) * TYK;
    b = r / ncy;
    return true;
  }
};

// One range per CTA, the CTAs dealt out to the tile columns as evenly as integers allow and
// each column's planes cut into that many ranges.
template <int TXK, int TYK>
__device__ __forceinline__ void march_even(const GridDesc& g, int& b, int& x0, int& y0, int& kz0, int& kz1) {
  const int ncx = (g.nx + TXK - 1) / TXK, ncy = (g.ny + TYK - 1) / TYK;
  const long long C = (long long)ncx * ncy * g.batch, G = gridDim.x, i = blockIdx.x;
  const int col = (int)(((i + 1) * C - 1) / G);
  const long long s0 = (long long)col * G / C, s1 = (long long)(col + 1) * G / C;
  const long long j = i - s0, m = s1 - s0;
  kz0 = (int)(g.nz * j / m);
  kz1 = (int)(g.nz * (j + 1) / m);
  x0 = (col % ncx) * TXK;
  const int r = col / ncx;
  y0 = (r % ncy) * TYK;
  b = r / ncy;
}

// One range per CTA under the split that MarchShape::get_ranges chose: even (g.split = 0),
// or g.split equal pieces of the columns laid end to end (see March), where CTA i < g.split
// takes the first range of piece i and the CTAs after them the beginnings of the columns
// that a piece reaches from the column before.  False, with an empty range of column 0,
// when there is none.
template <int TXK, int TYK>
__device__ __forceinline__ bool march_range(const GridDesc& g, int& b, int& x0, int& y0, int& kz0, int& kz1) {
  if (g.split == 0) {
    march_even<TXK, TYK>(g, b, x0, y0, kz0, kz1);
    return true;
  }
  const int ncx = (g.nx + TXK - 1) / TXK, ncy = (g.ny + TYK - 1) / TYK;
  const long long len = g.nz + MARCH_GAP, T = (long long)ncx * ncy * g.batch * len - MARCH_GAP, G = g.split,
                  i = blockIdx.x;
  int col;
  long long start, u0, u1;   // the column's start and the range's ends
  if (i < G) {
    u0 = T * i / G;
    u1 = T * (i + 1) / G;
    col = (int)(u0 / len);
    if (u0 - col * len >= g.nz) ++col;   // the piece begins in a gap
    start = col * len;
    if (u0 < start) u0 = start;
  } else {
    col = (int)(i - G) + 1;
    start = u0 = col * len;
    const long long q = ((start - MARCH_GAP) * G - 1) / T;   // piece of the last plane before
    u1 = T * (q + 1) / G;
  }
  kz0 = (int)(u0 - start);
  kz1 = u1 - start < g.nz ? (int)(u1 - start) : g.nz;
  if (kz0 >= kz1) {
    b = x0 = y0 = kz0 = kz1 = 0;
    return false;
  }
  x0 = (col % ncx) * TXK;
  const int r = col / ncx;
  y0 = (r % ncy) * TYK;
  b = r / ncy;
  return true;
}

// Launch shape of a plane-marching kernel: the CTA count (see the file comment).  The
// resident slots come from the occupancy calculator with the kernel's dynamic shared memory
// and are cached per device; the kernel's dynamic shared-memory limit is raised once.  The
// environment variable `env`, when set to a positive count, overrides the number of slots.
// At most one CTA per plane of a column.
template <int TXK, int TYK>
struct MarchShape {
  static constexpr int NTK = TXK * TYK;
  int per_dev[16] = {0};
  template <class K>
  cudaError_t slots_of(K kern, size_t smem, const char* env, long long& n) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int slots = (dev >= 0 && dev < 16) ? per_dev[dev] : 0;
    if (slots == 0) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      int per_sm = 0, sms = 0;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NTK, smem);
      if (e != cudaSuccess) return e;
      e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) return e;
      slots = (per_sm > 0 ? per_sm : 1) * sms;
      if (dev >= 0 && dev < 16) per_dev[dev] = slots;
    }
    n = slots;
    const char* ov = env ? getenv(env) : nullptr;
    if (ov && atoll(ov) > 0) n = atoll(ov);
    return cudaSuccess;
  }
  static long long columns(const GridDesc& g) {
    return (long long)((g.nx + TXK - 1) / TXK) * ((g.ny + TYK - 1) / TYK) * g.batch;
  }
  // kernels that march pieces (March)
  template <class K>
  cudaError_t get(K kern, size_t smem, const GridDesc& g, const char* env, int& ctas) {
    long long n = 0;
    const cudaError_t e = slots_of(kern, smem, env, n);
    if (e != cudaSuccess) return e;
    const long long cols = columns(g);
    if (cols > (1LL << 26)) return cudaErrorInvalidConfiguration;
    ctas = (int)(n < cols * g.nz ? n : cols * g.nz);
    return cudaSuccess;
  }
  // kernels that march one range per CTA: also sets g.split for march_range (pieces: the
  // kernel takes the split into pieces; otherwise it uses march_even; fixed_cuts: see
  // k_adj_stage; most_ctas: the most CTAs of a split in whole waves).  The pieces' second
  // parts are further CTAs that start as slots fall free; they pay while there are few of
  // them (one per column) and the pieces are longer than a range's priming.  128x64x64,
  // adjoint step: 211 us even, 203 us in pieces; with 144 columns on 304 slots (eight
  // 96x48x48 boxes) 605 us even, 781 us in pieces.  Even ranges are as many as the slots or,
  // when the columns are too many for that, the number of ranges per column with the
  // shortest whole waves: the 512 columns of a 512x256x128 box took 2310 us per primal step
  // in one range each (456 slots: a second wave with 56 CTAs), 1850 us in this split.
  template <class K>
  cudaError_t get_ranges(K kern, size_t smem, GridDesc& g, const char* env, int& ctas, bool pieces = true,
                         bool fixed_cuts = false, long long most_ctas = 0x7FFFFFFF) {
    long long n = 0;
    const cudaError_t e = slots_of(kern, smem, env, n);
    if (e != cudaSuccess) return e;
    const long long cols = columns(g);
    if (cols > (1LL << 26)) return cudaErrorInvalidConfiguration;
    g.split = 0;
    if (fixed_cuts) {
      // one wave of even ranges of at least four planes
      const long long most = cols * (g.nz / 4 > 1 ? g.nz / 4 : 1);
      ctas = (int)(n < cols ? cols : (n < most ? n : most));
      return cudaSuccess;
    }
    if (pieces && cols <= n / 8 && cols * g.nz >= 4 * n) {
      g.split = (int)n;
      ctas = (int)(n + cols - 1);
      return cudaSuccess;
    }
    // planes a slot marches: one wave of all slots, or whole waves of m ranges per column
    long long best = cols <= n ? (g.nz + n / cols - 1) / (n / cols) + MARCH_GAP : 1LL << 62, count = n;
    const int most = g.nz < MARCH_SPLIT ? g.nz : MARCH_SPLIT;
    for (int m = 1; m <= most && (m == 1 || cols * m <= most_ctas); ++m) {
      const long long cost = ((cols * m + n - 1) / n) * ((g.nz + m - 1) / m + MARCH_GAP);
      if (cost < best) {
        best = cost;
        count = cols * m;
      }
    }
    ctas = (int)(count < cols * g.nz ? count : cols * g.nz);
    return cudaSuccess;
  }
};

// Launch shape of the 2D (nz = 1) stage kernels: one CTA per tile of TX x TYF cells; the
// kernel's dynamic shared-memory limit is raised once per device.
template <int TYF>
struct FlatShape {
  bool ready[16] = {false};
  template <class K>
  cudaError_t get(K kern, size_t smem, const GridDesc& g, int& ctas) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 16 || !ready[dev]) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      if (dev >= 0 && dev < 16) ready[dev] = true;
    }
    const long long n = (long long)((g.nx + TX - 1) / TX) * ((g.ny + TYF - 1) / TYF) * g.batch;
    if (n > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    ctas = (int)n;
    return cudaSuccess;
  }
};

// Rows per tile of the 2D kernels: single rows spread a small box over the most SMs and
// keep the chain of a CTA shortest, but compute each y-face twice; four rows share them.
// Single rows up to two CTAs per SM: one FP64 step at 64x64 (128 single-row tiles) takes
// 23 us with single rows and 42 us with four, at 128x128 (512 tiles) 61 and 42 us.
inline int flat_rows(const GridDesc& g) {
  const long long rows = (long long)((g.nx + TX - 1) / TX) * g.ny * g.batch;
  return rows <= 2 * 152 ? 1 : 4;
}

template <class T>
struct Coef {
  T gamma, gm1, mu, alpha;
  T roe_delta;  // Harten's entropy-fix fraction of the Roe sound speed
  int roe;      // 1: Roe dissipation on the convective face flux
  T idx[3];    // 1 / dx_d
  T i4dx[3];   // 1 / (4 dx_d): tangential face gradient = mean of two central diffs
  T hidx[3];   // 1 / (2 dx_d): cell-centred central difference
};

__device__ __forceinline__ int wrap(int i, int n) {
  if (i >= 0 && i < n) return i;
  i %= n;
  return i < 0 ? i + n : i;
}

// ---------------------------------------------------------------------------------
// IEEE-754 binary64 <-> binary32 conversions in integer arithmetic.  GB300 issues
// FP64 instructions at a small fraction of the FP32 rate, so the mixed-precision path
// converts with integer ALU operations instead, from the field layout of the formats
// (sign, biased exponent, fraction):
//   d2f: round to nearest, ties to even; results below the smallest normal float
//        (2^-126) flush to signed zero; overflow gives infinity; NaN stays NaN.
//   f2d: exact for normal floats and zero; subnormal floats flush to signed zero.
// ---------------------------------------------------------------------------------
// Normal and zero values take a straight line of integer instructions (about a dozen; a
// form that branched on each range took twice as many); infinities, NaN and overflow
// branch off.
__device__ __forceinline__ float d2f(double x) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned sign = hi & 0x80000000u;
  const int m = (int)(hi & 0x7FFFFFFFu) - (896 << 20);   // biased exponent of the result above 20 fraction bits
  unsigned r = __funnelshift_l(lo, (unsigned)m, 3);       // the result's 31 bits before rounding
  // up when the 29 dropped bits exceed one half, or equal it and the result is odd
  r += ((lo & 0x1FFFFFFFu) + (r & 1u) + 0x0FFFFFFFu) >> 29;   // a carry may reach infinity
  if (m < (1 << 20)) r = 0u;                                   // zero, subnormal, underflow
  if (m >= (255 << 20)) {
    const bool nan = (hi & 0x7FFFFFFFu) > 0x7FF00000u || ((hi & 0x7FFFFFFFu) == 0x7FF00000u && lo != 0u);
    r = 0x7F800000u | (nan ? 0x00400000u : 0u);
  }
  return __uint_as_float(sign | r);
}

__device__ __forceinline__ double f2d(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned sign = u & 0x80000000u, a = u & 0x7FFFFFFFu;
  unsigned hi = (a >> 3) + (896u << 20), lo = u << 29;
  if (a < 0x00800000u) {   // zero, subnormal
    hi = 0u;
    lo = 0u;
  }
  if (a >= 0x7F800000u) {   // infinity, NaN (kept, made quiet)
    const unsigned m = u & 0x7FFFFFu;
    hi = 0x7FF00000u | (m >> 3) | (m ? 0x80000u : 0u);
  }
  return __hiloint2double((int)(sign | hi), (int)lo);
}

// 1/x = y / (1 - e), e = 1 - x y, from the FP32 reciprocal y by the geometric series to e^2
// (Halley's iteration for the reciprocal), which cubes y's relative error of 2^-22: three FP64
// instructions, the quotient takes some eight, and its value (no difference in 2^24 samples of
// each of several ranges of exponents); the quotient itself outside FP32's range.
__device__ __forceinline__ double recip(double x) {
  const float s = d2f(x), a = fabsf(s);
  if (!(a > 1e-30f && a < 1e30f)) return 1.0 / x;
  const double y = f2d(1.0f / s);
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// sqrt(x) in the same way: t = x y with y = rsqrt(x) of FP32, and t (1 - e)^(-1/2), e = 1 - t y,
// by the binomial series to 3 e^2/8; within 0.75 units of the last place
__device__ __forceinline__ double root(double x) {
  const float s = d2f(x);
  if (!(s > 1e-30f && s < 1e30f)) return sqrt(x);
  const double y = f2d(rsqrtf(s));
  const double t = x * y;
  const double e = fma(-t, y, 1.0);
  return fma(t * e, fma(0.375, e, 0.5), t);
}

// conversions used by the templated kernels: to the compute type / back to FP64
template <class T> __device__ __forceinline__ T cvt(double x);
template <> __device__ __forceinline__ double cvt<double>(double x) { return x; }
template <> __device__ __forceinline__ float cvt<float>(double x) { return d2f(x); }
template <class T> __device__ __forceinline__ T cvt(float x) { return T(x); }
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) { return f2d(x); }
// a caller's float (the added viscosity of FP64 products) exactly, subnormal values too, by
// the conversion instruction, which issues at FP64's rate
__device__ __forceinline__ bool subnormal(double) { return false; }   // (doubles are taken as they are)
__device__ __forceinline__ bool subnormal(float x) {
  const unsigned a = __float_as_uint(x) << 1;
  return a - 1u < 0x00FFFFFFu;
}
template <class T>
__device__ __forceinline__ double widen_exact(T x) {
  return subnormal(x) ? (double)x : widen(x);
}

// ---------------------------------------------------------------------------------
// forward-mode dual number (value, tangent) used to build the tangent kernel from
// the primal one
// ---------------------------------------------------------------------------------
struct Dual {
  double v, d;
  __host__ __device__ __forceinline__ Dual() {}
  __host__ __device__ __forceinline__ Dual(double a) : v(a), d(0.0) {}
  __host__ __device__ __forceinline__ Dual(double a, double b) : v(a), d(b) {}
};
__device__ __forceinline__ Dual operator+(Dual a, Dual b) { return Dual(a.v + b.v, a.d + b.d); }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return Dual(a.v - b.v, a.d - b.d); }
__device__ __forceinline__ Dual operator-(Dual a) { return Dual(-a.v, -a.d); }
__device__ __forceinline__ Dual operator*(Dual a, Dual b) {
  return Dual(a.v * b.v, a.d * b.v + a.v * b.d);
}
__device__ __forceinline__ Dual operator/(Dual a, Dual b) {
  double q = a.v / b.v;
  return Dual(q, (a.d - q * b.d) / b.v);
}
__device__ __forceinline__ Dual& operator+=(Dual& a, Dual b) { a = a + b; return a; }
__device__ __forceinline__ Dual& operator-=(Dual& a, Dual b) { a = a - b; return a; }

template <class T> struct ValueOf { typedef T type; };
template <> struct ValueOf<Dual> { typedef double type; };

__device__ __forceinline__ double val(double a) { return a; }
__device__ __forceinline__ float val(float a) { return a; }
__device__ __forceinline__ double val(Dual a) { return a.v; }
__device__ __forceinline__ double tan_of(Dual a) { return a.d; }

template <class T> __device__ __forceinline__ T one_over(T a) { return T(1) / a; }

// ---------------------------------------------------------------------------------
// Paired FP32 arithmetic (sm_100 family): one instruction does two independent FP32
// operations.  t2 = ((a - b) + c - d) * s for two such expressions at once, with the
// same rounding as the scalar left-to-right evaluation (a - b is fma(b, -1, a)).
// ---------------------------------------------------------------------------------
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

template <class CT>
__device__ __forceinline__ void diff4_pair(CT a1, CT b1, CT c1, CT d1, CT s1, CT a2, CT b2, CT c2, CT d2, CT s2,
                                           CT& r1, CT& r2) {
  if constexpr (std::is_same<CT, float>::value) {
    float2 t = sub2(f2(a1, a2), f2(b1, b2));
    t = __fadd2_rn(t, f2(c1, c2));
    t = sub2(t, f2(d1, d2));
    t = __fmul2_rn(t, f2(s1, s2));
    r1 = t.x;
    r2 = t.y;
  } else {
    r1 = (a1 - b1 + c1 - d1) * s1;
    r2 = (a2 - b2 + c2 - d2) * s2;
  }
}

// (hi, lo) += (bhi, blo) for unevaluated float pairs hi + lo: Knuth's two-sum of the high
// parts, the low parts added to its error, then a renormalising fast two-sum.  The pair
// keeps the sum of float terms to about 2^-44 relative; the result does not depend on
// the order of the two operands.
// (The explicit roundings keep a product in an operand from being fused into the sums,
// which would break the error-free transformation.)
__device__ __forceinline__ void df_add(float& hi, float& lo, float bhi, float blo) {
  const float s = __fadd_rn(hi, bhi);
  const float bb = __fsub_rn(s, hi);
  float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(bhi, bb));
  e = __fadd_rn(e, __fadd_rn(lo, blo));
  hi = __fadd_rn(s, e);
  lo = __fsub_rn(e, __fsub_rn(hi, s));
}

// ---------------------------------------------------------------------------------
// programmatic dependent launch.  The stencil and per-step diagnostic kernels of the
// sweep go out with programmatic stream serialisation: the next kernel's CTAs may be
// scheduled while the current kernel drains, so the launch latency between dependent
// kernels overlaps the tail of the previous one.  Each such kernel starts with
// pdl_enter(): griddepcontrol.wait blocks until the preceding grid has completed and
// its memory is visible (a no-op for a launch without the attribute), and only then
// does griddepcontrol.launch_dependents release the kernel after it, so every kernel
// still sees all earlier kernels' results.  The dependent grid starts only after every
// CTA of this one has started, so the early launch cannot starve this grid.  NS_PDL=0
// launches without the attribute.
// ---------------------------------------------------------------------------------
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

inline bool pdl_enabled() {
  static const bool on = [] {
    const char* e = getenv("NS_PDL");
    return !(e && e[0] == '0');
  }();
  return on;
}

// launch k (whose first statement is pdl_enter()) on st with the PDL attribute
template <class... KArgs, class... Args>
cudaError_t launch_pdl(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
}

// ---------------------------------------------------------------------------------
// error word bits (sticky, OR-ed by kernels, read by ns_last_error)
// ---------------------------------------------------------------------------------
constexpr unsigned ERRBIT_NONFINITE = 1u;
constexpr unsigned ERRBIT_UNSTABLE = 2u;
constexpr unsigned ERRBIT_CORRUPT = 4u;
constexpr unsigned ERRBIT_BOUNDS = 8u;

// An added adjoint viscosity v against the explicit stability limit: held at the limit
// where it exceeds it when cap is set; otherwise left, and flagged (NS_ERR_UNSTABLE) when
// above the limit or not finite.
template <class T>
__device__ __forceinline__ T nu_checked(T v, T limit, bool cap, unsigned* err) {
  if (cap && v > limit) return limit;
  if (!(v <= limit)) atomicOr(err, ERRBIT_UNSTABLE);
  return v;
}

// ---------------------------------------------------------------------------------
// Field accesses of the stencil kernels.  A field element is addressed as a base (box,
// plane and component: uniform over the CTA) plus the thread's in-plane offset.  Debug
// builds (NS_DEBUG_BOUNDS) check the element index base + off against the field's
// extent n before every access: an index outside [0, n) sets ERRBIT_BOUNDS in the
// sticky error word and the access is skipped (a load reads zero), so a wrong index
// shows as an error code instead of a memory fault.  Release builds access directly.
// ---------------------------------------------------------------------------------
#ifdef NS_DEBUG_BOUNDS
__device__ __forceinline__ bool dbg_ok(const GridDesc& g, long long i, long long n) {
  if (i >= 0 && i < n) return true;
  if (g.dbg_err) atomicOr(g.dbg_err, ERRBIT_BOUNDS);
  return false;
}
#define NS_LD(g, p, base, off, n)                                                                  \
  (::ns::dbg_ok((g), (long long)(base) + (long long)(off), (long long)(n))                         \
       ? ((p) + (base))[(off)]                                                                     \
       : std::remove_cv_t<std::remove_reference_t<decltype((p)[0])>>(0))
#define NS_ST(g, p, base, off, n, val)                                                             \
  do {                                                                                             \
    if (::ns::dbg_ok((g), (long long)(base) + (long long)(off), (long long)(n))) ((p) + (base))[(off)] = (val); \
  } while (0)
#define NS_IN_BOUNDS(g, i, n) (::ns::dbg_ok((g), (long long)(i), (long long)(n)))
#else
#define NS_IN_BOUNDS(g, i, n) true
#define NS_LD(g, p, base, off, n) (((p) + (base))[(off)])
#define NS_ST(g, p, base, off, n, val) (((p) + (base))[(off)] = (val))
#endif

}  // namespace ns
