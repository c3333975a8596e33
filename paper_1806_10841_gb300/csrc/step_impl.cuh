// The MD-step kernels of the AdResS library (templates; instantiated by step.cu for the
// WCA model and by step_ljrf.cu for the water-like Lennard-Jones + reaction-field model).
//
// One group of four consecutive threads handles one molecule (work item t), thread g
// owning atom g.  Kernels:
//   k_map      positions -> centre of mass, resolution value, COM-relative offsets
//   k_prologue first half kick + drift + wrap, then k_map's mapping
//   k_step     forces of Eq. 1 (Sec. "Force interpolation") + bonded (never interpolated)
//              + thermodynamic force (Sec. "Free energy corrections and the thermodynamic
//              force") and, by MODE:
//                MODE_FORCES   store the conservative force
//                MODE_LAST     + Langevin force, second half kick, store v and f
//                MODE_FUSED    + Langevin force, second half kick of this step, first half
//                              kick and drift of the next, wrap, and the next mapping
//                              (written to the other half of the double-buffered
//                              molecule arrays), so a step is one kernel.
//
// GB300 has 1.2 TFLOP/s of FP64 against ~70 TFLOP/s of FP32, so the FP32 mixed path keeps
// its FP64 work to the state update itself (kick and drift FMAs on double x and v):
// conversions, periodic wraps and the centre-of-mass mapping run on the integer pipes
// using the bit patterns of the doubles, and every pair force is FP32.  Positions enter
// the pair kernel as exact 32-bit fixed-point centres (so minimum-image differences are
// plain integer subtractions) plus float offsets.
#pragma once
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "internal.cuh"
#include "lists_impl.cuh"

namespace adress {

constexpr int MODE_FORCES = 0;
constexpr int MODE_LAST = 1;
constexpr int MODE_FUSED = 2;

// ---------------- bit-level conversions (integer pipes) -------------------------------

// Exact float -> double for finite floats (float denormals become signed zeros).
__device__ __forceinline__ double f2d_bits(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned e = (b >> 23) & 0xffu;
  const unsigned long long sg = (unsigned long long)(b >> 31) << 63;
  const unsigned long long m = (unsigned long long)(b & 0x7fffffu) << 29;
  const unsigned long long d = e ? (sg | ((unsigned long long)(e + 896u) << 52) | m) : sg;
  return __longlong_as_double((long long)d);
}

// double -> float rounding half away from zero (ties only differ from round-to-nearest-even).
__device__ __forceinline__ float d2f_bits(double x) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const unsigned sg = (unsigned)(bits >> 63) << 31;
  const unsigned long long a = (bits & 0x7fffffffffffffffull) + 0x10000000ull;
  const int e = (int)(a >> 52) - 896;
  if (e <= 0) return __uint_as_float(sg);
  if (e >= 255) return __uint_as_float(sg | 0x7f800000u);
  return __uint_as_float(sg | ((unsigned)e << 23) | (unsigned)((a >> 29) & 0x7fffffu));
}

// Rare path of the periodic wrap, kept out of line so the common path has no FP64 add.
static __device__ __noinline__ double wrap_slow(double y, double L) {
  if (y < 0.0) y += L;
  if (y >= L) y -= L;
  return y;
}

// y wrapped into [0, L): compare the bit patterns (non-negative doubles order like their bits).
__device__ __forceinline__ double wrap_bits(double y, double L, long long Lbits) {
  const long long bits = __double_as_longlong(y);
  if (bits < 0 || bits >= Lbits) y = wrap_slow(y, L);
  return y;
}

// Parameters as the pair loop's real type (float copies precomputed on the host).
template <class T>
__device__ __forceinline__ T par(double d, float f);
template <>
__device__ __forceinline__ double par<double>(double d, float) { return d; }
template <>
__device__ __forceinline__ float par<float>(double, float f) { return f; }

__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// floor(x 2^32 / L) for 0 <= x < L from the bits of x: the 53-bit significand times
// K = floor(2^q / L) (exact 128-bit product, high word kept), shifted by the exponent.
__device__ __forceinline__ unsigned fixed32(double x, unsigned long long K, int q) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((bits >> 52) & 0x7ff);
  const unsigned long long M = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = q - 44 - (e - 1023);
  const unsigned long long hi = __umul64hi(M, K);
  return (e == 0 || sh >= 64 || sh < 0) ? 0u : (unsigned)(hi >> sh);
}

// ---------------- Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) -------------------
__device__ __forceinline__ void philox4x32_10(unsigned c[4], unsigned k0, unsigned k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const unsigned lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
    const unsigned lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
    const unsigned n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
  }
}

// ---------------- FP64 reciprocal and square root ----------------------------------------
// Newton-Raphson from the hardware's approximations (about 20 bits).  Two steps leave an error far
// below the last place, and the rounding of the second: the reciprocal is within one unit in the
// last place of the correctly rounded one, the reciprocal square root (whose residual is rounded
// too) within two.  The FP64 pipe runs 2 lanes a clock per SM here, and the library's division and
// square root cost 2-3 times as many of its instructions.

__device__ __forceinline__ double rcp_nr(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(fma(-x, y, 1.0), y, y);
  return fma(fma(-x, y, 1.0), y, y);
}
__device__ __forceinline__ double rsqrt_nr(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = 0.5 * x;
  y = fma(fma(-h * y, y, 0.5), y, y);
  return fma(fma(-h * y, y, 0.5), y, y);
}
// ---------------- precision policies for the pair loop --------------------------------

template <class P>
struct Prec;

template <>
struct Prec<P64> {
  using real = double;
  struct V3 {
    double x, y, z;
  };
  static __device__ __forceinline__ double4_32a com(const Bufs& b, int cur, int a) { return b.com64[cur][a]; }
  static __device__ __forceinline__ double w(const double4_32a& c) { return c.w; }
  static __device__ __forceinline__ V3 dR(const Box& X, const double4_32a& A, const double4_32a& B) {
    return {minimg_bits(A.x - B.x, X.L[0], X.halfL[0]), minimg_bits(A.y - B.y, X.L[1], X.halfL[1]),
            minimg_bits(A.z - B.z, X.L[2], X.halfL[2])};
  }
  // offset of atom k of molecule a (NA atoms per molecule)
  template <int NA>
  static __device__ __forceinline__ double4_32a off(const Bufs& b, int cur, int a, int k) {
    return b.off64[cur][a * NA + k];
  }
  static __device__ __forceinline__ double cg(const Bufs& b, int cg_n, double r, double inv_dr, double* V) {
    const double u = r * inv_dr;
    int k = (int)u;
    if (k > cg_n - 1) k = cg_n - 1;
    const double t = u - k;
    *V = b.cgV64[k] * (1.0 - t) + b.cgV64[k + 1] * t;
    return b.cgF64[k] * (1.0 - t) + b.cgF64[k + 1] * t;
  }
  static __device__ __forceinline__ double tf(const Bufs& b, int k) { return b.tf64[k]; }
  static __device__ __forceinline__ double fec(const Bufs& b, int k) { return b.fec64[k]; }
  static __device__ __forceinline__ double sin_(double x) { return sin(x); }
  static __device__ __forceinline__ double rcp_(double x) { return rcp_nr(x); }
  static __device__ __forceinline__ double rsqrt_(double x) { return rsqrt_nr(x); }
  static __device__ __forceinline__ double acos_(double x) { return acos(x); }
  static __device__ __forceinline__ double div_(double a, double x) { return a * rcp_nr(x); }
};

template <>
struct Prec<P32> {
  using real = float;
  struct V3 {
    float x, y, z;
  };
  static __device__ __forceinline__ int4 com(const Bufs& b, int cur, int a) { return b.com_fx[cur][a]; }
  static __device__ __forceinline__ float w(const int4& c) { return __int_as_float(c.w); }
  // exact integer difference of fixed-point centres (periodic wrap for free), then float
  static __device__ __forceinline__ V3 dR(const Box& X, const int4& A, const int4& B) {
    return {(float)(int)((unsigned)A.x - (unsigned)B.x) * X.fx_scale[0],
            (float)(int)((unsigned)A.y - (unsigned)B.y) * X.fx_scale[1],
            (float)(int)((unsigned)A.z - (unsigned)B.z) * X.fx_scale[2]};
  }
  template <int NA>
  static __device__ __forceinline__ V3 off(const Bufs& b, int cur, int a, int k) {
    const float* o = (const float*)(b.off32[cur] + 3 * (size_t)a) + k;
    return {o[0], o[4], o[8]};
  }
  static __device__ __forceinline__ float cg(const Bufs& b, int cg_n, float r, float inv_dr, float* V) {
    const float u = r * inv_dr;
    int k = (int)u;
    if (k > cg_n - 1) k = cg_n - 1;
    const float t = u - (float)k;
    const float2 lo = b.cgFV32[k], hi = b.cgFV32[k + 1];
    *V = fmaf(t, hi.y - lo.y, lo.y);
    return fmaf(t, hi.x - lo.x, lo.x);
  }
  static __device__ __forceinline__ float tf(const Bufs& b, int k) { return b.tf32[k]; }
  static __device__ __forceinline__ float fec(const Bufs& b, int k) { return b.fec32[k]; }
  static __device__ __forceinline__ float sin_(float x) { return sinf(x); }
  // hardware approximations (a few ulp): the FP32 path's error budget is 2e-5 relative; in the
  // forms that take subnormal numbers for zero, which cost two to four instructions less.  A
  // quotient is a product, so that the compiler can join it with a following sum.
  static __device__ __forceinline__ float rsqrt_(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
  static __device__ __forceinline__ float sqrt_(float x) { return x * rsqrt_(x); }
  static __device__ __forceinline__ float rcp_(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
  static __device__ __forceinline__ float acos_(float x) { return acosf(x); }
  static __device__ __forceinline__ float div_(float a, float x) { return a * rcp_(x); }
};

// ---------------- energy sums ----------------------------------------------------------------
// Energies and the virial are sums of FP32 terms in double precision.  Where the terms are FP32
// (the WCA model's) a lane keeps its sum as two floats (error-free additions, Knuth's TwoSum;
// products exact through an FMA) and only the block totals are doubles: as doubles from the start,
// conversions and additions on the FP64 pipe and the double logarithm of every bond made the
// force kernel with energies 252 us at 800k atoms where it takes 33 without.
struct Sum2 {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float a) {
    const float s = __fadd_rn(hi, a), bb = __fadd_rn(s, -hi);
    lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(hi, -__fadd_rn(s, -bb)), __fadd_rn(a, -bb)));
    hi = s;
  }
  __device__ __forceinline__ void operator+=(double x) {
    const float h = (float)x;
    add(h);
    lo = __fadd_rn(lo, (float)(x - (double)h));
  }
  // (an infinite or undefined sum leaves lo undefined)
  __device__ __forceinline__ double value() const { return isfinite(hi) ? (double)hi + (double)lo : (double)hi; }
};
__device__ __forceinline__ void acc(double& s, double x) { s += x; }
__device__ __forceinline__ void acc(Sum2& s, float x) { s.add(x); }
// the exact product of two floats
__device__ __forceinline__ void acc_product(Sum2& s, float a, float b) {
  const float p = __fmul_rn(a, b);
  s.add(p);
  s.lo = __fadd_rn(s.lo, __fmaf_rn(a, b, -p));
}
// log g (normal g > 0 table-driven, after P. T. P. Tang, "Table-driven implementation of
// the logarithm function", 1990): g = 2^e m, c = tab.x a nine-bit reciprocal of m's interval, so
// r = m c - 1 is exact in two floats and |r| < 2^-7; log g = e ln 2 - log c + log1p(r), -log c as two
// floats (tab.y, tab.z) and the series of log1p to r^5.  What the series leaves out is below 4e-14;
// the error is that of evaluating its small terms in single floats, and of ln 2 and the low parts,
// some 3e-5 each, rounded to floats: at most 1e-11 + 8e-12 |e| (measured 7e-12 for g in 0.5 .. 1,
// where the mean error is 1.6e-12, and 1.3e-11 in 0.2 .. 0.5).  g itself, a float, stands for a bond
// length known to 6e-8.
__device__ __forceinline__ void acc_log(Sum2& s, float g, const float4* tab) {
  const unsigned u = __float_as_uint(g);
  if (u - 0x00800000u >= 0x7f000000u) {  // zero, subnormal, negative, infinite or undefined
    s.add(logf(g));
    return;
  }
  const float m = __uint_as_float((u & 0x7fffffu) | 0x3f800000u);
  const float4 T = tab[(u >> 16) & 127u];
  const float e = (float)((int)(u >> 23) - 127);
  const float p = __fmul_rn(m, T.x), rl = __fmaf_rn(m, T.x, -p), r = p - 1.f;
  const float q = r * r * fmaf(r, fmaf(r, fmaf(r, 0.2f, -0.25f), 1.f / 3.f), -0.5f);
  constexpr float kLn2Hi = 0.693115234375f, kLn2Lo = 3.1946183e-05f;  // ln 2, the first to 13 bits
  s.add(e * kLn2Hi);
  s.add(T.y);
  s.add(r);
  s.lo = __fadd_rn(s.lo, fmaf(e, kLn2Lo, T.z) + (rl + q - r * rl));
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum(Sum2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h = __shfl_xor_sync(0xffffffffu, v.hi, o), l = __shfl_xor_sync(0xffffffffu, v.lo, o);
    v.add(h);
    v.lo = __fadd_rn(v.lo, l);
  }
  return v.value();
}

// ---------------- mapping of a molecule (group of four lanes) --------------------------

__device__ __forceinline__ double shfl_d(unsigned mask, double v, int src) {
  return __hiloint2double(__shfl_sync(mask, __double2hiint(v), src), __shfl_sync(mask, __double2loint(v), src));
}
__device__ __forceinline__ double shfl_xor_d(unsigned mask, double v, int o) {
  return __hiloint2double(__shfl_xor_sync(mask, __double2hiint(v), o), __shfl_xor_sync(mask, __double2loint(v), o));
}

// Centre of mass in double exactly as R = sum_k m_k (x_0 + minimg(x_k - x_0)) / M, then
// wrapped; all lanes of the group get the x component.  Used where a decision must be
// taken in FP64 (region boundaries).
template <int NA>
__device__ __forceinline__ double com_x_fp64(const Sys& s, const Box& B, unsigned gmask, int base, int g, double xk) {
  const double x0 = shfl_d(gmask, xk, base);
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < NA; ++k) {
    const double xkk = shfl_d(gmask, xk, base + k);
    acc += s.mass[k] * (x0 + minimg_cmp(xkk - x0, B.L[0], B.halfL[0]));
  }
  double r = acc / s.Mtot;
  r -= B.L[0] * floor(r / B.L[0]);
  if (r >= B.L[0]) r -= B.L[0];
  return r;
}

// Nearest resolution centre of a molecule (self-adjusting geometry): the group's four lanes
// take every fourth centre, then reduce (distance, index) so that the first of equal
// distances wins, as the definition states.  FP32: from the fixed-point centres.
__device__ __forceinline__ float nearest_center32(const Sys& s, const Box& B, const Bufs& b, unsigned gmask, int g,
                                                  const unsigned R[3], int& kmin) {
  float best = INFINITY;
  int kb = 0x7fffffff;
  for (int k = g; k < s.n_centers; k += 4) {
    const int4 C = b.cen32[k];
    const float r = sqrtf(pair_r2((float)(int)(R[0] - (unsigned)C.x) * B.fx_scale[0],
                                  (float)(int)(R[1] - (unsigned)C.y) * B.fx_scale[1],
                                  (float)(int)(R[2] - (unsigned)C.z) * B.fx_scale[2]));
    if (r < best) {
      best = r;
      kb = k;
    }
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    const float ob = __shfl_xor_sync(gmask, best, o);
    const int ok = __shfl_xor_sync(gmask, kb, o);
    if (ob < best || (ob == best && ok < kb)) {
      best = ob;
      kb = ok;
    }
  }
  kmin = kb;
  return best;
}

// FP64: from a double centre of mass, the sum of squares in the definition's order.
__device__ __forceinline__ double nearest_center64(const Sys& s, const Box& B, const Bufs& b, unsigned gmask, int g,
                                                   const double R[3], int& kmin) {
  double best = INFINITY;
  int kb = 0x7fffffff;
  for (int k = g; k < s.n_centers; k += 4) {
    const double4_32a C = b.cen64[k];
    const double t0 = minimg_cmp(R[0] - C.x, B.L[0], B.halfL[0]);
    const double t1 = minimg_cmp(R[1] - C.y, B.L[1], B.halfL[1]);
    const double t2 = minimg_cmp(R[2] - C.z, B.L[2], B.halfL[2]);
    const double r = sqrt(__dadd_rn(__dadd_rn(__dmul_rn(t0, t0), __dmul_rn(t1, t1)), __dmul_rn(t2, t2)));
    if (r < best) {
      best = r;
      kb = k;
    }
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    const double ob = shfl_xor_d(gmask, best, o);
    const int ok = __shfl_xor_sync(gmask, kb, o);
    if (ob < best || (ob == best && ok < kb)) {
      best = ob;
      kb = ok;
    }
  }
  kmin = kb;
  return best;
}

// Centre of mass in double exactly as the definition forms it (all lanes of the group get it).
template <int NA>
__device__ __forceinline__ void com_fp64(const Sys& s, const Box& B, unsigned gmask, int base, const double x[3],
                                         double R[3]) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double x0 = shfl_d(gmask, x[d], base);
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < NA; ++k) {
      const double xkk = shfl_d(gmask, x[d], base + k);
      acc += s.mass[k] * (x0 + minimg_cmp(xkk - x0, B.L[d], B.halfL[d]));
    }
    double r = acc / s.Mtot;
    r -= B.L[d] * floor(r / B.L[d]);
    if (r >= B.L[d]) r -= B.L[d];
    R[d] = r;
  }
}

// Map one molecule: fixed-point centre, resolution value, offsets, region flag.
// P32: integer fixed-point arithmetic (exact, periodic) on the bits of the doubles.
template <int NA, bool SAMPLE>
__device__ __forceinline__ void map_group32(const Sys& s, const Box& B, const Bufs& b, int nxt, int a, int g, unsigned gmask,
                                            int base, bool live, const double x[3], const int4 ref, int sample, float& ext2,
                                            float& disp2) {
  const bool own = live && g < NA;
  unsigned Pk[3], P0[3], R[3];
  int o32[3];
  float cs[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Pk[d] = fixed32(x[d], B.fxK[d], B.fxq[d]);
    P0[d] = __shfl_sync(gmask, Pk[d], base);
    const int dl = own ? (int)(Pk[d] - P0[d]) : 0;
    o32[d] = dl;
    cs[d] = s.f.frac[g < NA ? g : 0] * (float)dl;
    if (!own) cs[d] = 0.f;
    cs[d] += __shfl_xor_sync(gmask, cs[d], 1);
    cs[d] += __shfl_xor_sync(gmask, cs[d], 2);
    const int c32 = __float2int_rn(cs[d]);
    o32[d] -= c32;
    R[d] = P0[d] + (unsigned)c32;
  }
  const float3 o = make_float3((float)o32[0] * B.fx_scale[0], (float)o32[1] * B.fx_scale[1],
                               (float)o32[2] * B.fx_scale[2]);
  if (own) {
    float* of = (float*)(b.off32[nxt] + 3 * (size_t)a) + g;
    of[0] = o.x;
    of[4] = o.y;
    of[8] = o.z;
    ext2 = fmaxf(ext2, o.x * o.x + o.y * o.y + o.z * o.z);
  }
  // signed x distance to the slab centre (spheres: distance to the nearest centre); region
  // decided in FP64 near a boundary
  int kmin = 0;
  const float dxc = s.n_centers > 0 ? nearest_center32(s, B, b, gmask, g, R, kmin)
                                    : (float)(int)(R[0] - B.xc32) * B.fx_scale[0];
  float dd = fabsf(dxc);
  const bool near = fabsf(dd - B.d_at_f) < B.near_at || fabsf(dd - B.d_hyend_f) < B.near_hyend;
  // the distance in FP64 as the definition forms it (all lanes of the group call)
  auto exact_distance = [&]() -> double {
    if (s.n_centers > 0) {
      double R64[3];
      com_fp64<NA>(s, B, gmask, base, x, R64);
      int k64;
      return nearest_center64(s, B, b, gmask, g, R64, k64);
    }
    const double rx = com_x_fp64<NA>(s, B, gmask, base, g, x[0]);
    return fabs(minimg_cmp(rx - B.xc, B.L[0], B.halfL[0]));
  };
  if (SAMPLE && sample) {
    // density profile: the bin of |dxc|, decided in FP64 within 1e-4 of a bin edge (global
    // atomics: right for the run kernel's few molecules; 200,000 of them cost 20 us a sample,
    // k_density's shared-memory counts 8)
    const float u = dd * s.f.tf_inv_dx, fl = floorf(u), fr = u - fl;
    int k = (int)fl;
    if (__any_sync(gmask, live && (fr < 1e-4f || fr > 1.f - 1e-4f))) k = (int)floor(exact_distance() / s.tf_dx);
    if (live && g == 0 && k < s.tf_n) atomicAdd(&b.hist[B.tf0 + k], 1ull);
  }
  int region;  // 0 AT, 1 hybrid, 2 CG
  if (__any_sync(gmask, live && near)) {
    const double dxd = exact_distance();
    region = dxd < B.d_at ? 0 : (dxd >= B.d_at + B.d_hy ? 2 : 1);
  } else {
    region = dd < B.d_at_f ? 0 : (dd >= B.d_hyend_f ? 2 : 1);
  }
  if (live && g == 0) {
    float w = region == 0 ? 1.f : 0.f;
    if (region == 1) {
      const float c = cosf((dd - B.d_at_f) * B.pi_half_over_dhy_f);
      w = c * c;
    }
    if (s.lam_uniform_on) {
      w = s.f.lam_uniform;
      region = 0;  // no hybrid-layer forces
    }
    b.com_fx[nxt][a] = make_int4((int)R[0], (int)R[1], (int)R[2], __float_as_int(w));
    b.molf[nxt][a] = make_float2(dxc, region == 1 ? 1.f : 0.f);
    if (s.n_centers > 0) b.kcen[nxt][a] = kmin;
    const float d0 = (float)(int)(R[0] - (unsigned)ref.x) * B.fx_scale[0];
    const float d1 = (float)(int)(R[1] - (unsigned)ref.y) * B.fx_scale[1];
    const float d2 = (float)(int)(R[2] - (unsigned)ref.z) * B.fx_scale[2];
    disp2 = d0 * d0 + d1 * d1 + d2 * d2;
  }
}

// P64: the mapping in double precision; comparisons and the fixed-point copy run on the integer
// pipe (the FP64 one runs 2 lanes a clock per SM).
template <int NA, bool SAMPLE>
__device__ __forceinline__ void map_group64(const Sys& s, const Box& B, const Bufs& b, int nxt, int a, int g, unsigned gmask,
                                            int base, bool live, const double x[3], const int4 ref, int sample, float& ext2,
                                            float& disp2) {
  const bool own = live && g < NA;
  double dl[3], c[3], R[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double x0 = shfl_d(gmask, x[d], base);
    dl[d] = own ? minimg_bits(x[d] - x0, B.L[d], B.halfL[d]) : 0.0;
    double cs = own ? s.frac[g] * dl[d] : 0.0;
    cs += shfl_xor_d(gmask, cs, 1);
    cs += shfl_xor_d(gmask, cs, 2);
    c[d] = cs;
    R[d] = wrap_bits(x0 + cs, B.L[d], B.Lbits[d]);
  }
  if (own) {
    const double o0 = dl[0] - c[0], o1 = dl[1] - c[1], o2 = dl[2] - c[2];
    b.off64[nxt][a * NA + g] = make_double4_32a(o0, o1, o2, 0.0);
    // as float for the pair tests that decide where FP64 is needed
    float* of = (float*)(b.off32[nxt] + 3 * (size_t)a) + g;
    const float f0 = d2f_bits(o0), f1 = d2f_bits(o1), f2 = d2f_bits(o2);
    of[0] = f0;
    of[4] = f1;
    of[8] = f2;
    // (an undefined coordinate is left to the force's check, as fmaxf leaves out a NaN)
    auto nan = [](double v) { return ((unsigned long long)__double_as_longlong(v) << 1) > 0xFFE0000000000000ull; };
    if (!(nan(o0) || nan(o1) || nan(o2))) ext2 = fmaxf(ext2, f0 * f0 + f1 * f1 + f2 * f2);
  }
  int kmin = 0;
  const double dxc = s.n_centers > 0 ? nearest_center64(s, B, b, gmask, g, R, kmin)
                                     : minimg_cmp(R[0] - B.xc, B.L[0], B.halfL[0]);
  if (live && g == 0) {
    const double dd = fabs(dxc);
    if (SAMPLE && sample) {
      const int k = (int)floor(dd / s.tf_dx);
      if (k < s.tf_n) atomicAdd(&b.hist[B.tf0 + k], 1ull);
    }
    double w;
    if (dd < B.d_at) w = 1.0;
    else if (dd >= B.d_at + B.d_hy) w = 0.0;
    else {
      const double cs = cos((dd - B.d_at) * B.pi_half_over_dhy);
      w = cs * cs;
    }
    if (s.lam_uniform_on) w = s.lam_uniform;
    b.com64[nxt][a] = make_double4_32a(R[0], R[1], R[2], w);
    b.dxc64[nxt][a] = dxc;
    if (s.n_centers > 0) b.kcen[nxt][a] = kmin;
    unsigned X[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) X[d] = fixed32(R[d], B.fxK[d], B.fxq[d]);
    // the float weight is 0 or 1 only where the double one is
    float wf = (float)w;
    if (w < 1.0 && wf >= 1.f) wf = 0x1.fffffep-1f;
    if (w > 0.0 && !(wf > 0.f)) wf = 0x1p-126f;
    b.com_fx[nxt][a] = make_int4((int)X[0], (int)X[1], (int)X[2], __float_as_int(wf));
    const float d0 = (float)(int)(X[0] - (unsigned)ref.x) * B.fx_scale[0];
    const float d1 = (float)(int)(X[1] - (unsigned)ref.y) * B.fx_scale[1];
    const float d2 = (float)(int)(X[2] - (unsigned)ref.z) * B.fx_scale[2];
    disp2 = d0 * d0 + d1 * d1 + d2 * d2;
  }
}

// Block maximum of the molecule extent and of the displacement since the last list
// build, merged into the control block with one fire-and-forget atomic per block (no
// fence, no returned value, so blocks retire at once) into slot blockIdx mod kExtSlots:
// spread over 32 slots the blocks' atomics rarely meet at one address (one address for
// all blocks cost ~2 us of the fused step at 800k atoms); whoever takes the rebuild decision folds them.
__device__ __forceinline__ void publish_extent(const Bufs& b, int set, float ext2, float disp2) {
  __shared__ unsigned red[2][kMaxForceBlock / 32];
  const unsigned e = __reduce_max_sync(0xffffffffu, __float_as_uint(ext2));
  const unsigned dm = __reduce_max_sync(0xffffffffu, __float_as_uint(disp2));
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[0][w] = e;
    red[1][w] = dm;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned me = red[0][0], md = red[1][0];
#pragma unroll
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
      me = max(me, red[0][k]);
      md = max(md, red[1][k]);
    }
    atomicMax(&b.ctrl->ext_slot[set][0][blockIdx.x & (kExtSlots - 1)], me);
    atomicMax(&b.ctrl->ext_slot[set][1][blockIdx.x & (kExtSlots - 1)], md);
  }
}

// ---------------- k_map / k_prologue ---------------------------------------------------

template <class P, int NA, bool INTEGRATE, bool MULTI>
__global__ void __launch_bounds__(kMaxForceBlock) k_prologue(const __grid_constant__ Sys s, Bufs b) {
  const int lane = threadIdx.x & 31, g = threadIdx.x & 3, base = lane & ~3;
  const unsigned gmask = 0xFu << base;
  const int a = (blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const bool live = a < s.M;
  const int i = (live ? a : 0) * NA + (g < NA ? g : 0);
  const int nxt = b.ctrl->parity ^ 1;
  const Box& B = box_t<MULTI>(s, b, live ? a : 0);
  const size_t N = (size_t)s.N;
  const int4 ref = live && g == 0 ? b.com_ref[a] : make_int4(0, 0, 0, 0);  // centre at the last build
  double x[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    x[d] = b.x[d * N + i];
    if (INTEGRATE && live && g < NA) {
      const double fv = P::fp64 ? ((const double*)b.f)[d * N + i] : f2d_bits(((const float*)b.f)[d * N + i]);
      const double v = fma(s.hdt_m[g], fv, b.v[d * N + i]);
      x[d] = P::fp64 ? [&] {
        double y = fma(s.dt, v, x[d]);
        if (y < 0.0) y += B.L[d];
        if (y >= B.L[d]) y -= B.L[d];
        return y;
      }()
                     : wrap_bits(fma(s.dt, v, x[d]), B.L[d], B.Lbits[d]);
      b.v[d * N + i] = v;
      b.x[d * N + i] = x[d];
    }
  }
  float ext2 = 0.f, disp2 = 0.f;
  if (P::fp64) map_group64<NA, false>(s, B, b, nxt, a, g, gmask, base, live, x, ref, 0, ext2, disp2);
  else map_group32<NA, false>(s, B, b, nxt, a, g, gmask, base, live, x, ref, 0, ext2, disp2);
  publish_extent(b, 0, ext2, disp2);
}

// ---------------- k_step ----------------------------------------------------------------

// MODEL 0: WCA between atoms of different molecules (the tetrahedral fluid);
// MODEL 1: Lennard-Jones + reaction-field Coulomb per site pair (the water-like fluid).
// Resident blocks per SM the FP32 kernels are compiled for: 9 (56 registers) for the WCA model
// (200,000 molecules: 8 blocks 65.8, 9 blocks 64.1, 10 blocks 66.2 us a step), 8 with energy
// interpolation, 6 (80 registers) for the water-like model (5: 153, 6: 144, 8: 163 us).
template <class P, int MODEL, bool MULTI, bool HS>
constexpr int step_min_blocks() {
  return P::fp64 ? 1 : MODEL == 1 ? 6 : HS ? 8 : 9;
}

// How a step kernel deals out a work item's neighbours (its template parameter FORM): one lane
// per atom (four lanes an item; FP64 water-like items two such groups); one lane per neighbour
// with the lanes per item chosen by the host; the same fixed to eight and four lanes; one lane per
// atom with every force added to the atom's sum one by one, in list and bond order.  The last is
// for the learned force of the tetrahedral model: its inputs are rounded to bfloat16, which turns a
// last-bit difference of a position into 2^-9 of an input, so a trajectory should not depend on how
// sums are grouped (outliers of 1e-3 of the force RMS after 50 steps with grouped sums, none with
// ordered ones; 50 steps of 200,000 molecules 6136 us grouped, 6014 ordered).  The water-like
// model has no lane per atom in FP32: with a learned force too its sums are grouped by lanes.
constexpr int FORM_ATOM = 0, FORM_NEIGHBOUR = 1, FORM_NEIGHBOUR_8_4 = 2, FORM_ORDERED = 3;
template <int FORM, class P, int MODEL>
__device__ __forceinline__ Lanes lanes_of(Lanes chosen) {
  if (FORM == FORM_NEIGHBOUR) return chosen;
  return FORM == FORM_NEIGHBOUR_8_4 ? Lanes{3, 2} : Lanes{atom_lanes(P::fp64, MODEL) == 8 ? 3 : 2, 2};
}

// Lanes of this lane's aligned group of G (a power of two).
__device__ __forceinline__ unsigned lane_group(int G, int lane) { return (0xffffffffu >> (32 - G)) << (lane & ~(G - 1)); }

// WCA force over distance of two atom pairs, 24 eps (2 sr^12 - sr^6) / r^2 w, in the rounding order
// of the scalar expression.
__device__ __forceinline__ float2 wca_fr2(const Sys& s, float2 sr6, float2 ir2, float wab) {
  const float e24 = 24.f * s.f.eps;
  const float2 t = __ffma2_rn(__fadd2_rn(sr6, sr6), sr6, make_float2(-sr6.x, -sr6.y));
  return __fmul2_rn(__fmul2_rn(__fmul2_rn(make_float2(e24, e24), t), ir2), make_float2(wab, wab));
}

// Eq. 1 on a high-resolution molecule a of the FP32 path: lane lig of the item's G lanes takes
// every G-th neighbour, evaluates all its atom pairs with the molecule (two of the molecule's
// atoms per instruction: packed float2 arithmetic) and its coarse-grained force once, and the
// lanes' sums are exchanged at the end so that lane g holds atom g's force.  One lane per
// neighbour keeps several neighbours' loads in flight per molecule, where one lane per atom
// walked the whole list as one dependent chain (13 neighbours deep in the tetrahedral fluid,
// ~300 in the water-like one), tests each neighbour once instead of once per atom and leaves no
// lane idle for three-atom molecules.  Water-like fluid, 64,000 molecules: 189 -> 138 us a step
// (126 with later changes); tetrahedral, 1000 molecules in the run kernel: 16.9 -> 9.4
// us (8.9).
template <int NA, bool ENERGY, int MODEL, bool HS, class Acc>
__device__ __forceinline__ void hr_forces32(const Sys& s, const Box& B, const Bufs& b, int cur, int t, int a, int G, int lig, int nnb,
                                            int m_first, bool live_item, const int4 Ca, float wa, float reach_at2, float sw,
                                            bool slow, bool drift, float& fx, float& fy, float& fz, float& dv, Acc& e_at,
                                            Acc& e_cg, Acc& vir) {
  using Q = Prec<P32>;
  static_assert(MODEL == 1 || !ENERGY, "the tetrahedral model's energies: one lane per atom");
  constexpr int NP = (NA + 1) / 2;  // pairs of the molecule's atoms, an odd last one by itself
  const int lane = threadIdx.x & 31;
  const int* row = b.nbr + (size_t)(live_item ? t : 0) * s.cap;
  const float4* off = b.off32[cur];
  // everything below is minus the separation and minus the force: partner minus own
  float2 nx[NP], ny[NP], nz[NP], ax[NP], ay[NP], az[NP];
  {
    const float4 X = off[3 * (size_t)a], Y = off[3 * (size_t)a + 1], Z = off[3 * (size_t)a + 2];
    const float x[4] = {X.x, X.y, X.z, X.w}, y[4] = {Y.x, Y.y, Y.z, Y.w}, z[4] = {Z.x, Z.y, Z.z, Z.w};
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int i1 = 2 * p + 1 < NA ? 2 * p + 1 : 2 * p;
      nx[p] = make_float2(-x[2 * p], -x[i1]);
      ny[p] = make_float2(-y[2 * p], -y[i1]);
      nz[p] = make_float2(-z[2 * p], -z[i1]);
      ax[p] = ay[p] = az[p] = make_float2(0.f, 0.f);
    }
  }
  float Fx = 0.f, Fy = 0.f, Fz = 0.f;
  const float rc_at2 = s.f.rc_at2, rc_cg2 = s.f.rc_cg2;
  constexpr bool EAGER = MODEL == 0;  // short lists: fetch the offsets with the centre
  int m_n = 0;
  int4 C_n = Ca;
  float4 Xn = {}, Yn = {}, Zn = {};
  if (lig < nnb) {
    m_n = m_first;
    C_n = Q::com(b, cur, m_n);
    if (EAGER) {
      Xn = off[3 * (size_t)m_n];
      Yn = off[3 * (size_t)m_n + 1];
      Zn = off[3 * (size_t)m_n + 2];
    }
  }
  for (int q = lig; q < nnb; q += G) {
    const int m = m_n;
    const int4 Cb = C_n;
    float4 X = Xn, Y = Yn, Z = Zn;
    if (q + G < nnb) {
      m_n = row[q + G];
      C_n = Q::com(b, cur, m_n);
      if (EAGER) {
        Xn = off[3 * (size_t)m_n];
        Yn = off[3 * (size_t)m_n + 1];
        Zn = off[3 * (size_t)m_n + 2];
      }
    }
    const auto R = Q::dR(B, Cb, Ca);
    const float r2 = pair_r2(R.x, R.y, R.z);
    const float wab = HS ? 0.5f * (wa + Q::w(Cb)) : wa * Q::w(Cb);
    if (wab > 0.f && r2 < reach_at2) {
      if (!EAGER) {
        X = off[3 * (size_t)m];
        Y = off[3 * (size_t)m + 1];
        Z = off[3 * (size_t)m + 2];
      }
      const float xj[4] = {X.x, X.y, X.z, X.w}, yj[4] = {Y.x, Y.y, Y.z, Y.w}, zj[4] = {Z.x, Z.y, Z.z, Z.w};
      // two atom pairs (ia, ja), (ib, jb) with the separations dx, dy, dz; `both`: the second one
      // counts; the forces go to (fx2, fy2, fz2)
      auto pairs = [&](float2 dx, float2 dy, float2 dz, int ia, int ja, int ib, int jb, bool both, float2& fx2, float2& fy2,
                       float2& fz2) {
        const float2 d2 = __ffma2_rn(dz, dz, __ffma2_rn(dx, dx, __fmul2_rn(dy, dy)));
        const bool h0 = d2.x < rc_at2, h1 = both && d2.y < rc_at2;
        if (h0 || h1) {
          float2 fr;
          if (MODEL == 0) {
            const float2 ir2 = make_float2(Q::rcp_(d2.x), Q::rcp_(d2.y));
            const float2 sr2 = __fmul2_rn(make_float2(s.f.sig2, s.f.sig2), ir2);
            const float2 sr6 = __fmul2_rn(__fmul2_rn(sr2, sr2), sr2);
            fr = wca_fr2(s, sr6, ir2, wab);
            if (drift) {
              const float v0 = h0 ? 4.f * s.f.eps * (sr6.x * sr6.x - sr6.x) + s.f.eps : 0.f;
              const float v1 = h1 ? 4.f * s.f.eps * (sr6.y * sr6.y - sr6.y) + s.f.eps : 0.f;
              dv += v0 + v1;
            }
          } else {
            // LJ (c12 r^-12 - c6 r^-6, shifted) for the site pairs that have one + reaction
            // field q_i q_j f (1/r + k_rf r^2 - c_rf)
            const float2 ir = make_float2(Q::rsqrt_(d2.x), Q::rsqrt_(d2.y));
            const float2 ir2 = __fmul2_rn(ir, ir);
            const float2 qq = make_float2(s.f.qq[ia][ja], s.f.qq[ib][jb]);
            float2 flj = make_float2(0.f, 0.f);
            float vl0 = 0.f, vl1 = 0.f;
            if ((s.lj_pairs >> (4 * ia + ja)) & 1) {
              const float ir6 = ir2.x * ir2.x * ir2.x;
              flj.x = (12.f * s.f.c12[ia][ja] * ir6 - 6.f * s.f.c6[ia][ja]) * ir6 * ir2.x;
              if (ENERGY || drift) vl0 = (s.f.c12[ia][ja] * ir6 - s.f.c6[ia][ja]) * ir6;
            }
            if (both && ((s.lj_pairs >> (4 * ib + jb)) & 1)) {
              const float ir6 = ir2.y * ir2.y * ir2.y;
              flj.y = (12.f * s.f.c12[ib][jb] * ir6 - 6.f * s.f.c6[ib][jb]) * ir6 * ir2.y;
              if (ENERGY || drift) vl1 = (s.f.c12[ib][jb] * ir6 - s.f.c6[ib][jb]) * ir6;
            }
            fr = __ffma2_rn(qq, __ffma2_rn(ir2, ir, make_float2(-s.f.krf2, -s.f.krf2)), flj);
            fr = __fmul2_rn(fr, make_float2(wab, wab));
            if (ENERGY) {
              if (h0)
                acc(e_at, 0.5 * (double)wab *
                              ((double)vl0 + s.vsh[ia][ja] + (double)qq.x * ((double)ir.x + s.krf * (double)d2.x - s.crf)));
              if (h1)
                acc(e_at, 0.5 * (double)wab *
                              ((double)vl1 + s.vsh[ib][jb] + (double)qq.y * ((double)ir.y + s.krf * (double)d2.y - s.crf)));
            }
            if (drift) {
              if (h0) dv += vl0 + s.f.vsh[ia][ja] + qq.x * (ir.x + s.f.krf * d2.x - s.f.crf);
              if (h1) dv += vl1 + s.f.vsh[ib][jb] + qq.y * (ir.y + s.f.krf * d2.y - s.f.crf);
            }
          }
          fr.x = h0 ? fr.x : 0.f;
          fr.y = h1 ? fr.y : 0.f;
          fx2 = __ffma2_rn(fr, dx, fx2);
          fy2 = __ffma2_rn(fr, dy, fy2);
          fz2 = __ffma2_rn(fr, dz, fz2);
          if (ENERGY) {
            acc(vir, 0.5f * (fr.x * d2.x));
            acc(vir, 0.5f * (fr.y * d2.y));
          }
        }
      };
#pragma unroll
      for (int p = 0; p < NA / 2; ++p) {
        const float2 px = __fadd2_rn(nx[p], make_float2(R.x, R.x)), py = __fadd2_rn(ny[p], make_float2(R.y, R.y)),
                     pz = __fadd2_rn(nz[p], make_float2(R.z, R.z));
#pragma unroll
        for (int j = 0; j < NA; ++j)
          pairs(__fadd2_rn(px, make_float2(xj[j], xj[j])), __fadd2_rn(py, make_float2(yj[j], yj[j])),
                __fadd2_rn(pz, make_float2(zj[j], zj[j])), 2 * p, j, 2 * p + 1, j, true, ax[p], ay[p], az[p]);
      }
      if (NA & 1) {  // the odd atom takes the neighbour's atoms two at a time
        constexpr int p = NA / 2 < NP ? NA / 2 : 0;
        const float px = nx[p].x + R.x, py = ny[p].x + R.y, pz = nz[p].x + R.z;
        const float2 p2 = make_float2(px, px), q2 = make_float2(py, py), r2p = make_float2(pz, pz);
#pragma unroll
        for (int j = 0; j < NA; j += 2) {
          const int j1 = j + 1 < NA ? j + 1 : j;
          pairs(__fadd2_rn(p2, make_float2(xj[j], xj[j1])), __fadd2_rn(q2, make_float2(yj[j], yj[j1])),
                __fadd2_rn(r2p, make_float2(zj[j], zj[j1])), NA - 1, j, NA - 1, j1, j1 != j, ax[p], ay[p], az[p]);
        }
      }
    }
    if (wab < 1.f && r2 < rc_cg2 && slow) {
      const float r = Q::sqrt_(r2);
      float V = 0.f;
      const float F = s.cg_mode ? b.fpair[(size_t)t * s.cap + q] : Q::cg(b, s.cg_n, r, s.f.cg_inv_dr, &V);
      const float fw = (1.f - wab) * F;
      const float c = Q::div_(fw * sw, r);
      Fx += c * R.x;
      Fy += c * R.y;
      Fz += c * R.z;
      if (ENERGY) {
        acc(e_cg, 0.5f * ((1.f - wab) * V));
        acc(vir, 0.5f * (Q::div_(fw, r) * r2));
      }
      if (drift) dv -= sw * V;
    }
  }
  // the atoms' sums with their share of the coarse-grained force, then exchanged within the
  // group: first halves (atoms 0, 1 / 2, 3), then single atoms, then the groups of four
  float f4[4][3];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int p = i / 2 < NP ? i / 2 : 0;
    // (an odd last atom's sums lie in both halves)
    auto of = [&](float2 v) { return (NA & 1) && i == NA - 1 ? v.x + v.y : (i & 1) ? v.y : v.x; };
    f4[i][0] = i < NA ? fmaf(s.f.frac[i], Fx, of(ax[p])) : 0.f;
    f4[i][1] = i < NA ? fmaf(s.f.frac[i], Fy, of(ay[p])) : 0.f;
    f4[i][2] = i < NA ? fmaf(s.f.frac[i], Fz, of(az[p])) : 0.f;
  }
  const unsigned mk = lane_group(G, lane);
  float r[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const bool up = lane & 2, odd = lane & 1;
    float k0 = up ? f4[2][c] : f4[0][c], k1 = up ? f4[3][c] : f4[1][c];
    k0 += __shfl_xor_sync(mk, up ? f4[0][c] : f4[2][c], 2);
    k1 += __shfl_xor_sync(mk, up ? f4[1][c] : f4[3][c], 2);
    r[c] = (odd ? k1 : k0) + __shfl_xor_sync(mk, odd ? k0 : k1, 1);
  }
  for (int o = kGroup; o < G; o <<= 1) {
#pragma unroll
    for (int c = 0; c < 3; ++c) r[c] += __shfl_xor_sync(mk, r[c], o);
  }
  fx = -r[0];
  fy = -r[1];
  fz = -r[2];
  if (HS) {  // V_AT_a - V_CG_a = half the group's sum (every pair is listed from both sides)
    for (int o = 1; o < G; o <<= 1) dv += __shfl_xor_sync(mk, dv, o);
    dv *= 0.5f;
  }
}

// The same with one lane per atom: lane g evaluates its atom against every listed neighbour
// (two of the neighbour's atoms per packed instruction), the next neighbour's index and centre
// fetched while the current one is evaluated.  Fewer registers than one lane per neighbour (56
// against the 128 it has in the run kernel, so twice the warps): the faster way once there are
// enough molecules to fill the device.
// ORDERED: one sum per component, every term added to it by itself.
template <int NA, bool ENERGY, bool HS, bool ORDERED, class Acc>
__device__ __forceinline__ void hr_forces32_atom(const Sys& s, const Box& B, const Bufs& b, int cur, int t, int g, int nnb,
                                                 int m_first, const int* row, const int4 Ca, float wa, float3 oi, float frac_g,
                                                 float reach_at2, float sw, bool slow, bool drift, float& fx, float& fy,
                                                 float& fz, float& dv, Acc& e_at, Acc& e_cg, Acc& vir) {
  using Q = Prec<P32>;
  constexpr int NP = (NA + 1) / 2;  // pairs of the neighbour's atoms (an odd last one is doubled)
  const float4* off = b.off32[cur];
  const float rc_at2 = s.f.rc_at2, rc_cg2 = s.f.rc_cg2;
  float2 ax = make_float2(0.f, 0.f), ay = ax, az = ax;
  float Fx = 0.f, Fy = 0.f, Fz = 0.f;
  int m_n = m_first;
  int4 C_n = Ca;
  if (nnb > 0) C_n = Q::com(b, cur, m_n);
  for (int q = 0; q < nnb; ++q) {
    const int m = m_n;
    const int4 Cb = C_n;
    if (q + 1 < nnb) {
      m_n = row[q + 1];
      C_n = Q::com(b, cur, m_n);
    }
    const auto R = Q::dR(B, Cb, Ca);  // minus the separation, as everything below
    const float r2 = pair_r2(R.x, R.y, R.z);
    const float wab = HS ? 0.5f * (wa + Q::w(Cb)) : wa * Q::w(Cb);
    if (wab > 0.f && r2 < reach_at2 && g < NA) {
      const float4 X = off[3 * (size_t)m], Y = off[3 * (size_t)m + 1], Z = off[3 * (size_t)m + 2];
      const float xj[4] = {X.x, X.y, X.z, X.w}, yj[4] = {Y.x, Y.y, Y.z, Y.w}, zj[4] = {Z.x, Z.y, Z.z, Z.w};
      const float px = R.x - oi.x, py = R.y - oi.y, pz = R.z - oi.z;
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const int j0 = 2 * p, j1 = 2 * p + 1 < NA ? 2 * p + 1 : 2 * p;
        const float2 dx = __fadd2_rn(make_float2(xj[j0], xj[j1]), make_float2(px, px));
        const float2 dy = __fadd2_rn(make_float2(yj[j0], yj[j1]), make_float2(py, py));
        const float2 dz = __fadd2_rn(make_float2(zj[j0], zj[j1]), make_float2(pz, pz));
        const float2 d2 = __ffma2_rn(dz, dz, __ffma2_rn(dx, dx, __fmul2_rn(dy, dy)));
        const bool h0 = d2.x < rc_at2, h1 = j1 != j0 && d2.y < rc_at2;
        if (h0 || h1) {
          const float2 ir2 = make_float2(Q::rcp_(d2.x), Q::rcp_(d2.y));
          const float2 sr2 = __fmul2_rn(make_float2(s.f.sig2, s.f.sig2), ir2);
          const float2 sr6 = __fmul2_rn(__fmul2_rn(sr2, sr2), sr2);
          float2 fr = wca_fr2(s, sr6, ir2, wab);
          if (ENERGY || drift) {
            const float v0 = h0 ? 4.f * s.f.eps * (sr6.x * sr6.x - sr6.x) + s.f.eps : 0.f;
            const float v1 = h1 ? 4.f * s.f.eps * (sr6.y * sr6.y - sr6.y) + s.f.eps : 0.f;
            if (ENERGY) {
              acc_product(e_at, 0.5f * wab, v0);
              acc_product(e_at, 0.5f * wab, v1);
            }
            if (drift) dv += v0 + v1;
          }
          fr.x = h0 ? fr.x : 0.f;
          fr.y = h1 ? fr.y : 0.f;
          if (ORDERED) {
            ax.x = fmaf(fr.y, dx.y, fmaf(fr.x, dx.x, ax.x));
            ay.x = fmaf(fr.y, dy.y, fmaf(fr.x, dy.x, ay.x));
            az.x = fmaf(fr.y, dz.y, fmaf(fr.x, dz.x, az.x));
          } else {
            ax = __ffma2_rn(fr, dx, ax);
            ay = __ffma2_rn(fr, dy, ay);
            az = __ffma2_rn(fr, dz, az);
          }
          if (ENERGY) {
            acc(vir, 0.5f * (fr.x * d2.x));
            acc(vir, 0.5f * (fr.y * d2.y));
          }
        }
      }
    }
    if (wab < 1.f && r2 < rc_cg2 && slow && g < NA) {
      const float r = Q::sqrt_(r2);
      float V = 0.f;
      const float F = s.cg_mode ? b.fpair[(size_t)t * s.cap + q] : Q::cg(b, s.cg_n, r, s.f.cg_inv_dr, &V);
      const float fw = (1.f - wab) * F;
      const float c = Q::div_(fw * sw, r);
      if (ORDERED) {
        const float cf = frac_g * c;
        ax.x = fmaf(cf, R.x, ax.x);
        ay.x = fmaf(cf, R.y, ay.x);
        az.x = fmaf(cf, R.z, az.x);
      } else {
        Fx += c * R.x;
        Fy += c * R.y;
        Fz += c * R.z;
      }
      if (ENERGY && g == 0) {
        acc(e_cg, 0.5f * ((1.f - wab) * V));
        acc(vir, 0.5f * (Q::div_(fw, r) * r2));
      }
      if (drift && g == 0) dv -= sw * V;
    }
  }
  fx = ORDERED ? -ax.x : -fmaf(frac_g, Fx, ax.x + ax.y);
  fy = ORDERED ? -ay.x : -fmaf(frac_g, Fy, ay.x + ay.y);
  fz = ORDERED ? -az.x : -fmaf(frac_g, Fz, az.x + az.y);
  if (HS) {  // V_AT_a - V_CG_a = half the group's sum (every pair is listed from both sides)
    const unsigned gmask = 0xFu << (threadIdx.x & 28);
    dv += __shfl_xor_sync(gmask, dv, 1);
    dv += __shfl_xor_sync(gmask, dv, 2);
    dv *= 0.5f;
  }
}

// Eq. 1 on a high-resolution molecule a of the FP64 path: lane g has atom g, lane group `sub` of
// SPLIT every SPLIT-th neighbour.  The FP64 pipe is the bound (2 lanes a clock per SM against
// 128 in FP32), and nine of ten listed atom pairs are beyond the cutoff, so a batch of
// neighbours is first tested in FP32 with a margin (fixed-point centres and float offsets; the
// margin, Sys::f.pretest, covers both and grows with the box) and only what passes is evaluated,
// and tested again, in FP64; the coarse-grained force of a pair is evaluated by one lane of the
// group.  800k atoms: 930 -> 516 us a step, 80k atoms all-atomistic 216 -> 80 us (400 and
// 64 us with the bonds evaluated once and positions wrapped in integers).
template <int NA, bool ENERGY, int MODEL, bool HS, int SPLIT>
__device__ __forceinline__ void hr_forces64(const Sys& s, const Box& B, const Bufs& b, int cur, int t, int a, int g, int sub, int nnb,
                                            bool live_item, const int* row, const double4_32a Ca, const double4_32a oi,
                                            double frac_g, double reach_at2, double sw, bool slow, bool drift,
                                            const double (&c12r)[NA], const double (&c6r)[NA], const double (&qqr)[NA],
                                            double& fx, double& fy, double& fz, double& dv, double& e_at, double& e_cg,
                                            double& vir) {
  using Q = Prec<P64>;
  constexpr int kBatch = 16;  // neighbours per batch: four hit bits each
  const float rcf = s.f.rc_at2 * s.f.pretest, rcgf = s.f.rc_cg2 * s.f.pretest, reachf = (float)reach_at2 * s.f.pretest;
  const int4 Cf = b.com_fx[cur][a];
  const float waf = __int_as_float(Cf.w);
  const float* of = (const float*)(b.off32[cur] + 3 * (size_t)a) + (g < NA ? g : 0);
  const float ox = of[0], oy = of[4], oz = of[8];
  const int gg = g < NA ? g : 0;
  double Fx = 0.0, Fy = 0.0, Fz = 0.0;
  for (int q0 = sub; q0 < nnb; q0 += kBatch * SPLIT) {
    unsigned long long hits = 0ull;
    unsigned cgs = 0u;
    int m_n = row[q0];
    int4 C_n = b.com_fx[cur][m_n];
    for (int k = 0; k < kBatch; ++k) {
      const int q = q0 + k * SPLIT;
      if (q >= nnb) break;
      const int m = m_n;
      const int4 Cb = C_n;
      if (k + 1 < kBatch && q + SPLIT < nnb) {
        m_n = row[q + SPLIT];
        C_n = b.com_fx[cur][m_n];
      }
      const float Rx = (float)(int)((unsigned)Cf.x - (unsigned)Cb.x) * B.fx_scale[0];
      const float Ry = (float)(int)((unsigned)Cf.y - (unsigned)Cb.y) * B.fx_scale[1];
      const float Rz = (float)(int)((unsigned)Cf.z - (unsigned)Cb.z) * B.fx_scale[2];
      const float r2 = pair_r2(Rx, Ry, Rz), wbf = __int_as_float(Cb.w);
      if (g < NA && r2 < reachf && (HS ? waf > 0.f || wbf > 0.f : waf > 0.f && wbf > 0.f)) {
        const float4* off = b.off32[cur] + 3 * (size_t)m;
        const float4 X = off[0], Y = off[1], Z = off[2];
        const float xj[4] = {X.x, X.y, X.z, X.w}, yj[4] = {Y.x, Y.y, Y.z, Y.w}, zj[4] = {Z.x, Z.y, Z.z, Z.w};
        const float px = Rx + ox, py = Ry + oy, pz = Rz + oz;
#pragma unroll
        for (int j = 0; j < NA; ++j) {
          const float dx = px - xj[j], dy = py - yj[j], dz = pz - zj[j];
          if (dx * dx + dy * dy + dz * dz < rcf) hits |= 1ull << (4 * k + j);
        }
      }
      if ((k & 3) == g && slow && r2 < rcgf && (waf < 1.f || wbf < 1.f)) cgs |= 1u << k;
    }
    while (hits) {
      const int bit = __ffsll((long long)hits) - 1;
      hits &= hits - 1;
      const int m = row[q0 + (bit >> 2) * SPLIT], j = bit & 3;
      const double4_32a Cb = b.com64[cur][m], oj = b.off64[cur][m * NA + j];
      const auto R = Q::dR(B, Ca, Cb);
      const double wab = HS ? 0.5 * (Ca.w + Cb.w) : Ca.w * Cb.w;
      const double dx = R.x + oi.x - oj.x, dy = R.y + oi.y - oj.y, dz = R.z + oi.z - oj.z;
      const double d2 = dx * dx + dy * dy + dz * dz;
      if (d2 < s.rc_at2) {
        double fr;
        if (MODEL == 0) {
          const double ir2 = rcp_nr(d2);
          const double sr2 = s.sig2 * ir2;
          const double sr6 = sr2 * sr2 * sr2;
          fr = 24.0 * s.eps * (2.0 * sr6 * sr6 - sr6) * ir2 * wab;
          if (ENERGY) e_at += 0.5 * wab * (4.0 * s.eps * (sr6 * sr6 - sr6) + s.eps);
          if (drift) dv += 4.0 * s.eps * (sr6 * sr6 - sr6) + s.eps;
        } else {
          // LJ (c12 r^-12 - c6 r^-6, shifted) + reaction field q_i q_j f (1/r + k_rf r^2 - c_rf);
          // this atom's coefficients with site j
          double c12 = c12r[0], c6 = c6r[0], qq = qqr[0];
#pragma unroll
          for (int e = 1; e < NA; ++e)
            if (j == e) {
              c12 = c12r[e];
              c6 = c6r[e];
              qq = qqr[e];
            }
          const double ir = rsqrt_nr(d2), ir2 = ir * ir;
          double flj = 0.0, vlj = 0.0;
          if ((s.lj_cols >> j) & 1) {
            const double ir6 = ir2 * ir2 * ir2;
            flj = (12.0 * c12 * ir6 - 6.0 * c6) * ir6 * ir2;
            if (ENERGY || drift) vlj = (c12 * ir6 - c6) * ir6;
          }
          fr = (flj + qq * (ir2 * ir - 2.0 * s.krf)) * wab;
          if (ENERGY || drift) {
            const double v = vlj + s.vsh[gg][j] + qq * (ir + s.krf * d2 - s.crf);
            if (ENERGY) e_at += 0.5 * wab * v;
            if (drift) dv += v;
          }
        }
        fx += fr * dx;
        fy += fr * dy;
        fz += fr * dz;
        if (ENERGY) vir += 0.5 * (fr * d2);
      }
    }
    while (cgs) {
      const int k = __ffs((int)cgs) - 1;
      cgs &= cgs - 1;
      const int q = q0 + k * SPLIT;
      const double4_32a Cb = b.com64[cur][row[q]];
      const auto R = Q::dR(B, Ca, Cb);
      const double r2 = pair_r2(R.x, R.y, R.z);
      const double wab = HS ? 0.5 * (Ca.w + Cb.w) : Ca.w * Cb.w;
      if (wab < 1.0 && r2 < s.rc_cg2) {
        const double ir = rsqrt_nr(r2), r = r2 * ir;
        double V = 0.0;
        const double F = s.cg_mode ? (double)b.fpair[(size_t)t * s.cap + q] : Q::cg(b, s.cg_n, r, s.cg_inv_dr, &V);
        const double fw = (1.0 - wab) * F, c = fw * sw * ir;
        Fx += c * R.x;
        Fy += c * R.y;
        Fz += c * R.z;
        if (ENERGY) {
          e_cg += 0.5 * (1.0 - wab) * V;
          vir += 0.5 * (fw * r);
        }
        if (drift) dv -= sw * V;
      }
    }
  }
  const unsigned gmask = 0xFu << (threadIdx.x & 28);
#pragma unroll
  for (int o = 1; o < kGroup; o <<= 1) {
    Fx += shfl_xor_d(gmask, Fx, o);
    Fy += shfl_xor_d(gmask, Fy, o);
    Fz += shfl_xor_d(gmask, Fz, o);
  }
  fx += frac_g * Fx;
  fy += frac_g * Fy;
  fz += frac_g * Fz;
}

// The step of the molecules of one tile of the grid (a block's worth of threads): thread gtid
// of the whole grid.  cur: current half of the molecule arrays; step: the time level of the
// forces; ext_now: the largest atom-to-COM distance; sample (SAMPLE): add the next mapping's
// molecules to the density profile; its maxima are merged into ext2 and disp2 (MODE_FUSED).  Every thread of a block calls.
//
// A high-resolution work item takes 2^ln.h lanes and a coarse-grained one 2^ln.c (32 >= 2^h >=
// 2^c >= 4, so that no item's lanes straddle a warp); the first four integrate and map the
// molecule, one lane per atom.  LPN: one lane per neighbour (hr_forces32), else per atom (ORDERED:
// FORM_ORDERED).
template <class P, int NA, int MODE, bool ENERGY, bool MULTI, int MODEL, bool HS, bool LPN, bool SAMPLE, bool ORDERED>
__device__ __forceinline__ void step_tile(const Sys& s, const Bufs& b, const Lanes ln, const int gtid, const int cur,
                                          const long long step, const float ext_now, const int sample, float& ext2,
                                          float& disp2) {
  using Q = Prec<P>;
  using real = typename Q::real;
  const int lane = threadIdx.x & 31, g = threadIdx.x & 3, base = lane & ~3;
  const unsigned gmask = 0xFu << base;
  const int n_hr = b.ctrl->n_hr, GC = 1 << ln.c;
  const bool hr_item = gtid < (n_hr << ln.h);
  // work item and this lane's place in its group
  const int u = hr_item || ln.h == ln.c ? gtid : gtid - (n_hr << ln.h);
  const int t = hr_item || ln.h == ln.c ? u >> ln.h : n_hr + (u >> ln.c);
  const int lig = u & ((1 << (hr_item ? ln.h : ln.c)) - 1);
  const bool live_item = t < s.M;
  const bool live = live_item && lig < kGroup;  // the lanes that integrate and map the molecule
  const bool own = live && g < NA;
  // the first list slot this lane reads is fetched together with the item, before the count
  // is known (slots below the capacity lie inside the list array; the value is used only
  // when the count covers the slot)
  // (one lane per atom: the four lanes of a group share a slot)
  const int j0 = !LPN && hr_item ? lig / kGroup : lig;
  const int* row = b.nbr + (size_t)(live_item ? t : 0) * s.cap;
  const int m_first = live_item && j0 < s.cap ? row[j0] : 0;

  const real eps = par<real>(s.eps, s.f.eps), sig2 = par<real>(s.sig2, s.f.sig2);
  const real rc_at2 = par<real>(s.rc_at2, s.f.rc_at2), rc_cg2 = par<real>(s.rc_cg2, s.f.rc_cg2);
  const real inv_dr = par<real>(s.cg_inv_dr, s.f.cg_inv_dr);
  const real reach = par<real>(s.rc_at, s.f.rc_at) + (real)2 * (real)ext_now;
  const real reach_at2 = reach * reach;
  const int gg0 = g < NA ? g : 0;
  const real frac_g = par<real>(s.frac[gg0], s.f.frac[gg0]);
  // MODEL 1: this atom's row of the site-pair coefficients (FP64 path)
  real c12r[NA], c6r[NA], qqr[NA];
  real krf2 = 0;
  if (MODEL == 1) {
#pragma unroll
    for (int j = 0; P::fp64 && j < NA; ++j) {
      c12r[j] = par<real>(s.c12[gg0][j], s.f.c12[gg0][j]);
      c6r[j] = par<real>(s.c6[gg0][j], s.f.c6[gg0][j]);
      qqr[j] = par<real>(s.qq[gg0][j], s.f.qq[gg0][j]);
    }
    krf2 = par<real>(2.0 * s.krf, s.f.krf2);
  }

  real fx = 0, fy = 0, fz = 0;
  using Acc = std::conditional_t<!P::fp64 && MODEL == 0, Sum2, double>;
  Acc e_at{}, e_cg{}, e_b{}, vir{}, e_log{};  // e_log: sum of the FENE logarithms

  const int a = live_item ? b.items[t] : 0;
  const Box& B = box_t<MULTI>(s, b, a);
  // centre at the last list build, for the displacement the next mapping reports: fetched
  // now so that its latency hides behind the force loops
  const int4 ref = MODE == MODE_FUSED && live && g == 0 ? b.com_ref[a] : make_int4(0, 0, 0, 0);
  const int i = a * NA + (g < NA ? g : 0);
  const auto Ca = Q::com(b, cur, a);
  const real wa = Q::w(Ca);
  const auto oi = Q::template off<NA>(b, cur, a, g < NA ? g : 0);
  const int nnb = live_item ? b.nn[t] : 0;
  // energy interpolation: a hybrid molecule sums its unweighted pair energies (AT per atom
  // lane, CG on lane 0 of its group) for the drift force
  constexpr bool hs = HS;
  const bool drift = hs && wa > (real)0 && wa < (real)1 && !s.lam_uniform_on;
  real dv = 0;
  // slow-force weight at this time level (1 without multiple time stepping)
  real sw = 1;
  if (s.respa_n > 1) sw = step % s.respa_n == 0 ? (real)s.respa_n : (real)0;
  const bool slow = sw != (real)0 || ENERGY;

  if (hr_item) {
    if constexpr (!P::fp64 && !LPN) {
      static_assert(MODEL == 0, "one lane per atom");
      hr_forces32_atom<NA, ENERGY, HS, ORDERED>(s, B, b, cur, t, g, nnb, m_first, row, Ca, wa, make_float3(oi.x, oi.y, oi.z), frac_g,
                                       reach_at2, sw, slow, drift, fx, fy, fz, dv, e_at, e_cg, vir);
    } else if constexpr (!P::fp64) {
      hr_forces32<NA, ENERGY, MODEL, HS>(s, B, b, cur, t, a, 1 << ln.h, lig, nnb, m_first, live_item, Ca, wa, reach_at2, sw, slow, drift,
                                             fx, fy, fz, dv, e_at, e_cg, vir);
    } else {
    constexpr int SPLIT = atom_lanes(true, MODEL) / kGroup;
    hr_forces64<NA, ENERGY, MODEL, HS, SPLIT>(s, B, b, cur, t, a, g, lig / kGroup, nnb, live_item, row, Ca, oi, frac_g, reach_at2,
                                              sw, slow, drift, c12r, c6r, qqr, fx, fy, fz, dv, e_at, e_cg, vir);
    if (SPLIT > 1) {  // the groups' shares of the force (energies are summed per warp)
      const unsigned mk = SPLIT == 2 ? 0xFFu << (lane & 24) : 0xFFFFu << (lane & 16);
#pragma unroll
      for (int o = kGroup; o < kGroup * SPLIT; o <<= 1) {
        fx += __shfl_xor_sync(mk, fx, o);
        fy += __shfl_xor_sync(mk, fy, o);
        fz += __shfl_xor_sync(mk, fz, o);
        if (hs) dv += __shfl_xor_sync(mk, dv, o);
      }
    }
    if (hs) {  // V_AT_a - V_CG_a = half the group's sum (every pair is listed from both sides)
      dv += __shfl_xor_sync(gmask, dv, 1);
      dv += __shfl_xor_sync(gmask, dv, 2);
      dv *= (real)0.5;
    }
    }
  } else {
    // coarse-grained item (l_a = 0, so w_ab = 0): neighbour list split over the group
    if (live && g == 0 && wa != (real)0) set_error(b.ctrl, ADRESS_ERR_STATE, a);
    real Fx = 0, Fy = 0, Fz = 0;
    const int nnb_cg = slow ? nnb : 0;  // no CG force at inner levels of multiple time stepping
    auto pair_cg = [&](int q, const typename Q::V3& R, real r2) {
      // (the FP64 path has 1/r at hand and divides by multiplying)
      const real ir = P::fp64 ? Q::rsqrt_(r2) : (real)0, r = P::fp64 ? r2 * ir : (real)Prec<P32>::sqrt_((float)r2);
      real V = 0;
      const real F = s.cg_mode ? (real)b.fpair[(size_t)t * s.cap + q] : Q::cg(b, s.cg_n, r, inv_dr, &V);
      const real c = P::fp64 ? F * ir : Q::div_(F, r);
      Fx += c * R.x;
      Fy += c * R.y;
      Fz += c * R.z;
      if (ENERGY) {
        acc(e_cg, (real)0.5 * V);
        acc(vir, (real)0.5 * (c * r2));
      }
    };
    // centres of the next two neighbours in flight (long lists: the water-like fluid); the FP64
    // path tests the fixed-point ones in FP32 with a margin first (see hr_forces64)
    const int4* cfx = b.com_fx[cur];
    const int4 Cf = P::fp64 ? cfx[a] : (const int4&)Ca;
    const float rcgf = P::fp64 ? s.f.rc_cg2 * s.f.pretest : s.f.rc_cg2;
    int m_n = m_first, m_n2 = 0;
    int4 C_n = Cf, C_n2 = Cf;
    if (lig < nnb_cg) C_n = cfx[m_n];
    if (lig + GC < nnb_cg) {
      m_n2 = row[lig + GC];
      C_n2 = cfx[m_n2];
    }
    for (int q = lig; q < nnb_cg; q += GC) {
      const int m = m_n;
      const int4 Cb = C_n;
      m_n = m_n2;
      C_n = C_n2;
      if (q + 2 * GC < nnb_cg) {
        m_n2 = row[q + 2 * GC];
        C_n2 = cfx[m_n2];
      }
      const auto Rf = Prec<P32>::dR(B, Cf, Cb);
      const float r2f = pair_r2(Rf.x, Rf.y, Rf.z);
      if (r2f < rcgf) {
        if constexpr (P::fp64) {
          const auto R = Q::dR(B, Ca, Q::com(b, cur, m));
          const real r2 = pair_r2(R.x, R.y, R.z);
          if (r2 < rc_cg2) pair_cg(q, R, r2);
        } else {
          pair_cg(q, Rf, r2f);
        }
      }
    }
    const unsigned mk = lane_group(GC, lane);
    for (int o = 1; o < GC; o <<= 1) {
      Fx += __shfl_xor_sync(mk, Fx, o);
      Fy += __shfl_xor_sync(mk, Fy, o);
      Fz += __shfl_xor_sync(mk, Fz, o);
    }
    const real fs = frac_g * sw;
    fx = fs * Fx;
    fy = fs * Fy;
    fz = fs * Fz;
  }

  // own state for the update, fetched before the bonded terms so the loads overlap them
  const size_t N = (size_t)s.N;
  double xo[3] = {0.0, 0.0, 0.0}, vo[3] = {0.0, 0.0, 0.0};
  if (MODE != MODE_FORCES && own) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      vo[d] = b.v[d * N + i];
      if (MODE == MODE_FUSED) xo[d] = b.x[d * N + i];
    }
  }

  // offset of atom k of this molecule: from its lane on the FP32 path (every lane of the group
  // calls), from memory on the FP64 path
  auto atom_off = [&](int k) {
    if constexpr (P::fp64) {
      return Q::template off<NA>(b, cur, a, k);
    } else {
      return typename Q::V3{__shfl_sync(gmask, oi.x, base + k), __shfl_sync(gmask, oi.y, base + k),
                            __shfl_sync(gmask, oi.z, base + k)};
    }
  };
  if (live) {
    // bonded terms: harmonic bonds and angles, or FENE + WCA, on the listed intramolecular
    // pairs.  A bond is evaluated once, by one of its atoms, in one of bond_rounds rounds (six
    // bonds of a tetrahedron: two); the other atom gets the force by a shuffle.  Every lane of the
    // group takes part in the shuffles.
    const unsigned send = own ? s.bond_send[gg0] : 0u, recv = own ? s.bond_recv[gg0] : 0u;
    auto give = [&](int q, real bx, real by, real bz) {
      const int rv = (recv >> (4 * q)) & 15;
      real tx, ty, tz;
      if constexpr (P::fp64) {
        tx = shfl_d(gmask, bx, base + (rv & 3));
        ty = shfl_d(gmask, by, base + (rv & 3));
        tz = shfl_d(gmask, bz, base + (rv & 3));
      } else {
        tx = __shfl_sync(gmask, bx, base + (rv & 3));
        ty = __shfl_sync(gmask, by, base + (rv & 3));
        tz = __shfl_sync(gmask, bz, base + (rv & 3));
      }
      if (rv & 8) {
        fx -= tx;
        fy -= ty;
        fz -= tz;
      }
    };
    if (s.bond_model == 1) {
      const real kb = par<real>(s.bond_k, s.f.bond_k), r0 = par<real>(s.bond_r0, s.f.bond_r0);
#pragma unroll
      for (int q = 0; q < kMaxBonds; ++q) {
        if (q >= s.bond_rounds) break;
        const int e = (send >> (4 * q)) & 15;
        const auto oo = atom_off(e & 3);
        real bx = 0, by = 0, bz = 0;
        if (e & 8) {
          const real dx = (real)oi.x - (real)oo.x, dy = (real)oi.y - (real)oo.y, dz = (real)oi.z - (real)oo.z;
          const real d2 = dx * dx + dy * dy + dz * dz;
          const real ird = Q::rsqrt_(d2);
          const real dl = d2 * ird;
          const real fr = -kb * (dl - r0) * ird;  // V = k/2 (r - r0)^2
          bx = fr * dx;
          by = fr * dy;
          bz = fr * dz;
          fx = fma_(fr, dx, fx);
          fy = fma_(fr, dy, fy);
          fz = fma_(fr, dz, fz);
          if (ENERGY) {
            e_b += 0.5 * (double)kb * (double)(dl - r0) * (double)(dl - r0);
            acc(vir, fr * d2);
          }
        }
        give(q, bx, by, bz);
      }
      // harmonic angles (i, vertex j, k): V = k/2 (theta - theta0)^2; the force on i is
      // dV/dtheta (v/(|u||v|) - cos(theta) u/|u|^2) / sin(theta), u = x_i - x_j, v = x_k - x_j,
      // likewise on k, and minus their sum on the vertex
      const real ka = par<real>(s.angle_k, s.f.angle_k), th0 = par<real>(s.angle_theta0, s.f.angle_theta0);
#pragma unroll
      for (int q = 0; q < kMaxAngles; ++q) {
        if (q >= s.n_angles) break;
        const int ai = s.angles[3 * q], aj = s.angles[3 * q + 1], ak = s.angles[3 * q + 2];
        const auto Oi = atom_off(ai), Oj = atom_off(aj), Ok = atom_off(ak);
        if (g != ai && g != aj && g != ak) continue;
        const real ux = (real)Oi.x - (real)Oj.x, uy = (real)Oi.y - (real)Oj.y, uz = (real)Oi.z - (real)Oj.z;
        const real vx = (real)Ok.x - (real)Oj.x, vy = (real)Ok.y - (real)Oj.y, vz = (real)Ok.z - (real)Oj.z;
        const real uu = ux * ux + uy * uy + uz * uz, vv = vx * vx + vy * vy + vz * vz;
        const real uv = ux * vx + uy * vy + uz * vz;
        const real iuv = Q::rsqrt_(uu * vv);
        real c = uv * iuv;
        c = c > (real)1 ? (real)1 : (c < (real)-1 ? (real)-1 : c);
        const real th = Q::acos_(c);
        const real s2 = (real)1 - c * c;
        const real gq = s2 > (real)0 ? ka * (th - th0) * Q::rsqrt_(s2) : (real)0;
        const real iu = Q::rcp_(uu), iv = Q::rcp_(vv);
        const real fix = gq * (vx * iuv - c * ux * iu), fiy = gq * (vy * iuv - c * uy * iu), fiz = gq * (vz * iuv - c * uz * iu);
        const real fkx = gq * (ux * iuv - c * vx * iv), fky = gq * (uy * iuv - c * vy * iv), fkz = gq * (uz * iuv - c * vz * iv);
        if (g == ai) {
          fx += fix;
          fy += fiy;
          fz += fiz;
        } else if (g == ak) {
          fx += fkx;
          fy += fky;
          fz += fkz;
        } else {
          fx -= fix + fkx;
          fy -= fiy + fky;
          fz -= fiz + fkz;
          if (ENERGY) {
            e_b += 0.5 * (double)ka * (double)(th - th0) * (double)(th - th0);
            acc(vir, ux * fix + uy * fiy + uz * fiz + vx * fkx + vy * fky + vz * fkz);
          }
        }
      }
    } else {
      const real R02 = par<real>(s.fene_r02, s.f.fene_r02), K = par<real>(s.fene_k, s.f.fene_k);
      // FENE + WCA with the atom at oo, added to this atom's force; its energy if it counts; the
      // force itself, for the other atom
      auto fene = [&](auto oo, bool counts, real& bx, real& by, real& bz) {
        const real dx = (real)oi.x - (real)oo.x, dy = (real)oi.y - (real)oo.y, dz = (real)oi.z - (real)oo.z;
        const real d2 = dx * dx + dy * dy + dz * dz;
        if (d2 >= R02) {
          set_error(b.ctrl, ADRESS_ERR_BOND_BROKEN, a);
        } else {
          const real gg = (real)1 - (P::fp64 ? d2 * (real)s.fene_inv_r02 : Q::div_(d2, R02));
          real fr = Q::div_(-K, gg);
          if (ENERGY && counts) {
            if constexpr (std::is_same_v<Acc, Sum2>) acc_log(e_log, gg, b.log_tab);
            else e_log += log((double)gg);
          }
          if (s.intra_wca && d2 < rc_at2) {
            const real ir2 = Q::rcp_(d2);
            const real sr2 = sig2 * ir2;
            const real sr6 = sr2 * sr2 * sr2;
            fr += (real)24 * eps * ((real)2 * sr6 * sr6 - sr6) * ir2;
            if (ENERGY && counts) acc(e_b, (real)4 * eps * (sr6 * sr6 - sr6) + eps);
          }
          bx = fr * dx;
          by = fr * dy;
          bz = fr * dz;
          fx = fma_(fr, dx, fx);
          fy = fma_(fr, dy, fy);
          fz = fma_(fr, dz, fz);
          if (ENERGY && counts) acc(vir, fr * d2);
        }
      };
      if constexpr (ORDERED) {  // every atom its own bonds, in bond order
        const unsigned bw = own ? s.bond_word[gg0] : 0u;
#pragma unroll
        for (int q = 0; q < kMaxBonds; ++q) {
          if (q >= s.bond_max) break;
          const int e = (bw >> (4 * q)) & 15;
          const auto oo = atom_off(e & 3);
          real bx, by, bz;
          if (q < (int)(bw >> 28)) fene(oo, e & 8, bx, by, bz);
        }
      } else {
#pragma unroll
        for (int q = 0; q < kMaxBonds; ++q) {
          if (q >= s.bond_rounds) break;
          const int e = (send >> (4 * q)) & 15;
          const auto oo = atom_off(e & 3);
          real bx = 0, by = 0, bz = 0;
          if (e & 8) fene(oo, true, bx, by, bz);
          give(q, bx, by, bz);
        }
      }
    }
  }
  if (own) {
    // thermodynamic force on hybrid-layer molecules (region decided at mapping time), and
    // energy interpolation's drift force -(V_AT_a - V_CG_a - g(l_a)) l'(d) along grad d
    if (s.tf_n > 0 || hs) {
      real dxc;
      bool hy;
      if (P::fp64) {
        const double dd = b.dxc64[cur][a], ad = fabs(dd);
        dxc = (real)dd;
        hy = ad >= B.d_at && ad < B.d_at + B.d_hy && !s.lam_uniform_on;
      } else {
        const float2 mf = b.molf[cur][a];
        dxc = (real)mf.x;
        hy = mf.y != 0.f;
      }
      if (hy) {
        const real d = dxc < (real)0 ? -dxc : dxc;
        real F = 0;
        if (s.tf_n > 0) {
          const real u = d * par<real>(s.tf_inv_dx, s.f.tf_inv_dx);
          const int k = (int)u;
          if (k + 1 < s.tf_n) {
            const real tt = u - (real)k;
            F = Q::tf(b, B.tf0 + k) * ((real)1 - tt) + Q::tf(b, B.tf0 + k + 1) * tt;
          } else if (k + 1 == s.tf_n && u == (real)k) {
            F = Q::tf(b, B.tf0 + k);
          }
          F *= sw;
        }
        if (hs) {
          real gl = 0;
          if (s.fec_n > 0) {  // free-energy correction dDF/dl at l_a
            const real ul = wa * par<real>(s.fec_scale, s.f.fec_scale);
            const int kl = (int)ul;
            if (kl + 1 < s.fec_n) {
              const real tl = ul - (real)kl;
              gl = Q::fec(b, kl) * ((real)1 - tl) + Q::fec(b, kl + 1) * tl;
            } else {
              gl = Q::fec(b, s.fec_n - 1);
            }
          }
          // l'(d) = -(pi/(2 d_hy)) sin(pi (d - d_at)/d_hy)
          const real c = par<real>(B.pi_half_over_dhy, B.pi_half_over_dhy_f);
          const real sn = Q::sin_((real)2 * c * (d - par<real>(B.d_at, B.d_at_f)));
          F += (dv - sw * gl) * c * sn;
        }
        if (s.n_centers > 0) {
          // along the direction from the nearest centre
          const int kc = b.kcen[cur][a];
          real ux, uy, uz;
          if (P::fp64) {
            const double4_32a C = b.cen64[kc];
            const auto& R64 = Ca;
            ux = (real)minimg_cmp(R64.x - C.x, B.L[0], B.halfL[0]);
            uy = (real)minimg_cmp(R64.y - C.y, B.L[1], B.halfL[1]);
            uz = (real)minimg_cmp(R64.z - C.z, B.L[2], B.halfL[2]);
          } else {
            const int4 C = b.cen32[kc];
            const auto& R32 = Ca;
            ux = (real)((float)(int)((unsigned)R32.x - (unsigned)C.x) * B.fx_scale[0]);
            uy = (real)((float)(int)((unsigned)R32.y - (unsigned)C.y) * B.fx_scale[1]);
            uz = (real)((float)(int)((unsigned)R32.z - (unsigned)C.z) * B.fx_scale[2]);
          }
          const real fd = frac_g * Q::div_(F, d);
          fx += fd * ux;
          fy += fd * uy;
          fz += fd * uz;
        } else {
          fx += frac_g * (dxc < (real)0 ? -F : F);
        }
      }
    }
  }

  if (MODE == MODE_FORCES) {
    if (own) {
      real* fo = (real*)b.f;
      fo[i] = fx;
      fo[N + i] = fy;
      fo[2 * N + i] = fz;
    }
  } else {
    double x[3] = {0.0, 0.0, 0.0};
    if (own) {
      // Langevin force with the half-step velocity, noise keyed by (seed, time level n)
      const unsigned ia = (unsigned)(i - B.mol0 * NA);  // atom index within its replica
      unsigned c[4] = {ia, (unsigned)step, (unsigned)((unsigned long long)step >> 32), (unsigned)(2 * B.replica)};
      philox4x32_10(c, s.seed_lo, s.seed_hi);
      const double vx = vo[0], vy = vo[1], vz = vo[2];
      if (P::fp64) {
        unsigned lo[4] = {ia, (unsigned)step, (unsigned)((unsigned long long)step >> 32),
                          (unsigned)(2 * B.replica + 1)};
        philox4x32_10(lo, s.seed_lo, s.seed_hi);
        const double k53 = 1.0 / 9007199254740992.0, amp = s.amp[g], gm = s.gm[g];
        const double u0 = (double)(((unsigned long long)c[0] << 21) | (lo[0] >> 11)) * k53;
        const double u1 = (double)(((unsigned long long)c[1] << 21) | (lo[1] >> 11)) * k53;
        const double u2 = (double)(((unsigned long long)c[2] << 21) | (lo[2] >> 11)) * k53;
        fx += -gm * vx + amp * (u0 - 0.5);
        fy += -gm * vy + amp * (u1 - 0.5);
        fz += -gm * vz + amp * (u2 - 0.5);
      } else {
        const float k24 = 1.0f / 16777216.0f, af = s.ampf[g], gm = s.gmf[g];
        fx += -gm * d2f_bits(vx) + af * ((float)(c[0] >> 8) * k24 - 0.5f);
        fy += -gm * d2f_bits(vy) + af * ((float)(c[1] >> 8) * k24 - 0.5f);
        fz += -gm * d2f_bits(vz) + af * ((float)(c[2] >> 8) * k24 - 0.5f);
      }
      if (!(isfinite(fx) && isfinite(fy) && isfinite(fz))) set_error(b.ctrl, ADRESS_ERR_NONFINITE, i);
      const double h = s.hdt_m[g];
      const double fdx = P::fp64 ? (double)fx : f2d_bits((float)fx);
      const double fdy = P::fp64 ? (double)fy : f2d_bits((float)fy);
      const double fdz = P::fp64 ? (double)fz : f2d_bits((float)fz);
      if (MODE == MODE_LAST) {
        b.v[i] = fma(h, fdx, vx);
        b.v[N + i] = fma(h, fdy, vy);
        b.v[2 * N + i] = fma(h, fdz, vz);
        real* fo = (real*)b.f;
        fo[i] = fx;
        fo[N + i] = fy;
        fo[2 * N + i] = fz;
      } else {
        // second half kick of this step and first half kick of the next in one FMA,
        // then the drift; the force stays in registers
        const double h2 = s.dt_m[g];
        const double nvx = fma(h2, fdx, vx), nvy = fma(h2, fdy, vy), nvz = fma(h2, fdz, vz);
        double y0 = fma(s.dt, nvx, xo[0]), y1 = fma(s.dt, nvy, xo[1]), y2 = fma(s.dt, nvz, xo[2]);
        y0 = wrap_bits(y0, B.L[0], B.Lbits[0]);
        y1 = wrap_bits(y1, B.L[1], B.Lbits[1]);
        y2 = wrap_bits(y2, B.L[2], B.Lbits[2]);
        b.v[i] = nvx;
        b.v[N + i] = nvy;
        b.v[2 * N + i] = nvz;
        b.x[i] = y0;
        b.x[N + i] = y1;
        b.x[2 * N + i] = y2;
        x[0] = y0;
        x[1] = y1;
        x[2] = y2;
      }
    }
    if (MODE == MODE_FUSED) {
      // the next step's mapping, into the other buffer half (lanes without an atom take atom 0)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double x0 = P::fp64 ? shfl_d(gmask, x[d], base) : shfl_d(gmask, x[d], base);
        if (!own) x[d] = x0;
      }
      const int nxt = cur ^ 1;
      float d2 = 0.f;
      if (P::fp64) map_group64<NA, SAMPLE>(s, B, b, nxt, a, g, gmask, base, live, x, ref, sample, ext2, d2);
      else map_group32<NA, SAMPLE>(s, B, b, nxt, a, g, gmask, base, live, x, ref, sample, ext2, d2);
      disp2 = fmaxf(disp2, d2);
    }
  }

  if (ENERGY) {  // one record per block
    __shared__ double part[kMaxForceBlock / 32][4];
    const double sums[4] = {warp_sum(e_at), warp_sum(e_cg),
                            warp_sum(e_b) - 0.5 * (double)par<real>(s.fene_k, s.f.fene_k) * (double)par<real>(s.fene_r02, s.f.fene_r02) *
                                                warp_sum(e_log),
                            warp_sum(vir)};
    if (lane < 4) part[threadIdx.x >> 5][lane] = lane == 0 ? sums[0] : lane == 1 ? sums[1] : lane == 2 ? sums[2] : sums[3];
    __syncthreads();
    if (threadIdx.x < 4) {
      double v = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += part[w][threadIdx.x];
      b.part[(size_t)blockIdx.x * 4 + threadIdx.x] = v;
    }
  }
}

template <class P, int NA, int MODE, bool ENERGY, bool MULTI, int MODEL, bool HS, int FORM = FORM_ATOM>
__global__ void __launch_bounds__(kMaxForceBlock, step_min_blocks<P, MODEL, MULTI, HS>()) k_step(const __grid_constant__ Sys s, Bufs b) {
  const Ctrl* c = b.ctrl;
  float ext2 = 0.f, disp2 = 0.f;
  constexpr bool LPN = FORM == FORM_NEIGHBOUR || FORM == FORM_NEIGHBOUR_8_4;
  const Lanes ln = lanes_of<FORM, P, MODEL>(s.step_lanes);
  // blocks past the last item (the host does not know the number of high-resolution items)
  if (!ENERGY && ln.h != ln.c && blockIdx.x * blockDim.x >= (unsigned)((c->n_hr << ln.h) + ((s.M - c->n_hr) << ln.c))) return;
  step_tile<P, NA, MODE, ENERGY, MULTI, MODEL, HS, LPN, false, FORM == FORM_ORDERED>(s, b, ln, blockIdx.x * blockDim.x + threadIdx.x, c->parity, c->step,
                                                        c->ext_now, 0, ext2, disp2);
  if (MODE == MODE_FUSED) publish_extent(b, 0, ext2, disp2);
}

// ---------------- k_run ------------------------------------------------------------------

// Resident blocks per SM of the run kernel: its systems are bound by latency, so registers
// (128 a thread) come before warps.
template <class P>
constexpr int run_min_blocks() {
  return P::fp64 ? 3 : 4;
}

// nsteps fused steps after mapping `done` in one cooperative launch (a density sample after every
// sample_every-th mapping): every block takes its tiles of the step, a
// grid barrier ends the mapping, every block takes the rebuild decision itself and the grid
// rebuilds the lists when needed.  For small systems (run_kernel_pays).
template <class P, int NA, bool MULTI, int MODEL, bool HS>
__global__ void __launch_bounds__(kMaxForceBlock, run_min_blocks<P>()) k_run(const __grid_constant__ Sys s, const __grid_constant__ Bufs b, int done, int nsteps,
                                                                              int sample_every) {
  Ctrl* c = b.ctrl;
  if (__syncthreads_or(threadIdx.x == 0 && __ldcg(&c->dead) != 0)) return;  // a grid barrier gave up earlier
  int cur = c->parity, set = 0, dirty = 0, rebuilt = 0;
  long long step = c->step;
  float ext_now = c->ext_now;
  constexpr bool LPN = !P::fp64;
  const Lanes ln = lanes_of<LPN ? FORM_NEIGHBOUR : FORM_ATOM, P, MODEL>(s.run_lanes);
  GridBarrier bar(b, &c->bar[1]);
  for (int k = 0; k < nsteps; ++k) {
    float ext2 = 0.f, disp2 = 0.f;
    const int sample = sample_every > 0 && (done + k + 1) % sample_every == 0;
    const int n_hr = c->n_hr;
    const int ntiles = ((n_hr << ln.h) + ((s.M - n_hr) << ln.c) + blockDim.x - 1) / blockDim.x;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
      step_tile<P, NA, MODE_FUSED, false, MULTI, MODEL, HS, LPN, true, false>(s, b, ln, tile * blockDim.x + threadIdx.x, cur, step, ext_now,
                                                                sample, ext2, disp2);
    publish_extent(b, set, ext2, disp2);
    if (!bar.sync()) return;
    const Decision d = decide_rebuild(s, c, set, 0);
    if (blockIdx.x == 0 && threadIdx.x < 32) {
      // the set of the previous step: every block has read it, and the step after the next
      // publishes to it
      c->ext_slot[(set + 2) % 3][0][threadIdx.x] = 0u;
      c->ext_slot[(set + 2) % 3][1][threadIdx.x] = 0u;
      if (threadIdx.x == 0 && sample) *b.nsamples += 1;
      if (threadIdx.x == 0 && d.too_wide) set_error(c, ADRESS_ERR_EXTENT, (int)(d.ext * 1000));
    }
    cur ^= 1;
    ++step;
    dirty = set;
    set = (set + 1) % 3;
    ext_now = d.ext;
    if (d.rebuild) {
      ++rebuilt;
      if (!rebuild_lists<kMaxForceBlock / 32>(s, b, cur, bar)) return;
      if (!bar.sync()) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) c->force_rebuild = 0;
    }
  }
  if (threadIdx.x < 32 && last_to_arrive(c)) {
    c->ext_slot[dirty][0][threadIdx.x] = 0u;
    c->ext_slot[dirty][1][threadIdx.x] = 0u;
    if (threadIdx.x == 0) {
      c->parity = cur;
      c->step = step;
      c->ext_now = ext_now;
      c->rebuilds += rebuilt;
    }
  }
}

// ---------------- launchers ----------------------------------------------------------

template <class P, int NA, int MODEL, bool HS, int FORM, bool MULTI>
static void launch_step_form(const Sys& s, const Bufs& b, int mode, int energy, cudaStream_t st) {
  const int blocks = ceil_div((long long)s.M * step_lanes(s), s.force_block), threads = s.force_block;
  switch (mode) {
    case MODE_FORCES:
      if (energy) k_step<P, NA, MODE_FORCES, true, MULTI, MODEL, HS, FORM><<<blocks, threads, 0, st>>>(s, b);
      else k_step<P, NA, MODE_FORCES, false, MULTI, MODEL, HS, FORM><<<blocks, threads, 0, st>>>(s, b);
      break;
    case MODE_LAST: k_step<P, NA, MODE_LAST, false, MULTI, MODEL, HS, FORM><<<blocks, threads, 0, st>>>(s, b); break;
    default: k_step<P, NA, MODE_FUSED, false, MULTI, MODEL, HS, FORM><<<blocks, threads, 0, st>>>(s, b); break;
  }
}

template <class P, int NA, int MODEL, bool HS, int FORM>
static void launch_step_boxes(const Sys& s, const Bufs& b, int mode, int energy, cudaStream_t st) {
  if (s.nbox > 1) launch_step_form<P, NA, MODEL, HS, FORM, true>(s, b, mode, energy, st);
  else launch_step_form<P, NA, MODEL, HS, FORM, false>(s, b, mode, energy, st);
}

template <class P, int NA, int MODEL, bool HS>
static void launch_step_na(const Sys& s, const Bufs& b, int mode, int energy, cudaStream_t st) {
  if constexpr (!P::fp64 && MODEL == 1) {
    // eight and four lanes as constants where the host chose them (4% at 64,000 molecules)
    if (s.step_lanes.h == 3 && s.step_lanes.c == 2) launch_step_boxes<P, NA, MODEL, HS, FORM_NEIGHBOUR_8_4>(s, b, mode, energy, st);
    else launch_step_boxes<P, NA, MODEL, HS, FORM_NEIGHBOUR>(s, b, mode, energy, st);
  } else {
    if constexpr (!P::fp64 && !HS) {  // (energy interpolation has no learned force)
      if (s.cg_mode) return launch_step_boxes<P, NA, MODEL, HS, FORM_ORDERED>(s, b, mode, energy, st);
    }
    launch_step_boxes<P, NA, MODEL, HS, FORM_ATOM>(s, b, mode, energy, st);
  }
}

// As many blocks as fit on the device at once, at most one per tile.  Their size is fixed: at a force
// kernel's 32 threads the four blocks an SM are four warps (us a step with 32 / 64 / 128 threads: 4000
// molecules 17.4 / 13.6 / 10.3, 20,000 32.8 / 21.6 / 18.0, where launches at 32 took 28.1).
template <class P, int NA, int MODEL, bool HS>
static cudaError_t launch_run_na(const Sys& s, const Bufs& b, int done, int nsteps, int sample_every, cudaStream_t st) {
  const int tiles = ceil_div((long long)s.M << (P::fp64 ? 2 : s.run_lanes.h), kMaxForceBlock);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(std::min(tiles, s.n_sm * run_min_blocks<P>()));
  cfg.blockDim = dim3(kMaxForceBlock);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (s.nbox > 1) return cudaLaunchKernelEx(&cfg, k_run<P, NA, true, MODEL, HS>, s, b, done, nsteps, sample_every);
  return cudaLaunchKernelEx(&cfg, k_run<P, NA, false, MODEL, HS>, s, b, done, nsteps, sample_every);
}

}  // namespace adress
