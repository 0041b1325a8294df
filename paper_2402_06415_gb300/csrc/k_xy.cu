// Checkerboard Metropolis sweep of the 2D XY model: the paper's own Monte Carlo
// workload (arXiv 2402.06415, Eq. 1; Supplementary "Detail of the MC
// calculation for the XY model").  Each site holds the unit vector
// u = (cos theta, sin theta).  Per site: theta' = 2 pi U1, p = U2 (two 24-bit
// uniforms from one half of a Philox block), dE = -(u' - u) . h with h the sum
// of the four neighbour vectors (Eq. S1, sign corrected, in local-field form),
// accept iff dE <= 0 or p < exp(-beta dE).  Sublattice (x + y) even, then odd.
//
// cos, sin and exp are evaluated by this file's own routines: Cody-Waite
// reduction by pi/2 (two-part constant) or ln 2, then Taylor polynomials in
// Horner form with explicit fused multiply-adds.  All other arithmetic is
// single IEEE operations in a fixed order, so every decision is reproducible
// bit for bit by any implementation of the same recipe.
//
// Layout: two colour planes of [L][L/2] vectors (T2 = float2 or double2);
// site (x, y) of colour c = (x + y) & 1 is element y (L/2) + (x >> 1) of plane c.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <new>
#include <vector>

#include "internal.h"
#include "ising.h"
#include "ising_device.cuh"

namespace ising {
namespace {

constexpr uint32_t kTagXYInit = 8, kTagXYMet = 9;

template <typename T> struct Vec;
template <> struct Vec<float> { using type = float2; };
template <> struct Vec<double> { using type = double2; };

// ---- own elementary functions (double) ----
__device__ __forceinline__ void sincos_small(double r, double& s, double& c) {
  const double z = __dmul_rn(r, r);
  double pc = 1.0 / 20922789888000.0;
  pc = fma(pc, z, -1.0 / 87178291200.0);
  pc = fma(pc, z, 1.0 / 479001600.0);
  pc = fma(pc, z, -1.0 / 3628800.0);
  pc = fma(pc, z, 1.0 / 40320.0);
  pc = fma(pc, z, -1.0 / 720.0);
  pc = fma(pc, z, 1.0 / 24.0);
  pc = fma(pc, z, -0.5);
  pc = fma(pc, z, 1.0);
  double ps = 1.0 / 355687428096000.0;
  ps = fma(ps, z, -1.0 / 1307674368000.0);
  ps = fma(ps, z, 1.0 / 6227020800.0);
  ps = fma(ps, z, -1.0 / 39916800.0);
  ps = fma(ps, z, 1.0 / 362880.0);
  ps = fma(ps, z, -1.0 / 5040.0);
  ps = fma(ps, z, 1.0 / 120.0);
  ps = fma(ps, z, -1.0 / 6.0);
  ps = fma(ps, z, 1.0);
  c = pc;
  s = __dmul_rn(ps, r);
}

__device__ __forceinline__ double own_exp(double x) {
  if (x < -700.0) return 0.0;
  const double k = rint(__dmul_rn(x, 1.4426950408889634));
  double r = fma(-k, 0.6931471805599453, x);
  r = fma(-k, 2.3190468138462996e-17, r);
  double p = 1.0 / 6227020800.0;
  p = fma(p, r, 1.0 / 479001600.0);
  p = fma(p, r, 1.0 / 39916800.0);
  p = fma(p, r, 1.0 / 3628800.0);
  p = fma(p, r, 1.0 / 362880.0);
  p = fma(p, r, 1.0 / 40320.0);
  p = fma(p, r, 1.0 / 5040.0);
  p = fma(p, r, 1.0 / 720.0);
  p = fma(p, r, 1.0 / 120.0);
  p = fma(p, r, 1.0 / 24.0);
  p = fma(p, r, 1.0 / 6.0);
  p = fma(p, r, 0.5);
  p = fma(p, r, 1.0);
  p = fma(p, r, 1.0);
  // p 2^k with 2^k built from its exponent field (k in [-1010, 0], a normal
  // number): a multiplication by a power of two is exact, or correctly rounded
  // when the product is subnormal, i.e. the same result as ldexp
  return p * __longlong_as_double((long long)((int)k + 1023) << 52);
}

// ---- own elementary functions (float) ----
__device__ __forceinline__ void sincos_small(float r, float& s, float& c) {
  const float z = __fmul_rn(r, r);
  float pc = 1.0f / 40320.0f;
  pc = fmaf(pc, z, -1.0f / 720.0f);
  pc = fmaf(pc, z, 1.0f / 24.0f);
  pc = fmaf(pc, z, -0.5f);
  pc = fmaf(pc, z, 1.0f);
  float ps = 1.0f / 362880.0f;
  ps = fmaf(ps, z, -1.0f / 5040.0f);
  ps = fmaf(ps, z, 1.0f / 120.0f);
  ps = fmaf(ps, z, -1.0f / 6.0f);
  ps = fmaf(ps, z, 1.0f);
  c = pc;
  s = __fmul_rn(ps, r);
}

__device__ __forceinline__ void own_sincos(float x, float& s, float& c) {
  const float k = rintf(__fmul_rn(x, 0.636619747f));
  float r = fmaf(-k, 1.57079637f, x);
  r = fmaf(-k, -4.37113883e-08f, r);
  float ss, cc;
  sincos_small(r, ss, cc);
  const int q = ((int)k) & 3;
  s = q == 0 ? ss : (q == 1 ? cc : (q == 2 ? -ss : -cc));
  c = q == 0 ? cc : (q == 1 ? -ss : (q == 2 ? -cc : ss));
}

__device__ __forceinline__ float own_exp(float x) {
  if (x < -87.0f) return 0.0f;
  const float k = rintf(__fmul_rn(x, 1.44269502f));
  float r = fmaf(-k, 0.693147182f, x);
  r = fmaf(-k, -1.90465421e-09f, r);
  float p = 1.0f / 40320.0f;
  p = fmaf(p, r, 1.0f / 5040.0f);
  p = fmaf(p, r, 1.0f / 720.0f);
  p = fmaf(p, r, 1.0f / 120.0f);
  p = fmaf(p, r, 1.0f / 24.0f);
  p = fmaf(p, r, 1.0f / 6.0f);
  p = fmaf(p, r, 0.5f);
  p = fmaf(p, r, 1.0f);
  p = fmaf(p, r, 1.0f);
  // p 2^k, 2^k from its exponent field (k in [-126, 0]): same result as ldexpf
  return p * __int_as_float(((int)k + 127) << 23);
}

template <typename T> __device__ __forceinline__ T mul_rn(T a, T b);
template <> __device__ __forceinline__ double mul_rn<double>(double a, double b) { return __dmul_rn(a, b); }
template <> __device__ __forceinline__ float mul_rn<float>(float a, float b) { return __fmul_rn(a, b); }
template <typename T> __device__ __forceinline__ T add_rn(T a, T b);
template <> __device__ __forceinline__ double add_rn<double>(double a, double b) { return __dadd_rn(a, b); }
template <> __device__ __forceinline__ float add_rn<float>(float a, float b) { return __fadd_rn(a, b); }
template <typename T> __device__ __forceinline__ T sub_rn(T a, T b);
template <> __device__ __forceinline__ double sub_rn<double>(double a, double b) { return __dsub_rn(a, b); }
template <> __device__ __forceinline__ float sub_rn<float>(float a, float b) { return __fsub_rn(a, b); }

// sin and cos of the angle of a random word, theta = 2 pi (m 2^-24) with m its top 24
// bits: theta rounded, k = rint(theta 2 / pi), r = theta - k pi / 2 (two-part
// constant), the polynomials at r, and the quadrant k & 3.  In double every
// operation holds this part's FP64 unit for 64 cycles per warp and sub-partition,
// so five of those steps are done otherwise with the same values: the conversion
// is integer work, the exact scaling by 2^-24 sits in the constant, and k is the
// integer (m + 2^21) >> 22 unless m / 2^22 is exactly a half integer (m / 2^22
// differs from theta 2 / pi by less than 2e-15, and otherwise lies at least 2^-22
// from a half integer).
__device__ __forceinline__ void word_sincos(uint32_t w, float& s, float& c) {
  own_sincos(__fmul_rn(6.28318548f, __fmul_rn((float)(w >> 8), 1.0f / 16777216.0f)), s, c);
}
__device__ __forceinline__ void word_sincos(uint32_t w, double& s, double& c) {
  const uint32_t m = w >> 8;
  // m and k as doubles from their (exact) floats; no branches: the lanes differ
  const uint32_t mf = __float_as_uint((float)m);
  const double md = __hiloint2double(m ? (int)((mf >> 3) + 0x38000000u) : 0, (int)(mf << 29));
  const double x = __dmul_rn(6.283185307179586 / 16777216.0, md);
  uint32_t k = (m + (1u << 21)) >> 22;
  if ((m & 0x3fffffu) == 0x200000u) k = (uint32_t)rint(__dmul_rn(x, 0.6366197723675814));
  const uint32_t kf = __float_as_uint((float)k);
  const double kd = __hiloint2double(k ? (int)((kf >> 3) + 0xb8000000u) : (int)0x80000000u, 0);  // -k
  double r = fma(kd, 1.5707963267948966, x);
  r = fma(kd, 6.123233995736766e-17, r);
  double ss, cc;
  sincos_small(r, ss, cc);
  // quadrant k & 3: swap sin and cos, then flip their sign bits
  const bool swap = (k & 1u) != 0;
  const int s_hi = __double2hiint(swap ? cc : ss) ^ (int)((k & 2u) << 30);
  const int c_hi = __double2hiint(swap ? ss : cc) ^ (int)(((k + 1u) & 2u) << 30);
  s = __hiloint2double(s_hi, __double2loint(swap ? cc : ss));
  c = __hiloint2double(c_hi, __double2loint(swap ? ss : cc));
}

template <typename T>
__global__ void k_xy_init(typename Vec<T>::type* __restrict__ u, int L, RngParams rng) {
  const long long N = (long long)L * L;
  const int half = L / 2;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    const int y = (int)(n / L), x = (int)(n - (n / L) * L);
    const uint4 r = philox10_rk(make_uint4((uint32_t)(n >> 2), 0u, rng.replica, kTagXYInit << 16),
                                rng.rk0, rng.rk1);
    const uint32_t w = (n & 3) == 0 ? r.x : ((n & 3) == 1 ? r.y : ((n & 3) == 2 ? r.z : r.w));
    T s, c;
    word_sincos(w, s, c);
    const int col = (x + y) & 1;
    typename Vec<T>::type v;
    v.x = c;
    v.y = s;
    u[(size_t)col * L * half + (size_t)y * half + (x >> 1)] = v;
  }
}

// The acceptance decision p < own_exp(x) (x = -beta dE < 0), decided first from
// the hardware exponential __expf: its documented error on this range is at most
// 2 + 1.173 |x| ulp (about 1e-5 relative for x >= -80), the rounding of x to
// float adds at most |x| 2^-24 relative, so when p lies outside
// e (1 -+ 1e-4) the exact own_exp gives the same answer and is skipped; inside
// that band (rare), or for x < -80 with p = 0, own_exp decides.  For x < -80,
// exp(x) < 2^-115 < p whenever p > 0 (p is a multiple of 2^-24).
__device__ __forceinline__ bool accept_exp(float p, float x) {
  if (x >= -80.f) {
    const float e = __expf(x);
    if (p < e * 0.9999f) return true;
    if (p > e * 1.0001f) return false;
  } else if (p > 0.f) {
    return false;
  }
  return p < own_exp(x);
}

// The trial's decision: dE <= 0 or p < exp(-beta dE), p = the top 24 bits of w2.
__device__ __forceinline__ bool accept_move(uint32_t w2, float dE, float beta, float) {
  return dE <= 0.f || accept_exp((float)(w2 >> 8) * (1.0f / 16777216.0f), mul_rn<float>(-beta, dE));
}
// beta for the estimate below; NaN (every trial decided exactly) where dE's cut to
// float range or beta's overflow would spoil it.
__host__ __device__ __forceinline__ float beta_estimate(double beta) {
  return beta <= 1e30 ? (float)beta : (float)(0.0 * INFINITY);
}
// In double, the sign and the estimate that decides all but a band of 1e-4 need
// no FP64 operation: -beta dE is formed in float (beta_f = beta) from dE's bits cut to 24
// (relative error below 2^-22, so below 2e-5 in exp for -beta dE >= -80, next to
// the 1e-5 of __expf); the band, and p = 0 below -80, are decided exactly.
__device__ __forceinline__ bool accept_move(uint32_t w2, double dE, double beta, float beta_f) {
  const int hi = __double2hiint(dE), lo = __double2loint(dE);
  const int mag = hi & 0x7fffffff;
  if (mag <= 0x7ff00000 && (hi < 0 || (mag | lo) == 0)) return true;
  const int ex = (mag >> 20) - 1023 + 127;
  const float d = ex <= 0 ? 0.f : ex >= 255 ? __int_as_float(0x7f800000)
                                            : __uint_as_float(((uint32_t)ex << 23) | ((uint32_t)(hi & 0xfffff) << 3) |
                                                              ((uint32_t)lo >> 29));
  const float x = -beta_f * d, p = (float)(w2 >> 8) * (1.0f / 16777216.0f);
  if (x >= -80.f) {
    const float e = __expf(x);
    if (p < e * 0.9999f) return true;
    if (p > e * 1.0001f) return false;
  } else if (x < -80.f && p > 0.f) {
    return false;
  }
  return dE <= 0.0 || (double)p < own_exp(__dmul_rn(-beta, dE));
}

// Loads and stores of the state: plain in the one-launch-per-half-sweep
// kernels; through L2 only (no L1) in the persistent kernel, whose CTAs read
// what other SMs wrote after a grid barrier.
template <bool CG, typename V>
__device__ __forceinline__ V ld_state(const V* p) {
  if (CG) return __ldcg(p);
  return *p;
}
template <bool CG, typename V>
__device__ __forceinline__ void st_state(V* p, V v) {
  if (CG) __stcg(p, v);
  else *p = v;
}

// Metropolis trials of the two colour-compact sites k = 2b, 2b + 1 of colour
// c (one Philox block); returns how many were accepted.
template <typename T, bool CG>
__device__ __forceinline__ unsigned int xy_pair(typename Vec<T>::type* __restrict__ own,
                                                const typename Vec<T>::type* __restrict__ oth, int L,
                                                uint32_t nk, uint32_t b, int c, uint32_t t, T beta,
                                                const RngParams& rng, const FastDiv& fh) {
  using V = typename Vec<T>::type;
  const int half = L / 2;
  unsigned int acc = 0;
  const uint4 r = philox10_rk(make_uint4(b, t, rng.replica, (kTagXYMet << 16) | ((uint32_t)c << 8)),
                              rng.rk0, rng.rk1);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t k = 2 * b + h;
    if (k >= nk) break;
    const int y = (int)fdiv(k, fh), j = (int)(k - (uint32_t)y * (uint32_t)half);
    const int o = (y + c) & 1;  // x = 2 j + o
    const int jr = o == 0 ? j : (j + 1 == half ? 0 : j + 1);   // x + 1
    const int jl = o == 0 ? (j == 0 ? half - 1 : j - 1) : j;   // x - 1
    const int yd = y + 1 == L ? 0 : y + 1, yu = y == 0 ? L - 1 : y - 1;
    const V a = ld_state<CG>(oth + (size_t)y * half + jr);
    const V bl = ld_state<CG>(oth + (size_t)y * half + jl);
    const V d = ld_state<CG>(oth + (size_t)yd * half + j);
    const V e = ld_state<CG>(oth + (size_t)yu * half + j);
    T hx = add_rn<T>(a.x, bl.x);
    hx = add_rn<T>(hx, d.x);
    hx = add_rn<T>(hx, e.x);
    T hy = add_rn<T>(a.y, bl.y);
    hy = add_rn<T>(hy, d.y);
    hy = add_rn<T>(hy, e.y);
    const uint32_t w1 = h == 0 ? r.x : r.z, w2 = h == 0 ? r.y : r.w;
    T sn, cs;
    word_sincos(w1, sn, cs);
    V me = ld_state<CG>(own + k);
    const T dE = -fma(sub_rn<T>(cs, me.x), hx, mul_rn<T>(sub_rn<T>(sn, me.y), hy));
    if (accept_move(w2, dE, beta, beta_estimate((double)beta))) {
      me.x = cs;
      me.y = sn;
      st_state<CG>(own + k, me);
      ++acc;
    }
  }
  return acc;
}

__device__ __forceinline__ void add_accepted(unsigned long long* accepted, unsigned int acc) {
  if (!accepted) return;
  unsigned int s = acc;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(accepted, (unsigned long long)s);
}

// One half sweep of colour c: thread = one Philox block = colour-compact sites
// k = 2b and 2b + 1.
template <typename T>
__global__ void __launch_bounds__(256) k_xy_half(typename Vec<T>::type* __restrict__ u, int L,
                                                 int c, uint32_t t, T beta, RngParams rng, FastDiv fh,
                                                 unsigned long long* __restrict__ accepted) {
  const int half = L / 2;
  const uint32_t nk = (uint32_t)L * (uint32_t)half;  // < 2^29 for L <= 32768
  typename Vec<T>::type* own = u + (size_t)c * L * half;
  const typename Vec<T>::type* oth = u + (size_t)(1 - c) * L * half;
  unsigned int acc = 0;
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; 2 * b < nk; b += gridDim.x * blockDim.x)
    acc += xy_pair<T, false>(own, oth, L, nk, b, c, t, beta, rng, fh);
  add_accepted(accepted, acc);
}

// E = -sum over colour-0 sites of u . (sum of its four neighbours) (every bond
// once), M = sum u; per-thread partials over a grid-stride range, accumulated
// in double and added to out3 by one atomic per warp.
template <typename T, bool CG>
__device__ __forceinline__ void xy_measure_part(const typename Vec<T>::type* __restrict__ u, int L,
                                                double* __restrict__ out3, const FastDiv& fh) {
  using V = typename Vec<T>::type;
  const int half = L / 2;
  const uint32_t nk = (uint32_t)L * (uint32_t)half;
  const V* p0 = u;
  const V* p1 = u + (size_t)L * half;
  double e = 0, mx = 0, my = 0;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < nk; k += gridDim.x * blockDim.x) {
    const int y = (int)fdiv(k, fh), j = (int)(k - (uint32_t)y * (uint32_t)half);
    const int o = y & 1;
    const int jr = o == 0 ? j : (j + 1 == half ? 0 : j + 1);
    const int jl = o == 0 ? (j == 0 ? half - 1 : j - 1) : j;
    const int yd = y + 1 == L ? 0 : y + 1, yu = y == 0 ? L - 1 : y - 1;
    const V s = ld_state<CG>(p0 + k);
    const V a = ld_state<CG>(p1 + (size_t)y * half + jr), b = ld_state<CG>(p1 + (size_t)y * half + jl);
    const V d = ld_state<CG>(p1 + (size_t)yd * half + j), f = ld_state<CG>(p1 + (size_t)yu * half + j);
    const double hx = (double)a.x + b.x + d.x + f.x, hy = (double)a.y + b.y + d.y + f.y;
    e -= (double)s.x * hx + (double)s.y * hy;
    const V s1 = ld_state<CG>(p1 + k);
    mx += (double)s.x + (double)s1.x;
    my += (double)s.y + (double)s1.y;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    e += __shfl_xor_sync(0xffffffffu, e, off);
    mx += __shfl_xor_sync(0xffffffffu, mx, off);
    my += __shfl_xor_sync(0xffffffffu, my, off);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&out3[0], e);
    atomicAdd(&out3[1], mx);
    atomicAdd(&out3[2], my);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_xy_measure(const typename Vec<T>::type* __restrict__ u,
                                                    int L, double* __restrict__ out3, FastDiv fh) {
  xy_measure_part<T, false>(u, L, out3, fh);
}

// Persistent form for small lattices: n sweeps (from sweep t0) in one launch,
// a barrier after each half sweep and each measurement.  PM = kOneCTA: one
// CTA, __syncthreads(), state through L1; kCluster: one thread-block cluster,
// the hardware cluster barrier (release / acquire), state through L2;
// kGrid: a cooperative grid (every CTA co-resident), the bounded grid barrier,
// state through L2.  Records go to ring slots rec0, rec0 + 1, ...; each slot is
// zeroed by CTA 0 in the half sweep before it is filled.
enum PersistMode { kOneCTA = 0, kCluster = 1, kGrid = 2 };

template <int PM>
__device__ __forceinline__ bool persist_sync(GridCtl* ctl, long long limit) {
  if (PM == kGrid) return grid_sync_bounded(ctl, limit);
  if (PM == kCluster) cooperative_groups::this_cluster().sync();
  else __syncthreads();
  return true;
}

template <typename T, int PM>
__global__ void __launch_bounds__(PM == kGrid ? 256 : 1024) k_xy_persist(typename Vec<T>::type* __restrict__ u, int L,
                                                    T beta, RngParams rng, uint32_t t0, int n, int m,
                                                    double* __restrict__ rec, long long rec0,
                                                    long long rec_cap,
                                                    unsigned long long* __restrict__ accepted,
                                                    GridCtl* ctl, long long limit, FastDiv fh) {
  using V = typename Vec<T>::type;
  const int half = L / 2;
  const uint32_t nk = (uint32_t)L * (uint32_t)half;
  unsigned int acc = 0;
  long long ri = rec0;
  for (int s = 0; s < n; ++s) {
    const uint32_t t = t0 + (uint32_t)s;
    const bool meas = m > 0 && ((long long)t + 1) % m == 0;
    double* slot = rec + 3 * (ri % rec_cap);
    bool ok = true;
    for (int c = 0; c < 2 && ok; ++c) {
      V* own = u + (size_t)c * L * half;
      const V* oth = u + (size_t)(1 - c) * L * half;
      for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; 2 * b < nk; b += gridDim.x * blockDim.x)
        acc += xy_pair<T, PM != kOneCTA>(own, oth, L, nk, b, c, t, beta, rng, fh);
      if (meas && c == 1 && blockIdx.x == 0 && threadIdx.x == 0) slot[0] = slot[1] = slot[2] = 0.0;
      ok = persist_sync<PM>(ctl, limit);
    }
    if (ok && meas) {
      xy_measure_part<T, PM != kOneCTA>(u, L, slot, fh);
      ++ri;
      ok = persist_sync<PM>(ctl, limit);
    }
    if (!ok) break;
  }
  add_accepted(accepted, acc);
}

// Resident strips: many sweeps in one launch for lattices whose half sweep is
// too short for a launch or a grid barrier of its own.  G CTAs own row strips of
// full width, both colours in shared memory, with a halo of `gh` rows; gh half
// sweeps run with CTA barriers only (each invalidates one more halo row), then
// the strips hand their outer rows to their neighbours as (tag, word) pairs
// through L2.  G = 1 keeps the whole lattice in one CTA.  A thread updates the
// two sites of one Philox block (k = 2b, 2b + 1; their parity survives the wrap
// because L^2 / 2 is even).  AHEAD (at most one block per thread): the proposals
// of the next half sweep, which do not depend on spins, are drawn before the
// barrier or while the neighbours' rows are on their way; in FP64 their sines
// and cosines are most of the work of this part's slow FP64 pipe.
// E, Mx, My of a recorded sweep are summed (in double) in the colour-1 half
// sweep itself: every bond joins a colour-1 site to a colour-0 neighbour.
// Per sweep with a record each, before (a grid barrier or launch per half sweep
// and per measurement) and now: FP64 L = 32 17.1 -> 5.2 us, FP32 L = 512 (a record
// every 10 sweeps) 14.9 -> 5.6 us.  What bounds it: FP64, the 31 FP64 operations of a
// trial at 64 cycles per warp and sub-partition; FP32, the dependent chain of a
// half sweep, at L = 512 still (16 warps an SM, ALU pipe 28 %, FMA 20 %).
template <typename T>
struct XYStripArgs {
  typename Vec<T>::type* u;
  int L, G, gh;
  T beta;
  float beta_f;
  uint32_t t0;
  int n, m, to_rec;  // sweeps; record every m; sweeps until the first record (0: none)
  double* rec;
  long long rec0, rec_cap;
  unsigned long long* accepted;
  unsigned long long* xbuf;  // xy_strip_words(...) pairs, zeroed by the launcher (G > 1)
  int* status;
  long long limit;
  FastDiv fh;
};
constexpr int kXYStripThreads = 512;

template <typename T>
size_t xy_strip_words(int L, int G, int gh) {
  return G == 1 ? 0 : (size_t)G * (8 * (size_t)gh * (L / 2) * (sizeof(typename Vec<T>::type) / 4) + 1);
}
template <typename T>
size_t xy_strip_smem(int L, int G, int gh) {
  return 2 * (size_t)((L + G - 1) / G + (G == 1 ? 0 : 2 * gh)) * (L / 2) * sizeof(typename Vec<T>::type);
}

template <typename T, bool WHOLE, bool AHEAD>
__global__ void __launch_bounds__(kXYStripThreads) k_xy_strip(XYStripArgs<T> a, RngParams rng) {
  using V = typename Vec<T>::type;
  constexpr int VW = sizeof(V) / 4;
  extern __shared__ uint4 xy_smem[];
  const int L = a.L, half = L / 2, G = WHOLE ? 1 : a.G, H = WHOLE ? 0 : a.gh;
  const int b = blockIdx.x, tid = threadIdx.x, nth = blockDim.x;
  const int y0 = (int)((long long)b * L / G), R = (int)((long long)(b + 1) * L / G) - y0;
  const int rows = R + 2 * H, ns = rows * half, N2 = L * half;
  const int plane = ((L + G - 1) / G + 2 * H) * half;
  V* const S = reinterpret_cast<V*>(xy_smem);
  auto P = [&](int c) { return S + c * plane; };
  const int koff = (y0 - H) * half;  // local site i is site i + koff of its colour, modulo N2
  auto global_k = [&](int i) {
    int k = i + koff;
    if (!WHOLE) {
      k += k < 0 ? N2 : 0;
      k -= k >= N2 ? N2 : 0;
    }
    return k;
  };
  for (int i = tid; i < 2 * ns; i += nth) {
    const int c = i >= ns, k = i - c * ns;
    P(c)[k] = __ldcg(&a.u[(size_t)c * N2 + global_k(k)]);
  }
  __syncthreads();
  const int hw = H * half * VW;  // 32-bit words of H rows of one colour
  const size_t per_cta = 8 * (size_t)hw + 1;
  const int up = b == 0 ? G - 1 : b - 1, dn = b == G - 1 ? 0 : b + 1;
  unsigned long long* const mine = WHOLE ? nullptr : a.xbuf + b * per_cta;
  if (!WHOLE && tid == 0) send_word(mine + 8 * hw, 1u, 0u);  // "lattice read"
  // an item is one site (SPT = 1) or the two sites of a block (item j: local sites
  // 2 j - par, 2 j - par + 1)
  constexpr int SPT = (AHEAD || sizeof(T) == 8) ? 1 : 2;
  const int par = SPT == 2 ? koff & 1 : 0;
  // AHEAD: one item per thread, in rows 1 .. rows - 2 (the outermost halo rows are only read)
  const int item = tid + (WHOLE ? 0 : half), items_end = ns - (WHOLE ? 0 : half);
  auto in_rows = [&](int i, int lo) { return i >= lo * half && i < ns - lo * half; };

  struct Prop {
    T cs[SPT], sn[SPT];
    uint32_t w2[SPT];
  };
  auto propose = [&](int j, uint32_t t, int c, Prop& q) {
    const uint32_t k = (uint32_t)global_k(SPT * j - par);
    const uint4 r = philox10_rk(make_uint4(k >> 1, t, rng.replica, (kTagXYMet << 16) | ((uint32_t)c << 8)), rng.rk0,
                                rng.rk1);
#pragma unroll
    for (int h = 0; h < SPT; ++h) {
      const bool second = SPT == 2 ? h == 1 : (k & 1u) != 0;
      word_sincos(second ? r.z : r.x, q.sn[h], q.cs[h]);
      q.w2[h] = second ? r.w : r.y;
    }
  };
  unsigned int acc = 0;
  double e = 0, mx = 0, my = 0;
  // trials of item j in the rows [lo, rows - lo) of colour c
  auto update = [&](int j, int c, int lo, bool meas, const Prop& q) {
    V* const So = P(c);
    const V* const Sn = P(1 - c);
#pragma unroll
    for (int h = 0; h < SPT; ++h) {
      const int i = SPT * j - par + h;
      if (!in_rows(i, lo)) continue;
      const int r = (int)fdiv((uint32_t)i, a.fh), x = i - r * half, row = i - x;
      const int o = (y0 - H + r + c) & 1;
      const int ir = o == 0 ? i : row + (x + 1 == half ? 0 : x + 1);
      const int il = o == 0 ? row + (x == 0 ? half - 1 : x - 1) : i;
      int id = i + half, iu = i - half;
      if (WHOLE) {
        id -= id >= ns ? ns : 0;
        iu += iu < 0 ? ns : 0;
      }
      const V va = Sn[ir], vb = Sn[il], vd = Sn[id], ve = Sn[iu];
      T hx = add_rn<T>(va.x, vb.x);
      hx = add_rn<T>(hx, vd.x);
      hx = add_rn<T>(hx, ve.x);
      T hy = add_rn<T>(va.y, vb.y);
      hy = add_rn<T>(hy, vd.y);
      hy = add_rn<T>(hy, ve.y);
      V me = So[i];
      const T dE = -fma(sub_rn<T>(q.cs[h], me.x), hx, mul_rn<T>(sub_rn<T>(q.sn[h], me.y), hy));
      const bool own = WHOLE || (r >= H && r < H + R);
      if (accept_move(q.w2[h], dE, a.beta, a.beta_f)) {
        me.x = q.cs[h];
        me.y = q.sn[h];
        So[i] = me;
        acc += own;
      }
      if (meas && own) {
        double b2;  // u . h: in double from the neighbours themselves when T is float
        if (sizeof(T) == 8) {
          b2 = (double)me.x * (double)hx + (double)me.y * (double)hy;
        } else {
          const double dx = (double)va.x + vb.x + vd.x + ve.x, dy = (double)va.y + vb.y + vd.y + ve.y;
          b2 = (double)me.x * dx + (double)me.y * dy;
        }
        const V s0 = Sn[i];
        const double tx = (double)me.x + (double)s0.x, ty = (double)me.y + (double)s0.y;
        e = AHEAD ? -b2 : e - b2;  // AHEAD: the thread's only site
        mx = AHEAD ? tx : mx + tx;
        my = AHEAD ? ty : my + ty;
      }
    }
  };

  Prop q;
  if (AHEAD && item < items_end) propose(item, a.t0, 0, q);
  int to_rec = a.to_rec, g = 0;
  long long slot = a.rec0;
  uint32_t exchanges = 0;
  const int halves = 2 * a.n;
  for (int hh = 0; hh < halves; ++hh) {
    const int c = hh & 1;
    const uint32_t t = a.t0 + (uint32_t)(hh >> 1), t_next = a.t0 + (uint32_t)((hh + 1) >> 1);
    const bool meas = c == 1 && to_rec == 1;
    const int lo = WHOLE ? 0 : g + 1;
    const bool swap = !WHOLE && g + 1 == H && hh + 1 < halves;
    if (AHEAD) {
      if (in_rows(item, lo)) update(item, c, lo, meas, q);
      if (!swap && in_rows(item, WHOLE ? 0 : lo + 1)) propose(item, t_next, 1 - c, q);
    } else {
      for (int j = (lo * half + par) / SPT + tid; SPT * j - par < ns - lo * half; j += nth) {
        propose(j, t, c, q);
        update(j, c, lo, meas, q);
      }
    }
    if (meas) {
      // warp sums of the three values with 6 additions instead of 15: after the
      // first exchange the lower lanes hold (e, mx), the upper ones (my, -), after
      // the second lanes 0, 8, 16 ... hold one value each
      const bool up4 = (tid & 16) != 0, up3 = (tid & 8) != 0;
      const double p = (up4 ? my : e) + __shfl_xor_sync(0xffffffffu, up4 ? e : my, 16);
      const double r = (up4 ? 0.0 : mx) + __shfl_xor_sync(0xffffffffu, up4 ? mx : 0.0, 16);
      double v = (up3 ? r : p) + __shfl_xor_sync(0xffffffffu, up3 ? p : r, 8);
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      const int which = (up4 ? 2 : 0) + (up3 ? 1 : 0);  // 0: E, 1: Mx, 2: My
      if ((tid & 7) == 0 && which < 3) atomicAdd(&a.rec[3 * slot + which], v);
      e = mx = my = 0;
    }
    if (c == 1 && to_rec > 0 && --to_rec == 0) {
      to_rec = a.m;
      slot = slot + 1 == a.rec_cap ? 0 : slot + 1;
    }
    __syncthreads();
    ++g;
    if (!swap) continue;
    g = 0;
    // own rows [H, 2H) go up, [R, R + H) go down; with one half sweep between
    // exchanges only the colour just updated changed
    const uint32_t tag = ++exchanges;
    const size_t buf = (size_t)(tag & 1) * 4 * hw;
    const int c_first = H == 1 ? c : 0, c_count = H == 1 ? 1 : 2;
    const uint32_t* const words = reinterpret_cast<const uint32_t*>(S);
    for (int i = tid; i < 2 * c_count * hw; i += nth) {
      const int lower = i >= c_count * hw, rem = i - lower * c_count * hw;
      const int cc = c_first + (rem >= hw), k = rem - (rem >= hw ? hw : 0);
      send_word(mine + buf + (lower * 2 + cc) * (size_t)hw + k, tag,
                words[(size_t)(cc * plane + (lower ? R : H) * half) * VW + k]);
    }
    if (AHEAD && item < items_end) propose(item, t_next, 1 - c, q);
    bool ok = true;
    const int total = 2 * c_count * hw;
    // the upper neighbour's lower rows, the lower neighbour's upper rows; four
    // loads in flight per thread
    auto src = [&](int i) {
      const int lower = i >= c_count * hw, rem = i - lower * c_count * hw;
      const int cc = c_first + (rem >= hw), k = rem - (rem >= hw ? hw : 0);
      return a.xbuf + (lower ? dn : up) * per_cta + buf + ((1 - lower) * 2 + cc) * (size_t)hw + k;
    };
    recv_words<4>(tid, nth, total, src, tag, a.limit, a.status, ok, [&](int i, uint32_t word) {
      const int lower = i >= c_count * hw, rem = i - lower * c_count * hw;
      const int cc = c_first + (rem >= hw), k = rem - (rem >= hw ? hw : 0);
      reinterpret_cast<uint32_t*>(S)[(size_t)(cc * plane + (lower ? H + R : 0) * half) * VW + k] = word;
    });
    if (!__syncthreads_and(ok)) return;
  }
  // in place: both neighbours must have read their halos
  if (!WHOLE && exchanges == 0) {
    uint32_t word;
    bool ok = true;
    if (tid < 2) ok = recv_word(a.xbuf + (tid ? dn : up) * per_cta + 8 * hw, 1u, a.limit, a.status, word);
    if (!__syncthreads_and(ok)) return;
  }
  for (int i = tid; i < 2 * R * half; i += nth) {
    const int c = i >= R * half, k = i - c * R * half;
    a.u[(size_t)c * N2 + (size_t)y0 * half + k] = P(c)[H * half + k];
  }
  add_accepted(a.accepted, acc);
}

// Self-test of the persistent kernels' barrier: CTA 0 never arrives, so every
// other CTA must give up after `limit` cycles and record the time-out.
__global__ void k_grid_barrier_selftest(GridCtl* ctl, long long limit) {
  if (blockIdx.x == 0) return;
  grid_sync_bounded(ctl, limit);
}

template <typename T>
__global__ void k_xy_to_host_layout(const typename Vec<T>::type* __restrict__ u, int L, long long n0, long long count,
                                    double* __restrict__ out, int to_dev) {
  // sites [n0, n0 + count); to_dev = 0: planes -> [count][2] double; 1: the reverse (out is the source)
  using V = typename Vec<T>::type;
  const int half = L / 2;
  V* uu = const_cast<V*>(u);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    const long long n = n0 + i;
    const int y = (int)(n / L), x = (int)(n - (n / L) * L);
    const size_t idx = (size_t)((x + y) & 1) * L * half + (size_t)y * half + (x >> 1);
    if (to_dev) {
      V v;
      v.x = (T)out[2 * i];
      v.y = (T)out[2 * i + 1];
      uu[idx] = v;
    } else {
      out[2 * i] = (double)u[idx].x;
      out[2 * i + 1] = (double)u[idx].y;
    }
  }
}

int xfail(int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  set_last_error(buf);
  return code;
}

#define XTRY(expr)                                                                        \
  do {                                                                                    \
    cudaError_t e__ = (expr);                                                             \
    if (e__ != cudaSuccess) return xfail(ISING_ECUDA, "%s: %s", #expr, cudaGetErrorString(e__)); \
  } while (0)

int grid_of(long long items) {
  long long g = (items + 255) / 256;
  return (int)std::max(1LL, std::min(g, 152LL * 32));
}

}  // namespace
}  // namespace ising

using namespace ising;

struct ising_xy {
  int L = 0, precision = 64;
  int mode = 0;                      // 0 auto, 1 one launch per half sweep, 2 persistent
  GridCtl* ctl = nullptr;            // persistent-kernel barrier and status
  int64_t launches = 0;
  double beta = 0;
  uint64_t seed = 0;
  int64_t sweep = 0;
  cudaStream_t stream = nullptr;
  void* u = nullptr;  // two colour planes of vectors
  double* rec = nullptr;  // ring [65536][3]
  int64_t rec_count = 0;
  unsigned long long* accepted = nullptr;
  bool grid_used = false;            // a grid barrier ran since the last seed: its status is worth reading
  double* host_layout = nullptr;     // spins in the host's layout, at most kXYLayoutSites at a time (xy_layout)
  // resident strips of the automatic mode (G = 0: one launch per half sweep)
  int strip_G = 0, strip_gh = 0;
  double strip_us = 0;  // modelled time of a sweep
  unsigned long long* strip_x = nullptr;
  StripStatus strip_status;
};

namespace {
constexpr int64_t kXYRec = 65536;
constexpr long long kXYLayoutSites = 2 << 20;  // 16 bytes a site in the host's layout

// Largest L for which the automatic mode runs the resident strips.
// (us per sweep, strips / one launch per half sweep: FP64 L = 256 8.9 / 17.6, 1024 76 / 78; FP32 L = 256 3.1 / 8.2,
// 1024 13.1 / 20.6)
constexpr int kXYStripMaxL = 1024;
constexpr long long kXYSpinLimit = 4000000000LL;  // ~2 s of SM clock per barrier

// Strips and half sweeps per exchange for an L x L lattice by a time model (us),
// fitted on GB300 (within 20 % of the measured times, L = 8 ... 1024): a half sweep
// with w warps of sites per SM sub-partition takes 0.5 + 1.05 w in FP64 (31
// operations at 64 cycles per warp) and 0.45 + 0.08 w in FP32 (0.5 + 0.0013 per site
// past one site per thread), an exchange 0.9 + 3e-4 per word.
struct XYStrip {
  int G, gh;
  double us;
};
template <typename T>
XYStrip choose_xy_strip(int L, int sms) {
  const int half = L / 2;
  XYStrip best{0, 0, 1e30};
  for (int G = 1; G <= sms && G <= L; ++G)
    for (int gh = 1; gh <= (G == 1 ? 1 : 4); gh *= 2) {
      if (L / G < gh || xy_strip_smem<T>(L, G, gh) > 200 * 1024) continue;
      const int R = (L + G - 1) / G;
      const bool ahead = (R + (G == 1 ? 0 : 2 * gh - 2)) * half <= kXYStripThreads;
      const int words = (gh == 1 ? 2 : 4) * gh * half * (int)(sizeof(T) / 2);
      double t = G == 1 ? 0.0 : 0.9 + 3e-4 * words;
      for (int g = 0; g < gh; ++g) {
        const double s = (double)(R + (G == 1 ? 0 : 2 * (gh - 1 - g))) * half;
        const double w = std::ceil(std::ceil(s / 32) / 4);
        t += sizeof(T) == 8 ? 0.5 + 1.05 * w : ahead ? 0.45 + 0.08 * w : 0.5 + 0.0013 * s;
      }
      t *= 2.0 / gh;
      if (t < best.us) best = {G, gh, t};
    }
  return best;
}

template <typename T>
cudaError_t xy_strip_t(ising_xy* x, int n, int m) {
  XYStripArgs<T> a{};
  a.u = (typename Vec<T>::type*)x->u;
  a.L = x->L;
  a.G = x->strip_G;
  a.gh = std::min(x->strip_gh, 2 * n);
  a.beta = (T)x->beta;
  a.beta_f = beta_estimate(x->beta);
  a.t0 = (uint32_t)x->sweep;
  a.n = n;
  a.m = m;
  a.rec = x->rec;
  a.rec0 = x->rec_count % kXYRec;
  a.rec_cap = kXYRec;
  a.accepted = x->accepted;
  a.xbuf = x->strip_x;
  a.status = x->strip_status.word();
  a.limit = x->strip_status.limit(kXYSpinLimit);
  a.fh = make_fastdiv((uint32_t)(x->L / 2));
  const bool whole = a.G == 1;
  const long long sites = (long long)((a.L + a.G - 1) / a.G + (whole ? 0 : 2 * a.gh)) * (a.L / 2);
  const long long active = sites - (whole ? 0 : a.L);  // without the two outermost rows
  const bool ahead = active <= kXYStripThreads;
  const long long items = ahead || sizeof(T) == 8 ? active : active / 2 + 2;
  const int threads = (int)std::min<long long>(kXYStripThreads, (items + 31) / 32 * 32);
  const size_t smem = xy_strip_smem<T>(a.L, a.G, a.gh);
  const void* fns[4] = {(const void*)k_xy_strip<T, false, false>, (const void*)k_xy_strip<T, true, false>,
                        (const void*)k_xy_strip<T, false, true>, (const void*)k_xy_strip<T, true, true>};
  const int which = (whole ? 1 : 0) + (ahead ? 2 : 0);
  static DeviceCache configured[4];
  cudaError_t e = allow_dynamic_smem(fns[which], configured[which]);
  if (e) return e;
  // records of this launch: zeroed, then summed into by every CTA
  int64_t n_rec = 0;
  if (m > 0) {
    const int64_t before = x->sweep / m;
    n_rec = (x->sweep + n) / m - before;
    a.to_rec = n_rec ? (int)((before + 1) * m - x->sweep) : 0;
    const int64_t n1 = std::min<int64_t>(n_rec, kXYRec - a.rec0);
    if (n1 > 0 && (e = cudaMemsetAsync(x->rec + 3 * a.rec0, 0, (size_t)n1 * 24, x->stream))) return e;
    if (n_rec > n1 && (e = cudaMemsetAsync(x->rec, 0, (size_t)(n_rec - n1) * 24, x->stream))) return e;
  }
  RngParams r = make_rng(x->seed, 0, 0, 0);
  void* args[] = {&a, &r};
  if (whole) {
    e = cudaLaunchKernel(fns[which], dim3(1), dim3(threads), args, smem, x->stream);
  } else {
    e = cudaMemsetAsync(a.xbuf, 0, xy_strip_words<T>(a.L, a.G, a.gh) * 8, x->stream);
    if (!e) e = launch_strips(fns[which], a.G, threads, args, smem, x->strip_status.refuse, x->stream);
  }
  if (e) return e;
  ++x->launches;
  x->rec_count += n_rec;
  return cudaSuccess;
}

template <typename T>
cudaError_t xy_persist_t(ising_xy* x, int n, int m) {
  using V = typename Vec<T>::type;
  const RngParams rng = make_rng(x->seed, 0, 0, 0);
  const long long pairs = ((long long)x->L * (x->L / 2) + 1) / 2;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (!e) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e) return e;
  // FP32: one CTA up to 256 site pairs, one cluster of 8 CTAs up to 8192;
  // FP64, which runs at a small fraction of the FP32 rate on this part: one CTA
  // only up to 32 pairs.  Beyond, a cooperative grid spreading the pairs over
  // the SMs (32 threads per CTA in FP64, 64 in FP32).
  const bool fp64 = sizeof(T) == 8;
  const int pm = pairs <= (fp64 ? 32 : 256) ? kOneCTA : (!fp64 && pairs <= 8192 ? kCluster : kGrid);
  int threads;
  long long grid;
  const void* fn;
  if (pm == kOneCTA) {
    threads = (int)(((pairs + 31) / 32) * 32);
    grid = 1;
    fn = (const void*)k_xy_persist<T, kOneCTA>;
  } else if (pm == kCluster) {
    threads = (int)std::min<long long>(1024, ((pairs + 8 * 32 - 1) / (8 * 32)) * 32);
    grid = 8;
    fn = (const void*)k_xy_persist<T, kCluster>;
  } else {
    threads = fp64 ? 32 : 64;
    grid = std::max(1LL, std::min((pairs + threads - 1) / threads, (long long)sms));
    fn = (const void*)k_xy_persist<T, kGrid>;
    x->grid_used = true;
    e = cudaMemsetAsync(&x->ctl->count, 0, sizeof(unsigned int), x->stream);
    if (e) return e;
  }
  V* u = (V*)x->u;
  int L = x->L;
  T beta = (T)x->beta;
  uint32_t t0 = (uint32_t)x->sweep;
  long long rec0 = x->rec_count, cap = kXYRec, limit = kXYSpinLimit;
  double* rec = x->rec;
  unsigned long long* acc = x->accepted;
  GridCtl* ctl = x->ctl;
  RngParams r = rng;
  FastDiv fh = make_fastdiv((uint32_t)(x->L / 2));
  void* args[] = {&u, &L, &beta, &r, &t0, &n, &m, &rec, &rec0, &cap, &acc, &ctl, &limit, &fh};
  if (pm == kOneCTA) {
    e = cudaLaunchKernel(fn, dim3(1), dim3(threads), args, 0, x->stream);
  } else if (pm == kCluster) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = x->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)grid;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelExC(&cfg, fn, args);
  } else {
    e = cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(threads), args, 0, x->stream);
  }
  if (e) return e;
  ++x->launches;
  if (m > 0) {
    for (int s = 0; s < n; ++s)
      if (((int64_t)x->sweep + s + 1) % m == 0) ++x->rec_count;
  }
  return cudaSuccess;
}

// Single-precision calls of one sweep that the strips make slower than the forms before
// them.  us per call: half sweeps / strips (which clear their exchange buffer first) L = 64 8.2 /
// 10.3, 512 12.3 / 14.4, 1024 20.5 / 22.6; with a record, one CTA or one cluster: separate measurement /
// in the sweep L = 8 6.2 / 6.9, 10 to 20 8.2 / 6.9, 32 10.3 / 11.4, on strips 48 12.3 / 11.4, 50 11.3 / 12.5, 64 11.4 / 12.5, 72 12.3 /
// 12.6, 80 13.3 / 12.4 (FP64: at most even).
int xy_one_sweep_mode(const ising_xy* x, bool recorded) {
  if (x->mode != 0 || x->precision != 32) return x->mode;
  if (x->strip_G > 1 && !recorded) return 1;
  if (!recorded) return 0;
  return x->L < 10 || (x->strip_G == 1 && x->L > 24) || (x->L >= 50 && x->L <= 72) ? 2 : 0;
}

template <typename T>
cudaError_t xy_sweep_t(ising_xy* x, int n, int m) {
  const int mode = n == 1 ? xy_one_sweep_mode(x, m > 0 && (x->sweep + 1) % m == 0) : x->mode;
  if (mode == 0 && x->strip_G > 0) {
    // chunks whose records fit the ring, of about 20 ms
    const int launch = strip_launch_sweeps(x->strip_us);
    const int most = m > 0 ? (int)std::min<int64_t>(kXYRec * (int64_t)m, launch) : launch;
    cudaError_t e = cudaSuccess;
    int done = 0;
    for (; done < n && !e;) {
      const int k = std::min(most, n - done);
      e = xy_strip_t<T>(x, k, m);
      if (strips_refused(e)) {
        x->strip_G = 0;
        e = xy_sweep_t<T>(x, n - done, m);
        break;
      }
      x->sweep += k;
      done += k;
    }
    x->sweep -= done;  // the caller advances the counter
    return e;
  }
  if (mode == 2) return n > 0 ? xy_persist_t<T>(x, n, m) : cudaSuccess;
  const RngParams rng = make_rng(x->seed, 0, 0, 0);
  const long long blocks = ((long long)x->L * (x->L / 2) + 1) / 2;
  using V = typename Vec<T>::type;
  for (int s = 0; s < n; ++s) {
    const uint32_t t = (uint32_t)(x->sweep + s);
    for (int c = 0; c < 2; ++c) {
      k_xy_half<T><<<grid_of(blocks), 256, 0, x->stream>>>((V*)x->u, x->L, c, t, (T)x->beta, rng,
                                                            make_fastdiv((uint32_t)(x->L / 2)), x->accepted);
      cudaError_t e = cudaGetLastError();
      if (e) return e;
      ++x->launches;
    }
    if (m > 0 && ((int64_t)t + 1) % m == 0) {
      double* slot = x->rec + 3 * (x->rec_count % kXYRec);
      cudaError_t e = cudaMemsetAsync(slot, 0, 3 * sizeof(double), x->stream);
      if (e) return e;
      k_xy_measure<T><<<grid_of((long long)x->L * (x->L / 2)), 256, 0, x->stream>>>(
          (const V*)x->u, x->L, slot, make_fastdiv((uint32_t)(x->L / 2)));
      e = cudaGetLastError();
      if (e) return e;
      ++x->launches;
      ++x->rec_count;
    }
  }
  return cudaSuccess;
}
}  // namespace

extern "C" {

int ising_xy_create(ising_xy** out, int L, double beta, int precision, void* stream) {
  if (!out) return xfail(ISING_EINVAL, "null output pointer");
  *out = nullptr;
  if (L < 2 || L > 32768 || (L & 1)) return xfail(ISING_EINVAL, "L must be even and in [2, 32768]");
  if (!std::isfinite(beta) || beta <= 0) return xfail(ISING_EINVAL, "beta must be finite and > 0");
  if (precision != 32 && precision != 64) return xfail(ISING_EINVAL, "precision must be 32 or 64");
  ising_xy* x = new (std::nothrow) ising_xy();
  if (!x) return xfail(ISING_ENOMEM, "host allocation failed");
  x->L = L;
  x->beta = beta;
  x->precision = precision;
  x->stream = (cudaStream_t)stream;
  const size_t bytes = (size_t)L * L * (precision == 64 ? 16 : 8);
  int dev = 0, sms = 0;
  size_t strip_words = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (!e) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (!e && L <= kXYStripMaxL) {
    const XYStrip st = precision == 64 ? choose_xy_strip<double>(L, sms) : choose_xy_strip<float>(L, sms);
    x->strip_G = st.G;
    x->strip_gh = st.gh;
    x->strip_us = st.us;
    if (st.G > 1) {
      strip_words = precision == 64 ? xy_strip_words<double>(L, st.G, st.gh) : xy_strip_words<float>(L, st.G, st.gh);
      e = x->strip_status.ensure();
    }
  }
  // one allocation: each that starts a 2 MB page of its own takes 80 us
  const size_t sizes[5] = {bytes, kXYRec * 3 * sizeof(double), strip_words * sizeof(unsigned long long),
                           sizeof(unsigned long long), sizeof(GridCtl)};
  size_t at[6] = {0};
  for (int k = 0; k < 5; ++k) at[k + 1] = at[k] + (sizes[k] + 255) / 256 * 256;
  if (!e) e = cudaMalloc(&x->u, at[5]);
  if (!e) {
    char* const m = (char*)x->u;
    x->rec = (double*)(m + at[1]);
    if (strip_words) x->strip_x = (unsigned long long*)(m + at[2]);
    x->accepted = (unsigned long long*)(m + at[3]);
    x->ctl = (GridCtl*)(m + at[4]);
    e = cudaMemset(x->accepted, 0, at[5] - at[3]);
  }
  if (e) {
    cudaGetLastError();
    x->strip_status.release();
    cudaFree(x->u);
    delete x;
    return xfail(ISING_ENOMEM, "XY allocation: %s", cudaGetErrorString(e));
  }
  *out = x;
  return ising_xy_seed(x, 0);
}

int ising_xy_seed(ising_xy* x, uint64_t seed) {
  if (!x) return xfail(ISING_EINVAL, "null context");
  x->seed = seed;
  x->sweep = 0;
  x->rec_count = 0;
  x->grid_used = false;
  XTRY(x->strip_status.begin(x->stream));
  const RngParams rng = make_rng(seed, 0, 0, 0);
  const long long N = (long long)x->L * x->L;
  if (x->precision == 64)
    k_xy_init<double><<<grid_of(N), 256, 0, x->stream>>>((double2*)x->u, x->L, rng);
  else
    k_xy_init<float><<<grid_of(N), 256, 0, x->stream>>>((float2*)x->u, x->L, rng);
  XTRY(cudaGetLastError());
  XTRY(cudaMemsetAsync(x->accepted, 0, sizeof(unsigned long long), x->stream));
  XTRY(cudaMemsetAsync(x->ctl, 0, sizeof(GridCtl), x->stream));
  set_last_error("");
  return ISING_OK;
}

int ising_xy_sweep(ising_xy* x, int n_sweeps, int measure_every) {
  if (!x) return xfail(ISING_EINVAL, "null context");
  if (n_sweeps < 0 || measure_every < 0) return xfail(ISING_EINVAL, "negative count");
  if (x->sweep + n_sweeps >= ((int64_t)1 << 32)) return xfail(ISING_EINVAL, "sweep counter overflow");
  NvtxRange nvtx("ising_xy_sweep");
  XTRY(x->precision == 64 ? xy_sweep_t<double>(x, n_sweeps, measure_every)
                          : xy_sweep_t<float>(x, n_sweeps, measure_every));
  x->sweep += n_sweeps;
  set_last_error("");
  return ISING_OK;
}

// After a synchronising call: ETIMEOUT if a persistent kernel's grid barrier
// or a strip's wait gave up (until the lattice is seeded or set again).
static int xy_status(ising_xy* x) {
  if (x->strip_status.failed())
    return xfail(ISING_ETIMEOUT, "a strip's wait for its neighbour timed out in the XY kernel");
  if (!x->grid_used) return ISING_OK;
  int st = 0;
  XTRY(cudaMemcpy(&st, &x->ctl->status, sizeof(int), cudaMemcpyDeviceToHost));
  if (st) return xfail(ISING_ETIMEOUT, "grid barrier timed out in the persistent XY kernel");
  return ISING_OK;
}

int ising_selftest_grid_barrier(double timeout_s, int* timed_out) {
  if (!timed_out || !(timeout_s > 0) || timeout_s > 10) return xfail(ISING_EINVAL, "bad arguments");
  GridCtl* ctl = nullptr;
  XTRY(cudaMalloc((void**)&ctl, sizeof(GridCtl)));
  cudaError_t e = cudaMemset(ctl, 0, sizeof(GridCtl));
  if (!e) {
    GridCtl* c = ctl;
    long long limit = (long long)(timeout_s * 2.1e9);  // SM clock cycles (<= 2.1 GHz)
    void* args[] = {&c, &limit};
    e = cudaLaunchCooperativeKernel((const void*)k_grid_barrier_selftest, dim3(4), dim3(32), args, 0, 0);
  }
  if (!e) e = cudaDeviceSynchronize();
  GridCtl h{};
  if (!e) e = cudaMemcpy(&h, ctl, sizeof(GridCtl), cudaMemcpyDeviceToHost);
  cudaFree(ctl);
  if (e) return xfail(ISING_ECUDA, "barrier self-test: %s", cudaGetErrorString(e));
  *timed_out = h.status;
  set_last_error("");
  return ISING_OK;
}

int ising_xy_set_mode(ising_xy* x, int mode) {
  if (!x) return xfail(ISING_EINVAL, "null context");
  if (mode < 0 || mode > 2) return xfail(ISING_EINVAL, "mode must be 0 (auto), 1 (per half sweep) or 2 (persistent)");
  x->mode = mode;
  set_last_error("");
  return ISING_OK;
}

int ising_xy_launch_count(ising_xy* x, int64_t* count) {
  if (!x || !count) return xfail(ISING_EINVAL, "null argument");
  *count = x->launches;
  return ISING_OK;
}

int ising_xy_series(ising_xy* x, double* E, double* Mx, double* My, int n) {
  if (!x) return xfail(ISING_EINVAL, "null context");
  if (n < 0 || n > std::min<int64_t>(x->rec_count, kXYRec)) return xfail(ISING_EINVAL, "n exceeds records");
  std::vector<double> h((size_t)3 * n);
  const int64_t s0 = (x->rec_count - n) % kXYRec, n1 = std::min<int64_t>(n, kXYRec - s0);
  if (n1 > 0) XTRY(cudaMemcpyAsync(h.data(), x->rec + 3 * s0, (size_t)n1 * 24, cudaMemcpyDeviceToHost, x->stream));
  if (n > n1)
    XTRY(cudaMemcpyAsync(h.data() + 3 * n1, x->rec, (size_t)(n - n1) * 24, cudaMemcpyDeviceToHost, x->stream));
  XTRY(cudaStreamSynchronize(x->stream));
  if (int st = xy_status(x)) return st;
  for (int i = 0; i < n; ++i) {
    if (E) E[i] = h[3 * i];
    if (Mx) Mx[i] = h[3 * i + 1];
    if (My) My[i] = h[3 * i + 2];
  }
  set_last_error("");
  return ISING_OK;
}

// Spins between the planes and the host's layout, through a device buffer of at most 32 MB
// that the context keeps (an allocation per call took 100 us; one for the whole lattice
// would hold 17 GB at L = 32768).
static cudaError_t xy_layout(ising_xy* x, double* host, bool to_dev) {
  const long long N = (long long)x->L * x->L, most = std::min(N, kXYLayoutSites);
  cudaError_t e = cudaSuccess;
  if (!x->host_layout) {
    e = cudaMalloc((void**)&x->host_layout, most * 2 * sizeof(double));
    if (e) return e;
  }
  double* const d = x->host_layout;
  for (long long n0 = 0; n0 < N && !e; n0 += most) {
    const long long count = std::min(most, N - n0);
    const size_t bytes = (size_t)count * 2 * sizeof(double);
    if (to_dev) e = cudaMemcpyAsync(d, host + 2 * n0, bytes, cudaMemcpyHostToDevice, x->stream);
    if (e) return e;
    if (x->precision == 64)
      k_xy_to_host_layout<double><<<grid_of(count), 256, 0, x->stream>>>((const double2*)x->u, x->L, n0, count, d, to_dev);
    else
      k_xy_to_host_layout<float><<<grid_of(count), 256, 0, x->stream>>>((const float2*)x->u, x->L, n0, count, d, to_dev);
    e = cudaGetLastError();
    if (!e && !to_dev) e = cudaMemcpyAsync(host + 2 * n0, d, bytes, cudaMemcpyDeviceToHost, x->stream);
  }
  return e ? e : cudaStreamSynchronize(x->stream);
}

int ising_xy_get_spins(ising_xy* x, double* host_uv) {
  if (!x || !host_uv) return xfail(ISING_EINVAL, "null argument");
  cudaError_t e = xy_layout(x, host_uv, false);
  if (e) return xfail(ISING_ECUDA, "get spins: %s", cudaGetErrorString(e));
  if (int st = xy_status(x)) return st;
  set_last_error("");
  return ISING_OK;
}

int ising_xy_set_spins(ising_xy* x, const double* host_uv) {
  if (!x || !host_uv) return xfail(ISING_EINVAL, "null argument");
  XTRY(x->strip_status.begin(x->stream));
  XTRY(cudaMemsetAsync(x->ctl, 0, sizeof(GridCtl), x->stream));
  cudaError_t e = xy_layout(x, const_cast<double*>(host_uv), true);
  if (e) return xfail(ISING_ECUDA, "set spins: %s", cudaGetErrorString(e));
  set_last_error("");
  return ISING_OK;
}

int ising_xy_accepted(ising_xy* x, int64_t* accepted) {
  if (!x || !accepted) return xfail(ISING_EINVAL, "null argument");
  unsigned long long h = 0;
  XTRY(cudaMemcpyAsync(&h, x->accepted, 8, cudaMemcpyDeviceToHost, x->stream));
  XTRY(cudaStreamSynchronize(x->stream));
  if (int st = xy_status(x)) return st;
  *accepted = (int64_t)h;
  set_last_error("");
  return ISING_OK;
}

int ising_xy_destroy(ising_xy* x) {
  if (!x) return ISING_OK;
  cudaStreamSynchronize(x->stream);
  cudaFree(x->u);
  cudaFree(x->host_layout);
  x->strip_status.release();
  delete x;
  return ISING_OK;
}

}  // extern "C"
