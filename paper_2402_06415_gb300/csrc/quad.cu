// Quadripartite Metropolis sweep of the Ising model on lattices with a
// four-site unit cell (arXiv 2402.06415, Results "optimising the partition",
// Fig. 5b/5d; Supplementary Fig. S4a-c): the four sites of a cell belong to four
// sublattices, none of which has an internal bond, so a sweep is four parallel
// steps (sublattice 0, 1, 2, 3).
//
// Lattices on Lc x Lc periodic cells:
//   SQUARE: square lattice of side 2 Lc, site (2X + i, 2Y + j) in sublattice
//     q = i + 2j; J1 on nearest neighbours, J2 on the diagonal (next-nearest)
//     neighbours.
//   SQOCT: square-octagon (4.8.8) lattice; cell sites A, B, C, D (q = 0..3)
//     form a J1 square A-B-C-D-A; J2 octagon bonds B(X,Y)-D(X+1,Y), A(X,Y)-C(X,Y+1).
// Flip of a site with a1 / a2 antiparallel J1 / J2 neighbours (z1, z2 of them):
// dE = 2 J1 (z1 - 2 a1) + 2 J2 (z2 - 2 a2); flip iff dE <= 0 or u < T(a1, a2) =
// floor(exp(-beta dE) 2^32), computed once on the host.
//
// Layout: one bit plane per sublattice, [4][Lc][Wq] u32 words, Wq = ceil(Lc/32),
// bit b of word w of row Y = cell X = 32 w + b (1 = spin up); padding bits 0.
// One thread per word: neighbour words of the other three planes (a one-bit
// funnel shift for the x-offset cells), bit-sliced counts of antiparallel J1 and
// J2 neighbours, class masks, then a lazy bit-serial compare u < T against the
// per-lane threshold, MSB first, generating Philox planes only while lanes are
// undecided.  Uniform of lane b: u = sum_k bit_b(P_k) 2^(31-k), P_{4m+k} = word
// k of Philox(g, t, replica, QUAD_MET << 16 | q << 8 | m), g = Y Wq + w.
#include <cuda_runtime.h>

#include <algorithm>
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

constexpr uint32_t kTagQuadInit = 12, kTagQuadMet = 13;
constexpr int kMaxClasses = 25;

struct QuadGeom {
  int Lc, Wq, nlast;  // nlast: valid bits of a row's last word (1..32)
  FastDiv fw;         // division by Wq
};

// Decision table of one (lattice, beta, J1, J2): class c = a1 (z2 + 1) + a2.
struct QuadTable {
  uint32_t always;            // classes with dE <= 0
  int n_vals;                 // distinct thresholds of the other classes
  uint32_t val[kMaxClasses];  // the thresholds
  uint32_t cls[kMaxClasses];  // bitset of the classes holding val[d]
  uint32_t lm[kMaxClasses][32];  // all ones iff bit 31 - k of val[d] is set
};

struct Count3 {  // bit-sliced 3-bit counter per lane (counts 0..4)
  uint32_t c0 = 0, c1 = 0, c2 = 0;
  __device__ __forceinline__ void add(uint32_t x) {
    const uint32_t k0 = c0 & x;
    c0 ^= x;
    const uint32_t k1 = c1 & k0;
    c1 ^= k0;
    c2 |= k1;
  }
  __device__ __forceinline__ uint32_t eq(int v) const {
    return ((v & 1) ? c0 : ~c0) & ((v & 2) ? c1 : ~c1) & ((v & 4) ? c2 : ~c2);
  }
};

// Neighbour-plane loads: through the read-only path from global memory (G), or
// plain loads from shared memory in the persistent single-CTA kernel.
template <bool G>
__device__ __forceinline__ uint32_t ldw(const uint32_t* p) {
  if (G) return __ldg(p);
  return *p;
}

// Word whose bit b holds the spin of cell X = 32 w + b + DX (periodic in X) of a row.
template <int DX, bool G = true>
__device__ __forceinline__ uint32_t xword(const uint32_t* __restrict__ row, const QuadGeom& g, int w) {
  const uint32_t cur = ldw<G>(row + w);
  if (DX == 0) return cur;
  if (DX > 0) {
    const bool last = w == g.Wq - 1;
    const uint32_t nxt = ldw<G>(row + (last ? 0 : w + 1));
    const int valid = last ? g.nlast : 32;
    return (cur >> 1) | ((nxt & 1u) << (valid - 1));
  }
  const bool first = w == 0;
  const uint32_t prv = ldw<G>(row + (first ? g.Wq - 1 : w - 1));
  const int pvalid = first ? g.nlast : 32;
  return (cur << 1) | ((prv >> (pvalid - 1)) & 1u);
}

template <bool G>
__device__ __forceinline__ uint32_t xword_dir(const uint32_t* row, const QuadGeom& g, int w, int dx) {
  return dx > 0 ? xword<1, G>(row, g, w) : xword<-1, G>(row, g, w);
}

// Antiparallel J1 / J2 neighbour counts of the 32 sites of word (q, Y, w).
template <int LAT, bool G = true>
__device__ __forceinline__ void count_anti(const uint32_t* __restrict__ planes, const QuadGeom& g,
                                           int q, int Y, int w, uint32_t me, Count3& n1, Count3& n2) {
  const size_t plane = (size_t)g.Lc * g.Wq;
  const int Yp = Y + 1 == g.Lc ? 0 : Y + 1, Ym = Y == 0 ? g.Lc - 1 : Y - 1;
  if (LAT == ISING_QUAD_SQUARE) {
    const int sx = (q & 1) ? 1 : -1;
    const int Yn = (q & 2) ? Yp : Ym;
    const uint32_t* rx = planes + (size_t)(q ^ 1) * plane + (size_t)Y * g.Wq;
    const uint32_t* ry0 = planes + (size_t)(q ^ 2) * plane + (size_t)Y * g.Wq;
    const uint32_t* ry1 = planes + (size_t)(q ^ 2) * plane + (size_t)Yn * g.Wq;
    const uint32_t* rd0 = planes + (size_t)(q ^ 3) * plane + (size_t)Y * g.Wq;
    const uint32_t* rd1 = planes + (size_t)(q ^ 3) * plane + (size_t)Yn * g.Wq;
    n1.add(me ^ xword<0, G>(rx, g, w));
    n1.add(me ^ xword_dir<G>(rx, g, w, sx));
    n1.add(me ^ xword<0, G>(ry0, g, w));
    n1.add(me ^ xword<0, G>(ry1, g, w));
    n2.add(me ^ xword<0, G>(rd0, g, w));
    n2.add(me ^ xword_dir<G>(rd0, g, w, sx));
    n2.add(me ^ xword<0, G>(rd1, g, w));
    n2.add(me ^ xword_dir<G>(rd1, g, w, sx));
  } else {
    const int nxt = (q + 1) & 3, prv = (q + 3) & 3;
    n1.add(me ^ xword<0, G>(planes + (size_t)nxt * plane + (size_t)Y * g.Wq, g, w));
    n1.add(me ^ xword<0, G>(planes + (size_t)prv * plane + (size_t)Y * g.Wq, g, w));
    uint32_t o;
    if (q == 0) o = xword<0, G>(planes + 2 * plane + (size_t)Yp * g.Wq, g, w);
    else if (q == 1) o = xword<1, G>(planes + 3 * plane + (size_t)Y * g.Wq, g, w);
    else if (q == 2) o = xword<0, G>(planes + 0 * plane + (size_t)Ym * g.Wq, g, w);
    else o = xword<-1, G>(planes + 1 * plane + (size_t)Y * g.Wq, g, w);
    n2.add(me ^ o);
  }
}

__device__ __forceinline__ uint32_t valid_bits(const QuadGeom& g, int w) {
  return (w == g.Wq - 1 && g.nlast < 32) ? ((1u << g.nlast) - 1u) : 0xffffffffu;
}

// Metropolis trials of the 32 sites of word i = Y Wq + w of sublattice q.
// All 32 lanes of the warp call it together (warp vote); lanes past the end pass
// active = false (any in-range i) and change nothing.
// grp is the word's index in the whole lattice (its Philox counter).  The first NB
// Philox blocks are drawn for every word and compared as one 4 NB-bit borrow chain;
// the rest while a lane of the warp is tied.
template <int LAT, int NV, bool G, int NB>
__device__ __forceinline__ void quad_word(uint32_t* __restrict__ planes, const QuadGeom& g, int q,
                                          long long i, uint32_t grp, bool active, uint32_t t, const RngParams& rng,
                                          const QuadTable& tab) {
  constexpr int Z2 = LAT == ISING_QUAD_SQUARE ? 4 : 1;
  constexpr int Z1 = LAT == ISING_QUAD_SQUARE ? 4 : 2;
  if (!active) i = 0;
  const int Y = (int)fdiv((uint32_t)i, g.fw), w = (int)((uint32_t)i - (uint32_t)Y * (uint32_t)g.Wq);
  uint32_t* own = planes + (size_t)q * g.Lc * g.Wq + i;
  const uint32_t me = *own;
  const uint32_t valid = active ? valid_bits(g, w) : 0u;
  Count3 n1, n2;
  count_anti<LAT, G>(planes, g, q, Y, w, me, n1, n2);
  uint32_t e2[Z2 + 1];
#pragma unroll
  for (int a2 = 0; a2 <= Z2; ++a2) e2[a2] = n2.eq(a2);
  uint32_t always = 0, vm[NV];
#pragma unroll
  for (int d = 0; d < NV; ++d) vm[d] = 0;
#pragma unroll
  for (int a1 = 0; a1 <= Z1; ++a1) {
    const uint32_t e1 = n1.eq(a1);
#pragma unroll
    for (int a2 = 0; a2 <= Z2; ++a2) {
      const int c = a1 * (Z2 + 1) + a2;
      const uint32_t cm = e1 & e2[a2];
      always |= cm & (0u - ((tab.always >> c) & 1u));
#pragma unroll
      for (int d = 0; d < NV; ++d) vm[d] |= cm & (0u - ((tab.cls[d] >> c) & 1u));
    }
  }
  uint32_t und = ~always & valid, lt = 0;
  // the level is a compile-time index, so each threshold-bit mask is a constant operand
  auto level_mask = [&](int lvl) {
    uint32_t tm = 0;
#pragma unroll
    for (int d = 0; d < NV; ++d) tm |= vm[d] & tab.lm[d][lvl];
    return tm;
  };
  auto block = [&](int m) {
    return philox10_rk(make_uint4(grp, t, rng.replica, (kTagQuadMet << 16) | ((uint32_t)q << 8) | (uint32_t)m),
                       rng.rk0, rng.rk1);
  };
  {
    uint32_t bor = 0, eq = und;
#pragma unroll
    for (int m = NB - 1; m >= 0; --m) {
      const uint4 r = block(m);
      const uint32_t pw[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
      for (int k = 3; k >= 0; --k) {
        const uint32_t tm = level_mask(4 * m + k);
        bor = (~pw[k] & tm) | (~pw[k] & bor) | (tm & bor);
        eq &= ~(tm ^ pw[k]);
      }
    }
    lt = und & bor;
    und = eq;
  }
#pragma unroll
  for (int m = NB; m < 8; ++m) {
    if (!__any_sync(0xffffffffu, und != 0u)) break;
    const uint4 r = block(m);
    const uint32_t pw[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t tm = level_mask(4 * m + k);
      lt |= und & ~pw[k] & tm;
      und &= ~(pw[k] ^ tm);
    }
  }
  const uint32_t flip = (always | lt) & valid;
  if (active && flip) *own = me ^ flip;
}

template <int LAT, int NV>
__global__ void __launch_bounds__(256) k_quad_quarter(uint32_t* __restrict__ planes, QuadGeom g, int q,
                                                      uint32_t t, RngParams rng, QuadTable tab) {
  const long long words = (long long)g.Lc * g.Wq;
  const int lane = threadIdx.x & 31;
  for (long long base = (blockIdx.x * (long long)blockDim.x + threadIdx.x) - lane; base < words;
       base += (long long)gridDim.x * blockDim.x)
    quad_word<LAT, NV, true, 2>(planes, g, q, base + lane, (uint32_t)(base + lane), base + lane < words, t, rng, tab);
}

__global__ void k_quad_init(uint32_t* __restrict__ planes, QuadGeom g, RngParams rng) {
  const long long words = (long long)g.Lc * g.Wq;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 4 * words;
       i += (long long)gridDim.x * blockDim.x) {
    const int q = (int)(i / words);
    const long long gi = i - (long long)q * words;
    const int w = (int)(gi % g.Wq);
    const uint4 r = philox10_rk(make_uint4((uint32_t)gi, 0u, rng.replica, (kTagQuadInit << 16) | ((uint32_t)q << 8)),
                                rng.rk0, rng.rk1);
    planes[i] = r.x & valid_bits(g, w);
  }
}

// Bond sums of word i of the 4 Lc Wq words: (2 B1, 2 B2, M) contributions (each
// bond is seen from both ends).
template <int LAT, bool G>
__device__ __forceinline__ void quad_measure_word(const uint32_t* __restrict__ planes, const QuadGeom& g,
                                                  long long i, long long& b1, long long& b2, long long& m) {
  constexpr int Z1 = LAT == ISING_QUAD_SQUARE ? 4 : 2;
  constexpr int Z2 = LAT == ISING_QUAD_SQUARE ? 4 : 1;
  const long long words = (long long)g.Lc * g.Wq;
  const int q = (int)(i / words);
  const long long gi = i - (long long)q * words;
  const int Y = (int)fdiv((uint32_t)gi, g.fw), w = (int)((uint32_t)gi - (uint32_t)Y * (uint32_t)g.Wq);
  const uint32_t v = valid_bits(g, w);
  const uint32_t me = planes[i];
  Count3 n1, n2;
  count_anti<LAT, G>(planes, g, q, Y, w, me, n1, n2);
  const int nv = __popc(v);
  const int anti1 = __popc(n1.c0 & v) + 2 * __popc(n1.c1 & v) + 4 * __popc(n1.c2 & v);
  const int anti2 = __popc(n2.c0 & v) + 2 * __popc(n2.c1 & v) + 4 * __popc(n2.c2 & v);
  b1 += (long long)Z1 * nv - 2LL * anti1;
  b2 += (long long)Z2 * nv - 2LL * anti2;
  m += 2LL * __popc(me & v) - nv;
}

// rec[0] += 2 B1, rec[1] += 2 B2, rec[2] += M.
template <int LAT>
__global__ void __launch_bounds__(256) k_quad_measure(const uint32_t* __restrict__ planes, QuadGeom g,
                                                      unsigned long long* __restrict__ rec) {
  const long long words = (long long)g.Lc * g.Wq;
  long long b1 = 0, b2 = 0, m = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 4 * words;
       i += (long long)gridDim.x * blockDim.x)
    quad_measure_word<LAT, true>(planes, g, i, b1, b2, m);
  const unsigned long long s1 = warp_sum_u64((unsigned long long)b1);
  const unsigned long long s2 = warp_sum_u64((unsigned long long)b2);
  const unsigned long long s3 = warp_sum_u64((unsigned long long)m);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&rec[0], s1);
    atomicAdd(&rec[1], s2);
    atomicAdd(&rec[2], s3);
  }
}

// Small lattices (the paper's N = 16 ... 4096 and up to 256^2 cells): the whole
// lattice in shared memory, one CTA, n sweeps in one launch with __syncthreads()
// between quarter sweeps; records (2 B1, 2 B2, M) written to ring slots rec0, ...
template <int LAT, int NV>
__global__ void __launch_bounds__(1024) k_quad_persist(uint32_t* __restrict__ planes, QuadGeom g, uint32_t t0,
                                                       int n, int meas_every, RngParams rng, QuadTable tab,
                                                       unsigned long long* __restrict__ rec, long long rec0,
                                                       long long rec_cap) {
  extern __shared__ uint32_t sp[];
  __shared__ long long red[3][32];
  const long long words = (long long)g.Lc * g.Wq;
  for (long long i = threadIdx.x; i < 4 * words; i += blockDim.x) sp[i] = planes[i];
  __syncthreads();
  long long ri = rec0;
  for (int s = 0; s < n; ++s) {
    const uint32_t t = t0 + (uint32_t)s;
    for (int q = 0; q < 4; ++q) {
      for (long long base = threadIdx.x & ~31; base < words; base += blockDim.x)
        quad_word<LAT, NV, false, 2>(sp, g, q, base + (threadIdx.x & 31), (uint32_t)(base + (threadIdx.x & 31)),
                                     base + (threadIdx.x & 31) < words, t, rng, tab);
      __syncthreads();
    }
    if (meas_every > 0 && ((long long)t + 1) % meas_every == 0) {
      long long b1 = 0, b2 = 0, m = 0;
      for (long long i = threadIdx.x; i < 4 * words; i += blockDim.x) quad_measure_word<LAT, false>(sp, g, i, b1, b2, m);
      b1 = (long long)warp_sum_u64((unsigned long long)b1);
      b2 = (long long)warp_sum_u64((unsigned long long)b2);
      m = (long long)warp_sum_u64((unsigned long long)m);
      const int wid = threadIdx.x >> 5;
      if ((threadIdx.x & 31) == 0) {
        red[0][wid] = b1;
        red[1][wid] = b2;
        red[2][wid] = m;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        long long a = 0, b = 0, c = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
          a += red[0][k];
          b += red[1][k];
          c += red[2][k];
        }
        unsigned long long* slot = rec + 3 * (ri % rec_cap);
        slot[0] = (unsigned long long)a;
        slot[1] = (unsigned long long)b;
        slot[2] = (unsigned long long)c;
      }
      ++ri;
      __syncthreads();
    }
  }
  for (long long i = threadIdx.x; i < 4 * words; i += blockDim.x) planes[i] = sp[i];
}

// Resident strips (as the two-sublattice sweep's): G CTAs own row strips of full
// width, the four planes in shared memory, K sweeps between exchanges of boundary
// rows.  A sweep invalidates one more halo row on each side: two of the quarter
// sweeps read the row below, two the row above, so the first pair runs one row
// further than the second on the side it does not read from.  The halo has
// H = K + 1 rows, because the bond sums of a recorded sweep read one row beyond
// the strip.
// Bound by the dependent chain of a quarter sweep (~0.6 us) up to 1024^2 cells (there two
// warps a sub-partition, ALU pipe 40 % busy), then by the ALU pipe.  The 4.8.8 form for up to
// 8 classes spills 56 bytes at its 64 registers.  us per sweep, before (one CTA up to 256^2 cells, else a launch per
// quarter sweep) and with strips: 4.8.8 at 256^2 19.5 -> 2.7, 1024^2 16.5 -> 4.5, 4096^2
// 49.8 -> 34.5; square J2 = 0.5 at 1024^2 24.7 -> 8.8.  8192^2 does not fit and keeps
// the launches (152 us, ALU pipe bound).
struct QuadStripArgs {
  uint32_t* planes;
  QuadGeom g;
  int G, K;
  uint32_t t0;
  int n, m, to_rec;  // sweeps; record every m; sweeps until the first record (0: none)
  unsigned long long* rec;
  long long rec0, rec_cap;
  unsigned long long* xbuf;  // quad_strip_words(...) pairs, zeroed by the launcher
  int* status;
  long long limit;
};
constexpr int kQuadStripThreads = 512, kQuadStripMaxK = 4;

size_t quad_strip_words(const QuadGeom& g, int G, int K) { return (size_t)G * (16 * (size_t)(K + 1) * g.Wq + 1); }
size_t quad_strip_smem(const QuadGeom& g, int G, int K) {
  return 4 * (size_t)((g.Lc + G - 1) / G + 2 * (K + 1)) * g.Wq * sizeof(uint32_t);
}

template <int LAT, int NV>
__global__ void __launch_bounds__(kQuadStripThreads) k_quad_strip(QuadStripArgs a, RngParams rng, QuadTable tab) {
  extern __shared__ uint32_t sp[];
  const int Lc = a.g.Lc, Wq = a.g.Wq, G = a.G, H = a.K + 1;
  const int b = blockIdx.x, tid = threadIdx.x, nth = blockDim.x, lane = tid & 31;
  const int y0 = (int)((long long)b * Lc / G), R = (int)((long long)(b + 1) * Lc / G) - y0;
  const int rows = R + 2 * H, plane = rows * Wq, LW = Lc * Wq;
  const QuadGeom gl{rows, Wq, a.g.nlast, a.g.fw};
  const int goff = (y0 - H) * Wq;  // local word i is word i + goff of its plane, modulo LW
  auto group_of = [&](int i) {
    int k = i + goff;
    k += k < 0 ? LW : 0;
    k -= k >= LW ? LW : 0;
    return k;
  };
  for (int q = 0; q < 4; ++q)
    for (int i = tid; i < plane; i += nth) sp[q * plane + i] = __ldcg(&a.planes[(size_t)q * LW + group_of(i)]);
  __syncthreads();
  const int hw = H * Wq;
  const size_t per_cta = 16 * (size_t)hw + 1;
  const int up = b == 0 ? G - 1 : b - 1, dn = b == G - 1 ? 0 : b + 1;
  unsigned long long* const mine = a.xbuf + b * per_cta;
  if (tid == 0) send_word(mine + 16 * hw, 1u, 0u);  // "lattice read"
  int to_rec = a.to_rec;
  long long slot = a.rec0;
  uint32_t exchanges = 0;
  for (int done = 0; done < a.n;) {
    const int kk = min(a.K, a.n - done);
    // the outermost halo rows are needed only if a sweep of this group is recorded
    const int skip = to_rec > 0 && to_rec <= kk ? a.K - kk : a.K - kk + 1;
    for (int s = 0; s < kk; ++s) {
      const uint32_t t = a.t0 + (uint32_t)(done + s);
      const int e = skip + s;  // halo rows already invalid (or not needed) on each side
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        // square: q = 0, 1 read the row above, 2, 3 the row below; 4.8.8: 0 the row below, 2 the row above
        const int lo = LAT == ISING_QUAD_SQUARE ? e + 1 : (q < 2 ? e : e + 1);
        const int hi = LAT == ISING_QUAD_SQUARE ? (q < 2 ? rows - e : rows - e - 1) : rows - e - 1;
        const int count = (hi - lo) * Wq;
        for (int base = tid & ~31; base < count; base += nth) {
          const bool active = base + lane < count;
          const int i = lo * Wq + (active ? base + lane : 0);
          quad_word<LAT, NV, false, 3>(sp, gl, q, i, (uint32_t)group_of(i), active, t, rng, tab);
        }
        __syncthreads();
      }
      if (to_rec > 0 && --to_rec == 0) {
        to_rec = a.m;
        long long b1 = 0, b2 = 0, m = 0;
        for (int i = tid; i < 4 * R * Wq; i += nth) {
          const int q = i / (R * Wq);
          quad_measure_word<LAT, false>(sp, gl, (long long)q * plane + hw + (i - q * R * Wq), b1, b2, m);
        }
        const unsigned long long s1 = warp_sum_u64((unsigned long long)b1);
        const unsigned long long s2 = warp_sum_u64((unsigned long long)b2);
        const unsigned long long s3 = warp_sum_u64((unsigned long long)m);
        if (lane == 0) {
          atomicAdd(&a.rec[3 * slot], s1);
          atomicAdd(&a.rec[3 * slot + 1], s2);
          atomicAdd(&a.rec[3 * slot + 2], s3);
        }
        slot = slot + 1 == a.rec_cap ? 0 : slot + 1;
        __syncthreads();
      }
    }
    done += kk;
    if (done >= a.n) break;
    const uint32_t tag = ++exchanges;
    const size_t buf = (size_t)(tag & 1) * 8 * hw;
    for (int i = tid; i < 8 * hw; i += nth) {  // [upper / lower rows][plane][H rows]
      const int lower = i >= 4 * hw, rem = i - lower * 4 * hw, q = rem / hw;
      send_word(mine + buf + i, tag, sp[q * plane + (lower ? R * Wq : hw) + rem - q * hw]);
    }
    bool ok = true;
    auto src = [&](int i) {  // the upper neighbour's lower rows, the lower neighbour's upper rows
      const int lower = i >= 4 * hw;
      return a.xbuf + (lower ? dn : up) * per_cta + buf + (lower ? i - 4 * hw : i + 4 * hw);
    };
    recv_words<4>(tid, nth, 8 * hw, src, tag, a.limit, a.status, ok, [&](int i, uint32_t word) {
      const int lower = i >= 4 * hw, rem = i - lower * 4 * hw, q = rem / hw;
      sp[q * plane + (lower ? (H + R) * Wq : 0) + rem - q * hw] = word;
    });
    if (!__syncthreads_and(ok)) return;
  }
  // in place: both neighbours must have read their halos
  if (exchanges == 0) {
    uint32_t word;
    bool ok = true;
    if (tid < 2) ok = recv_word(a.xbuf + (tid ? dn : up) * per_cta + 16 * hw, 1u, a.limit, a.status, word);
    if (!__syncthreads_and(ok)) return;
  }
  for (int q = 0; q < 4; ++q)
    for (int i = tid; i < R * Wq; i += nth) a.planes[(size_t)q * LW + (size_t)y0 * Wq + i] = sp[q * plane + hw + i];
}

// Rows [row0, row0 + rows) of the bit planes (row q Lc + Y) -> one int8 (+-1) per site.
__global__ void __launch_bounds__(256) k_quad_unpack(const uint32_t* __restrict__ planes, QuadGeom g, long long row0,
                                                     int rows, int8_t* __restrict__ out) {
  const long long words = (long long)rows * g.Wq;
  planes += row0 * g.Wq;
  const int lane = threadIdx.x & 31;
  // one warp per word, one lane per site
  for (long long i = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; i < words;
       i += ((long long)gridDim.x * blockDim.x) >> 5) {
    const long long row = i / g.Wq;
    const int X = 32 * (int)(i - row * g.Wq) + lane;
    const uint32_t v = __ldg(&planes[i]);
    if (X < g.Lc) out[row * g.Lc + X] = (v >> lane) & 1u ? 1 : -1;
  }
}

int qfail(int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  set_last_error(buf);
  return code;
}

#define QTRY(expr)                                                                        \
  do {                                                                                    \
    cudaError_t e__ = (expr);                                                             \
    if (e__ != cudaSuccess) return qfail(ISING_ECUDA, "%s: %s", #expr, cudaGetErrorString(e__)); \
  } while (0)

int qgrid(long long items) {
  long long g = (items + 255) / 256;
  return (int)std::max(1LL, std::min(g, 152LL * 32));
}

// Classes and thresholds for one (lattice, beta, J1, J2).  The products are
// kept in volatile temporaries so that no compiler contracts them into a fused
// multiply-add: the table must round exactly as written.
bool build_table(int lattice, double beta, double J1, double J2, QuadTable* tab) {
  const int z1 = lattice == ISING_QUAD_SQUARE ? 4 : 2, z2 = lattice == ISING_QUAD_SQUARE ? 4 : 1;
  QuadTable t{};
  for (int a1 = 0; a1 <= z1; ++a1)
    for (int a2 = 0; a2 <= z2; ++a2) {
      const int c = a1 * (z2 + 1) + a2;
      volatile double p1 = 2.0 * J1 * (double)(z1 - 2 * a1);
      volatile double p2 = 2.0 * J2 * (double)(z2 - 2 * a2);
      const double dE = p1 + p2;
      if (dE <= 0.0) {
        t.always |= 1u << c;
        continue;
      }
      volatile double x = -beta * dE;
      const double f = std::floor(std::exp(x) * 4294967296.0);
      const uint32_t thr = f >= 4294967295.0 ? 0xffffffffu : (uint32_t)f;
      int d = 0;
      while (d < t.n_vals && t.val[d] != thr) ++d;
      if (d == t.n_vals) {
        if (t.n_vals == kMaxClasses) return false;
        t.val[t.n_vals++] = thr;
      }
      t.cls[d] |= 1u << c;
    }
  for (int d = 0; d < t.n_vals; ++d)
    for (int k = 0; k < 32; ++k) t.lm[d][k] = ((t.val[d] >> (31 - k)) & 1u) ? 0xffffffffu : 0u;
  *tab = t;
  return true;
}

}  // namespace
}  // namespace ising

using namespace ising;

struct ising_quad {
  int lattice = 0, Lc = 0;
  QuadGeom geom{};
  double beta = 0, J1 = 1, J2 = 0;
  QuadTable tab{};
  uint64_t seed = 0;
  uint32_t replica = 0;
  int64_t sweep = 0;
  cudaStream_t stream = nullptr;
  uint32_t* planes = nullptr;
  unsigned long long* rec = nullptr;  // ring [65536][3]
  int64_t rec_count = 0;
  int64_t launches = 0;
  int strip_G = 0, strip_K = 0;  // resident strips (G = 0: not used)
  double strip_us = 0;           // modelled time of a sweep
  unsigned long long* strip_x = nullptr;
  StripStatus strip_status;
  int8_t* spins = nullptr;       // unpacked rows for get_spins, at most kQuadUnpackBytes
};

namespace {
constexpr int64_t kQuadRec = 65536;
constexpr long long kQuadUnpackBytes = 32 << 20;
constexpr long long kQuadSpinLimit = 4000000000LL;  // ~2 s of SM clock per wait

// Strips of an Lc x Lc lattice by a time model (us per sweep, GB300): a quarter
// sweep takes 0.45 + 0.25 per resident warp of an SM sub-partition, an exchange
// 1.0; G = 0 where one CTA (the same time per quarter, no exchange) is as fast
// or the strips do not fit.
void choose_quad_strip(const QuadGeom& g, int sms, int* G_out, int* K_out, double* us_out) {
  auto quarter = [](double words) { return 0.45 + 0.25 * std::ceil(std::ceil(words / 32) / 4); };
  double best = g.Lc <= 256 ? 4 * quarter((double)g.Lc * g.Wq) : 1e30;
  *G_out = *K_out = 0;
  for (int G = 2; G <= sms && G <= g.Lc; ++G)
    for (int K = 1; K <= kQuadStripMaxK; ++K) {
      if (g.Lc / G < K + 1 || quad_strip_smem(g, G, K) > 200 * 1024) break;
      const int R = (g.Lc + G - 1) / G;
      double t = 1.0;
      for (int s = 0; s < K; ++s) t += 4 * quarter((double)(R + 2 * (K - 1 - s) + 1) * g.Wq);
      if (t / K < best) {
        best = t / K;
        *G_out = G;
        *K_out = K;
        *us_out = best;
      }
    }
}

template <int LAT, int NV>
cudaError_t launch_quad_strip(ising_quad* x, int n, int m, const RngParams& rng) {
  QuadStripArgs a{};
  a.planes = x->planes;
  a.g = x->geom;
  a.G = x->strip_G;
  a.K = std::min(x->strip_K, n);
  a.t0 = (uint32_t)x->sweep;
  a.n = n;
  a.m = m;
  a.rec = x->rec;
  a.rec0 = x->rec_count % kQuadRec;
  a.rec_cap = kQuadRec;
  a.xbuf = x->strip_x;
  a.status = x->strip_status.word();
  a.limit = x->strip_status.limit(kQuadSpinLimit);
  cudaError_t e;
  int64_t n_rec = 0;
  if (m > 0) {
    const int64_t before = x->sweep / m;
    n_rec = (x->sweep + n) / m - before;
    a.to_rec = n_rec ? (int)((before + 1) * m - x->sweep) : 0;
    const int64_t n1 = std::min<int64_t>(n_rec, kQuadRec - a.rec0);
    if (n1 > 0 && (e = cudaMemsetAsync(x->rec + 3 * a.rec0, 0, (size_t)n1 * 24, x->stream))) return e;
    if (n_rec > n1 && (e = cudaMemsetAsync(x->rec, 0, (size_t)(n_rec - n1) * 24, x->stream))) return e;
  }
  const size_t smem = quad_strip_smem(a.g, a.G, a.K);
  const void* fn = (const void*)k_quad_strip<LAT, NV>;
  static DeviceCache configured;
  if ((e = allow_dynamic_smem(fn, configured))) return e;
  const long long words = (long long)((a.g.Lc + a.G - 1) / a.G + 2 * a.K - 1) * a.g.Wq;
  const int threads = (int)std::min<long long>(kQuadStripThreads, std::max(64LL, (words + 31) / 32 * 32));
  if ((e = cudaMemsetAsync(a.xbuf, 0, quad_strip_words(a.g, a.G, a.K) * 8, x->stream))) return e;
  RngParams r = rng;
  QuadTable tab = x->tab;
  void* args[] = {&a, &r, &tab};
  if ((e = launch_strips(fn, a.G, threads, args, smem, x->strip_status.refuse, x->stream))) return e;
  ++x->launches;
  x->rec_count += n_rec;
  return cudaSuccess;
}

template <int LAT>
cudaError_t strip_dispatch(ising_quad* x, int n, int m, const RngParams& rng) {
  const int nv = x->tab.n_vals;
  if (nv <= 2) return launch_quad_strip<LAT, 2>(x, n, m, rng);
  if (nv <= 8) return launch_quad_strip<LAT, 8>(x, n, m, rng);
  if (LAT == ISING_QUAD_SQUARE) return launch_quad_strip<LAT, kMaxClasses>(x, n, m, rng);
  return cudaErrorInvalidValue;
}

template <int LAT, int NV>
cudaError_t launch_quarter(ising_quad* x, int q, uint32_t t, const RngParams& rng) {
  k_quad_quarter<LAT, NV><<<qgrid((long long)x->Lc * x->geom.Wq), 256, 0, x->stream>>>(
      x->planes, x->geom, q, t, rng, x->tab);
  return cudaGetLastError();
}

template <int LAT>
cudaError_t quarter_dispatch(ising_quad* x, int q, uint32_t t, const RngParams& rng) {
  const int nv = x->tab.n_vals;
  if (nv <= 2) return launch_quarter<LAT, 2>(x, q, t, rng);
  if (nv <= 8) return launch_quarter<LAT, 8>(x, q, t, rng);
  if (LAT == ISING_QUAD_SQUARE) return launch_quarter<LAT, kMaxClasses>(x, q, t, rng);
  return cudaErrorInvalidValue;  // the square-octagon lattice has at most 6 classes
}

constexpr int kQuadPersistMaxLc = 256;  // shared memory: 4 Lc ceil(Lc/32) words <= 32 KB

template <int LAT, int NV>
cudaError_t launch_persist(ising_quad* x, int n, int m, const RngParams& rng) {
  const long long words = (long long)x->Lc * x->geom.Wq;
  const int threads = (int)std::min<long long>(1024, ((words + 31) / 32) * 32);
  const size_t smem = (size_t)4 * words * sizeof(uint32_t);
  k_quad_persist<LAT, NV><<<1, threads, smem, x->stream>>>(x->planes, x->geom, (uint32_t)x->sweep, n, m, rng,
                                                           x->tab, x->rec, x->rec_count, kQuadRec);
  return cudaGetLastError();
}

template <int LAT>
cudaError_t persist_dispatch(ising_quad* x, int n, int m, const RngParams& rng) {
  const int nv = x->tab.n_vals;
  if (nv <= 2) return launch_persist<LAT, 2>(x, n, m, rng);
  if (nv <= 8) return launch_persist<LAT, 8>(x, n, m, rng);
  if (LAT == ISING_QUAD_SQUARE) return launch_persist<LAT, kMaxClasses>(x, n, m, rng);
  return cudaErrorInvalidValue;
}

// Calls of few sweeps that one CTA finishes before strips, which are launched cooperatively and
// clear their exchange buffer first.  us per call, strips / one CTA: one sweep, 4.8.8 Lc = 65 10.3 / 8.3, 128 12.3 /
// 10.1, 129 11.3 / 12.3; square J2 = 0 66 11.7 / 8.3, 128 14.3 / 12.3, 129 11.4 / 16.2; J2 = 0.5 66 16.0 / 12.3, 96 14.4 / 14.4, 97 14.4 /
// 18.4; two sweeps, in the same order, 84 12.4 / 10.3, 14.6 / 14.4, 22.7 / 20.5, 89 12.3 / 12.4, 14.5 / 16.5, 22.6 /
// 26.6; three at 76 15.9 / 14.4, 19.9 / 18.5, 32.3 / 28.7; five 20.5 / 20.5, 28.3 / 28.0, 47.1 / 44.8, 20 strips from 65 on.
bool quad_one_cta(const ising_quad* x, int n) {
  const bool more_classes = x->tab.n_vals > 2;
  if (n > (more_classes ? 5 : 3)) return false;
  return x->Lc < (n > 1 ? 88 : more_classes && x->lattice == ISING_QUAD_SQUARE ? 97 : 129);
}

cudaError_t quad_sweeps(ising_quad* x, int n, int m) {
  const RngParams rng = make_rng(x->seed, x->replica, 0, 0);
  if (x->strip_G > 0 && n > 0 && !quad_one_cta(x, n)) {
    // chunks whose records fit the ring, of about 20 ms
    const int launch = strip_launch_sweeps(x->strip_us);
    const int most = m > 0 ? (int)std::min<int64_t>(kQuadRec * (int64_t)m, launch) : launch;
    cudaError_t e = cudaSuccess;
    int done = 0;
    for (; done < n && !e;) {
      const int k = std::min(most, n - done);
      e = x->lattice == ISING_QUAD_SQUARE ? strip_dispatch<ISING_QUAD_SQUARE>(x, k, m, rng)
                                          : strip_dispatch<ISING_QUAD_SQOCT>(x, k, m, rng);
      if (strips_refused(e)) {
        x->strip_G = 0;
        e = quad_sweeps(x, n - done, m);
        break;
      }
      x->sweep += k;
      done += k;
    }
    x->sweep -= done;  // the caller advances the counter
    return e;
  }
  if (x->Lc <= kQuadPersistMaxLc && n > 0) {
    cudaError_t e = x->lattice == ISING_QUAD_SQUARE ? persist_dispatch<ISING_QUAD_SQUARE>(x, n, m, rng)
                                                    : persist_dispatch<ISING_QUAD_SQOCT>(x, n, m, rng);
    if (e) return e;
    ++x->launches;
    if (m > 0)
      for (int s = 0; s < n; ++s)
        if ((x->sweep + s + 1) % m == 0) ++x->rec_count;
    return cudaSuccess;
  }
  for (int s = 0; s < n; ++s) {
    const uint32_t t = (uint32_t)(x->sweep + s);
    for (int q = 0; q < 4; ++q) {
      cudaError_t e = x->lattice == ISING_QUAD_SQUARE ? quarter_dispatch<ISING_QUAD_SQUARE>(x, q, t, rng)
                                                      : quarter_dispatch<ISING_QUAD_SQOCT>(x, q, t, rng);
      if (e) return e;
      ++x->launches;
    }
    if (m > 0 && ((int64_t)t + 1) % m == 0) {
      unsigned long long* slot = x->rec + 3 * (x->rec_count % kQuadRec);
      cudaError_t e = cudaMemsetAsync(slot, 0, 3 * sizeof(unsigned long long), x->stream);
      if (e) return e;
      const int grid = qgrid(4LL * x->Lc * x->geom.Wq);
      if (x->lattice == ISING_QUAD_SQUARE)
        k_quad_measure<ISING_QUAD_SQUARE><<<grid, 256, 0, x->stream>>>(x->planes, x->geom, slot);
      else
        k_quad_measure<ISING_QUAD_SQOCT><<<grid, 256, 0, x->stream>>>(x->planes, x->geom, slot);
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

int ising_quad_create(ising_quad** out, int lattice, int Lc, double beta, double J1, double J2,
                      void* stream) {
  if (!out) return qfail(ISING_EINVAL, "null output pointer");
  *out = nullptr;
  if (lattice != ISING_QUAD_SQUARE && lattice != ISING_QUAD_SQOCT)
    return qfail(ISING_EINVAL, "unknown lattice %d", lattice);
  if (Lc < 2 || Lc > 16384) return qfail(ISING_EINVAL, "Lc must be in [2, 16384] (got %d)", Lc);
  if (!std::isfinite(beta) || beta <= 0) return qfail(ISING_EINVAL, "beta must be finite and > 0");
  if (!std::isfinite(J1) || !std::isfinite(J2)) return qfail(ISING_EINVAL, "couplings must be finite");
  ising_quad* x = new (std::nothrow) ising_quad();
  if (!x) return qfail(ISING_ENOMEM, "host allocation failed");
  x->lattice = lattice;
  x->Lc = Lc;
  x->geom.Lc = Lc;
  x->geom.Wq = (Lc + 31) / 32;
  x->geom.nlast = Lc - 32 * (x->geom.Wq - 1);
  x->geom.fw = make_fastdiv((uint32_t)x->geom.Wq);
  x->beta = beta;
  x->J1 = J1;
  x->J2 = J2;
  x->stream = (cudaStream_t)stream;
  if (!build_table(lattice, beta, J1, J2, &x->tab)) {
    delete x;
    return qfail(ISING_EINTERNAL, "threshold table overflow");
  }
  const size_t bytes = (size_t)4 * Lc * x->geom.Wq * sizeof(uint32_t);
  int dev = 0, sms = 0;
  size_t strip_words = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (!e) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (!e) choose_quad_strip(x->geom, sms, &x->strip_G, &x->strip_K, &x->strip_us);
  if (!e && x->strip_G > 0) {
    strip_words = quad_strip_words(x->geom, x->strip_G, x->strip_K);
    e = x->strip_status.ensure();
  }
  // one allocation: each that starts a 2 MB page of its own takes 80 us
  const size_t at_rec = (bytes + 255) / 256 * 256, at_x = at_rec + kQuadRec * 3 * sizeof(unsigned long long);
  if (!e) e = cudaMalloc((void**)&x->planes, at_x + strip_words * sizeof(unsigned long long));
  if (!e) {
    x->rec = (unsigned long long*)((char*)x->planes + at_rec);
    if (strip_words) x->strip_x = (unsigned long long*)((char*)x->planes + at_x);
  }
  if (e) {
    cudaGetLastError();
    x->strip_status.release();
    cudaFree(x->planes);
    delete x;
    return qfail(ISING_ENOMEM, "quad allocation: %s", cudaGetErrorString(e));
  }
  *out = x;
  return ising_quad_seed(x, 0);
}

int ising_quad_seed(ising_quad* x, uint64_t seed) {
  if (!x) return qfail(ISING_EINVAL, "null context");
  x->seed = seed;
  x->sweep = 0;
  x->rec_count = 0;
  QTRY(x->strip_status.begin(x->stream));
  const RngParams rng = make_rng(seed, x->replica, 0, 0);
  k_quad_init<<<qgrid(4LL * x->Lc * x->geom.Wq), 256, 0, x->stream>>>(x->planes, x->geom, rng);
  QTRY(cudaGetLastError());
  set_last_error("");
  return ISING_OK;
}

int ising_quad_set_replica(ising_quad* x, uint32_t replica) {
  if (!x) return qfail(ISING_EINVAL, "null context");
  x->replica = replica;
  return ising_quad_seed(x, x->seed);
}

int ising_quad_sweep(ising_quad* x, int n_sweeps, int measure_every) {
  if (!x) return qfail(ISING_EINVAL, "null context");
  if (n_sweeps < 0 || measure_every < 0) return qfail(ISING_EINVAL, "negative count");
  if (x->sweep + n_sweeps >= ((int64_t)1 << 32)) return qfail(ISING_EINVAL, "sweep counter overflow");
  NvtxRange nvtx("ising_quad_sweep");
  QTRY(quad_sweeps(x, n_sweeps, measure_every));
  x->sweep += n_sweeps;
  set_last_error("");
  return ISING_OK;
}

// After a synchronising call: ETIMEOUT if a strip's wait gave up (until the lattice is set again).
static int quad_status(ising_quad* x) {
  if (x->strip_status.failed())
    return qfail(ISING_ETIMEOUT, "a strip's wait for its neighbour timed out");
  return ISING_OK;
}

int ising_quad_series(ising_quad* x, int64_t* B1, int64_t* B2, int64_t* M, int n) {
  if (!x) return qfail(ISING_EINVAL, "null context");
  if (n < 0 || n > std::min<int64_t>(x->rec_count, kQuadRec)) return qfail(ISING_EINVAL, "n exceeds records");
  std::vector<unsigned long long> h((size_t)3 * n);
  const int64_t s0 = (x->rec_count - n) % kQuadRec, n1 = std::min<int64_t>(n, kQuadRec - s0);
  if (n1 > 0) QTRY(cudaMemcpyAsync(h.data(), x->rec + 3 * s0, (size_t)n1 * 24, cudaMemcpyDeviceToHost, x->stream));
  if (n > n1)
    QTRY(cudaMemcpyAsync(h.data() + 3 * n1, x->rec, (size_t)(n - n1) * 24, cudaMemcpyDeviceToHost, x->stream));
  QTRY(cudaStreamSynchronize(x->stream));
  if (int st = quad_status(x)) return st;
  for (int i = 0; i < n; ++i) {
    if (B1) B1[i] = (int64_t)h[3 * i] / 2;
    if (B2) B2[i] = (int64_t)h[3 * i + 1] / 2;
    if (M) M[i] = (int64_t)h[3 * i + 2];
  }
  set_last_error("");
  return ISING_OK;
}

int ising_quad_get_spins(ising_quad* x, int8_t* host_out) {
  if (!x || !host_out) return qfail(ISING_EINVAL, "null argument");
  const int Lc = x->Lc, Wq = x->geom.Wq;
  const long long rows = 4LL * Lc, most = std::min(rows, std::max(1LL, kQuadUnpackBytes / Lc));
  if (Lc <= 48) {
    // unpacked here: a launch and a copy after it take longer (us, Lc = 8 11.5 / 16.8, 32 13.6 / 17.5, 64
    // 20.2 / 17.7, 1024 1800 / 119)
    std::vector<uint32_t> h((size_t)rows * Wq);
    QTRY(cudaMemcpyAsync(h.data(), x->planes, h.size() * 4, cudaMemcpyDeviceToHost, x->stream));
    QTRY(cudaStreamSynchronize(x->stream));
    for (long long r = 0; r < rows; ++r)
      for (int X = 0; X < Lc; ++X) host_out[r * Lc + X] = (h[r * Wq + (X >> 5)] >> (X & 31)) & 1u ? 1 : -1;
  } else {
    // through a buffer that the context keeps, so many rows at a time
    if (!x->spins) QTRY(cudaMalloc((void**)&x->spins, most * Lc));
    for (long long r0 = 0; r0 < rows; r0 += most) {
      const int n = (int)std::min(most, rows - r0);
      k_quad_unpack<<<qgrid((long long)n * Wq * 32), 256, 0, x->stream>>>(x->planes, x->geom, r0, n, x->spins);
      QTRY(cudaGetLastError());
      QTRY(cudaMemcpyAsync(host_out + r0 * Lc, x->spins, (size_t)n * Lc, cudaMemcpyDeviceToHost, x->stream));
    }
    QTRY(cudaStreamSynchronize(x->stream));
  }
  if (int st = quad_status(x)) return st;
  set_last_error("");
  return ISING_OK;
}

int ising_quad_set_spins(ising_quad* x, const int8_t* host_in) {
  if (!x || !host_in) return qfail(ISING_EINVAL, "null argument");
  const int Lc = x->Lc, Wq = x->geom.Wq;
  std::vector<uint32_t> h((size_t)4 * Lc * Wq, 0u);
  for (int q = 0; q < 4; ++q)
    for (int Y = 0; Y < Lc; ++Y)
      for (int X = 0; X < Lc; ++X) {
        const int8_t v = host_in[((size_t)q * Lc + Y) * Lc + X];
        if (v != 1 && v != -1) return qfail(ISING_EINVAL, "spins must be +1 or -1");
        if (v == 1) h[((size_t)q * Lc + Y) * Wq + (X >> 5)] |= 1u << (X & 31);
      }
  QTRY(x->strip_status.begin(x->stream));
  QTRY(cudaMemcpyAsync(x->planes, h.data(), h.size() * 4, cudaMemcpyHostToDevice, x->stream));
  QTRY(cudaStreamSynchronize(x->stream));
  set_last_error("");
  return ISING_OK;
}

int ising_quad_launch_count(ising_quad* x, int64_t* count) {
  if (!x || !count) return qfail(ISING_EINVAL, "null argument");
  *count = x->launches;
  return ISING_OK;
}

int ising_quad_destroy(ising_quad* x) {
  if (!x) return ISING_OK;
  cudaStreamSynchronize(x->stream);
  cudaFree(x->planes);
  x->strip_status.release();
  cudaFree(x->spins);
  delete x;
  return ISING_OK;
}

}  // extern "C"
