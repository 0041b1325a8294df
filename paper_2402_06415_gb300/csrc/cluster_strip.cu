// Cluster steps (Swendsen-Wang and Wolff) on resident row strips: all steps of a
// call in one cooperative launch, one CTA per SM owning R full rows in shared
// memory.  Same bonds, seeds, coins and therefore the same configurations as
// sw.cu, wolff.cu and cluster_persist.cu.  One step:
//   1. bond draws (one Philox block per site pair) and horizontal runs: a warp
//      takes 64 consecutive sites of a row and labels each with the first site of
//      its run by two ballots and a count of leading zeros;
//   2. vertical bonds, bonds between 64-site blocks and wrap bonds unite labels in
//      shared memory (links from the larger to the smaller index), then every
//      site stores its root;
//   3. the roots that touch the strip's first or last row enter a forest in global
//      memory (two forests used in turn, so that the next step may fill one while
//      others still read this one); grid barrier; bonds to the next strip's first
//      row unite roots there; grid barrier;
//   4. each local root walks to its global root m (the cluster's smallest site)
//      and takes its coin (SW) or compares it with the seed's root (Wolff); sites
//      flip by their local root's verdict;
//   5. the first row goes to the previous strip as (tag, word) pairs.
// Only boundary bonds pay L2 round trips; with every bond and label in global memory
// (cluster_persist.cu) each site did.  Bound by the two grid barriers (~1.3 us each), the
// dependent walks of the boundary forest and, for long strips, the shared-memory
// unions: three of four warp cycles are spent at a barrier behind them (L = 256), no pipe is
// above 8 %.  At beta 0.2 to 1.0 it is as far ahead of the forms before as at beta_c.  us per SW step at beta_c, before (cluster_persist.cu up to L = 766, then
// sw.cu) and now: L = 128 28 -> 13, 256 34 -> 19, 512 71 -> 27, 1024 134 -> 51.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "ising_device.cuh"

namespace ising {
namespace {

constexpr uint32_t kTagSWBond = 10, kTagSWFlip = 11, kTagWolffSeed = 16, kTagWolffBond = 17;
constexpr int kThreads = 1024;
constexpr int kSolveMaxL = 160;

struct ClusterStripArgs {
  uint32_t* planes;
  int L, Wc, G;
  uint32_t step0;
  int n, m, to_rec;
  uint32_t thr;
  unsigned long long* rec;
  long long rec0, rec_cap;
  uint32_t* forest;   // 2 x L * L
  uint32_t* row_root; // G x L: global root of every site of a strip's first row
  uint32_t* seed_root;  // 2
  uint32_t* edges;      // G x L packed pairs of roots (SOLVE)
  // zeroed by the launcher: G x 2 x ceil(L / 32) boundary pairs, G barrier flags, 4 edge counters
  unsigned long long* xbuf;
  unsigned int* flags;
  unsigned int* n_edges;
  WolffCtl* wctl;
  int* status;
  long long limit;
  FastDiv fL;
};

__device__ __forceinline__ uint32_t groot_ro(const uint32_t* parent, uint32_t a) {
  while (true) {
    const uint32_t p = __ldcg(&parent[a]);
    if (p == a) return a;
    a = p;
  }
}
// Unions walk both trees in step (two loads in flight: 22 -> 19 us per step at L = 256,
// 56 -> 51 at 1024) with path halving, which stores only ancestors, and link the larger
// root below the smaller.
__device__ __forceinline__ void gunite(uint32_t* parent, uint32_t a, uint32_t b) {
  while (true) {
    uint32_t pa = __ldcg(&parent[a]), pb = __ldcg(&parent[b]);
    while (pa != a || pb != b) {
      if (pa == pb) return;
      const uint32_t ga = __ldcg(&parent[pa]), gb = __ldcg(&parent[pb]);
      if (ga != pa) __stcg(&parent[a], ga);
      if (gb != pb) __stcg(&parent[b], gb);
      a = ga;
      b = gb;
      pa = __ldcg(&parent[a]);
      pb = __ldcg(&parent[b]);
    }
    if (a == b) return;
    if (a < b) {
      const uint32_t t = a;
      a = b;
      b = t;
    }
    const uint32_t old = atomicCAS(&parent[a], a, b);
    if (old == a) return;
    a = old;
  }
}
__device__ __forceinline__ void lunite(uint32_t* lab, uint32_t a, uint32_t b) {
  volatile uint32_t* v = lab;
  while (true) {
    uint32_t pa = v[a], pb = v[b];
    while (pa != a || pb != b) {
      if (pa == pb) return;
      const uint32_t ga = v[pa], gb = v[pb];
      if (ga != pa) v[a] = ga;
      if (gb != pb) v[b] = gb;
      a = ga;
      b = gb;
      pa = v[a];
      pb = v[b];
    }
    if (a == b) return;
    if (a < b) {
      const uint32_t t = a;
      a = b;
      b = t;
    }
    const uint32_t old = atomicCAS(&lab[a], a, b);
    if (old == a) return;
    a = old;
  }
}
__device__ __forceinline__ uint32_t sroot16(uint16_t* par, uint32_t a) {
  volatile uint16_t* v = par;
  while (true) {
    const uint32_t p = v[a];
    if (p == a) return a;
    const uint32_t gp = v[p];
    if (gp != p) v[a] = (uint16_t)gp;
    a = gp;
  }
}
__device__ __forceinline__ void sunite16(uint16_t* par, uint32_t a, uint32_t b) {
  while (true) {
    a = sroot16(par, a);
    b = sroot16(par, b);
    if (a == b) return;
    if (a < b) {
      const uint32_t t = a;
      a = b;
      b = t;
    }
    const uint32_t old = atomicCAS(reinterpret_cast<unsigned short*>(&par[a]), (unsigned short)a, (unsigned short)b);
    if (old == a) return;
    a = old;
  }
}

// Grid barrier of up to kThreads CTAs, all resident: every CTA raises its flag and
// polls everybody's, one thread per CTA, so it takes one store and one load through
// L2 instead of an atomic, its answer and a load.  False after `limit` cycles
// (and *status = 1).
__device__ __forceinline__ bool flag_barrier(unsigned int* flags, int G, unsigned int epoch, long long limit,
                                             int* status) {
  __syncthreads();
  const int tid = threadIdx.x;
  if (tid == 0) {
    __threadfence();
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(flags + blockIdx.x), "r"(epoch) : "memory");
  }
  bool ok = true;
  if (tid < G) {
    const long long start = clock64();
    while (ld_acquire_gpu(flags + tid) < epoch) {
      if (clock64() - start > limit) {
        *reinterpret_cast<volatile int*>(status) = 1;
        ok = false;
        break;
      }
    }
  }
  return __syncthreads_and(ok) != 0;
}

// st[] per site: bit 0 spin, 1 bond to x + 1, 2 bond to y + 1, 3 root of a cluster
// that touches the strip's first or last row, 4 verdict of a root (flip)
// SOLVE (up to 160 x 160 sites): after the first barrier every CTA lists the pairs of
// roots its boundary bonds join, and after the second every CTA solves all of them in
// a 16-bit forest of its own in shared memory, where a hop costs 30 cycles and not 700.
// Beyond, the thousands of pairs that every CTA repeats cost more than the global
// forest (L = 256: 24 us at best against 21).  Two other forms measured slower there:
// the pairs taken level by level of a binary tree over the strips (29 us), and the
// global forest linked in a pseudo-random order of the sites, which needs a third
// barrier for each cluster's smallest site (28 us).
template <bool WOLFF, bool SOLVE>
__global__ void __launch_bounds__(kThreads) k_cluster_strip(ClusterStripArgs a, RngParams rng) {
  extern __shared__ uint32_t cs_smem[];
  __shared__ uint32_t s_seed, s_count, s_ne, s_base;
  __shared__ uint32_t s_edges[SOLVE ? kSolveMaxL : 1];  // this strip's pairs
  const int L = a.L, G = a.G, b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kThreads / 32;
  const int y0 = (int)((long long)b * L / G), R = (int)((long long)(b + 1) * L / G) - y0;
  const uint32_t n_own = (uint32_t)R * (uint32_t)L, g0 = (uint32_t)y0 * (uint32_t)L;
  uint32_t* const lab = cs_smem;
  uint8_t* const st = reinterpret_cast<uint8_t*>(lab + (size_t)((L + G - 1) / G) * L);  // R + 1 rows
  uint16_t* const par = reinterpret_cast<uint16_t*>(
      reinterpret_cast<unsigned char*>(cs_smem) + (((size_t)((L + G - 1) / G) * L * 5 + L + 15) & ~(size_t)15));
  const int blocks_x = (L + 63) / 64, words_x = (L + 31) / 32;
  const int next = b == G - 1 ? 0 : b + 1;
  const uint32_t bond_tag = WOLFF ? kTagWolffBond : kTagSWBond;
  const size_t N = (size_t)L * (size_t)L;
  // spins of the own rows and of the next strip's first row
  for (uint32_t i = tid; i < n_own + L; i += kThreads) {
    const uint32_t r = fdiv(i, a.fL), x = i - r * (uint32_t)L;
    const uint32_t y = y0 + r >= (uint32_t)L ? y0 + r - L : y0 + r;
    const uint32_t c = (x + y) & 1u, j = x >> 1;
    st[i] = (uint8_t)((__ldcg(&a.planes[(size_t)c * L * a.Wc + (size_t)y * a.Wc + (j >> 5)]) >> (j & 31)) & 1u);
  }
  // nobody writes the planes before everyone has read them: the first step's barriers
  __syncthreads();
  int to_rec = a.to_rec;
  long long slot = a.rec0;
  unsigned int epoch = 0;
  for (int s = 0; s < a.n; ++s) {
    const uint32_t t = a.step0 + (uint32_t)s;
    uint32_t* const forest = SOLVE ? nullptr : a.forest + (s & 1) * N;
    // ---- 1. bonds and runs, one warp per 64 sites of a row (lane: sites 2 lane, 2 lane + 1) ----
    for (int k = warp; k < R * blocks_x; k += kWarps) {
      const int r = k / blocks_x, x = 64 * (k - r * blocks_x) + 2 * lane;
      const bool in = x < L;  // L is even: a pair is whole
      const uint32_t li = (uint32_t)r * (uint32_t)L + (uint32_t)(in ? x : 0);
      bool h0 = false, h1 = false;
      if (in) {
        const uint4 w = philox10_rk(make_uint4((g0 + li) >> 1, t, rng.replica, bond_tag << 16), rng.rk0, rng.rk1);
        const uint32_t s0 = st[li] & 1u, s1 = st[li + 1] & 1u;
        const uint32_t s2 = st[x + 2 == L ? li + 2 - (uint32_t)L : li + 2] & 1u;
        const uint32_t d0 = st[li + L] & 1u, d1 = st[li + L + 1] & 1u;
        h0 = w.x < a.thr && s0 == s1;
        h1 = w.z < a.thr && s1 == s2;
        const bool v0 = w.y < a.thr && s0 == d0, v1 = w.w < a.thr && s1 == d1;
        st[li] = (uint8_t)(s0 | (h0 ? 2u : 0u) | (v0 ? 4u : 0u));
        st[li + 1] = (uint8_t)(s1 | (h1 ? 2u : 0u) | (v1 ? 4u : 0u));
      }
      // sites that start a run: even ones without a bond from the previous pair, odd ones without h0
      const uint32_t even = ~(__ballot_sync(0xffffffffu, h1) << 1), odd = ~__ballot_sync(0xffffffffu, h0);
      if (in) {
        const uint32_t le = 0xffffffffu >> (31 - lane), lt = le >> 1;
        const int se = 2 * (31 - __clz((int)(even & le)));  // even bit 0 is always set
        const uint32_t ob = odd & lt;
        const int so = ob ? 2 * (31 - __clz((int)ob)) + 1 : -1;
        const int start = max(se, so);
        const uint32_t row0 = li - 2u * (uint32_t)lane;  // first site of the 64
        lab[li] = row0 + (uint32_t)start;
        lab[li + 1] = h0 ? row0 + (uint32_t)start : li + 1;
      }
    }
    __syncthreads();
    // ---- 2. unions inside the strip ----
    for (uint32_t i = tid; i < n_own; i += kThreads) {
      const uint32_t v = st[i];
      if (!(v & 6u)) continue;
      const uint32_t r = fdiv(i, a.fL), x = i - r * (uint32_t)L;
      if ((v & 4u) && r + 1 < (uint32_t)R) {
        // skipped if the left neighbour's vertical bond already joined the same two runs
        const bool skip = x > 0 && (st[i - 1] & 6u) == 6u && (st[i - 1 + L] & 2u);
        if (!skip) lunite(lab, i, i + L);
      }
      if (v & 2u) {
        if (x + 1 == (uint32_t)L) lunite(lab, i, i - x);
        else if ((x & 63u) == 63u) lunite(lab, i, i + 1);
      }
    }
    __syncthreads();
    for (uint32_t i = tid; i < n_own; i += kThreads) {
      // read-only walk: a halving store could overwrite a site's root with an ancestor
      volatile uint32_t* v = lab;
      uint32_t p = i;
      while (v[p] != p) p = v[p];
      v[i] = p;
    }
    __syncthreads();
    // ---- 3. the forest of the roots that touch the strip's first or last row ----
    for (uint32_t x = tid; x < (uint32_t)L; x += kThreads) {
      const uint32_t top = lab[x], bot = lab[n_own - L + x];
      st[top] |= 8u;  // several threads store the same byte
      st[bot] |= 8u;
      if (!SOLVE) {
        __stcg(&forest[g0 + top], g0 + top);
        __stcg(&forest[g0 + bot], g0 + bot);
      } else {
        par[g0 + top] = (uint16_t)(g0 + top);
        par[g0 + bot] = (uint16_t)(g0 + bot);
      }
      __stcg(&a.row_root[(size_t)b * L + x], g0 + top);
    }
    uint32_t seed = 0;
    if (WOLFF && tid == 0) {
      seed = __umulhi(philox10_rk(make_uint4(0u, t, rng.replica, kTagWolffSeed << 16), rng.rk0, rng.rk1).x, (uint32_t)N);
      if (seed >= g0 && seed - g0 < n_own) {
        const uint32_t r = g0 + lab[seed - g0];
        if (!SOLVE) __stcg(&forest[r], r);
        __stcg(&a.seed_root[s & 1], r);
        a.wctl->seed_site = seed;
      }
    }
    if (tid == 0) {
      s_count = 0;
      s_ne = 0;
    }
    if (!flag_barrier(a.flags, G, ++epoch, a.limit, a.status)) return;
    // between the barriers nobody adds to the last step's count or to this one's
    if (WOLFF && b == 0 && tid == 0) a.wctl->last_size = 0;
    // the counter of the next step: last read two steps ago
    if (SOLVE && b == 0 && tid == 0) a.n_edges[(s + 1) % 3] = 0;
    for (uint32_t x = tid; x < (uint32_t)L; x += kThreads) {
      const uint32_t i = n_own - L + x;
      if (!(st[i] & 4u)) continue;
      const uint32_t other = __ldcg(&a.row_root[(size_t)next * L + x]);
      // skipped if the left neighbour's bond joins the same two clusters
      if (x > 0 && (st[i - 1] & 4u) && lab[i - 1] == lab[i] && __ldcg(&a.row_root[(size_t)next * L + x - 1]) == other)
        continue;
      if (SOLVE)
        s_edges[atomicAdd(&s_ne, 1u)] = (g0 + lab[i]) | (other << 16);
      else
        gunite(forest, g0 + lab[i], other);
    }
    if (SOLVE) {
      __syncthreads();
      if (tid == 0) s_base = atomicAdd(&a.n_edges[s % 3], s_ne);
      __syncthreads();
      for (uint32_t e = tid; e < s_ne; e += kThreads) __stcg(&a.edges[s_base + e], s_edges[e]);
    }
    if (!flag_barrier(a.flags, G, ++epoch, a.limit, a.status)) return;
    if (SOLVE) {
      const uint32_t total = __ldcg(&a.n_edges[s % 3]);
      for (uint32_t e = tid; e < total; e += kThreads) {  // the roots of every pair start as their own parents
        const uint32_t uv = __ldcg(&a.edges[e]);
        par[uv & 0xffffu] = (uint16_t)(uv & 0xffffu);
        par[uv >> 16] = (uint16_t)(uv >> 16);
      }
      if (WOLFF && tid == 0) {  // the seed's root may touch no boundary
        const uint32_t r = __ldcg(&a.seed_root[s & 1]);
        par[r] = (uint16_t)r;
      }
      __syncthreads();
      for (uint32_t e = tid; e < total; e += kThreads) {
        const uint32_t uv = __ldcg(&a.edges[e]);
        sunite16(par, uv & 0xffffu, uv >> 16);
      }
      __syncthreads();
    }
    // ---- 4. verdicts of the local roots, then flips ----
    if (WOLFF) {
      if (tid == 0) {
        const uint32_t r = __ldcg(&a.seed_root[s & 1]);
        s_seed = SOLVE ? sroot16(par, r) : groot_ro(forest, r);
      }
      __syncthreads();
    }
    for (uint32_t i = tid; i < n_own; i += kThreads) {
      if (lab[i] != i) continue;
      const uint32_t v = st[i];
      const uint32_t m = v & 8u ? (SOLVE ? sroot16(par, g0 + i) : groot_ro(forest, g0 + i)) : g0 + i;
      bool f;
      if (WOLFF) {
        f = m == s_seed;
      } else {
        const uint4 w = philox10_rk(make_uint4(m >> 2, t, rng.replica, kTagSWFlip << 16), rng.rk0, rng.rk1);
        const uint32_t q = m & 3u;
        f = ((q == 0 ? w.x : q == 1 ? w.y : q == 2 ? w.z : w.w) >> 31) != 0;
      }
      if (f) st[i] = (uint8_t)(v | 16u);
    }
    __syncthreads();
    uint32_t count = 0;
    for (uint32_t i = tid; i < n_own; i += kThreads)
      if (st[lab[i]] & 16u) {
        st[i] ^= 1u;  // the owner's byte; others read only its bit 4
        ++count;
      }
    if (WOLFF) {
      count = __reduce_add_sync(0xffffffffu, count);
      if (lane == 0 && count) atomicAdd(&s_count, count);
    }
    __syncthreads();
    if (WOLFF && tid == 0) {
      if (s_count) {
        atomicAdd(&a.wctl->last_size, s_count);
        atomicAdd(&a.wctl->flipped, (unsigned long long)s_count);
      }
      if (b == 0) {
        a.wctl->labelled += 1;
        a.wctl->need_label = 0;
      }
    }
    // ---- 5. first row to the previous strip ----
    const bool meas = to_rec == 1;
    if (s + 1 < a.n || meas) {
      const uint32_t tag = (uint32_t)s + 1u;
      const size_t half = (size_t)(s & 1) * words_x;
      for (int w = warp; w < words_x; w += kWarps) {
        const int x = 32 * w + lane;
        const uint32_t bits = __ballot_sync(0xffffffffu, x < L && (st[x] & 1u));
        if (lane == 0) send_word(a.xbuf + (size_t)b * 2 * words_x + half + w, tag, bits);
      }
      bool ok = true;
      for (int w = warp; w < words_x; w += kWarps) {
        uint32_t bits = 0;
        ok = ok && recv_word(a.xbuf + (size_t)next * 2 * words_x + half + w, tag, a.limit, a.status, bits);
        const int x = 32 * w + lane;
        if (x < L) st[n_own + x] = (uint8_t)((bits >> lane) & 1u);
      }
      if (!__syncthreads_and(ok)) return;
    }
    if (meas) {
      unsigned int anti = 0, ones = 0;
      for (uint32_t i = tid; i < n_own; i += kThreads) {
        const uint32_t r = fdiv(i, a.fL), x = i - r * (uint32_t)L;
        const uint32_t v = st[i] & 1u;
        anti += (v ^ (st[x + 1 == (uint32_t)L ? i - x : i + 1] & 1u)) + (v ^ (st[i + L] & 1u));
        ones += v;
      }
      anti = __reduce_add_sync(0xffffffffu, anti);
      ones = __reduce_add_sync(0xffffffffu, ones);
      if (lane == 0 && (anti | ones)) {
        atomicAdd(&a.rec[2 * slot], (unsigned long long)anti);
        atomicAdd(&a.rec[2 * slot + 1], (unsigned long long)ones);
      }
      __syncthreads();
    }
    if (to_rec > 0 && --to_rec == 0) {
      to_rec = a.m;
      slot = slot + 1 == a.rec_cap ? 0 : slot + 1;
    }
  }
  // write the own rows back: one thread per packed word
  const int n = L / 2;
  for (int i = tid; i < 2 * R * a.Wc; i += kThreads) {
    const int c = i / (R * a.Wc), rem = i - c * R * a.Wc, r = rem / a.Wc, w = rem - r * a.Wc, y = y0 + r;
    uint32_t word = 0;
    for (int k = 0; k < 32 && 32 * w + k < n; ++k)
      word |= (uint32_t)(st[(uint32_t)r * L + 2 * (32 * w + k) + ((y + c) & 1)] & 1u) << k;
    a.planes[(size_t)c * L * a.Wc + (size_t)y * a.Wc + w] = word;
  }
}

bool solves(int L) { return L <= kSolveMaxL; }

size_t strip_smem(int L, int G) {
  const size_t R = (size_t)(L + G - 1) / G;
  return ((R * L * 5 + L + 15) & ~(size_t)15) + (solves(L) ? 2 * (size_t)L * L : 0);
}
size_t zeroed_bytes(int L, int G) {  // boundary pairs, barrier flags, edge counters
  return (size_t)G * 2 * ((L + 31) / 32) * 8 + ((size_t)G + 5) / 2 * 8;
}

}  // namespace

// Number of strips: more of them shorten the work inside a strip and lengthen the
// boundary forest.  us per SW step at beta_c for 16 / 32 / 64 / 152 strips: L = 128 (SOLVE)
// 12.9 / 16.0 / 22.7 / -, 256 28.9 / 20.3 / 18.8 / 22.4 (128), 384 52 / 34 / 24.4 / 24.4, 512 82 / 50 /
// 32 / 27, 1024 - / 151 / 88 / 51.
int cluster_strip_grid(int L, int sms) {
  const int want = solves(L) ? 16 : L < 448 ? std::min(64, L / 4) : sms;
  const int G = std::min(std::min(want, sms), std::min(L / 2, kThreads));
  return G >= 2 && strip_smem(L, G) <= 200 * 1024 ? G : 0;
}

size_t cluster_strip_bytes(int L, int G) {
  const size_t words = (solves(L) ? (size_t)G * L : 2 * (size_t)L * L) + (size_t)G * L + 2;
  return (words + 1) / 2 * 8 + zeroed_bytes(L, G);
}

cudaError_t launch_cluster_strip(const BitsLattice& lat, bool wolff, uint32_t step0, int n_steps, int measure_every,
                                 int to_rec, uint32_t thr, const RngParams& rng, int G, void* scratch,
                                 unsigned long long* rec, long long rec0, long long rec_cap, WolffCtl* wctl,
                                 const StripStatus& status, cudaStream_t s) {
  ClusterStripArgs a{};
  a.planes = lat.planes;
  a.L = lat.L;
  a.Wc = lat.Wc;
  a.G = G;
  a.step0 = step0;
  a.n = n_steps;
  a.m = measure_every;
  a.to_rec = to_rec;
  a.thr = thr;
  a.rec = rec;
  a.rec0 = rec0;
  a.rec_cap = rec_cap;
  const bool solve = solves(a.L);
  a.forest = a.edges = (uint32_t*)scratch;
  a.row_root = a.forest + (solve ? (size_t)G * a.L : 2 * (size_t)a.L * a.L);
  a.seed_root = a.row_root + (size_t)G * a.L;
  const size_t xwords = (size_t)G * 2 * ((a.L + 31) / 32), zeroed = zeroed_bytes(a.L, G);
  a.xbuf = (unsigned long long*)((char*)scratch + cluster_strip_bytes(a.L, G) - zeroed);
  a.flags = (unsigned int*)(a.xbuf + xwords);
  a.n_edges = a.flags + G;
  a.wctl = wctl;
  a.status = status.word();
  a.limit = status.limit(kClusterSpinLimit);
  a.fL = make_fastdiv((uint32_t)a.L);
  const size_t smem = strip_smem(a.L, G);
  const void* fns[4] = {(const void*)k_cluster_strip<false, false>, (const void*)k_cluster_strip<true, false>,
                        (const void*)k_cluster_strip<false, true>, (const void*)k_cluster_strip<true, true>};
  const int which = (wolff ? 1 : 0) + (solve ? 2 : 0);
  const void* fn = fns[which];
  static DeviceCache configured[4];
  cudaError_t e;
  if ((e = allow_dynamic_smem(fn, configured[which]))) return e;
  if ((e = cudaMemsetAsync(a.xbuf, 0, zeroed, s))) return e;
  RngParams r = rng;
  void* args[] = {&a, &r};
  return launch_strips(fn, G, kThreads, args, smem, status.refuse, s);
}

}  // namespace ising
