// Resident strips: many checkerboard Metropolis sweeps of one lattice per
// launch (arXiv 2402.06415, Results A: the two sublattices updated in turn),
// for lattices whose sweep is too short for a launch of its own.
//
// G CTAs (one per SM, all co-resident) own G row strips of full width and keep
// them as two bit planes in shared memory, with a halo of H = 2K rows above
// and below.  A group of K sweeps runs with CTA barriers only: every half
// sweep invalidates one more halo row on each side, and halo sites are updated
// with their owners' (sweep, site) random numbers, so after K sweeps exactly
// the own rows are correct.  Then each CTA hands its H outer rows to its two
// neighbours through global memory and waits for theirs (a flag per CTA; there
// is no grid barrier).  G = 1 keeps the whole lattice in one CTA without halo.
// Rows are whole, so any even L works: the x wrap and a ragged last word are a
// select per word.
//
// What bounds it: up to L ~ 500 the dependent chain of a half sweep (shared
// loads, neighbour classes, one Philox block, the plane test, a CTA barrier) and
// the exchange (0.9 us).  There four threads share a word, one Philox block
// each (SPLIT), and draw the next half sweep's block while this one's loads and
// shuffles are in flight: a half sweep of 32 words takes 0.19 us against 0.62
// with one thread per word.  Above, three blocks per word on the multiply pipe
// (4 cycles per 32 x 32 -> 64 product and sub-partition).  Time per sweep, before
// (launches per sweep or half sweep; int8: one CTA) and with strips: L = 64 int8
// 16.4 -> 0.55 us, L = 256 8.3 -> 1.04, L = 1000 8.2 -> 1.85, L = 2048 21 -> 2.5 (k_strip_edge).
#include <algorithm>

#include "internal.h"
#include "ising_device.cuh"

namespace ising {
namespace {

// NB Philox blocks (4 NB planes) of a word, and one strict comparison over them
// (planes8 with a variable number of blocks).
template <int NB>
__device__ __forceinline__ void draw_planes(uint4 (&pl)[NB], uint32_t g, uint32_t t, uint32_t rep, uint32_t colour,
                                            const RngParams& rng) {
#pragma unroll
  for (int b = 0; b < NB; ++b)
    pl[b] = philox10_rk(make_uint4(g, t, rep, ctr_w(kTagMet, colour, b)), rng.rk0, rng.rk1);
}
template <int NB>
__device__ __forceinline__ void compare_planes(const uint4 (&pl)[NB], const RngParams& rng, uint32_t& D, uint32_t cls,
                                               uint32_t& acc) {
  uint32_t bor = 0u, eq = D;
#pragma unroll
  for (int b = NB - 1; b >= 0; --b) {
    const uint32_t p[4] = {pl[b].x, pl[b].y, pl[b].z, pl[b].w};
#pragma unroll
    for (int q = 3; q >= 0; --q) {
      const int k = 4 * b + q;
      const uint32_t tm = (cls & rng.tm4[k]) | (~cls & rng.tm8[k]);  // lane's threshold bit
      bor = (~p[q] & tm) | (~p[q] & bor) | (tm & bor);
      eq &= ~(tm ^ p[q]);
    }
  }
  acc |= D & bor;
  D = eq;
}

// Words of a strip's planes (P(c)[i] = word group_of(i) of colour c), and its own rows
// back to the lattice.  With int8 spins a warp takes a word, lane j site j's byte.
template <bool I8, typename Plane, typename Group>
__device__ __forceinline__ void strip_load(const StripArgs& a, int n_words, Plane P, Group group_of) {
  const int tid = threadIdx.x, nth = blockDim.x, L = a.L, Wc = a.Wc;
  if (I8) {
    // kWords loads of a warp in flight: one word after the other, and the edge words of
    // k_strip_edge byte after byte, a call of one sweep at L = 1000 (224 words and 4 warps a
    // strip) took 32.8 us, so 24.6
    constexpr int kWords = 8;
    const int warps = nth >> 5;
    for (int i0 = tid >> 5; i0 < 2 * n_words; i0 += kWords * warps) {
      bool up[kWords];
#pragma unroll
      for (int u = 0; u < kWords; ++u) {
        const int i = min(i0 + u * warps, 2 * n_words - 1);
        const int c = i >= n_words, g = group_of(i - c * n_words);
        const int y = (int)fdiv((uint32_t)g, a.fwc), w = g - y * Wc;
        const int j = 32 * w + (tid & 31);
        up[u] = j < L / 2 && a.spins[(size_t)y * L + 2 * j + ((y + c) & 1)] > 0;
      }
#pragma unroll
      for (int u = 0; u < kWords; ++u) {
        const int i = i0 + u * warps;
        const uint32_t v = __ballot_sync(0xffffffffu, up[u]);
        if (i < 2 * n_words && (tid & 31) == 0) P(i >= n_words)[i >= n_words ? i - n_words : i] = v;
      }
    }
  } else {
    for (int i = tid; i < 2 * n_words; i += nth) {
      const int c = i >= n_words, k = i - c * n_words;
      P(c)[k] = __ldcg(&a.planes[(size_t)c * L * Wc + group_of(k)]);
    }
  }
}
template <bool I8, typename Plane>
__device__ __forceinline__ void strip_store(const StripArgs& a, int y0, int R, int off, Plane P) {
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, L = a.L, Wc = a.Wc, n = R * Wc;
  if (I8) {
    for (int i = tid >> 5; i < 2 * n; i += nth >> 5) {
      const int c = i >= n, k = i - c * n;
      const int r = (int)fdiv((uint32_t)k, a.fwc), w = k - r * Wc, y = y0 + r;
      const uint32_t v = P(c)[off + k];
      const int j = 32 * w + lane;
      if (j < L / 2) a.spins[(size_t)y * L + 2 * j + ((y + c) & 1)] = (v >> lane) & 1u ? 1 : -1;
    }
  } else {
    for (int i = tid; i < 2 * n; i += nth) {
      const int c = i >= n, k = i - c * n;
      a.planes[(size_t)c * L * Wc + (size_t)y0 * Wc + k] = P(c)[off + k];
    }
  }
}

template <bool WHOLE, bool I8, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? kSplitThreads : kStripThreads) k_strip(StripArgs a, RngParams rng) {
  extern __shared__ uint32_t strip_smem[];
  const int L = a.L, Wc = a.Wc, n_half = L / 2;
  const int nb = n_half - 32 * (Wc - 1);                       // valid bits of a row's last word
  const uint32_t last_mask = nb >= 32 ? 0xffffffffu : ((1u << nb) - 1u);
  const int G = WHOLE ? 1 : a.G, H = WHOLE ? 0 : 2 * a.K;
  const int b = blockIdx.x, tid = threadIdx.x, nth = blockDim.x, lane = tid & 31;
  const int y0 = (int)((long long)b * L / G), y1 = (int)((long long)(b + 1) * L / G);
  const int R = y1 - y0, rows = R + 2 * H;
  const int plane = ((L + G - 1) / G + 2 * H) * Wc;
  auto P = [plane](int c) { return strip_smem + c * plane; };
  const int LW = L * Wc, n_words = rows * Wc;
  // word i of the strip is group g = i + goff of the lattice, modulo L * Wc
  const int goff = (y0 - H) * Wc;
  auto group_of = [&](int i) {
    int g = i + goff;
    if (!WHOLE) {
      g += g < 0 ? LW : 0;
      g -= g >= LW ? LW : 0;
    }
    return g;
  };
  strip_load<I8>(a, n_words, P, group_of);
  __syncthreads();
  // slots of this strip: 2 x 4 hw boundary pairs (two buffers used in turn), then
  // one "lattice read" token
  const int hw = H * Wc;
  const size_t per_cta = 8 * (size_t)hw + 1;
  unsigned long long* const mine = WHOLE ? nullptr : a.xbuf + b * per_cta;
  const unsigned long long* const up_slots = WHOLE ? nullptr : a.xbuf + (b == 0 ? G - 1 : b - 1) * per_cta;
  const unsigned long long* const dn_slots = WHOLE ? nullptr : a.xbuf + (b == G - 1 ? 0 : b + 1) * per_cta;
  if (!WHOLE && tid == 0) send_word(mine + 8 * hw, 1u, 0u);
  uint32_t exchanges = 0;
  int to_rec = a.to_rec;  // sweeps until the next record (counting this one), 0 = never
  long long slot = a.rec0;
  // SPLIT: four threads per word, one Philox block each (planes 4q .. 4q + 3),
  // always the same word, whose two spin words stay in registers
  const int q = tid & 3;
  const int wi = (WHOLE ? 0 : Wc) + (tid >> 2);
  const bool mine_w = SPLIT && wi < n_words - (WHOLE ? 0 : Wc);
  const int i1 = mine_w ? wi : (WHOLE ? 0 : Wc);
  const int r1 = (int)fdiv((uint32_t)i1, a.fwc), w1 = i1 - r1 * Wc;
  const uint32_t g1 = (uint32_t)group_of(i1);
  const bool first1 = w1 == 0, last1 = w1 == Wc - 1;
  const int o1 = (y0 + r1) & 1;  // x offset of colour 0
  int iu1 = i1 - Wc, id1 = i1 + Wc;
  if (WHOLE) {
    iu1 += iu1 < 0 ? n_words : 0;
    id1 -= id1 >= n_words ? n_words : 0;
  }
  const int il1 = first1 ? i1 + Wc - 1 : i1 - 1, ir1 = last1 ? i1 - Wc + 1 : i1 + 1;
  const int shl1 = first1 ? nb - 1 : 31, shr1 = last1 ? nb - 1 : 31;
  const uint32_t valid1 = mine_w ? (last1 ? last_mask : 0xffffffffu) : 0u;
  const bool inner1 = mine_w && q == 0 && r1 >= H && r1 < H + R;
  uint32_t m4[4], m8[4], own[2] = {0u, 0u};
  uint4 pl = make_uint4(0u, 0u, 0u, 0u);
  if (SPLIT) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      m4[k] = rng.tm4[4 * q + k];
      m8[k] = rng.tm8[4 * q + k];
    }
    own[0] = P(0)[i1];
    own[1] = P(1)[i1];
    pl = philox10_rk(make_uint4(g1, a.t0, rng.replica, ctr_w(kTagMet, 0u, (uint32_t)q)), rng.rk0, rng.rk1);
  }
  for (int done = 0; done < a.n;) {
    const int kk = min(a.K, a.n - done);
    if (SPLIT) {
      for (int s2 = 0; s2 < kk; ++s2) {
        const uint32_t t = a.t0 + (uint32_t)(done + s2);
        unsigned int anti = 0, ones = 0;
        const bool meas = to_rec == 1;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t* const So = P(c);
          const uint32_t* const Sn = P(1 - c);
          const bool left = ((o1 ^ c) & 1) == 0;
          const uint32_t s = own[c], mid = own[1 - c];
          const uint32_t up = Sn[iu1], dn = Sn[id1], x = Sn[left ? il1 : ir1];
          // the next half sweep's planes do not depend on spins: drawn while
          // this one's loads and shuffles are in flight
          const uint4 nx = philox10_rk(make_uint4(g1, t + (uint32_t)c, rng.replica,
                                                  ctr_w(kTagMet, (uint32_t)(1 - c), (uint32_t)q)),
                                       rng.rk0, rng.rk1);
          const uint32_t side = left ? (mid << 1) | ((x >> shl1) & 1u) : (mid >> 1) | ((x & 1u) << shr1);
          const HalfClasses k = classify_hs(s, up ^ dn, up, dn, mid, side);
          const uint32_t p[4] = {pl.x, pl.y, pl.z, pl.w};
          uint32_t bor = 0u, eq = 0xffffffffu;
#pragma unroll
          for (int j = 3; j >= 0; --j) {
            const uint32_t tm = (k.cls & m4[j]) | (~k.cls & m8[j]);
            bor = (~p[j] & tm) | (~p[j] & bor) | (tm & bor);
            eq &= ~(tm ^ p[j]);
          }
          // merge the four blocks' verdicts: the more significant block decides
          // unless it is tied (eq)
#pragma unroll
          for (int st = 1; st <= 2; st <<= 1) {
            const uint32_t ob = __shfl_xor_sync(0xffffffffu, bor, st), oe = __shfl_xor_sync(0xffffffffu, eq, st);
            const bool hi = (q & st) == 0;
            const uint32_t hb = hi ? bor : ob, he = hi ? eq : oe, lb = hi ? ob : bor;
            bor = hb | (he & lb);
            eq &= oe;
          }
          uint32_t D = ~k.ge2 & valid1;
          uint32_t acc = D & bor;
          D &= eq;
          // a tie over 16 planes (1 word in 2500): the other blocks.  By the lane alone
          // (no vote: 1.14 -> 1.04 us per sweep at L = 256), in one CTA by vote (0.56 -> 0.53
          // at L = 64)
          if (WHOLE) {
            if (__any_sync(0xffffffffu, D != 0u))
              lazy_planes<4, 8>(g1, t, rng.replica, (uint32_t)c, rng, D, k.cls, acc);
          } else if (D != 0u) {
            acc |= finish_word<4>(g1, t, rng.replica, (uint32_t)c, rng, D, k.cls);
          }
          const uint32_t ns = s ^ ((k.ge2 & valid1) | acc);
          own[c] = ns;
          if (mine_w && q == 0) So[i1] = ns;
          if (c == 1 && meas && inner1) {
            anti = __popc((ns ^ up) & valid1) + __popc((ns ^ dn) & valid1) + __popc((ns ^ mid) & valid1) +
                   __popc((ns ^ side) & valid1);
            ones = __popc(ns & valid1) + __popc(mid & valid1);
          }
          pl = nx;
          __syncthreads();
        }
        if (meas) {
          anti = __reduce_add_sync(0xffffffffu, anti);
          ones = __reduce_add_sync(0xffffffffu, ones);
          if (lane == 0 && (anti | ones)) {
            atomicAdd(&a.rec[2 * slot], (unsigned long long)anti);
            atomicAdd(&a.rec[2 * slot + 1], (unsigned long long)ones);
          }
        }
        if (to_rec > 0 && --to_rec == 0) {
          to_rec = a.m;
          slot = slot + 1 == a.rec_cap ? 0 : slot + 1;
        }
      }
    } else {
      for (int h = 0; h < 2 * kk; ++h) {
        const int c = h & 1;
        const uint32_t t = a.t0 + (uint32_t)(done + (h >> 1));
        const bool meas = c == 1 && to_rec == 1;
        uint32_t* const So = P(c);
        const uint32_t* const Sn = P(1 - c);
        // rows still correct after this half sweep (a short last group starts further in)
        const int margin = WHOLE ? 0 : h + 1 + 2 * (a.K - kk);
        const int lo = margin * Wc, count = n_words - 2 * lo;
        unsigned int anti = 0, ones = 0;
        for (int base = tid & ~31; base < count; base += nth) {
          const bool active = base + lane < count;
          const int i = lo + (active ? base + lane : 0);
          const int r = (int)fdiv((uint32_t)i, a.fwc), w = i - r * Wc;
          int iu = i - Wc, id = i + Wc;
          if (WHOLE) {
            iu += iu < 0 ? n_words : 0;
            id -= id >= n_words ? n_words : 0;
          }
          const bool first = w == 0, last = w == Wc - 1;
          const int o = (y0 + r + c) & 1;  // H is even
          const int ix = o == 0 ? (first ? i + Wc - 1 : i - 1) : (last ? i - Wc + 1 : i + 1);
          const uint32_t s = So[i], up = Sn[iu], dn = Sn[id], mid = Sn[i], x = Sn[ix];
          const uint32_t side = o == 0 ? (mid << 1) | ((x >> (first ? nb - 1 : 31)) & 1u)
                                       : (mid >> 1) | ((x & 1u) << (last ? nb - 1 : 31));
          const uint32_t valid = active ? (last ? last_mask : 0xffffffffu) : 0u;
          const HalfClasses k = classify_hs(s, up ^ dn, up, dn, mid, side);
          uint32_t D = ~k.ge2 & valid, acc = 0;
          const uint32_t g = (uint32_t)group_of(i);
          uint4 p[kStripBlocks];
          draw_planes(p, g, t, rng.replica, (uint32_t)c, rng);
          compare_planes(p, rng, D, k.cls, acc);
          lazy_planes<kStripBlocks, 8>(g, t, rng.replica, (uint32_t)c, rng, D, k.cls, acc);
          const uint32_t ns = s ^ ((k.ge2 & valid) | acc);
          if (active) So[i] = ns;
          if (meas && r >= H && r < H + R) {
            anti += __popc((ns ^ up) & valid) + __popc((ns ^ dn) & valid) + __popc((ns ^ mid) & valid) +
                    __popc((ns ^ side) & valid);
            ones += __popc(ns & valid) + __popc(mid & valid);
          }
        }
        if (meas) {
          anti = __reduce_add_sync(0xffffffffu, anti);
          ones = __reduce_add_sync(0xffffffffu, ones);
          if (lane == 0 && (anti | ones)) {
            atomicAdd(&a.rec[2 * slot], (unsigned long long)anti);
            atomicAdd(&a.rec[2 * slot + 1], (unsigned long long)ones);
          }
        }
        if (c == 1 && to_rec > 0 && --to_rec == 0) {
          to_rec = a.m;
          slot = slot + 1 == a.rec_cap ? 0 : slot + 1;
        }
        __syncthreads();
      }
    }
    done += kk;
    if (WHOLE || done >= a.n) continue;
    // exchange: own rows [H, 2H) go up, [R, R + H) go down; buffers alternate
    const uint32_t tag = ++exchanges;
    const size_t buf = (size_t)(tag & 1) * 4 * hw;
    for (int i = tid; i < 4 * hw; i += nth) {
      const int lower = i >= 2 * hw, rem = i - lower * 2 * hw;
      const int c = rem >= hw, k = rem - c * hw;
      send_word(mine + buf + i, tag, P(c)[(lower ? R * Wc : H * Wc) + k]);
    }
    bool ok = true;
    // the upper neighbour's lower rows, the lower neighbour's upper rows
    auto src = [&](int i) {
      const int lower = i >= 2 * hw;
      return (lower ? dn_slots : up_slots + 2 * hw) + buf + (i - lower * 2 * hw);
    };
    recv_words<SPLIT ? 1 : 4>(tid, nth, 4 * hw, src, tag, a.limit, a.status, ok, [&](int i, uint32_t word) {
      const int lower = i >= 2 * hw, rem = i - lower * 2 * hw;
      const int c = rem >= hw, k = rem - c * hw;
      P(c)[(lower ? (H + R) * Wc : 0) + k] = word;
    });
    if (!__syncthreads_and(ok)) return;
    if (SPLIT) {
      own[0] = P(0)[i1];
      own[1] = P(1)[i1];
    }
  }
  // the lattice is updated in place: both neighbours must have read their halos
  if (!WHOLE && exchanges == 0) {
    uint32_t word;
    bool ok = true;
    if (tid < 2) ok = recv_word((tid ? dn_slots : up_slots) + 8 * hw, 1u, a.limit, a.status, word);
    if (!__syncthreads_and(ok)) return;
  }
  strip_store<I8>(a, y0, R, H * Wc, P);
}

// Strips without a halo in shared memory, for rows long enough that a half sweep
// takes about as long as an exchange: the first and the last row's words belong to
// threads of their own, which send each new word and wait for the neighbour's one in a
// register, while the other warps update the inner rows.  A half sweep then costs the
// longer of the two instead of their sum, and no row is updated twice.  Every thread
// draws the planes of its (first) word of the next half sweep ahead, edge warps once
// they have sent; words beyond the CTA's threads are taken in a loop.  us per sweep,
// k_strip -> here: L = 1300 2.32 -> 2.11, 2048 3.49 -> 2.49, 3072 5.7 -> 4.5, 4096 8.4 -> 7.4; with
// the planes drawn before the wait 2048 took 2.63, drawn by all after the update 2.60.
// Bound by the round trip of an edge word (0.85 us per half sweep) up to L ~ 1800, then
// by the logic and multiply pipes.
template <bool I8>
__global__ void __launch_bounds__(kStripThreads) k_strip_edge(StripArgs a, RngParams rng) {
  extern __shared__ uint32_t strip_smem[];
  const int L = a.L, Wc = a.Wc, G = a.G, n_half = L / 2;
  const int nb = n_half - 32 * (Wc - 1);                       // valid bits of a row's last word
  const uint32_t last_mask = nb >= 32 ? 0xffffffffu : ((1u << nb) - 1u);
  const int b = blockIdx.x, tid = threadIdx.x, nth = blockDim.x, lane = tid & 31;
  const int y0 = (int)((long long)b * L / G), y1 = (int)((long long)(b + 1) * L / G);
  const int R = y1 - y0, n_words = R * Wc;
  const int plane = ((L + G - 1) / G) * Wc;
  auto P = [plane](int c) { return strip_smem + c * plane; };
  strip_load<I8>(a, n_words, P, [&](int i) { return y0 * Wc + i; });
  // words in the order first row, last row, inner rows: row and index of the k-th
  auto row_of = [&](int k, int& w) {
    const int q = (int)fdiv((uint32_t)k, a.fwc);
    w = k - q * Wc;
    return q == 0 ? 0 : q == 1 ? R - 1 : q - 1;
  };
  const bool active1 = tid < n_words, edge = tid < 2 * Wc, top = tid < Wc;
  const bool edge_warp = (tid & ~31) < 2 * Wc;
  int w1;
  const int r1 = row_of(active1 ? tid : 0, w1), i1 = r1 * Wc + w1;
  const uint32_t g1 = (uint32_t)(y0 * Wc + i1);
  // the neighbour's row that an edge word needs: colour 1 as the call found it
  uint32_t beyond = 0;
  if (edge) {
    const int y = top ? (y0 == 0 ? L - 1 : y0 - 1) : (y1 == L ? 0 : y1);
    if (I8) {
      // all 32 loads in flight
      const int8_t* const row = a.spins + (size_t)y * L + 64 * w1 + ((y + 1) & 1);
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (32 * w1 + j < n_half) beyond |= (uint32_t)(row[2 * j] > 0) << j;
    } else {
      beyond = __ldcg(&a.planes[(size_t)L * Wc + (size_t)y * Wc + w1]);
    }
  }
  __syncthreads();
  // slots: two buffers used in turn of 2 Wc pairs, first row and last row.  A strip writes
  // one again only after it received what its neighbour sent having read it
  unsigned long long* const mine = a.xbuf + (size_t)b * 4 * Wc + tid;
  const unsigned long long* const theirs =
      a.xbuf + (size_t)(top ? (b == 0 ? G - 1 : b - 1) : (b == G - 1 ? 0 : b + 1)) * 4 * Wc + (top ? Wc : 0) + w1;
  uint32_t own[2] = {P(0)[i1], P(1)[i1]};
  uint4 pl[kStripBlocks];
  draw_planes(pl, g1, a.t0, rng.replica, 0u, rng);
  uint32_t sent = 0;
  int to_rec = a.to_rec;
  long long slot = a.rec0;
  for (int s2 = 0; s2 < a.n; ++s2) {
    const uint32_t t = a.t0 + (uint32_t)s2;
    const bool meas = to_rec == 1;
    unsigned int anti = 0, ones = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      uint32_t* const So = P(c);
      const uint32_t* const Sn = P(1 - c);
      // word w of row r, index i; up / dn: the words above and below
      auto update = [&](int w, int r, int i, bool active, uint32_t g, uint32_t s, uint32_t mid, uint32_t up,
                        uint32_t dn, const uint4(&p)[kStripBlocks]) {
        const bool first = w == 0, last = w == Wc - 1, left = ((y0 + r + c) & 1) == 0;
        const uint32_t x = Sn[left ? (first ? i + Wc - 1 : i - 1) : (last ? i - Wc + 1 : i + 1)];
        const uint32_t side = left ? (mid << 1) | ((x >> (first ? nb - 1 : 31)) & 1u)
                                   : (mid >> 1) | ((x & 1u) << (last ? nb - 1 : 31));
        const uint32_t valid = active ? (last ? last_mask : 0xffffffffu) : 0u;
        const HalfClasses k = classify_hs(s, up ^ dn, up, dn, mid, side);
        uint32_t D = ~k.ge2 & valid, acc = 0;
        compare_planes(p, rng, D, k.cls, acc);
        if (D != 0u) acc |= finish_word<kStripBlocks>(g, t, rng.replica, (uint32_t)c, rng, D, k.cls);
        const uint32_t ns = s ^ ((k.ge2 & valid) | acc);
        if (active) So[i] = ns;
        if (c == 1 && meas) {
          anti += __popc((ns ^ up) & valid) + __popc((ns ^ dn) & valid) + __popc((ns ^ mid) & valid) +
                  __popc((ns ^ side) & valid);
          ones += __popc(ns & valid) + __popc(mid & valid);
        }
        return ns;
      };
      // the next half sweep's planes: edge warps first wait, update and send
      uint4 nx[kStripBlocks];
      if (!edge_warp) draw_planes(nx, g1, t + (uint32_t)c, rng.replica, (uint32_t)(1 - c), rng);
      bool ok = true;
      if (edge && sent > 0)
        ok = recv_word(theirs + (sent & 1 ? 2 * Wc : 0), sent, a.limit, a.status, beyond);
      ++sent;
      const uint32_t up = edge && top ? beyond : Sn[r1 == 0 ? i1 : i1 - Wc];
      const uint32_t dn = edge && !top ? beyond : Sn[r1 == R - 1 ? i1 : i1 + Wc];
      own[c] = update(w1, r1, i1, active1, g1, own[c], own[1 - c], up, dn, pl);
      if (edge) send_word(mine + (sent & 1 ? 2 * Wc : 0), sent, own[c]);
      if (edge_warp) draw_planes(nx, g1, t + (uint32_t)c, rng.replica, (uint32_t)(1 - c), rng);
#pragma unroll
      for (int j = 0; j < kStripBlocks; ++j) pl[j] = nx[j];
      // the last warps, which have no edge words, first
      for (int base = 2 * nth - 32 - (tid & ~31); base < n_words; base += nth) {
        const bool active = base + lane < n_words;
        int w;
        const int r = row_of(active ? base + lane : 2 * Wc, w), i = r * Wc + w;
        const uint32_t g = (uint32_t)(y0 * Wc + i);
        uint4 p[kStripBlocks];
        draw_planes(p, g, t, rng.replica, (uint32_t)c, rng);
        update(w, r, i, active, g, So[i], Sn[i], Sn[i - Wc], Sn[i + Wc], p);
      }
      // (a plain barrier and a failure that is carried to the end: 2 to 7 % slower)
      if (!__syncthreads_and(ok)) return;
    }
    if (meas) {
      anti = __reduce_add_sync(0xffffffffu, anti);
      ones = __reduce_add_sync(0xffffffffu, ones);
      if (lane == 0 && (anti | ones)) {
        atomicAdd(&a.rec[2 * slot], (unsigned long long)anti);
        atomicAdd(&a.rec[2 * slot + 1], (unsigned long long)ones);
      }
    }
    if (to_rec > 0 && --to_rec == 0) {
      to_rec = a.m;
      slot = slot + 1 == a.rec_cap ? 0 : slot + 1;
    }
  }
  // in place: a neighbour's edge threads read this strip's rows before they sent the
  // words that its own edge threads have received
  strip_store<I8>(a, y0, R, 0, P);
}

}  // namespace

size_t strip_smem_bytes(int L, int G, int K) {
  const int Wc = (L / 2 + 31) / 32;
  const int H = G == 1 ? 0 : 2 * K;  // K = 0: k_strip_edge, no halo
  return 2ull * (size_t)((L + G - 1) / G + 2 * H) * (size_t)Wc * sizeof(uint32_t);
}

size_t strip_xbuf_words(int L, int G, int K) {
  const int Wc = (L / 2 + 31) / 32;
  return G == 1 ? 0 : K == 0 ? (size_t)G * 4 * Wc : (size_t)G * (16 * (size_t)K * Wc + 1);
}

// Time model of one sweep in microseconds, fitted to sweeps of (G, K) on GB300
// for L = 32 ... 6144 (within 15 %): per half sweep 0.10 + 0.085 us per resident
// warp of an SM sub-partition with four threads per word (SPLIT), 0.33 + 0.23 us
// with one, and 0.9 us per exchange; without a halo (K = 0) the longer of 0.85 + 0.08 us
// and 0.25 + 0.25 us per half sweep, and never below the other forms up to L ~ 900.
static double strip_model_us(int L, int Wc, int G, int K) {
  const int R = (L + G - 1) / G;
  const bool whole = G == 1;
  if (K == 0) {
    const int wps = ((R * Wc + 31) / 32 + 3) / 4;
    return 2 * std::max(0.85 + 0.08 * wps, 0.25 + 0.25 * wps);
  }
  const int most = (R + (whole ? 0 : 4 * K - 2)) * Wc;
  double t = whole ? 0.0 : 0.9;
  if (4 * most <= kSplitThreads) {
    const int wps = ((most + 7) / 8 + 3) / 4;
    t += 2 * K * (0.10 + 0.085 * wps);
  } else {
    for (int h = 0; h < 2 * K; ++h) {
      const int words = (R + (whole ? 0 : 2 * (2 * K - 1 - h))) * Wc;
      t += 0.33 + 0.23 * (((words + 31) / 32 + 3) / 4);
    }
  }
  return t / K;
}

StripShape choose_strip(int L, int sms) {
  const int Wc = (L / 2 + 31) / 32;
  StripShape best{0, 0, 1e30};
  for (int G = 1; G <= sms && G <= L / 2; ++G)
    for (int K = G == 1 ? 1 : 0; K <= (G == 1 ? 1 : kStripMaxK); ++K) {
      // k_strip_edge: two rows at least, and a thread for each edge word
      if (K == 0 && (L / G < 2 || 2 * Wc > kStripThreads)) continue;
      if (G > 1 && L / G < 2 * K) break;  // the halo comes from the next strip only
      if (strip_smem_bytes(L, G, K) > 200 * 1024) break;
      const double t = strip_model_us(L, Wc, G, K);
      // without a halo, equal warps a sub-partition: more strips from two warps on (us per sweep
      // for 128 / 152 strips: L = 1000 1.78 / 1.85, 1600 2.27 / 2.17, 2048 2.58 / 2.49)
      const bool finer = K == 0 && best.K == 0 && t == best.us && (L + G - 1) / G * Wc > 128;
      if (t < best.us || finer) best = {G, G == 1 ? 1 << 30 : K, t};
    }
  return best;
}

cudaError_t launch_strip_sweep(StripArgs a, const RngParams& rng, bool refuse, cudaStream_t s) {
  const bool whole = a.G == 1, edge = a.K == 0, i8 = a.spins != nullptr;
  if (a.K > a.n) a.K = a.n;
  const size_t smem = strip_smem_bytes(a.L, a.G, a.K);
  const int words = (int)(((a.L + a.G - 1) / a.G + (whole || edge ? 0 : 4 * a.K - 2)) * (long long)a.Wc);
  const bool split = !edge && 4 * words <= kSplitThreads;
  const void* fns[10] = {(const void*)k_strip<false, false, false>, (const void*)k_strip<true, false, false>,
                         (const void*)k_strip<false, true, false>,  (const void*)k_strip<true, true, false>,
                         (const void*)k_strip<false, false, true>,  (const void*)k_strip<true, false, true>,
                         (const void*)k_strip<false, true, true>,   (const void*)k_strip<true, true, true>,
                         (const void*)k_strip_edge<false>, (const void*)k_strip_edge<true>};
  a.fwc = make_fastdiv((uint32_t)a.Wc);
  const int which = edge ? (i8 ? 9 : 8) : (whole ? 1 : 0) + (i8 ? 2 : 0) + (split ? 4 : 0);
  static DeviceCache configured[10];
  cudaError_t e = allow_dynamic_smem(fns[which], configured[which]);
  if (e != cudaSuccess) return e;
  int threads = (((split ? 4 : 1) * words + 31) / 32) * 32;
  if (threads < 64) threads = 64;
  if (!split && threads > kStripThreads) threads = kStripThreads;
  RngParams r = rng;
  void* args[] = {&a, &r};
  if (whole) return cudaLaunchKernel(fns[which], dim3(1), dim3(threads), args, smem, s);
  e = cudaMemsetAsync(a.xbuf, 0, strip_xbuf_words(a.L, a.G, a.K) * 8, s);
  if (e != cudaSuccess) return e;
  return launch_strips(fns[which], a.G, threads, args, smem, refuse, s);
}

}  // namespace ising
