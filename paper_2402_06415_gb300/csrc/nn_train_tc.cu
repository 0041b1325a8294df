// CNN training on the tensor cores: loss and gradients of the block proposal's
// maximum-likelihood objective (the same samples, inputs, loss terms and
// normalisation as the FP32 kernel k_nn_train in nn.cu) with the three
// contractions of the 32 -> 32 convolution on warp-level mma.sync
// (m16n8k16, BF16 operands, FP32 accumulation):
//   forward        z2[p][o]  = sum_{t,c} h1[p + d_t][c] W2[o][c][t]
//   input gradient g1[q][c]  = sum_{t,o} gz2[q - d_t][o] W2[o][c][t]
//   weight gradient dW2[o][c][t] += sum_p gz2[p][o] h1[p + d_t][c]
// (p, q frame positions, d_t the offset of tap t, zero outside the frame).
// Activations and dL/dz2 are rounded to BF16 for the MMA operands (the master
// weights stay FP32, the operands see them in BF16), so gradients agree with the
// FP32 kernel to BF16 rounding, not bit for bit.  Layers 1 and 3 (2 -> 32 and
// 32 -> 1 channels) are FP32: layer 3 on the CUDA cores; layer 1 and its weight
// gradient on mma.sync as well, with the FP32 operand (W1, dL/dz1) split into
// three BF16 terms that hold it exactly; the other operand, the spins and the
// known mask, is exact in BF16, so products are exact and sums FP32.
//
// A stage's loss terms sit at a few sites, so only the positions next to them
// carry a gradient: h2 matters at the sites' 3 x 3 neighbourhoods (list l2 of the
// plan), h1 at their 5 x 5 neighbourhoods (list l1); everywhere else the
// gradients are exactly zero.  Over the 8 network stages of a 16 x 16 block that
// is 666 and 1196 positions instead of 8 x 324 each.  A CTA takes up to kMaxW
// windows of one stage at a time and keeps their activations packed in list
// order, so the matrix rows are dense; tables per stage give, for every list
// entry and tap, the row to gather (a zero row where there is none).  512 layer-1
// rows at a time give each of the 16 warps one unit of 32 rows x 32 channels.
// The windows of all stages are dealt to the CTAs in contiguous ranges of equal
// estimated work, so a CTA builds the tables of one or two stages.
//
// What bounds it: the barriers between phases and the latency of ldmatrix, with 4
// warps a sub-partition (stalls per instruction: barrier 2.6, fixed latency 2.2, shared
// memory 2.0); the tensor pipe is 29 % busy, the load / store unit, through which every warp
// reads the weights again, 18 %.  128 registers, 100 bytes of them spilled.
// 512 windows x 8 stages: kernel 1520 -> 192 us, loss and gradients through the
// API 1560 -> 236 us (before: full frames, one sample at a time, and one thread
// listing the loss sites).
// Each CTA keeps its weight-gradient sums in registers over all its windows and
// adds them to the global gradient once.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "nn_common.cuh"

namespace ising {
namespace nnc {
namespace {

constexpr int kTcWarps = 16, kTcThreads = 32 * kTcWarps;
constexpr int kCap1 = 512, kCap2 = 336, kCap3 = kMaxB * kMaxB;  // packed rows of layers 1, 2, 3
constexpr int kMaxW = 12;                                        // windows of a stage at a time
// layer-1 inputs of a row: columns 0 .. 15 (spin, known) of taps 0 .. 7; then, three
// times (once per BF16 term of the weights), (spin, known) of tap 8, a one for the
// bias and a zero; zeros up to 32
constexpr int kXP = 40, kW1K = 64;  // row stride, K of the layer-1 product
constexpr uint16_t kNone = 0xffff;
static_assert(kCap1 >= kMaxFrame && kCap2 >= kMaxFrame, "one full-frame window must fit");
static_assert(kCap1 == 32 * kTcWarps, "one unit of 32 layer-1 rows per warp");

struct TrainTcSmem {
  __nv_bfloat16 w2f[kC * kK2P];          // W2 as [o][t * 32 + c]
  __nv_bfloat16 h1[(kCap1 + 1) * kCP];   // layer-1 output rows (the last row is zero)
  __nv_bfloat16 h2[(kCap2 + 1) * kCP];   // layer-2 output rows
  __nv_bfloat16 gz2[(kCap2 + 1) * kCP];  // dL/dz2 rows (the last row is zero)
  __nv_bfloat16 x[kCap1 * kXP];          // layer-1 input rows
  // W1 and b1 in three BF16 terms, [c][K]: terms of taps 0 .. 7 at 0, 16, 32, of x columns 16 .. 27 at 48
  __nv_bfloat16 w1s[kC * (kW1K + 8)];
  uint32_t mask[kCap1];                  // layer-1 row: bit c set iff h1[c] > 0
  alignas(16) float w3t[9 * kC];         // W3 as [t][c]
  float b2[kC], b3;
  float g3[kCap3];                       // dL/dz3 at the sites
  // tables of the current stage
  uint32_t p1[kMaxFrame];       // l1 entry: frame position, known taps << 16
  uint16_t nb1[kMaxFrame * 9];  // l2 entry, tap -> l1 entry at p + d_t
  uint16_t nb2[kMaxFrame * 9];  // l1 entry, tap -> l2 entry at q - d_t
  uint16_t nb3[kMaxFrame * 9];  // l2 entry, tap -> site at p - d_t
  uint16_t nb4[kCap3 * 9];      // site, tap -> l2 entry at p + d_t
  uint16_t m3[kMaxFrame];       // l2 entry: taps of nb3 that exist
  uint2 l3s[kMaxFrame];         // l2 entry: its first four sites, 16 bits each: tap | site << 4 (kNone: no more)
  uint16_t at1[kMaxFrame], at2[kMaxFrame], at3[kMaxFrame];  // frame position -> list entry
  int8_t win[kMaxW * kMaxFrame];
};
constexpr int kRed = 30;  // per-warp sums added up at the end, rows of 32: 18 W1, b1, b2, 9 W3 (and one spare)
static_assert(kTcWarps * kRed * kC * 4 <= (kCap1 + kCap2) * kCP * 2, "the sums fit the h1 and h2 buffers");

__device__ __forceinline__ void ldm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
      "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldm_x2_t(uint32_t addr, uint32_t& r0, uint32_t& r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(addr));
}
// v0, v1 as a sum of three packed BF16 pairs, exactly (8 + 8 + 8 significand bits)
__device__ __forceinline__ void split3(float v0, float v1, uint32_t (&o)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
    o[i] = *reinterpret_cast<const uint32_t*>(&h);
    v0 -= __uint_as_float(o[i] << 16);
    v1 -= __uint_as_float(o[i] & 0xffff0000u);
  }
}

__device__ __forceinline__ void ldm_x4_row(const __nv_bfloat16* p, uint32_t (&r)[4]) {
  ldm_x4(smem_addr(p), r[0], r[1], r[2], r[3]);
}

// Work of one window of a stage in units of about one layer-1 row, for the
// division of the windows among the CTAs.
__device__ __forceinline__ long long window_cost(const StagedPlan* plan, int k) {
  return (plan->off1[k + 1] - plan->off1[k]) + (plan->off2[k + 1] - plan->off2[k]) +
         4 * (plan->off3[k + 1] - plan->off3[k]) + 16;
}

__global__ void __launch_bounds__(kTcThreads, 1) k_nn_train_tc(const int8_t* __restrict__ windows, int n,
                                                               const StagedPlan* __restrict__ plan,
                                                               const float* __restrict__ params,
                                                               float* __restrict__ grads, float* __restrict__ loss) {
  extern __shared__ uint4 smem_raw[];
  TrainTcSmem& S = *reinterpret_cast<TrainTcSmem*>(smem_raw);
  const int B = plan->B, F = frame_of(B), FF = F * F;
  const float invn = 1.f / (float)n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const __nv_bfloat16 z = __float2bfloat16_rn(0.f);
  // this CTA's windows of a stage: those whose start before + i cost lies in [b, b + 1) total / grid
  const int n_net = plan->n_net;
  long long total = 0;
  for (int s = 0; s < n_net; ++s) total += (long long)n * window_cost(plan, plan->net_ids[s]);
  auto windows_of = [&](long long before, long long cost, int& k_lo, int& k_hi) {
    auto first_of = [&](long long b) {
      const long long x = b * total - before * (long long)gridDim.x, d = cost * (long long)gridDim.x;
      const long long i = x <= 0 ? 0 : (x + d - 1) / d;
      return (int)(i < n ? i : n);
    };
    k_lo = first_of(blockIdx.x);
    k_hi = first_of((long long)blockIdx.x + 1);
    return k_lo < k_hi;
  };
  bool any = false;
  long long before = 0;
  for (int s = 0; s < n_net; ++s) {
    const long long cost = window_cost(plan, plan->net_ids[s]);
    int lo, hi;
    any = windows_of(before, cost, lo, hi) || any;
    before += (long long)n * cost;
  }
  if (!any) return;
  for (int i = tid; i < kC * kC * 9; i += kTcThreads) {
    const int o = i / (kC * 9), c = (i / 9) % kC, t = i % 9;  // W2[o][c][t]
    S.w2f[o * kK2P + t * kC + c] = __float2bfloat16_rn(params[kOffW2 + i]);
  }
  for (int i = tid; i < kC * (kW1K + 8); i += kTcThreads) S.w1s[i] = z;
  __syncthreads();
  for (int i = tid; i < kC * 19; i += kTcThreads) {
    const int c = i / 19, j = i % 19;  // column j = 2 t + ci; 18: the bias
    float v = j < 18 ? params[kOffW1 + c * 18 + (j & 1) * 9 + (j >> 1)] : params[kOffB1 + c];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const __nv_bfloat16 h = __float2bfloat16_rn(v);
      S.w1s[c * (kW1K + 8) + (j < 16 ? 16 * q + j : 48 + 4 * q + j - 16)] = h;
      v -= bf(h);
    }
  }
  for (int i = tid; i < kC * 9; i += kTcThreads) S.w3t[(i % 9) * kC + i / 9] = params[kOffW3 + i];
  for (int i = tid; i < kCap1 * kXP / 8; i += kTcThreads) {  // zeros, and ones in columns 18, 22 and 26
    const int j = i % (kXP / 8);
    reinterpret_cast<uint4*>(S.x)[i] = make_uint4(0u, j == 2 || j == 3 ? 0x3f80u : 0u, 0u, j == 2 ? 0x3f80u : 0u);
  }
  if (tid < kC) S.b2[tid] = params[kOffB2 + tid];
  if (tid == 0) S.b3 = params[kOffB3];
  if (tid < kCP) {
    S.h1[kCap1 * kCP + tid] = z;
    S.h2[kCap2 * kCP + tid] = z;
    S.gz2[kCap2 * kCP + tid] = z;
  }

  // gradient sums of this thread over all its CTA's windows.  dW2: tap warp & 7
  // (both halves of the output channels x four tiles of input channels) and one
  // tile of tap 8, over every second 16 rows; dW1 and db1: 32 channels x 24
  // columns (as x) over this warp's rows; W3[lane][tap] over this warp's sites.
  const int my_tap = warp & 7, my_half = warp >> 3, t8m = my_tap >> 2, t8n = my_tap & 3;
  float dw[9][4] = {}, dw1[2][3][4] = {}, gw3s[9] = {};
  float gb3s = 0.f, my_loss = 0.f;
  float4 gb2s = make_float4(0.f, 0.f, 0.f, 0.f);  // channels 4 (lane & 7) ..

  before = 0;
  for (int s = 0; s < n_net; ++s) {
    const int stage = plan->net_ids[s];
    const long long cost = window_cost(plan, stage);
    int k_lo, k_hi;
    const bool some = windows_of(before, cost, k_lo, k_hi);
    before += (long long)n * cost;
    if (!some) continue;
    const int16_t* l1 = plan->l1 + plan->off1[stage];
    const int16_t* l2 = plan->l2 + plan->off2[stage];
    const int16_t* l3 = plan->l3 + plan->off3[stage];
    const uint16_t* m1 = plan->m1 + plan->off1[stage];
    const int n1 = plan->off1[stage + 1] - plan->off1[stage], n2 = plan->off2[stage + 1] - plan->off2[stage];
    const int n3 = plan->off3[stage + 1] - plan->off3[stage];
    const int W = min(min(kMaxW, kCap1 / n1), min(kCap2 / n2, kCap3 / n3));
    const FastDiv f1 = make_fastdiv((uint32_t)n1), f2 = make_fastdiv((uint32_t)n2), f3 = make_fastdiv((uint32_t)n3);

    // ---- tables of the stage ----
    __syncthreads();
    for (int i = tid; i < FF; i += kTcThreads) S.at1[i] = S.at2[i] = S.at3[i] = kNone;
    __syncthreads();
    for (int e = tid; e < n1; e += kTcThreads) {
      S.at1[l1[e]] = (uint16_t)e;
      S.p1[e] = (uint32_t)l1[e] | ((uint32_t)m1[e] << 16);
    }
    for (int e = tid; e < n2; e += kTcThreads) S.at2[l2[e]] = (uint16_t)e;
    for (int e = tid; e < n3; e += kTcThreads) S.at3[(l3[e] / B + 1) * F + l3[e] % B + 1] = (uint16_t)e;
    __syncthreads();
    auto look = [&](const uint16_t* at, int p, int t, int sign) {
      const int y = p / F + sign * (t / 3 - 1), x = p % F + sign * (t % 3 - 1);
      return y >= 0 && y < F && x >= 0 && x < F ? at[y * F + x] : kNone;
    };
    for (int i = tid; i < n2 * 9; i += kTcThreads) {
      S.nb1[i] = look(S.at1, l2[i / 9], i % 9, +1);
      S.nb3[i] = look(S.at3, l2[i / 9], i % 9, -1);
    }
    for (int i = tid; i < n1 * 9; i += kTcThreads) S.nb2[i] = look(S.at2, l1[i / 9], i % 9, -1);
    for (int i = tid; i < n3 * 9; i += kTcThreads)
      S.nb4[i] = look(S.at2, (l3[i / 9] / B + 1) * F + l3[i / 9] % B + 1, i % 9, +1);
    __syncthreads();
    for (int e = tid; e < n2; e += kTcThreads) {
      uint32_t m = 0;
      uint32_t l[4] = {kNone, kNone, kNone, kNone};
      int q = 0;
      for (int t = 0; t < 9; ++t) {
        const uint32_t site = S.nb3[e * 9 + t];
        if (site == kNone) continue;
        m |= 1u << t;
        const uint32_t x = (uint32_t)t | (site << 4);
        if (q == 0) l[0] = x;
        else if (q == 1) l[1] = x;
        else if (q == 2) l[2] = x;
        else if (q == 3) l[3] = x;
        ++q;
      }
      S.m3[e] = (uint16_t)m;
      S.l3s[e] = make_uint2(l[0] | (l[1] << 16), l[2] | (l[3] << 16));
    }

    for (int k0 = k_lo; k0 < k_hi; k0 += W) {
      const int nw = min(W, k_hi - k0), R1 = nw * n1, R2 = nw * n2, R3 = nw * n3;
      for (int i = tid; i < nw * FF; i += kTcThreads) S.win[i] = windows[(size_t)k0 * FF + i];
      __syncthreads();
      // ---- layer-1 input rows ----
      if (tid < R1) {  // one row per thread (R1 <= kCap1)
        const int w = (int)fdiv((uint32_t)tid, f1);
        const uint32_t pm = S.p1[tid - w * n1];
        const int8_t* at = S.win + w * FF + (int)(pm & 0xffffu);
        uint32_t v[9];  // (spin, known)
#pragma unroll
        for (int t = 0; t < 9; ++t) {
          v[t] = 0u;
          if (pm & (0x10000u << t))  // an int8 is exact in BF16
            v[t] = (__float_as_uint((float)at[(t / 3 - 1) * F + t % 3 - 1]) >> 16) | 0x3f800000u;
        }
        uint4* row = reinterpret_cast<uint4*>(S.x + tid * kXP);
        row[0] = make_uint4(v[0], v[1], v[2], v[3]);
        row[1] = make_uint4(v[4], v[5], v[6], v[7]);
        uint32_t* tail = reinterpret_cast<uint32_t*>(row + 2);
        tail[0] = tail[2] = tail[4] = v[8];
      }
      __syncthreads();
      const int u0 = warp * 32;  // this warp's unit of 32 layer-1 rows
      // ---- layer 1: h1 = relu(W1 * x + b1), W1 in three BF16 terms (exact products, FP32 sums) ----
      if (u0 < R1) {
        float acc[2][4][4] = {};
        uint32_t ax[2][2][4];  // columns 0 .. 15 and 16 .. 31 of two times 16 rows
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int k = 0; k < 2; ++k)
            ldm_x4_row(S.x + (u0 + m * 16 + (lane & 15)) * kXP + k * 16 + (lane >> 4) * 8, ax[m][k]);
        const __nv_bfloat16* wr =
            S.w1s + ((lane & 7) + ((lane >> 4) << 3)) * (kW1K + 8) + ((lane >> 3) & 1) * 8;
#pragma unroll
        for (int q = 3; q >= 0; --q) {  // taps 0 .. 7 last, their smallest term first
          uint32_t bw[8];
          ldm_x4(smem_addr(wr + q * 16), bw[0], bw[1], bw[2], bw[3]);
          ldm_x4(smem_addr(wr + q * 16 + 16 * (kW1K + 8)), bw[4], bw[5], bw[6], bw[7]);
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
              const uint32_t(&a)[4] = ax[m][q == 3 ? 1 : 0];
              mma_bf16(acc[m][nt], a[0], a[1], a[2], a[3], bw[2 * nt], bw[2 * nt + 1]);
            }
        }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            const int row = u0 + m * 16 + (lane >> 2) + half * 8;
            uint32_t pos = 0u;
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
              const int c = nt * 8 + (lane & 3) * 2;
              const __nv_bfloat162 h = __floats2bfloat162_rn(fmaxf(acc[m][nt][2 * half], 0.f),
                                                             fmaxf(acc[m][nt][2 * half + 1], 0.f));
              *reinterpret_cast<__nv_bfloat162*>(&S.h1[row * kCP + c]) = h;
              pos |= (bf(h.x) > 0.f ? 1u << c : 0u) | (bf(h.y) > 0.f ? 2u << c : 0u);
            }
            pos |= __shfl_xor_sync(0xffffffffu, pos, 1);
            pos |= __shfl_xor_sync(0xffffffffu, pos, 2);
            if ((lane & 3) == 0) S.mask[row] = row < R1 ? pos : 0u;
          }
      }
      __syncthreads();
      // ---- layer 2 forward on the tensor cores: units of 32 rows x 32 channels ----
      for (int r0 = warp * 32; r0 < R2; r0 += kTcWarps * 32) {
        float acc[2][4][4] = {};
        int e9[2], base[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int row = r0 + m * 16 + (lane & 15), w = (int)fdiv((uint32_t)row, f2);
          e9[m] = row < R2 ? (row - w * n2) * 9 : -1;
          base[m] = w * n1;
        }
        const __nv_bfloat16* b_base = S.w2f + ((lane & 7) + ((lane >> 4) << 3)) * kK2P + ((lane >> 3) & 1) * 8;
        int nx[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) nx[m] = e9[m] < 0 ? kNone : S.nb1[e9[m]];
#pragma unroll 1
        for (int t = 0; t < 9; ++t) {
          const __nv_bfloat16* ar[2];
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const int i = nx[m];
            if (t < 8 && e9[m] >= 0) nx[m] = S.nb1[e9[m] + t + 1];
            ar[m] = S.h1 + (i == kNone ? kCap1 : base[m] + i) * kCP + (lane >> 4) * 8;
          }
#pragma unroll
          for (int k = 0; k < kC; k += 16) {
            uint32_t av[2][4], bv[8];
            ldm_x4_row(ar[0] + k, av[0]);
            ldm_x4_row(ar[1] + k, av[1]);
            ldm_x4(smem_addr(b_base + t * kC + k), bv[0], bv[1], bv[2], bv[3]);
            ldm_x4(smem_addr(b_base + 16 * kK2P + t * kC + k), bv[4], bv[5], bv[6], bv[7]);
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
              for (int nt = 0; nt < 4; ++nt)
                mma_bf16(acc[m][nt], av[m][0], av[m][1], av[m][2], av[m][3], bv[2 * nt], bv[2 * nt + 1]);
          }
        }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            const int row = r0 + m * 16 + (lane >> 2) + half * 8;
            if (row >= R2) continue;
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
              const int o = nt * 8 + (lane & 3) * 2;
              *reinterpret_cast<__nv_bfloat162*>(&S.h2[row * kCP + o]) =
                  __floats2bfloat162_rn(fmaxf(acc[m][nt][2 * half] + S.b2[o], 0.f),
                                        fmaxf(acc[m][nt][2 * half + 1] + S.b2[o + 1], 0.f));
            }
          }
      }
      __syncthreads();
      // ---- layer 3 and the loss: eight lanes per site ----
      for (int base = warp * 4; base < R3; base += kTcWarps * 4) {
        const int si = base + (lane >> 3);
        const int sub = lane & 7, c0 = 4 * sub;
        float zz = 0.f;
        int w = 0, j = 0;
        if (si < R3) {
          w = (int)fdiv((uint32_t)si, f3);
          j = si - w * n3;
#pragma unroll
          for (int t = 0; t < 9; ++t) {
            const __nv_bfloat16* h = &S.h2[(w * n2 + S.nb4[j * 9 + t]) * kCP + c0];
            const float* w3 = &S.w3t[t * kC + c0];
            zz += w3[0] * bf(h[0]) + w3[1] * bf(h[1]) + w3[2] * bf(h[2]) + w3[3] * bf(h[3]);
          }
        }
        zz += __shfl_xor_sync(0xffffffffu, zz, 4);
        zz += __shfl_xor_sync(0xffffffffu, zz, 2);
        zz += __shfl_xor_sync(0xffffffffu, zz, 1);
        if (si < R3 && sub == 0) {
          zz += S.b3;
          const float y = S.win[w * FF + (l3[j] / B + 1) * F + l3[j] % B + 1] > 0 ? 1.f : 0.f;
          my_loss += (fmaxf(zz, 0.f) - zz * y + log1pf(expf(-fabsf(zz)))) * invn;
          const float g = (1.f / (1.f + expf(-zz)) - y) * invn;
          S.g3[si] = g;
          gb3s += g;
        }
      }
      __syncthreads();
      // ---- layer 3 gradients (FP32): lane = channel, one site per warp ----
      for (int si = warp; si < R3; si += kTcWarps) {
        const int w = (int)fdiv((uint32_t)si, f3), j = si - w * n3;
        const float g = S.g3[si];
#pragma unroll
        for (int t = 0; t < 9; ++t) gw3s[t] += g * bf(S.h2[(w * n2 + S.nb4[j * 9 + t]) * kCP + lane]);
      }
      // dL/dz2 = (W3^T g3) . (h2 > 0) in BF16, and its FP32 sum for the bias: eight lanes per row, four
      // channels each; a row next to at most four sites (every staged one) reads them from one list entry
      for (int r = warp * 4 + (lane >> 3); r < R2; r += kTcWarps * 4) {
        const int w = (int)fdiv((uint32_t)r, f2), e = r - w * n2, c0 = (lane & 7) * 4;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        auto add = [&](int t, int site) {
          const float4 w3 = *reinterpret_cast<const float4*>(&S.w3t[t * kC + c0]);
          const float g = S.g3[w * n3 + site];
          v.x += w3.x * g;
          v.y += w3.y * g;
          v.z += w3.z * g;
          v.w += w3.w * g;
        };
        const uint32_t m = S.m3[e];
        if (__popc(m) <= 4) {
          const uint2 l = S.l3s[e];
          const uint32_t x[4] = {l.x & 0xffffu, l.x >> 16, l.y & 0xffffu, l.y >> 16};
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (x[q] != kNone) add((int)(x[q] & 15u), (int)(x[q] >> 4));
        } else {
          for (uint32_t mm = m; mm; mm &= mm - 1) {
            const int t = __ffs(mm) - 1;
            add(t, S.nb3[e * 9 + t]);
          }
        }
        const uint2 h = *reinterpret_cast<const uint2*>(&S.h2[r * kCP + c0]);
        v.x = __uint_as_float(h.x << 16) > 0.f ? v.x : 0.f;
        v.y = __uint_as_float(h.x & 0xffff0000u) > 0.f ? v.y : 0.f;
        v.z = __uint_as_float(h.y << 16) > 0.f ? v.z : 0.f;
        v.w = __uint_as_float(h.y & 0xffff0000u) > 0.f ? v.w : 0.f;
        const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        *reinterpret_cast<uint2*>(&S.gz2[r * kCP + c0]) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
        gb2s.x += v.x;
        gb2s.y += v.y;
        gb2s.z += v.z;
        gb2s.w += v.w;
      }
      __syncthreads();
      // ---- weight gradient of layer 2 on the tensor cores: K = rows ----
      for (int p0 = my_half * 16; p0 < R2; p0 += 32) {
        // this lane's rows in the A (gz2^T) and B (h1) tiles; past the end: zero rows
        const int pa = p0 + (lane & 7) + ((lane >> 4) << 3), pb = p0 + (lane & 15);
        const int w = (int)fdiv((uint32_t)pb, f2);
        const uint16_t* nb = &S.nb1[(pb - w * n2) * 9];
        const int i = pb < R2 ? nb[my_tap] : kNone, i8 = pb < R2 ? nb[8] : kNone;
        uint32_t av[2][4], bv[8], b8[2];
        const __nv_bfloat16* ga = S.gz2 + (pa < R2 ? pa : kCap2) * kCP + ((lane >> 3) & 1) * 8;
        ldm_x4_t(smem_addr(ga), av[0][0], av[0][1], av[0][2], av[0][3]);
        ldm_x4_t(smem_addr(ga + 16), av[1][0], av[1][1], av[1][2], av[1][3]);
        const __nv_bfloat16* hb = S.h1 + (i == kNone ? kCap1 : w * n1 + i) * kCP + (lane >> 4) * 8;
        ldm_x4_t(smem_addr(hb), bv[0], bv[1], bv[2], bv[3]);
        ldm_x4_t(smem_addr(hb + 16), bv[4], bv[5], bv[6], bv[7]);
        ldm_x2_t(smem_addr(S.h1 + (i8 == kNone ? kCap1 : w * n1 + i8) * kCP + t8n * 8), b8[0], b8[1]);
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int nt = 0; nt < 4; ++nt)
            mma_bf16(dw[m * 4 + nt], av[m][0], av[m][1], av[m][2], av[m][3], bv[2 * nt], bv[2 * nt + 1]);
        const uint32_t* a8 = av[0];
        mma_bf16(dw[8], t8m ? av[1][0] : a8[0], t8m ? av[1][1] : a8[1], t8m ? av[1][2] : a8[2], t8m ? av[1][3] : a8[3],
                 b8[0], b8[1]);
      }
      // ---- input gradient of layer 2, transposed: D[c][q] = sum_{t,o} W2[o][c][t] gz2[q - d_t][o], one
      // unit of 32 rows q per warp; masked with h1 > 0 it is dL/dz1^T, whose accumulator layout is the A
      // operand of the layer-1 weight gradient dW1[c][j] += sum_q dL/dz1[q][c] x[q][j] ----
      if (u0 < R1) {
        float acc[2][4][4] = {};
        int e9[2], base[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int q = u0 + h * 16 + (lane & 7) + ((lane >> 4) << 3), w = (int)fdiv((uint32_t)q, f1);
          e9[h] = q < R1 ? (q - w * n1) * 9 : -1;
          base[h] = w * n2;
        }
        const __nv_bfloat16* a_base = S.w2f + ((lane & 7) + ((lane >> 4) << 3)) * kK2P + ((lane >> 3) & 1) * 8;
        int nx[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) nx[h] = e9[h] < 0 ? kNone : S.nb2[e9[h]];
#pragma unroll 1
        for (int t = 0; t < 9; ++t) {
          const __nv_bfloat16* br[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int i = nx[h];
            if (t < 8 && e9[h] >= 0) nx[h] = S.nb2[e9[h] + t + 1];
            br[h] = S.gz2 + (i == kNone ? kCap2 : base[h] + i) * kCP + ((lane >> 3) & 1) * 8;
          }
#pragma unroll
          for (int k = 0; k < kC; k += 16) {
            uint32_t av[2][4], bv[8];
            ldm_x4_t(smem_addr(a_base + k * kK2P + t * kC), av[0][0], av[0][1], av[0][2], av[0][3]);
            ldm_x4_t(smem_addr(a_base + k * kK2P + t * kC + 16), av[1][0], av[1][1], av[1][2], av[1][3]);
            ldm_x4(smem_addr(br[0] + k), bv[0], bv[1], bv[2], bv[3]);
            ldm_x4(smem_addr(br[1] + k), bv[4], bv[5], bv[6], bv[7]);
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
              for (int nt = 0; nt < 4; ++nt)
                mma_bf16(acc[m][nt], av[m][0], av[m][1], av[m][2], av[m][3], bv[2 * nt], bv[2 * nt + 1]);
          }
        }
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {  // 16 rows at a time
          uint32_t xb[6];
          const __nv_bfloat16* xr = S.x + (u0 + kk * 16 + (lane & 15)) * kXP;
          ldm_x4_t(smem_addr(xr + (lane >> 4) * 8), xb[0], xb[1], xb[2], xb[3]);
          ldm_x2_t(smem_addr(xr + 16), xb[4], xb[5]);
          uint2 mk[2];
#pragma unroll
          for (int h = 0; h < 2; ++h)
            mk[h] = *reinterpret_cast<const uint2*>(&S.mask[u0 + kk * 16 + h * 8 + (lane & 3) * 2]);
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            uint32_t a[4][3];  // A registers (rows g, g + 8; columns of tile 2 kk, 2 kk + 1), three terms each
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const float* d = acc[m][2 * kk + (r >> 1)] + 2 * (r & 1);
              const uint32_t bit = 1u << (m * 16 + (lane >> 2) + (r & 1) * 8);
              split3(mk[r >> 1].x & bit ? d[0] : 0.f, mk[r >> 1].y & bit ? d[1] : 0.f, a[r]);
            }
            // summed over the rows so far by FP32 additions: the accumulator of an mma is cut and not rounded,
            // which left 1.0e-5 of the gradient over 16384 windows and 8e-5 over 131072, rounded sums 2e-7
#pragma unroll
            for (int nt = 0; nt < 3; ++nt) {
              float d[4] = {};
#pragma unroll
              for (int q = 2; q >= 0; --q)
                mma_bf16(d, a[0][q], a[1][q], a[2][q], a[3][q], xb[2 * nt], xb[2 * nt + 1]);
#pragma unroll
              for (int e = 0; e < 4; ++e) dw1[m][nt][e] += d[e];
            }
          }
        }
      }
      __syncthreads();
    }
  }
  // add this CTA's sums to the global gradient: the warps' sums meet in shared
  // memory (the h1 and h2 buffers)
  const int g = lane >> 2, t2 = (lane & 3) * 2;
  float* red = reinterpret_cast<float*>(S.h1);
  if (my_half == 1) {
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
      for (int e = 0; e < 4; ++e) red[((my_tap * 9 + q) * 4 + e) * 32 + lane] = dw[q][e];
  }
  __syncthreads();
  if (my_half == 0) {
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float v = dw[q][e] + red[((my_tap * 9 + q) * 4 + e) * 32 + lane];
        const int m = q < 8 ? q >> 2 : t8m, nt = q < 8 ? q & 3 : t8n, t = q < 8 ? my_tap : 8;
        const int o = m * 16 + g + (e >> 1) * 8, c = nt * 8 + t2 + (e & 1);
        if (v != 0.f) atomicAdd(&grads[kOffW2 + (o * kC + c) * 9 + t], v);
      }
  }
  __syncthreads();
  float* mine = red + warp * kRed * kC;
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int nt = 0; nt < 3; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int c = m * 16 + g + (e >> 1) * 8, j = nt * 8 + t2 + (e & 1);  // column j = 2 t + ci
        if (j < 19) mine[(j == 18 ? 18 : (j & 1) * 9 + (j >> 1)) * kC + c] = dw1[m][nt][e];
      }
#pragma unroll
  for (int o = 8; o <= 16; o <<= 1) {
    gb2s.x += __shfl_xor_sync(0xffffffffu, gb2s.x, o);
    gb2s.y += __shfl_xor_sync(0xffffffffu, gb2s.y, o);
    gb2s.z += __shfl_xor_sync(0xffffffffu, gb2s.z, o);
    gb2s.w += __shfl_xor_sync(0xffffffffu, gb2s.w, o);
  }
  if (lane < 8) *reinterpret_cast<float4*>(&mine[19 * kC + 4 * lane]) = gb2s;
#pragma unroll
  for (int t = 0; t < 9; ++t) mine[(20 + t) * kC + lane] = gw3s[t];
  __syncthreads();
  for (int i = tid; i < 29 * kC; i += kTcThreads) {
    float v = 0.f;
    for (int w = 0; w < kTcWarps; ++w) v += red[w * kRed * kC + i];
    const int j = i / kC, c = i % kC;
    const int at = j < 18 ? kOffW1 + c * 18 + j : j == 18 ? kOffB1 + c : j == 19 ? kOffB2 + c : kOffW3 + c * 9 + j - 20;
    if (v != 0.f) atomicAdd(&grads[at], v);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    my_loss += __shfl_xor_sync(0xffffffffu, my_loss, o);
    gb3s += __shfl_xor_sync(0xffffffffu, gb3s, o);
  }
  if (lane == 0) {
    atomicAdd(loss, my_loss);
    if (gb3s != 0.f) atomicAdd(&grads[kOffB3], gb3s);
  }
}

}  // namespace

size_t nn_train_tc_smem() { return sizeof(TrainTcSmem); }

cudaError_t nn_train_tc(const int8_t* windows, int count, const StagedPlan* d_plan,
                        const float* params, float* grads, float* loss, int grid, cudaStream_t s) {
  static DeviceCache attr;
  if (!attr.get()) {
    cudaError_t e = cudaFuncSetAttribute(k_nn_train_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(TrainTcSmem));
    if (e) return e;
    attr.set(1);
  }
  // every SM, also for fewer samples: the finer the ranges, the fewer CTAs take windows of two
  // stages and build two sets of tables (8 windows of 8 x 8 blocks 78.6 -> 66 us); the rest leave at once
  k_nn_train_tc<<<grid, kTcThreads, sizeof(TrainTcSmem), s>>>(windows, count, d_plan, params, grads, loss);
  return cudaGetLastError();
}

}  // namespace nnc
}  // namespace ising
