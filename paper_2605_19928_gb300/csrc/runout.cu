// All-in run-outs evaluated in one step: the win-minus-loss tables E and the values
// u E q at each run-out's top node (see runout.h).
#include <cuda_runtime.h>

#include <cstdint>

#include "runout.h"

namespace pcfr {
namespace {

constexpr int kBuildThreads = 256;

// Thread (o, h) of table blockIdx.z: E[h][o] over the table's boards, stored at [o][h] with
// the table's bias (padding hands h >= n_hands hold E = 0).
__global__ void __launch_bounds__(kBuildThreads) k_runout_build(const RunoutTable* __restrict__ tables,
                                                                const RunoutBoard* __restrict__ boards,
                                                                const int32_t* __restrict__ gs,
                                                                const uint64_t* __restrict__ hand_mask, int H,
                                                                int ld, unsigned char* __restrict__ pool) {
  const RunoutTable tb = tables[blockIdx.z];
  const int o = blockIdx.y, h = blockIdx.x * kBuildThreads + threadIdx.x;
  if (h >= ld) return;
  int e = 0;
  if (h < H) {
    const uint64_t mo = hand_mask[o], mh = hand_mask[h];
    if (!(mo & mh)) {
      for (int b = 0; b < tb.n_boards; ++b) {
        const RunoutBoard bd = boards[tb.board0 + b];
        if (bd.cards & (mo | mh)) continue;  // a card of the board is in one of the hands
        const int32_t* g = gs + (size_t)bd.table * H;
        const int d = g[h] - g[o];
        e += (d > 0) - (d < 0);
      }
    }
  }
  const size_t at = (size_t)o * ld + h;
  if (tb.wide)
    reinterpret_cast<uint16_t*>(pool + tb.offset)[at] = (uint16_t)(e + 32768);
  else
    pool[tb.offset + at] = (uint8_t)(e + 128);
}

// Values at the run-outs' top nodes: v(h) = u sum_o E[h][o] q(o), each (top, hand) one chain of
// FP32 FMAs over o in order.  Bound: the FP32 pipe (2 H^2 operations a top; the tables come from
// L2).  What the layout is for:
//   * a thread holds 4 hands x kTops tops of sums, so a table row's 4 entries (one load, turned
//     into floats exactly by placing them in the mantissa of 2^23) serve 4 x kTops FMAs;
//   * the FMAs are packed pairs (fma.rn.f32x2: the two hands of a pair are independent chains), so
//     the issue slots they leave carry the loads and conversions; q is staged doubled, (q, q), so
//     a broadcast load gives two tops' pair operands;
//   * table rows are loaded kAhead rows ahead, because a row's L2 latency is many times the
//     cycles its FMAs take, and q in chunks of kChunk rows, one chunk ahead;
//   * two warps a block: 980 blocks of the 1,470 turn tops spread over 152 SMs within 8 % of even.
// The few tops on 16-bit tables (flop all-ins: 10) would leave most SMs idle at 8 tops a thread:
// they take 2 tops a thread, and their blocks come first in the same launch, so that their
// longer chains run beside the others'.
// Measured on the 1176-hand flop (1,470 turn tops, 10 flop tops, one player): 350 + 340 us as two
// launches of 4-hand, 8-top threads loading two rows ahead; about 185 us as one launch of this form.
constexpr int kValueThreads = 64;  // 4 hands a thread: 256 hands a block
constexpr int kChunk = 64;         // opponent hands staged at a time (one a thread)
constexpr int kAhead = 8;          // table rows in flight per thread
static_assert(2 * kAhead <= kRunoutPadRows, "rows loaded past a table's end stay in the pool");
constexpr int kTops8 = kRunoutGroup, kTops16 = 2, kSubs16 = kRunoutGroup / kTops16;
static_assert(kChunk == kValueThreads && kChunk % kAhead == 0, "one staged hand per thread");

using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float2 unpack2(f32x2 x) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(x));
  return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Four entries of a table row; entries() gives them as two exact pairs of floats: the biased
// integer x goes into the mantissa of 2^23, then 2^23 and the bias come off in one exact step.
template <typename T>
struct Row4;
template <>
struct Row4<uint8_t> {
  uint32_t w;
  static __device__ __forceinline__ Row4 load(const uint8_t* p) { return {__ldg(reinterpret_cast<const uint32_t*>(p))}; }
  __device__ __forceinline__ void entries(f32x2& a, f32x2& b) const {
    const f32x2 off = pack2(-(8388608.f + 128.f), -(8388608.f + 128.f));
    a = add2(pack2(__uint_as_float(__byte_perm(w, 0x4b000000u, 0x7440)), __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7441))), off);
    b = add2(pack2(__uint_as_float(__byte_perm(w, 0x4b000000u, 0x7442)), __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7443))), off);
  }
};
template <>
struct Row4<uint16_t> {
  uint2 w;
  static __device__ __forceinline__ Row4 load(const uint16_t* p) { return {__ldg(reinterpret_cast<const uint2*>(p))}; }
  __device__ __forceinline__ void entries(f32x2& a, f32x2& b) const {
    const f32x2 off = pack2(-(8388608.f + 32768.f), -(8388608.f + 32768.f));
    a = add2(pack2(__uint_as_float(__byte_perm(w.x, 0x4b000000u, 0x7410)), __uint_as_float(__byte_perm(w.x, 0x4b000000u, 0x7432))), off);
    b = add2(pack2(__uint_as_float(__byte_perm(w.y, 0x4b000000u, 0x7410)), __uint_as_float(__byte_perm(w.y, 0x4b000000u, 0x7432))), off);
  }
};

// One step of the chains: E's row for opponent hand o times the tops' (q, q) at o.
template <typename T, int kTops>
__device__ __forceinline__ void runout_step(const Row4<T>& row, const ulonglong2* __restrict__ q, f32x2 (&acc)[kTops][2]) {
  f32x2 e0, e1;
  row.entries(e0, e1);
#pragma unroll
  for (int g = 0; g < kTops; g += 2) {
    const ulonglong2 qq = q[g / 2];
    acc[g][0] = fma2(e0, qq.x, acc[g][0]);
    acc[g][1] = fma2(e1, qq.x, acc[g][1]);
    acc[g + 1][0] = fma2(e0, qq.y, acc[g + 1][0]);
    acc[g + 1][1] = fma2(e1, qq.y, acc[g + 1][1]);
  }
}

// Tops items[0 .. count) (count <= kTops) of one table for this thread's hands h0 .. h0 + 3.
template <typename T, int kTops>
__device__ __forceinline__ void runout_tops(const GameDev& G, const RunoutItem* __restrict__ items, int count,
                                            const T* __restrict__ table, int h0, const float* __restrict__ reach,
                                            const int32_t* __restrict__ reach_row, float* __restrict__ out,
                                            ulonglong2* qs) {
  const int H = G.n_hands, tid = threadIdx.x;
  const size_t S = (size_t)G.hstride;
  const uint32_t ld = (uint32_t)S;
  uint32_t at = h0 < H ? (uint32_t)h0 : 0u;  // a thread past the hands computes hand 0's and drops them
  const float* src[kTops];
#pragma unroll
  for (int g = 0; g < kTops; ++g) src[g] = reach + (size_t)reach_row[items[g < count ? g : 0].node] * S;
  f32x2 acc[kTops][2];
#pragma unroll
  for (int g = 0; g < kTops; ++g) acc[g][0] = acc[g][1] = 0ull;
  float q[kTops];
  auto fetch = [&](int o) {
#pragma unroll
    for (int g = 0; g < kTops; ++g) q[g] = o < H && g < count ? src[g][o] : 0.f;
  };
  auto stage = [&](int buf) {
    ulonglong2* dst = qs + (size_t)(buf * kChunk + tid) * (kTops / 2);
#pragma unroll
    for (int g = 0; g < kTops; g += 2) dst[g / 2] = make_ulonglong2(pack2(q[g], q[g]), pack2(q[g + 1], q[g + 1]));
  };
  // rows past the last are loaded too (the pool has kRunoutPadRows rows of slack) and not used
  Row4<T> row[kAhead], next[kAhead];
  auto rows = [&](Row4<T> (&r)[kAhead]) {
#pragma unroll
    for (int k = 0; k < kAhead; ++k, at += ld) r[k] = Row4<T>::load(table + at);
  };
  rows(row);
  fetch(tid);
  stage(0);
  __syncthreads();
  for (int c0 = 0, buf = 0; c0 < H; c0 += kChunk, buf ^= 1) {
    if (c0 + kChunk < H) fetch(c0 + kChunk + tid);
    const ulonglong2* qc = qs + (size_t)buf * kChunk * (kTops / 2);
    const int n = min(kChunk, H - c0);
    for (int k0 = 0; k0 + kAhead <= n; k0 += kAhead) {
      rows(next);
#pragma unroll
      for (int k = 0; k < kAhead; ++k) runout_step<T, kTops>(row[k], qc + (k0 + k) * (kTops / 2), acc);
#pragma unroll
      for (int k = 0; k < kAhead; ++k) row[k] = next[k];
    }
    if (n % kAhead) {  // the last chunk's last rows
      const int k0 = n - n % kAhead;
#pragma unroll
      for (int k = 0; k < kAhead - 1; ++k)
        if (k < n % kAhead) runout_step<T, kTops>(row[k], qc + (k0 + k) * (kTops / 2), acc);
    }
    if (c0 + kChunk < H) stage(buf ^ 1);  // its readers finished before the last barrier
    __syncthreads();
  }
  if (h0 >= H) return;
#pragma unroll
  for (int g = 0; g < kTops; ++g) {
    if (g >= count) break;
    const RunoutItem it = items[g];
    float* dst = out + (size_t)it.node * S + h0;
    const float2 a = unpack2(acc[g][0]), b = unpack2(acc[g][1]);
    const float4 v = make_float4(it.u * a.x, it.u * a.y, it.u * b.x, it.u * b.y);
    if (h0 + 4 <= H) {  // rows start 128-byte aligned and h0 is a multiple of 4
      *reinterpret_cast<float4*>(dst) = v;
    } else {
      dst[0] = v.x;
      if (h0 + 1 < H) dst[1] = v.y;
      if (h0 + 2 < H) dst[2] = v.z;
    }
  }
}

// Blocks: (16-bit group, sub-group of kTops16 tops, hand block), then (8-bit group, hand block);
// blockIdx.y the player.
__global__ void __launch_bounds__(kValueThreads) k_runout_values(const GameDev* __restrict__ games,
                                                                 const RunoutItem* __restrict__ items,
                                                                 const RunoutGroup* __restrict__ groups8,
                                                                 const RunoutGroup* __restrict__ groups16, int n16,
                                                                 const RunoutTable* __restrict__ tables,
                                                                 const unsigned char* __restrict__ pool,
                                                                 const int32_t* __restrict__ row0,
                                                                 const int32_t* __restrict__ row1, int hand_blocks,
                                                                 int player_mask, int use_bar) {
  __shared__ __align__(16) ulonglong2 qs[2 * kChunk * kTops8 / 2];
  const GameDev& G = games[0];
  const int i = player_mask == 3 ? (int)blockIdx.y : (player_mask == 1 ? 0 : 1);
  const size_t S = (size_t)G.hstride, N = (size_t)G.n_nodes;
  const float* reach = static_cast<const float*>(use_bar ? G.reach_bar : G.reach) + (size_t)(1 - i) * N * S;
  float* out = static_cast<float*>(use_bar ? G.cfv_br : G.cfv) + (size_t)i * N * S;
  int b = blockIdx.x;
  const int blocks16 = n16 * kSubs16 * hand_blocks;
  if (b < blocks16) {
    const int h0 = 4 * ((b % hand_blocks) * kValueThreads + (int)threadIdx.x);
    b /= hand_blocks;
    const RunoutGroup gr = groups16[b / kSubs16];
    const int first = (b % kSubs16) * kTops16, count = min(gr.count - first, kTops16);
    if (count > 0)
      runout_tops<uint16_t, kTops16>(G, items + gr.item0 + first, count,
                                     reinterpret_cast<const uint16_t*>(pool + tables[gr.table].offset), h0, reach, i ? row0 : row1, out, qs);
  } else {
    b -= blocks16;
    const int h0 = 4 * ((b % hand_blocks) * kValueThreads + (int)threadIdx.x);
    const RunoutGroup gr = groups8[b / hand_blocks];
    runout_tops<uint8_t, kTops8>(G, items + gr.item0, gr.count, pool + tables[gr.table].offset, h0, reach, i ? row0 : row1, out, qs);
  }
}

}  // namespace

int launch_runout_build(const RunoutTable* tables, int n_tables, const RunoutBoard* boards, const int32_t* gs,
                        const uint64_t* hand_mask, int n_hands, int hstride, unsigned char* pool, void* stream) {
  if (n_tables == 0) return 0;
  const dim3 grid((unsigned)((hstride + kBuildThreads - 1) / kBuildThreads), (unsigned)n_hands, (unsigned)n_tables);
  k_runout_build<<<grid, kBuildThreads, 0, (cudaStream_t)stream>>>(tables, boards, gs, hand_mask, n_hands, hstride,
                                                                  pool);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_runout_values(const GameDev* games, const RunoutItem* items, const RunoutGroup* groups8, int n8,
                         const RunoutGroup* groups16, int n16, const RunoutTable* tables, const unsigned char* pool,
                         const int32_t* row0, const int32_t* row1, int n_hands, int player_mask, int use_bar,
                         void* stream) {
  if (n8 + n16 == 0) return 0;
  const int hand_blocks = (n_hands + 4 * kValueThreads - 1) / (4 * kValueThreads);
  const dim3 grid((unsigned)((n16 * kSubs16 + n8) * hand_blocks), player_mask == 3 ? 2u : 1u);
  k_runout_values<<<grid, kValueThreads, 0, (cudaStream_t)stream>>>(games, items, groups8, groups16, n16, tables, pool,
                                                                   row0, row1, hand_blocks, player_mask, use_bar);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace pcfr
