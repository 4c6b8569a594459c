// Gate of the MoE layer (paper Sec. 2.1 / Sec. 4.1: the gate yields each token's routed expert
// ids and gate scores), token->expert permutation, and the integer numerators of the expert
// reuse priority (Sec. 4.3 priority equation).
//
// Everything a keep/evict or routing decision depends on is computed in a fixed operation
// order so that it can be reproduced bit for bit elsewhere:
//   * logit(t,e): 32 chains, lane q owns h with (h/8) mod 32 == q, ascending h, one fused
//     multiply-add per term (bf16*bf16 is exact in fp32, so the fma rounds once, like a plain
//     add of the exact product); butterfly over xor distances 16,8,4,2,1; bias one rounded add.
//   * top-k: logit descending, ties to the lower expert index (a NaN logit counts as -inf).
//   * gate scores: z_j = exp_spec(L_j - L_0); S = ((z_0+z_1)+z_2)...; g_j = z_j / S.
//   * score numerators: v = g * psi(c) rounded once; floor(v * 2^32) summed as integers.
// The router stays off the tensor cores on purpose: their accumulation order is unspecified.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>

#include "kernels.h"
#include "fp8_split.h"
#include "route_math.h"

namespace oled {
namespace {

// Top-k (ties to the lower index), gate scores over the selected logits, counts and integer
// reuse-score numerators of one token; executed by one warp.  row: the token's E logits.
template <int kMaxEPerLane>  // E <= 32 * kMaxEPerLane: bounds the per-lane candidate scan
__device__ __forceinline__ void route_token_tail_n(const float* row, int t, int lane, int E, int K,
                                                 const float* __restrict__ conf, int32_t* __restrict__ ids,
                                                 float* __restrict__ gate, int32_t* __restrict__ counts,
                                                 unsigned long long* __restrict__ scores) {
    float v[kMaxEPerLane];
#pragma unroll
    for (int i = 0; i < kMaxEPerLane; ++i) {
      const int e = lane + 32 * i;
      const float x = e < E ? row[e] : 0.0f;
      // a NaN logit is read as -inf: the order stays total; -0 becomes +0 (they compare equal)
      v[i] = (x == x) ? __fadd_rn(x, 0.0f) : __int_as_float(0xff800000);
    }
    float c = conf[t];  // (arrives during the selection)
    uint32_t used = 0;
    int my_id = 0;
    float my_logit = 0.0f;
    for (int r = 0; r < K; ++r) {
      float bv = 0.0f;
      int be = 0x7fffffff;
#pragma unroll
      for (int i = 0; i < kMaxEPerLane; ++i) {
        const int e = lane + 32 * i;
        if (e < E && !((used >> i) & 1u)) {
          if (be == 0x7fffffff || v[i] > bv) {  // ascending e: strict > keeps the lower index
            bv = v[i];
            be = e;
          }
        }
      }
      // the warp's best: largest logit, then lowest index - two integer warp reductions (the logit
      // as an order-preserving unsigned key; a lane without a candidate holds key 0, below every
      // logit's key) and one broadcast of the winning logit
      const uint32_t bits = __float_as_uint(bv);
      const uint32_t key = be == 0x7fffffff ? 0u : ((bits & 0x80000000u) ? ~bits : (bits | 0x80000000u));
      const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
      be = (int)__reduce_min_sync(0xffffffffu, key == kmax ? (uint32_t)be : 0x7fffffffu);
      bv = __shfl_sync(0xffffffffu, bv, be & 31);
      if ((be & 31) == lane) used |= 1u << (be >> 5);
      if (lane == r) {
        my_id = be;
        my_logit = bv;
      }
    }
    const float top = __shfl_sync(0xffffffffu, my_logit, 0);
    const float z = lane < K ? exp_spec(__fsub_rn(my_logit, top)) : 0.0f;
    float s = __shfl_sync(0xffffffffu, z, 0);
    for (int j = 1; j < K; ++j) s = __fadd_rn(s, __shfl_sync(0xffffffffu, z, j));
    if (lane < K) {
      const float g = __fdiv_rn(z, s);
      ids[(size_t)t * K + lane] = my_id;
      gate[(size_t)t * K + lane] = g;
      c = (c != c) ? 0.0f : fminf(fmaxf(c, 0.0f), 1.0f);  // psi(c) = c, clamped; NaN -> 0
      const float pv = __fmul_rn(g, c);
      // a NaN product (non-finite activations) adds nothing; the 64-bit conversion of a NaN
      // would return 2^63
      const unsigned long long q = (pv == pv) ? __float2ull_rz(__fmul_rn(pv, 4294967296.0f)) : 0ull;
      atomicAdd(&counts[my_id], 1);
      atomicAdd(&scores[my_id], q);
    }
  }

// The same selection whatever the bound: a tighter bound only drops candidates that do not exist.
__device__ __forceinline__ void route_token_tail(const float* row, int t, int lane, int E, int K,
                                                 const float* __restrict__ conf, int32_t* __restrict__ ids,
                                                 float* __restrict__ gate, int32_t* __restrict__ counts,
                                                 unsigned long long* __restrict__ scores) {
  if (E <= 64) route_token_tail_n<2>(row, t, lane, E, K, conf, ids, gate, counts, scores);
  else if (E <= 128) route_token_tail_n<4>(row, t, lane, E, K, conf, ids, gate, counts, scores);
  else route_token_tail_n<OLED_MAX_EXPERTS / 32>(row, t, lane, E, K, conf, ids, gate, counts, scores);
}

// The previous layer's gate-weighted combine and residual, done by the gate kernel of the next
// layer for its own token (paper Sec. 2.1: the MoE output is the gate-score-weighted sum over the
// top-k experts; the stack adds it to the layer's input).  Arithmetic and order are those of
// combine_kernel: fp32 fused multiply-adds in rank order, out = bf16(sum), x = bf16(x_prev + out).
// n_rows tokens t0 .. t0 + n_rows - 1; their rows end up in s_x[row][H] as well, and in dense[t][H] where
// that is given.  Everything a thread needs for its columns - the rows of eight assignments, the gate
// scores, the residual - is requested at once: the kernel's time is its chain of memory round trips (with
// the gate scores fetched first this phase took 3.0 us at one token, 5.5 us at sixteen).
// kItems: groups of four columns in flight per thread (CTAs of several tokens).
template <int kItems>
__device__ __forceinline__ void combine_rows(const CombinePrev& p, int t0, int n_rows, int H, uint16_t* s_x,
                                             uint16_t* dense) {
  const int K = p.K, lane = threadIdx.x & 31;
  const int quads = H / 4, total = n_rows * quads;  // (a warp's 32 quads lie in one row: H is a multiple of 256)
  for (int i0 = (int)threadIdx.x; i0 < total; i0 += kItems * (int)blockDim.x) {
    float4 acc[kItems], v[kItems][8];
    uint2 xv[kItems];
    float g[kItems];
    size_t off[kItems];  // of the quad in a [T][H] array
    for (int j0 = 0; j0 < K; j0 += 8) {
#pragma unroll
      for (int u = 0; u < kItems; ++u) {
        const int i = i0 + u * (int)blockDim.x;
        if (i >= total) continue;  // (whole warps)
        const int row = i / quads, t = t0 + row, h = (i - row * quads) * 4;
        if (j0 == 0) {
          off[u] = (size_t)t * H + h;
          acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
          xv[u] = *reinterpret_cast<const uint2*>(p.x + off[u]);
          g[u] = lane < K ? p.gate[(size_t)t * K + lane] : 0.f;
        }
        int r = t * K + j0;
        int rr = 0;
        if (p.pos != nullptr) rr = lane < K ? p.pos[(size_t)t * K + lane] : 0;
#pragma unroll
        for (int jj = 0; jj < 8; ++jj)
          if (j0 + jj < K) {
            const int y_row = p.pos != nullptr ? __shfl_sync(0xffffffffu, rr, j0 + jj) : r + jj;
            v[u][jj] = *reinterpret_cast<const float4*>(p.y + (size_t)y_row * H + h);
          }
      }
#pragma unroll
      for (int u = 0; u < kItems; ++u) {
        if (i0 + u * (int)blockDim.x >= total) continue;
#pragma unroll
        for (int jj = 0; jj < 8; ++jj)
          if (j0 + jj < K) {
            const float gj = __shfl_sync(0xffffffffu, g[u], j0 + jj);
            acc[u].x = fmaf(gj, v[u][jj].x, acc[u].x);
            acc[u].y = fmaf(gj, v[u][jj].y, acc[u].y);
            acc[u].z = fmaf(gj, v[u][jj].z, acc[u].z);
            acc[u].w = fmaf(gj, v[u][jj].w, acc[u].w);
          }
      }
    }
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
      if (i0 + u * (int)blockDim.x >= total) continue;
      __nv_bfloat162 lo = __floats2bfloat162_rn(acc[u].x, acc[u].y);
      __nv_bfloat162 hi = __floats2bfloat162_rn(acc[u].z, acc[u].w);
      uint2 pk;
      pk.x = *reinterpret_cast<uint32_t*>(&lo);
      pk.y = *reinterpret_cast<uint32_t*>(&hi);
      *reinterpret_cast<uint2*>(p.out + off[u]) = pk;
      const float2 o0 = __bfloat1622float2(lo), o1 = __bfloat1622float2(hi);
      __nv_bfloat162 r0 = __floats2bfloat162_rn(__uint_as_float(xv[u].x << 16) + o0.x,
                                                __uint_as_float(xv[u].x & 0xffff0000u) + o0.y);
      __nv_bfloat162 r1 = __floats2bfloat162_rn(__uint_as_float(xv[u].y << 16) + o1.x,
                                                __uint_as_float(xv[u].y & 0xffff0000u) + o1.y);
      uint2 rk;
      rk.x = *reinterpret_cast<uint32_t*>(&r0);
      rk.y = *reinterpret_cast<uint32_t*>(&r1);
      *reinterpret_cast<uint2*>(p.x_next + off[u]) = rk;
      if (dense != nullptr) *reinterpret_cast<uint2*>(dense + off[u]) = rk;
      *reinterpret_cast<uint2*>(s_x + (off[u] - (size_t)t0 * H)) = rk;
    }
  }
}

// What the allocation-free routing entry point adds to the gate kernel: the counts, offsets and the stable permutation, by
// the gate kernel's CTA where there is one, else by a kernel of one CTA behind it (sort_kernel).
struct RouteFinish {
  int32_t* offsets = nullptr;  // nullptr: a gate kernel of a step
  int32_t* perm = nullptr;
};
// counts[E], offsets[E + 1] and the stable permutation by expert of n assignments, by one CTA of WARPS warps (E at most
// one expert per thread; a number that names no expert is passed over).  Every warp counts the experts of a contiguous part of the list, the counts are scanned over
// (expert, warp), and every warp hands out its part's rows in order.  s_hist: [WARPS][E].
template <int WARPS>
__device__ __forceinline__ void sort_assignments(const int32_t* ids, int n, int E, int32_t* __restrict__ counts,
                                                 int32_t* __restrict__ offsets, int32_t* __restrict__ perm, int* s_hist) {
  static_assert(WARPS * 32 >= OLED_MAX_EXPERTS, "a thread per expert");
  __shared__ int s_warp[WARPS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < WARPS * E; i += WARPS * 32) s_hist[i] = 0;
  __syncthreads();
  const int part = (n + WARPS * 32 - 1) / (WARPS * 32) * 32, first = warp * part, last = min(n, first + part);
  int* const hist = s_hist + warp * E;
  for (int i0 = first; i0 < last; i0 += 32) {
    int id = i0 + lane < last ? __ldcg(ids + i0 + lane) : -1;
    if ((unsigned)id >= (unsigned)E) id = -1;
    const uint32_t same = __match_any_sync(0xffffffffu, id);
    if (id >= 0 && lane == __ffs((int)same) - 1) hist[id] += __popc(same);
    __syncwarp();
  }
  __syncthreads();
  const int e = threadIdx.x;
  int total = 0;
  if (e < E)
    for (int w = 0; w < WARPS; ++w) {
      const int c = s_hist[w * E + e];
      s_hist[w * E + e] = total;
      total += c;
    }
  int incl = total;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  int before = incl - total;
  for (int w = 0; w < warp; ++w) before += s_warp[w];
  if (e < E) {
    counts[e] = total;
    offsets[e] = before;
    if (e == E - 1) offsets[E] = before + total;
    for (int w = 0; w < WARPS; ++w) s_hist[w * E + e] += before;
  }
  __syncthreads();
  for (int i0 = first; i0 < last; i0 += 32) {
    int id = i0 + lane < last ? __ldcg(ids + i0 + lane) : -1;
    if ((unsigned)id >= (unsigned)E) id = -1;
    const uint32_t same = __match_any_sync(0xffffffffu, id);
    const int rank = __popc(same & ((1u << lane) - 1u));
    if (id >= 0) perm[hist[id] + rank] = i0 + lane;
    __syncwarp();
    if (id >= 0 && rank == 0) hist[id] += __popc(same);
    __syncwarp();
  }
}

// Chunks of the router matrix that wait in registers (kAhead; the combine of two tokens has no registers left for them).
__host__ __device__ constexpr int router_tail(int tt) { return tt == 1 ? 2 : 0; }
// TT tokens per CTA, WARPS warps; each warp owns kEPerWarp experts per pass and all TT tokens.  Small
// blocks use TT = 1 with 16 warps (one pass covers 64 experts) and keep several 256-wide
// chunks of loads in flight; the chain order of every logit is the same in all variants.
// TT <= 4 (few-token steps): the tokens' rows are staged in shared memory - copied from x, or
// produced by the previous layer's combine (prev.y != nullptr), which this kernel then carries
// out for its tokens - and the top-k is a rank computation spread over all warps: expert e is
// selected iff fewer than K experts precede it in the order (logit descending, index ascending)
// - the same total order a round-by-round selection walks.
// One token per CTA while that gives at most one wave of CTAs; two or four beyond (every CTA
// streams the whole router matrix, so a second wave costs as much as the first).
// kAhead: the router matrix is on chip before the input is there, `ahead` chunks of 256 columns in shared memory and what is
// left, at most router_tail() chunks, in registers (router_chunks_ahead() says when; never in routing without a step, whose
// matrix is the caller's and may still be in the making).
// The kernel reports nothing to the host: the step's first FFN launch, which starts when it has completed,
// publishes the finished counts and scores without any ticket or fence.
template <int TT, int WARPS, int UNROLL, int kEPerWarp, bool kAhead = false>
__global__ void __launch_bounds__(WARPS * 32, 1)
route_kernel(const uint16_t* __restrict__ x, const uint16_t* __restrict__ wr,
             const float* __restrict__ bias, const float* __restrict__ conf, int T, int H, int E,
             int K, float* __restrict__ logits_out, int32_t* __restrict__ ids,
             float* __restrict__ gate, int32_t* __restrict__ counts,
             unsigned long long* __restrict__ scores, CombinePrev prev, StepTimeline* timeline,
             const __grid_constant__ ScatterRows scatter, const __grid_constant__ RouteFinish finish, int ahead) {
  extern __shared__ __align__(16) uint8_t s_dyn[];
  float* s_logits = reinterpret_cast<float*>(s_dyn);                       // [TT][E]
  constexpr bool staged = TT <= 4;
  constexpr int kST = staged ? TT : 1;
  // [TT][H] (staged forms only), on a 16-byte boundary: rows are moved with 16-byte vector accesses
  uint16_t* s_x = reinterpret_cast<uint16_t*>(s_dyn + (((size_t)TT * E * 4 + 15) & ~(size_t)15));
  // [TT][Ep] (staged forms only): the logits as order-preserving keys, rows padded with zeros, below every key
  const int Ep = (E + 3) & ~3;
  uint32_t* s_key = reinterpret_cast<uint32_t*>(s_x + (size_t)TT * H);
  __shared__ int s_sel_id[kST][OLED_MAX_TOPK];
  __shared__ float s_sel_logit[kST][OLED_MAX_TOPK];
  __shared__ int s_r[kST * OLED_MAX_TOPK];
  __shared__ float s_conf[kST];
  __shared__ uint32_t s_amax[kST];  // fp8 stores: the rows' largest magnitudes (bf16 bits)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t0 = blockIdx.x * TT;
  griddep_launch_dependents();
  if (threadIdx.x == 0) timeline_entry(timeline, 0);
  constexpr int kRouteWarps = WARPS;
  const int my_tokens = min(TT, T - t0);
  // The router matrix does not depend on the predecessor (the previous layer's expert FFN, which a CTA of this kernel
  // usually waits 4 to 8 us for).  What bounds the logits otherwise is one SM's share of L2, 64 bytes a cycle: 64 experts x
  // 2048 took 3.4-3.6 us after the input was there, from chip 2.6.
  // [E][ahead * 256], a row's 512 bytes of a chunk are read by a warp at a time
  uint16_t* const s_w = reinterpret_cast<uint16_t*>(s_key + (size_t)TT * Ep);
  const int w_cols = ahead * 256;
  constexpr int kTail = kAhead ? router_tail(TT) : 0;
  uint4 w_tail[kTail == 0 ? 1 : kTail][kEPerWarp];
  if (kAhead) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_w);
    const int pieces = w_cols / 8;  // of 16 bytes, per row
    for (int e = warp; e < E; e += kRouteWarps)
      for (int c = lane; c < pieces; c += 32)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)(e * pieces + c) * 16u),
                     "l"(wr + (size_t)e * H + c * 8)
                     : "memory");
#pragma unroll
    for (int i = 0; i < kTail; ++i)
#pragma unroll
      for (int b = 0; b < kEPerWarp; ++b)
        if (w_cols + i * 256 < H)
          w_tail[i][b] = *reinterpret_cast<const uint4*>(wr + (size_t)min(warp * kEPerWarp + b, E - 1) * H + w_cols + i * 256 + lane * 8);
  } else if (staged && gridDim.x <= 148) {
    // into L2, out of which the expert weights streamed since its last use may have pushed it
    for (int e = warp; e < E; e += kRouteWarps)
      for (int c = lane * 64; c < H; c += 32 * 64)  // 128-byte lines of the row
        asm volatile("prefetch.global.L2 [%0];" ::"l"(wr + (size_t)e * H + c));
  }
  uint16_t* const dense_rows = staged && scatter.cap > 0 && scatter.dense && scatter.split.amax_in == nullptr ? scatter.xp : nullptr;
  griddep_wait();
  if (threadIdx.x == 0) timeline_start(timeline, 0);
  if (staged) {
    if (prev.y != nullptr) {
      combine_rows<TT == 1 ? 1 : 2>(prev, t0, my_tokens, H, s_x, dense_rows);
      // CTA 0 also clears the control block the previous step used (its kernels have completed)
      if (blockIdx.x == 0 && prev.zero_words != nullptr)
        for (int i = threadIdx.x; i < prev.n_zero_words; i += blockDim.x) prev.zero_words[i] = 0u;
    } else {
      for (int c = threadIdx.x; c < my_tokens * (H / 8); c += blockDim.x) {
        const uint4 v = reinterpret_cast<const uint4*>(x + (size_t)t0 * H)[c];
        reinterpret_cast<uint4*>(s_x)[c] = v;
        if (dense_rows != nullptr) reinterpret_cast<uint4*>(dense_rows + (size_t)t0 * H)[c] = v;
      }
    }
    if ((int)threadIdx.x < my_tokens) s_conf[threadIdx.x] = conf[t0 + threadIdx.x];
    for (int i = threadIdx.x; i < TT * (Ep - E); i += blockDim.x) s_key[(i / (Ep - E)) * Ep + E + i % (Ep - E)] = 0u;
    if (threadIdx.x < kST) s_amax[threadIdx.x] = 0u;
    if (kAhead) asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (scatter.split.amax_in != nullptr)
      for (int a = 0; a < my_tokens; ++a) {
        uint32_t big = 0u;
        for (int c = threadIdx.x; c < H / 8; c += blockDim.x) {
          const uint4 v = reinterpret_cast<const uint4*>(s_x + (size_t)a * H)[c];
          big = __vmaxu2(__vmaxu2(big, __vmaxu2(v.x & 0x7fff7fffu, v.y & 0x7fff7fffu)),
                         __vmaxu2(v.z & 0x7fff7fffu, v.w & 0x7fff7fffu));
        }
        big = __reduce_max_sync(0xffffffffu, max(big & 0xffffu, big >> 16));
        if (lane == 0 && big != 0u) atomicMax(&s_amax[a], big);
      }
  }

  for (int eb = warp * kEPerWarp; eb < E; eb += kRouteWarps * kEPerWarp) {
    float acc[TT][kEPerWarp];
#pragma unroll
    for (int a = 0; a < TT; ++a)
#pragma unroll
      for (int b = 0; b < kEPerWarp; ++b) acc[a][b] = 0.0f;

    float bias_e[kEPerWarp];  // (requested ahead of the loop, not after it)
#pragma unroll
    for (int b = 0; b < kEPerWarp; ++b) bias_e[b] = bias != nullptr ? bias[min(eb + b, E - 1)] : 0.0f;
    // one chunk of 256 columns: weights ww, the tokens' rows from shared memory (or global memory)
    auto chunk = [&](int hc, const uint4 (&ww)[kEPerWarp]) {
      const int h = hc + lane * 8;
      uint4 xw[TT];
#pragma unroll
      for (int a = 0; a < TT; ++a)
        // (staged rows beyond the step's last token hold stale shared memory: their logits are never used)
        xw[a] = staged ? *reinterpret_cast<const uint4*>(s_x + (size_t)a * H + h)
                       : *reinterpret_cast<const uint4*>(x + (size_t)min(t0 + a, T - 1) * H + h);
      // elements in ascending h: word 0 low half, word 0 high half, word 1 low half, ...
      auto word = [&](auto get) {
#pragma unroll
        for (int a = 0; a < TT; ++a)
#pragma unroll
          for (int b = 0; b < kEPerWarp; ++b) fma_bf16_pair(acc[a][b], get(xw[a]), get(ww[b]));
      };
      word([](const uint4& v) { return v.x; });
      word([](const uint4& v) { return v.y; });
      word([](const uint4& v) { return v.z; });
      word([](const uint4& v) { return v.w; });
    };
    if constexpr (kAhead) {
      int hc = 0;
#pragma unroll 2
      for (; hc < w_cols; hc += 256) {
        uint4 ww[kEPerWarp];
#pragma unroll
        for (int b = 0; b < kEPerWarp; ++b)
          ww[b] = *reinterpret_cast<const uint4*>(s_w + (size_t)min(eb + b, E - 1) * w_cols + hc + lane * 8);
        chunk(hc, ww);
      }
#pragma unroll
      for (int i = 0; i < kTail; ++i, hc += 256)  // (there are any only where one pass takes all experts: these are its rows)
        if (hc < H) chunk(hc, w_tail[i]);
    } else {
#pragma unroll UNROLL
      for (int hc = 0; hc < H; hc += 256) {
        uint4 ww[kEPerWarp];
#pragma unroll
        for (int b = 0; b < kEPerWarp; ++b)
          ww[b] = *reinterpret_cast<const uint4*>(wr + (size_t)min(eb + b, E - 1) * H + hc + lane * 8);
        chunk(hc, ww);
      }
    }
#pragma unroll
    for (int a = 0; a < TT; ++a)
#pragma unroll
      for (int b = 0; b < kEPerWarp; ++b) {
        float v = acc[a][b];
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, d));
        const int e = eb + b;
        if (lane == 0 && e < E && t0 + a < T) {
          if (bias != nullptr) v = __fadd_rn(v, bias_e[b]);
          s_logits[a * E + e] = v;
          if (staged) s_key[a * Ep + e] = order_key(topk_value(v));
          if (logits_out != nullptr) logits_out[(size_t)(t0 + a) * E + e] = v;
        }
      }
  }
  __syncthreads();

  if (staged) {
    // top-k by rank: expert e is selected iff fewer than K experts precede it in the order (logit descending,
    // index ascending), and its rank is the number that do.  `parts` neighbouring threads per (token, expert)
    // count a share of the experts each, four keys at a time.  (A warp per expert at a time took 1.4 us for
    // one token and 64 experts, 6.5 us for two and 128; now 0.5 and 0.9.  Divisions by E had doubled that.)
    const int items = my_tokens * E;
    int parts = 1, parts_log2 = 0;
    for (; parts < 32 && items * parts * 2 <= WARPS * 32; parts <<= 1) ++parts_log2;
    const int part = threadIdx.x & (parts - 1);
    for (int i0 = 0; i0 < items; i0 += (WARPS * 32) >> parts_log2) {
      const int i = i0 + ((int)threadIdx.x >> parts_log2);
      int a = 0, e = min(i, items - 1);
#pragma unroll
      for (int j = 1; j < TT; ++j)
        if (e >= E) {
          e -= E;
          ++a;
        }
      const uint32_t ke = s_key[a * Ep + e];
      const uint4* row = reinterpret_cast<const uint4*>(s_key + a * Ep);
      int before = 0;
      for (int c = part; c < Ep / 4; c += parts) {
        const uint4 k = row[c];
        const int o = 4 * c;  // (an equal key precedes if its index is lower; no key of an expert is zero)
        before += (k.x > ke - (o < e)) + (k.y > ke - (o + 1 < e)) + (k.z > ke - (o + 2 < e)) + (k.w > ke - (o + 3 < e));
      }
      for (int d = parts >> 1; d >= 1; d >>= 1) before += __shfl_xor_sync(0xffffffffu, before, d);
      if (part == 0 && i < items && before < K) {
        s_sel_id[a][before] = e;
        s_sel_logit[a][before] = topk_value(s_logits[a * E + e]);
      }
    }
    __syncthreads();
    // scattered steps: every assignment of the CTA's tokens takes a row of its expert (the last warps
    // turn the selected logits into gate scores meanwhile)
    if (scatter.cap > 0) {
      for (int i = threadIdx.x; i < my_tokens * K; i += blockDim.x) {
        const int a = i / K, e = s_sel_id[a][i - a * K];
        const int row = e * scatter.cap + atomicAdd(&counts[e], 1);
        s_r[i] = row;
        scatter.assignment[row] = t0 * K + i;
        if (scatter.split.amax_in != nullptr) {
          // (dense steps: the input rows are the tokens', the intermediate rows the first T * K)
          scatter.split.amax_in[scatter.dense ? t0 + a : row] = s_amax[a] << 16;
          scatter.split.amax_mid[scatter.dense ? t0 * K + i : row] = 0u;
        }
      }
    }
    for (int a = kRouteWarps - 1 - warp; a < my_tokens; a += kRouteWarps) {
      const int t = t0 + a;
      const int my_id = lane < K ? s_sel_id[a][lane] : 0;
      const float my_logit = lane < K ? s_sel_logit[a][lane] : 0.0f;
      const float top = __shfl_sync(0xffffffffu, my_logit, 0);
      const float z = lane < K ? exp_spec(__fsub_rn(my_logit, top)) : 0.0f;
      float sum = __shfl_sync(0xffffffffu, z, 0);
      for (int j = 1; j < K; ++j) sum = __fadd_rn(sum, __shfl_sync(0xffffffffu, z, j));
      if (lane < K) {
        const float g = __fdiv_rn(z, sum);
        ids[(size_t)t * K + lane] = my_id;
        gate[(size_t)t * K + lane] = g;
        if (finish.offsets == nullptr) {
          if (scatter.cap == 0) atomicAdd(&counts[my_id], 1);
          atomicAdd(&scores[my_id], score_quantum(g, s_conf[a]));
        }
      }
    }
    if (scatter.cap > 0 && dense_rows == nullptr) {  // (dense rows of bf16 stores have been stored already)
      __syncthreads();  // the rows of all assignments are known
      const int vec_per_row = H / 8, total = my_tokens * vec_per_row;
      for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const int a = i / vec_per_row, c = i - a * vec_per_row;
        const uint4 v = reinterpret_cast<const uint4*>(s_x)[i];
        uint2 t1 = make_uint2(0u, 0u), t2 = t1;
        if (scatter.split.amax_in != nullptr) {
          const float scale = token_scale(s_amax[a] << 16);
          split_bf16x4(v.x, v.y, scale, t1.x, t2.x);
          split_bf16x4(v.z, v.w, scale, t1.y, t2.y);
        }
        for (int j = 0; j < (scatter.dense ? 1 : K); ++j) {
          const size_t row = scatter.dense ? (size_t)(t0 + a) : (size_t)s_r[a * K + j];
          if (scatter.split.amax_in == nullptr) {
            reinterpret_cast<uint4*>(scatter.xp)[row * vec_per_row + c] = v;
          } else {  // (the FFN reads the terms only: 8 layers of 250 tokens 748 -> 734 us without the copies)
            reinterpret_cast<uint2*>(scatter.split.terms_in)[row * vec_per_row + c] = t1;
            reinterpret_cast<uint2*>(scatter.split.terms_in)[((size_t)scatter.split.rows + row) * vec_per_row + c] = t2;
          }
        }
      }
    }
  } else {
    // one warp per token
    for (int a = warp; a < TT; a += kRouteWarps) {
      const int t = t0 + a;
      if (t >= T) continue;
      route_token_tail(s_logits + a * E, t, lane, E, K, conf, ids, gate, counts, scores);
    }
  }
  if (finish.offsets != nullptr && gridDim.x == 1) {
    __syncthreads();  // (the ids are stored)
    sort_assignments<WARPS>(ids, T * K, E, counts, finish.offsets, finish.perm, reinterpret_cast<int*>(s_dyn));
  }
  if (threadIdx.x == 0) timeline_end(timeline, 0);
}

// Many-token steps: TT tokens per CTA, eight warps, every warp a register tile of TT tokens x 8
// experts.  The plain kernel above re-reads the router matrix once per eight tokens through the L1
// path and spends an ALU instruction on every bf16 -> fp32 conversion; it reaches a third of the
// FP32 pipe.  Here
//  - the operands are staged in shared memory by cp.async, a ring of k-chunks of 256 elements (the
//    TT token rows and 64 router rows of a chunk), so that the warps read only shared memory
//    (conflict-free 16-byte reads) and the global loads of later chunks are always in flight;
//  - the multiply-adds take their bf16 operands directly (fma.rn.f32.bf16: exact product, one
//    rounding - bit for bit the fp32 fused multiply-add of the converted operands), which removes
//    the conversions;
//  - TT is chosen by the launcher so that the CTAs fill whole waves of SMs (4096 tokens: 14 per
//    CTA, 293 CTAs, two waves on 148 SMs), and a larger TT re-reads the router matrix less often.
// Same chains, same order: lane q still owns the elements h with (h/8) mod 32 == q and walks them
// in ascending order.  Experts beyond 64 take further passes over the rows.
constexpr int kManyWarps = 8, kManyExperts = 64, kManyStages = 4;
__host__ __device__ constexpr int many_stage_bytes(int tt) { return (tt + kManyExperts) * 512; }  // one k-chunk of 256 bf16 per row

template <int TT>
__global__ void __launch_bounds__(kManyWarps * 32, 1)
route_many_kernel(const uint16_t* __restrict__ x, const uint16_t* __restrict__ wr,
                  const float* __restrict__ bias, const float* __restrict__ conf, int T, int H, int E,
                  int K, float* __restrict__ logits_out, int32_t* __restrict__ ids,
                  float* __restrict__ gate, int32_t* __restrict__ counts,
                  unsigned long long* __restrict__ scores, StepTimeline* timeline,
                  int32_t* __restrict__ seg_counts, int seg_tokens) {
  constexpr int kStageBytes = many_stage_bytes(TT);
  constexpr int kRows = TT + kManyExperts;
  extern __shared__ __align__(16) uint8_t s_dyn[];
  uint8_t* s_ring = s_dyn;                                                        // [stages][TT + 64 rows][512 B]
  // the CTA's sums, added to the global words at the end: [E] scores, [2][E] counts (of the one or two segments that its
  // tokens lie in; a segment has at least TT tokens)
  unsigned long long* s_scores = reinterpret_cast<unsigned long long*>(s_dyn + kManyStages * kStageBytes);
  int32_t* s_counts = reinterpret_cast<int32_t*>(s_scores + E);
  float* s_logits = reinterpret_cast<float*>(s_counts + 2 * E);  // [TT][E]
  __shared__ const uint16_t* s_rowptr[kRows];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t0 = blockIdx.x * TT;
  griddep_launch_dependents();
  if (threadIdx.x == 0) timeline_entry(timeline, 0);
  griddep_wait();
  if (threadIdx.x == 0) timeline_start(timeline, 0);
  for (int e = threadIdx.x; e < E; e += kManyWarps * 32) {
    s_scores[e] = 0ull;
    s_counts[e] = s_counts[E + e] = 0;
  }
  const int n_chunks = H / 256;
  const uint32_t ring_base = (uint32_t)__cvta_generic_to_shared(s_ring);

  for (int e0 = 0; e0 < E; e0 += kManyExperts) {
    // one stage: rows 0..TT-1 = tokens t0.., rows TT.. = experts e0..; each row 32 pieces of 16 bytes.
    // The rows' addresses are looked up in a table (one 8-byte read instead of a clamp and a 64-bit
    // multiply per copy: the copies' own instructions are a tenth of the loop otherwise).
    __syncthreads();  // the previous pass has finished with the ring and the table
    for (int row = threadIdx.x; row < kRows; row += kManyWarps * 32)
      s_rowptr[row] = row < TT ? x + (size_t)min(t0 + row, T - 1) * H
                               : wr + (size_t)min(e0 + row - TT, E - 1) * H;
    auto issue = [&](int chunk) {
      const uint32_t dst0 = ring_base + (uint32_t)(chunk % kManyStages) * kStageBytes + (uint32_t)lane * 16u;
#pragma unroll
      for (int j = 0; j < (kRows + kManyWarps - 1) / kManyWarps; ++j) {
        const int row = warp + j * kManyWarps;
        if (row < kRows)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst0 + (uint32_t)row * 512u),
                       "l"(s_rowptr[row] + (size_t)chunk * 256 + lane * 8)
                       : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[TT][8];
#pragma unroll
    for (int a = 0; a < TT; ++a)
#pragma unroll
      for (int b = 0; b < 8; ++b) acc[a][b] = 0.0f;
    __syncthreads();  // the table is complete
    for (int c = 0; c < kManyStages - 1; ++c) {
      if (c < n_chunks) issue(c);
      else asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int c = 0; c < n_chunks; ++c) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kManyStages - 2) : "memory");  // chunk c has landed (this thread's part)
      __syncthreads();                                                            // ... everyone's; and chunk c-1 is consumed
      if (c + kManyStages - 1 < n_chunks) issue(c + kManyStages - 1);
      else asm volatile("cp.async.commit_group;" ::: "memory");
      const uint8_t* st = s_ring + (size_t)(c % kManyStages) * kStageBytes;
      uint4 xw[TT], ww[8];
#pragma unroll
      for (int a = 0; a < TT; ++a) xw[a] = *reinterpret_cast<const uint4*>(st + a * 512 + lane * 16);
#pragma unroll
      for (int b = 0; b < 8; ++b) ww[b] = *reinterpret_cast<const uint4*>(st + (TT + warp * 8 + b) * 512 + lane * 16);
      // elements in ascending h: word 0 low half, word 0 high half, word 1 low half, ...
#pragma unroll
      for (int a = 0; a < TT; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) fma_bf16_pair(acc[a][b], xw[a].x, ww[b].x);
#pragma unroll
      for (int a = 0; a < TT; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) fma_bf16_pair(acc[a][b], xw[a].y, ww[b].y);
#pragma unroll
      for (int a = 0; a < TT; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) fma_bf16_pair(acc[a][b], xw[a].z, ww[b].z);
#pragma unroll
      for (int a = 0; a < TT; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) fma_bf16_pair(acc[a][b], xw[a].w, ww[b].w);
    }
    // The 32 partial sums of every (token, expert) pair are added in the order of the xor butterfly
    // (offsets 16, 8, 4, 2, 1; at every step a lane adds its partner's value to its own).  Addition
    // is commutative bit for bit, so every lane of the butterfly ends with the same value, and the
    // 32 pairs of a group can share the steps: at offset d a lane keeps the half of its pairs
    // whose index has bit d equal to its own lane's bit and hands the other half to its partner -
    // 31 shuffles per 32 pairs instead of 160, and lane l ends with the sum of pair l.
#pragma unroll
    for (int g = 0; g < (TT * 8 + 31) / 32; ++g) {
      float v[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const int p = g * 32 + i;  // pair p: token p / 8, expert column p % 8
        v[i] = p < TT * 8 ? acc[p / 8][p % 8] : 0.0f;
      }
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) {
        const bool upper = (lane & d) != 0;
#pragma unroll
        for (int i = 0; i < d; ++i) {
          const float keep = upper ? v[i + d] : v[i];
          const float send = upper ? v[i] : v[i + d];
          v[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, d));
        }
      }
      const int p = g * 32 + lane, a = p / 8, e = e0 + warp * 8 + p % 8;
      if (p < TT * 8 && e < E && t0 + a < T) {
        float r = v[0];
        if (bias != nullptr) r = __fadd_rn(r, bias[e]);
        s_logits[a * E + e] = r;
        if (logits_out != nullptr) logits_out[(size_t)(t0 + a) * E + e] = r;
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // One warp per token.  Counts and scores are summed in shared memory (integers: the order does not matter) and each of
  // the experts' words receives one addition per CTA: with one per assignment the few words of the popular experts were
  // a queue (4096 tokens, 64 experts top-8: 89 us, now 81; a batch of 1000 tokens in 4 layers 808 us, now 795).
  const int seg0 = seg_counts != nullptr ? t0 / seg_tokens : 0;
  for (int a = warp; a < TT; a += kManyWarps) {
    const int t = t0 + a;
    if (t >= T) continue;
    const int second = seg_counts != nullptr && t >= (seg0 + 1) * seg_tokens ? E : 0;
    route_token_tail(s_logits + a * E, t, lane, E, K, conf, ids, gate, s_counts + second, s_scores);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < E; e += kManyWarps * 32) {
    const int c0 = s_counts[e], c1 = s_counts[E + e];
    if (c0 + c1 == 0) continue;
    atomicAdd(&counts[e], c0 + c1);
    if (s_scores[e] != 0ull) atomicAdd(&scores[e], s_scores[e]);
    if (seg_counts != nullptr && c0 != 0) atomicAdd(&seg_counts[seg0 * E + e], c0);
    if (seg_counts != nullptr && c1 != 0) atomicAdd(&seg_counts[(seg0 + 1) * E + e], c1);
  }
  if (threadIdx.x == 0) timeline_end(timeline, 0);
}

// One CTA per expert (blockIdx.x): offset = sum of the counts before it; then a stable scan of the
// flat assignment list (ascending t*K+j) hands out consecutive sorted rows.
// If xp != nullptr the expert's CTAs (gridDim.y of them) also copy its token rows into sorted
// order (xp[r,:] = x[perm[r]/K,:]); used for small steps and, segment by segment, in many-token steps.
// Each of those CTAs repeats the scan for itself - a few hundred ids - keeps the token of every
// sorted row in shared memory (reading the rows' numbers back from global memory would cost a
// round trip before the first load), and takes every gridDim.y-th batch of RB rows, so that an
// expert that received many tokens does not make the step wait for one CTA's chain of batches.
// Only the CTAs with blockIdx.y == 0 write offsets, perm and pos.
constexpr int kGatherTokMax = 4096;  // rows of one expert in a step that gathers here (T * K <= 4096), or in a segment
// RB: rows a CTA copies at a time.  Two, with eight CTAs per expert, in gathering launches of few-token steps: an
// expert's handful of rows is then spread over several SMs (with one CTA taking eight rows the
// step waited 3 us longer whenever an expert had more than eight, and the e4m3 terms of fp8
// steps, whose conversions are the long pole, came to 7 us).  Four where a segment's CTA copies its rows.  (Launches that
// do not gather take the smallest, for its registers: with eight, 152 of them, one CTA fits an SM and 4096 tokens took 18 us.)
template <int RB>
__global__ void __launch_bounds__(256)
permute_kernel(const int32_t* __restrict__ ids, const int32_t* __restrict__ counts, int n, int E,
               int32_t* __restrict__ offsets, int32_t* __restrict__ perm, int32_t* __restrict__ pos,
               const uint16_t* __restrict__ x, uint16_t* __restrict__ xp, int H, int K, StepTimeline* timeline,
               TokenSplit split, const int32_t* __restrict__ seg_counts, int seg_tokens) {
  uint32_t* const amax_in = split.amax_in;
  uint32_t* const amax_mid = split.amax_mid;
  __shared__ int s_red[8];
  __shared__ int s_base, s_seg;
  __shared__ int s_tok[kGatherTokMax];
  __shared__ uint32_t s_amax[3][RB];  // per batch of RB rows, three batches in rotation (see the gather loop)
  const int e = blockIdx.x;
  // segmented launches: CTA (e, s) scans segment s of the assignment list only and starts behind the expert's rows of
  // the earlier segments, whose number the gate kernel counted
  const bool segmented = seg_counts != nullptr;
  const bool writer = blockIdx.y == 0 || segmented;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  griddep_launch_dependents();
  if (threadIdx.x == 0) timeline_entry(timeline, 1);
  griddep_wait();
  if (threadIdx.x == 0) timeline_start(timeline, 1);
  int part = 0;
  if (segmented && warp == 1) {  // the expert's rows of the earlier segments (requested together: one after the other, 16 of
                                 // them were most of this kernel's 9 us at 1000 tokens)
    int s = lane < (int)blockIdx.y ? seg_counts[lane * E + e] : 0;
    s = __reduce_add_sync(0xffffffffu, s);
    if (lane == 0) s_seg = s;
  }
  for (int i = threadIdx.x; i < e; i += blockDim.x) part += counts[i];
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) part += __shfl_xor_sync(0xffffffffu, part, d);
  if (lane == 0) s_red[warp] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    int off = 0;
    for (int w = 0; w < 8; ++w) off += s_red[w];
    s_base = off;
    if (blockIdx.y == 0) {
      offsets[e] = off;
      if (e == E - 1) offsets[E] = off + counts[e];
    }
    if (segmented) s_base = off + s_seg;
  }
  __syncthreads();
  // (a CTA beyond the first of an expert has work only if the expert has a batch of rows for it)
  if (segmented ? seg_counts[blockIdx.y * E + e] == 0 : (counts[e] == 0 || (int)blockIdx.y * RB >= counts[e])) {
    if (threadIdx.x == 0) timeline_end(timeline, 1);
    return;
  }
  int base = s_base;
  const int a_first = segmented ? (int)blockIdx.y * seg_tokens * K : 0;
  const int a_end = segmented ? min(n, a_first + seg_tokens * K) : n;
  // stable scan, 8 consecutive assignments per thread and 2048 per round
  for (int a0 = a_first; a0 < a_end; a0 += 8 * blockDim.x) {
    const int first = a0 + threadIdx.x * 8;
    int v[8];
    if (first + 8 <= a_end) {
      const int4 lo = *reinterpret_cast<const int4*>(ids + first);
      const int4 hi = *reinterpret_cast<const int4*>(ids + first + 4);
      v[0] = lo.x; v[1] = lo.y; v[2] = lo.z; v[3] = lo.w;
      v[4] = hi.x; v[5] = hi.y; v[6] = hi.z; v[7] = hi.w;
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = first + i < a_end ? ids[first + i] : -1;
    }
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) m |= (v[i] == e ? 1u : 0u) << i;
    const int c = __popc(m);
    int incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    __syncthreads();  // previous round's s_red fully consumed
    if (lane == 31) s_red[warp] = incl;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const int cw = s_red[w];
      if (w < warp) before += cw;
      total += cw;
    }
    int r = base + before + incl - c;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if ((m >> i) & 1u) {
        if (writer) {
          perm[r] = first + i;
          pos[first + i] = r;
        }
        if (xp != nullptr) s_tok[r - s_base] = (first + i) / K;
        ++r;
      }
    base += total;
  }
  if (xp == nullptr) {
    if (threadIdx.x == 0) timeline_end(timeline, 1);
    return;
  }
  if (threadIdx.x < 3 * RB) s_amax[threadIdx.x / RB][threadIdx.x % RB] = 0u;
  __syncthreads();  // the tokens of this expert's rows are in shared memory
  // RB rows at a time: their token numbers, then their loads, are independent memory
  // operations in flight together (a row-by-row loop is a chain of dependent round trips)
  // (segmented launches: all rows of the segment are this CTA's)
  const int vec_per_row = H / 8, first = s_base, rows = segmented ? seg_counts[blockIdx.y * E + e] : counts[e];
  const int r_first = segmented ? 0 : (int)blockIdx.y * RB, r_step = segmented ? RB : RB * (int)gridDim.y;
  const uint4* src = reinterpret_cast<const uint4*>(x);
  uint4* dst = reinterpret_cast<uint4*>(xp);
  int batch = 0;
  for (int r0 = r_first; r0 < rows; r0 += r_step, ++batch) {
    int tok[RB];
#pragma unroll
    for (int j = 0; j < RB; ++j) tok[j] = r0 + j < rows ? s_tok[r0 + j] : -1;
    uint32_t big[RB];  // per row: max of |bf16| bit patterns, two per word
#pragma unroll
    for (int j = 0; j < RB; ++j) big[j] = 0u;
    uint4 v[RB];  // (the last vectors stay in registers for the e4m3 terms below)
    int c_last = -1;
    for (int c = threadIdx.x; c < vec_per_row; c += blockDim.x) {
      c_last = c;
#pragma unroll
      for (int j = 0; j < RB; ++j)
        if (tok[j] >= 0) v[j] = src[(size_t)tok[j] * vec_per_row + c];
#pragma unroll
      for (int j = 0; j < RB; ++j)
        if (tok[j] >= 0) {
          dst[(size_t)(first + r0 + j) * vec_per_row + c] = v[j];
          if (amax_in != nullptr)
            big[j] = __vmaxu2(__vmaxu2(big[j], __vmaxu2(v[j].x & 0x7fff7fffu, v[j].y & 0x7fff7fffu)),
                              __vmaxu2(v[j].z & 0x7fff7fffu, v[j].w & 0x7fff7fffu));
        }
    }
    if (amax_in != nullptr) {
      // the rows' largest magnitudes (a bf16 magnitude's bits order like the value) and a cleared
      // word per row for the intermediate rows' maxima.  One barrier per batch: a batch's words
      // were cleared two batches (two barriers) ago, and it clears the words of the batch after next.
      uint32_t* amax_now = s_amax[batch % 3];
#pragma unroll
      for (int j = 0; j < RB; ++j) {
        const uint32_t m = __reduce_max_sync(0xffffffffu, max(big[j] & 0xffffu, big[j] >> 16));
        if (lane == 0 && m != 0u) atomicMax(&amax_now[j], m);
      }
      __syncthreads();
      if (threadIdx.x < RB) {
        s_amax[(batch + 2) % 3][threadIdx.x] = 0u;
        if (r0 + (int)threadIdx.x < rows) {
          amax_in[first + r0 + threadIdx.x] = amax_now[threadIdx.x] << 16;
          amax_mid[first + r0 + threadIdx.x] = 0u;
        }
      }
      // the rows' two e4m3 terms (vectors of earlier rounds of the loop above are read back)
      for (int c = threadIdx.x; c < vec_per_row; c += blockDim.x) {
#pragma unroll
        for (int j = 0; j < RB; ++j)
          if (tok[j] >= 0) {
            const size_t r = (size_t)(first + r0 + j);
            const uint4 vv = c == c_last ? v[j] : dst[r * vec_per_row + c];
            const float scale = token_scale(amax_now[j] << 16);
            uint2 t1, t2;
            split_bf16x4(vv.x, vv.y, scale, t1.x, t2.x);
            split_bf16x4(vv.z, vv.w, scale, t1.y, t2.y);
            uint2* out1 = reinterpret_cast<uint2*>(split.terms_in + r * H);
            uint2* out2 = reinterpret_cast<uint2*>(split.terms_in + ((size_t)split.rows + r) * H);
            out1[c] = t1;
            out2[c] = t2;
          }
      }
    }
  }
  if (threadIdx.x == 0) timeline_end(timeline, 1);
}

// One warp per sorted row: the row's token number once, then the row's 16-byte vectors, four
// loads in flight per lane.
__global__ void __launch_bounds__(256)
gather_kernel(const uint16_t* __restrict__ x, const int32_t* __restrict__ perm, int n_rows, int H,
              int K, uint16_t* __restrict__ xp) {
  const int vec_per_row = H / 8;
  const int lane = threadIdx.x & 31;
  const int warps = gridDim.x * (blockDim.x >> 5);
  griddep_launch_dependents();
  griddep_wait();
  for (int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < n_rows; r += warps) {
    const int t = perm[r] / K;
    const uint4* src = reinterpret_cast<const uint4*>(x) + (size_t)t * vec_per_row;
    uint4* dst = reinterpret_cast<uint4*>(xp) + (size_t)r * vec_per_row;
    for (int c0 = lane; c0 < vec_per_row; c0 += 128) {
      uint4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (c0 + 32 * j < vec_per_row) v[j] = src[c0 + 32 * j];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (c0 + 32 * j < vec_per_row) dst[c0 + 32 * j] = v[j];
    }
  }
}

}  // namespace


static thread_local bool g_pdl_step = true;
static std::atomic<bool> g_pdl_allowed{true};
void pdl_set_step(bool on) { g_pdl_step = on; }
void pdl_set_allowed(bool on) { g_pdl_allowed.store(on); }
bool pdl_enabled() { return g_pdl_allowed.load() && g_pdl_step; }

// The staged gate kernel takes few-token steps, where it brings the rows to their experts and may carry out a
// combine; beyond two tokens per SM it re-reads the router matrix too often (64 experts x 2048, 1000 tokens: 35 us
// against 16 in the many-token kernel), so it stays there only for what the other does not do.
constexpr int kStagedWarps = 16;
static size_t staged_smem(int tt, int H, int E) {  // logits, rows, keys
  return ((((size_t)tt * E * sizeof(float)) + 15) & ~(size_t)15) + (size_t)tt * H * 2 + (size_t)tt * ((E + 3) & ~3) * 4;
}
constexpr size_t kStagedSmem = 224 * 1024;  // (of 227 KB; the rest holds the kernel's static arrays)
// Chunks of the router matrix to fetch into shared memory ahead of the input, 0: none.  Only where
//  * the whole matrix is on chip then (64 experts of 2048, 128 of 512): a part of it is the same wait for the copies and the
//    same reads of L2 for the rest (6 chunks of 16 at 64 x 4096 from fp8 stores: a lone step of one token 42.5 us, without them 40.7,
//    stacks of four such layers 150 / 139); what shared memory has no room for waits in registers where one pass of the warps
//    takes all experts;
//  * a CTA has one token or two (four, stacks of 400 tokens at 16 x 512: bf16 / fp8 stores 183.9 / 218.6 us with it, 181.3 / 217.0 without);
//  * there is an FFN launch to wait for - the kernel carries its combine out -, or the CTAs are so few that the copies are no
//    queue in front of the logits (lone steps at 64 x 2048 of 1 / 4 / 16 / 32 / 100 tokens: 28.1 / 54.0 / 111.0 / 118.4 / 127.2 us with it,
//    28.7 / 54.0 / 110.7 / 117.5 / 125.0 without; from fp8 stores 26.1 / 38.5 / 64.5 / 71.6 / 75.2 and 26.8 / 39.0 / 65.0 / 70.6 / 73.4).
// Stacks of four layers without / with it: 64 x 2048, 1 token 113.4 / 109.6 us, 32 tokens 469.8 / 468.3; 128 x 512, 1 / 16 / 100 tokens
// 90.8 / 212.9 / 287.7 and 85.7 / 209.0 / 284.9; 160 x 512 from fp8 stores, 32 tokens 151.4 / 149.0; of six layers 16 x 512, 250 tokens (two
// a CTA) 158.4 / 157.5, from fp8 stores 184.9 / 181.3.
static int router_chunks_ahead(int T, int H, int E, bool combines) {
  if (T > 296 || !(combines || T <= 16)) return 0;
  const int tt = T <= 148 ? 1 : 2;
  const int chunks = (int)std::min<size_t>(H / 256, (kStagedSmem - staged_smem(tt, H, E)) / ((size_t)E * 512));
  return H / 256 - chunks <= (E <= kStagedWarps * 4 ? router_tail(tt) : 0) ? chunks : 0;
}
static bool staged_attributes() {  // the staged rows: up to 4 x 16 K elements
  static const bool ok = [] {
    const bool done =
        cudaFuncSetAttribute(route_kernel<1, kStagedWarps, 4, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmem) == cudaSuccess &&
        cudaFuncSetAttribute(route_kernel<2, kStagedWarps, 4, 4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmem) == cudaSuccess &&
        cudaFuncSetAttribute(route_kernel<1, kStagedWarps, 4, 4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmem) == cudaSuccess &&
        cudaFuncSetAttribute(route_kernel<2, kStagedWarps, 4, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmem) == cudaSuccess &&
        cudaFuncSetAttribute(route_kernel<4, kStagedWarps, 2, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmem) == cudaSuccess;
    if (!done) cudaGetLastError();
    return done;
  }();
  return ok;
}
bool route_staged(int T, int K) { return T <= 296 || (T <= 1024 && (size_t)T * K <= 4096); }

void launch_route(cudaStream_t st, const uint16_t* x, const uint16_t* w_router, const float* bias,
                  const float* conf, int T, int H, int E, int K, float* logits, int32_t* ids,
                  float* gate, int32_t* counts, unsigned long long* scores, const CombinePrev& prev,
                  StepTimeline* timeline, int32_t* seg_counts, int seg_tokens, const ScatterRows& scatter) {
  if (route_staged(T, K)) {
    constexpr int W = kStagedWarps;
    staged_attributes();
    // (the matrix is the context's copy, whose writer has been waited for: it is older than all that may still run on the stream)
    const int ahead = router_chunks_ahead(T, H, E, prev.y != nullptr);
    auto go = [&](auto kernel, int tt) {
      launch_pdl(kernel, dim3((T + tt - 1) / tt), dim3(W * 32), staged_smem(tt, H, E) + (size_t)ahead * E * 512, st, x, w_router,
                 bias, conf, T, H, E, K, logits, ids, gate, counts, scores, prev, timeline, scatter, RouteFinish{}, ahead);
    };
    if (T <= 148 && ahead > 0) go(route_kernel<1, W, 4, 4, true>, 1);
    else if (T <= 148) go(route_kernel<1, W, 4, 4>, 1);
    else if (ahead > 0) go(route_kernel<2, W, 4, 4, true>, 2);
    else if (T <= 296) go(route_kernel<2, W, 4, 4>, 2);  // (four tokens per CTA measured slower at 256 tokens x 128 experts: 33 against 20 us)
    else go(route_kernel<4, W, 2, 4>, 4);
  } else {
    // (re-tilings of the plain kernel - more tokens or experts per warp, more warps per CTA, deeper
    // unrolling - were all slower at 4096 tokens x 64 experts x 4096)
    // tokens per CTA: the time is (waves of CTAs) x (tokens per CTA); ties go to the larger tile,
    // which reads the router matrix less often
    static int n_sms = 0;
    if (n_sms == 0) {
      int dev = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev);
      if (n_sms <= 0) n_sms = 148;
    }
    int best_tt = 8;
    long best_cost = -1;
    for (int tt : {8, 10, 12, 14}) {
      const int ctas = (T + tt - 1) / tt;
      const long cost = (long)((ctas + n_sms - 1) / n_sms) * tt;
      if (best_cost < 0 || cost <= best_cost) {
        best_cost = cost;
        best_tt = tt;
      }
    }
    auto go = [&](auto kernel, int tt) {
      const size_t smem = (size_t)kManyStages * many_stage_bytes(tt) + (size_t)(tt + 4) * E * sizeof(float);
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
      launch_pdl(kernel, dim3((T + tt - 1) / tt), dim3(kManyWarps * 32), smem, st, x, w_router, bias, conf, T, H, E,
                 K, logits, ids, gate, counts, scores, timeline, seg_counts, seg_tokens);
    };
    switch (best_tt) {
      case 8: go(route_many_kernel<8>, 8); break;
      case 10: go(route_many_kernel<10>, 10); break;
      case 12: go(route_many_kernel<12>, 12); break;
      default: go(route_many_kernel<14>, 14); break;
    }
  }
}

void launch_permute(cudaStream_t st, const int32_t* ids, const int32_t* counts, int T, int E, int K,
                    int32_t* offsets, int32_t* perm, int32_t* pos, const uint16_t* x, uint16_t* xp, int H,
                    StepTimeline* timeline, const TokenSplit* split, const int32_t* seg_counts, int seg_tokens) {
  const TokenSplit sp = xp != nullptr && split != nullptr && split->complete() ? *split : TokenSplit{};
  if (xp != nullptr && seg_counts != nullptr) {
    // many-token steps: each segment's CTA copies its own rows (1000 tokens: a gather kernel behind this one took 6 us)
    launch_pdl(permute_kernel<4>, dim3(E, kPermuteSegments), dim3(256), 0, st, ids, counts, T * K, E, offsets, perm, pos, x, xp,
               H, K, timeline, sp, seg_counts, seg_tokens);
  } else if (xp != nullptr) {
    // gathering steps: two rows per CTA and batch, eight CTAs per expert (see the kernel) - fewer where
    // eight per expert would not be resident at once (four CTAs fit an SM; 128 experts take four each:
    // 7.2 instead of 8.9 us at 256 tokens, two each 9.5 us)
    int per_expert = 8;
    while (per_expert > 1 && E * per_expert > 4 * 148) per_expert >>= 1;
    launch_pdl(permute_kernel<2>, dim3(E, per_expert), dim3(256), 0, st, ids, counts, T * K, E, offsets, perm, pos, x, xp,
               H, K, timeline, sp, (const int32_t*)nullptr, 0);
  }
  else
    launch_pdl(permute_kernel<2>, dim3(E, seg_counts != nullptr ? kPermuteSegments : 1), dim3(256), 0, st, ids, counts,
               T * K, E, offsets, perm, pos, x, xp, H, K, timeline, sp, seg_counts, seg_tokens);
}

namespace {
__global__ void __launch_bounds__(128) report_kernel(RouteReport rep) {
  griddep_launch_dependents();
  griddep_wait();
  publish_report(rep, (int)threadIdx.x, (int)blockDim.x);
}
}  // namespace
void launch_report(cudaStream_t st, const RouteReport& rep) {
  launch_pdl(report_kernel, dim3(1), dim3(128), 0, st, rep);
}

void launch_gather(cudaStream_t st, const uint16_t* x, const int32_t* perm, int T, int H, int K,
                   uint16_t* xp) {
  const size_t total = (size_t)T * K * (H / 8);
  const int blocks = (int)std::min<size_t>((total + 255) / 256, 148 * 16);
  launch_pdl(gather_kernel, dim3(blocks), dim3(256), 0, st, x, perm, T * K, H, K, xp);
}

}  // namespace oled

// ---------------------------------------------------------------------------------------
// Allocation-free routing entry point (no counterpart in the paper).
//
// Some hosts cannot let a library allocate: an inference server that hands every byte of
// device memory to its own arena at start-up, or a latency-critical decode loop in which the
// implicit device-wide synchronisation of cudaMalloc / cudaFree is not acceptable.  For them
// this entry point runs the gate, top-k, gate scores and the token->expert permutation of one
// step without logits or scores in memory, and without scratch: a kernel of one CTA, which waits beside the gate kernel
// and starts when that ends, sorts the assignments, so calls share nothing and may overlap or be replayed in any order.  (As
// three memsets, the gate kernel and the permutation kernel a call of 32 tokens took 16 us, nearly all of it on the host; sorted
// by the gate kernel's last CTA, found by counting in a word that a kernel in front cleared, 9.96; now 8.51.)
namespace oled {
namespace {

__global__ void __launch_bounds__(kStagedWarps * 32)
sort_kernel(const int32_t* ids, int n, int E, int32_t* counts, int32_t* offsets, int32_t* perm) {
  extern __shared__ int s_hist[];
  griddep_launch_dependents();
  griddep_wait();
  sort_assignments<kStagedWarps>(ids, n, E, counts, offsets, perm, s_hist);
}

// Dynamic shared memory of the gate kernel in this role (the one-token form sorts in it).
size_t route_alone_smem(int T, int H, int E) {
  return std::max(staged_smem(T <= 148 ? 1 : 2, H, E), (size_t)kStagedWarps * E * sizeof(int));
}

// The sort indexes by what the gate kernel has stored: it is launched only behind a gate kernel that was.
cudaError_t launch_route_alone(cudaStream_t st, const uint16_t* x, const uint16_t* w_router, const float* bias, const float* conf,
                               int T, int H, int E, int K, int32_t* ids, float* gate, int32_t* counts, const RouteFinish& finish) {
  auto go = [&](auto kernel, int tt) {
    return launch_pdl(kernel, dim3((T + tt - 1) / tt), dim3(kStagedWarps * 32), route_alone_smem(T, H, E), st, x, w_router,
                      bias, conf, T, H, E, K, (float*)nullptr, ids, gate, counts, (unsigned long long*)nullptr, CombinePrev{},
                      (StepTimeline*)nullptr, ScatterRows{}, finish, 0);
  };
  const cudaError_t err = T <= 148 ? go(route_kernel<1, kStagedWarps, 4, 4>, 1) : go(route_kernel<2, kStagedWarps, 4, 4>, 2);
  if (err != cudaSuccess || T == 1) return err;
  return launch_pdl(sort_kernel, dim3(1), dim3(kStagedWarps * 32), (size_t)kStagedWarps * E * sizeof(int), st, (const int32_t*)ids,
                    T * K, E, counts, finish.offsets, finish.perm);
}

}  // namespace
}  // namespace oled

extern "C" int oled_route_noalloc(const void* hidden, const void* w_router, const float* bias,
                                  const float* confidences, int32_t n_tokens, int32_t hidden_dim,
                                  int32_t n_experts, int32_t top_k, void* cuda_stream, int32_t* ids,
                                  float* gate, int32_t* counts, int32_t* offsets, int32_t* perm) {
  using namespace oled;
  if (n_tokens < 0 || hidden_dim <= 0 || hidden_dim % 256 != 0 || n_experts <= 0 ||
      n_experts > OLED_MAX_EXPERTS || top_k <= 0 || top_k > OLED_MAX_TOPK || top_k > n_experts ||
      !counts || !offsets)
    return OLED_ERR_INVALID_ARG;
  if (n_tokens > OLED_NOALLOC_MAX_TOKENS) return OLED_ERR_TOO_MANY_TOKENS;
  if (n_tokens > 0 && (!hidden || !w_router || !confidences || !ids || !gate || !perm))
    return OLED_ERR_INVALID_ARG;
  {  // rows and ids are accessed with 16-byte vectors, everything else as 32-bit words
    auto off = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) != 0; };
    if (off(hidden, 16) || off(w_router, 16) || off(ids, 16) || off(bias, 4) || off(confidences, 4) ||
        off(gate, 4) || off(counts, 4) || off(offsets, 4) || off(perm, 4))
      return OLED_ERR_INVALID_ARG;
  }
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (n_tokens == 0) {
    if (cudaMemsetAsync(counts, 0, (size_t)n_experts * sizeof(int32_t), st) != cudaSuccess ||
        cudaMemsetAsync(offsets, 0, (size_t)(n_experts + 1) * sizeof(int32_t), st) != cudaSuccess) {
      cudaGetLastError();
      return OLED_ERR_CUDA;
    }
    return OLED_OK;
  }
  if (route_alone_smem(n_tokens, hidden_dim, n_experts) > kStagedSmem) return OLED_ERR_INVALID_ARG;
  RouteFinish finish;
  if (!staged_attributes()) return OLED_ERR_CUDA;
  finish.offsets = offsets;
  finish.perm = perm;
  const cudaError_t err = launch_route_alone(st, static_cast<const uint16_t*>(hidden), static_cast<const uint16_t*>(w_router), bias,
                                             confidences, n_tokens, hidden_dim, n_experts, top_k, ids, gate, counts, finish);
  return cudaGetLastError() == cudaSuccess && err == cudaSuccess ? OLED_OK : OLED_ERR_CUDA;
}
