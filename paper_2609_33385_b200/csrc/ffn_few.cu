// Grouped SwiGLU expert FFN of few-token steps (token tiles of at most 128 rows): a weight stream.
//
// Weights on M, tokens on N: the 128 rows of a weight tile fill the MMA's M dimension whatever the
// number of tokens an expert received, so every activated expert's weights cross HBM once.
//   gate/up items: 64 intermediate features, their gate and their up rows in ONE 128-row tile.  A 5-D
//     tensor map lays the rows down as four groups of 16 gate rows and the 16 up rows of the same
//     features, so a feature's two accumulators lie in the same TMEM lane quarter, 16 lanes apart: the
//     epilogue pairs them with a warp shuffle, and a k-block of weights is one copy instruction.
//     hbuf[row, f] = bf16(silu(gate) * up)
//   down items: 128 rows of Wd, y[assignment, c] = D
// KIND 1 / 2: one of the two; KIND 3: the gate/up items, then the down items of the same experts, in one
// launch (a down item's token rows wait, bounded, for its expert's completion counter).
//
// What bounds it: HBM.  At 63 activated experts of 12.6 MB the stream runs at the measured copy rate;
// what a layer loses, it loses BETWEEN streams, while the gate kernel decides who is activated.  So the
// kernel is launched dependent on the gate kernel, which follows the previous layer's FFN in the same way:
// a CTA starts as soon as its SM is free, and loads weights on a GUESS before it knows the routing - the
// experts that the layer activated at its previous execution lead the list (`n_guess` of them; adjacent
// iterations activate mostly the same experts, paper Sec. 3.3), CTA c takes item c of them, fills its ring of
// shared-memory stages with that item's weights and calls the rest of the item into L2.  Slots of
// resident experts are not written while they are resident, so these loads depend on nothing.  When the
// gate is through, the stages only lack their token rows; if the expert was not activated after
// all they are released unread and the CTA draws another item.
// Items other than guesses are drawn from a counter in global memory.
//
// One launch (KIND 3) makes no assumption about which of its CTAs run at the same time: kernels of other streams may hold
// SMs for as long as they like.  Everything a down item waits for is in the hands of a running CTA: counter-drawn
// gate/up items are all drawn before the first down item is, a guess belongs to its CTA only once that CTA has claimed
// it after the gate, and before its first down item a CTA looks whether every guess has been claimed and takes over those
// that have not (after a grace of 10 us; a late owner then drops what it has loaded).  The terms of fp8 rows are
// handed out the same way.  No gate/up item waits for another CTA.
//
// With few experts activated (8 at one token) it is bound by the chain of one CTA's item instead.  Hence the
// roles: one warp loads weights, one loads token rows (each TMA copy is 120 cycles of its thread; with both on one
// thread that thread was the limit: 8 layers of 1 token 282 us against 261 when they were parted; 8 layers of 16 similar tokens 421
// against 384), one issues MMAs, and the epilogue's warps build the work table while the first item already runs.
// A stage's token rows are one copy whatever their number (a tensor map per size of the tile, k-blocks as its slowest
// dimension), and those of a guess are requested as soon as the gate is through, before it is known whether the guess was
// right.  The two together: 8 layers of 1 token 241.2 -> 237.4 us, of 16 similar tokens 368.3 -> 365.6, 16 layers of 32 from fp8 stores
// 1235 -> 1226, 8 layers of 250 from fp8 stores 789 -> 781.
//
// Token rows (FfnRows): dense steps (at most 32 tokens) multiply EVERY expert with all rows of the step,
// stored once, in token order - the tile costs what a gathered one would (N is 16 or 32 either way) and
// no copy of a row per expert exists; the epilogue keeps the columns of the tokens routed to the expert.
// Their intermediate rows are compact (offsets by an exclusive scan of the counts, made by every CTA).
// Scattered and sorted steps find an expert's rows side by side; an item takes the fewest of 16, 32, 48, 64, 96 or
// 128 rows that hold its own.
//
// fp8 expert stores (FP8): the MMAs are kind::f8f6f4 and read the e4m3 codes as they are; the token operand
// is two e4m3 terms per row (fp8_split.h), the epilogue adds the two accumulators (D1 + D2 / 16), undoes the
// row's power-of-two scale and applies the weight row's scale.  The input rows' terms come from the gate
// kernel, those of the intermediate rows from four more warps per CTA (KIND 3) or from split_rows_kernel.  (An M = 128
// instruction consumes 128 weight rows x 32 bytes whatever the element size; widening the codes to bf16 first
// makes the thread that issues the MMAs the bound: 8 layers of 250 tokens 1459 us, now 735.)
//
// Warp roles: warps 0-7 the work table, then the epilogue (lane quarter = warp mod 4, interleaved 16-column
// chunks), warp 8 weights, warp 9 token rows, warp 10 MMA issue; in one
// launch warp 11 counts stored items, and with fp8 stores warps 12-15 make the intermediate rows' terms.  Every wait is bounded as in ffn_tc.cu.
// (Times that stand together in a comment were taken in turn on one machine; machines differ by 5 %, so they do not chain.)
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstddef>

#include "fp8_split.h"
#include "kernels.h"
#include "sm100_ptx.h"

namespace oled {
namespace {

constexpr int kFewEpiWarps = 8;
constexpr int kFewWeightWarp = kFewEpiWarps, kFewTokenWarp = kFewEpiWarps + 1, kFewMmaWarp = kFewEpiWarps + 2;
constexpr int kFewCountWarp = kFewEpiWarps + 3;                           // KIND 3
constexpr int kFewSplitWarp = kFewEpiWarps + 4, kFewSplitWarps = 4;       // KIND 3, fp8 stores
constexpr int few_threads(int kind, bool fp8) { return (kFewEpiWarps + 3 + (kind != 3 ? 0 : fp8 ? 1 + kFewSplitWarps : 1)) * 32; }
constexpr uint32_t kFewWTile = 128 * 128;  // a k-block of weights: 128 rows of 128 bytes (64 bf16 or 128 e4m3)
constexpr int kFewMaxStages = 12;
constexpr int kFewRing = 8;
constexpr uint32_t kFewSmemMax = 232448;  // 227 KB

struct __align__(16) FewCtl {
  unsigned long long full[kFewMaxStages];
  unsigned long long empty[kFewMaxStages];
  unsigned long long item_full[kFewRing];
  unsigned long long item_empty[kFewRing];
  unsigned long long item_stored[kFewRing];  // (one launch) the epilogue warps have stored the item's rows
  unsigned long long tmem_full[2];
  unsigned long long tmem_empty[2];
  unsigned long long table;   // the work table below is complete
  unsigned long long claimed; // (one launch) guess_lost is known
  unsigned long long looked;  // ... guesses_open is
  uint32_t tmem_base;
  int abort;
  int gate_through; // the weight warp is past its dependency wait
  int n_tiles;      // token tiles of the group
  int n_first;      // first-phase (or only) items that are drawn from the counter
  int guess_lost;   // another CTA has taken this one's guess over: its results are not stored
  int guesses_open; // some guess has not been claimed yet, after a grace
  int item_ring[kFewRing];                  // an item as the roles see it: expert of the group, kind, token tile
  int item_m[kFewRing];                     // ... and weight tile
  int count[OLED_MAX_EXPERTS];              // per expert: token rows
  int offsets[OLED_MAX_EXPERTS];            // sorted and dense steps: exclusive scan of the counts
  int tile_prefix[OLED_MAX_EXPERTS + 1];    // per expert of the group: exclusive scan of the token tiles
  int item_prefix[OLED_MAX_EXPERTS + 1];    // ... of the first-phase items left to the counter
};
constexpr uint32_t kFewCtlBytes = (sizeof(FewCtl) + 1023u) & ~1023u;

constexpr unsigned long long kGuessGraceNs = 10000;  // for a CTA to claim its guess after the gate's end
constexpr int kItemNone = -1, kItemAbort = -2, kItemDrop = -3;
// whole: the item multiplies with n_box rows (dense gate/up items, items loaded on a guess), not the fewest that do
__device__ __forceinline__ int pack_item(int g, int down, int whole, int nt) { return g | down << 9 | whole << 10 | nt << 11; }

// Token rows of an item: 16, 32, 48, 64, 96 or 128, and the tensor map whose box is that high.
__host__ __device__ constexpr int few_size(int rows) { return rows <= 64 ? (rows + 15) & ~15 : (rows + 31) & ~31; }
__host__ __device__ constexpr int few_map(int size) { return size <= 64 ? size / 16 - 1 : size / 32 + 1; }

struct FewArgs {
  CUtensorMap tm_w1;    // gate/up weights, 5-D (see ffn_few_setup)
  CUtensorMap tm_w2;    // down-projection weights
  CUtensorMap tm_x[kFewSizes];  // token rows, a box per size (fp8: of their terms)
  CUtensorMap tm_h[kFewSizes];  // intermediate rows
  FfnGroup grp;
  FfnRows rows;
  uint16_t* hbuf;
  float* y;
  int y_bf16;          // y holds bf16 rows (many-token steps)
  int H, I, E;
  int n_stages, k_atoms;
  int n_guess;         // experts at the head of the group that are expected to be activated (0: no guess)
  int early;           // KIND 2: everything but hbuf is known to be older than this kernel's predecessor
  const uint8_t* pool;
  unsigned long long slot_bytes;
  TokenSplit split;          // fp8: the token operands' terms and magnitudes (amax_mid is raised by the gate/up epilogue)
  uint32_t* status;
  uint32_t* work_counter;    // two words, zero at the start: items, and (KIND 3, fp8) rows to split
  uint32_t* claims;          // KIND 3: per CTA, zero at the start: its guess has been claimed (by itself or another)
  uint32_t* done;            // KIND 3: per expert of the group, zero at the start: its gate/up items that have been stored
  uint32_t* split_done;      // KIND 3, fp8: the same for its intermediate rows whose terms have been stored
  StepTimeline* timeline;
  int timeline_slot;
  RouteReport report;
};

__device__ __forceinline__ void few_load_w1(const CUtensorMap* map, uint32_t dst, uint32_t bar, int k, int m, int slot, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6, %7}], [%2], %8;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(k), "r"(0), "r"(0), "r"(m * 4), "r"(slot), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void few_prefetch_w1(const CUtensorMap* map, int k, int m, int slot, uint64_t policy) {
  asm volatile("cp.async.bulk.prefetch.tensor.5d.L2.global.L2::cache_hint [%0, {%1, %2, %3, %4, %5}], %6;"
               ::"l"(map), "r"(k), "r"(0), "r"(0), "r"(m * 4), "r"(slot), "l"(policy)
               : "memory");
}

// One intermediate row (bf16, its largest magnitude final) as two e4m3 terms per element; thread `rank` of `n`.
__device__ __forceinline__ void split_row(const uint16_t* hbuf, const TokenSplit& split, int row, int I, int rank, int n) {
  const float scale = token_scale(__ldcg(split.amax_mid + row));
  const uint4* src = reinterpret_cast<const uint4*>(hbuf + (size_t)row * I);
  uint2* out1 = reinterpret_cast<uint2*>(split.terms_mid + (size_t)row * I);
  uint2* out2 = reinterpret_cast<uint2*>(split.terms_mid + ((size_t)split.rows + row) * I);
  for (int c0 = rank; c0 < I / 8; c0 += 4 * n) {  // (four loads in flight)
    uint4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (c0 + i * n < I / 8) v[i] = __ldcg(src + c0 + i * n);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (c0 + i * n < I / 8) {
        uint2 t1, t2;
        split_bf16x4(v[i].x, v[i].y, scale, t1.x, t2.x);
        split_bf16x4(v[i].z, v[i].w, scale, t1.y, t2.y);
        out1[c0 + i * n] = t1;
        out2[c0 + i * n] = t2;
      }
  }
}

template <int KIND, bool FP8>
__global__ void __launch_bounds__(few_threads(KIND, FP8), 1)
ffn_few_kernel(const __grid_constant__ FewArgs p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  FewCtl* ctl = reinterpret_cast<FewCtl*>(smem_raw);
  const uint32_t tiles_base = (smem_u32(smem_raw) + kFewCtlBytes + 1023u) & ~1023u;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const FfnGroup& grp = p.grp;
  const int n_box = grp.n_box, H = p.H, I = p.I;
  constexpr bool fused = KIND == 3;
  constexpr int kK = FP8 ? 128 : 64;  // k-values of a k-block
  const bool dense = p.rows.dense != 0;
  constexpr uint32_t kRowBytes = FP8 ? 256u : 128u;  // of a token row in a k-block (fp8: two terms)
  // a stage: the weight tiles of its k-blocks, then their token rows (k-block by k-block; fp8: the rows' first terms
  // before the second ones)
  const uint32_t stage_tokens = (uint32_t)p.k_atoms * kFewWTile;
  const uint32_t stage_bytes = stage_tokens + (uint32_t)(p.k_atoms * n_box) * kRowBytes;
  const int k_blocks1 = H / (kK * p.k_atoms), k_blocks2 = I / (kK * p.k_atoms);  // stages per item
  const int m_tiles1 = KIND == 2 ? H / 128 : I / 64;  // weight tiles of the first-phase (or only) items
  const int m_tiles2 = H / 128;
  const int acc_cols = n_box * (FP8 ? 2 : 1);
  const int epi_warps = min(kFewEpiWarps, 4 * (n_box / 16));
  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < 2 * acc_cols) tmem_cols <<= 1;
  volatile int* abort_flag = &ctl->abort;
  // token rows an item multiplies with
  auto size_of = [&](int code) {
    return (code >> 10) & 1 ? n_box : few_size(min(n_box, ctl->count[grp.expert[code & 511]] - (code >> 11) * n_box));
  };
  // first row of an expert's intermediate rows (and of its token rows, unless dense)
  auto first_row = [&](int e) { return p.rows.offsets != nullptr || dense ? ctl->offsets[e] : e * p.rows.cap; };

  // ---- set-up that depends on no earlier kernel
  griddep_launch_dependents();
  const bool guess = KIND != 2 && p.n_guess > 0;
  const bool early = KIND == 2 && p.early != 0;
  const int spec_g = (int)blockIdx.x / m_tiles1, spec_m = (int)blockIdx.x - spec_g * m_tiles1;
  const bool spec = guess && spec_g < p.n_guess && !grp.withhold_loads;
  const int n_spec = guess ? min((int)gridDim.x, p.n_guess * m_tiles1) : 0;  // CTAs with a guess
  const int pre1 = min(p.n_stages, k_blocks1);  // stages that a first item loaded on a guess fills
  // The weights are read once per layer execution and leave L2 first: what the layers hand on and use again - hidden
  // states, outputs, router matrices - then survives the stream.  (Without it those were HBM reads queued behind the
  // next launch's weights: 16 layers of 32 tokens 1996 us, with it 1922; the same fp8 1395 / 1270; 8 layers of 16
  // similar tokens 380 / 356; 8 layers of 250 tokens fp8 894 / 811.)
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
  auto load_weights = [&](int st, int kb, bool down, int m, int slot) {  // one elected lane
    const uint32_t bar = full0 + (uint32_t)st * 8u;
    uint32_t dst = tiles_base + (uint32_t)st * stage_bytes;
    mbar_expect_tx(bar, (uint32_t)p.k_atoms * kFewWTile);
    int k0 = kb * p.k_atoms * kK;
    for (int a = 0; a < p.k_atoms; ++a, k0 += kK, dst += kFewWTile) {
      if (down) tma_load_3d_hint(&p.tm_w2, dst, bar, k0, m * 128, slot, policy);
      else few_load_w1(&p.tm_w1, dst, bar, k0, m, slot, policy);
    }
  };
  if (warp == kFewWeightWarp) {
    if (lane == 0) {
      timeline_entry(p.timeline, p.timeline_slot);
      for (int s = 0; s < p.n_stages; ++s) {
        mbar_init(smem_u32(&ctl->full[s]), 2);  // the weight warp's and the token warp's announcements
        mbar_init(smem_u32(&ctl->empty[s]), 1);
      }
      for (int s = 0; s < kFewRing; ++s) {
        mbar_init(smem_u32(&ctl->item_full[s]), 1);
        // token warp, MMA warp, epilogue warps, counting warp
        mbar_init(smem_u32(&ctl->item_empty[s]), (fused ? 3u : 2u) + (uint32_t)epi_warps);
        mbar_init(smem_u32(&ctl->item_stored[s]), (uint32_t)epi_warps);
      }
      for (int a = 0; a < 2; ++a) {
        mbar_init(smem_u32(&ctl->tmem_full[a]), 1);
        mbar_init(smem_u32(&ctl->tmem_empty[a]), (uint32_t)epi_warps);
      }
      mbar_init(smem_u32(&ctl->table), kFewEpiWarps);
      mbar_init(smem_u32(&ctl->claimed), 1);
      mbar_init(smem_u32(&ctl->looked), 1);
      ctl->abort = 0;
      ctl->gate_through = 0;
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    if (spec && elect_one()) {
      for (int i = 0; i < pre1; ++i) load_weights(i, i, false, spec_m, grp.slot[spec_g]);
    }
    __syncwarp();
  }
  if (warp == kFewTokenWarp) {  // the maps of the loads to come (a guess's own map goes with its loads)
    const int size = few_map(n_box);
    const CUtensorMap* const map = lane == 0 ? &p.tm_w2 : lane == 1 ? p.tm_x + size : lane == 2 ? p.tm_h + size : p.tm_h;
    if (lane < 4) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
  }
  if (warp == kFewMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  auto done_target = [&](int g) { return (uint32_t)m_tiles1 * (uint32_t)(ctl->tile_prefix[g + 1] - ctl->tile_prefix[g]); };
  // (a whole warp) waits until a counter in global memory has reached `target`
  auto wait_count = [&](const uint32_t* counter, uint32_t target, uint32_t sleep_ns) {
    unsigned long long t0 = 0;
    for (uint32_t spin = 0;; ++spin) {
      uint32_t seen;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
      if (__all_sync(0xffffffffu, seen >= target)) return true;
      if (sleep_ns) __nanosleep(sleep_ns);
      if ((spin & 255u) == 255u) {
        const unsigned long long now = globaltimer();
        if (t0 == 0) t0 = now;
        if (now - t0 > kWaitLimitNs) {
          *abort_flag = 1;
          atomicExch(p.status, (uint32_t)kStatusWaitTimeout);
        }
        if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
      }
    }
  };
  auto wait_table = [&]() { return warp_wait(smem_u32(&ctl->table), 0u, abort_flag, p.status); };

  // While the gate kernel runs, a warp with nothing to do before the first item (the counting warp, in two launches the MMA warp)
  // calls the rest of the guessed item into L2: paced, all at once it was a queue that the gate's own loads stood in, and no
  // further once the gate is through, when the ring is to have the memory to itself.  (By the weight warp, on a fixed schedule,
  // it held the first item back: that / this, both with twelve k-blocks in flight, four layers of 64 experts x 2048, 64 tokens 497.6 / 491.8 us,
  // 100 tokens 508.6 / 496.0, x 4096, 100 tokens from fp8 stores 454.4 / 442.6.)  148 CTAs take a k-block each off HBM in 0.37 us; not
  // at all / a pause of 75 / 150 / 300 ns (450 as 300): 8 layers of 1 token 226.5 / 222.9 / 220.3 / 215.1 us, of 16 similar tokens 346.1 /
  // 345.1 / 339.2 / 335.3; 16 layers of 32 tokens 1943 / 1949 / 1939 / 1925, from fp8 stores 1170 / 1175 / 1172 / 1172; 8 layers of 250
  // from fp8 stores 726 / 733 / 733 / 733.  Nothing beyond the item: a line that waits in L2 is read there twice (16 layers of 32 from fp8
  // stores, 64 MB of the following items during the gate 1164 -> 1181; the CTA's next item all along the stream -> 1415).
  auto call_rest_of_guess = [&]() {
    if (!spec) return;
    for (int a = pre1 * p.k_atoms; a < k_blocks1 * p.k_atoms; ++a) {
      if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&ctl->gate_through) != 0)) break;
      if (elect_one()) few_prefetch_w1(&p.tm_w1, a * kK, spec_m, grp.slot[spec_g], policy);
      __nanosleep(300);
    }
    __syncwarp();
  };

  if (warp == kFewWeightWarp) {
    // ------------------------------------------------------------ weights (TMA), and who does what
    int stage = 0, g1 = 0, g2 = 0, seq = 0;
    uint32_t phase = 0;
    bool ok = true;
    if (!early) griddep_wait();
    if (lane == 0) *reinterpret_cast<volatile int*>(&ctl->gate_through) = 1;
    if (lane == 0) timeline_start(p.timeline, p.timeline_slot);
    const bool spec_ok = spec && __ldcg(p.rows.counts + grp.expert[spec_g]) > 0;
    auto publish = [&](int code, int m) {
      const int slot = seq % kFewRing;
      if (!warp_wait(smem_u32(&ctl->item_empty[slot]), ((uint32_t)(seq / kFewRing) & 1u) ^ 1u, abort_flag, p.status))
        return false;
      if (lane == 0) {
        *reinterpret_cast<volatile int*>(&ctl->item_ring[slot]) = code;
        *reinterpret_cast<volatile int*>(&ctl->item_m[slot]) = m;
        mbar_arrive(smem_u32(&ctl->item_full[slot]));
      }
      ++seq;
      return true;
    };
    auto load_item = [&](int kb, int k_blocks, bool down, int m, int slot) {
      for (; kb < k_blocks; ++kb) {
        if (!warp_wait(empty0 + (uint32_t)stage * 8u, phase ^ 1u, abort_flag, p.status)) return false;
        if (elect_one()) load_weights(stage, kb, down, m, slot);
        __syncwarp();
        if (++stage == p.n_stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      return true;
    };
    // First item: the guess, or (two launches, without one) the CTA's own number; later ones from the counter, each
    // number fetched an item ahead.  (With loads withheld - the test of the bounded waits - nothing is published.)
    if (!grp.withhold_loads) {
      const bool drawn_first = guess || fused;
      const int counter_base = drawn_first ? 0 : (int)gridDim.x;
      int item = 0;
      bool guesses_claimed = !(fused && guess);
      if (spec) {
        ok = spec_ok ? publish(pack_item(spec_g, 0, 1, 0), spec_m) : publish(kItemDrop, 0);
        if (lane == 0) item = (int)atomicAdd(p.work_counter, 1u);  // (in flight under the guess's loads)
        stage = pre1 == p.n_stages ? 0 : pre1;
        phase = pre1 == p.n_stages ? 1u : 0u;
        if (ok && spec_ok) ok = load_item(pre1, k_blocks1, false, spec_m, grp.slot[spec_g]);
      } else if (lane == 0) {
        item = drawn_first ? (int)atomicAdd(p.work_counter, 1u) : (int)blockIdx.x;
      }
      item = __shfl_sync(0xffffffffu, item, 0);
      ok = ok && wait_table();
      const int n_first = ctl->n_first, n_items = n_first + (fused ? ctl->n_tiles * m_tiles2 : 0);
      int steal_c0 = 0;          // guesses to take over: looked through so far, and those of the last 32 that are ours
      uint32_t steal_mask = 0;
      while (ok) {
        int g, nt, m, next = item;
        bool down = KIND == 2, whole = false;
        if (item >= n_items) {
          publish(kItemNone, 0);
          break;
        }
        if (item >= n_first && !guesses_claimed) {
          // before the CTA's first down item: every guess that turned out right must have a running CTA
          if (!warp_wait(smem_u32(&ctl->looked), 0u, abort_flag, p.status)) {
            ok = false;
            break;
          }
          if (*reinterpret_cast<volatile int*>(&ctl->guesses_open) != 0)
            for (; steal_mask == 0u && steal_c0 < n_spec; steal_c0 += 32) {
              const int c = steal_c0 + lane;
              const bool needed = c < n_spec && ctl->count[grp.expert[c / m_tiles1]] > 0;
              steal_mask = __ballot_sync(0xffffffffu, needed && atomicExch(p.claims + c, 1u) == 0u);
            }
          guesses_claimed = steal_mask == 0u;
        }
        if (fused && !guesses_claimed && steal_mask != 0u) {
          const int c = steal_c0 - 32 + __ffs((int)steal_mask) - 1;
          steal_mask &= steal_mask - 1u;
          g = c / m_tiles1;
          m = c - g * m_tiles1;
          nt = 0;
          whole = true;
        } else {
          if (item < n_first) {
            while (ctl->item_prefix[g1 + 1] <= item) ++g1;
            g = g1;
            int in = item - ctl->item_prefix[g];
            if (guess && g < p.n_guess) in += min(max((int)gridDim.x - g * m_tiles1, 0), m_tiles1);
            nt = in / m_tiles1;
            m = in - nt * m_tiles1;
          } else {
            const int q = (item - n_first) / m_tiles2;
            m = item - n_first - q * m_tiles2;
            while (ctl->tile_prefix[g2 + 1] <= q) ++g2;
            g = g2;
            nt = q - ctl->tile_prefix[g];
            down = true;
          }
          whole = dense && !down;
          if (lane == 0) next = (int)atomicAdd(p.work_counter, 1u) + counter_base;  // (in flight under this item's loads)
        }
        ok = publish(pack_item(g, down, whole, nt), m) &&
             load_item(0, down ? k_blocks2 : k_blocks1, down, m, grp.slot[g]);
        item = __shfl_sync(0xffffffffu, next, 0);
      }
    }
    if (!ok) {  // let copies already issued land before the CTA's shared memory is released
      const unsigned long long t0 = globaltimer();
      while (globaltimer() - t0 < 2000000ull) {
      }
    }
  } else if (warp == kFewTokenWarp) {
    // ------------------------------------------------------------ token rows (TMA)
    int stage = 0, ready_g = -1;
    uint32_t phase = 0;
    bool ok = true;
    auto load_tokens = [&](int st, int kb, const CUtensorMap* map, int row0, int n) {  // one elected lane
      const uint32_t bar = full0 + (uint32_t)st * 8u;
      const uint32_t dst = tiles_base + (uint32_t)st * stage_bytes + stage_tokens;
      mbar_expect_tx(bar, (uint32_t)(p.k_atoms * n) * kRowBytes);
      if (FP8) tma_load_4d(map, dst, bar, 0, row0, 0, kb * p.k_atoms);
      else tma_load_3d(map, dst, bar, 0, row0, kb * p.k_atoms);
    };
    griddep_wait();
    // A guess: the rows that its expert would have are requested at once, before it is known whether there are any (if not,
    // the stages are completed all the same and released unread).
    const int guess_row0 = spec && !dense ? grp.expert[spec_g] * p.rows.cap : 0;
    if (spec) {
      if (elect_one())
        for (int i = 0; i < pre1; ++i) load_tokens(i, i, p.tm_x + few_map(n_box), guess_row0, n_box);
      __syncwarp();
      stage = pre1 == p.n_stages ? 0 : pre1;
      phase = pre1 == p.n_stages ? 1u : 0u;
    }
    for (int seq = 0; ok; ++seq) {
      const int slot = seq % kFewRing;
      if (!warp_wait(smem_u32(&ctl->item_full[slot]), (uint32_t)(seq / kFewRing) & 1u, abort_flag, p.status)) break;
      const int code = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&ctl->item_ring[slot]), 0);
      if (lane == 0) mbar_arrive(smem_u32(&ctl->item_empty[slot]));
      if (code == kItemNone) break;
      if (code == kItemDrop) continue;
      int k_blocks = k_blocks1, n = n_box, row0 = guess_row0, kb = pre1;
      const bool down = (code >> 9) & 1;
      if (seq != 0 || !spec) {
        const int g = code & 511, nt = code >> 11, e = grp.expert[g];
        if (!(ok = wait_table())) break;
        n = size_of(code);
        if (down) k_blocks = k_blocks2;
        row0 = dense && !down ? 0 : first_row(e) + nt * n_box;
        kb = 0;
        if (fused && down && g != ready_g) {
          // the intermediate rows of every token tile of this expert (fp8: their terms) must be in memory
          ok = FP8 ? wait_count(p.split_done + g, (uint32_t)ctl->count[e], 0u) : wait_count(p.done + g, done_target(g), 0u);
          if (!ok) break;
          ready_g = g;
          // The rows were written through the generic proxy, the loads below read through the async proxy: the one
          // proxy fence between the two stands here.  (On the writers' side as well, and for all state spaces, it
          // waited for the CTA's copies in flight: 6000 to 12800 cycles per item.)
          asm volatile("fence.proxy.async.global;" ::: "memory");
        }
      }
      const CUtensorMap* const map = (down ? p.tm_h : p.tm_x) + few_map(n);
      for (; kb < k_blocks; ++kb) {
        if (!warp_wait(empty0 + (uint32_t)stage * 8u, phase ^ 1u, abort_flag, p.status)) {
          ok = false;
          break;
        }
        if (elect_one()) load_tokens(stage, kb, map, row0, n);
        __syncwarp();
        if (++stage == p.n_stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok) {
      const unsigned long long t0 = globaltimer();
      while (globaltimer() - t0 < 2000000ull) {
      }
    }
  } else if (warp == kFewMmaWarp) {
    // ------------------------------------------------------------ MMA issuer
    // The whole warp runs the loop and one elected lane issues: the operands' descriptors then stay in uniform
    // registers (with a single lane in a divergent branch every MMA instruction cost 79 cycles, most of them
    // spent moving its operands there; now 55).  The two load warps are built the same way.
    int stage = 0, local = 0;
    uint32_t phase = 0;
    bool ok = true;
    const uint32_t stage_step = stage_bytes >> 4;  // descriptor addresses count 16 bytes
    const uint64_t a_desc0 = make_smem_desc(tiles_base), b_desc0 = make_smem_desc(tiles_base + stage_tokens);
    if (!fused) call_rest_of_guess();
    for (int seq = 0; ok; ++seq) {
      const int slot = seq % kFewRing;
      if (!warp_wait(smem_u32(&ctl->item_full[slot]), (uint32_t)(seq / kFewRing) & 1u, abort_flag, p.status)) break;
      const int code = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&ctl->item_ring[slot]), 0);
      if (lane == 0) mbar_arrive(smem_u32(&ctl->item_empty[slot]));
      if (code == kItemNone) break;
      if (code == kItemDrop) {  // a wrong guess: its stages are released unread
        for (int i = 0; i < pre1 && ok; ++i) {
          ok = warp_wait(full0 + (uint32_t)stage * 8u, phase, abort_flag, p.status);
          if (lane == 0) mbar_arrive(empty0 + (uint32_t)stage * 8u);
          if (++stage == p.n_stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        continue;
      }
      const bool whole = (code >> 10) & 1;
      if (!whole && !wait_table()) break;
      const bool down = (code >> 9) & 1;
      const int k_blocks = down ? k_blocks2 : k_blocks1;
      const int acc = local & 1;
      if (!warp_wait(smem_u32(&ctl->tmem_empty[acc]), ((uint32_t)(local >> 1) & 1u) ^ 1u, abort_flag, p.status)) break;
      ++local;
      tc_fence_after();
      const int n = size_of(code);
      const uint32_t idesc = __shfl_sync(0xffffffffu, FP8 ? make_idesc_e4m3(2 * n) : make_idesc(n), 0);
      const uint32_t d0 = __shfl_sync(0xffffffffu, tmem_base + (uint32_t)(acc * acc_cols), 0);
      const uint32_t b_step = __shfl_sync(0xffffffffu, ((uint32_t)n * kRowBytes) >> 4, 0);  // to a stage's second k-block
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!warp_wait(full0 + (uint32_t)stage * 8u, phase, abort_flag, p.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (elect_one()) {
          const uint64_t a0 = a_desc0 + (uint64_t)((uint32_t)stage * stage_step);
          const uint64_t b0 = b_desc0 + (uint64_t)((uint32_t)stage * stage_step);
          // 32 bytes along K = 2 address units
          if (kb == 0) tc_mma_desc<FP8, false>(d0, a0, b0, idesc);
          else tc_mma_desc<FP8, true>(d0, a0, b0, idesc);
#pragma unroll
          for (int k = 1; k < 4; ++k) tc_mma_desc<FP8, true>(d0, a0 + k * 2, b0 + k * 2, idesc);
          if (p.k_atoms == 2) {
#pragma unroll
            for (int k = 0; k < 4; ++k) tc_mma_desc<FP8, true>(d0, a0 + (kFewWTile >> 4) + k * 2, b0 + b_step + k * 2, idesc);
          }
          tc_commit(empty0 + (uint32_t)stage * 8u);
          if (kb + 1 == k_blocks) tc_commit(smem_u32(&ctl->tmem_full[acc]));
        }
        __syncwarp();
        if (++stage == p.n_stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
  } else if (fused && warp == kFewCountWarp) {
    // ------------------------------------------------------------ counts stored gate/up items (one launch)
    // The down items of an expert wait until all of its gate/up items are counted.  The count is a release: it waits
    // until the stores before it are visible device-wide, 2 to 5 us while the stream saturates the memory, so a warp
    // of its own waits and not the epilogue.  Before that it claims the CTA's guess and looks whether every other one is
    // claimed: the weight warp, had it to wait for those answers, would not keep the stream going (a look by it before
    // its first down item cost 0.7 us per layer at one token, 2 us at 32 from fp8 stores).
    bool lost = false;
    if (guess) {
      call_rest_of_guess();
      griddep_wait();
      if (spec) {
        uint32_t taken = 0;
        if (lane == 0) taken = atomicExch(p.claims + blockIdx.x, 1u);
        lost = __shfl_sync(0xffffffffu, taken, 0) != 0u;
      }
      if (lane == 0) {
        *reinterpret_cast<volatile int*>(&ctl->guess_lost) = lost ? 1 : 0;
        mbar_arrive(smem_u32(&ctl->claimed));
      }
      __nanosleep(800);  // (looks that find the others' claims on their way cost 0.2 us per layer)
      const unsigned long long t0 = globaltimer();
      bool open = true, late = false;
      while (open && !late) {
        late = __any_sync(0xffffffffu, globaltimer() - t0 > kGuessGraceNs);
        open = false;
        for (int c = lane; c < n_spec; c += 32) open |= __ldcg(p.claims + c) == 0u;
        open = __any_sync(0xffffffffu, open);
      }
      if (lane == 0) {
        *reinterpret_cast<volatile int*>(&ctl->guesses_open) = open ? 1 : 0;
        mbar_arrive(smem_u32(&ctl->looked));
      }
    }
    for (int seq = 0;; ++seq) {
      const int slot = seq % kFewRing;
      const uint32_t parity = (uint32_t)(seq / kFewRing) & 1u;
      if (!warp_wait(smem_u32(&ctl->item_full[slot]), parity, abort_flag, p.status)) break;
      const int code = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&ctl->item_ring[slot]), 0);
      if (code == kItemNone) break;
      if (!warp_wait(smem_u32(&ctl->item_stored[slot]), parity, abort_flag, p.status)) break;
      if (lane == 0 && code != kItemDrop && !((code >> 9) & 1) && !(lost && seq == 0)) red_release_add(p.done + (code & 511), 1u);
      // (handed back only now: the barrier above is not used again before this warp has seen its phase)
      if (lane == 0) mbar_arrive(smem_u32(&ctl->item_empty[slot]));
    }
  } else if (FP8 && fused && warp >= kFewSplitWarp) {
    // ------------------------------------------------------------ terms of the intermediate rows (fp8, one launch)
    // A task is every `workers`-th row of one expert, and the warps draw them from a counter (a fixed share per CTA
    // would wait for CTAs that have no SM yet): as soon as all of the expert's gate/up items are stored, the rows'
    // magnitudes are final and the rows become two e4m3 terms each.  All gate/up items are handed out before the
    // first down item, so that is over long before most down items need it, and the weight stream runs on.  (As a kernel
    // between two launches it cost 8 of 80 us per layer of 32 tokens.)
    if (wait_table() && !grp.withhold_loads) {
      const int workers = max(1, (int)gridDim.x / grp.n) * kFewSplitWarps;  // warps per expert
      for (;;) {
        const int task = __shfl_sync(0xffffffffu, lane == 0 ? (int)atomicAdd(p.work_counter + 1, 1u) : 0, 0);
        if (task >= grp.n * workers) break;
        const int w = task / grp.n, g = task - w * grp.n;
        const int e = grp.expert[g], count = ctl->count[e], row0 = first_row(e);
        if (w >= count) continue;  // (no row of this expert is this task's)
        if (!wait_count(p.done + g, done_target(g), 500u)) break;
        uint32_t mine = 0;
        for (int r = w; r < count; r += workers, ++mine) split_row(p.hbuf, p.split, row0 + r, I, lane, 32);
        __syncwarp();
        if (lane == 0) red_release_add(p.split_done + g, mine);
      }
    }
  } else {
    // ------------------------------------------------------------ the work table, then the epilogue
    if (!early) griddep_wait();
    const int tid = threadIdx.x;
    for (int e = tid; e < p.E; e += kFewEpiWarps * 32) {
      if (p.rows.offsets != nullptr) {
        const int o = __ldcg(p.rows.offsets + e);
        ctl->offsets[e] = o;
        ctl->count[e] = __ldcg(p.rows.offsets + e + 1) - o;
      } else {
        ctl->count[e] = __ldcg(p.rows.counts + e);
      }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kFewEpiWarps * 32) : "memory");
    if (warp == 0) {  // token tiles and counter-drawn items of the group, 32 experts at a time
      int tiles_before = 0, items_before = 0;
      for (int g0 = 0; g0 < grp.n; g0 += 32) {
        const int g = g0 + lane;
        const int tiles = g < grp.n ? (ctl->count[grp.expert[g]] + n_box - 1) / n_box : 0;
        // items of this expert that a CTA has taken on a guess: those of its first token tile below the grid size
        int items = tiles * m_tiles1;
        if (guess && g < p.n_guess && tiles > 0) items -= min(max((int)gridDim.x - g * m_tiles1, 0), m_tiles1);
        int ti = tiles, ii = items;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int o = __shfl_up_sync(0xffffffffu, ti, d), q = __shfl_up_sync(0xffffffffu, ii, d);
          if (lane >= d) {
            ti += o;
            ii += q;
          }
        }
        if (g < grp.n) {
          ctl->tile_prefix[g] = tiles_before + ti - tiles;
          ctl->item_prefix[g] = items_before + ii - items;
        }
        tiles_before += __shfl_sync(0xffffffffu, ti, 31);
        items_before += __shfl_sync(0xffffffffu, ii, 31);
      }
      if (lane == 0) {
        ctl->tile_prefix[grp.n] = tiles_before;
        ctl->item_prefix[grp.n] = items_before;
        ctl->n_tiles = tiles_before;
        ctl->n_first = items_before;
      }
    } else if (warp == 1 && dense) {  // compact intermediate rows: the scan over all experts
      int carry = 0;
      for (int e0 = 0; e0 < p.E; e0 += 32) {
        const int c = e0 + lane < p.E ? ctl->count[e0 + lane] : 0;
        int incl = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int o = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += o;
        }
        if (e0 + lane < p.E) ctl->offsets[e0 + lane] = carry + incl - c;
        carry += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&ctl->table));
    // the step's report to the host: its trip across the link ends long before this kernel does
    if (KIND != 2 && blockIdx.x == 0 && warp == kFewEpiWarps - 1) publish_report(p.report, lane, 32);
    const bool live = warp < epi_warps && wait_table();
    const int quarter = warp & 3;  // this warp's lanes; its columns: every epi_warps / 4-th chunk of 16
    if (early) griddep_wait();  // (the rows' magnitudes below are products of the predecessor)
    int local = 0;
    for (int seq = 0; live; ++seq) {
      int code = kItemAbort, m = 0;
      if (lane == 0) {
        const int slot = seq % kFewRing;
        if (mbar_wait(smem_u32(&ctl->item_full[slot]), (uint32_t)(seq / kFewRing) & 1u, abort_flag, p.status)) {
          code = *reinterpret_cast<volatile int*>(&ctl->item_ring[slot]);
          m = *reinterpret_cast<volatile int*>(&ctl->item_m[slot]);
          mbar_arrive(smem_u32(&ctl->item_empty[slot]));
        }
      }
      code = __shfl_sync(0xffffffffu, code, 0);
      m = __shfl_sync(0xffffffffu, m, 0);
      if (code == kItemDrop) {
        if (fused && lane == 0) mbar_arrive(smem_u32(&ctl->item_stored[seq % kFewRing]));
        continue;
      }
      if (code < 0) break;
      const int g = code & 511, nt = code >> 11;
      const bool down = KIND == 2 || (fused && ((code >> 9) & 1));
      const int e = grp.expert[g], count = ctl->count[e], row1 = first_row(e);
      const int n = size_of(code);
      const int acc = local & 1;
      const uint32_t acc_phase = (uint32_t)(local >> 1) & 1u;
      ++local;
      const int valid = min(n_box, count - nt * n_box);
      // the columns of a chunk: `row` = the intermediate row of the calling lane's column (-1: none), `inv` (fp8) the
      // inverse of its token row's power-of-two scale, `dst` (down) where its output goes
      //   dense gate/up: column t is token t; its place among the expert's rows is looked up
      //   otherwise: column j is row first + nt * n_box + j
      auto columns = [&](int c, int& row, int& dst, float& inv) {
        const int my_col = c + (lane & 15);
        row = my_col < valid ? row1 + nt * n_box + my_col : -1;
        dst = row;
        if (p.rows.assignment != nullptr) {
          if (dense && !down) {
            const int tok = lane < count ? __ldcg(p.rows.assignment + e * p.rows.cap + lane) / p.rows.K : -1;
            row = -1;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const uint32_t hit = __ballot_sync(0xffffffffu, tok == c + j);
              if ((lane & 15) == j && hit != 0u) row = row1 + __ffs((int)hit) - 1;
            }
          } else if (down && row >= 0) {
            dst = __ldcg(p.rows.assignment + e * p.rows.cap + nt * n_box + my_col);
          }
        }
        if (FP8) inv = row >= 0 ? token_scale_inverse(__ldcg(down ? p.split.amax_mid + row : p.split.amax_in + (dense ? my_col : row))) : 0.0f;
      };
      // fp8 stores: one fp32 scale per weight row behind the codes (s_gate[I] | s_up[I] | s_down[H])
      float s0 = 1.0f;
      if (FP8) {
        const float* sc = reinterpret_cast<const float*>(p.pool + (size_t)grp.slot[g] * p.slot_bytes + (size_t)3 * H * I);
        s0 = down ? sc[2 * I + m * 128 + quarter * 32 + lane]
                  : sc[(lane >= 16 ? I : 0) + m * 64 + quarter * 16 + (lane & 15)];
      }
      const int step = 4 * epi_warps;
      int c = (warp >> 2) * 16;
      int row = -1, dst = 0;
      float inv = 0.0f;
      // looked up while the MMAs still run - but the magnitudes of intermediate rows that this launch itself makes
      // are final only once the item's MMAs are through
      const bool ahead = !(FP8 && fused && down);
      if (c < n && ahead) columns(c, row, dst, inv);
      int ready = 0;
      if (lane == 0) ready = mbar_wait(smem_u32(&ctl->tmem_full[acc]), acc_phase, abort_flag, p.status) ? 1 : 0;
      ready = __shfl_sync(0xffffffffu, ready, 0);
      if (!ready) break;
      tc_fence_after();
      bool lost = false;  // (another CTA computes and stores this guess)
      if (fused && spec && seq == 0) {
        if (!warp_wait(smem_u32(&ctl->claimed), 0u, abort_flag, p.status)) break;
        lost = *reinterpret_cast<volatile int*>(&ctl->guess_lost) != 0;
        if (lost) row = -1;
      }
      for (bool first = true; first || c < n; first = false, c += step) {
        const bool last = c + step >= n;
        uint32_t ra[16];
        if (c < n) {
          const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * acc_cols + c);
          tmem_ld16(t_row, ra);
          if (!first || !ahead) {
            columns(c, row, dst, inv);
            if (lost) row = -1;
          }
          if (FP8) {  // D = (D1 + D2 / 16) / row scale of the token
            uint32_t rt[16];
            tmem_ld16(t_row + (uint32_t)n, rt);  // (the second terms' columns lie behind the first ones')
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 16; ++j)
              ra[j] = __float_as_uint(__fmaf_rn(__uint_as_float(rt[j]), 0.0625f, __uint_as_float(ra[j])) *
                                      __shfl_sync(0xffffffffu, inv, j) * s0);
          } else {
            tmem_ld_wait();
          }
        }
        if (last) {  // the accumulators are in registers: the MMAs of the item after next may have the columns
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&ctl->tmem_empty[acc]));
        }
        if (c >= n) break;
        if (!down) {
          // lane l < 16 holds the gate row of feature l of this quarter, lane l + 16 its up row: the lower half
          // of the warp finishes columns 0-7 of the chunk, the upper half columns 8-15
          const bool up_half = lane >= 16;
          const int f = m * 64 + quarter * 16 + (lane & 15);
          uint32_t mag[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float mine = __uint_as_float(up_half ? ra[8 + j] : ra[j]);
            const float got = __shfl_xor_sync(0xffffffffu, __uint_as_float(up_half ? ra[j] : ra[8 + j]), 16);
            const int r = __shfl_sync(0xffffffffu, row, (up_half ? 8 : 0) + j);
            const float a = up_half ? got : mine, u = up_half ? mine : got;
            const float hm = __fdividef(a, 1.0f + __expf(-a)) * u;
            const __nv_bfloat16 b = __float2bfloat16_rn(hm);
            mag[j] = 0u;
            if (r >= 0) {
              p.hbuf[(size_t)r * I + f] = *reinterpret_cast<const uint16_t*>(&b);
              mag[j] = (uint32_t)(*reinterpret_cast<const uint16_t*>(&b) & 0x7fffu);
            }
          }
          if (FP8) {
            // the rows' largest magnitudes, for the down projection's token scaling: 8 columns over 16 lanes,
            // half of the columns handed over at every step
#pragma unroll
            for (int d = 8, k = 4; d >= 2; d >>= 1, k >>= 1) {
              const bool hi = (lane & d) != 0;
#pragma unroll
              for (int i = 0; i < k; ++i) {
                const uint32_t keep = hi ? mag[i + k] : mag[i], send = hi ? mag[i] : mag[i + k];
                mag[i] = max(keep, __shfl_xor_sync(0xffffffffu, send, d));
              }
            }
            const uint32_t top = max(mag[0], __shfl_xor_sync(0xffffffffu, mag[0], 1));
            // lane bits 3, 2, 1 = bits 2, 1, 0 of the column within the half
            const int r = __shfl_sync(0xffffffffu, row, (up_half ? 8 : 0) + ((lane >> 1) & 7));
            if ((lane & 1) == 0 && r >= 0 && top != 0u) atomicMax(p.split.amax_mid + r, top << 16);
          }
        } else if (c < valid) {
          const size_t col = (size_t)(m * 128 + quarter * 32 + lane);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const size_t o = (size_t)__shfl_sync(0xffffffffu, dst, j) * H + col;
            if (c + j < valid) {
              if (p.y_bf16) reinterpret_cast<__nv_bfloat16*>(p.y)[o] = __float2bfloat16_rn(__uint_as_float(ra[j]));
              else p.y[o] = __uint_as_float(ra[j]);
            }
          }
        }
      }
      if (fused) {
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctl->item_stored[seq % kFewRing]));
      }
    }
  }

  // ---- teardown.  Every way out passes the dependency wait, so that no kernel of a step completes before
  // its predecessors have (an early-start CTA without an item reaches it only here).
  if (early) griddep_wait();
  tc_fence_before();
  __syncthreads();
  if (warp == kFewMmaWarp) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
  if (threadIdx.x == 0) timeline_end(p.timeline, p.timeline_slot);
}

// fp8 stores, between the two projections as two launches: the intermediate rows of the group's experts (bf16,
// written by the gate/up epilogue together with every row's largest magnitude) as two e4m3 terms
// per element.  Four CTAs per expert of the group (a quarter of the columns each); a warp takes a
// row at a time.
__global__ void __launch_bounds__(256)
split_rows_kernel(const __grid_constant__ FfnGroup grp, const __grid_constant__ FfnRows rows,
                  const uint16_t* __restrict__ hbuf, const __grid_constant__ TokenSplit split, int I) {
  griddep_launch_dependents();
  griddep_wait();
  const int e = grp.expert[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int first = rows.first(e);
  const int count = rows.count(e);
  if (rows.dense) {  // compact rows: the counts of the experts before this one (each warp adds them up for itself)
    first = 0;
    for (int i = lane; i < e; i += 32) first += rows.counts[i];
    first = __reduce_add_sync(0xffffffffu, first);
  }
  for (int r = first + warp; r < first + count; r += 8)
    split_row(hbuf, split, r, I, lane + 32 * (int)blockIdx.y, 32 * (int)gridDim.y);
}

// Stage shape and count: two k-blocks per stage where at least three such stages fit and both contractions
// have an even number of them (half the waits and commits on the MMA thread); ten bf16 k-blocks in flight
// at most, eight of e4m3 codes (16 tokens, 8 layers: 557 us, with ten 569).  Tiles of 16 rows have room for twelve bf16 ones, which
// gains at hidden 2048 with 64 experts only (layers of 1 token with twelve / ten 26.5 / 26.7 us, of 16 similar tokens 41.4 / 42.1); elsewhere it costs:
// four layers of 64 experts, 4096 x 768, 1 token 173.2 / 155.8 us, 3072 x 768, 5 tokens 308.5 / 300.6, 768 x 1024, 16 tokens 187.6 / 183.8,
// of 128 experts, 2048 x 768, 8 tokens 316.1 / 309.9.
struct FewRings {
  int stages, k_atoms;
  uint32_t smem;
};
FewRings few_rings(int n_box, bool fp8, int H, int I) {
  const uint32_t atom = kFewWTile + (uint32_t)n_box * 128u * (fp8 ? 2u : 1u);
  const int kblocks = (int)std::min<uint32_t>(fp8 ? 8u : 10u, (kFewSmemMax - kFewCtlBytes - 1024u) / atom);
  const int kk = fp8 ? 128 : 64;
  FewRings r;
  r.k_atoms = kblocks >= 6 && (H / kk) % 2 == 0 && (I / kk) % 2 == 0 ? 2 : 1;
  r.stages = std::min(kblocks / r.k_atoms, kFewMaxStages);
  r.smem = kFewCtlBytes + 1024u + (uint32_t)(r.stages * r.k_atoms) * atom;
  return r;
}

}  // namespace

int ffn_few_setup(FfnTcMaps* maps, const uint8_t* pool, size_t slot_bytes, int n_slots, int H, int I, bool fp8,
                  const uint16_t* xp, const uint16_t* hbuf, int rows, const TokenSplit* split) {
  const cuuint64_t esz = fp8 ? 1 : 2;
  const cuuint32_t k_box = fp8 ? 128u : 64u;
  {
    // [slot][I / 16 groups][gate | up][16 rows][H]: a box of four groups is the 64 gate and 64 up rows of 64 features
    const cuuint64_t dims[5] = {(cuuint64_t)H, 16, 2, (cuuint64_t)(I / 16), (cuuint64_t)n_slots};
    const cuuint64_t strides[4] = {(cuuint64_t)H * esz, (cuuint64_t)I * H * esz, (cuuint64_t)16 * H * esz, (cuuint64_t)slot_bytes};
    const cuuint32_t box[5] = {k_box, 16, 2, 4, 1};
    if (!encode_tensor_map(&maps->few_w1, 5, pool, dims, strides, box, fp8)) return OLED_ERR_CUDA;
  }
  {
    const cuuint64_t dims[3] = {(cuuint64_t)I, (cuuint64_t)H, (cuuint64_t)n_slots};
    const cuuint64_t strides[2] = {(cuuint64_t)I * esz, (cuuint64_t)slot_bytes};
    const cuuint32_t box[3] = {k_box, 128, 1};
    if (!encode_tensor_map(&maps->few_w2, 3, pool + (size_t)2 * I * H * esz, dims, strides, box, fp8)) return OLED_ERR_CUDA;
  }
  for (int atoms = 1; atoms <= 2; ++atoms)  // token rows, intermediate rows: k-blocks as the slowest dimension, so that a
    for (int size : {16, 32, 48, 64, 96, 128})  // stage's rows are one copy (fp8: [k-block][term][row][k])
      for (int op = 0; op < 2; ++op) {
        const cuuint64_t width = (cuuint64_t)(op == 0 ? H : I);
        const void* base = fp8 ? (const void*)(op == 0 ? split->terms_in : split->terms_mid) : (const void*)(op == 0 ? xp : hbuf);
        const cuuint64_t k_blocks = width / k_box, term_stride = width * (cuuint64_t)rows;
        const cuuint64_t dims[4] = {k_box, (cuuint64_t)rows, fp8 ? 2 : k_blocks, k_blocks};
        const cuuint64_t strides[3] = {width * esz, fp8 ? term_stride : 128, 128};
        const cuuint32_t box[4] = {k_box, (cuuint32_t)size, fp8 ? 2u : (cuuint32_t)atoms, (cuuint32_t)atoms};
        CUtensorMap* const m = (op == 0 ? maps->few_x : maps->few_h)[atoms - 1] + few_map(size);
        if (!encode_tensor_map(m, fp8 ? 4 : 3, base, dims, strides, box, fp8)) return OLED_ERR_CUDA;
      }
  maps->few = true;
  static const bool attr_ok = [] {
    return cudaFuncSetAttribute(ffn_few_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess &&
           cudaFuncSetAttribute(ffn_few_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess &&
           cudaFuncSetAttribute(ffn_few_kernel<3, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess &&
           cudaFuncSetAttribute(ffn_few_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess &&
           cudaFuncSetAttribute(ffn_few_kernel<3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess &&
           cudaFuncSetAttribute(ffn_few_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess;
  }();
  return attr_ok ? OLED_OK : OLED_ERR_CUDA;
}

int launch_ffn_few(cudaStream_t st, const FfnTcMaps& maps, const FfnGroup& group, int max_count, int kind,
                   const int32_t* host_counts, const FfnRows& rows, uint16_t* hbuf, float* y, int y_bf16, int H, int I, int n_sms,
                   uint32_t* status, uint32_t* work_counter, bool behind_event_wait, StepTimeline* timeline,
                   int timeline_slot, const RouteReport& report, uint32_t* done, const TokenSplit* split,
                   uint32_t* split_done, uint32_t* claims) {
  const bool fp8 = maps.fp8;
  if (kind == 3 && (done == nullptr || claims == nullptr || (fp8 && split_done == nullptr))) return OLED_ERR_INVALID_ARG;  // callers ask ffn_tc_can_fuse() first
  FewArgs a;
  a.tm_w1 = maps.few_w1;
  a.tm_w2 = maps.few_w2;
  a.grp = group;
  const FfnGroup& grp = a.grp;
  a.grp.n_box = few_size(std::min(max_count, kFewMaxRows));
  const FewRings r = few_rings(grp.n_box, fp8, H, I);
  for (int i = 0; i < kFewSizes; ++i) {
    a.tm_x[i] = maps.few_x[r.k_atoms - 1][i];
    a.tm_h[i] = maps.few_h[r.k_atoms - 1][i];
  }
  a.y_bf16 = y_bf16;
  a.rows = rows;
  a.hbuf = hbuf;
  a.y = y;
  a.H = H;
  a.I = I;
  a.E = rows.E;
  a.n_stages = r.stages;
  a.k_atoms = r.k_atoms;
  // a guess needs to know at once whether the expert has tokens (counts), and every CTA of the full grid
  a.n_guess = kind != 2 && host_counts == nullptr && rows.offsets == nullptr ? std::min(grp.n_guess, grp.n) : 0;
  // A kind 2 launch reads everything but hbuf ahead of its dependency wait where nothing else can still
  // be in the making: either every SM holds a CTA of the kind 1 launch before it (full grid; two CTAs do
  // not share an SM, so a kind 2 CTA runs only where a kind 1 CTA, which waited for the gate, has left),
  // or the launch pair sits behind an event wait, which completes everything enqueued before it.
  a.early = kind == 2 && (behind_event_wait || host_counts == nullptr) && 2 * r.smem > 228u * 1024u ? 1 : 0;
  a.pool = maps.pool;
  a.slot_bytes = (unsigned long long)maps.slot_bytes;
  if (fp8) a.split = *split;
  a.status = status;
  a.work_counter = work_counter;
  a.done = done;
  a.split_done = split_done;
  a.claims = claims;
  a.timeline = timeline;
  a.timeline_slot = timeline_slot;
  a.report = report;
  int grid = n_sms;
  if (host_counts != nullptr) {  // fewer CTAs if the group has fewer items than SMs
    long long tiles = 0;
    for (int g = 0; g < grp.n; ++g) tiles += (host_counts[grp.expert[g]] + grp.n_box - 1) / grp.n_box;
    const int per_tile = (kind != 2 ? I / 64 : 0) + (kind != 1 ? H / 128 : 0);
    grid = (int)std::max<long long>(1, std::min<long long>(n_sms, tiles * per_tile));
  }
  if (kind == 2 && fp8)  // the intermediate rows as e4m3 terms, now that their magnitudes are complete
    launch_pdl(split_rows_kernel, dim3(grp.n, 4), dim3(256), 0, st, grp, rows, (const uint16_t*)hbuf,
               *split, I);
  launch_pdl(fp8 ? (kind == 3 ? ffn_few_kernel<3, true> : kind == 2 ? ffn_few_kernel<2, true> : ffn_few_kernel<1, true>)
                 : (kind == 3 ? ffn_few_kernel<3, false> : kind == 2 ? ffn_few_kernel<2, false> : ffn_few_kernel<1, false>),
             dim3(grid), dim3(few_threads(kind, fp8)), r.smem, st, a);
  return cudaGetLastError() == cudaSuccess ? OLED_OK : OLED_ERR_CUDA;
}

}  // namespace oled
