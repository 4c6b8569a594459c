// Grouped SwiGLU expert FFN of few-token steps (token tiles of at most 32 rows): a weight stream.
//
// Weights on M, tokens on N: the 128 rows of a weight tile fill the MMA's M dimension whatever the
// number of tokens an expert received, so every activated expert's weights cross HBM once.
//   gate/up items: 64 intermediate features, their gate and their up rows in ONE 128-row tile.  A 5-D
//     tensor map lays the rows down as four groups of 16 gate rows and the 16 up rows of the same
//     features, so a feature's two accumulators lie in the same TMEM lane quarter, 16 lanes apart: the
//     epilogue pairs them with a warp shuffle, and a k-block of weights is one copy instruction.
//     hbuf[row, f] = bf16(silu(gate) * up)
//   down items: 128 rows of Wd, y[assignment, c] = D (fp32)
// KIND 1 / 2: one of the two; KIND 3: the gate/up items, then the down items of the same experts, in one
// launch (a down item waits, bounded, for its expert's completion counter).
//
// What bounds it: HBM.  At 63 activated experts of 12.6 MB the stream runs at the measured copy rate;
// what a layer loses, it loses BETWEEN streams, while the gate kernel decides who is activated.  So:
//   * the CTA is small (320 threads; a gate CTA fits beside it) and the kernel is launched dependent on
//     the gate kernel, which follows the previous layer's FFN in the same way: a CTA starts as soon as
//     its SM is free, and loads weights on a GUESS before it knows the routing - the experts that the
//     layer activated at its previous execution lead the list (`n_guess` of them; adjacent iterations
//     activate mostly the same experts, paper Sec. 3.3), CTA c takes item c of them, fills its ring of
//     shared-memory stages with that item's weights and calls the rest of the item into L2.  Slots of
//     resident experts are not written while they are resident, so these loads depend on nothing.  When the
//     gate is through, the stages only lack their token tiles; if the expert was not activated after
//     all they are dropped (the MMA thread releases them unread) and the CTA draws another item.
// Items other than the first are drawn from a counter in global memory and published to the CTA's other
// roles through a ring in shared memory, as in ffn_tc.cu.
//
// Token rows (FfnRows): dense steps (at most 32 tokens) multiply EVERY expert with all rows of the step,
// stored once, in token order - the tile costs what a gathered one would (N is 16 or 32 either way) and
// no copy of a row per expert exists; the epilogue keeps the columns of the tokens routed to the expert.
// Their intermediate rows are compact (offsets by an exclusive scan of the counts, made by every CTA).
// Scattered and sorted steps find an expert's rows side by side.
//
// fp8 expert stores (FP8): the MMAs are kind::f8f6f4 and read the e4m3 codes as they are; the token operand
// is two e4m3 terms per row (fp8_split.h), the epilogue adds the two accumulators (D1 + D2 / 16), undoes the
// row's power-of-two scale and applies the weight row's scale.  The input rows' terms come from the gate
// kernel, those of the intermediate rows from split_rows_kernel between the two projections.
//
// Warp roles: warps 0-7 epilogue (lane quarter = warp mod 4, 16-column chunk = warp / 4), warp 8 lane 0 TMA
// producer, warp 9 MMA issuer.  Every wait is bounded as in ffn_tc.cu.
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
constexpr int kFewProducerWarp = kFewEpiWarps, kFewMmaWarp = kFewEpiWarps + 1;
constexpr int kFewThreads = (kFewEpiWarps + 2) * 32;
constexpr uint32_t kFewWTile = 128 * 128;  // a k-block of weights: 128 rows of 128 bytes (64 bf16 or 128 e4m3)
constexpr int kFewMaxStages = 12;
constexpr int kFewRing = 8;
constexpr uint32_t kFewSmemMax = 232448;  // 227 KB

struct __align__(16) FewCtl {
  unsigned long long full[kFewMaxStages];
  unsigned long long empty[kFewMaxStages];
  unsigned long long item_full[kFewRing];
  unsigned long long item_empty[kFewRing];
  unsigned long long tmem_full[2];
  unsigned long long tmem_empty[2];
  uint32_t tmem_base;
  int abort;
  int n_tiles;      // token tiles of the group
  int n_first;      // first-phase (or only) items that are drawn from the counter
  int item_ring[kFewRing];
  int count[OLED_MAX_EXPERTS];              // per expert of the group: token rows
  int first[OLED_MAX_EXPERTS];              // first row of its intermediate rows (and of its token rows, unless dense)
  int tile_prefix[OLED_MAX_EXPERTS + 1];    // exclusive scan of the token tiles
  int item_prefix[OLED_MAX_EXPERTS + 1];    // exclusive scan of the first-phase items left to the counter
  int offsets[OLED_MAX_EXPERTS];            // dense steps: exclusive scan of ALL experts' counts
};
constexpr uint32_t kFewCtlBytes = (sizeof(FewCtl) + 1023u) & ~1023u;

// An item as the roles see it, packed for the ring: expert of the group, kind, token tile, weight tile.
constexpr int kItemNone = -1, kItemAbort = -2, kItemDrop = -3;
__device__ __forceinline__ int pack_item(int g, int down, int nt, int m) { return g | down << 9 | nt << 10 | m << 20; }

struct FewArgs {
  CUtensorMap tm_w1;   // gate/up weights, 5-D (see ffn_few_setup)
  CUtensorMap tm_x;    // token rows (fp8: their terms)
  CUtensorMap tm_w2;   // down-projection weights
  CUtensorMap tm_h;    // intermediate rows (fp8: their terms)
  FfnGroup grp;
  FfnRows rows;
  uint16_t* hbuf;
  float* y;
  int H, I, E;
  int n_stages, k_atoms;
  int n_guess;         // experts at the head of the group that are expected to be activated (0: no guess)
  int early;           // KIND 2: everything but hbuf is known to be older than this kernel's predecessor
  const uint8_t* pool;
  unsigned long long slot_bytes;
  const uint32_t* amax_act;  // fp8: magnitudes of the token operand's rows (kind 1: input, kind 2: intermediate)
  uint32_t* amax_out;        // fp8, kind 1: raised by the epilogue
  uint32_t* status;
  uint32_t* work_counter;    // zero at the start
  uint32_t* done;            // KIND 3: per expert of the group, zero at the start
  StepTimeline* timeline;
  int timeline_slot;
  RouteReport report;
};

__device__ __forceinline__ void few_load_w1(const CUtensorMap* map, uint32_t dst, uint32_t bar, int k, int m, int slot) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(k), "r"(0), "r"(0), "r"(m * 4), "r"(slot)
      : "memory");
}
__device__ __forceinline__ void few_prefetch_w1(const CUtensorMap* map, int k, int m, int slot) {
  asm volatile("cp.async.bulk.prefetch.tensor.5d.L2.global [%0, {%1, %2, %3, %4, %5}];"
               ::"l"(map), "r"(k), "r"(0), "r"(0), "r"(m * 4), "r"(slot)
               : "memory");
}

template <int KIND, bool FP8>
__global__ void __launch_bounds__(kFewThreads, 1)
ffn_few_kernel(const __grid_constant__ FewArgs p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  FewCtl* ctl = reinterpret_cast<FewCtl*>(smem_raw);
  const uint32_t tiles_base = (smem_u32(smem_raw) + kFewCtlBytes + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const FfnGroup& grp = p.grp;
  const int n_box = grp.n_box, H = p.H, I = p.I;
  constexpr bool fused = KIND == 3;
  static_assert(!(fused && FP8), "fp8 stores need the split kernel between the two projections");
  constexpr int kK = FP8 ? 128 : 64;  // k-values of a k-block
  const bool dense = p.rows.dense != 0;
  const uint32_t act_bytes = (uint32_t)n_box * 128u * (FP8 ? 2u : 1u);
  const uint32_t atom_bytes = kFewWTile + act_bytes;
  const uint32_t stage_bytes = (uint32_t)p.k_atoms * atom_bytes;
  const int k_blocks1 = H / (kK * p.k_atoms), k_blocks2 = I / (kK * p.k_atoms);  // stages per item
  const int m_tiles1 = KIND == 2 ? H / 128 : I / 64;  // weight tiles of the first-phase (or only) items
  const int m_tiles2 = H / 128;
  const int acc_cols = n_box * (FP8 ? 2 : 1);
  const int epi_warps = min(kFewEpiWarps, 4 * (n_box / 16));
  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < 2 * acc_cols) tmem_cols <<= 1;
  volatile int* abort_flag = &ctl->abort;

  // ---- set-up that depends on no earlier kernel
  griddep_launch_dependents();
  const bool guess = KIND != 2 && p.n_guess > 0;
  const bool early = KIND == 2 && p.early != 0;
  const int spec_g = (int)blockIdx.x / m_tiles1, spec_m = (int)blockIdx.x - spec_g * m_tiles1;
  const bool spec = guess && spec_g < p.n_guess && !grp.withhold_loads;
  const int pre1 = min(p.n_stages, KIND == 2 ? k_blocks2 : k_blocks1);  // stages a first item can fill
  auto load_weights = [&](int st, int kb, bool down, int m, int slot) {
    const uint32_t bar = smem_u32(&ctl->full[st]);
    mbar_expect_tx(bar, stage_bytes);
    for (int a = 0; a < p.k_atoms; ++a) {
      const uint32_t dst = tiles_base + (uint32_t)st * stage_bytes + (uint32_t)a * atom_bytes;
      const int k0 = (kb * p.k_atoms + a) * kK;
      if (down) tma_load_3d(&p.tm_w2, dst, bar, k0, m * 128, slot);
      else few_load_w1(&p.tm_w1, dst, bar, k0, m, slot);
    }
  };
  auto load_tokens = [&](int st, int kb, bool down, int row0) {
    const uint32_t bar = smem_u32(&ctl->full[st]);
    for (int a = 0; a < p.k_atoms; ++a) {
      const uint32_t dst = tiles_base + (uint32_t)st * stage_bytes + (uint32_t)a * atom_bytes + kFewWTile;
      const int k0 = (kb * p.k_atoms + a) * kK;
      if (FP8) tma_load_3d(down ? &p.tm_h : &p.tm_x, dst, bar, k0, row0, 0);  // (both terms in one box)
      else tma_load_2d(down ? &p.tm_h : &p.tm_x, dst, bar, k0, row0);
    }
  };
  if (warp == kFewProducerWarp && lane == 0) {
    timeline_entry(p.timeline, p.timeline_slot);
    for (int s = 0; s < kFewMaxStages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int s = 0; s < kFewRing; ++s) {
      mbar_init(smem_u32(&ctl->item_full[s]), 1);
      mbar_init(smem_u32(&ctl->item_empty[s]), 1u + (uint32_t)epi_warps);  // the MMA thread, a lane of every epilogue warp
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&ctl->tmem_full[a]), 1);
      mbar_init(smem_u32(&ctl->tmem_empty[a]), (uint32_t)epi_warps);
    }
    ctl->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (spec) {
      for (int i = 0; i < pre1; ++i) load_weights(i, i, false, spec_m, grp.slot[spec_g]);
      for (int a = pre1 * p.k_atoms; a < k_blocks1 * p.k_atoms; ++a)
        few_prefetch_w1(&p.tm_w1, a * kK, spec_m, grp.slot[spec_g]);
    }
  }
  if (warp == kFewMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (!early) griddep_wait();
  if (threadIdx.x == 0) timeline_start(p.timeline, p.timeline_slot);
  // ---- the routing is known: the guessed item's token tiles go at once, the work table follows
  if (KIND != 2 && blockIdx.x == 0 && warp == kFewProducerWarp && lane != 0) publish_report(p.report, lane - 1, 31);
  bool spec_ok = false;
  uint32_t drawn = 0;  // (producer) the next item number
  if (warp == kFewProducerWarp && lane == 0) {
    if (!grp.withhold_loads) drawn = guess ? atomicAdd(p.work_counter, 1u) : 0u;
    if (spec) {
      const int e = grp.expert[spec_g];
      spec_ok = __ldcg(p.rows.counts + e) > 0;
      const int row0 = spec_ok && !dense ? e * p.rows.cap : 0;
      for (int i = 0; i < pre1; ++i) load_tokens(i, i, false, row0);  // (dropped stages are completed, too)
    }
  }
  if (p.rows.offsets != nullptr) {
    for (int g = threadIdx.x; g < grp.n; g += kFewThreads) {
      const int e = grp.expert[g], o = __ldcg(p.rows.offsets + e);
      ctl->first[g] = o;
      ctl->count[g] = __ldcg(p.rows.offsets + e + 1) - o;
    }
  } else {
    for (int g = threadIdx.x; g < grp.n; g += kFewThreads) {
      ctl->count[g] = __ldcg(p.rows.counts + grp.expert[g]);
      ctl->first[g] = grp.expert[g] * p.rows.cap;
    }
    if (dense && warp == 1) {  // compact intermediate rows: the scan over all experts
      int carry = 0;
      for (int e0 = 0; e0 < p.E; e0 += 32) {
        const int c = e0 + lane < p.E ? __ldcg(p.rows.counts + e0 + lane) : 0;
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
  }
  __syncthreads();
  if (warp == 0) {  // token tiles and counter-drawn items of the group, 32 experts at a time
    int tiles_before = 0, items_before = 0;
    for (int g0 = 0; g0 < grp.n; g0 += 32) {
      const int g = g0 + lane;
      const int tiles = g < grp.n ? (ctl->count[g] + n_box - 1) / n_box : 0;
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
        if (dense) ctl->first[g] = ctl->offsets[grp.expert[g]];
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
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  const int n_first = ctl->n_first, n_items = n_first + (fused ? ctl->n_tiles * m_tiles2 : 0);
  // KIND 3: epilogue warps that store intermediate rows per gate/up item, times the items of a token tile
  const uint32_t done_per_tile = (uint32_t)(m_tiles1 * epi_warps);

  if (warp == kFewProducerWarp && lane == 0) {
    // ------------------------------------------------------------ TMA producer
    int stage = 0, ready_g = -1, g1 = 0, g2 = 0;
    uint32_t phase = 0;
    bool ok = true;
    auto advance = [&]() {
      if (++stage == p.n_stages) {
        stage = 0;
        phase ^= 1u;
      }
    };
    int seq = 0;
    auto publish = [&](int code) {
      const int slot = seq % kFewRing;
      if (!mbar_wait(smem_u32(&ctl->item_empty[slot]), ((uint32_t)(seq / kFewRing) & 1u) ^ 1u, abort_flag, p.status))
        return false;
      *reinterpret_cast<volatile int*>(&ctl->item_ring[slot]) = code;
      mbar_arrive(smem_u32(&ctl->item_full[slot]));
      ++seq;
      return true;
    };
    // first item: the guess, or (without one) the CTA's own number; later ones from the counter
    int item = guess ? (int)drawn : (int)blockIdx.x;
    const int counter_base = guess ? 0 : (int)gridDim.x;
    bool first_guess = spec && spec_ok;
    if (spec)
      for (int i = 0; i < pre1; ++i) advance();
    if (spec && !spec_ok) ok = publish(kItemDrop);
    // (with loads withheld - the test of the bounded waits - nothing is published either)
    while (ok && !grp.withhold_loads) {
      int g, nt, m, kb = 0;
      bool down = KIND == 2;
      if (first_guess) {
        g = spec_g;
        nt = 0;
        m = spec_m;
        kb = pre1;
      } else {
        if (item >= n_items) {
          publish(kItemNone);
          break;
        }
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
        // the number after this one is fetched now: the atomic's latency lies under this item's loads
        item = (int)atomicAdd(p.work_counter, 1u) + counter_base;
      }
      first_guess = false;
      if (!publish(pack_item(g, down, nt, m))) {
        ok = false;
        break;
      }
      const int slot = grp.slot[g];
      const int row0 = (dense && !down ? 0 : ctl->first[g]) + nt * n_box;
      const int k_blocks = down ? k_blocks2 : k_blocks1;
      if (early && seq == 1) {
        // weights of the first stages now, token tiles once the predecessor is done
        for (int i = 0; i < pre1; ++i) load_weights(i, i, true, m, slot);
        griddep_wait();
        for (int i = 0; i < pre1; ++i) {
          load_tokens(i, i, true, row0);
          advance();
        }
        kb = pre1;
      }
      if (fused && down) {
        // The intermediate rows of every token tile of this expert must be in memory.  If they are not
        // yet, the weights of as many stages as the ring holds go first, then the wait, then their tokens.
        const uint32_t* flag = p.done + g;
        const uint32_t target = done_per_tile * (uint32_t)(ctl->tile_prefix[g + 1] - ctl->tile_prefix[g]);
        uint32_t seen = target;
        if (g != ready_g) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(flag) : "memory");
        int pre = 0;
        const int stage0 = stage;
        if (seen < target) {
          pre = min(p.n_stages, k_blocks);
          for (int i = 0; i < pre && ok; ++i) {
            if (!mbar_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag, p.status)) {
              ok = false;
              break;
            }
            load_weights(stage, i, true, m, slot);
            advance();
          }
          unsigned long long t0 = 0;
          for (uint32_t spin = 0; ok; ++spin) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(flag) : "memory");
            if (seen >= target) break;
            if ((spin & 255u) == 255u) {
              if (*abort_flag) ok = false;
              const unsigned long long now = globaltimer();
              if (t0 == 0) t0 = now;
              if (now - t0 > kWaitLimitNs) {
                *abort_flag = 1;
                atomicExch(p.status, (uint32_t)kStatusWaitTimeout);
                ok = false;
              }
            }
          }
          if (!ok) break;
        }
        ready_g = g;
        // the rows were written through the generic proxy; the loads below read through the async proxy
        asm volatile("fence.proxy.async;" ::: "memory");
        for (int i = 0, st = stage0; i < pre; ++i) {
          load_tokens(st, i, true, row0);
          if (++st == p.n_stages) st = 0;
        }
        kb = pre;
      }
      for (; kb < k_blocks; ++kb) {
        if (!mbar_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag, p.status)) {
          ok = false;
          break;
        }
        load_weights(stage, kb, down, m, slot);
        load_tokens(stage, kb, down, row0);
        advance();
      }
    }
    if (!ok) {  // let copies already issued land before the CTA's shared memory is released
      const unsigned long long t0 = globaltimer();
      while (globaltimer() - t0 < 2000000ull) {
      }
    }
  } else if (warp == kFewMmaWarp) {
    // ------------------------------------------------------------ MMA issuer
    // The whole warp runs the loop and one elected lane issues: the operands' descriptors then stay in uniform
    // registers (with a single lane in a divergent branch every MMA instruction cost 79 cycles, most of them
    // spent moving its operands there).
    int stage = 0, local = 0;
    uint32_t phase = 0;
    bool ok = true;
    const uint32_t ring_step = atom_bytes >> 4, stage_step = stage_bytes >> 4;  // descriptor addresses count 16 bytes
    const uint64_t a_desc0 = make_smem_desc(tiles_base), b_desc0 = make_smem_desc(tiles_base + kFewWTile);
    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
    for (int seq = 0; ok; ++seq) {
      const int slot = seq % kFewRing;
      if (!mbar_wait(smem_u32(&ctl->item_full[slot]), (uint32_t)(seq / kFewRing) & 1u, abort_flag, p.status)) break;
      const int code = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&ctl->item_ring[slot]), 0);
      if (lane == 0) mbar_arrive(smem_u32(&ctl->item_empty[slot]));
      if (code == kItemNone) break;
      if (code == kItemDrop) {  // a wrong guess: its stages are released unread
        for (int i = 0; i < pre1 && ok; ++i) {
          ok = mbar_wait(full0 + (uint32_t)stage * 8u, phase, abort_flag, p.status);
          __syncwarp();
          if (lane == 0) mbar_arrive(empty0 + (uint32_t)stage * 8u);
          if (++stage == p.n_stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        continue;
      }
      const int g = code & 511, nt = (code >> 10) & 1023;
      const bool down = (code >> 9) & 1;
      const int k_blocks = down ? k_blocks2 : k_blocks1;
      const int acc = local & 1;
      if (!mbar_wait(smem_u32(&ctl->tmem_empty[acc]), ((uint32_t)(local >> 1) & 1u) ^ 1u, abort_flag, p.status)) break;
      ++local;
      tc_fence_after();
      const int valid = min(n_box, ctl->count[g] - nt * n_box);
      const int n_mma = dense && !down ? n_box : max(16, (valid + 15) & ~15);
      const uint32_t idesc = __shfl_sync(0xffffffffu, FP8 ? make_idesc_e4m3(2 * n_box) : make_idesc(n_mma), 0);
      const uint32_t d0 = __shfl_sync(0xffffffffu, tmem_base + (uint32_t)(acc * acc_cols), 0);
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait(full0 + (uint32_t)stage * 8u, phase, abort_flag, p.status)) {
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
            for (int k = 0; k < 4; ++k) tc_mma_desc<FP8, true>(d0, a0 + ring_step + k * 2, b0 + ring_step + k * 2, idesc);
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
  } else if (warp < epi_warps) {
    // ------------------------------------------------------------ epilogue
    const int quarter = warp & 3, c = (warp >> 2) * 16;  // this warp's lanes and its 16 columns
    if (early) griddep_wait();  // (the rows' magnitudes below are products of the predecessor)
    int local = 0;
    for (int seq = 0;; ++seq) {
      int code = kItemAbort;
      if (lane == 0) {
        const int slot = seq % kFewRing;
        if (mbar_wait(smem_u32(&ctl->item_full[slot]), (uint32_t)(seq / kFewRing) & 1u, abort_flag, p.status)) {
          code = *reinterpret_cast<volatile int*>(&ctl->item_ring[slot]);
          mbar_arrive(smem_u32(&ctl->item_empty[slot]));
        }
      }
      code = __shfl_sync(0xffffffffu, code, 0);
      if (code == kItemDrop) continue;
      if (code < 0) break;
      const int g = code & 511, nt = (code >> 10) & 1023, m = code >> 20;
      const bool down = KIND == 2 || (fused && ((code >> 9) & 1));
      const int e = grp.expert[g], count = ctl->count[g];
      const int acc = local & 1;
      const uint32_t acc_phase = (uint32_t)(local >> 1) & 1u;
      ++local;
      // what the columns are: `row` = the intermediate row of the calling lane's column (-1: none)
      //   dense gate/up: column t is token t; its place among the expert's rows is looked up
      //   otherwise: column j is row first + nt * n_box + j
      const int valid = min(n_box, count - nt * n_box);
      const int my_col = c + (lane & 15);
      int row = my_col < valid ? ctl->first[g] + nt * n_box + my_col : -1;
      int dst = row;  // down: where the row's output goes
      if (p.rows.assignment != nullptr) {
        if (dense && !down) {
          const int tok = lane < count ? __ldcg(p.rows.assignment + e * p.rows.cap + lane) / p.rows.K : -1;
          row = -1;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const uint32_t hit = __ballot_sync(0xffffffffu, tok == c + j);
            if ((lane & 15) == j && hit != 0u) row = ctl->first[g] + __ffs((int)hit) - 1;
          }
        } else if (down && row >= 0) {
          dst = __ldcg(p.rows.assignment + e * p.rows.cap + nt * n_box + my_col);
        }
      }
      // fp8 stores: one fp32 scale per weight row behind the codes (s_gate[I] | s_up[I] | s_down[H]), and the
      // inverse of the token row's power-of-two scale
      float s0 = 1.0f, inv = 0.0f;
      if (FP8) {
        const float* sc = reinterpret_cast<const float*>(p.pool + (size_t)grp.slot[g] * p.slot_bytes + (size_t)3 * H * I);
        s0 = down ? sc[2 * I + m * 128 + quarter * 32 + lane]
                  : sc[(lane >= 16 ? I : 0) + m * 64 + quarter * 16 + (lane & 15)];
        const int arow = dense && !down ? my_col : row;
        if (row >= 0) inv = token_scale_inverse(__ldcg(p.amax_act + arow));
      }
      int ready = 0;
      if (lane == 0) ready = mbar_wait(smem_u32(&ctl->tmem_full[acc]), acc_phase, abort_flag, p.status) ? 1 : 0;
      ready = __shfl_sync(0xffffffffu, ready, 0);
      if (!ready) break;
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * acc_cols + c);
      // (columns that no row of this item uses are not read; the MMA did not write those beyond its N)
      const bool any = dense && !down ? true : c < valid;
      uint32_t ra[16];
      if (any) {
        tmem_ld16(t_row, ra);
        if (FP8) {  // D = (D1 + D2 / 16) / row scale of the token
          uint32_t rt[16];
          tmem_ld16(t_row + (uint32_t)n_box, rt);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j)
            ra[j] = __float_as_uint(__fmaf_rn(__uint_as_float(rt[j]), 0.0625f, __uint_as_float(ra[j])) *
                                    __shfl_sync(0xffffffffu, inv, j) * s0);
        } else {
          tmem_ld_wait();
        }
      }
      // the accumulators are in registers: the MMAs of the item after next may have the columns
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl->tmem_empty[acc]));
      if (any && !down) {
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
          for (int d = 8, n = 4; d >= 2; d >>= 1, n >>= 1) {
            const bool hi = (lane & d) != 0;
#pragma unroll
            for (int i = 0; i < n; ++i) {
              const uint32_t keep = hi ? mag[i + n] : mag[i], send = hi ? mag[i] : mag[i + n];
              mag[i] = max(keep, __shfl_xor_sync(0xffffffffu, send, d));
            }
          }
          const uint32_t top = max(mag[0], __shfl_xor_sync(0xffffffffu, mag[0], 1));
          // lane bits 3, 2, 1 = bits 2, 1, 0 of the column within the half
          const int r = __shfl_sync(0xffffffffu, row, (up_half ? 8 : 0) + ((lane >> 1) & 7));
          if ((lane & 1) == 0 && r >= 0 && top != 0u) atomicMax(p.amax_out + r, top << 16);
        }
        if (fused) {
          // this warp's intermediate rows of the item are stored: make them visible device-wide
          __threadfence();
          asm volatile("fence.proxy.async;" ::: "memory");
        }
      } else if (any) {
        float* const y = p.y + m * 128 + quarter * 32 + lane;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int d = __shfl_sync(0xffffffffu, dst, j);
          if (c + j < valid) y[(size_t)d * H] = __uint_as_float(ra[j]);
        }
      }
      if (fused && !down) {  // ... and count the warp in (the down items of this expert wait for the full count)
        __syncwarp();
        if (lane == 0) atomicAdd(p.done + g, 1u);
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

// fp8 stores, between the two projections: the intermediate rows of the group's experts (bf16,
// written by the gate/up epilogue together with every row's largest magnitude) as two e4m3 terms
// per element.  Four CTAs per expert of the group (a quarter of the columns each); a warp takes a
// row at a time.
__global__ void __launch_bounds__(256)
split_rows_kernel(const __grid_constant__ FfnGroup grp, const __grid_constant__ FfnRows rows,
                  const uint16_t* __restrict__ hbuf, const uint32_t* __restrict__ amax_mid,
                  uint8_t* __restrict__ terms_mid, int I, int rows_total) {
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
  for (int r = first + warp; r < first + count; r += 8) {
    const float scale = token_scale(amax_mid[r]);
    const uint4* src = reinterpret_cast<const uint4*>(hbuf + (size_t)r * I);
    uint2* out1 = reinterpret_cast<uint2*>(terms_mid + (size_t)r * I);
    uint2* out2 = reinterpret_cast<uint2*>(terms_mid + ((size_t)rows_total + r) * I);
    for (int c = lane + 32 * (int)blockIdx.y; c < I / 8; c += 32 * (int)gridDim.y) {
      const uint4 v = src[c];
      uint2 t1, t2;
      split_bf16x4(v.x, v.y, scale, t1.x, t2.x);
      split_bf16x4(v.z, v.w, scale, t1.y, t2.y);
      out1[c] = t1;
      out2[c] = t2;
    }
  }
}

// Stage shape and count: two k-blocks per stage where at least four such stages fit and both contractions
// have an even number of them (half the waits and commits on the MMA thread); ten bf16 k-blocks in flight
// at most (eleven measured slower), twelve of e4m3 codes.
struct FewRings {
  int stages, k_atoms;
  uint32_t smem;
};
FewRings few_rings(int n_box, bool fp8, int H, int I) {
  const uint32_t atom = kFewWTile + (uint32_t)n_box * 128u * (fp8 ? 2u : 1u);
  const int kblocks = (int)std::min<uint32_t>(fp8 ? 12u : 10u, (kFewSmemMax - kFewCtlBytes - 1024u) / atom);
  const int kk = fp8 ? 128 : 64;
  FewRings r;
  r.k_atoms = kblocks >= 8 && (H / kk) % 2 == 0 && (I / kk) % 2 == 0 ? 2 : 1;
  r.stages = std::min(kblocks / r.k_atoms, kFewMaxStages);
  r.smem = kFewCtlBytes + 1024u + (uint32_t)(r.stages * r.k_atoms) * atom;
  return r;
}

}  // namespace

int ffn_few_setup(FfnTcMaps* maps, const uint8_t* pool, size_t slot_bytes, int n_slots, int H, int I, bool fp8) {
  // [slot][I / 16 groups][gate | up][16 rows][H]: a box of four groups is the 64 gate and 64 up rows of 64 features
  const cuuint64_t esz = fp8 ? 1 : 2;
  const cuuint64_t dims[5] = {(cuuint64_t)H, 16, 2, (cuuint64_t)(I / 16), (cuuint64_t)n_slots};
  const cuuint64_t strides[4] = {(cuuint64_t)H * esz, (cuuint64_t)I * H * esz, (cuuint64_t)16 * H * esz, (cuuint64_t)slot_bytes};
  const cuuint32_t box[5] = {fp8 ? 128u : 64u, 16, 2, 4, 1};
  if (!encode_tensor_map(fp8 ? &maps->w13_few_e4m3 : &maps->w13_few, 5, pool, dims, strides, box, fp8)) return OLED_ERR_CUDA;
  static const bool attr_ok = [] {
    return cudaFuncSetAttribute(ffn_few_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess &&
           cudaFuncSetAttribute(ffn_few_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess &&
           cudaFuncSetAttribute(ffn_few_kernel<3, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess &&
           cudaFuncSetAttribute(ffn_few_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess &&
           cudaFuncSetAttribute(ffn_few_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax) == cudaSuccess;
  }();
  return attr_ok ? OLED_OK : OLED_ERR_CUDA;
}

int launch_ffn_few(cudaStream_t st, const FfnTcMaps& maps, const FfnGroup& grp, int box_index, int kind,
                   const int32_t* host_counts, const FfnRows& rows, uint16_t* hbuf, float* y, int H, int I, int n_sms,
                   uint32_t* status, uint32_t* work_counter, bool behind_event_wait, StepTimeline* timeline,
                   int timeline_slot, const RouteReport& report, uint32_t* done, const TokenSplit* split) {
  const bool fp8 = maps.fp8;
  if (kind == 3 && (fp8 || done == nullptr)) return OLED_ERR_INVALID_ARG;  // callers ask ffn_tc_can_fuse() first
  const FewRings r = few_rings(grp.n_box, fp8, H, I);
  FewArgs a;
  a.tm_w1 = fp8 ? maps.w13_few_e4m3 : maps.w13_few;
  a.tm_x = fp8 ? maps.xp_terms[box_index] : maps.xp[box_index];
  a.tm_w2 = fp8 ? maps.w2_e4m3 : maps.w2;
  a.tm_h = fp8 ? maps.hbuf_terms[box_index] : maps.hbuf[box_index];
  a.grp = grp;
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
  a.amax_act = !fp8 ? nullptr : kind == 2 ? split->amax_mid : split->amax_in;
  a.amax_out = fp8 && kind == 1 ? split->amax_mid : nullptr;
  a.status = status;
  a.work_counter = work_counter;
  a.done = done;
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
               (const uint32_t*)split->amax_mid, split->terms_mid, I, split->rows);
  if (fp8) launch_pdl(kind == 2 ? ffn_few_kernel<2, true> : ffn_few_kernel<1, true>, dim3(grid), dim3(kFewThreads), r.smem, st, a);
  else
    launch_pdl(kind == 3 ? ffn_few_kernel<3, false> : kind == 2 ? ffn_few_kernel<2, false> : ffn_few_kernel<1, false>,
               dim3(grid), dim3(kFewThreads), r.smem, st, a);
  return cudaGetLastError() == cudaSuccess ? OLED_OK : OLED_ERR_CUDA;
}

}  // namespace oled
