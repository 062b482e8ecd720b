// Tensor-core ST-SpAttn prefill (Sec. 3.2) for bf16, head_dim 128, on sm_100a.
//
// Persistent kernel: one CTA per SM walks the list of work units the plan assigned to it.  A unit is a
// 128-row query tile of a PAIR of query heads that share a KV head ("slots") and a chunk of that tile's
// list of kept key tiles, so every K/V tile staged in shared memory feeds two heads and key blocks the
// mask removes are never read.  With an odd number of heads per KV head the group's last head is worked on by both
// slots for two consecutive query tiles over the union of their lists (a twin unit), each slot with its own tile
// classes and bit masks.  Roles:
//   warp 8      producer: per unit Q of both slots, then per key tile the tile's class word and, for
//               general tiles, its bit mask (bulk copy) into a small ring, and K and V (TMA, 128-byte
//               swizzle, two 64-column panels each) into a ring of stages.  It runs ahead across units.
//   warp 9      owns the 512 TMEM columns; one lane issues tcgen05.mma, alternating slots:
//               S = Q K^T (K-major A and B from shared memory) and
//               O += P V (A = bf16 P from TMEM, B = V as MN-major shared-memory operand),
//               so the tensor pipe works on one slot while the other slot's rows are in softmax.
//   warps 0-7   one thread per query row of a slot (registers raised with setmaxnreg at the expense of
//               warps 8-11): the row of S from TMEM into registers, the
//               tile's predicate (none / causal / bit mask), online softmax in the log2 domain against a
//               reference that moves only when exp2 would overflow (then O is rescaled), bf16 P written
//               over S; at the end of a unit either the normalised output (whole list in one unit; whole query
//               tiles go to shared memory for warp 10 to copy out) or an unnormalised fp32 partial result plus (max, sum) per row
//               into the workspace.  The warp that finishes its rows of a split list last (a counter in the plan)
//               combines the partial results in chunk order, so the result does not depend on timing.
// Every wait on an mbarrier is bounded in time; on expiry the CTA raises a shared abort flag,
// sets the device status word, drains, frees TMEM and exits.
#include <type_traits>

#include "prefill.cuh"
#include "tc_util.cuh"

namespace purekv {
namespace tc {

constexpr int kBQ = 128;
constexpr int kThreads = 384;  // warps 0-3 softmax of slot 0, warps 4-7 of slot 1, warp 8 producer, warp 9 MMA, warp 10 output, 11 idle
constexpr int kWarpProducer = 8, kWarpMma = 9, kWarpStore = 10;
// Per-thread registers after the warpgroups trade them.  setmaxnreg only moves registers inside the CTA's launch
// allocation (kThreads x the count ptxas gives the kernel, 168 at 384 threads); asking for more would block forever,
// so the launch code checks the budget against the compiled register count.
constexpr int kRegsSoftmax = 208, kRegsOther = 88;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColO = 256;
constexpr int kUnitRing = 4;  // units in flight between the producer's publication and the other roles' copies

template <int BK>
struct Cfg {
  static constexpr int kStages = 2;                 // K/V ring depth (64 KB per stage)
  static constexpr int kMeta = 2 * kStages;         // ring of per-tile class words and bit masks
  static constexpr uint32_t kMaskBytes = kBQ * BK / 8;
};

template <int BK>
struct __align__(8) Barriers {
  static constexpr int ST = Cfg<BK>::kStages, MR = Cfg<BK>::kMeta;
  uint64_t q_full, q_empty;
  uint64_t k_full[ST], k_empty[ST], v_full[ST], v_empty[ST];
  uint64_t m_full[MR];     // producer -> softmax: class word (and bit mask) of a tile are in place
  uint64_t s_full[2];      // MMA -> softmax: S of the slot is complete
  uint64_t p_part[2];      // softmax -> MMA: P of the first 96 keys written (and O rescaled) by the slot's four row warps
  uint64_t p_full[2];      // softmax -> MMA: all of P written
  uint64_t o_final[2];     // one completion per unit, after the slot's last P.V product
  uint64_t u_full[kUnitRing];   // the producer published a unit (or the end mark) in unit_s[]
  uint64_t u_empty[kUnitRing];  // the MMA thread, the eight softmax warps and the storing thread have copied it
  uint64_t o_staged[2][ST];  // softmax -> storing thread: the slot's output tile is in that stage.  A barrier per stage, because
                             // a slot may be a unit of one tile (in the other stage) ahead of the copies; a stage is its own
                             // again only when the storing thread has given it back, which is after its wait
  uint64_t drain;
};

// TMEM columns: S(slot) at slot*128 (P aliases its first BK/2 columns), O(slot) at 256 + slot*128.
template <int BK>
__global__ void __launch_bounds__(kThreads, 1) prefill_tc_kernel(
    const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
    const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_k64,
    const __grid_constant__ CUtensorMap tm_v64, const __grid_constant__ CUtensorMap tm_o, __nv_bfloat16* __restrict__ o, float* __restrict__ lse,
    uint8_t* __restrict__ plan, float* __restrict__ ws, int32_t n_q_heads, int32_t n_kv_heads, float scale_log2,
    int32_t* __restrict__ status, uint64_t wait_ns, int64_t plan_bytes, int64_t ws_floats, int32_t n_units, int32_t n_layers,
    int64_t o_stride, int64_t lse_stride) {
  constexpr int ST = Cfg<BK>::kStages, MR = Cfg<BK>::kMeta;
  constexpr uint32_t kPanelQ = kBQ * 128;  // bytes of one 64-column panel of a Q tile
  constexpr uint32_t kTileQ = 2 * kPanelQ;
  constexpr uint32_t kPanelKV = BK * 128;  // bytes of one 64-column panel of a K or V tile
  constexpr uint32_t kTileKV = 2 * kPanelKV;
  constexpr uint32_t kMaskBytes = Cfg<BK>::kMaskBytes;
  extern __shared__ uint8_t smem_raw[];
  __shared__ Barriers<BK> bars;
  __shared__ int2 meta_s[MR][2];  // per slot: the entry word, and the byte offset in shared memory of the slot's bit mask plus the halves loaded
  __shared__ Unit unit_s[kUnitRing];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  __shared__ int abort_code_s;  // what the status word becomes if the CTA gives up: an expired wait unless set otherwise

  const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = smem0;                 // [2 slots][2 panels][128 rows x 128 B]
  const uint32_t sK = sQ + 2 * kTileQ;       // [ST][2 panels][BK rows x 128 B]
  const uint32_t sV = sK + ST * kTileKV;
  const uint32_t sM = sV + ST * kTileKV;     // [MR][2 slots][128 rows x BK/8 B]

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // Programmatic dependent launch: the next kernel in the stream may start its CTAs as ours retire and set up its
  // barriers and TMEM meanwhile; nothing the previous kernel may have written is read before griddep_wait below.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  volatile int* abort_flag = &abort_s;

  if (tid == 0) {
    mbar_init(smem_u32(&bars.q_full), 1);
    mbar_init(smem_u32(&bars.q_empty), 1);
    for (int s = 0; s < ST; ++s) {
      mbar_init(smem_u32(&bars.k_full[s]), 1);
      mbar_init(smem_u32(&bars.k_empty[s]), 1);
      mbar_init(smem_u32(&bars.v_full[s]), 1);
      mbar_init(smem_u32(&bars.v_empty[s]), 1);
    }
    for (int s = 0; s < MR; ++s) mbar_init(smem_u32(&bars.m_full[s]), 1);
    for (int sl = 0; sl < 2; ++sl) {
      mbar_init(smem_u32(&bars.s_full[sl]), 1);
      mbar_init(smem_u32(&bars.p_full[sl]), 4);
      mbar_init(smem_u32(&bars.p_part[sl]), 4);
      mbar_init(smem_u32(&bars.o_final[sl]), 1);
      for (int s = 0; s < ST; ++s) mbar_init(smem_u32(&bars.o_staged[sl][s]), 4);
    }
    for (int s = 0; s < kUnitRing; ++s) {
      mbar_init(smem_u32(&bars.u_full[s]), 1);
      mbar_init(smem_u32(&bars.u_empty[s]), 10);
    }
    mbar_init(smem_u32(&bars.drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kWarpMma) {
    tmem_alloc(smem_u32(&tmem_base_s), kTmemCols);
    tmem_relinquish();
  }
  // The maps' descriptors are fetched beside the barriers' set-up, not by the first copies (64 units 15.5 -> 15.4 us, 512 35.4 -> 35.3).
  if (warp == 11 && lane < 6) {
    const CUtensorMap* map = lane == 0 ? &tm_q : lane == 1 ? &tm_k : lane == 2 ? &tm_v : lane == 3 ? &tm_k64 : lane == 4 ? &tm_v64 : &tm_o;
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the stream's earlier work is complete and visible from here on
  if (tid == 0) {
    abort_s = *reinterpret_cast<volatile int32_t*>(status) != 0;  // an earlier CTA or launch already failed
    abort_code_s = (int)PUREKV_ERR_TIMEOUT;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  const PlanHeader* hdr = reinterpret_cast<const PlanHeader*>(plan);
  // The plan is checked before anything is read through it: the header's own fields here (by every thread, on the
  // same values, so the decision is uniform), each unit and each list entry by the producer before it publishes or
  // uses them.  A plan that fails is not used: the status word becomes PUREKV_ERR_BAD_PLAN and the CTA leaves.
  bool plan_ok = plan_bytes >= (int64_t)sizeof(PlanHeader);
  if (plan_ok) {
    const int64_t G_ = n_kv_heads > 0 ? n_q_heads / n_kv_heads : 0;
    auto section = [&](int64_t off, int64_t count, int64_t elem) {
      return off >= (int64_t)sizeof(PlanHeader) && (off & 15) == 0 && count >= 0 && count <= plan_bytes / elem &&
             off <= plan_bytes - count * elem;
    };
    plan_ok = hdr->magic == kPlanMagic && hdr->tile_q == kBQ && hdr->tile_k == BK && hdr->words_per_row == BK / 32 &&
              hdr->n_q_heads == n_q_heads && hdr->n_kv_heads == n_kv_heads && G_ >= 1 &&
              hdr->n_ctas == (int32_t)gridDim.x && hdr->n_units == n_units && hdr->n_counters >= 0 &&
              section(hdr->off_entries, hdr->n_entries, 8) && section(hdr->off_masks, hdr->n_mask_words, 4) &&
              hdr->n_mask_words >= hdr->n_entries &&
              section(hdr->off_units, hdr->n_units, (int64_t)sizeof(Unit)) &&
              section(hdr->off_counters, (int64_t)hdr->n_counters + 2, 4) && hdr->part_slots >= 0 &&
              hdr->part_slots <= ws_floats / kPartFloats && hdr->total_tokens >= 0;
  }
  if (!plan_ok) {
    if (tid == 0 && abort_s == 0) atomicExch(status, (int32_t)PUREKV_ERR_BAD_PLAN);
    hdr = nullptr;
  }
  const int2* entries = reinterpret_cast<const int2*>(plan + (plan_ok ? hdr->off_entries : 0));
  const uint32_t* masks = reinterpret_cast<const uint32_t*>(plan + (plan_ok ? hdr->off_masks : 0));
  const uint32_t* kept_halves = masks + (plan_ok ? hdr->n_mask_words - hdr->n_entries : 0);  // one word per entry
  const Unit* units = reinterpret_cast<const Unit*>(plan + (plan_ok ? hdr->off_units : 0));
  int32_t* counters = reinterpret_cast<int32_t*>(plan + (plan_ok ? hdr->off_counters : 0));
  const int32_t G = n_q_heads / n_kv_heads, ppg = (G + 1) >> 1;
  // Units are handed out at run time: CTA c starts with unit c of the list (sorted by decreasing cost) and draws
  // every further one from a counter behind the merge counters, so the CTAs finish within one small unit of one
  // another whatever the units really cost.  The producer draws and publishes; the other roles follow unit_s[].
  // With several layers the list is gone through once per layer, one after another: the CTAs pass from a layer's last (and
  // smallest) units to the next layer's first without meeting, so a launch's start and its uneven end are paid for once.
  const int32_t n_work = n_units * n_layers;  // (the launch code knows that it is no more than an int32 holds)
  int32_t* sched = counters + (plan_ok ? hdr->n_counters : 0);  // [0] units drawn beyond the first round, [1] CTAs that drew their last
  const int64_t n_entries = plan_ok ? hdr->n_entries : 0, n_mask_words = plan_ok ? hdr->n_mask_words - n_entries : 0;
  const int64_t total_tokens = plan_ok ? hdr->total_tokens : 0;
  const int32_t n_counters = plan_ok ? hdr->n_counters : 0;
  const int64_t part_slots = plan_ok ? hdr->part_slots : 0;
  const bool withhold_first_k = plan_ok && (hdr->test_flags & 1u) != 0u;
  const bool start_ok = abort_s == 0 && plan_ok;
  // Whether a unit's output leaves through shared memory: whole query tiles of whole lists.  The rows of a tile lie thousands of
  // bytes apart; stored from registers each warp store touches 32 lines, and a unit's output took 2250-3400 clk of its rows' time.
  // Through shared memory it is one copy per slot that the copy engine makes beside the next unit's first tile.  The room is the
  // stages of the unit's last tile, whose next contents are not wanted before the next unit's second tile: K's for slot 0
  // (both slots' S of that tile are long complete), V's for slot 1 (its last product is the unit's last).  Ragged batch of 8, sparse
  // layer: 618 -> 595 us at full clock, 725 -> 701 in a row; 37 120 tokens 653 -> 643 and 762 -> 749; the copies by rolled loops,
  // because of the instruction cache.  It is the faster way for launches of few units too (one sparse layer, 32 heads: 2432 tokens
  // 45.4 us from registers, 42.2 so; 384 units 29.8 and 28.1, 512 units 37.1 and 35.4, 64 and 256 units the same), so the shape of
  // the unit alone decides.  The roles read the answer in the unit's record, as a bit (384 units 27.8 -> 27.7, 512 35.2 -> 34.7).
  auto output_staged = [](const Unit& u) { return u.n_chunks == 1 && u.q_rows == kBQ && (u.q_rows1 == 0 || u.q_rows1 == kBQ); };

  // the two softmax warpgroups take registers from the warpgroup of the producer and MMA warps

  if (warp >= 8) {
    setmaxnreg_dec<kRegsOther>();
  if (start_ok && warp == kWarpProducer) {
    // ---------------- producer (whole warp; lane 0 issues) ----------------
    uint32_t it = 0;  // key tiles issued so far by this CTA, over all units
    int32_t issued_k = 0, issued_v = 0;
    bool ok = true;
    // unit idx of the list, or the end mark (ent_count 0) past its end
    // Also checks the unit: a unit whose fields point outside the plan's sections, the batch or the workspace is not
    // published; the CTA gives up with PUREKV_ERR_BAD_PLAN instead.
    auto fetch = [&](int32_t idx) -> Unit {
      Unit uu = {};
      if (idx < n_work) {
        const int32_t layer = idx < n_units ? 0 : idx / n_units;
        uu = units[idx - layer * n_units];
        uu.layer = layer;
        const int32_t n_pairs = n_kv_heads * ppg;
        const bool split = uu.n_chunks > 1, twin = uu.q_rows1 != 0;
        const int32_t group = uu.pair / ppg, in_group = 2 * (uu.pair - group * ppg);
        uu.heads = (group * G + in_group) * 4 + (output_staged(uu) ? 2 : 0) + (twin || in_group + 1 < G ? 1 : 0);
        const bool good = uu.ent_count >= 1 && uu.ent_begin >= 0 &&
                          (int64_t)uu.ent_begin + (int64_t)uu.ent_count * (twin ? 2 : 1) <= n_entries &&
                          uu.q_rows >= 1 && uu.q_rows <= kBQ && uu.req_start >= 0 && uu.q_start >= uu.req_start &&
                          (int64_t)uu.q_start + uu.q_rows <= total_tokens && uu.pair >= 0 && uu.pair < n_pairs &&
                          uu.n_chunks >= 1 && uu.n_chunks <= 255 && uu.chunk >= 0 && uu.chunk < uu.n_chunks &&
                          (!split || n_layers == 1) &&  // (the plan has merge counters and slots for one layer at a time)
                          (!twin || (uu.q_rows1 >= 1 && uu.q_rows1 <= kBQ && uu.q_start1 >= uu.req_start &&
                                     (int64_t)uu.q_start1 + uu.q_rows1 <= total_tokens && (G & 1) != 0 &&
                                     in_group == 2 * (ppg - 1) &&
                                     (!split || (uu.part_base1 >= 0 && ((int64_t)uu.part_base1 + uu.n_chunks) * n_q_heads <= part_slots &&
                                                 uu.counter_base1 >= 0 && (int64_t)uu.counter_base1 + n_q_heads <= n_counters)))) &&
                          (!split || (uu.part_base >= 0 && ((int64_t)uu.part_base + uu.n_chunks) * n_q_heads <= part_slots &&
                                      uu.counter_base >= 0 && (int64_t)uu.counter_base + n_q_heads <= n_counters));
        if (!good) {
          abort_code_s = (int)PUREKV_ERR_BAD_PLAN;
          *abort_flag = 1;
          uu = Unit{};
        }
      }
      return uu;
    };
    // lane 0: put a fetched unit into the ring as the CTA's unit number uo
    auto publish = [&](const Unit& uu, uint32_t uo) -> bool {
      if (*abort_flag) return false;
      const uint32_t us = uo % kUnitRing;
      if (uo >= (uint32_t)kUnitRing && !mbar_wait(smem_u32(&bars.u_empty[us]), ((uo / kUnitRing) - 1u) & 1u, abort_flag, wait_ns))
        return false;
      unit_s[us] = uu;
      mbar_arrive(smem_u32(&bars.u_full[us]));
      if (uu.ent_count == 0) {
        // This CTA has drawn for the last time.  The CTA that does so last of all rewinds both counters for the
        // plan's next launch (nobody reads them any more in this one).
        __threadfence();
        if (atomicAdd(sched + 1, 1) == (int32_t)gridDim.x - 1) {
          sched[0] = 0;
          sched[1] = 0;
        }
      }
      return true;
    };
    if (lane == 0) ok = publish(fetch((int32_t)blockIdx.x), 0u);
    for (uint32_t uo = 0;; ++uo) {
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      __syncwarp();
      const Unit u = unit_s[uo % kUnitRing];
      if (u.ent_count == 0) break;
      // The next unit is drawn as late as the latencies allow: when this unit's last tile goes out (the other roles
      // still have about two tiles of it to work through, which covers the counter's and the list's round trips).
      // Drawn at the start of a unit it would be reserved for as long as that unit runs, and the CTAs with the
      // longest units would keep work from those that finish early.
      int32_t idx_next = 0;
      const int32_t nt = u.ent_count;
      const int32_t g = u.pair / ppg, hq0 = u.heads >> 2;
      const bool twin = u.q_rows1 != 0;  // both slots on head hq0, slot 1 on the query tile at q_start1
      const int32_t n_slots = 1 + (u.heads & 1);
      // A tile's entry as slot 0 and as slot 1 see it, 32 tiles at a time, one per lane; of the halves an entry claims only
      // those that hold a kept pair are loaded and multiplied (with a skip granularity of 128 keys the entries claim both;
      // 64 frames of 24 x 24 under the paper's mask: 12 % fewer halves, 833 -> 780 us; a 64-key half costs 0.78 of a tile).
      int2 e_l, f_l;
      auto load_entries = [&](int32_t n) {
        e_l = f_l = make_int2(0, -1);
        if (n < nt) {
          const int32_t at = u.ent_begin + (twin ? 2 * n : n);
          e_l = __ldg(entries + at);
          if (twin) f_l = __ldg(entries + at + 1);
          const uint32_t he = __ldg(kept_halves + at), hf = twin ? __ldg(kept_halves + at + 1) : 0u;
          e_l.x &= (int32_t)(~12u | ((he & 3u) << 2));
          if (twin) f_l.x &= (int32_t)(~12u | ((hf & 3u) << 2));
          if (!twin) f_l = e_l;
          // The entry is checked before its mask offset or key-tile index is used for a copy: a class the slot knows (none only
          // in a twin unit, and then without halves), a bit mask inside the table.
          auto entry_ok = [&](const int2& x) {
            const int32_t c = x.x & 3;
            const uint32_t h = (uint32_t)(x.x >> 2) & 3u;
            if (x.x < 0 || (c == kTileNone ? (!twin || h != 0u) : h == 0u)) return false;
            return c != kTileGeneral || (x.y >= 0 && (int64_t)x.y + (int64_t)(kMaskBytes / 4) <= n_mask_words && (x.y & 3) == 0);
          };
          if (!entry_ok(e_l) || !entry_ok(f_l) || (e_l.x >> 4) != (f_l.x >> 4) || ((e_l.x | f_l.x) & 12) == 0 ||
              (int64_t)u.req_start + (int64_t)(e_l.x >> 4) * BK >= total_tokens) {
            abort_code_s = (int)PUREKV_ERR_BAD_PLAN;
            *abort_flag = 1;
            return false;
          }
        }
        return true;
      };
      if (lane == 0) {
        if (uo > 0) ok = mbar_wait(smem_u32(&bars.q_empty), (uo - 1u) & 1u, abort_flag, wait_ns);
        if (ok) {
          mbar_expect_tx(smem_u32(&bars.q_full), n_slots * kTileQ);
          for (int sl = 0; sl < n_slots; ++sl) {
            const int32_t hq = twin ? hq0 : hq0 + sl, qs = (twin && sl) ? u.q_start1 : u.q_start;
            tma_load_4d(sQ + sl * kTileQ, &tm_q, smem_u32(&bars.q_full), 0, hq, qs, u.layer);
            tma_load_4d(sQ + sl * kTileQ + kPanelQ, &tm_q, smem_u32(&bars.q_full), 64, hq, qs, u.layer);
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      for (int32_t n0 = 0; ok && n0 < nt; n0 += 32) {
        ok = __all_sync(0xffffffffu, load_entries(n0 + lane));
        const int32_t n1 = min(nt, n0 + 32);
        for (int32_t n = n0; ok && n < n1; ++n) {
          int2 e, f;
          e.x = __shfl_sync(0xffffffffu, e_l.x, n - n0);
          e.y = __shfl_sync(0xffffffffu, e_l.y, n - n0);
          f.x = __shfl_sync(0xffffffffu, f_l.x, n - n0);
          f.y = __shfl_sync(0xffffffffu, f_l.y, n - n0);
          if (lane == 0) {
            if (n == nt - 1) idx_next = atomicAdd(sched, 1) + (int32_t)gridDim.x;  // used after the loop
            const uint32_t s = it % ST, par = ((it / ST) - 1u) & 1u, ms = it % MR;
            const uint32_t hm = (uint32_t)((e.x | f.x) >> 2) & 3u;  // which 64-key halves of the tile are present
            // a whole tile, or one half: 64 rows into their place inside each panel
            const int32_t hh = hm == 2u ? 1 : 0, row = u.req_start + (e.x >> 4) * BK + 64 * hh;
            const uint32_t off = (uint32_t)hh * (kPanelKV / 2), bytes = hm == 3u ? kTileKV : kTileKV / 2;
            const CUtensorMap *map_k = hm == 3u ? &tm_k : &tm_k64, *map_v = hm == 3u ? &tm_v : &tm_v64;
            if (ok && it >= (uint32_t)ST) ok = mbar_wait(smem_u32(&bars.k_empty[s]), par, abort_flag, wait_ns);
            if (ok) {
              // a slot's bit mask goes to its own buffer; outside twin units both slots read the first one
              const uint32_t m_off = (sM - smem_u32(smem_raw)) + ms * 2u * kMaskBytes;
              const bool mask0 = (e.x & 3) == kTileGeneral, mask1 = twin && (f.x & 3) == kTileGeneral;
              meta_s[ms][0] = make_int2(e.x, (int32_t)(m_off + hm));
              meta_s[ms][1] = make_int2(f.x, (int32_t)(m_off + hm + (twin ? kMaskBytes : 0u)));
              if (mask0 || mask1) {
                mbar_expect_tx(smem_u32(&bars.m_full[ms]), (mask0 && mask1) ? 2u * kMaskBytes : kMaskBytes);
                if (mask0) bulk_load(sM + ms * 2u * kMaskBytes, masks + e.y, kMaskBytes, smem_u32(&bars.m_full[ms]));
                if (mask1)
                  bulk_load(sM + ms * 2u * kMaskBytes + kMaskBytes, masks + f.y, kMaskBytes, smem_u32(&bars.m_full[ms]));
              } else {
                mbar_arrive(smem_u32(&bars.m_full[ms]));
              }
              // (test plans withhold the first tile's K: whoever waits for it runs into the limit)
              if (!(withhold_first_k && it == 0u)) {
                mbar_expect_tx(smem_u32(&bars.k_full[s]), bytes);
                tma_load_4d(sK + s * kTileKV + off, map_k, smem_u32(&bars.k_full[s]), 0, g, row, u.layer);
                tma_load_4d(sK + s * kTileKV + kPanelKV + off, map_k, smem_u32(&bars.k_full[s]), 64, g, row, u.layer);
              }
              if (!(withhold_first_k && it == 0u)) issued_k = (int32_t)it + 1;
              if (it >= (uint32_t)ST) ok = mbar_wait(smem_u32(&bars.v_empty[s]), par, abort_flag, wait_ns);
            }
            if (ok) {
              mbar_expect_tx(smem_u32(&bars.v_full[s]), bytes);
              tma_load_4d(sV + s * kTileKV + off, map_v, smem_u32(&bars.v_full[s]), 0, g, row, u.layer);
              tma_load_4d(sV + s * kTileKV + kPanelKV + off, map_v, smem_u32(&bars.v_full[s]), 64, g, row, u.layer);
              issued_v = (int32_t)it + 1;
            }
          }
          ++it;
          ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        }
      }
      if (lane == 0 && ok) ok = publish(fetch(idx_next), uo + 1u);
    }
    if (lane == 0 && *abort_flag) {
      // drain: every issued copy must have landed before shared memory is released
      const uint64_t t0 = global_ns();
      for (int32_t n = max(0, issued_k - ST); n < issued_k; ++n)
        while (!mbar_try_wait(smem_u32(&bars.k_full[n % ST]), (n / ST) & 1) && global_ns() - t0 < wait_ns) {}
      for (int32_t n = max(0, issued_v - ST); n < issued_v; ++n)
        while (!mbar_try_wait(smem_u32(&bars.v_full[n % ST]), (n / ST) & 1) && global_ns() - t0 < wait_ns) {}
      for (int32_t n = max(0, issued_k - MR); n < issued_k; ++n)
        while (!mbar_try_wait(smem_u32(&bars.m_full[n % MR]), (n / MR) & 1) && global_ns() - t0 < wait_ns) {}
      __nanosleep(20000);  // a Q tile possibly still in flight (its barrier's phase is not known here)
    }
  } else if (start_ok && warp == kWarpMma) {
    // ---------------- MMA issuer ----------------
    // elect.sync tells the compiler that one thread runs this (a comparison with the lane number does not), so that
    // descriptors live in uniform registers: 8320 tokens, dense causal 477 -> 448 us
    if (elect_one()) {
      constexpr uint32_t idesc_qk = instr_desc(BK, false);
      constexpr uint32_t idesc_qk_half = instr_desc(BK / 2, false);
      constexpr uint32_t idesc_pv = instr_desc(kD, true);
      static_assert(BK == 128 && ST == 2, "S of a tile is issued behind P V of the tile before, which frees its columns");
      uint32_t it = 0;   // the CTA's key tiles so far, which are slot 0's
      uint32_t tp1 = 0;  // slot 1's
      // Descriptor words.  High word: stride between 8-row groups 1024 B, descriptor version 1, 128-byte swizzle.
      // Low word: start address / 16 and the leading-dimension offset / 16 (used by the MN-major V operand only).
      constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
      const uint32_t q_lo0 = ((sQ & 0x3FFFFu) >> 4) | (1u << 16);
      const uint32_t k_lo0 = ((sK & 0x3FFFFu) >> 4) | (1u << 16);
      const uint32_t v_lo0 = ((sV & 0x3FFFFu) >> 4) | ((kPanelKV >> 4) << 16);
      auto halves_of = [&](uint32_t i) {  // written before the stage's barrier was armed
        return (uint32_t)meta_s[i % MR][0].y & 3u;
      };
      // One body of code for first and later tiles, whole tiles and halves.  What the roles run in a tile's time goes through
      // the SM's instruction cache; what misses there comes from the cache that an SM shares with its neighbours, which was 78 %
      // busy with it (ragged batch of 8: 3.3 M lines a launch, now 2.7 M, and 625 -> 613 us at full clock; dense causal 12.0 M,
      // now 7.5 M, time unchanged: products by a rolled loop as well leave 2.8 M there and are 4 % slower).
      bool ok = true;
      for (uint32_t uo = 0; ok; ++uo) {
        const uint32_t us = uo % kUnitRing;
        ok = mbar_wait(smem_u32(&bars.u_full[us]), (uo / kUnitRing) & 1u, abort_flag, wait_ns);
        if (!ok) break;
        const int32_t nt = unit_s[us].ent_count;
        const uint32_t last_slot = (uint32_t)unit_s[us].heads & 1u;
        const bool staged = (unit_s[us].heads & 2) != 0;
        mbar_arrive(smem_u32(&bars.u_empty[us]));
        if (nt == 0) break;
        ok = mbar_wait(smem_u32(&bars.q_full), uo & 1u, abort_flag, wait_ns);
        // Step n: P V of tile n and S of tile n + 1, slot 0 before slot 1; step -1 is the first S alone.
        uint32_t hm = 0u;
#pragma unroll 1
        for (int32_t n = -1; ok && n < nt; ++n) {
          const bool pv = n >= 0, qk = n + 1 < nt;
          const uint32_t s = it % ST, sn = (pv ? it + 1u : it) % ST;  // stages of tile n, and of tile n + 1
          uint32_t hn = 3u;
          if (pv) ok = mbar_wait(smem_u32(&bars.v_full[s]), (it / ST) & 1u, abort_flag, wait_ns);
          if (ok && qk) {
            ok = mbar_wait(smem_u32(&bars.k_full[sn]), ((pv ? it + 1u : it) / ST) & 1u, abort_flag, wait_ns);
            hn = halves_of(pv ? it + 1u : it);
          }
#pragma unroll
          for (uint32_t sl = 0; sl < 2u; ++sl) {
            if (sl > last_slot) break;
            const uint32_t p_addr = tmem + sl * 128u;
            if (pv) {
              // O(slot) += P V, when P has come: the K steps of the first 96 keys as soon as those have, the others behind.  P of the
              // unit's first tile also implies that the previous unit's output has left TMEM.
              // B = V tile, MN-major: per K step 16 key rows (2 groups of 8, 1024 B apart) x 128 dims (2 panels)
              const uint32_t par = (sl == 0u ? it : tp1) & 1u, v_lo = v_lo0 + s * (kTileKV >> 4);
              bool part, full;
              mbar_test2(smem_u32(&bars.p_part[sl]), par, smem_u32(&bars.p_full[sl]), par, &part, &full);
              if (hm != 3u) part = full;
              if (!part) ok = mbar_wait(smem_u32(hm == 3u ? &bars.p_part[sl] : &bars.p_full[sl]), par, abort_flag, wait_ns);
              if (!ok) break;
              tc_fence_after();
              const uint32_t acc = n > 0 ? 1u : 0u;  // the unit's first product overwrites O
              if (hm == 3u) {
#pragma unroll
                for (int ks = 0; ks < 6; ++ks)
                  mma_ts_lh(p_addr + kColO, p_addr + ks * 8, v_lo + ks * (2048 >> 4), kDescHi, idesc_pv, ks > 0 ? 1u : acc);
                if (!full) {
                  ok = mbar_wait(smem_u32(&bars.p_full[sl]), par, abort_flag, wait_ns);
                  if (!ok) break;
                  tc_fence_after();
                }
#pragma unroll
                for (int ks = 6; ks < 8; ++ks)
                  mma_ts_lh(p_addr + kColO, p_addr + ks * 8, v_lo + ks * (2048 >> 4), kDescHi, idesc_pv, 1u);
              } else {  // the K steps of the present half only
                const uint32_t k0 = (hm >> 1) * (BK / 32);
#pragma unroll
                for (int ks = 0; ks < BK / 32; ++ks)
                  mma_ts_lh(p_addr + kColO, p_addr + (k0 + ks) * 8, v_lo + (k0 + ks) * (2048 >> 4), kDescHi, idesc_pv, ks > 0 ? 1u : acc);
              }
            } else {
              tc_fence_after();
            }
            if (qk) {
              // S = Q K^T of tile n + 1; of one 64-key half with N = 64, into that half's columns of S
              const uint32_t hh = hn == 2u ? 1u : 0u, q_lo = q_lo0 + sl * (kTileQ >> 4);
              const uint32_t k_lo = k_lo0 + sn * (kTileKV >> 4) + hh * (kPanelKV >> 5);
              const uint32_t d_addr = p_addr + hh * 64u, idesc = hn == 3u ? idesc_qk : idesc_qk_half;
#pragma unroll
              for (int ks = 0; ks < kD / 16; ++ks)
                mma_ss_lh(d_addr, q_lo + (ks >> 2) * (kPanelQ >> 4) + (ks & 3) * 2, kDescHi,
                          k_lo + (ks >> 2) * (kPanelKV >> 4) + (ks & 3) * 2, kDescHi, idesc, ks > 0 ? 1u : 0u);
            }
            // announced to the slot's rows first (they are waiting for it), the releases of the stages follow behind
            tc_commit(smem_u32(qk ? &bars.s_full[sl] : &bars.o_final[sl]));
          }
          if (!ok) break;
          // (the last tile's stages: the output goes through them, see output_staged)
          if (pv && (qk || !staged || last_slot == 0u)) tc_commit(smem_u32(&bars.v_empty[s]));
          if (qk && (n + 2 < nt || !staged)) tc_commit(smem_u32(&bars.k_empty[sn]));
          if (n + 2 == nt) tc_commit(smem_u32(&bars.q_empty));  // the unit's last read of Q
          if (pv) {
            ++it;
            tp1 += last_slot;
          }
          hm = hn;
        }
      }
      if (!ok) {
        // leaving early: let every issued MMA finish before TMEM is released
        tc_commit(smem_u32(&bars.drain));
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(smem_u32(&bars.drain), 0) && global_ns() - t0 < wait_ns) {}
      }
    }
  } else if (start_ok && warp == kWarpStore) {
    // ---------------- output: staged tiles to global memory ----------------
    if (lane == 0) {
      uint32_t it = 0, phases = 0u;  // key tiles so far; bit sl * ST + s: the parity of the next phase of o_staged[sl][s]
      bool ok = true;
      for (uint32_t uo = 0; ok; ++uo) {
        const uint32_t us = uo % kUnitRing;
        ok = mbar_wait(smem_u32(&bars.u_full[us]), (uo / kUnitRing) & 1u, abort_flag, wait_ns);
        if (!ok) break;
        const Unit& u = unit_s[us];
        const int32_t nt = u.ent_count;
        if (nt == 0) break;
        it += (uint32_t)nt;
        if ((u.heads & 2) != 0) {
          const uint32_t s = (it - 1u) % ST;
          const bool twin = u.q_rows1 != 0;
#pragma unroll
          for (int sl = 0; sl < 2; ++sl) {
            if (sl > (u.heads & 1)) break;
            const uint32_t bit = (uint32_t)sl * ST + s;
            ok = mbar_wait(smem_u32(&bars.o_staged[sl][s]), (phases >> bit) & 1u, abort_flag, wait_ns);
            if (!ok) break;
            phases ^= 1u << bit;
            const uint32_t buf = (sl == 0 ? sK : sV) + s * kTileKV;
            const int32_t hq = (u.heads >> 2) + (twin ? 0 : sl), q_first = twin && sl == 1 ? u.q_start1 : u.q_start;
            tma_store_4d(&tm_o, buf, 0, hq, q_first, u.layer);
            tma_store_4d(&tm_o, buf + kPanelKV, 64, hq, q_first, u.layer);
            asm volatile("cp.async.bulk.commit_group;\n cp.async.bulk.wait_group.read 0;" ::: "memory");
            mbar_arrive(smem_u32(sl == 0 ? &bars.k_empty[s] : &bars.v_empty[s]));  // in the MMA thread's place
          }
        }
        if (ok) mbar_arrive(smem_u32(&bars.u_empty[us]));
      }
      asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
  }
  } else {
    setmaxnreg_inc<kRegsSoftmax>();
  if (start_ok) {
    // ---------------- softmax / epilogue: one thread per query row of one slot ----------------
    const int sl = warp >> 2;
    const int quad = warp & 3;  // TMEM lane quadrant this warp may access
    const int row = quad * 32 + lane;
    const uint32_t t_lane = tmem + ((uint32_t)(quad * 32) << 16);
    // waits are made warp-uniform: the TMEM loads/stores below need the whole warp
    auto wait_w = [&](uint32_t bar, uint32_t parity) -> bool {
      return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, wait_ns) ? 1 : 0) != 0;
    };
    uint32_t it = 0;          // key tiles of the CTA so far (both slots)
    uint32_t t = 0;           // tiles this slot has processed, over all units
    uint32_t slot_units = 0;  // units this slot took part in
    bool ok = true;
    for (uint32_t uo = 0; ok; ++uo) {
      const uint32_t us = uo % kUnitRing;
      if (!wait_w(smem_u32(&bars.u_full[us]), (uo / kUnitRing) & 1u)) { ok = false; break; }
      // read in place (the fields wanted after the tile loop are not held in registers meanwhile); the ring slot is
      // given back at the end of the unit
      const Unit& u = unit_s[us];
      auto release_unit = [&]() {
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars.u_empty[us]));
      };
      const int32_t nt = u.ent_count;
      if (nt == 0) break;
      if (sl > (u.heads & 1)) {
        // A single-head unit: this slot sits it out.  It takes no part in the tile ring meanwhile: a parity wait only
        // tells a barrier's current phase from the one before, and a slot with nothing to deliver is held back by
        // nobody, so it could fall (or run) a whole ring away from the producer.  The unit ring is a full handshake
        // instead, and the next unit is published only after every tile of this one has been issued, which puts the
        // slot's next tile within the ring's reach again.
        it += (uint32_t)nt;
        release_unit();
        continue;
      }
      const int32_t i_rel = (u.q_rows1 != 0 && sl == 1 ? u.q_start1 : u.q_start) - u.req_start + row;
      float m_ref = 0.f, l_sum = 0.f;
      for (const uint32_t it_end = it + (uint32_t)nt; it != it_end; ++it) {
        if (!wait_w(smem_u32(&bars.m_full[it % MR]), (it / MR) & 1u)) { ok = false; break; }
        const int2 e = meta_s[it % MR][sl];
        const int32_t cls = e.x & 3, j0 = (e.x >> 4) * BK;
        // hm: the 64-key halves that were loaded and multiplied (chunk c belongs to half c / 2); hm_own: those in which
        // this slot's query tile keeps anything (they differ in twin units only)
        const uint32_t hm_own = (uint32_t)(e.x >> 2) & 3u, hm = (uint32_t)e.y & 3u;
        uint32_t keep[BK / 32];
        if (cls == kTileGeneral) {  // this row's bits of the tile's mask
          const uint32_t* mrow = reinterpret_cast<const uint32_t*>(smem_raw + (e.y & ~3)) + row * (BK / 32);
          static_assert(BK == 128, "a mask row is four 32-bit words");
          const uint4 w4 = *reinterpret_cast<const uint4*>(mrow);
          keep[0] = w4.x; keep[1] = w4.y; keep[2] = w4.z; keep[3] = w4.w;
        } else if (cls == kTileDiag) {
          const int32_t n_ok = min(BK, max(0, i_rel - j0 + 1));  // causal: columns 0 .. n_ok-1
#pragma unroll
          for (int c = 0; c < BK / 32; ++c) {
            const int32_t k_in = min(32, max(0, n_ok - 32 * c));
            keep[c] = k_in >= 32 ? 0xFFFFFFFFu : ((1u << k_in) - 1u);
          }
        } else {
#pragma unroll
          for (int c = 0; c < BK / 32; ++c) keep[c] = 0xFFFFFFFFu;
        }
        if (hm_own != 3u) {  // columns of a half the slot keeps nothing of (or that is absent altogether): masked
#pragma unroll
          for (int c = 0; c < BK / 32; ++c)
            if (!((hm_own >> (c >> 1)) & 1u)) keep[c] = 0u;
        }
        // The 32-key chunks of which some row of the warp keeps a key.  Not asked of causal tiles, where warps 2 and 3 need three and
        // four of them and the products wait for all four warps: with warps 0 and 1 on the other way below, one layer of 6 x 600
        // tokens (28 heads) 33.3 us, without 31.9; 8 x 460 (32 heads) 34.9 and 33.9; long lists the same.
        uint32_t some = 15u;
        if (cls >= kTileGeneral) {
          some = 0u;
#pragma unroll
          for (int c = 0; c < BK / 32; ++c) some |= keep[c] != 0u ? 1u << c : 0u;
          some = __reduce_or_sync(0xffffffffu, some);
        }
        if (!wait_w(smem_u32(&bars.s_full[sl]), t & 1u)) { ok = false; break; }
        tc_fence_after();
        const uint32_t s_addr = t_lane + sl * 128;
        // Fast path: exponentials against the row's standing reference m_ref, no maximum taken.  Softmax does not depend
        // on the reference, and fp32 / bf16 carry 8 exponent bits, so the reference (0 at the start of a unit) only has
        // to keep exp2 in range: it moves when a tile overflows, or when everything kept so far has underflowed; those
        // tiles take the exact path below.  P goes to the tensor cores in two parts, 96 keys and 32: six of the eight K steps
        // of P V run during the last quarter's exponentials instead of behind them (8320 tokens: dense causal 421 -> 406 us,
        // paper mask 122 -> 116 us; handing over half of P instead was measured slower, the wait between the parts then
        // holds the MMA thread up for the other slot).
        uint32_t pk[BK / 2];
        float l_tile = 0.f;
        auto p_stored = [&]() {  // the warp's P is in TMEM; lane 0 may say so, one arrival per warp: 4 per slot
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
        };
        const uint32_t part_bar = smem_u32(&bars.p_part[sl]), full_bar = smem_u32(&bars.p_full[sl]);
        bool exact = false;
        {
          float2 ls2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
          const float2 sc2 = make_float2(scale_log2, scale_log2), mm2 = make_float2(-m_ref, -m_ref);
          // Masked columns are set to -inf first, all of them, so that the exponentials behind are one straight run of
          // code: with a branch per 32 columns the MUFU unit drained four times per tile (1650 clk for the exponentials of a
          // tile against 1200 for the same code alone; 8320 tokens, dense causal 448 -> 420 us, paper mask 126 -> 123 us).
          auto mask64 = [&](uint32_t (&r)[64], uint32_t k0, uint32_t k1) {
            if (__any_sync(0xffffffffu, (k0 & k1) != 0xFFFFFFFFu)) {  // warp-uniform
#pragma unroll
              for (int x = 0; x < 32; ++x) {
                if (!((k0 >> x) & 1u)) r[x] = 0xFF800000u;  // -inf: exp2 gives 0
                if (!((k1 >> x) & 1u)) r[32 + x] = 0xFF800000u;
              }
            }
          };
          auto exps = [&](const uint32_t (&r)[64], auto x0_c, auto x1_c, auto off_c) {  // columns x0 .. x1 - 1 -> pk[off ..]
            constexpr int x0 = decltype(x0_c)::value, x1 = decltype(x1_c)::value, off = decltype(off_c)::value;
#pragma unroll
            for (int x = x0; x < x1; x += 2) {
              const float2 a = __ffma2_rn(make_float2(__uint_as_float(r[x]), __uint_as_float(r[x + 1])), sc2, mm2);
              const float2 pp = make_float2(ex2(a.x), ex2(a.y));
              ls2[(x >> 1) & 1] = __fadd2_rn(ls2[(x >> 1) & 1], pp);
              pk[off + ((x - x0) >> 1)] = pack_bf16(pp.x, pp.y);
            }
          };
          constexpr std::integral_constant<int, 0> i0{};
          constexpr std::integral_constant<int, 32> i32{};
          constexpr std::integral_constant<int, 16> i16{};
          constexpr std::integral_constant<int, 48> i48{};
          constexpr std::integral_constant<int, 64> i64{};
          bool has_kept = cls == kTileFull;  // (a full tile has both halves)
#pragma unroll
          for (int c = 0; c < BK / 32; ++c) has_kept |= keep[c] != 0u;
          // overflow (inf or NaN), or kept keys and still nothing representable: redo against the true maximum.  Settled
          // before P of the first 96 keys goes out, from its sum and the largest logit of the last 32 keys (32 terms below
          // 2^94 stay below 1e30; one of 2^-96 or more is representable).
          auto bad = [&](float top) {
            return __any_sync(0xffffffffu, !(l_tile <= 1.0e30f) || !(top < 94.f) ||
                                               (has_kept && l_sum + l_tile < 1.0e-30f && top < -96.f));
          };
          if (__popc(some) > 2) {  // all loads in flight before the one wait
            uint32_t r0[64], r1[64];
            tmem_ld32_at<0>(s_addr, r0);
            tmem_ld32_at<32>(s_addr + 32, r0);
            tmem_ld32_at<0>(s_addr + 64, r1);
            tmem_ld32_at<32>(s_addr + 96, r1);
            tc_wait_ld();
            if (cls != kTileFull) {
              mask64(r0, keep[0], keep[1]);
              mask64(r1, keep[2], keep[3]);
            }
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int x = 32; x < 64; x += 2) mx[(x >> 1) & 3] = max3(mx[(x >> 1) & 3], __uint_as_float(r1[x]), __uint_as_float(r1[x + 1]));
            exps(r0, i0, i64, i0);
            exps(r1, i0, i32, i32);
            l_tile = (ls2[0].x + ls2[0].y) + (ls2[1].x + ls2[1].y);
            exact = bad(fmaf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])), scale_log2, -m_ref));  // scale > 0
            if (!exact) {
              tmem_st32(s_addr, reinterpret_cast<const uint32_t(&)[32]>(pk[0]));  // over columns of S that have been read
              tmem_st16(s_addr + 32, reinterpret_cast<const uint32_t(&)[16]>(pk[32]));
              p_stored();
              if (lane == 0) mbar_arrive(part_bar);
              exps(r1, i32, i64, i48);
              l_tile = (ls2[0].x + ls2[0].y) + (ls2[1].x + ls2[1].y);
              tmem_st16(s_addr + 48, reinterpret_cast<const uint32_t(&)[16]>(pk[48]));
            }
          } else {
            // The warp's rows keep keys of two 32-key chunks at most: those are read and exponentiated, one after another, and the
            // others' P is zero.  (The cell of the previous frame is a diagonal, one chunk per warp of a tile that costs four;
            // 8320 tokens x 28 layers 4070 -> 3890 us, 37 120 tokens one layer 785 -> 766, ragged batch of 8 751 -> 739.  With three
            // chunks, or with the loads of both in flight at once, which spills, the straight run above is faster.)
            const int ca = __ffs((int)some) - 1, cb = 31 - __clz((int)some);  // (-1: none, for a slot that sits a twin unit's tile out)
            auto pick = [&](int c) { return c == 0 ? keep[0] : c == 1 ? keep[1] : c == 2 ? keep[2] : keep[3]; };
            auto chunk = [&](int c, auto off_c) {
              constexpr int off = decltype(off_c)::value;
              uint32_t r[32];
              tmem_ld32(s_addr + 32 * c, r);
              tc_wait_ld();
              const uint32_t k = pick(c);
#pragma unroll
              for (int x = 0; x < 32; ++x)
                if (!((k >> x) & 1u)) r[x] = 0xFF800000u;
#pragma unroll
              for (int x = 0; x < 32; x += 2) {
                const float2 a = __ffma2_rn(make_float2(__uint_as_float(r[x]), __uint_as_float(r[x + 1])), sc2, mm2);
                const float2 pp = make_float2(ex2(a.x), ex2(a.y));
                ls2[(x >> 1) & 1] = __fadd2_rn(ls2[(x >> 1) & 1], pp);
                pk[off + (x >> 1)] = pack_bf16(pp.x, pp.y);
              }
            };
            if (ca >= 0) chunk(ca, i0);
            if (ca != cb) chunk(cb, i16);
            l_tile = (ls2[0].x + ls2[0].y) + (ls2[1].x + ls2[1].y);
            exact = bad(-INFINITY);
            if (!exact) {
              const uint32_t zeros[16] = {};
#pragma unroll
              for (int c = 0; c < BK / 32; ++c)
                if (((hm >> (c >> 1)) & 1u) && !((some >> c) & 1u)) tmem_st16(s_addr + 16 * c, zeros);
              if (ca >= 0) tmem_st16(s_addr + 16 * ca, reinterpret_cast<const uint32_t(&)[16]>(pk[0]));
              if (ca != cb) tmem_st16(s_addr + 16 * cb, reinterpret_cast<const uint32_t(&)[16]>(pk[16]));
            }
          }
        }
        if (exact) {
          // Exact path (rare): re-reference the row; O and the running sum are rescaled.  S is still intact in TMEM
          // (P has not been stored yet).
          float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int c = 0; c < BK / 32; ++c) {
            uint32_t r[32];
            tmem_ld32(s_addr + 32 * c, r);
            tc_wait_ld();
#pragma unroll
            for (int x = 0; x < 32; ++x)
              if ((keep[c] >> x) & 1u) mx[x & 3] = fmaxf(mx[x & 3], __uint_as_float(r[x]));
          }
          const float m_tile = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale_log2;  // scale > 0
          // the new reference: the larger of this tile's maximum and the log-sum of what has been accumulated
          const float m_eff = l_sum > 0.f ? m_ref + log2f(l_sum) : -INFINITY;
          const float m_max = fmaxf(m_eff, m_tile);
          const float m_new = m_max == -INFINITY ? m_ref : m_max;  // nothing kept yet and nothing accumulated: stay
          const float alpha = l_sum > 0.f ? ex2(m_ref - m_new) : 1.f;  // with l_sum == 0 every earlier P was 0, so O is 0
          const float m_sub = m_new;
          if (__any_sync(0xffffffffu, alpha != 1.f)) {  // (not in a unit's first tile: alpha is 1 there)
            // O is quiescent: S of a tile is issued behind P V of the one before, and it is complete.
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < kD / 32; ++c) {
              uint32_t tt[32];
              tmem_ld32(t_lane + kColO + sl * 128 + 32 * c, tt);
              tc_wait_ld();
#pragma unroll
              for (int x = 0; x < 32; ++x) tt[x] = __float_as_uint(__uint_as_float(tt[x]) * alpha);
              tmem_st32(t_lane + kColO + sl * 128 + 32 * c, tt);
            }
          }
          float ls[2] = {0.f, 0.f};
#pragma unroll
          for (int c = 0; c < BK / 32; ++c) {
            uint32_t r[32], pc[16];
            tmem_ld32(s_addr + 32 * c, r);
            tc_wait_ld();
#pragma unroll
            for (int x = 0; x < 32; x += 2) {
              const float p0 = ((keep[c] >> x) & 1u) ? ex2(fmaf(__uint_as_float(r[x]), scale_log2, -m_sub)) : 0.f;
              const float p1 = ((keep[c] >> (x + 1)) & 1u) ? ex2(fmaf(__uint_as_float(r[x + 1]), scale_log2, -m_sub)) : 0.f;
              ls[(x >> 1) & 1] += p0 + p1;
              pc[x >> 1] = pack_bf16(p0, p1);
            }
            // (over columns of S that have been read: chunk c of P lies inside chunk c / 2 of S)
            if ((hm >> (c >> 1)) & 1u) tmem_st16(s_addr + 16 * c, pc);
          }
          l_tile = ls[0] + ls[1];
          l_sum *= alpha;
          m_ref = m_new;
        }
        l_sum += l_tile;
        p_stored();
        if (lane == 0) {
          // Every tile counts on both barriers, and on p_part first: the MMA thread waits for p_full in every tile but for p_part
          // only where both halves are present, so p_full has to imply p_part.  (The other way round a late arrival could leave
          // p_part a phase behind, and the parity of the next tile's wait would match the phase before it.)
          if (exact || __popc(some) <= 2) mbar_arrive(part_bar);
          mbar_arrive(full_bar);
        }
        ++t;
      }
      if (!ok) break;
      // (one completion per unit, behind the slot's last P V)
      if (!wait_w(smem_u32(&bars.o_final[sl]), slot_units & 1u)) { ok = false; break; }
      ++slot_units;
      tc_fence_after();
      // (the unit's fields are read again rather than held through the tile loop: the softmax uses every register it has)
      const bool twin = u.q_rows1 != 0, second = twin && sl == 1;  // this slot works on the unit's second query tile
      const int32_t hq = (u.heads >> 2) + (twin ? 0 : sl), q_first = second ? u.q_start1 : u.q_start;
      const bool row_valid = row < (second ? u.q_rows1 : u.q_rows);
      if ((u.heads & 2) != 0) {
        const float inv = 1.f / l_sum;
        const uint32_t buf = (sl == 0 ? sK : sV) + ((it - 1u) % ST) * kTileKV + (uint32_t)row * 128u;
#pragma unroll 1
        for (int c = 0; c < kD / 32; ++c) {
          uint32_t tt[32];
          tmem_ld32(t_lane + kColO + sl * 128 + 32 * c, tt);
          tc_wait_ld();
#pragma unroll
          for (int y = 0; y < 4; ++y) {  // 16 bytes each, placed as the 128-byte swizzle has them
            uint32_t w[4];
#pragma unroll
            for (int z = 0; z < 4; ++z)
              w[z] = pack_bf16(__uint_as_float(tt[8 * y + 2 * z]) * inv, __uint_as_float(tt[8 * y + 2 * z + 1]) * inv);
            st_shared_v4(buf + (uint32_t)(c >> 1) * kPanelKV + ((uint32_t)((4 * (c & 1) + y) ^ (row & 7)) << 4), w);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the copy out reads what these stores wrote
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars.o_staged[sl][(it - 1u) % ST]));
        if (lse) lse[u.layer * lse_stride + (int64_t)hq * hdr->total_tokens + q_first + row] = (m_ref + log2f(l_sum)) * 0.6931471805599453f;
      } else if (u.n_chunks == 1) {
        const float inv = 1.f / l_sum;
        __nv_bfloat16* dst = o + u.layer * o_stride + ((int64_t)(q_first + row) * n_q_heads + hq) * kD;
#pragma unroll 1
        for (int c = 0; c < kD / 32; ++c) {
          uint32_t tt[32];
          tmem_ld32(t_lane + kColO + sl * 128 + 32 * c, tt);
          tc_wait_ld();
          if (row_valid) {
#pragma unroll
            for (int x = 0; x < 32; x += 16) {
              uint32_t w[8];
#pragma unroll
              for (int y = 0; y < 8; ++y)
                w[y] = pack_bf16(__uint_as_float(tt[x + 2 * y]) * inv, __uint_as_float(tt[x + 2 * y + 1]) * inv);
              st_global_v8(dst + 32 * c + x, w);
            }
          }
        }
        if (lse && row_valid)
          lse[u.layer * lse_stride + (int64_t)hq * hdr->total_tokens + q_first + row] = (m_ref + log2f(l_sum)) * 0.6931471805599453f;
      } else {
        // one chunk of a split list: leave the unnormalised result for whoever arrives last
        const int32_t part_base = second ? u.part_base1 : u.part_base;
        float* part = ws + ((int64_t)(part_base + u.chunk) * n_q_heads + hq) * kPartFloats;
#pragma unroll
        for (int c = 0; c < kD / 32; ++c) {
          uint32_t tt[32];
          tmem_ld32(t_lane + kColO + sl * 128 + 32 * c, tt);
          tc_wait_ld();
#pragma unroll
          for (int x = 0; x < 32; x += 4)
            *reinterpret_cast<uint4*>(part + ((c * 8 + (x >> 2)) * 128 + row) * 4) =
                make_uint4(tt[x], tt[x + 1], tt[x + 2], tt[x + 3]);
        }
        part[128 * 128 + row] = m_ref;
        part[128 * 128 + 128 + row] = l_sum;
        // A row's partial results are read by the thread of the same row in another CTA, so each warp publishes and counts for
        // itself: a byte of the head's counter per warp (one release / acquire update at GPU scope by lane 0; release is
        // cumulative over what __syncwarp ordered before it, so no thread needs a fence of its own).  Whichever warp finds all
        // chunks of its 32 rows there merges them.
        __syncwarp();
        int32_t last = 0;
        if (lane == 0) {
          int32_t* cnt = counters + (second ? u.counter_base1 : u.counter_base) + hq;
          last = ((atom_add_acq_rel(cnt, 1 << (8 * quad)) >> (8 * quad)) & 255) == u.n_chunks - 1;
          if (last) atomicSub(reinterpret_cast<uint32_t*>(cnt), (uint32_t)u.n_chunks << (8 * quad));  // ready for the next launch
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        __syncwarp();
        if (last) {
          const float* p0 = ws + ((int64_t)part_base * n_q_heads + hq) * kPartFloats;
          const int64_t cstride = (int64_t)n_q_heads * kPartFloats;
          const int32_t own = u.chunk, n_ch = u.n_chunks;
          // The merge is a chain of L2 round trips: row statistics four chunks at a time, then 32 columns of two chunks at a
          // time, the CTA's own chunk from TMEM; always summed in chunk order.  (2432 tokens, lists in three chunks, one layer:
          // two chunks at a time and the slot's warps together 45.6 us, this way 44.0.)
          float m_all = -INFINITY, l_all = 0.f;
          for (int32_t c0 = 0; c0 < n_ch; c0 += 4) {
            float mc[4], lc[4];
#pragma unroll
            for (int y = 0; y < 4; ++y) {
              const float* pc = p0 + (int64_t)min(c0 + y, n_ch - 1) * cstride + 128 * 128 + row;
              mc[y] = __ldcg(pc);
              lc[y] = __ldcg(pc + 128);
            }
#pragma unroll
            for (int y = 0; y < 4; ++y) {
              if (c0 + y < n_ch && lc[y] > 0.f) {
                if (mc[y] > m_all) {
                  l_all *= ex2(m_all - mc[y]);  // (l_all is 0 while m_all is -inf)
                  m_all = mc[y];
                }
                l_all += lc[y] * ex2(mc[y] - m_all);
              }
            }
          }
          const float inv = 1.f / l_all, w_own = l_sum > 0.f ? ex2(m_ref - m_all) : 0.f;
          __nv_bfloat16* dst = o + ((int64_t)(q_first + row) * n_q_heads + hq) * kD;
#pragma unroll 1
          for (int cc = 0; cc < kD / 32; ++cc) {
            uint32_t tt[32];
            tmem_ld32(t_lane + kColO + sl * 128 + 32 * cc, tt);
            float acc[32];
#pragma unroll
            for (int x = 0; x < 32; ++x) acc[x] = 0.f;
            bool own_in = false;
            auto add = [&](float w, const float4 (&v)[8]) {
#pragma unroll
              for (int x = 0; x < 8; ++x) {
                acc[4 * x] = fmaf(w, v[x].x, acc[4 * x]);
                acc[4 * x + 1] = fmaf(w, v[x].y, acc[4 * x + 1]);
                acc[4 * x + 2] = fmaf(w, v[x].z, acc[4 * x + 2]);
                acc[4 * x + 3] = fmaf(w, v[x].w, acc[4 * x + 3]);
              }
            };
            auto add_own = [&]() {
#pragma unroll
              for (int x = 0; x < 32; ++x) acc[x] = fmaf(w_own, __uint_as_float(tt[x]), acc[x]);
              own_in = true;
            };
#pragma unroll 1
            for (int32_t k = 0; k < n_ch - 1; k += 2) {  // the others, in order
              const int32_t ca = k + (k >= own), cb = min(k + 1 + (k + 1 >= own), n_ch - 1);
              const bool two = k + 1 < n_ch - 1;
              const float* pa = p0 + ca * cstride;
              const float* pb = p0 + cb * cstride;
              float4 va[8], vb[8];
              const float ma = __ldcg(pa + 128 * 128 + row), la = __ldcg(pa + 128 * 128 + 128 + row);
              const float mb = __ldcg(pb + 128 * 128 + row), lb = __ldcg(pb + 128 * 128 + 128 + row);
#pragma unroll
              for (int x = 0; x < 8; ++x) va[x] = __ldcg(reinterpret_cast<const float4*>(pa + ((cc * 8 + x) * 128 + row) * 4));
#pragma unroll
              for (int x = 0; x < 8; ++x)
                vb[x] = two ? __ldcg(reinterpret_cast<const float4*>(pb + ((cc * 8 + x) * 128 + row) * 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
              const float wa = la > 0.f ? ex2(ma - m_all) : 0.f, wb = two && lb > 0.f ? ex2(mb - m_all) : 0.f;
              if (k == 0) tc_wait_ld();
              if (!own_in && own < ca) add_own();
              add(wa, va);
              if (two) {
                if (!own_in && own < cb) add_own();
                add(wb, vb);
              }
            }
            if (!own_in) add_own();
            if (row_valid) {
#pragma unroll
              for (int x = 0; x < 32; x += 16) {
                uint32_t w[8];
#pragma unroll
                for (int y = 0; y < 8; ++y) w[y] = pack_bf16(acc[x + 2 * y] * inv, acc[x + 2 * y + 1] * inv);
                st_global_v8(dst + 32 * cc + x, w);
              }
            }
          }
          if (lse && row_valid)
            lse[(int64_t)hq * hdr->total_tokens + q_first + row] = (m_all + log2f(l_all)) * 0.6931471805599453f;
        }
      }
      release_unit();
    }
  }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
  if (tid == 0 && abort_s && start_ok) atomicCAS(status, 0, (int32_t)abort_code_s);  // the first code raised stays
}

static purekv_status launch(const PrefillArgs& a, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,
                            const CUtensorMap& mk64, const CUtensorMap& mv64, const CUtensorMap& mo, int32_t* status) {
  constexpr int BK = 128;
  const size_t smem = 1024 + 2 * 2 * (size_t)kBQ * 128 + 2 * (size_t)Cfg<BK>::kStages * 2 * BK * 128 +
                      2 * (size_t)Cfg<BK>::kMeta * Cfg<BK>::kMaskBytes;
  static std::atomic<int> launch_regs{0};  // the compiled register count: the same on every device, read once
  int regs = launch_regs.load(std::memory_order_relaxed);
  if (regs == 0) {
    cudaFuncAttributes fa;
    PK_CUDA(cudaFuncGetAttributes(&fa, prefill_tc_kernel<BK>));
    regs = fa.numRegs;
    launch_regs.store(regs, std::memory_order_relaxed);
  }
  PK_REQUIRE(256 * kRegsSoftmax + 128 * kRegsOther <= kThreads * regs, PUREKV_ERR_UNSUPPORTED,
             "prefill kernel was compiled with %d registers per thread, too few for its register hand-over", regs);
  {
    static std::atomic<uint64_t> smem_allowed{0};
    const purekv_status st_smem = allow_max_dynamic_smem(prefill_tc_kernel<BK>, smem_allowed);
    if (st_smem != PUREKV_OK) return st_smem;
  }
  dim3 grid((unsigned)a.info->n_ctas);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = a.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see griddepcontrol in the kernel
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  PK_CUDA(cudaLaunchKernelEx(&cfg, prefill_tc_kernel<BK>, mq, mk, mv, mk64, mv64, mo, (__nv_bfloat16*)a.o, a.lse,
                             (uint8_t*)a.plan, (float*)a.ws, a.n_q_heads, a.n_kv_heads,
                             a.scale * 1.4426950408889634f, status, wait_limit_ns(), (int64_t)a.info->bytes_used,
                             (int64_t)(a.ws_bytes / sizeof(float)), a.info->n_units, a.n_layers, a.o_stride, a.lse_stride));
  PK_CUDA(cudaGetLastError());
  return PUREKV_OK;
}

}  // namespace tc

purekv_status launch_prefill_tc(const PrefillArgs& a) {
  using namespace tc;
  PK_REQUIRE(a.info->tile_q == kBQ && (a.info->tile_k == 64 || a.info->tile_k == 128) && a.head_dim == kD,
             PUREKV_ERR_UNSUPPORTED, "tensor-core prefill needs tile_q 128, tile_k 64/128, head_dim 128");
  PK_REQUIRE(a.info->n_ctas >= 1 && a.info->n_units >= 1, PUREKV_ERR_INVALID_ARG, "plan holds no schedule");
  PK_REQUIRE((uintptr_t)a.o % 32 == 0, PUREKV_ERR_INVALID_ARG, "O must be 32-byte aligned for the tensor-core kernel");
  const int64_t T = a.batch->total_tokens;
  CUtensorMap mq, mk, mv, mk64, mv64, mo;
  purekv_status st;
  const int32_t L = a.n_layers;
  const int64_t q_stride = L > 1 ? a.q_stride : T * a.n_q_heads * kD, kv_stride = L > 1 ? a.kv_stride : T * a.n_kv_heads * kD;
  if ((st = make_map_layers(&mq, a.q, T, a.n_q_heads, kBQ, L, q_stride)) != PUREKV_OK) return st;
  if ((st = make_map_layers(&mk, a.k, T, a.n_kv_heads, 128, L, kv_stride)) != PUREKV_OK) return st;
  if ((st = make_map_layers(&mv, a.v, T, a.n_kv_heads, 128, L, kv_stride)) != PUREKV_OK) return st;
  if ((st = make_map_layers(&mk64, a.k, T, a.n_kv_heads, 64, L, kv_stride)) != PUREKV_OK) return st;
  if ((st = make_map_layers(&mv64, a.v, T, a.n_kv_heads, 64, L, kv_stride)) != PUREKV_OK) return st;
  if ((st = make_map_layers(&mo, a.o, T, a.n_q_heads, kBQ, L, L > 1 ? a.o_stride : T * a.n_q_heads * kD)) != PUREKV_OK) return st;
  int32_t* status = a.status;
  if (!status) {
    const purekv_status st_w = default_status_word(&status);
    if (st_w != PUREKV_OK) return st_w;
  }
  return launch(a, mq, mk, mv, mk64, mv64, mo, status);
}

}  // namespace purekv
