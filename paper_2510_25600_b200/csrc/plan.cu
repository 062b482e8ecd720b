// Host-side planning for ST-SpAttn prefill (Sec. 3.2): turns the batch shape and the mask
// parameters into per-query-tile lists of kept key tiles, each classified as
//   full    -- every (row, key) pair of the tile is kept: no predicate in the kernel,
//   diag    -- exactly the causal pairs j <= i are kept: only the causal compare,
//   general -- the kernel reads a bit mask (one bit per row and key) stored in the plan.
// Work per query tile is O(rows x intervals): each row's kept keys are a union of a few
// position intervals (prefix + first frames, spans of the current frame, spans or single cells
// of linked earlier frames), accumulated into per-key-tile pair counts; general tiles get their
// bits from the same intervals.  The kernels therefore never evaluate the mask's definition.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "common.cuh"

namespace purekv {

static thread_local char g_err[512] = "";
static std::atomic<uint64_t> g_wait_limit_ns{1000ull * 1000ull * 1000ull};

uint64_t wait_limit_ns() { return g_wait_limit_ns.load(std::memory_order_relaxed); }

void set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
}

purekv_status check_batch(const purekv_batch* b, bool need_device) {
  PK_REQUIRE(b != nullptr, PUREKV_ERR_INVALID_ARG, "batch is null");
  PK_REQUIRE(b->n_req >= 0 && b->total_tokens >= 0, PUREKV_ERR_INVALID_ARG, "negative batch size");
  PK_REQUIRE(b->h_cu_seqlens != nullptr, PUREKV_ERR_INVALID_ARG, "h_cu_seqlens is null");
  PK_REQUIRE(!need_device || b->cu_seqlens != nullptr || b->n_req == 0 || b->total_tokens == 0, PUREKV_ERR_INVALID_ARG,
             "cu_seqlens (device) is null");
  PK_REQUIRE(b->h_cu_seqlens[0] == 0, PUREKV_ERR_INVALID_ARG, "cu_seqlens[0] must be 0");
  for (int r = 0; r < b->n_req; ++r)
    PK_REQUIRE(b->h_cu_seqlens[r + 1] >= b->h_cu_seqlens[r], PUREKV_ERR_INVALID_ARG,
               "cu_seqlens must be non-decreasing (request %d)", r);
  PK_REQUIRE(b->h_cu_seqlens[b->n_req] == b->total_tokens, PUREKV_ERR_INVALID_ARG,
             "total_tokens %lld != cu_seqlens[n_req] %d", (long long)b->total_tokens,
             b->h_cu_seqlens[b->n_req]);
  return PUREKV_OK;
}

static int64_t align16(int64_t x) { return (x + 15) & ~int64_t(15); }

static purekv_status check_params(const purekv_batch* b, const purekv_st_params* p, purekv_dtype dtype,
                                  int32_t head_dim, int* tile_q, int* tile_k) {
  purekv_status st = check_batch(b, false);
  if (st != PUREKV_OK) return st;
  PK_REQUIRE(p != nullptr, PUREKV_ERR_INVALID_ARG, "params is null");
  PK_REQUIRE(b->h_n_prefix && b->h_n_frames, PUREKV_ERR_INVALID_ARG, "h_n_prefix / h_n_frames is null");
  PK_REQUIRE(p->grid_h >= 1 && p->grid_w >= 1 && p->grid_h <= 32767 && p->grid_w <= 32767,
             PUREKV_ERR_INVALID_ARG, "grid %dx%d out of range", p->grid_h, p->grid_w);
  PK_REQUIRE(p->tile == 16 || p->tile == 32 || p->tile == 64 || p->tile == 128, PUREKV_ERR_UNSUPPORTED,
             "tile %d not in {16,32,64,128}", p->tile);
  PK_REQUIRE(p->anchor_frames >= 0 && p->spatial_radius >= -1 && p->temporal_depth >= -1 &&
                 p->temporal_radius >= -1 && p->temporal_stride >= 1 && p->temporal_stride <= 32767 &&
                 p->temporal_depth <= 32767 && p->local_window >= 0 && p->atrous_dilation >= 0,
             PUREKV_ERR_INVALID_ARG, "mask parameter out of range");
  PK_REQUIRE(dtype == PUREKV_BF16 || dtype == PUREKV_FP32, PUREKV_ERR_INVALID_ARG, "unknown dtype");
  const int64_t n = (int64_t)p->grid_h * p->grid_w;
  for (int r = 0; r < b->n_req; ++r) {
    const int64_t len = b->h_cu_seqlens[r + 1] - b->h_cu_seqlens[r];
    PK_REQUIRE(b->h_n_prefix[r] >= 0 && b->h_n_frames[r] >= 0 && b->h_n_frames[r] <= 32767 &&
                   b->h_n_prefix[r] + b->h_n_frames[r] * n <= len,
               PUREKV_ERR_INVALID_ARG, "request %d: prefix %d + %d frames of %lld tokens exceed length %lld", r,
               b->h_n_prefix[r], b->h_n_frames[r], (long long)n, (long long)len);
  }
  // Tensor-core kernel: 128 query rows per tile, keys per tile = the skip granularity.
  const bool tc = dtype == PUREKV_BF16 && head_dim == 128 && (p->tile == 64 || p->tile == 128);
  *tile_k = p->tile;
  *tile_q = tc ? 128 : std::min(p->tile, 64);  // CUDA-core kernel: at most 64 rows per tile
  return PUREKV_OK;
}

struct Span { int32_t a, b; };  // inclusive request-relative positions

// The status word of calls made without one.  In host code this name is only a stand-in for the symbol: the device
// address comes from cudaGetSymbolAddress, once per device.
static __device__ int32_t g_default_status;

purekv_status default_status_word(int32_t** out) {
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static int32_t* ptrs[kMaxDevices] = {};
  int dev = -1;
  PK_CUDA(cudaGetDevice(&dev));
  PK_REQUIRE(dev >= 0 && dev < kMaxDevices, PUREKV_ERR_UNSUPPORTED, "device ordinal %d is beyond %d", dev, kMaxDevices);
  std::lock_guard<std::mutex> lock(mu);
  if (!ptrs[dev]) {
    int32_t* p = nullptr;
    PK_CUDA(cudaGetSymbolAddress((void**)&p, g_default_status));
    PK_REQUIRE(p != nullptr, PUREKV_ERR_CUDA, "cudaGetSymbolAddress returned a null status address");
    ptrs[dev] = p;
  }
  *out = ptrs[dev];
  return PUREKV_OK;
}

}  // namespace purekv

using namespace purekv;

extern "C" {

const char* purekv_version(void) { return "purekv-b200 0.2.0 (sm_100a)"; }

void purekv_set_wait_limit_ns(uint64_t ns) {
  g_wait_limit_ns.store(ns ? ns : 1000ull * 1000ull * 1000ull, std::memory_order_relaxed);
}

void purekv_last_error(char* buf, size_t n) {
  if (!buf || n == 0) return;
  strncpy(buf, g_err, n - 1);
  buf[n - 1] = 0;
}

purekv_status purekv_budget(int32_t len, int32_t window, double keep_ratio, int32_t* h_out, int32_t* k_out) {
  PK_REQUIRE(len >= 0 && window >= 0 && keep_ratio >= 0.0 && h_out && k_out, PUREKV_ERR_INVALID_ARG,
             "purekv_budget: bad argument");
  const int32_t w = std::min(window, len);
  const double kf = keep_ratio * (double)len;
  int32_t k = kf >= (double)len ? len : (int32_t)kf;  // floor of a non-negative value
  k = std::min(len, std::max(w, k));
  *h_out = k - w;
  *k_out = k;
  return PUREKV_OK;
}

// What a schedule takes in a plan.
struct ScheduleSize {
  int64_t units = 0, twin_entries = 0, counters = 0;
};

// Splits long kept-key lists into chunks and orders the (query tile, head pair, chunk) units by decreasing cost:
// the kernel's n_ctas persistent CTAs start with the first n_ctas units and draw the rest from a counter as they
// finish, so the order is longest-first list scheduling carried out at run time.  The costs also decide how finely
// long lists are cut.  They are in quarters of a 64-key half of a list entry: 4 per
// half that the entry lists (5 when it carries a bit mask), 6 per unit (query load, pipeline fill, epilogue) and 14 more for a
// chunk of a split list (fp32 partial result written out, and the merge).  The constants were fitted to unit times of an
// earlier form of the kernel, which also loaded the listed halves that hold no pair; today a half costs 0.78 of a whole entry
// rather than half of it, a chunk's merge less, and an entry with a bit mask of which a warp keeps one or two 32-key chunks less
// than one without.  The order they give is still the one measured.
//
// With an odd group size the group's last head has no partner; a unit for it alone takes as long as a unit for two
// heads.  Consecutive query tiles of a request whose lists are not split therefore share that head's unit (a twin
// unit, see Unit): the merged lists are appended to `entries`.
//
// `apart_size`: of the schedule that one layer a launch would get (where n_layers > 1; the plan's own otherwise).
static void schedule_units(const std::vector<QTile>& qtiles, std::vector<int2>& entries, int32_t H, int32_t Hkv,
                           int32_t n_ctas, int32_t n_layers,
                           std::vector<Unit>& units, int32_t* n_counters,
                           int64_t* part_slots, int32_t* max_chunks, ScheduleSize* apart_size) {
  const int32_t G = H / Hkv, ppg = (G + 1) / 2, n_pairs = Hkv * ppg;
  const bool odd = (G & 1) != 0;
  const int32_t overhead = 6, split_extra = 14;
  const int32_t nq = (int32_t)qtiles.size();
  // running cost of the entries: a run's cost is a difference
  std::vector<int32_t> pre(entries.size() + 1, 0);
  for (size_t i = 0; i < entries.size(); ++i)
    pre[i + 1] = pre[i] + ((((entries[i].x >> 2) & 3) == 3) ? 2 : 1) * ((entries[i].x & 3) == kTileGeneral ? 5 : 4);
  auto halves = [&](int32_t first, int32_t last) { return pre[last] - pre[first]; };  // cost of entries [first, last)
  // The union of two runs of entries (of two query tiles' lists) in key-tile order: its cost and length; the entry
  // pairs go to `out` if given.
  auto merge_lists = [&](int32_t ia, int32_t ea, int32_t ib, int32_t eb, std::vector<int2>* out, int32_t* count) {
    int32_t cost = 0, n = 0;
    while (ia < ea || ib < eb) {
      const int32_t ka = ia < ea ? (entries[ia].x >> 4) : INT32_MAX, kb = ib < eb ? (entries[ib].x >> 4) : INT32_MAX;
      const int32_t kt = std::min(ka, kb);
      const int2 none = make_int2((kt << 4) | kTileNone, -1);
      const int2 xa = ka == kt ? entries[ia++] : none, xb = kb == kt ? entries[ib++] : none;
      const bool both = (((xa.x | xb.x) >> 2) & 3) == 3;
      const bool bits = (xa.x & 3) == kTileGeneral || (xb.x & 3) == kTileGeneral;
      cost += (both ? 2 : 1) * (bits ? 5 : 4);
      if (out) { out->push_back(xa); out->push_back(xb); }
      ++n;
    }
    *count = n;
    return cost;
  };
  // (the kernel counts a list's chunks in a byte per warp)
  auto chunks_of = [&](const QTile& q, int32_t l_max) { return std::min(255, std::max(1, (q.entry_count + l_max - 1) / l_max)); };
  // chunk c of nch of a tile's list, as a range of entries[]
  auto chunk_range = [&](const QTile& q, int32_t c, int32_t nch, int32_t* first, int32_t* last) {
    *first = q.entry_begin + (int32_t)((int64_t)q.entry_count * c / nch);
    *last = q.entry_begin + (int32_t)((int64_t)q.entry_count * (c + 1) / nch);
  };
  // partner[i]: the tile that shares tile i's odd-head units (i leads the twin), -2 if tile i is the second of a
  // twin, -1 if it stays alone.  Twins have the same number of chunks, and a merged chunk may be a quarter longer
  // than the cap on a chunk.  twin_cost, twin_len: the merged chunks' costs and lengths, leader by leader, chunk by chunk.
  std::vector<int32_t> partner, twin_cost, twin_len;
  struct Merged { int32_t n = -1, cost = 0; };
  std::vector<Merged> whole((size_t)nq);  // tile i's whole list merged with tile i + 1's: the same under every cap that leaves both whole
  auto merge_chunk = [&](int32_t i, int32_t c, int32_t nch) {
    Merged m;
    if (nch == 1 && whole[i].n >= 0) return whole[i];
    int32_t a0, a1, b0, b1;
    chunk_range(qtiles[i], c, nch, &a0, &a1);
    chunk_range(qtiles[i + 1], c, nch, &b0, &b1);
    m.cost = merge_lists(a0, a1, b0, b1, nullptr, &m.n);
    if (nch == 1) whole[i] = m;
    return m;
  };
  auto find_twins = [&](int32_t l_max) {
    partner.assign((size_t)nq, -1);
    twin_cost.clear();
    twin_len.clear();
    if (!odd) return;
    for (int32_t i = 0; i + 1 < nq; ++i) {
      const QTile &a = qtiles[i], &b = qtiles[i + 1];
      const int32_t nch = chunks_of(a, l_max);
      if (partner[i] != -1 || a.req_start != b.req_start || nch != chunks_of(b, l_max)) continue;
      const size_t at = twin_cost.size();
      bool fits = true;
      for (int32_t c = 0; c < nch && fits; ++c) {
        const Merged m = merge_chunk(i, c, nch);
        twin_cost.push_back(m.cost);
        twin_len.push_back(m.n);
        fits = m.n <= l_max + l_max / 4;
      }
      if (!fits) {
        twin_cost.resize(at);
        twin_len.resize(at);
        continue;
      }
      partner[i] = i + 1;
      partner[i + 1] = -2;
    }
  };
  std::vector<Unit> items;
  std::vector<int32_t> item_cost;
  std::vector<int2> twin_entries;
  std::vector<int32_t> part_of, counter_of;  // per query tile: first workspace slot and merge counter, -1 if unsplit
  int32_t counters = 0, mc = 1;
  int64_t slots = 0;
  // the units when no chunk of a list may be longer than l_max entries, by decreasing cost (equal costs as they come)
  auto make_items = [&](int32_t l_max) {
    find_twins(l_max);
    part_of.assign((size_t)nq, -1);
    counter_of.assign((size_t)nq, -1);
    for (int32_t qi = 0; qi < nq; ++qi) {
      const int32_t nch = chunks_of(qtiles[qi], l_max);
      mc = std::max(mc, nch);
      if (nch > 1) {
        part_of[qi] = (int32_t)slots;
        counter_of[qi] = counters;
        slots += nch;
        counters += H;
      }
    }
    size_t twin_at = 0;
    for (int32_t qi = 0; qi < nq; ++qi) {
      const QTile& q = qtiles[qi];
      const int32_t nch = chunks_of(q, l_max);
      for (int32_t c = 0; c < nch; ++c) {
        int32_t a, e;
        chunk_range(q, c, nch, &a, &e);
        const int32_t extra = overhead + (nch > 1 ? split_extra : 0), cost = halves(a, e) + extra;
        for (int32_t pr = 0; pr < n_pairs; ++pr) {
          if (partner[qi] != -1 && pr % ppg == ppg - 1) continue;  // the odd head goes into a twin unit
          Unit u = {};
          u.q_start = q.q_start; u.q_rows = q.q_rows; u.req_start = q.req_start;
          u.ent_begin = a; u.ent_count = e - a;
          u.pair = pr; u.chunk = c; u.n_chunks = nch;
          u.part_base = part_of[qi]; u.counter_base = counter_of[qi];
          u.part_base1 = u.counter_base1 = -1;
          items.push_back(u);
          item_cost.push_back(cost);
        }
        if (partner[qi] >= 0) {
          const QTile& q1 = qtiles[partner[qi]];
          int32_t a1, e1, n = 0;
          chunk_range(q1, c, nch, &a1, &e1);
          const int32_t at = (int32_t)(entries.size() + twin_entries.size());
          merge_lists(a, e, a1, e1, &twin_entries, &n);
          const int32_t cost2 = twin_cost[twin_at++] + extra;
          for (int32_t g = 0; g < Hkv; ++g) {
            Unit u = {};
            u.q_start = q.q_start; u.q_rows = q.q_rows; u.req_start = q.req_start;
            u.q_start1 = q1.q_start; u.q_rows1 = q1.q_rows;
            u.ent_begin = at; u.ent_count = n;
            u.pair = g * ppg + ppg - 1; u.chunk = c; u.n_chunks = nch;
            u.part_base = part_of[qi]; u.counter_base = counter_of[qi];
            u.part_base1 = part_of[partner[qi]]; u.counter_base1 = counter_of[partner[qi]];
            items.push_back(u);
            item_cost.push_back(cost2);
          }
        }
      }
    }
    // counting sort (costs are small numbers: ten per entry of a chunk at most, and the overheads)
    int32_t top = 0;
    for (int32_t c : item_cost) top = std::max(top, c);
    std::vector<int32_t> at((size_t)top + 2, 0);  // at[c]: where the units of cost c begin
    for (int32_t c : item_cost) ++at[c];
    int32_t run = 0;
    for (int32_t c = top; c >= 0; --c) {
      const int32_t n = at[c];
      at[c] = run;
      run += n;
    }
    units.resize(items.size());
    for (size_t i = 0; i < items.size(); ++i) units[at[item_cost[i]]++] = items[i];
  };
  // The time the last CTA ends when the CTAs draw units in decreasing order of cost, each as it becomes free; anything
  // above `limit` is answered as soon as it is known.  Units of one cost and CTAs free at the same time are counted, not
  // listed: the earliest free time only grows, so one pass over the times serves all units.
  std::vector<int32_t> n_of_cost, n_free;
  int64_t total = 0;  // the units' costs
  ScheduleSize size;
  auto makespan = [&](int32_t l_max, int64_t limit) {
    find_twins(l_max);
    n_of_cost.clear();
    total = 0;
    size = ScheduleSize{};
    auto add = [&](int32_t cost, int32_t n) {
      size.units += n;
      if ((size_t)cost >= n_of_cost.size()) n_of_cost.resize((size_t)cost + 1, 0);
      n_of_cost[cost] += n;
      total += (int64_t)cost * n;
    };
    size_t twin_at = 0;
    for (int32_t qi = 0; qi < nq; ++qi) {
      const QTile& q = qtiles[qi];
      const int32_t nch = chunks_of(q, l_max), extra = overhead + (nch > 1 ? split_extra : 0);
      if (nch > 1) size.counters += H;
      for (int32_t c = 0; c < nch; ++c) {
        int32_t a, e;
        chunk_range(q, c, nch, &a, &e);
        add(halves(a, e) + extra, partner[qi] != -1 ? n_pairs - Hkv : n_pairs);
        if (partner[qi] >= 0) {
          size.twin_entries += 2 * twin_len[twin_at];
          add(twin_cost[twin_at++] + extra, Hkv);
        }
      }
    }
    n_free.assign((size_t)(total / n_ctas) + n_of_cost.size() + 1, 0);  // CTAs that become free at each time
    n_free[0] = n_ctas;
    int64_t end = 0, now = 0;
    for (int32_t cost = (int32_t)n_of_cost.size() - 1; cost > 0; --cost) {
      for (int32_t m = n_of_cost[cost]; m > 0;) {
        while (n_free[now] == 0) ++now;
        const int32_t k = std::min(m, n_free[now]);
        n_free[now] -= k;
        n_free[now + cost] += k;
        m -= k;
        end = std::max(end, now + cost);
        if (end > limit) return end;
      }
    }
    return end;
  };
  // Splitting shortens the units the CTAs end on but costs a partial result and a merge per chunk.  With few units
  // per CTA the trade is decided by trying: the cap on a chunk's length that ends soonest under the cost model wins.
  // With many units the ends even out by themselves and only the very longest lists are cut.
  int32_t l_best = 64;
  if ((int64_t)qtiles.size() * n_pairs < 12 * (int64_t)n_ctas) {
    int64_t t_best = -1;
    for (int32_t l_max : {64, 24, 12, 9, 7, 5}) {
      const int64_t t = makespan(l_max, t_best < 0 ? INT64_MAX : t_best);
      if (t_best < 0 || t <= t_best) { t_best = t; l_best = l_max; }  // on a tie the finer cut
    }
  }
  // Launches of several layers need whole lists, and pass from one layer to the next without waiting for its end: layers but
  // the last cost the CTAs' share of the units.  Taken if that ends before n_layers launches of the lists as cut above would,
  // a launch's start (8 us, of which a 128-key entry takes 1.6) counted in.  Few layers of long lists fall to the other side:
  // one CTA would be on the longest list when the others are done.
  if (n_layers > 1) {
    const int32_t l_whole = 1 << 28, launch = 40;
    const int64_t apart = n_layers * (makespan(l_best, INT64_MAX) + launch);
    *apart_size = size;
    const int64_t last = makespan(l_whole, INT64_MAX);
    if ((n_layers - 1) * (total + n_ctas - 1) / n_ctas + last + launch <= apart) l_best = l_whole;
  }
  make_items(l_best);
  if (n_layers == 1) *apart_size = ScheduleSize{(int64_t)units.size(), (int64_t)twin_entries.size(), counters};
  entries.insert(entries.end(), twin_entries.begin(), twin_entries.end());
  *n_counters = counters;
  *part_slots = slots * H;
  *max_chunks = mc;
}

// A plan on the host: its sections, and their layout in the buffer.
struct HostPlan {
  PlanHeader h;
  int64_t total = 0;  // bytes
  int64_t room = 0;   // bytes, also for the plan of the same layers one a launch
  std::vector<QTile> qtiles;
  std::vector<int32_t> order;
  std::vector<int2> entries;
  std::vector<uint32_t> masks;
  std::vector<Unit> units;

  void write(uint8_t* dst) const {  // total bytes; gaps between sections and the counters are zero
    int64_t at = 0;
    auto section = [&](int64_t off, const void* src, size_t bytes) {
      memset(dst + at, 0, (size_t)(off - at));
      if (bytes) memcpy(dst + off, src, bytes);
      at = off + (int64_t)bytes;
    };
    section(0, &h, sizeof(h));
    section(h.off_qtiles, qtiles.data(), qtiles.size() * sizeof(QTile));
    section(h.off_order, order.data(), order.size() * 4);
    section(h.off_entries, entries.data(), entries.size() * 8);
    section(h.off_masks, masks.data(), masks.size() * 4);
    section(h.off_units, units.data(), units.size() * sizeof(Unit));
    section(total, nullptr, 0);
  }
};

static purekv_status build_plan(const purekv_batch* b, const purekv_st_params* p, purekv_dtype dtype,
                                int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, int32_t n_ctas, int32_t n_layers,
                                purekv_plan_info* info, HostPlan& plan) {
  int tq, gk;  // rows per query tile; skip granularity in keys (the mask parameter `tile`)
  purekv_status st = check_params(b, p, dtype, head_dim, &tq, &gk);
  if (st != PUREKV_OK) return st;
  // The tensor-core kernel always works on 128-key entries; with a 64-key skip granularity an entry carries a
  // 2-bit mask of the halves that hold kept pairs, and an absent half is neither loaded nor computed.
  const int32_t tk = tq == 128 ? 128 : gk;  // keys per list entry
  const int32_t hpe = tk / gk;              // key blocks of the skip granularity per entry (1 or 2)
  PK_REQUIRE(info, PUREKV_ERR_INVALID_ARG, "info is null");
  PK_REQUIRE(n_q_heads >= 1 && n_kv_heads >= 1 && n_q_heads % n_kv_heads == 0 && n_q_heads <= 65535,
             PUREKV_ERR_INVALID_ARG, "n_q_heads %d must be a positive multiple of n_kv_heads %d", n_q_heads,
             n_kv_heads);
  PK_REQUIRE(n_ctas >= 0 && n_ctas <= 4096, PUREKV_ERR_INVALID_ARG, "n_ctas %d outside [0, 4096]", n_ctas);
  PK_REQUIRE(n_layers >= 1 && n_layers <= 65535, PUREKV_ERR_INVALID_ARG, "n_layers %d outside [1, 65535]", n_layers);
  if (n_ctas == 0) n_ctas = 148;  // one persistent CTA per SM of a B200
  const bool dense = (p->flags & PUREKV_FLAG_DENSE_CAUSAL) != 0;
  const int32_t gw = p->grid_w, gh = p->grid_h, n = gw * gh;
  const int64_t T = b->total_tokens;
  const int32_t wpr = std::max(1, tk / 32);  // mask words per row of a general tile

  const int32_t gsh = 31 - __builtin_clz((unsigned)gk), tsh = 31 - __builtin_clz((unsigned)tk);  // gk and tk are powers of two
  std::vector<QTile>& qtiles = plan.qtiles;
  std::vector<int2>& entries = plan.entries;
  std::vector<uint32_t>& masks = plan.masks;
  std::vector<uint32_t> mask_halves;  // per mask of a tensor-core plan: bit h set when its keys 64h .. 64h+63 hold any kept pair
  memset(info, 0, sizeof(*info));

  std::vector<int64_t> cnt, diff, cg;  // kept pairs per gk-key block of the current query tile
  std::vector<Span> spans, row_spans, merged;
  std::vector<char> blk_kept;
  std::vector<int32_t> mask_of;  // per key tile of the current query tile: first word of its bit mask, or -1
  const bool coarse = (p->flags & PUREKV_FLAG_COARSE_BLOCKS) != 0 && !dense;
  std::vector<int32_t> row_off;
  for (int r = 0; r < b->n_req; ++r) {
    const int32_t base = b->h_cu_seqlens[r];
    const int32_t len = b->h_cu_seqlens[r + 1] - base;
    const int32_t npre = b->h_n_prefix[r], nfr = b->h_n_frames[r];
    const int32_t vis_end = npre + nfr * n;
    const int32_t nkt = (len + gk - 1) / gk + 2;
    cnt.assign((size_t)nkt + 2, 0);
    diff.assign((size_t)nkt + 3, 0);
    cg.assign((size_t)nkt + 3, 0);
    const int32_t anchor_end = (int32_t)std::min<int64_t>(vis_end, npre + (int64_t)p->anchor_frames * n);  // exclusive
    // the token-level mask of row i as disjoint ascending spans of kept key positions
    int32_t at_i = -2, at_f = 0, at_c = 0, at_y = 0, at_x = 0;  // frame, cell and its coordinates of the last visual row asked for
    auto token_spans = [&](int32_t i, std::vector<Span>& out) {
      out.clear();
      const bool visual = i >= npre && i < vis_end;
      if (dense || !visual) {
        out.push_back({0, i});  // text rows and the dense mask: plain causal
        return;
      }
      spans.clear();
      if (anchor_end > 0) spans.push_back({0, std::min(i, anchor_end - 1)});  // prefix + first frame(s)
      if (i == at_i + 1) {  // rows mostly come in order: step instead of dividing
        if (++at_x == gw) { at_x = 0; ++at_y; }
        if (++at_c == n) { at_c = at_y = at_x = 0; ++at_f; }
      } else {
        at_f = (i - npre) / n; at_c = (i - npre) % n; at_y = at_c / gw; at_x = at_c % gw;
      }
      at_i = i;
      const int32_t f = at_f, y = at_y, x = at_x;
      const int32_t fs = npre + f * n;
      if (p->spatial_radius < 0) {
        spans.push_back({fs, i});  // the current frame, causal
      } else {
        const int32_t rr = p->spatial_radius;
        for (int32_t yy = std::max(0, y - rr); yy <= y; ++yy) {
          const int32_t xa = std::max(0, x - rr), xb = yy == y ? x : std::min(gw - 1, x + rr);
          spans.push_back({fs + yy * gw + xa, fs + yy * gw + xb});
        }
      }
      for (int32_t m = 1;; ++m) {  // linked earlier frames: the corresponding cell (or a window / the frame)
        const int64_t fj = (int64_t)f - (int64_t)m * p->temporal_stride;
        if (fj < 0 || (p->temporal_depth >= 0 && m > p->temporal_depth)) break;
        const int32_t fjs = npre + (int32_t)fj * n;
        if (p->temporal_radius < 0) {
          spans.push_back({fjs, fjs + n - 1});
        } else {
          const int32_t rr = p->temporal_radius;
          for (int32_t yy = std::max(0, y - rr); yy <= std::min(gh - 1, y + rr); ++yy)
            spans.push_back({fjs + yy * gw + std::max(0, x - rr), fjs + yy * gw + std::min(gw - 1, x + rr)});
        }
      }
      if (p->local_window > 0) spans.push_back({std::max(npre, i - p->local_window + 1), i});  // the most recent positions
      if (p->atrous_dilation > 0)                                                             // every D-th position back
        for (int32_t j = i; j >= npre; j -= p->atrous_dilation) spans.push_back({j, j});
      if (spans.size() <= 12) {  // a few spans, nearly in order: insertion
        for (size_t x = 1; x < spans.size(); ++x) {
          const Span sp = spans[x];
          size_t y = x;
          for (; y > 0 && spans[y - 1].a > sp.a; --y) spans[y] = spans[y - 1];
          spans[y] = sp;
        }
      } else {
        std::sort(spans.begin(), spans.end(), [](const Span& u, const Span& v) { return u.a < v.a; });
      }
      int32_t ca = spans[0].a, cb = spans[0].b;
      for (size_t s = 1; s < spans.size(); ++s) {
        if (spans[s].a <= cb + 1) cb = std::max(cb, spans[s].b);
        else { out.push_back({ca, cb}); ca = spans[s].a; cb = spans[s].b; }
      }
      out.push_back({ca, cb});
    };
    int32_t cached_rb = -1;          // block of rows whose kept key blocks are in blk_kept (coarse masks)
    for (int32_t q0 = 0; q0 < len; q0 += tq) {
      const int32_t q1 = std::min(len, q0 + tq);  // exclusive
      const int32_t kt_hi = (q1 - 1) / tk;        // last list entry a causal mask reaches
      const int32_t kg_hi = (q1 - 1) / gk;        // last gk-key block a causal mask reaches
      std::fill(cnt.begin(), cnt.begin() + kg_hi + 3, 0);
      std::fill(diff.begin(), diff.begin() + kg_hi + 4, 0);
      row_spans.clear();
      row_off.assign(1, 0);
      auto add_span = [&](int32_t a, int32_t bb) {  // inclusive, a <= bb
        row_spans.push_back({a, bb});
        const int32_t ta = a >> gsh, tb = bb >> gsh;
        if (ta == tb) { cnt[ta] += bb - a + 1; return; }
        cnt[ta] += (ta + 1) * gk - a;
        cnt[tb] += bb - tb * gk + 1;
        diff[ta + 1] += gk;
        diff[tb] -= gk;
      };
      // each row's kept keys as disjoint ascending spans (Sec. 3.2; App. A.3 for the local and atrous terms)
      // (a tile of plain causal rows needs none: its counts follow from the diagonal alone)
      const bool plain = dense || (!coarse && (q1 <= npre || q0 >= vis_end || npre == vis_end));
      for (int32_t i = q0; i < q1 && !plain; ++i) {
        if (!coarse) {
          token_spans(i, merged);
          for (const Span& sp : merged) add_span(sp.a, sp.b);
        } else {
          // block-level widening: the key blocks in which any row of this row's block keeps a pair (found once per
          // block of rows), each taken whole up to the diagonal
          const int32_t rb = i / gk;
          if (rb != cached_rb) {
            cached_rb = rb;
            const int32_t r_hi = std::min(len, rb * gk + gk);
            blk_kept.assign((size_t)(r_hi - 1) / gk + 1, 0);
            for (int32_t ii = rb * gk; ii < r_hi; ++ii) {
              token_spans(ii, merged);
              for (const Span& sp : merged)
                for (int32_t kb = sp.a / gk; kb <= sp.b / gk; ++kb) blk_kept[kb] = 1;
            }
          }
          for (int32_t kb = 0; kb <= i / gk; ++kb) {
            if (!blk_kept[kb]) continue;
            int32_t ke = kb;
            while (ke + 1 <= i / gk && blk_kept[ke + 1]) ++ke;
            add_span(kb * gk, std::min(ke * gk + gk - 1, i));
            kb = ke;
          }
        }
        row_off.push_back((int32_t)row_spans.size());
      }
      QTile qt;
      qt.q_start = base + q0;
      qt.q_rows = q1 - q0;
      qt.req_start = base;
      qt.req_len = len;
      qt.entry_begin = (int32_t)entries.size();
      qt.pad[0] = qt.pad[1] = 0;
      int64_t run = 0;
      int32_t n_general = 0;  // tiles of this row of tiles with a bit mask
      if (mask_of.size() < (size_t)kt_hi + 1) mask_of.resize((size_t)kt_hi + 1);
      std::fill(mask_of.begin(), mask_of.begin() + kt_hi + 1, -1);
      for (int32_t kg = 0; kg <= kg_hi + 1; ++kg) {
        run += diff[kg];
        cg[kg] = cnt[kg] + run;
      }
      if (plain)
        for (int32_t kg = 0; kg <= kg_hi; ++kg) {
          const int32_t j0 = kg * gk;
          cg[kg] = (int64_t)(q1 - q0) * gk;
          if (j0 + gk - 1 > q0) {
            cg[kg] = 0;
            for (int32_t i = std::max(q0, j0); i < q1; ++i) cg[kg] += std::min(gk, i - j0 + 1);
          }
        }
      info->tiles_causal += kg_hi + 1;
      for (int32_t kt = 0; kt <= kt_hi; ++kt) {
        int64_t c = 0;
        int32_t half_mask = 0;
        for (int32_t hh = 0; hh < hpe; ++hh) {
          const int32_t kg = kt * hpe + hh;
          if (kg <= kg_hi && cg[kg] > 0) { c += cg[kg]; half_mask |= 1 << hh; info->tiles_kept++; }
        }
        if (c == 0) continue;
        if (hpe == 1) half_mask = 3;  // one block per entry: both bits set by convention
        const int32_t j0 = kt * tk;
        const int64_t full = (int64_t)(q1 - q0) * tk;
        int64_t causal = full;  // pairs with j <= i inside this tile
        if (j0 + tk - 1 > q0) {
          causal = 0;
          for (int32_t i = q0; i < q1; ++i) causal += std::max(0, std::min(tk, i - j0 + 1));
        }
        int32_t cls = kTileGeneral, mask_at = -1;
        if (c == full && j0 + tk <= len) cls = kTileFull;
        else if (c == causal) cls = kTileDiag;
        if (cls == kTileGeneral) {
          // one bit per (row, key) of the tile, rows past q_rows stay zero; the bits follow once the tile's masks are known
          PK_REQUIRE(masks.size() + (size_t)n_general * tq * wpr + (size_t)tq * wpr < (size_t)INT32_MAX, PUREKV_ERR_UNSUPPORTED,
                     "mask table exceeds 2^31 words");
          mask_at = (int32_t)(masks.size() + (size_t)n_general++ * tq * wpr);
        }
        mask_of[kt] = mask_at;
        entries.push_back(make_int2((kt << 4) | (half_mask << 2) | cls, mask_at));
        info->pairs_kept += c;
        (cls == kTileFull ? info->tiles_full : cls == kTileDiag ? info->tiles_diag : info->tiles_general)++;
      }
      if (n_general) {  // row by row, each span into the masks of the tiles it crosses
        masks.resize(masks.size() + (size_t)n_general * tq * wpr, 0u);
        if (tq == 128) mask_halves.resize(mask_halves.size() + (size_t)n_general, 0u);
        for (int32_t i = q0; i < q1; ++i)
          for (int32_t s = row_off[i - q0]; s < row_off[i - q0 + 1]; ++s) {
            const int32_t a = row_spans[s].a, bb = row_spans[s].b;
            for (int32_t kt = a >> tsh; kt <= bb >> tsh; ++kt) {
              if (mask_of[kt] < 0) continue;
              const int32_t j0 = kt << tsh, lo = std::max(a - j0, 0), hi = std::min(bb - j0, tk - 1);  // bit range inside the tile row
              uint32_t* rw = masks.data() + mask_of[kt] + (size_t)(i - q0) * wpr;
              if (tq == 128) mask_halves[(size_t)mask_of[kt] / (128 * 4)] |= (1u << (lo >> 6)) | (1u << (hi >> 6));
              for (int32_t w = lo >> 5; w <= (hi >> 5); ++w) {
                const int32_t b0 = std::max(lo - 32 * w, 0), b1 = std::min(hi - 32 * w, 31);
                rw[w] |= (b1 - b0 == 31) ? 0xFFFFFFFFu : (((1u << (b1 - b0 + 1)) - 1u) << b0);
              }
            }
          }
      }
      qt.entry_count = (int32_t)entries.size() - qt.entry_begin;
      info->max_list = std::max(info->max_list, qt.entry_count);
      qtiles.push_back(qt);
    }
  }
  const int32_t nq = (int32_t)qtiles.size();
  std::vector<int32_t>& order = plan.order;
  order.resize((size_t)nq);
  for (int32_t i = 0; i < nq; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(),
                   [&](int32_t u, int32_t v) { return qtiles[u].entry_count > qtiles[v].entry_count; });

  // tensor-core plans carry the persistent kernel's schedule
  std::vector<Unit>& units = plan.units;
  int32_t n_counters = 0, max_chunks = 1;
  int64_t part_slots = 0;
  ScheduleSize apart;
  const int64_t n_listed = (int64_t)entries.size();
  const size_t n_masks = masks.size();
  if (tq == 128 && nq > 0) {
    schedule_units(qtiles, entries, n_q_heads, n_kv_heads, n_ctas, n_layers, units, &n_counters, &part_slots, &max_chunks, &apart);
    PK_REQUIRE(n_masks + entries.size() < (size_t)INT32_MAX, PUREKV_ERR_UNSUPPORTED, "mask table exceeds 2^31 words");
    masks.resize(n_masks + entries.size());
    for (size_t i = 0; i < entries.size(); ++i) {
      const uint32_t listed = ((uint32_t)entries[i].x >> 2) & 3u;
      masks[n_masks + i] = (entries[i].x & 3) == kTileGeneral ? listed & mask_halves[(size_t)entries[i].y / (128 * 4)] : listed;
    }
  } else {
    n_ctas = 0;
  }

  PlanHeader& h = plan.h;
  memset(&h, 0, sizeof(h));
  h.magic = kPlanMagic;
  h.tile_q = tq;
  h.tile_k = tk;
  h.n_qtiles = nq;
  h.total_tokens = T;
  h.n_entries = (int64_t)entries.size();
  h.n_mask_words = (int64_t)masks.size();
  h.words_per_row = wpr;
  h.n_ctas = units.empty() ? 0 : n_ctas;
  h.n_units = (int32_t)units.size();
  h.n_counters = n_counters;
  h.n_q_heads = n_q_heads;
  h.n_kv_heads = n_kv_heads;
  h.part_slots = part_slots;
  // Lays the sections out and returns the bytes they take.
  auto layout = [&](int64_t n_entries, int64_t n_mask_words, int64_t n_units, int64_t counters) {
    h.off_qtiles = align16(sizeof(PlanHeader));
    h.off_order = h.off_qtiles + align16((int64_t)nq * sizeof(QTile));
    h.off_entries = h.off_order + align16((int64_t)nq * 4);
    h.off_masks = h.off_entries + align16(n_entries * 8);
    h.off_units = h.off_masks + align16(n_mask_words * 4);
    h.off_counters = h.off_units + align16(n_units * (int64_t)sizeof(Unit));
    // the merge counters, then the kernel's two scheduling counters; all start at zero and the kernel leaves them so
    return h.off_counters + align16((counters + 2) * 4);
  };
  const int64_t apart_entries = n_listed + apart.twin_entries;
  const int64_t apart_total =
      layout(apart_entries, (int64_t)n_masks + (tq == 128 && nq > 0 ? apart_entries : 0), apart.units, apart.counters);
  const int64_t total = layout(h.n_entries, h.n_mask_words, h.n_units, n_counters);

  plan.total = total;
  plan.room = std::max(total, apart_total);

  info->tile_q = tq;
  info->tile_k = gk;
  info->n_qtiles = nq;
  info->bytes_used = total;
  info->dtype = (int32_t)dtype;
  info->head_dim = head_dim;
  info->n_q_heads = n_q_heads;
  info->n_kv_heads = n_kv_heads;
  info->n_ctas = h.n_ctas;
  info->n_units = h.n_units;
  info->max_chunks = max_chunks;
  info->ws_bytes = part_slots * kPartFloats * (int64_t)sizeof(float);
  return PUREKV_OK;
}

size_t purekv_plan_bytes(const purekv_batch* b, const purekv_st_params* p, purekv_dtype dtype, int32_t head_dim,
                         int32_t n_q_heads, int32_t n_kv_heads, int32_t n_ctas) {
  return purekv_plan_layers_bytes(b, p, dtype, head_dim, n_q_heads, n_kv_heads, n_ctas, 1);
}

size_t purekv_plan_layers_bytes(const purekv_batch* b, const purekv_st_params* p, purekv_dtype dtype, int32_t head_dim,
                                int32_t n_q_heads, int32_t n_kv_heads, int32_t n_ctas, int32_t n_layers) {
  purekv_plan_info info;
  HostPlan host;
  if (build_plan(b, p, dtype, head_dim, n_q_heads, n_kv_heads, n_ctas, n_layers, &info, host) != PUREKV_OK) return 0;
  return (size_t)host.room;
}

purekv_status purekv_plan_build_host(const purekv_batch* b, const purekv_st_params* p, purekv_dtype dtype,
                                     int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, int32_t n_ctas,
                                     void* h_plan, size_t plan_bytes, purekv_plan_info* info) {
  return purekv_plan_build_layers_host(b, p, dtype, head_dim, n_q_heads, n_kv_heads, n_ctas, 1, h_plan, plan_bytes, info);
}

purekv_status purekv_plan_build_layers_host(const purekv_batch* b, const purekv_st_params* p, purekv_dtype dtype,
                                            int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, int32_t n_ctas,
                                            int32_t n_layers, void* h_plan, size_t plan_bytes, purekv_plan_info* info) {
  PK_REQUIRE(h_plan, PUREKV_ERR_INVALID_ARG, "h_plan is null");
  HostPlan host;
  purekv_status st = build_plan(b, p, dtype, head_dim, n_q_heads, n_kv_heads, n_ctas, n_layers, info, host);
  if (st != PUREKV_OK) return st;
  PK_REQUIRE((size_t)host.total <= plan_bytes, PUREKV_ERR_WORKSPACE, "plan needs %zu bytes, buffer has %zu", (size_t)host.total,
             plan_bytes);
  host.write((uint8_t*)h_plan);
  return PUREKV_OK;
}

purekv_status purekv_plan_build(const purekv_batch* b, const purekv_st_params* p, purekv_dtype dtype,
                                int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, int32_t n_ctas, void* plan,
                                size_t plan_bytes, purekv_plan_info* info, void* stream) {
  PK_REQUIRE(plan, PUREKV_ERR_INVALID_ARG, "plan is null");
  HostPlan built;
  purekv_status st = build_plan(b, p, dtype, head_dim, n_q_heads, n_kv_heads, n_ctas, 1, info, built);
  if (st != PUREKV_OK) return st;
  PK_REQUIRE((size_t)built.total <= plan_bytes, PUREKV_ERR_WORKSPACE, "plan needs %zu bytes, buffer has %zu", (size_t)built.total,
             plan_bytes);
  std::vector<uint8_t> host((size_t)built.total);
  built.write(host.data());
  cudaStream_t s = (cudaStream_t)stream;
  PK_CUDA(cudaMemcpyAsync(plan, host.data(), host.size(), cudaMemcpyHostToDevice, s));
  PK_CUDA(cudaStreamSynchronize(s));
  return PUREKV_OK;
}

purekv_status purekv_poll_status(const int32_t* status, int32_t* h_out, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  PK_CUDA(cudaStreamSynchronize(s));
  int32_t v = 0;
  if (status) {
    PK_CUDA(cudaMemcpy(&v, status, sizeof(v), cudaMemcpyDeviceToHost));
  } else {
    // the library's own word, used by calls made with status == NULL: report it and clear it, so that one expired
    // wait does not block every later call of that kind
    int32_t* own = nullptr;
    purekv_status st = default_status_word(&own);
    if (st != PUREKV_OK) return st;
    PK_CUDA(cudaMemcpy(&v, own, sizeof(v), cudaMemcpyDeviceToHost));
    if (v != 0) PK_CUDA(cudaMemset(own, 0, sizeof(v)));
  }
  if (h_out) *h_out = v;
  PK_REQUIRE(v != (int32_t)PUREKV_ERR_BAD_PLAN, PUREKV_ERR_BAD_PLAN,
             "device status word is %d: a kernel refused the plan it was handed", v);
  PK_REQUIRE(v == 0, PUREKV_ERR_TIMEOUT, "device status word is %d: a bounded device-side wait expired", v);
  return PUREKV_OK;
}

}  // extern "C"
