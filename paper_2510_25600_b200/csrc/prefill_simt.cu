// CUDA-core ST-SpAttn prefill (Sec. 3.2) for the shapes the tensor-core kernel does not take:
// fp32 inputs (computed in fp32 throughout) and bf16 with head_dim other than 128.
//
// One CTA (128 threads) = R rows of a query tile of one query head, walking the plan's list of kept key tiles in chunks of
// NK keys: short tiles are put together, long ones taken in parts, so that the chunk, not the plan's tile, sets the work
// between two barriers.  K and V of the next chunk are copied with cp.async while the current one is used.  TPR threads
// share a row: for S = Q K^T each takes every TPR-th key of the chunk (float4 reads of a Q row that the threads of a row
// share and of K rows padded so that eight rows fall into different banks), the row's online-softmax state is kept by all
// of them, probabilities pass through shared memory inside the warp, and for P V each takes every TPR-th group of four
// dimensions.  RPT rows per thread reuse what is read of K and V.
// What bounds it: for large inputs the FMA pipe and the shared-memory reads that feed it (RPT = 4: 12 reads per 128
// FMAs); for a short prompt the chain of a row block's chunks, which is why the rows per CTA (R = 128 / TPR * RPT) come
// down until the CTAs cover the SMs.  Before (a warp per row, lanes along the keys, a plan tile between barriers) and now,
// dense causal: 288 tokens, 2 heads, fp32, head_dim 64: 114 -> 19 us; 1184 tokens, 8 heads, fp32, head_dim 64: 657 -> 140;
// 2336 tokens, 32 heads, head_dim 64 in bf16: 3706 -> 970, head_dim 128 in fp32: 5976 -> 2170.
#include "common.cuh"
#include "prefill.cuh"

namespace purekv {

constexpr int kSimtThreads = 128;

__device__ __forceinline__ float4 simt_load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 simt_load4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xFFFF0000u));
}
__device__ __forceinline__ void simt_store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void simt_store4(__nv_bfloat16* p, float4 v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
}

// A run of `u` keys of a chunk: one entry of the plan's list or a part of one.
struct SimtSeg {
  int32_t j0, cls, word;  // first key, TileClass or -1 (nothing there), first mask word of the query tile's row 0
};

template <typename T, int D, int NK>
struct SimtCfg {
  static constexpr int kLd = D + 16 / (int)sizeof(T);  // elements of a staged K or V row
  static constexpr int kLdQ = D + 4, kLdP = NK + 4;
  static size_t smem(int rows) {
    return 2 * 2 * (size_t)NK * kLd * sizeof(T) + (size_t)rows * (kLdQ + kLdP) * sizeof(float);
  }
};

__device__ __forceinline__ void simt_store1(float* p, float x) { *p = x; }
__device__ __forceinline__ void simt_store1(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }

// One row by one warp, straight from the plan's list and global memory: a row takes nothing from a key tile of which it keeps
// nothing, whatever stands there.  (The kernel below multiplies every V of a chunk of several tiles by the row's weights, zeros
// where the row keeps nothing; an infinity or a NaN there survives that, and such rows come here.)  `tile`: the query tile's place
// in the plan's order, `row`: the row in it, `q`: its query in shared memory.
template <typename T, int D>
__device__ __noinline__ void prefill_simt_row(const float* q, const T* k, const T* v, T* o, float* lse, const uint8_t* plan, int32_t tile,
                                              int32_t row, int32_t n_q_heads, int32_t n_kv_heads, float scale_log2) {
  const PlanHeader* hdr = reinterpret_cast<const PlanHeader*>(plan);
  const int32_t tk = hdr->tile_k, wpr = hdr->words_per_row, hq = blockIdx.y, g = hq / (n_q_heads / n_kv_heads);
  const QTile qt = reinterpret_cast<const QTile*>(plan + hdr->off_qtiles)[reinterpret_cast<const int32_t*>(plan + hdr->off_order)[tile]];
  const int2* entries = reinterpret_cast<const int2*>(plan + hdr->off_entries) + qt.entry_begin;
  const uint32_t* masks = reinterpret_cast<const uint32_t*>(plan + hdr->off_masks);
  const int lane = threadIdx.x & 31;
  const int32_t i = qt.q_start - qt.req_start + row;
  float m = -INFINITY, l = 0.f, acc[D / 32];
  for (int c = 0; c < D / 32; ++c) acc[c] = 0.f;
  for (int32_t e = 0; e < qt.entry_count; ++e) {
    const int2 ent = entries[e];
    const int32_t cls = ent.x & 3, j0 = (ent.x >> 4) * tk;
    float s[4], tmax = -INFINITY;  // (tk <= 128: at most four keys per lane)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int32_t c = lane + 32 * x, j = j0 + c;
      s[x] = -INFINITY;
      if (c < tk && j < qt.req_len) {
        const bool keep = cls == kTileGeneral ? (masks[ent.y + row * wpr + (c >> 5)] >> (c & 31)) & 1u : cls == kTileFull || j <= i;
        if (keep) {
          const T* kr = k + ((int64_t)(qt.req_start + j) * n_kv_heads + g) * D;
          float a = 0.f;
          for (int dd = 0; dd < D; ++dd) a = fmaf(q[dd], to_f32(kr[dd]), a);
          s[x] = a * scale_log2;
        }
      }
      tmax = fmaxf(tmax, s[x]);
    }
    for (int off = 16; off >= 1; off >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, off));
    if (tmax == -INFINITY) continue;
    const float mn = fmaxf(m, tmax), alpha = exp2f(m - mn);
    float sum = 0.f;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      s[x] = exp2f(s[x] - mn);
      sum += s[x];
    }
    for (int off = 16; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    l = l * alpha + sum;
    m = mn;
    for (int c = 0; c < D / 32; ++c) acc[c] *= alpha;
#pragma unroll
    for (int x = 0; x < 4; ++x)
      for (int c = 32 * x; c < min(tk, 32 * x + 32) && j0 + c < qt.req_len; ++c) {
        const float p = __shfl_sync(0xffffffffu, s[x], c & 31);
        const T* vr = v + ((int64_t)(qt.req_start + j0 + c) * n_kv_heads + g) * D + lane;
        for (int dd = 0; dd < D / 32; ++dd) acc[dd] = fmaf(p, to_f32(vr[32 * dd]), acc[dd]);
      }
  }
  const float inv = 1.f / l;
  const int64_t token = qt.q_start + row;
  for (int c = 0; c < D / 32; ++c) simt_store1(o + (token * n_q_heads + hq) * D + lane + 32 * c, acc[c] * inv);
  if (lse && lane == 0) lse[(int64_t)hq * hdr->total_tokens + token] = (m + log2f(l)) * 0.6931471805599453f;
}

template <typename T, int D, int NK, int TPR, int RPT>
__global__ void __launch_bounds__(kSimtThreads) prefill_simt_kernel(
    const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, T* __restrict__ o,
    float* __restrict__ lse, const uint8_t* __restrict__ plan, int32_t n_q_heads, int32_t n_kv_heads,
    float scale_log2) {
  using Cfg = SimtCfg<T, D, NK>;
  constexpr int LD = Cfg::kLd, LDQ = Cfg::kLdQ, LDP = Cfg::kLdP;
  constexpr int kGroups = kSimtThreads / TPR, R = kGroups * RPT, KPT = NK / TPR, ND = D / (4 * TPR);
  constexpr int kSegs = NK / 16;
  constexpr int CPR = D * (int)sizeof(T) / 16;  // 16-byte copies per row
  extern __shared__ __align__(16) uint8_t smem_raw[];
  __shared__ SimtSeg segs[3][kSegs];
  __shared__ uint32_t redo[2];  // rows with a value that is not finite
  T* kv = reinterpret_cast<T*>(smem_raw);                      // [2 stages][K, V][NK][LD]
  float* qs = reinterpret_cast<float*>(kv + 2 * 2 * NK * LD);  // [R][LDQ]
  float* ps = qs + R * LDQ;                                    // [R][LDP]

  const PlanHeader* hdr = reinterpret_cast<const PlanHeader*>(plan);
  const int32_t tq = hdr->tile_q, tk = hdr->tile_k, wpr = hdr->words_per_row;
  const int32_t n_sub = tq / R;  // row blocks of a query tile
  const int32_t* order = reinterpret_cast<const int32_t*>(plan + hdr->off_order);
  const QTile qt = reinterpret_cast<const QTile*>(plan + hdr->off_qtiles)[order[blockIdx.x / n_sub]];
  const int2* entries = reinterpret_cast<const int2*>(plan + hdr->off_entries) + qt.entry_begin;
  const uint32_t* masks = reinterpret_cast<const uint32_t*>(plan + hdr->off_masks);
  const int32_t row0 = (int32_t)(blockIdx.x % n_sub) * R;  // this CTA's first row of the query tile
  if (row0 >= qt.q_rows) return;
  const int32_t hq = blockIdx.y, g = hq / (n_q_heads / n_kv_heads);
  const int32_t i0 = qt.q_start - qt.req_start + row0;
  const int32_t u = min(tk, NK), ush = 31 - __clz(u), parts = tk / u, spc = NK / u;  // keys, parts of an entry, runs of a chunk
  const int32_t n_runs = qt.entry_count * parts, n_chunks = (n_runs + spc - 1) / spc;
  const int tid = threadIdx.x, grp = tid / TPR, kx = tid % TPR;

  auto seg_of = [&](int32_t chunk) -> SimtSeg {  // run number `tid` of the chunk
    const int32_t run = chunk * spc + tid;
    SimtSeg sg = {0, -1, 0};
    if (run < n_runs) {
      const int2 e = __ldg(entries + run / parts);
      const int32_t p0 = (run % parts) * u;
      sg = {(e.x >> 4) * tk + p0, e.x & 3, e.y + (p0 >> 5)};
    }
    return sg;
  };
  auto stage = [&](int32_t chunk) {
    if (chunk < n_chunks) {
      T* dst = kv + (chunk & 1) * 2 * NK * LD;
#pragma unroll 4
      for (int x = tid; x < NK * CPR; x += kSimtThreads) {
        const int row = x / CPR, c = (x % CPR) * (16 / (int)sizeof(T));
        const SimtSeg& sg = segs[chunk % 3][row >> ush];
        const int32_t j = sg.j0 + (row & (u - 1));
        const uint32_t bytes = sg.cls >= 0 && j < qt.req_len ? 16u : 0u;  // (0: zero fill)
        const int64_t src = bytes ? ((int64_t)(qt.req_start + j) * n_kv_heads + g) * D + c : 0;
        const uint32_t sa = (uint32_t)__cvta_generic_to_shared(dst + row * LD + c);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(k + src), "r"(bytes) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa + NK * LD * (int)sizeof(T)), "l"(v + src), "r"(bytes) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  if (tid < 2) redo[tid] = 0u;
  if (tid < spc) {
    segs[0][tid] = seg_of(0);
    segs[1][tid] = seg_of(1);
  }
  __syncthreads();
  stage(0);
  for (int x = tid; x < R * (D / 4); x += kSimtThreads) {
    const int row = x / (D / 4), c = 4 * (x % (D / 4));
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row0 + row < qt.q_rows) f = simt_load4(q + ((int64_t)(qt.q_start + row0 + row) * n_q_heads + hq) * D + c);
    simt_store4(qs + row * LDQ + c, f);
  }

  float m[RPT], l[RPT];
  float4 acc[RPT][ND];
#pragma unroll
  for (int rr = 0; rr < RPT; ++rr) {
    m[rr] = -INFINITY;
    l[rr] = 0.f;
#pragma unroll
    for (int nd = 0; nd < ND; ++nd) acc[rr][nd] = make_float4(0.f, 0.f, 0.f, 0.f);
  }

  for (int32_t ch = 0; ch < n_chunks; ++ch) {
    stage(ch + 1);
    SimtSeg ahead;
    if (tid < spc) ahead = seg_of(ch + 2);  // on its way while this chunk is used
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const T* ks = kv + (ch & 1) * 2 * NK * LD;
    const T* vs = ks + NK * LD;
    const SimtSeg* sg = segs[ch % 3];
    const int32_t n_keys = min(spc, n_runs - ch * spc) << ush;  // keys of the chunk that a run covers

    // S
    float s[RPT][KPT];
#pragma unroll
    for (int rr = 0; rr < RPT; ++rr)
#pragma unroll
      for (int j = 0; j < KPT; ++j) s[rr][j] = 0.f;
#pragma unroll 4
    for (int d = 0; d < D; d += 4) {
      float4 qv[RPT];
#pragma unroll
      for (int rr = 0; rr < RPT; ++rr) qv[rr] = simt_load4(qs + (grp + kGroups * rr) * LDQ + d);
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        const float4 kk = simt_load4(ks + (kx + TPR * j) * LD + d);  // (zeros where the chunk has no run)
#pragma unroll
        for (int rr = 0; rr < RPT; ++rr) {
          s[rr][j] = fmaf(qv[rr].x, kk.x, s[rr][j]);
          s[rr][j] = fmaf(qv[rr].y, kk.y, s[rr][j]);
          s[rr][j] = fmaf(qv[rr].z, kk.z, s[rr][j]);
          s[rr][j] = fmaf(qv[rr].w, kk.w, s[rr][j]);
        }
      }
    }
    // the mask and the rows' softmax state
#pragma unroll
    for (int rr = 0; rr < RPT; ++rr) {
      const int32_t row = grp + kGroups * rr, i = i0 + row;
      float tmax = -INFINITY;
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        const int32_t c = kx + TPR * j, in = c & (u - 1);
        const SimtSeg& e = sg[(TPR * j) >> ush];  // the same run for the whole block
        bool keep = TPR * j < n_keys;
        if (keep) {
          if (e.cls == kTileDiag) keep = e.j0 + in <= i;
          else if (e.cls == kTileGeneral) keep = (__ldg(masks + e.word + (row0 + row) * wpr + (in >> 5)) >> (in & 31)) & 1u;
        }
        s[rr][j] = keep ? s[rr][j] * scale_log2 : -INFINITY;
        tmax = fmaxf(tmax, s[rr][j]);
      }
#pragma unroll
      for (int off = TPR / 2; off >= 1; off >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, off));
      const float mn = fmaxf(m[rr], tmax), ref = mn == -INFINITY ? 0.f : mn;  // (nothing kept so far: all weights 0)
      const float alpha = exp2f(m[rr] - ref);                                // 0 when m was -inf
      float psum = 0.f;
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        const float p = exp2f(s[rr][j] - ref);  // exp2(-inf) = 0 for masked keys
        ps[row * LDP + kx + TPR * j] = p;
        psum += p;
      }
#pragma unroll
      for (int off = TPR / 2; off >= 1; off >>= 1) psum += __shfl_xor_sync(0xffffffffu, psum, off);
      l[rr] = l[rr] * alpha + psum;
      m[rr] = mn;
#pragma unroll
      for (int nd = 0; nd < ND; ++nd) {
        acc[rr][nd].x *= alpha; acc[rr][nd].y *= alpha; acc[rr][nd].z *= alpha; acc[rr][nd].w *= alpha;
      }
    }
    __syncwarp();  // a row's threads are one part of a warp
    // O += P V
#pragma unroll 4
    for (int kc = 0; kc < n_keys; kc += 4) {
      float4 p4[RPT];
#pragma unroll
      for (int rr = 0; rr < RPT; ++rr) p4[rr] = simt_load4(ps + (grp + kGroups * rr) * LDP + kc);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
#pragma unroll
        for (int nd = 0; nd < ND; ++nd) {
          const float4 vv = simt_load4(vs + (kc + x) * LD + 4 * kx + 4 * TPR * nd);
#pragma unroll
          for (int rr = 0; rr < RPT; ++rr) {
            const float p = x == 0 ? p4[rr].x : x == 1 ? p4[rr].y : x == 2 ? p4[rr].z : p4[rr].w;
            acc[rr][nd].x = fmaf(p, vv.x, acc[rr][nd].x);
            acc[rr][nd].y = fmaf(p, vv.y, acc[rr][nd].y);
            acc[rr][nd].z = fmaf(p, vv.z, acc[rr][nd].z);
            acc[rr][nd].w = fmaf(p, vv.w, acc[rr][nd].w);
          }
        }
      }
    }
    if (tid < spc) segs[(ch + 2) % 3][tid] = ahead;
    __syncthreads();  // the stage may be overwritten, and the runs after the next are known
  }
  bool any = false;
#pragma unroll
  for (int rr = 0; rr < RPT; ++rr) {
    const int32_t row = grp + kGroups * rr;
    if (row0 + row >= qt.q_rows) continue;
    const float inv = 1.f / l[rr];
    T* dst = o + ((int64_t)(qt.q_start + row0 + row) * n_q_heads + hq) * D + 4 * kx;
    float zero = 0.f;  // 0 unless a value is infinite or NaN
#pragma unroll
    for (int nd = 0; nd < ND; ++nd) {
      const float4 a = make_float4(acc[rr][nd].x * inv, acc[rr][nd].y * inv, acc[rr][nd].z * inv, acc[rr][nd].w * inv);
      simt_store4(dst + 4 * TPR * nd, a);
      zero = fmaf(a.x, 0.f, zero); zero = fmaf(a.y, 0.f, zero); zero = fmaf(a.z, 0.f, zero); zero = fmaf(a.w, 0.f, zero);
    }
    if (lse && kx == 0)
      lse[(int64_t)hq * hdr->total_tokens + qt.q_start + row0 + row] = (m[rr] + log2f(l[rr])) * 0.6931471805599453f;
    if (zero != 0.f) {
      any = true;
      atomicOr(&redo[row >> 5], 1u << (row & 31));
    }
  }
  if (!__syncthreads_or(any)) return;
  for (int32_t row = tid >> 5; row < R; row += kSimtThreads / 32)
    if ((redo[row >> 5] >> (row & 31)) & 1u)
      prefill_simt_row<T, D>(qs + row * LDQ, k, v, o, lse, plan, blockIdx.x / n_sub, row0 + row, n_q_heads, n_kv_heads, scale_log2);
}

template <typename T, int D, int TPR, int RPT>
static purekv_status launch(const PrefillArgs& a) {
  constexpr int NK = D > 128 ? 32 : 64;  // keys per chunk: two stages of K and V take at most 135 KB
  constexpr int R = kSimtThreads / TPR * RPT;
  auto kernel = prefill_simt_kernel<T, D, NK, TPR, RPT>;
  const size_t smem = SimtCfg<T, D, NK>::smem(R);
  static std::atomic<uint64_t> smem_allowed{0};
  const purekv_status st_smem = allow_max_dynamic_smem(kernel, smem_allowed);
  if (st_smem != PUREKV_OK) return st_smem;
  dim3 grid((unsigned)(a.info->n_qtiles * (a.info->tile_q / R)), (unsigned)a.n_q_heads);
  kernel<<<grid, kSimtThreads, smem, a.stream>>>((const T*)a.q, (const T*)a.k, (const T*)a.v, (T*)a.o, a.lse,
                                                 (const uint8_t*)a.plan, a.n_q_heads, a.n_kv_heads,
                                                 a.scale * 1.4426950408889634f);
  PK_CUDA(cudaGetLastError());
  return PUREKV_OK;
}

// Rows per CTA: the most that leave two CTAs per SM (and that the query tile and the registers take); a smaller job takes
// the fewest.
template <typename T, int D>
static purekv_status launch_rows(const PrefillArgs& a) {
  const int64_t rows = (int64_t)a.info->n_qtiles * a.info->tile_q * a.n_q_heads;
  const int32_t tq = a.info->tile_q;
  if constexpr (D <= 128)
    if (tq >= 64 && rows >= 64 * 2 * 148) return launch<T, D, 8, 4>(a);
  if (tq >= 32 && rows >= 32 * 2 * 148) return launch<T, D, 8, 2>(a);
  if constexpr (D >= 64)
    if (rows < 16 * 2 * 148) return launch<T, D, 16, 1>(a);
  return launch<T, D, 8, 1>(a);
}

purekv_status launch_prefill_simt(const PrefillArgs& a) {
  PK_REQUIRE(a.info->tile_q <= 64 && a.info->tile_q >= 16 && a.info->tile_q % 16 == 0 && a.info->tile_k <= 128,
             PUREKV_ERR_UNSUPPORTED, "CUDA-core prefill needs a plan with tile_q 16, 32 or 64");
  const bool bf = a.dtype == PUREKV_BF16;
  switch (a.head_dim) {
    case 32: return bf ? launch_rows<__nv_bfloat16, 32>(a) : launch_rows<float, 32>(a);
    case 64: return bf ? launch_rows<__nv_bfloat16, 64>(a) : launch_rows<float, 64>(a);
    case 128: return bf ? launch_rows<__nv_bfloat16, 128>(a) : launch_rows<float, 128>(a);
    case 256: return bf ? launch_rows<__nv_bfloat16, 256>(a) : launch_rows<float, 256>(a);
    default: break;
  }
  set_error("head_dim %d has no prefill kernel (supported: 32, 64, 128, 256)", a.head_dim);
  return PUREKV_ERR_UNSUPPORTED;
}

}  // namespace purekv
