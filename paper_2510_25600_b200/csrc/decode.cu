// purekv_decode_attention: one decoding step over the compacted cache of one layer (Sec. 3.1: later tokens attend
// to the compressed cache; the stage Table 3 times as decode latency).  Every request brings one new query per head;
// query head hq reads KV head hq / G of the request's kept rows.
//
// Split-KV, HBM bound: a CTA owns a chunk of one (request, KV head)'s kept keys and serves all G query heads of the
// group from one read of K and one of V.  bf16 runs on tensor cores (decode_cluster_kernel, further down); the kernel
// described next serves fp32.  Rows are 256 bytes (bf16 d = 128 or fp32 d = 64): a half-warp covers a
// row with one 16-byte load per lane, so a warp instruction fetches two rows.  Pass 1 forms the G logits of every
// key (q slices in registers; the 16 lanes' partial dot products are folded by a butterfly that halves the number of
// values per step) into shared memory; the chunk's maxima and exp2 weights are then taken once per element; pass 2
// streams V and accumulates G x d outputs in registers.  One chunk per (request, KV head): the CTA normalises and
// writes O itself; several: it leaves (unnormalised O, max, sum) per head and a second small kernel merges them.
#include <algorithm>

#include "cluster.cuh"
#include "common.cuh"

namespace purekv {

constexpr int kDecThreads = 128;
constexpr int kUnroll = 8;         // rows a half-warp has in flight
constexpr int kDecChunkMax = 512;  // keys per CTA: logits of 8 heads x 512 keys take 16 KB of shared memory

template <typename T>
struct Row16;  // the elements of one 16-byte chunk as fp32
template <>
struct Row16<float> {
  static constexpr int E = 4;
  static __device__ __forceinline__ void unpack(uint4 u, float (&f)[4]) {
    f[0] = __uint_as_float(u.x); f[1] = __uint_as_float(u.y); f[2] = __uint_as_float(u.z); f[3] = __uint_as_float(u.w);
  }
};
__device__ __forceinline__ float dec_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Folds v[0..N) of the 16 lanes of a half-warp: each step a lane hands half of its values to the partner across
// `mask` and adds the partner's other half, so the values halve while the lanes summed double.  Afterwards v[0] of
// lane ch is the full 16-lane sum for head ch >> (4 - log2 N).
template <int N>
__device__ __forceinline__ void fold16(float (&v)[N], int ch) {
  int mask = 8;
  int n = N;
#pragma unroll
  for (int step = 0; step < 4; ++step) {
    if (n > 1) {
      const int half = n >> 1;
      const bool up = (ch & mask) != 0;
#pragma unroll
      for (int i = 0; i < N / 2; ++i) {
        if (i < half) {
          const float send = up ? v[i] : v[i + half];
          const float keep = up ? v[i + half] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, mask);
        }
      }
      n = half;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], mask);
    }
    mask >>= 1;
  }
}

// grid (n_splits, H_kv, n_req), 128 threads.  part: [n_req][H][n_splits][D + 2] floats when n_splits > 1.
template <typename T, int GP>
__global__ void __launch_bounds__(kDecThreads) decode_partial_kernel(
    const uint4* __restrict__ q, const uint4* __restrict__ kc, const uint4* __restrict__ vc,
    const int32_t* __restrict__ cu_kept, int32_t n_q_heads, int32_t n_kv_heads, int32_t chunk, float scale_log2,
    T* __restrict__ o, float* __restrict__ lse, float* __restrict__ part, int32_t n_splits) {
  constexpr int E = Row16<T>::E, D = 16 * E;
  constexpr int kShift = GP == 8 ? 1 : GP == 4 ? 2 : GP == 2 ? 3 : 4;  // head of lane ch after fold16 = ch >> kShift
  __shared__ float s_sc[GP][kDecChunkMax];
  __shared__ float s_red[kDecThreads / 32][GP][D];
  __shared__ float s_m[GP], s_l[GP];

  const int32_t sp = blockIdx.x, g = blockIdx.y, r = blockIdx.z;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // the merge kernel may be placed meanwhile
  const int32_t G = n_q_heads / n_kv_heads;
  const int32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, hw = lane >> 4, ch = lane & 15;
  const int64_t j0 = (int64_t)cu_kept[r] + (int64_t)sp * chunk;
  const int32_t n = (int32_t)max((int64_t)0, min((int64_t)cu_kept[r + 1], j0 + chunk) - j0);

  // this lane's slice of the group's queries, already in log2 units
  float qf[GP][E];
#pragma unroll
  for (int h = 0; h < GP; ++h) {
    float t[E];
#pragma unroll
    for (int e = 0; e < E; ++e) t[e] = 0.f;
    if (h < G) Row16<T>::unpack(__ldg(q + ((int64_t)r * n_q_heads + g * G + h) * 16 + ch), t);
#pragma unroll
    for (int e = 0; e < E; ++e) qf[h][e] = t[e] * scale_log2;
  }

  // pass 1: logits.  kUnroll rows per half-warp are requested before the first is used (bytes in flight); the bound
  // is rounded up to a pair of rows so that both halves of a warp make the same trips (the fold shuffles).
  constexpr int kStride = (kDecThreads / 32) * 2;
  const int32_t n_up = (n + 1) & ~1;
  for (int32_t p = warp * 2 + hw; p < n_up; p += kStride * kUnroll) {
    uint4 raw[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      raw[u] = __ldg(kc + ((j0 + min(p + u * kStride, n - 1)) * n_kv_heads + g) * 16 + ch);
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int32_t pu = p + u * kStride;
      if (pu < n_up) {  // the same for every lane of the warp
        float kf[E];
        Row16<T>::unpack(raw[u], kf);
        float dot[GP];
#pragma unroll
        for (int h = 0; h < GP; ++h) {
          float a = 0.f;
#pragma unroll
          for (int e = 0; e < E; ++e) a = fmaf(qf[h][e], kf[e], a);
          dot[h] = a;
        }
        fold16<GP>(dot, ch);
        if ((ch & ((1 << kShift) - 1)) == 0 && pu < n) s_sc[ch >> kShift][pu] = dot[0];
      }
    }
  }
  __syncthreads();

  // per head: the chunk's maximum, then the weights 2^(s - max) in place and their sum (16 threads per head)
  {
    const int32_t h_t = tid >> 4, i0 = tid & 15;
    const int32_t h = min(h_t, GP - 1);  // surplus threads repeat the last head (whole warps stay in the shuffles)
    {
      float m = -INFINITY;
      for (int32_t i = i0; i < n; i += 16) m = fmaxf(m, s_sc[h][i]);
#pragma unroll
      for (int mask = 8; mask >= 1; mask >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, mask));
      float l = 0.f;
      for (int32_t i = i0; i < n; i += 16) {
        const float pw = dec_ex2(s_sc[h][i] - m);
        if (h_t < GP) s_sc[h][i] = pw;
        l += pw;
      }
#pragma unroll
      for (int mask = 8; mask >= 1; mask >>= 1) l += __shfl_xor_sync(0xffffffffu, l, mask);
      if (i0 == 0 && h_t < GP) {
        s_m[h] = m;
        s_l[h] = l;
      }
    }
  }
  __syncthreads();

  // pass 2: O += P V
  float acc[GP][E];
#pragma unroll
  for (int h = 0; h < GP; ++h)
#pragma unroll
    for (int e = 0; e < E; ++e) acc[h][e] = 0.f;
  for (int32_t p = warp * 2 + hw; p < n; p += kStride * kUnroll) {
    uint4 raw[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      raw[u] = __ldg(vc + ((j0 + min(p + u * kStride, n - 1)) * n_kv_heads + g) * 16 + ch);
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int32_t pu = p + u * kStride;
      if (pu < n) {
        float vf[E];
        Row16<T>::unpack(raw[u], vf);
#pragma unroll
        for (int h = 0; h < GP; ++h) {
          const float pw = s_sc[h][pu];
#pragma unroll
          for (int e = 0; e < E; ++e) acc[h][e] = fmaf(pw, vf[e], acc[h][e]);
        }
      }
    }
  }
  // the two half-warps, then the four warps
#pragma unroll
  for (int h = 0; h < GP; ++h)
#pragma unroll
    for (int e = 0; e < E; ++e) acc[h][e] += __shfl_xor_sync(0xffffffffu, acc[h][e], 16);
  if (hw == 0) {
#pragma unroll
    for (int h = 0; h < GP; ++h)
#pragma unroll
      for (int e = 0; e < E; ++e) s_red[warp][h][ch * E + e] = acc[h][e];
  }
  __syncthreads();
  for (int32_t x = tid; x < G * D; x += kDecThreads) {
    const int32_t h = x / D, c = x % D;
    const float a = (s_red[0][h][c] + s_red[1][h][c]) + (s_red[2][h][c] + s_red[3][h][c]);
    const int32_t hq = g * G + h;
    if (n_splits == 1) {
      const float l = s_l[h];
      o[((int64_t)r * n_q_heads + hq) * D + c] = (T)(l > 0.f ? a / l : 0.f);
      if (c == 0 && lse) lse[(int64_t)r * n_q_heads + hq] = l > 0.f ? (s_m[h] + log2f(l)) * 0.6931471805599453f : -INFINITY;
    } else {
      float* dst = part + (((int64_t)r * n_q_heads + hq) * n_splits + sp) * (D + 2);
      dst[c] = a;
      if (c == 0) {
        dst[D] = s_m[h];
        dst[D + 1] = s_l[h];
      }
    }
  }
}

// ---- bf16, d = 128 on tensor cores ---------------------------------------------------------------------------
__device__ __forceinline__ void dec_mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t dec_pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// A row's reference maximum moves when a logit exceeds it by this (log2).  At 0 it is the largest logit so far, and the heaviest
// weights are powers of two, exact in bf16: error against 64 bits 1.87e-3 of the norm of the result for 8 requests of 5000 rows, 1.90
// for 64 of 700, 1.79 for one of 3000 with 16 heads per KV head; at 8, 2.29, 2.31 and 1.97e-3.  (The chunk kernel of before, at 8 but
// with a single trip per warp for short requests: 2.28, 2.25 and 1.77.)  Up to 5 % slower with 16 heads per KV head, otherwise equal.
constexpr float kDecRescale = 0.f;

// One launch.  A cluster of C CTAs (grid (C, H_kv, n_req)) owns one (request, KV head); CTA `rank` takes the rank-th share
// of the request's rows, so ragged requests are cut evenly, and the CTAs' partial results meet in distributed shared
// memory instead of in a workspace that a second kernel merges (chunk kernel + merge kernel before: 12.0 us for one
// request of 1664 rows with 28 / 4 heads, now 5.5; 128 requests of 2900-5100 rows 214 us = 5.0 TB/s, now 167 us = 6.4 TB/s in a row
// and 5.6 TB/s with a cold L2).
// Bound by HBM for large batches and by a chain of latencies for small ones: launch (1 us behind a programmatic
// predecessor), the offsets, the rows, the products, one cluster barrier.
// A warp takes 16 keys per trip: with mma.sync the group's heads are the 16 rows of an m16n8k16 tile (M = 16 is far below a
// tcgen05 tile's 128 rows), S = Q K^T is two n8 tiles, and the softmax on their accumulators leaves the A operand of
// O += P V.  Each warp streams its trips through a private ring of ST stages with cp.async (rows padded to 272 bytes, so
// that ldmatrix reads eight rows without bank conflicts): two further trips are in flight while one is multiplied, and no
// warp waits for another before the end.
constexpr int kClRow = 272;                     // bytes of a row in shared memory
constexpr int kClStageBytes = 2 * 16 * kClRow;  // 16 K rows, then 16 V rows
constexpr int kClMax = 16;                      // CTAs per cluster

// Dynamic shared memory of one warp: its ring, over which its partial results (rows of 128 + 8 floats) are laid at the end.
template <int RW, int ST>
__host__ __device__ constexpr int cl_warp_bytes() {
  return ST * kClStageBytes > 8 * RW * (128 + 8) * 4 ? ST * kClStageBytes : 8 * RW * (128 + 8) * 4;
}

__device__ __forceinline__ void dec_ldsm(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void dec_ldsm_t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint32_t dec_mapa(const void* local, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
  return a;
}

// RW: row groups of eight heads in use (1: G <= 8, 2: G <= 16); W warps; ST stages of each warp's ring.
template <int RW, int W, int ST>
__global__ void __launch_bounds__(W * 32, (ST == 1 ? 12 : 8) / W) decode_cluster_kernel(
    const uint4* __restrict__ q, const uint4* __restrict__ kc, const uint4* __restrict__ vc,
    const int32_t* __restrict__ cu_kept, int32_t n_q_heads, int32_t n_kv_heads, float scale_log2,
    __nv_bfloat16* __restrict__ o, float* __restrict__ lse) {
  constexpr int D = 128, R = 8 * RW, kThreads = W * 32, kWarpBytes = cl_warp_bytes<RW, ST>();
  extern __shared__ __align__(16) uint8_t cl_smem[];
  __shared__ float s_ml[W][R][2];
  __shared__ __align__(16) float s_part[R * D];       // what the cluster's CTAs send this one: [source][head][its columns]
  __shared__ __align__(8) float s_pml[kClMax][R][2];  // every CTA's (reference, sum) per head

  const uint32_t C = gridDim.x, rank = blockIdx.x;  // the cluster spans the grid's x dimension
  const int32_t g = blockIdx.y, r = blockIdx.z;
  const int32_t G = n_q_heads / n_kv_heads;
  const int32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g8 = lane >> 2, t = lane & 3;
  // The next kernel of the stream may be placed meanwhile (the calls of consecutive layers follow one another); what the
  // previous one wrote is complete and visible behind the wait.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (C > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // "started": awaited before the sends
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t kept0 = cu_kept[r];
  const int32_t n_all = cu_kept[r + 1] - (int32_t)kept0;
  const int32_t share = ((n_all + (int32_t)C - 1) / (int32_t)C + 15) & ~15;
  const int64_t j0 = kept0 + (int64_t)rank * share;
  const int32_t n = max(0, min(n_all - (int32_t)rank * share, share));

  // 16-row trip `trip` of this warp into stage trip % ST: a warp request covers two rows; rows past the end repeat the
  // last one (weight 0)
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(cl_smem) + (uint32_t)warp * kWarpBytes;
  const int64_t row_stride = (int64_t)n_kv_heads * 16;  // 16-byte words
  const int32_t n_trips = n > warp * 16 ? (n - warp * 16 + W * 16 - 1) / (W * 16) : 0;
  auto fetch = [&](int32_t trip) {
    if (trip < n_trips) {
      const int32_t k0 = warp * 16 + trip * (W * 16);
      const uint32_t dst = ring + (uint32_t)(trip % ST) * kClStageBytes + (uint32_t)(lane >> 4) * kClRow + (lane & 15) * 16;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int64_t src = (j0 + min(k0 + 2 * i + (lane >> 4), n - 1)) * row_stride + g * 16 + (lane & 15);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 2 * i * kClRow), "l"(kc + src) : "memory");
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int64_t src = (j0 + min(k0 + 2 * i + (lane >> 4), n - 1)) * row_stride + g * 16 + (lane & 15);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (16 + 2 * i) * kClRow), "l"(vc + src) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");  // (empty past the end: the group count stays in step)
  };
#pragma unroll
  for (int s = 0; s < (ST > 1 ? ST - 1 : 1); ++s) fetch(s);

  // A fragments of Q: rows g8 and g8 + 8 (heads of the group; rows past G are zero)
  uint32_t qa[8][4];
  {
    const uint32_t* q32 = reinterpret_cast<const uint32_t*>(q) + ((int64_t)r * n_q_heads + g * G) * 64 + t;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      qa[ks][0] = g8 < G ? __ldg(q32 + g8 * 64 + ks * 8) : 0u;
      qa[ks][2] = g8 < G ? __ldg(q32 + g8 * 64 + ks * 8 + 4) : 0u;
      qa[ks][1] = RW == 2 && g8 + 8 < G ? __ldg(q32 + (g8 + 8) * 64 + ks * 8) : 0u;
      qa[ks][3] = RW == 2 && g8 + 8 < G ? __ldg(q32 + (g8 + 8) * 64 + ks * 8 + 4) : 0u;
    }
  }
  float oacc[16][4];
#pragma unroll
  for (int nt = 0; nt < 16; ++nt)
#pragma unroll
    for (int x = 0; x < 4; ++x) oacc[nt][x] = 0.f;
  float m_ref[2] = {-INFINITY, -INFINITY}, l_part[2] = {0.f, 0.f};  // rows g8 and g8 + 8

  // ldmatrix: lane l addresses row l % 8 (+ 8 for the third and fourth matrix of K, the second and fourth of V)
  const uint32_t k_off = (uint32_t)((lane & 7) + 8 * (lane >> 4)) * kClRow + ((lane >> 3) & 1) * 16;
  const uint32_t v_off = (uint32_t)(16 + (lane & 7) + 8 * ((lane >> 3) & 1)) * kClRow + (lane >> 4) * 16;
  for (int32_t trip = 0; trip < n_trips; ++trip) {
    const int32_t k0 = warp * 16 + trip * (W * 16);
    if constexpr (ST > 1) fetch(trip + ST - 1);
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 1) : "memory");
    __syncwarp();
    const uint32_t st = ring + (uint32_t)(trip % ST) * kClStageBytes;
    float sc[2][4];
#pragma unroll
    for (int tl = 0; tl < 2; ++tl)
#pragma unroll
      for (int x = 0; x < 4; ++x) sc[tl][x] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      uint32_t b[4];
      dec_ldsm(st + k_off + ks * 32, b);
      dec_mma(sc[0], qa[ks], b[0], b[1]);
      dec_mma(sc[1], qa[ks], b[2], b[3]);
    }
    // log2 units; keys past the end weigh nothing.  sc[tl][0..1]: row g8, keys 2t, 2t+1 of tile tl; [2..3]: row g8 + 8
#pragma unroll
    for (int tl = 0; tl < 2; ++tl)
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int32_t key = k0 + 8 * tl + 2 * t + (x & 1);
        sc[tl][x] = key < n ? sc[tl][x] * scale_log2 : -INFINITY;
      }
    uint32_t pa[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int rw = 0; rw < RW; ++rw) {
      float mx = fmaxf(fmaxf(sc[0][2 * rw], sc[0][2 * rw + 1]), fmaxf(sc[1][2 * rw], sc[1][2 * rw + 1]));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      if (mx > m_ref[rw] + kDecRescale) {  // the same for the four threads of the row
        const float alpha = m_ref[rw] == -INFINITY ? 0.f : dec_ex2(m_ref[rw] - mx);
        l_part[rw] *= alpha;
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) {
          oacc[nt][2 * rw] *= alpha;
          oacc[nt][2 * rw + 1] *= alpha;
        }
        m_ref[rw] = mx;
      }
      const float p00 = dec_ex2(sc[0][2 * rw] - m_ref[rw]), p01 = dec_ex2(sc[0][2 * rw + 1] - m_ref[rw]);
      const float p10 = dec_ex2(sc[1][2 * rw] - m_ref[rw]), p11 = dec_ex2(sc[1][2 * rw + 1] - m_ref[rw]);
      l_part[rw] += (p00 + p01) + (p10 + p11);
      pa[rw] = dec_pack_bf16(p00, p01);      // k slots 2t, 2t+1: keys 2t, 2t+1 of tile 0
      pa[2 + rw] = dec_pack_bf16(p10, p11);  // k slots 2t+8, 2t+9: the same keys of tile 1
    }
#pragma unroll
    for (int nt = 0; nt < 16; nt += 2) {
      uint32_t b[4];
      dec_ldsm_t(st + v_off + nt * 16, b);
      dec_mma(oacc[nt], pa, b[0], b[1]);
      dec_mma(oacc[nt + 1], pa, b[2], b[3]);
    }
    __syncwarp();  // every lane has read the stage before the next fetch overwrites it
    if constexpr (ST == 1) fetch(trip + 1);
  }

  // the warps' results side by side in shared memory (a warp's over its own ring, which nobody else reads)
#pragma unroll
  for (int rw = 0; rw < RW; ++rw) {
    l_part[rw] += __shfl_xor_sync(0xffffffffu, l_part[rw], 1);
    l_part[rw] += __shfl_xor_sync(0xffffffffu, l_part[rw], 2);
    if (t == 0) {
      s_ml[warp][g8 + 8 * rw][0] = m_ref[rw];
      s_ml[warp][g8 + 8 * rw][1] = l_part[rw];
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  constexpr int LD = D + 8;  // rows start eight banks apart: the 8-byte stores of a half-warp do not collide
  {
    float* s_o = reinterpret_cast<float*>(cl_smem + warp * kWarpBytes);  // [R][LD]
#pragma unroll
    for (int nt = 0; nt < 16; ++nt)
#pragma unroll
      for (int rw = 0; rw < RW; ++rw)
        *reinterpret_cast<float2*>(s_o + (g8 + 8 * rw) * LD + nt * 8 + 2 * t) = make_float2(oacc[nt][2 * rw], oacc[nt][2 * rw + 1]);
  }
  __syncthreads();
  if (C > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  const int32_t cols = D / (int32_t)C;  // columns of every head that each CTA of the cluster finishes
  // one thread per four columns of a head
  for (int32_t x = tid; x < G * (D / 4); x += kThreads) {
    const int32_t h = x / (D / 4), c = 4 * (x % (D / 4));
    float m_w[W], m_all = -INFINITY;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      m_w[w] = s_ml[w][h][1] > 0.f ? s_ml[w][h][0] : -INFINITY;
      m_all = fmaxf(m_all, m_w[w]);
    }
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    float l = 0.f;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const float wgt = m_w[w] > -INFINITY ? dec_ex2(m_w[w] - m_all) : 0.f;
      const float4 v4 = *reinterpret_cast<const float4*>(cl_smem + w * kWarpBytes + (h * LD + c) * 4);
      a.x = fmaf(wgt, v4.x, a.x); a.y = fmaf(wgt, v4.y, a.y); a.z = fmaf(wgt, v4.z, a.z); a.w = fmaf(wgt, v4.w, a.w);
      l = fmaf(wgt, s_ml[w][h][1], l);
    }
    if (C == 1) {
      const int64_t hq = (int64_t)r * n_q_heads + g * G + h;
      const float inv = l > 0.f ? 1.f / l : 0.f;
      *reinterpret_cast<uint2*>(o + hq * D + c) = make_uint2(dec_pack_bf16(a.x * inv, a.y * inv), dec_pack_bf16(a.z * inv, a.w * inv));
      if (c == 0 && lse) lse[hq] = l > 0.f ? (m_all + log2f(l)) * 0.6931471805599453f : -INFINITY;
    } else {
      const uint32_t to = (uint32_t)(c / cols);
      asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dec_mapa(s_part + ((int32_t)rank * G + h) * cols + c % cols, to)),
                   "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w) : "memory");
      if (c % cols == 0)
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dec_mapa(s_pml[rank][h], to)), "f"(m_all), "f"(l) : "memory");
    }
  }
  if (C == 1) return;
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  // four threads per output value, each over every fourth CTA's share (G * cols * 4 is a multiple of 32: whole warps)
  const int32_t part = tid & 3;
  for (int32_t x = tid; x < G * cols * 4; x += kThreads) {
    const int32_t h = (x >> 2) / cols, c = (x >> 2) % cols;
    float m_all = -INFINITY, mi[kClMax / 4], li[kClMax / 4];
#pragma unroll
    for (int k = 0; k < kClMax / 4; ++k) {
      const int32_t i = part + 4 * k;
      const float2 ml = i < (int32_t)C ? *reinterpret_cast<const float2*>(s_pml[i][h]) : make_float2(0.f, 0.f);
      li[k] = ml.y;
      mi[k] = ml.y > 0.f ? ml.x : -INFINITY;
      m_all = fmaxf(m_all, mi[k]);
    }
    m_all = fmaxf(m_all, __shfl_xor_sync(0xffffffffu, m_all, 1));
    m_all = fmaxf(m_all, __shfl_xor_sync(0xffffffffu, m_all, 2));
    float a = 0.f, l = 0.f;
#pragma unroll
    for (int k = 0; k < kClMax / 4; ++k) {
      if (mi[k] > -INFINITY) {
        const float wgt = dec_ex2(mi[k] - m_all);
        a = fmaf(wgt, s_part[((part + 4 * k) * G + h) * cols + c], a);
        l = fmaf(wgt, li[k], l);
      }
    }
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    if (part == 0) {
      const int64_t hq = (int64_t)r * n_q_heads + g * G + h;
      o[hq * D + (int32_t)rank * cols + c] = __float2bfloat16(l > 0.f ? a / l : 0.f);
      if (rank == 0 && c == 0 && lse) lse[hq] = l > 0.f ? (m_all + log2f(l)) * 0.6931471805599453f : -INFINITY;
    }
  }
}

// fp32: grid (H, n_req), D threads: merges the chunks' partial results of one (request, head).  The
// chunks' weights 2^(m_s - m) are formed once, 128 chunks at a time, in shared memory; thread c then sums column c
// with independent loads.
__global__ void decode_merge_kernel(const float* __restrict__ part, int32_t n_q_heads, int32_t n_splits, int32_t D,
                                    float* __restrict__ o, float* __restrict__ lse) {
  __shared__ float s_w[128];
  __shared__ float s_red[4];
  __shared__ float s_m;
  const int32_t hq = blockIdx.x, r = blockIdx.y, c = threadIdx.x, lane = c & 31, warp = c >> 5;
  const int32_t n_warps = (int32_t)blockDim.x >> 5;
  // launched with programmatic stream serialization: placed while the chunk kernel still runs, its partial results
  // are complete and visible from here on
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const float* src = part + ((int64_t)r * n_q_heads + hq) * n_splits * (D + 2);
  // the largest chunk maximum among chunks that hold anything
  float m = -INFINITY;
  for (int32_t s = c; s < n_splits; s += (int32_t)blockDim.x)
    if (src[(int64_t)s * (D + 2) + D + 1] > 0.f) m = fmaxf(m, src[(int64_t)s * (D + 2) + D]);
#pragma unroll
  for (int mask = 16; mask >= 1; mask >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, mask));
  if (lane == 0) s_red[warp] = m;
  __syncthreads();
  if (c == 0) {
    float mm = s_red[0];
    for (int32_t w = 1; w < n_warps; ++w) mm = fmaxf(mm, s_red[w]);
    s_m = mm;
  }
  __syncthreads();
  const float m_all = s_m;
  float a = 0.f, l = 0.f;
  for (int32_t s0 = 0; s0 < n_splits; s0 += 128) {
    const int32_t ns = min(128, n_splits - s0);
    __syncthreads();
    for (int32_t i = c; i < ns; i += (int32_t)blockDim.x) {
      const float ls = src[(int64_t)(s0 + i) * (D + 2) + D + 1];
      const float wgt = ls > 0.f ? dec_ex2(src[(int64_t)(s0 + i) * (D + 2) + D] - m_all) : 0.f;
      s_w[i] = wgt;
      l = fmaf(wgt, ls, l);  // this thread's share of the row sum
    }
    __syncthreads();
    const float* col = src + (int64_t)s0 * (D + 2) + c;
    int32_t i = 0;
    for (; i + 4 <= ns; i += 4) {
      const float v0 = col[(int64_t)i * (D + 2)], v1 = col[(int64_t)(i + 1) * (D + 2)];
      const float v2 = col[(int64_t)(i + 2) * (D + 2)], v3 = col[(int64_t)(i + 3) * (D + 2)];
      a = fmaf(s_w[i], v0, a); a = fmaf(s_w[i + 1], v1, a); a = fmaf(s_w[i + 2], v2, a); a = fmaf(s_w[i + 3], v3, a);
    }
    for (; i < ns; ++i) a = fmaf(s_w[i], col[(int64_t)i * (D + 2)], a);
  }
#pragma unroll
  for (int mask = 16; mask >= 1; mask >>= 1) l += __shfl_xor_sync(0xffffffffu, l, mask);
  __syncthreads();
  if (lane == 0) s_red[warp] = l;
  __syncthreads();
  l = 0.f;
  for (int32_t w = 0; w < n_warps; ++w) l += s_red[w];
  o[((int64_t)r * n_q_heads + hq) * D + c] = l > 0.f ? a / l : 0.f;
  if (c == 0 && lse) lse[(int64_t)r * n_q_heads + hq] = l > 0.f ? (m_all + log2f(l)) * 0.6931471805599453f : -INFINITY;
}

// keys per CTA and CTAs per (request, KV head): enough CTAs for two per SM when the batch alone does not give them
// (more and shorter chunks were measured slower: the merge kernel walks a head's chunks one after the other)
static void decode_split(int32_t n_req, int32_t max_kept, int32_t n_kv_heads, int32_t* chunk, int32_t* n_splits) {
  const int64_t base = std::max<int64_t>(1, (int64_t)n_req * n_kv_heads);
  const int64_t want = std::max<int64_t>(1, (2 * 148 + base - 1) / base);
  int64_t c = (std::max(1, max_kept) + want - 1) / want;
  c = std::min<int64_t>(kDecChunkMax, std::max<int64_t>(64, c));
  c = (c + 7) / 8 * 8;
  *chunk = (int32_t)c;
  *n_splits = (int32_t)((std::max(1, max_kept) + c - 1) / c);
}

template <int RW, int W, int ST>
static purekv_status launch_cluster_as(int32_t cl, cudaStream_t sm, const void* q, const void* kc, const void* vc,
                                       const int32_t* cu_kept, int32_t n_req, int32_t H, int32_t Hkv, float scale_log2,
                                       void* o, float* lse) {
  auto kernel = decode_cluster_kernel<RW, W, ST>;
  static std::atomic<uint64_t> smem_allowed{0}, wide_allowed{0};
  const purekv_status st = allow_max_dynamic_smem(kernel, smem_allowed);
  if (st != PUREKV_OK) return st;
  if (cl > 8) {  // clusters of more than eight CTAs are opt-in, once per device
    int dev = -1;
    PK_CUDA(cudaGetDevice(&dev));
    if (!(wide_allowed.load(std::memory_order_acquire) & (1ull << dev))) {
      PK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
      wide_allowed.fetch_or(1ull << dev, std::memory_order_release);
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(W * 32);
  cfg.dynamicSmemBytes = (size_t)W * cl_warp_bytes<RW, ST>();
  cfg.stream = sm;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see griddepcontrol in the kernel
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  auto set_size = [&](int32_t c) {
    cfg.gridDim = dim3((unsigned)c, (unsigned)Hkv, (unsigned)n_req);
    attr[1].val.clusterDim.x = (unsigned)c;
  };
  set_size(cluster_that_fits(cl, [&](int32_t c) {
    set_size(c);
    return clusters_at_once(kernel, cfg);
  }));
  PK_CUDA(cudaLaunchKernelEx(&cfg, kernel, (const uint4*)q, (const uint4*)kc, (const uint4*)vc, cu_kept, H, Hkv, scale_log2,
                             (__nv_bfloat16*)o, lse));
  return PUREKV_OK;
}

template <int RW>
static purekv_status launch_cluster(int32_t max_kept, int64_t total_kept, cudaStream_t sm, const void* q, const void* kc,
                                    const void* vc, const int32_t* cu_kept, int32_t n_req, int32_t H, int32_t Hkv,
                                    float scale_log2, void* o, float* lse) {
  const int64_t base = (int64_t)n_req * Hkv;
  const bool skewed = max_kept > 256 && 2 * (int64_t)max_kept * n_req > 3 * total_kept;
  int32_t cl = 1;  // CTAs per cluster
  if (skewed) {
    // One long request among short ones: more CTAs each shorten what the last one streams, and the short requests' clusters
    // take turns on the GPU.  Times in ns as measured with an SM per CTA: 4 us for a cluster that has little to do, 6.9 ns a
    // row for a CTA that streams among idle ones, 6.3 TB/s for all; so many clusters fit at once.  (Chosen by this rule against
    // the one for even batches, 28 / 4 heads: 20 000 rows among 63 x 100: 40 against 132 us; 60 000 among 7 x 100: 35 against
    // 105; 4 x 30 000 among 60 x 1000: 81 against 202; 64 x 300-9000 at random: 106 either way.)
    const int32_t at_once[5] = {148, 74, 33, 15, 7};
    double best = 0.;
    for (int32_t i = 0; i < 5; ++i) {
      const int32_t c = 1 << i;
      const double row = std::max(6.9, 0.0813 * (double)(std::min<int64_t>(base, at_once[i]) * c));
      const double waves = (double)((base + at_once[i] - 1) / at_once[i]);
      const double t = std::max(waves * (4000. + (double)total_kept / n_req / c * row), 4000. + (double)max_kept / c * 6.9);
      if (i == 0 || t < best) { best = t; cl = c; }
    }
  } else if (max_kept > 256) {
    // Even batches, measured over 1-256 requests of 1-500 000 rows: shares of down to 64 rows pay (256 rows are two trips of one
    // CTA's eight warps, 4.9 us, and a cluster costs 1 us), as long as every CTA finds an SM of its own -- 128 CTAs for
    // clusters of up to four, 64 beyond (clusters of 8 or 16 CTAs with all of an SM's memory do not fill the GPCs: two
    // requests, 4 KV heads, 1664 rows: 7.2 us as 8 clusters of 8, 11.5 as 8 of 16).  Where each CTA still has thousands of rows
    // to stream, up to the 15 or 7 such clusters that fit at once (three requests of 60 000 rows, 4 KV heads: 105 -> 65 us).
    auto room = [&](int32_t c) {
      if (c < 8) return base * c <= 128;
      return base * c <= 64 || (max_kept > 4096 * (c / 2) && base <= (c == 8 ? 15 : 7));
    };
    while (cl < kClMax && max_kept > 64 * cl && room(2 * cl)) cl *= 2;
  }
  const int32_t share = (max_kept + cl - 1) / cl;
  // Eight warps and the SM to themselves for CTAs that are alone on it (four requests of 20 000 rows: 41 against 47 us; one of
  // 500, 16 heads per KV head: 6.4 against 7.7) or stream long shares (128 x 5000 rows: 167 against 174 us); otherwise two CTAs
  // of four warps, so that one streams while the other starts or ends (128 requests of up to 700 rows: 39 against 52 us).  One
  // stage when a share is a single trip.
  if (skewed || base * cl <= 148 || share > 2048)
    return share <= 128 ? launch_cluster_as<RW, 8, 1>(cl, sm, q, kc, vc, cu_kept, n_req, H, Hkv, scale_log2, o, lse)
                        : launch_cluster_as<RW, 8, 3>(cl, sm, q, kc, vc, cu_kept, n_req, H, Hkv, scale_log2, o, lse);
  return share <= 64 ? launch_cluster_as<RW, 4, 1>(cl, sm, q, kc, vc, cu_kept, n_req, H, Hkv, scale_log2, o, lse)
                     : launch_cluster_as<RW, 4, 3>(cl, sm, q, kc, vc, cu_kept, n_req, H, Hkv, scale_log2, o, lse);
}

template <typename T, int GP>
static void launch_decode(dim3 grid, cudaStream_t sm, const void* q, const void* kc, const void* vc, const int32_t* cu_kept,
                          int32_t H, int32_t Hkv, int32_t chunk, float scale_log2, void* o, float* lse, float* part,
                          int32_t n_splits) {
  decode_partial_kernel<T, GP><<<grid, kDecThreads, 0, sm>>>((const uint4*)q, (const uint4*)kc, (const uint4*)vc, cu_kept, H,
                                                            Hkv, chunk, scale_log2, (T*)o, lse, part, n_splits);
}

}  // namespace purekv

using namespace purekv;

extern "C" {

size_t purekv_decode_ws_bytes(int32_t n_req, int32_t max_kept, int32_t n_q_heads, int32_t n_kv_heads, int32_t head_dim) {
  if (n_req <= 0 || max_kept <= 0 || n_q_heads <= 0 || n_kv_heads <= 0 || head_dim <= 0) return 0;
  int32_t chunk, n_splits;
  decode_split(n_req, max_kept, n_kv_heads, &chunk, &n_splits);
  if (n_splits == 1) return 0;
  return (size_t)n_req * n_q_heads * n_splits * (head_dim + 2) * sizeof(float) + 256;
}

purekv_status purekv_decode_attention(const void* q, const void* k_cache, const void* v_cache, void* o, float* lse,
                                      const int32_t* cu_kept, const int32_t* h_cu_kept, int32_t n_req, int32_t n_q_heads,
                                      int32_t n_kv_heads, int32_t head_dim, purekv_dtype dtype, float softmax_scale,
                                      void* ws, size_t ws_bytes, void* stream) {
  PK_REQUIRE(n_req >= 0 && h_cu_kept, PUREKV_ERR_INVALID_ARG, "purekv_decode_attention: bad batch");
  PK_REQUIRE(n_q_heads > 0 && n_kv_heads > 0 && n_q_heads % n_kv_heads == 0, PUREKV_ERR_INVALID_ARG,
             "purekv_decode_attention: n_q_heads must be a positive multiple of n_kv_heads");
  PK_REQUIRE(dtype == PUREKV_BF16 || dtype == PUREKV_FP32, PUREKV_ERR_INVALID_ARG, "purekv_decode_attention: bad dtype");
  const int32_t G = n_q_heads / n_kv_heads;
  PK_REQUIRE((dtype == PUREKV_BF16 && head_dim == 128) || (dtype == PUREKV_FP32 && head_dim == 64), PUREKV_ERR_UNSUPPORTED,
             "purekv_decode_attention: rows must be 256 bytes (bf16 with head_dim 128, or fp32 with head_dim 64)");
  PK_REQUIRE(G <= (dtype == PUREKV_BF16 ? 16 : 8), PUREKV_ERR_UNSUPPORTED,
             "purekv_decode_attention: at most 16 (bf16) or 8 (fp32) query heads per KV head");
  if (n_req == 0) return PUREKV_OK;
  int32_t max_kept = 0;
  PK_REQUIRE(h_cu_kept[0] == 0, PUREKV_ERR_INVALID_ARG, "purekv_decode_attention: cu_kept must start at 0");
  for (int32_t r = 0; r < n_req; ++r) {
    PK_REQUIRE(h_cu_kept[r + 1] >= h_cu_kept[r], PUREKV_ERR_INVALID_ARG, "purekv_decode_attention: cu_kept must not decrease");
    max_kept = std::max(max_kept, h_cu_kept[r + 1] - h_cu_kept[r]);
  }
  PK_REQUIRE(q && o && cu_kept, PUREKV_ERR_INVALID_ARG, "purekv_decode_attention: null pointer");
  PK_REQUIRE(h_cu_kept[n_req] == 0 || (k_cache && v_cache), PUREKV_ERR_INVALID_ARG, "purekv_decode_attention: null cache");
  PK_REQUIRE(((uintptr_t)q | (uintptr_t)k_cache | (uintptr_t)v_cache | (uintptr_t)o) % 16 == 0, PUREKV_ERR_INVALID_ARG,
             "purekv_decode_attention: pointers must be 16-byte aligned");
  const float scale = softmax_scale > 0.f ? softmax_scale : 1.f / sqrtf((float)head_dim);
  const float scale_log2 = scale * 1.4426950408889634f;
  cudaStream_t sm = (cudaStream_t)stream;
  PK_REQUIRE(n_kv_heads <= 65535 && n_req <= 65535, PUREKV_ERR_UNSUPPORTED, "too many heads or requests");
  if (dtype == PUREKV_BF16)
    return G <= 8 ? launch_cluster<1>(max_kept, h_cu_kept[n_req], sm, q, k_cache, v_cache, cu_kept, n_req, n_q_heads, n_kv_heads, scale_log2, o, lse)
                  : launch_cluster<2>(max_kept, h_cu_kept[n_req], sm, q, k_cache, v_cache, cu_kept, n_req, n_q_heads, n_kv_heads, scale_log2, o, lse);
  int32_t chunk, n_splits;
  decode_split(n_req, max_kept, n_kv_heads, &chunk, &n_splits);
  float* part = nullptr;
  if (n_splits > 1) {
    PK_REQUIRE(ws && ws_bytes >= purekv_decode_ws_bytes(n_req, max_kept, n_q_heads, n_kv_heads, head_dim), PUREKV_ERR_WORKSPACE,
               "purekv_decode_attention: workspace of %zu bytes is too small", ws_bytes);
    part = (float*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
  }
  dim3 grid((unsigned)n_splits, (unsigned)n_kv_heads, (unsigned)n_req);
  const int GP = G <= 1 ? 1 : G <= 2 ? 2 : G <= 4 ? 4 : 8;
#define PK_DECODE(T)                                                                                                     \
  switch (GP) {                                                                                                          \
    case 1: launch_decode<T, 1>(grid, sm, q, k_cache, v_cache, cu_kept, n_q_heads, n_kv_heads, chunk, scale_log2, o, lse, part, n_splits); break; \
    case 2: launch_decode<T, 2>(grid, sm, q, k_cache, v_cache, cu_kept, n_q_heads, n_kv_heads, chunk, scale_log2, o, lse, part, n_splits); break; \
    case 4: launch_decode<T, 4>(grid, sm, q, k_cache, v_cache, cu_kept, n_q_heads, n_kv_heads, chunk, scale_log2, o, lse, part, n_splits); break; \
    default: launch_decode<T, 8>(grid, sm, q, k_cache, v_cache, cu_kept, n_q_heads, n_kv_heads, chunk, scale_log2, o, lse, part, n_splits); break; \
  }
  PK_DECODE(float)
#undef PK_DECODE
  PK_CUDA(cudaGetLastError());
  if (n_splits > 1) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_q_heads, (unsigned)n_req);
    cfg.blockDim = dim3((unsigned)head_dim);
    cfg.stream = sm;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see griddepcontrol in the kernels
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const float* part_c = part;
    PK_CUDA(cudaLaunchKernelEx(&cfg, decode_merge_kernel, part_c, n_q_heads, n_splits, head_dim, (float*)o, lse));
    PK_CUDA(cudaGetLastError());
  }
  return PUREKV_OK;
}

}  // extern "C"
