// purekv_lowlayer_score: window attention scores of the low layer (Eq. 1-2).
//
// For each request and KV head g the G*w query rows of the recent window (G query heads of
// the group x w positions) are stacked; row (hl, iw) is query head g*G+hl at position
// i = l-w+iw.  Pass 1 streams the keys once per 32-row block and keeps a running
// (max, sum of exponentials) per row -> log-sum-exp over all causal keys j <= i (Eq. 1's row
// normaliser).  Pass 2 gives each CTA one block of 64 non-recent keys: it recomputes the
// logits of every stacked row against those keys, forms exp(s - lse) and sums down the rows
// (Eq. 2), so the attention matrix never leaves the SM and no atomics are needed.
// Logits are fp32 FMA chains over exact products; exponentials use exp2f.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "cluster.cuh"
#include "common.cuh"

namespace purekv {

// Scratch of purekv_lowlayer_score_noalloc: the window rows' log-sum-exp values and their per-key-block
// parts, i.e. what purekv_lowlayer_score keeps in its workspace.  It lives in the library's device image, so every GPU that
// loads the library holds this 1 MiB until the process exits.  Host code may not pass this name to
// a kernel (on the host it is only a stand-in for the symbol); the device address comes from
// cudaGetSymbolAddress, looked up once per device.
constexpr size_t kNoallocScoreFloats = PUREKV_NOALLOC_SCORE_MAX_ROWS;
static __device__ __align__(256) float g_noalloc_score_scratch[kNoallocScoreFloats + 64];  // + the 256 bytes of alignment slack the workspace rule asks for

constexpr int kRB = 32;        // stacked rows per block
constexpr int kKB = 64;        // keys per block
constexpr int kThreads = 256;  // thread (ty, tx): rows 2*ty, 2*ty+1; keys tx, tx+16, tx+32, tx+48

template <typename T>
__device__ __forceinline__ void load_row_f32(float* dst, const T* src, int d, int lane_in_group, int group_size) {
  for (int c = lane_in_group; c < d; c += group_size) dst[c] = to_f32(src[c]);
}

// s[a][b] = <q row 2*ty+a, key tx+16*b> over d, both tiles in shared memory with row stride ld.
__device__ __forceinline__ void tile_dots(const float* qs, const float* ks, int d, int ld, int ty, int tx,
                                          float s[2][4]) {
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) s[a][b] = 0.f;
  const float4* q0 = reinterpret_cast<const float4*>(qs + (2 * ty) * ld);
  const float4* q1 = reinterpret_cast<const float4*>(qs + (2 * ty + 1) * ld);
  for (int c = 0; c < d / 4; ++c) {
    const float4 a0 = q0[c], a1 = q1[c];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float4 kk = reinterpret_cast<const float4*>(ks + (tx + 16 * b) * ld)[c];
      s[0][b] = fmaf(a0.x, kk.x, s[0][b]);
      s[0][b] = fmaf(a0.y, kk.y, s[0][b]);
      s[0][b] = fmaf(a0.z, kk.z, s[0][b]);
      s[0][b] = fmaf(a0.w, kk.w, s[0][b]);
      s[1][b] = fmaf(a1.x, kk.x, s[1][b]);
      s[1][b] = fmaf(a1.y, kk.y, s[1][b]);
      s[1][b] = fmaf(a1.z, kk.z, s[1][b]);
      s[1][b] = fmaf(a1.w, kk.w, s[1][b]);
    }
  }
}

// Pass 1.  grid (row blocks, n_kv_heads, n_req).  lse2 [n_req][H][window] in log2 units of the
// scaled logits (s * scale * log2 e).
template <typename T>
__global__ void __launch_bounds__(kThreads) score_lse_kernel(const T* __restrict__ q, const T* __restrict__ k,
                                                             const int32_t* __restrict__ cu_seqlens, int32_t window,
                                                             int32_t n_q_heads, int32_t n_kv_heads, int32_t d,
                                                             float scale_log2, float* __restrict__ lse2) {
  extern __shared__ __align__(16) float smem[];
  const int ld = d + 4;
  float* qs = smem;             // [kRB][ld]
  float* ks = smem + kRB * ld;  // [kKB][ld]
  const int32_t r = blockIdx.z, g = blockIdx.y;
  const int32_t G = n_q_heads / n_kv_heads;
  const int32_t base = cu_seqlens[r], len = cu_seqlens[r + 1] - base;
  const int32_t w = min(window, len);
  const int32_t n_rows = G * w;
  const int32_t row0 = blockIdx.x * kRB;
  if (row0 >= n_rows) return;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  // stage the query rows (rows past n_rows are zero)
  for (int rr = tid >> 3; rr < kRB; rr += kThreads / 8) {
    const int32_t row = row0 + rr;
    float* dst = qs + rr * ld;
    if (row < n_rows) {
      const int32_t hq = g * G + row / w, i = len - w + row % w;
      load_row_f32(dst, q + ((int64_t)(base + i) * n_q_heads + hq) * d, d, tid & 7, 8);
    } else {
      for (int c = tid & 7; c < d; c += 8) dst[c] = 0.f;
    }
  }
  int32_t my_i[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int32_t row = row0 + 2 * ty + a;
    my_i[a] = row < n_rows ? len - w + row % w : -1;
  }
  // last key any row of this block needs
  const int32_t last_row = min(n_rows, row0 + kRB) - 1;
  int32_t i_max = 0;
  if (row0 / w == last_row / w) i_max = len - w + last_row % w; else i_max = len - 1;
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
  for (int32_t j0 = 0; j0 <= i_max; j0 += kKB) {
    __syncthreads();
    for (int rr = tid >> 3; rr < kKB; rr += kThreads / 8) {
      const int32_t j = j0 + rr;
      float* dst = ks + rr * ld;
      if (j < len) load_row_f32(dst, k + ((int64_t)(base + j) * n_kv_heads + g) * d, d, tid & 7, 8);
      else for (int c = tid & 7; c < d; c += 8) dst[c] = 0.f;
    }
    __syncthreads();
    float s[2][4];
    tile_dots(qs, ks, d, ld, ty, tx, s);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      float tmax = -INFINITY;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int32_t j = j0 + tx + 16 * b;
        s[a][b] = j <= my_i[a] ? s[a][b] * scale_log2 : -INFINITY;
        tmax = fmaxf(tmax, s[a][b]);
      }
      if (tmax > -INFINITY) {
        const float mn = fmaxf(m[a], tmax);
        float add = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) add += exp2f(s[a][b] - mn);
        l[a] = l[a] * exp2f(m[a] - mn) + add;
        m[a] = mn;
      }
    }
  }
  // combine the 16 threads (tx) that share a row: lanes differ in the low 4 bits
#pragma unroll
  for (int a = 0; a < 2; ++a) {
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) {
      const float mo = __shfl_xor_sync(0xffffffffu, m[a], off), lo = __shfl_xor_sync(0xffffffffu, l[a], off);
      const float mn = fmaxf(m[a], mo);
      if (mn > -INFINITY) {
        l[a] = l[a] * exp2f(m[a] - mn) + lo * exp2f(mo - mn);
        m[a] = mn;
      }
    }
    const int32_t row = row0 + 2 * ty + a;
    if (tx == 0 && row < n_rows)
      lse2[((int64_t)r * n_q_heads + g * G + row / w) * window + row % w] = m[a] + log2f(l[a]);
  }
}

// Pass 2.  grid (key blocks over the longest request, n_kv_heads, n_req).
template <typename T>
__global__ void __launch_bounds__(kThreads) score_colsum_kernel(const T* __restrict__ q, const T* __restrict__ k,
                                                                const int32_t* __restrict__ cu_seqlens,
                                                                int32_t window, int32_t obs, int32_t n_q_heads,
                                                                int32_t n_kv_heads, int32_t d, float scale_log2,
                                                                const float* __restrict__ lse2, int64_t n_tokens,
                                                                float* __restrict__ c_out) {
  extern __shared__ __align__(16) float smem[];
  __shared__ float red[kThreads / 16][kKB];
  const int ld = d + 4;
  float* qs = smem;
  float* ks = smem + kRB * ld;
  const int32_t r = blockIdx.z, g = blockIdx.y;
  const int32_t G = n_q_heads / n_kv_heads;
  const int32_t base = cu_seqlens[r], len = cu_seqlens[r + 1] - base;
  const int32_t w = min(window, len);
  const int32_t nr = len - w;  // non-recent keys
  const int32_t wo = min(obs, len);  // rows that are accumulated: the last wo of the request (Eq. 2: wo = w)
  const int32_t j0 = blockIdx.x * kKB;
  if (j0 >= len) return;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  float* cg = c_out + (int64_t)g * n_tokens + base;
  if (j0 >= nr) {  // block inside the window: defined as 0
    for (int c = tid; c < kKB; c += kThreads)
      if (j0 + c < len) cg[j0 + c] = 0.f;
    return;
  }
  for (int rr = tid >> 3; rr < kKB; rr += kThreads / 8) {
    const int32_t j = j0 + rr;
    float* dst = ks + rr * ld;
    if (j < len) load_row_f32(dst, k + ((int64_t)(base + j) * n_kv_heads + g) * d, d, tid & 7, 8);
    else for (int c = tid & 7; c < d; c += 8) dst[c] = 0.f;
  }
  const int32_t n_rows = G * wo;
  float col[4] = {0.f, 0.f, 0.f, 0.f};
  for (int32_t row0 = 0; row0 < n_rows; row0 += kRB) {
    __syncthreads();
    for (int rr = tid >> 3; rr < kRB; rr += kThreads / 8) {
      const int32_t row = row0 + rr;
      float* dst = qs + rr * ld;
      if (row < n_rows) {
        const int32_t hq = g * G + row / wo, i = len - wo + row % wo;
        load_row_f32(dst, q + ((int64_t)(base + i) * n_q_heads + hq) * d, d, tid & 7, 8);
      } else {
        for (int c = tid & 7; c < d; c += 8) dst[c] = 0.f;
      }
    }
    __syncthreads();
    float s[2][4];
    tile_dots(qs, ks, d, ld, ty, tx, s);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const int32_t row = row0 + 2 * ty + a;
      if (row < n_rows) {
        const float lse = __ldg(lse2 + ((int64_t)r * n_q_heads + g * G + row / wo) * obs + row % wo);
        // with wo = w every non-recent key precedes every accumulated row; a longer observation reaches rows that
        // lie before some of the block's keys, and a row only counts for the keys it can see
        const int32_t i = len - wo + row % wo;
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (j0 + tx + 16 * b <= i) col[b] += exp2f(s[a][b] * scale_log2 - lse);
      }
    }
  }
#pragma unroll
  for (int b = 0; b < 4; ++b) red[ty][tx + 16 * b] = col[b];
  __syncthreads();
  if (tid < kKB) {
    float sum = 0.f;
#pragma unroll
    for (int t = 0; t < kThreads / 16; ++t) sum += red[t][tid];
    const int32_t j = j0 + tid;
    if (j < len) cg[j] = j < nr ? sum / (float)G : 0.f;
  }
}

static int32_t max_len(const purekv_batch* b) {
  int32_t m = 0;
  for (int r = 0; r < b->n_req; ++r) m = std::max(m, b->h_cu_seqlens[r + 1] - b->h_cu_seqlens[r]);
  return m;
}

// ---- bf16 path on tensor cores ------------------------------------------------------------------
// Both passes use the same tiling: a CTA owns one block of 128 keys of one (request, KV head) and walks the
// G*w stacked window rows in blocks of 128; its 8 warps form a 4 x 2 grid, warp (wr, wc) computing the 32 x 64
// logits of rows 32*wr .. +31 against keys 64*wc .. +63 with mma.sync m16n8k16 (bf16 x bf16 -> fp32: products
// exact, fp32 accumulation).  Pass 1 leaves, per 64-key block and row, the maximum and the sum of exponentials of
// the causal logits; a small kernel folds those into the row's log-sum-exp; pass 2 forms exp(s - lse) and sums down
// the rows.  Every key block is an independent CTA, so the grid is (key blocks) x (KV heads) x (requests) in both
// passes.
constexpr int kMmaKeys = 64;    // keys per warp column, and the granularity of the pass-1 (max, sum) pairs
constexpr int kCtaKeys = 128;   // keys per CTA
constexpr int kMmaRows = 128;
constexpr int kMmaThreads = 256;

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x2(uint32_t addr, uint32_t (&r)[2]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16_16x8x16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Copies `rows` rows of d bf16 (global row r at src + row_of(r)) into shared memory with a row stride of d + 8
// elements (conflict-free for ldmatrix); rows for which row_of gives a negative offset are zero-filled.
template <typename RowOf>
__device__ __forceinline__ void stage_rows_bf16(__nv_bfloat16* dst, const __nv_bfloat16* src, int rows, int d, RowOf row_of) {
  const int cpr = d / 8;  // 16-byte chunks per row
  for (int x = threadIdx.x; x < rows * cpr; x += kMmaThreads) {
    const int r = x / cpr, c = x % cpr;
    const int64_t off = row_of(r);
    uint4 v = make_uint4(0, 0, 0, 0);
    if (off >= 0) v = __ldg(reinterpret_cast<const uint4*>(src + off) + c);
    *reinterpret_cast<uint4*>(dst + r * (d + 8) + c * 8) = v;
  }
}

// The same copy with cp.async (16 bytes per request, zero fill for absent rows): returns at once, the data is
// there after cp_async_wait.  Used to load the next block of query rows while the current one is multiplied.
template <typename RowOf>
__device__ __forceinline__ void stage_rows_bf16_async(__nv_bfloat16* dst, const __nv_bfloat16* src, int rows, int d, RowOf row_of) {
  const int cpr = d / 8;
  for (int x = threadIdx.x; x < rows * cpr; x += kMmaThreads) {
    const int r = x / cpr, c = x % cpr;
    const int64_t off = row_of(r);
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(dst + r * (d + 8) + c * 8);
    const void* ga = off >= 0 ? (const void*)(reinterpret_cast<const uint4*>(src + off) + c) : (const void*)src;
    const uint32_t bytes = off >= 0 ? 16u : 0u;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(ga), "r"(bytes) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// acc[mb][nb][0..3] = logits of rows (32*wr + 16*mb + lane/4, +8) x keys (64*wc + 8*nb + 2*(lane%4), +1) of the
// staged tiles: per 16-wide K step two A fragments and four ldmatrix.x4 of K feed sixteen MMAs.
__device__ __forceinline__ void logits_32x64(const __nv_bfloat16* qs, const __nv_bfloat16* ks, int d, float (&acc)[2][8][4]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wr = warp >> 1, wc = warp & 1, ld = d + 8;
#pragma unroll
  for (int mb = 0; mb < 2; ++mb)
#pragma unroll
    for (int nb = 0; nb < 8; ++nb)
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[mb][nb][x] = 0.f;
  const uint32_t qa = (uint32_t)__cvta_generic_to_shared(qs + (32 * wr + (lane & 7) + 8 * ((lane >> 3) & 1)) * ld + 8 * (lane >> 4));
  // K: one x4 covers two 8-key blocks: matrices (keys +0, k 0-7), (keys +0, k 8-15), (keys +8, k 0-7), (keys +8, k 8-15)
  const uint32_t ka = (uint32_t)__cvta_generic_to_shared(ks + (64 * wc + (lane & 7) + 8 * (lane >> 4)) * ld + 8 * ((lane >> 3) & 1));
  for (int k0 = 0; k0 < d; k0 += 16) {
    uint32_t a0[4], a1[4];
    ldmatrix_x4(qa + k0 * 2, a0);
    ldmatrix_x4(qa + (16 * ld + k0) * 2, a1);
#pragma unroll
    for (int nb = 0; nb < 8; nb += 2) {
      uint32_t b4[4];
      ldmatrix_x4(ka + (nb * 8 * ld + k0) * 2, b4);
      const uint32_t b0[2] = {b4[0], b4[1]}, b1[2] = {b4[2], b4[3]};
      mma_bf16_16x8x16(acc[0][nb], a0, b0);
      mma_bf16_16x8x16(acc[1][nb], a1, b0);
      mma_bf16_16x8x16(acc[0][nb + 1], a0, b1);
      mma_bf16_16x8x16(acc[1][nb + 1], a1, b1);
    }
  }
}

// Pass 1.  partial[((r * Hkv + g) * n_kb + kb64) * rows_max + row] = (max, sum of exp2) of the causal logits of the
// stacked row against the 64-key block kb64, in log2 units of the scaled logits.
__global__ void __launch_bounds__(kMmaThreads) score_mma_partial_kernel(
    const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, const int32_t* __restrict__ cu_seqlens,
    int32_t window, int32_t n_q_heads, int32_t n_kv_heads, int32_t d, float scale_log2, int32_t n_kb, int32_t rows_max,
    float2* __restrict__ partial) {
  extern __shared__ __align__(16) uint8_t smem_mma[];
  __nv_bfloat16* ks = reinterpret_cast<__nv_bfloat16*>(smem_mma);
  __nv_bfloat16* qs = ks + kCtaKeys * (d + 8);
  const int32_t r = blockIdx.z, g = blockIdx.y;
  const int32_t G = n_q_heads / n_kv_heads;
  const int32_t base = cu_seqlens[r], len = cu_seqlens[r + 1] - base;
  const int32_t w = min(window, len), n_rows = G * w, j0 = blockIdx.x * kCtaKeys;
  if (j0 >= len) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wr = warp >> 1, wc = warp & 1;
  stage_rows_bf16(ks, k, kCtaKeys, d, [&](int rr) -> int64_t {
    return j0 + rr < len ? ((int64_t)(base + j0 + rr) * n_kv_heads + g) * d : -1;
  });
  const int32_t kb64 = 2 * blockIdx.x + wc;  // this warp's 64-key block
  float2* out = partial + ((int64_t)(r * n_kv_heads + g) * n_kb + kb64) * rows_max;
  const bool block_live = j0 + 64 * wc < len;  // the second half of the last CTA may lie past the request
  auto q_row = [&](int32_t row) -> int64_t {
    return row < n_rows ? ((int64_t)(base + len - w + row % w) * n_q_heads + g * G + row / w) * d : -1;
  };
  __nv_bfloat16* qbuf[2] = {qs, qs + kMmaRows * (d + 8)};
  stage_rows_bf16_async(qbuf[0], q, kMmaRows, d, [&](int rr) { return q_row(rr); });
  for (int32_t row0 = 0, it = 0; row0 < n_rows; row0 += kMmaRows, ++it) {
    __syncthreads();  // everyone is done with the buffer the next copy overwrites (and, first time, K is staged)
    if (row0 + kMmaRows < n_rows) {
      stage_rows_bf16_async(qbuf[(it + 1) & 1], q, kMmaRows, d, [&](int rr) { return q_row(row0 + kMmaRows + rr); });
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const __nv_bfloat16* qcur = qbuf[it & 1];
    float acc[2][8][4];
    logits_32x64(qcur, ks, d, acc);
#pragma unroll
    for (int mb = 0; mb < 2; ++mb)
#pragma unroll
      for (int h = 0; h < 2; ++h) {  // the thread's four rows
        const int32_t row = row0 + 32 * wr + 16 * mb + (lane >> 2) + 8 * h;
        const int32_t i = row < n_rows ? len - w + row % w : -1;  // causal limit of the row (-1: no row)
        float m = -INFINITY;
#pragma unroll
        for (int nb = 0; nb < 8; ++nb)
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const int32_t j = j0 + 64 * wc + 8 * nb + 2 * (lane & 3) + x;
            const float sv = j <= i ? acc[mb][nb][2 * h + x] * scale_log2 : -INFINITY;
            acc[mb][nb][2 * h + x] = sv;
            m = fmaxf(m, sv);
          }
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        float l = 0.f;
        if (m > -INFINITY) {
#pragma unroll
          for (int nb = 0; nb < 8; ++nb) l += exp2f(acc[mb][nb][2 * h] - m) + exp2f(acc[mb][nb][2 * h + 1] - m);
        }
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        if ((lane & 3) == 0 && row < n_rows && block_live) out[row] = make_float2(m, l);
      }
  }
}

// Folds the per-key-block (max, sum) pairs into each stacked row's log-sum-exp.  One thread per (request, query
// head, window position).
__global__ void __launch_bounds__(256) score_lse_merge_kernel(const float2* __restrict__ partial,
                                                              const int32_t* __restrict__ cu_seqlens, int32_t window,
                                                              int32_t n_q_heads, int32_t n_kv_heads, int32_t n_kb,
                                                              int32_t rows_max, int32_t n_req, float* __restrict__ lse2) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= (int64_t)n_req * n_q_heads * window) return;
  const int32_t iw = (int32_t)(x % window), hq = (int32_t)((x / window) % n_q_heads), r = (int32_t)(x / ((int64_t)window * n_q_heads));
  const int32_t G = n_q_heads / n_kv_heads, g = hq / G, hl = hq % G;
  const int32_t len = cu_seqlens[r + 1] - cu_seqlens[r];
  const int32_t w = min(window, len);
  if (iw >= w) return;
  const int32_t row = hl * w + iw, kbs = (len + kMmaKeys - 1) / kMmaKeys;
  const float2* p = partial + ((int64_t)(r * n_kv_heads + g) * n_kb) * rows_max + row;
  float m = -INFINITY;
  for (int32_t kb = 0; kb < kbs; ++kb) m = fmaxf(m, p[(int64_t)kb * rows_max].x);
  float l = 0.f;
  for (int32_t kb = 0; kb < kbs; ++kb) {
    const float2 v = p[(int64_t)kb * rows_max];
    if (v.y > 0.f) l += v.y * exp2f(v.x - m);
  }
  lse2[((int64_t)r * n_q_heads + hq) * window + iw] = m + log2f(l);
}

// Pass 2 (Eq. 2).  C[g, j] = (1/G) * sum over the stacked rows of exp2(s - lse) for the non-recent keys of the CTA's block.
__global__ void __launch_bounds__(kMmaThreads) score_mma_colsum_kernel(
    const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, const int32_t* __restrict__ cu_seqlens,
    int32_t window, int32_t obs, int32_t n_q_heads, int32_t n_kv_heads, int32_t d, float scale_log2,
    const float* __restrict__ lse2, int64_t n_tokens, float* __restrict__ c_out) {
  extern __shared__ __align__(16) uint8_t smem_mma[];
  __shared__ float red[4][kCtaKeys];  // per row group of warps
  __nv_bfloat16* ks = reinterpret_cast<__nv_bfloat16*>(smem_mma);
  __nv_bfloat16* qs = ks + kCtaKeys * (d + 8);
  const int32_t r = blockIdx.z, g = blockIdx.y, j0 = blockIdx.x * kCtaKeys;
  const int32_t G = n_q_heads / n_kv_heads;
  const int32_t base = cu_seqlens[r], len = cu_seqlens[r + 1] - base;
  const int32_t w = min(window, len), nr = len - w;
  const int32_t wo = min(obs, len), n_rows = G * wo;  // accumulated rows: the last wo of the request (Eq. 2: wo = w)
  if (j0 >= len) return;
  float* cg = c_out + (int64_t)g * n_tokens + base;
  if (j0 >= nr) {  // block inside the window: defined as 0
    for (int c = threadIdx.x; c < kCtaKeys; c += kMmaThreads)
      if (j0 + c < len) cg[j0 + c] = 0.f;
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wr = warp >> 1, wc = warp & 1;
  stage_rows_bf16(ks, k, kCtaKeys, d, [&](int rr) -> int64_t {
    return j0 + rr < len ? ((int64_t)(base + j0 + rr) * n_kv_heads + g) * d : -1;
  });
  float col[8][2];
#pragma unroll
  for (int nb = 0; nb < 8; ++nb) col[nb][0] = col[nb][1] = 0.f;
  auto q_row = [&](int32_t row) -> int64_t {
    return row < n_rows ? ((int64_t)(base + len - wo + row % wo) * n_q_heads + g * G + row / wo) * d : -1;
  };
  __nv_bfloat16* qbuf[2] = {qs, qs + kMmaRows * (d + 8)};
  stage_rows_bf16_async(qbuf[0], q, kMmaRows, d, [&](int rr) { return q_row(rr); });
  for (int32_t row0 = 0, it = 0; row0 < n_rows; row0 += kMmaRows, ++it) {
    __syncthreads();  // everyone is done with the buffer the next copy overwrites (and, first time, K is staged)
    if (row0 + kMmaRows < n_rows) {
      stage_rows_bf16_async(qbuf[(it + 1) & 1], q, kMmaRows, d, [&](int rr) { return q_row(row0 + kMmaRows + rr); });
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const __nv_bfloat16* qcur = qbuf[it & 1];
    float acc[2][8][4];
    logits_32x64(qcur, ks, d, acc);
#pragma unroll
    for (int mb = 0; mb < 2; ++mb)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int32_t row = row0 + 32 * wr + 16 * mb + (lane >> 2) + 8 * h;
        if (row < n_rows) {
          const float lse = __ldg(lse2 + ((int64_t)r * n_q_heads + g * G + row / wo) * obs + row % wo);
          if (wo == w) {
            // every non-recent key precedes every window row, so causality holds for all of them
#pragma unroll
            for (int nb = 0; nb < 8; ++nb) {
              col[nb][0] += exp2f(fmaf(acc[mb][nb][2 * h], scale_log2, -lse));
              col[nb][1] += exp2f(fmaf(acc[mb][nb][2 * h + 1], scale_log2, -lse));
            }
          } else {
            // a longer observation reaches rows that lie before some keys: a row only counts for the keys it sees
            const int32_t i = len - wo + row % wo, jb = j0 + 64 * wc + 2 * (lane & 3);
#pragma unroll
            for (int nb = 0; nb < 8; ++nb) {
              if (jb + 8 * nb <= i) col[nb][0] += exp2f(fmaf(acc[mb][nb][2 * h], scale_log2, -lse));
              if (jb + 8 * nb + 1 <= i) col[nb][1] += exp2f(fmaf(acc[mb][nb][2 * h + 1], scale_log2, -lse));
            }
          }
        }
      }
  }
  // sum over the 8 row groups of the warp (lanes with equal lane % 4 hold the same columns), then over the 4 row warps
#pragma unroll
  for (int nb = 0; nb < 8; ++nb)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      float v = col[nb][x];
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      if (lane < 4) red[wr][64 * wc + 8 * nb + 2 * lane + x] = v;
    }
  __syncthreads();
  if (threadIdx.x < kCtaKeys) {
    const float sum = (red[0][threadIdx.x] + red[1][threadIdx.x]) + (red[2][threadIdx.x] + red[3][threadIdx.x]);
    const int32_t j = j0 + threadIdx.x;
    if (j < len) cg[j] = j < nr ? sum / (float)G : 0.f;
  }
}

// ---- bf16, both passes in one launch -------------------------------------------------------------------------------
// A cluster of C CTAs owns one (request, KV head): each keeps MB blocks of 128 keys in shared memory and walks the stacked
// rows in blocks of 128 like the two kernels above, but the logits are formed once: a CTA's (max, sum of exponentials) per
// row goes to every CTA of the cluster through distributed shared memory, and after one cluster barrier each has the rows'
// log-sum-exp and sums exp(s - lse) down the rows from the accumulators it still holds.  Pooling along the keys takes the
// few scores it needs beyond a CTA's keys from its neighbours the same way.  No workspace, one launch instead of three or
// four.  Requests of up to 16 x 256 keys; longer ones take the passes above, which read K twice but need no more than one
// block of keys per CTA.  Bound by latencies at these sizes (launch, staging, a cluster barrier per block of rows): 2432
// tokens, 32 / 8 heads, 32 voting rows, pool 7: 38 us with four kernels, now 15; window of 64
// rows: 45 -> 23.
constexpr int kClusterMax = 16;        // CTAs per cluster
constexpr int kClusterRowBlocks = 16;  // blocks of 128 stacked rows
constexpr int kPoolHalfMax = 64;       // scores taken from a neighbour on either side

struct ScoreClusterShared {
  float2 part[2][kClusterMax][kMmaRows];  // [parity of the block of rows][CTA][row]: (max, sum) in log2 units
  float2 half[2][kMmaRows];               // the same per 64-key column of warps
  float lse[kMmaRows];
};

// The mean over 2 * half + 1 keys of the scores in colbuf, a CTA's kKeys at j0 ..: `half` scores on either side come from the
// neighbouring CTAs (outside the request: 0).  All threads of the cluster take part.
template <int kKeys>
__device__ __forceinline__ void pool_in_cluster(const float* colbuf, float (*halo)[kPoolHalfMax], int32_t half, int32_t rank,
                                                int32_t C, int32_t j0, int32_t nr, int32_t len, float* cg) {
  const int tid = threadIdx.x;
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (tid < 2 * half) {
    const int32_t side = tid >= half, at = side ? tid - half : tid, from = rank + (side ? 1 : -1);
    float v = 0.f;
    if (from >= 0 && from < C) {
      uint32_t src;
      asm("mapa.shared::cluster.u32 %0, %1, %2;"
          : "=r"(src) : "r"((uint32_t)__cvta_generic_to_shared(colbuf + (side ? at : kKeys - half + at))), "r"(from));
      asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(src) : "memory");
    }
    halo[side][at] = v;
  }
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // done with the neighbours' memory
  if (tid < kKeys && j0 + tid < len) {
    float sum = 0.f;
    if (j0 + tid < nr)
      for (int32_t x = tid - half; x <= tid + half; ++x)
        sum += x < 0 ? halo[0][half + x] : x >= kKeys ? halo[1][x - kKeys] : colbuf[x];
    cg[j0 + tid] = sum / (float)(2 * half + 1);
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // a CTA's memory outlives its neighbours' reads
}

template <int MB>
__global__ void __launch_bounds__(kMmaThreads, 1) score_cluster_kernel(
    const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, const int32_t* __restrict__ cu_seqlens,
    int32_t window, int32_t obs, int32_t pool, int32_t n_q_heads, int32_t n_kv_heads, int32_t d, float scale_log2,
    int64_t n_tokens, float* __restrict__ c_out) {
  constexpr int kKeys = MB * kCtaKeys;
  extern __shared__ __align__(16) uint8_t smem_mma[];
  __shared__ ScoreClusterShared sh;
  __shared__ float red[4][kKeys];                      // per row group of warps
  __shared__ float colbuf[kKeys];                      // the CTA's scores before pooling, read by its neighbours too
  __shared__ float halo[2][kPoolHalfMax];
  __nv_bfloat16* ks = reinterpret_cast<__nv_bfloat16*>(smem_mma);
  __nv_bfloat16* qs = ks + kKeys * (d + 8);
  const int32_t C = gridDim.x, rank = blockIdx.x, r = blockIdx.z, g = blockIdx.y, j0 = rank * kKeys;
  const int32_t G = n_q_heads / n_kv_heads;
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // "started": awaited before the first exchange
  asm volatile("griddepcontrol.wait;" ::: "memory");  // (launched with programmatic stream serialization)
  const int32_t base = cu_seqlens[r], len = cu_seqlens[r + 1] - base;
  const int32_t w = min(window, len), nr = len - w, wo = min(obs, len), n_rows = G * wo;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wr = warp >> 1, wc = warp & 1;
  if (nr == 0) {  // (the same for all CTAs of the cluster) a request within its window: no key has a score
    for (int32_t j = j0 + tid; j < min(len, j0 + kKeys); j += kMmaThreads) c_out[(int64_t)g * n_tokens + base + j] = 0.f;
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    return;
  }
  auto q_row = [&](int32_t row) -> int64_t {
    return row < n_rows ? ((int64_t)(base + len - wo + row % wo) * n_q_heads + g * G + row / wo) * d : -1;
  };
  stage_rows_bf16_async(ks, k, kKeys, d, [&](int rr) -> int64_t {
    return j0 + rr < len ? ((int64_t)(base + j0 + rr) * n_kv_heads + g) * d : -1;
  });
  __nv_bfloat16* qbuf[2] = {qs, qs + kMmaRows * (d + 8)};
  stage_rows_bf16_async(qbuf[0], q, kMmaRows, d, [&](int rr) { return q_row(rr); });
  float col[MB][8][2];
#pragma unroll
  for (int m = 0; m < MB; ++m)
#pragma unroll
    for (int nb = 0; nb < 8; ++nb) col[m][nb][0] = col[m][nb][1] = 0.f;
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  for (int32_t row0 = 0, it = 0; row0 < n_rows; row0 += kMmaRows, ++it) {
    __syncthreads();  // everyone is done with the buffer the next copy overwrites
    if (row0 + kMmaRows < n_rows) {
      stage_rows_bf16_async(qbuf[(it + 1) & 1], q, kMmaRows, d, [&](int rr) { return q_row(row0 + kMmaRows + rr); });
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    float acc[MB][2][8][4];
#pragma unroll
    for (int m = 0; m < MB; ++m) logits_32x64(qbuf[it & 1], ks + m * kCtaKeys * (d + 8), d, acc[m]);
    // scaled logits, causal; the warp's (max, sum) per row over its keys
#pragma unroll
    for (int mb = 0; mb < 2; ++mb)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int32_t rl = 32 * wr + 16 * mb + (lane >> 2) + 8 * h, row = row0 + rl;
        const int32_t i = row < n_rows ? len - wo + row % wo : -1;  // causal limit of the row (-1: no row)
        float mx = -INFINITY;
#pragma unroll
        for (int m = 0; m < MB; ++m)
#pragma unroll
          for (int nb = 0; nb < 8; ++nb)
#pragma unroll
            for (int x = 0; x < 2; ++x) {
              const int32_t j = j0 + m * kCtaKeys + 64 * wc + 8 * nb + 2 * (lane & 3) + x;
              const float sv = j <= i ? acc[m][mb][nb][2 * h + x] * scale_log2 : -INFINITY;
              acc[m][mb][nb][2 * h + x] = sv;
              mx = fmaxf(mx, sv);
            }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        float l = 0.f;
        if (mx > -INFINITY) {
#pragma unroll
          for (int m = 0; m < MB; ++m)
#pragma unroll
            for (int nb = 0; nb < 8; ++nb) l += exp2f(acc[m][mb][nb][2 * h] - mx) + exp2f(acc[m][mb][nb][2 * h + 1] - mx);
        }
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        if ((lane & 3) == 0) sh.half[wc][rl] = make_float2(mx, l);
      }
    __syncthreads();
    // the CTA's pair per row, to every CTA of the cluster (two threads per row, each serves every other CTA)
    {
      const int32_t rl = tid >> 1;
      const float2 a = sh.half[0][rl], b = sh.half[1][rl];
      const float mx = fmaxf(a.x, b.x);
      float l = 0.f;
      if (a.y > 0.f) l += a.y * exp2f(a.x - mx);
      if (b.y > 0.f) l += b.y * exp2f(b.x - mx);
      const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&sh.part[it & 1][rank][rl]);
      for (int32_t to = tid & 1; to < C; to += 2) {
        uint32_t dst;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(mine), "r"(to));
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(mx), "f"(l) : "memory");
      }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    // the rows' log-sum-exp: two threads per row, each over every other CTA.  (The pairs of this parity are overwritten two
    // blocks of rows later, behind the next block's barrier, which everybody reaches after this read.)
    bool odd;  // a row of NaN logits (passed over by the maxima: -inf) or with a NaN sum
    {
      const int32_t rl = tid >> 1;
      float mx = -INFINITY;
      for (int32_t x = tid & 1; x < C; x += 2) mx = fmaxf(mx, sh.part[it & 1][x][rl].x);
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      float l = 0.f;
      for (int32_t x = tid & 1; x < C; x += 2) {
        const float2 p = sh.part[it & 1][x][rl];
        if (p.y > 0.f) l += p.y * exp2f(p.x - mx);
      }
      l += __shfl_xor_sync(0xffffffffu, l, 1);
      const float lse = row0 + rl < n_rows ? mx + log2f(l) : INFINITY;  // (+inf: an absent row adds nothing)
      if ((tid & 1) == 0) sh.lse[rl] = lse;
      odd = !(lse > -INFINITY);
    }
    const bool any_odd = __syncthreads_or(odd);
    auto add = [&](auto check_c) {
#pragma unroll
      for (int mb = 0; mb < 2; ++mb)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float lse = sh.lse[32 * wr + 16 * mb + (lane >> 2) + 8 * h];
#pragma unroll
          for (int m = 0; m < MB; ++m)
#pragma unroll
            for (int nb = 0; nb < 8; ++nb)
#pragma unroll
              for (int x = 0; x < 2; ++x) {
                const float sv = acc[m][mb][nb][2 * h + x];
                // keys the row does not see are -inf and add nothing, also where the row's sum is NaN
                if (!decltype(check_c)::value || sv != -INFINITY) col[m][nb][x] += exp2f(sv - lse);
              }
        }
    };
    if (any_odd) add(std::true_type{});
    else add(std::false_type{});
  }
  // sum over the 8 row groups of the warp (lanes with equal lane % 4 hold the same columns), then over the 4 row warps
#pragma unroll
  for (int m = 0; m < MB; ++m)
#pragma unroll
    for (int nb = 0; nb < 8; ++nb)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        float v = col[m][nb][x];
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 16);
        if (lane < 4) red[wr][m * kCtaKeys + 64 * wc + 8 * nb + 2 * lane + x] = v;
      }
  __syncthreads();
  float* cg = c_out + (int64_t)g * n_tokens + base;
  const int32_t half = pool / 2;
  if (tid < kKeys) {
    const float sum = (red[0][tid] + red[1][tid]) + (red[2][tid] + red[3][tid]);
    const int32_t j = j0 + tid;
    const float v = j < nr ? sum / (float)G : 0.f;  // (the window, and keys past the end: 0)
    if (half == 0 && j < len) cg[j] = v;
    colbuf[tid] = v;
  }
  if (half == 0) return;  // (no CTA reads another's shared memory behind the last barrier)
  pool_in_cluster<kKeys>(colbuf, halo, half, rank, C, j0, nr, len, cg);
}

// A launch of grid (C, Hkv, n_req) in clusters of C CTAs, behind the previous kernel by programmatic stream serialization.
struct ClusterLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  ClusterLaunch(int32_t C, int32_t Hkv, int32_t n_req, int threads, size_t smem, cudaStream_t sm) {
    cfg.gridDim = dim3((unsigned)C, (unsigned)Hkv, (unsigned)n_req);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = sm;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)C;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
  }
  ClusterLaunch(const ClusterLaunch&) = delete;
  ClusterLaunch& operator=(const ClusterLaunch&) = delete;
};

// Allows the kernel all of an SM's shared memory and clusters of more than eight CTAs (opt-in, once per device).
template <typename... Params>
static purekv_status allow_wide_clusters(void (*kernel)(Params...), std::atomic<uint64_t>& smem, std::atomic<uint64_t>& wide) {
  const purekv_status st = allow_max_dynamic_smem(kernel, smem);
  if (st != PUREKV_OK) return st;
  int dev = -1;
  PK_CUDA(cudaGetDevice(&dev));
  if (!(wide.load(std::memory_order_acquire) & (1ull << dev))) {
    PK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    wide.fetch_or(1ull << dev, std::memory_order_release);
  }
  return PUREKV_OK;
}

// Requests with a key outside their window: each is a cluster's work per KV head, the others are none.
static int64_t live_requests(const purekv_batch* b, int32_t window) {
  int64_t n = 0;
  for (int r = 0; r < b->n_req; ++r) n += b->h_cu_seqlens[r + 1] - b->h_cu_seqlens[r] > window;
  return n;
}

// Which form the scores take is decided by what each would take, in us, from times measured over 1-128 requests of 100-4200
// tokens, 1-8 query heads per KV head and 8-400 rows (d = 128); the estimates are within a fifth of them.  A cluster of C CTAs
// keeps C SMs through all its blocks of rows, whatever the request's length, and few of the large ones fit at once (7 of 16 CTAs,
// 15 of 8), so clusters run in waves: 6.4 us per block of rows and 2.5 more with 128 keys per CTA, 9.3 and 3 with 256.  The
// separate kernels take 9.4 us per block with up to one CTA per SM, 13.5 with two and so on, and 18 for three launches.
// In one wave the cluster is always the faster (1 x 2048, 28 / 4 heads, 64 rows: 31 against 54); in several it has to be so by a
// tenth.  (1 x 2048, 32 / 8 heads, 100 rows: 40 as 8 clusters of 8 against 51 and, as 8 of 16, 59; 2000 + 100 + 50 tokens, 64 rows:
// 42 against 43 and 62; 4 x 2432, 100 rows: 120 against 158; 4000 + 3 x 300, 16 rows: 58 against 46.)
static double cluster_us(int32_t keys_per_cta, int64_t live_clusters, int32_t at_once, int32_t row_blocks, double* waves) {
  *waves = (double)std::max<int64_t>(1, (live_clusters + at_once - 1) / at_once);
  return live_clusters == 0 ? 3. : *waves * (keys_per_cta == kCtaKeys ? 2.5 + 6.4 * row_blocks : 3. + 9.3 * row_blocks);
}
static double separate_us(const purekv_batch* b, int32_t window, int32_t Hkv, int32_t row_blocks) {
  int64_t all = 0, scored = 0;  // key blocks of the first pass, and of the second
  for (int r = 0; r < b->n_req; ++r) {
    const int32_t len = b->h_cu_seqlens[r + 1] - b->h_cu_seqlens[r];
    all += (len + kCtaKeys - 1) / kCtaKeys;
    scored += (std::max(0, len - window) + kCtaKeys - 1) / kCtaKeys;
  }
  const double per_sm = 0.5 * (double)((all + scored) * Hkv) / 148.;
  return 18. + 4. * per_sm + row_blocks * (per_sm > 2. ? 6.5 * per_sm + 3. : per_sm > 1. ? 13.5 : 9.4);
}

// One form of the cluster kernel for a call: its launch, and what it would take (infinity where it cannot run).
template <int MB>
struct ScoreCluster {
  int32_t C;
  ClusterLaunch l;
  double us = INFINITY, waves = 0.;
  ScoreCluster(const purekv_batch* b, int32_t Hkv, int32_t d, cudaStream_t sm)
      : C(std::max(1, (max_len(b) + MB * kCtaKeys - 1) / (MB * kCtaKeys))),
        l(C, Hkv, b->n_req, kMmaThreads, (size_t)(MB * kCtaKeys + 2 * kMmaRows) * (d + 8) * sizeof(__nv_bfloat16), sm) {}
  purekv_status weigh(int64_t live_clusters, int32_t row_blocks) {
    static std::atomic<uint64_t> smem_allowed{0}, wide_allowed{0};
    if (C > kClusterMax) return PUREKV_OK;
    const purekv_status st = allow_wide_clusters(score_cluster_kernel<MB>, smem_allowed, wide_allowed);
    if (st != PUREKV_OK) return st;
    const int32_t at_once = clusters_at_once(score_cluster_kernel<MB>, l.cfg);
    if (at_once >= 1) us = cluster_us(MB * kCtaKeys, live_clusters, at_once, row_blocks, &waves);
    return PUREKV_OK;
  }
};

// The bf16 scores in one cluster launch, if that is the form to take (*launched).
static purekv_status launch_score_cluster(const void* q, const void* k, float* c_out, const purekv_batch* b, int32_t window,
                                          int32_t obs, int32_t pool, int32_t H, int32_t Hkv, int32_t d, float scale,
                                          cudaStream_t sm, bool* launched) {
  const int32_t row_blocks = ((H / Hkv) * obs + kMmaRows - 1) / kMmaRows;
  const int64_t live = live_requests(b, window) * Hkv;
  ScoreCluster<1> one(b, Hkv, d, sm);
  ScoreCluster<2> two(b, Hkv, d, sm);
  purekv_status st = one.weigh(live, row_blocks);
  if (st == PUREKV_OK) st = two.weigh(live, row_blocks);
  if (st != PUREKV_OK) return st;
  const bool small = one.us <= two.us;
  const double us = small ? one.us : two.us, waves = small ? one.waves : two.waves;
  *launched = us < INFINITY && (waves <= 1. || us <= 0.9 * separate_us(b, window, Hkv, row_blocks));
  if (!*launched) return PUREKV_OK;
  const float scale_log2 = scale * 1.4426950408889634f;
  const auto *qb = (const __nv_bfloat16*)q, *kb = (const __nv_bfloat16*)k;
  if (small) PK_CUDA(cudaLaunchKernelEx(&one.l.cfg, score_cluster_kernel<1>, qb, kb, b->cu_seqlens, window, obs, pool, H, Hkv, d, scale_log2, b->total_tokens, c_out));
  else PK_CUDA(cudaLaunchKernelEx(&two.l.cfg, score_cluster_kernel<2>, qb, kb, b->cu_seqlens, window, obs, pool, H, Hkv, d, scale_log2, b->total_tokens, c_out));
  return PUREKV_OK;
}

// ---- fp32, both passes in one launch -------------------------------------------------------------------------------
// The cluster scheme above with fp32 products on CUDA cores: a CTA keeps 64 keys, a block is 32 stacked rows.  Requests of
// up to 16 x 64 keys; for a short prompt the two-kernel form spends its time in one CTA that walks all keys (288 tokens,
// 2 heads, window 16: 28 us for the two kernels, now 6).
struct ScoreClusterSharedF32 {
  float2 part[2][kClusterMax][kRB];
  float lse[kRB];
  float red[kThreads / 16][kKB];
  float colbuf[kKB];
  float halo[2][kPoolHalfMax];
};

template <typename RowOf>
__device__ __forceinline__ void stage_rows_f32_async(float* dst, const float* src, int rows, int d, RowOf row_of) {
  const int cpr = d / 4;
  for (int x = threadIdx.x; x < rows * cpr; x += kThreads) {
    const int r = x / cpr, c = 4 * (x % cpr);
    const int64_t off = row_of(r);
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(dst + r * (d + 4) + c);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(off >= 0 ? src + off + c : src), "r"(off >= 0 ? 16u : 0u)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

__global__ void __launch_bounds__(kThreads, 1) score_cluster_f32_kernel(
    const float* __restrict__ q, const float* __restrict__ k, const int32_t* __restrict__ cu_seqlens, int32_t window, int32_t obs,
    int32_t pool, int32_t n_q_heads, int32_t n_kv_heads, int32_t d, float scale_log2, int64_t n_tokens,
    float* __restrict__ c_out) {
  extern __shared__ __align__(16) float smem[];
  __shared__ ScoreClusterSharedF32 sh;
  const int ld = d + 4;
  float* ks = smem;             // [kKB][ld]
  float* qs = ks + kKB * ld;    // [2][kRB][ld]
  const int32_t C = gridDim.x, rank = blockIdx.x, r = blockIdx.z, g = blockIdx.y, j0 = rank * kKB;
  const int32_t G = n_q_heads / n_kv_heads;
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // "started": awaited before the first exchange
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int32_t base = cu_seqlens[r], len = cu_seqlens[r + 1] - base;
  const int32_t w = min(window, len), nr = len - w, wo = min(obs, len), n_rows = G * wo;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  if (nr == 0) {  // (the same for all CTAs of the cluster) a request within its window: no key has a score
    for (int32_t j = j0 + tid; j < min(len, j0 + kKB); j += kThreads) c_out[(int64_t)g * n_tokens + base + j] = 0.f;
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    return;
  }
  auto q_row = [&](int32_t row) -> int64_t {
    return row < n_rows ? ((int64_t)(base + len - wo + row % wo) * n_q_heads + g * G + row / wo) * d : -1;
  };
  stage_rows_f32_async(ks, k, kKB, d, [&](int rr) -> int64_t {
    return j0 + rr < len ? ((int64_t)(base + j0 + rr) * n_kv_heads + g) * d : -1;
  });
  stage_rows_f32_async(qs, q, kRB, d, q_row);
  float col[4] = {0.f, 0.f, 0.f, 0.f};
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  for (int32_t row0 = 0, it = 0; row0 < n_rows; row0 += kRB, ++it) {
    __syncthreads();  // everyone is done with the buffer the next copy overwrites
    if (row0 + kRB < n_rows) {
      stage_rows_f32_async(qs + ((it + 1) & 1) * kRB * ld, q, kRB, d, [&](int rr) { return q_row(row0 + kRB + rr); });
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    float s[2][4];
    tile_dots(qs + (it & 1) * kRB * ld, ks, d, ld, ty, tx, s);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const int32_t rl = 2 * ty + a, row = row0 + rl, i = row < n_rows ? len - wo + row % wo : -1;
      float mx = -INFINITY;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        s[a][b] = j0 + tx + 16 * b <= i ? s[a][b] * scale_log2 : -INFINITY;
        mx = fmaxf(mx, s[a][b]);
      }
#pragma unroll
      for (int off = 8; off >= 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      float l = 0.f;
      if (mx > -INFINITY) {
#pragma unroll
        for (int b = 0; b < 4; ++b) l += exp2f(s[a][b] - mx);
      } else {  // nothing seen, or NaN logits alone, which the maximum has passed over: the row's sum is NaN then
#pragma unroll
        for (int b = 0; b < 4; ++b) l += s[a][b] != -INFINITY ? s[a][b] : 0.f;
      }
#pragma unroll
      for (int off = 8; off >= 1; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
      // lane tx of the row's sixteen threads serves CTA tx of the cluster
      if (tx < C) {
        uint32_t dst;
        asm("mapa.shared::cluster.u32 %0, %1, %2;"
            : "=r"(dst) : "r"((uint32_t)__cvta_generic_to_shared(&sh.part[it & 1][rank][rl])), "r"(tx));
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(mx), "f"(l) : "memory");
      }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const int32_t rl = 2 * ty + a;
      const float2 p = tx < C ? sh.part[it & 1][tx][rl] : make_float2(-INFINITY, 0.f);
      float mx = p.x;
#pragma unroll
      for (int off = 8; off >= 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      float l = p.y != 0.f ? p.y * exp2f(p.x - mx) : 0.f;
#pragma unroll
      for (int off = 8; off >= 1; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
      const float lse = row0 + rl < n_rows ? mx + log2f(l) : INFINITY;  // (+inf: an absent row adds nothing)
      if (__any_sync(0xffffffffu, !(lse > -INFINITY))) {  // a row with a NaN sum: its NaN goes to the keys it sees alone
#pragma unroll
        for (int b = 0; b < 4; ++b) col[b] += s[a][b] == -INFINITY ? 0.f : exp2f(s[a][b] - lse);
      } else {
#pragma unroll
        for (int b = 0; b < 4; ++b) col[b] += exp2f(s[a][b] - lse);
      }
    }
  }
#pragma unroll
  for (int b = 0; b < 4; ++b) sh.red[ty][tx + 16 * b] = col[b];
  __syncthreads();
  float* cg = c_out + (int64_t)g * n_tokens + base;
  const int32_t half = pool / 2;
  if (tid < kKB) {
    float sum = 0.f;
#pragma unroll
    for (int t = 0; t < kThreads / 16; ++t) sum += sh.red[t][tid];
    const int32_t j = j0 + tid;
    const float v = j < nr ? sum / (float)G : 0.f;
    if (half == 0 && j < len) cg[j] = v;
    sh.colbuf[tid] = v;
  }
  if (half == 0) return;  // (no CTA reads another's shared memory behind the last barrier)
  pool_in_cluster<kKB>(sh.colbuf, sh.halo, half, rank, C, j0, nr, len, cg);
}

// The same choice for fp32, in us as measured over 1-64 requests of 100-1024 tokens, d = 64-256.  The cluster: a block of 32 rows
// 3.4-4.3 us (d = 64), more where clusters share SMs.  The separate kernels: one CTA walks all key blocks in the first pass and all
// row blocks in the second, 2.4 us (d = 64) a step, more where CTAs queue.  (288 tokens, 16 rows: 5.6 in a cluster, 25 separately;
// 64 x 300, 256 rows: 416 and 293; 8 x 1024, 8 / 2 heads, 64 rows: 101 and 86.)
static double cluster_f32_us(int32_t C, int32_t d, int64_t live_clusters, int32_t at_once, int32_t row_blocks) {
  auto wave = [&](int64_t clusters) {
    const double per_sm = (double)clusters * C / 148.;
    return 2. + row_blocks * (1.65 + 0.0262 * d + 0.055 * C) * (per_sm > 1. ? 1. + 0.8 * (per_sm - 1.) : 1.);
  };
  const int64_t last = live_clusters % at_once;
  return (double)(live_clusters / at_once) * wave(at_once) + (last ? wave(last) : 0.);
}
static double separate_f32_us(const purekv_batch* b, int32_t window, int32_t obs, int32_t H, int32_t Hkv, int32_t d, int32_t row_blocks) {
  int64_t rows = 0, keys = 0, scored = 0;  // CTAs of the first pass; of the second, and those that have work
  for (int r = 0; r < b->n_req; ++r) {
    const int32_t len = b->h_cu_seqlens[r + 1] - b->h_cu_seqlens[r];
    rows += ((int64_t)(H / Hkv) * std::min(obs, len) + kRB - 1) / kRB;
    keys += (len + kKB - 1) / kKB;
    scored += (std::max(0, len - window) + kKB - 1) / kKB;
  }
  const double queue1 = std::max(1., 0.8 * (double)(rows * Hkv) / 148.), queue2 = std::max(1., 0.8 * (double)(scored * Hkv) / 148.);
  const double steps = (double)((max_len(b) + kKB - 1) / kKB) * queue1 + 1.12 * row_blocks * queue2;
  return 9. + (0.4 + 0.031 * d) * steps + 0.8 * (double)((rows + keys) * Hkv) / 148.;
}

static purekv_status launch_score_cluster_f32(const float* q, const float* k, float* c_out, const purekv_batch* b,
                                              int32_t window, int32_t obs, int32_t pool, int32_t H, int32_t Hkv, int32_t d,
                                              float scale, cudaStream_t sm, bool* launched) {
  static std::atomic<uint64_t> smem_allowed{0}, wide_allowed{0};
  const purekv_status st = allow_wide_clusters(score_cluster_f32_kernel, smem_allowed, wide_allowed);
  if (st != PUREKV_OK) return st;
  const int32_t C = std::max(1, (max_len(b) + kKB - 1) / kKB), row_blocks = ((H / Hkv) * obs + kRB - 1) / kRB;
  ClusterLaunch l(C, Hkv, b->n_req, kThreads, (size_t)(kKB + 2 * kRB) * (d + 4) * sizeof(float), sm);
  const int32_t at_once = clusters_at_once(score_cluster_f32_kernel, l.cfg);
  *launched = at_once >= 1 && cluster_f32_us(C, d, live_requests(b, window) * Hkv, at_once, row_blocks) <=
                                  separate_f32_us(b, window, obs, H, Hkv, d, row_blocks);
  if (!*launched) return PUREKV_OK;
  PK_CUDA(cudaLaunchKernelEx(&l.cfg, score_cluster_f32_kernel, q, k, b->cu_seqlens, window, obs, pool, H, Hkv, d,
                             scale * 1.4426950408889634f, b->total_tokens, c_out));
  return PUREKV_OK;
}

// `obs` = accumulated rows per request and head (Eq. 2: the window itself); the first pass and the merge see only
// rows, so they take it in place of the window.
static purekv_status launch_score_mma(const void* q, const void* k, float* c_out, const purekv_batch* b, int32_t window,
                                      int32_t obs, int32_t H, int32_t Hkv, int32_t d, float scale, float* ws_f,
                                      cudaStream_t sm) {
  const int32_t ml = max_len(b);
  const int32_t n_kb = (ml + kMmaKeys - 1) / kMmaKeys, rows_max = (H / Hkv) * obs;
  float* lse2 = ws_f;                                                             // [n_req][H][obs]
  // the pairs start on a 256-byte boundary behind the log-sum-exp values
  float2* partial = reinterpret_cast<float2*>(ws_f + (((int64_t)b->n_req * H * obs + 63) & ~(int64_t)63));  // [n_req][Hkv][n_kb][rows_max]
  const size_t smem = (size_t)(kCtaKeys + 2 * kMmaRows) * (d + 8) * sizeof(__nv_bfloat16);  // K block + two Q blocks
  {
    static std::atomic<uint64_t> smem_allowed{0};
    const purekv_status st_smem = allow_max_dynamic_smem(score_mma_partial_kernel, smem_allowed);
    if (st_smem != PUREKV_OK) return st_smem;
  }
  {
    static std::atomic<uint64_t> smem_allowed{0};
    const purekv_status st_smem = allow_max_dynamic_smem(score_mma_colsum_kernel, smem_allowed);
    if (st_smem != PUREKV_OK) return st_smem;
  }
  const float scale_log2 = scale * 1.4426950408889634f;
  dim3 grid((unsigned)((ml + kCtaKeys - 1) / kCtaKeys), (unsigned)Hkv, (unsigned)b->n_req);
  score_mma_partial_kernel<<<grid, kMmaThreads, smem, sm>>>((const __nv_bfloat16*)q, (const __nv_bfloat16*)k, b->cu_seqlens,
                                                            obs, H, Hkv, d, scale_log2, n_kb, rows_max, partial);
  PK_CUDA(cudaGetLastError());
  const int64_t n_lse = (int64_t)b->n_req * H * obs;
  score_lse_merge_kernel<<<(unsigned)((n_lse + 255) / 256), 256, 0, sm>>>(partial, b->cu_seqlens, obs, H, Hkv, n_kb,
                                                                         rows_max, b->n_req, lse2);
  PK_CUDA(cudaGetLastError());
  score_mma_colsum_kernel<<<grid, kMmaThreads, smem, sm>>>((const __nv_bfloat16*)q, (const __nv_bfloat16*)k, b->cu_seqlens,
                                                           window, obs, H, Hkv, d, scale_log2, lse2, b->total_tokens, c_out);
  PK_CUDA(cudaGetLastError());
  return PUREKV_OK;
}

template <typename T>
static purekv_status launch_score(const void* q, const void* k, float* c_out, const purekv_batch* b, int32_t window,
                                  int32_t obs, int32_t H, int32_t Hkv, int32_t d, float scale, float* lse2,
                                  cudaStream_t sm) {
  const int32_t ml = max_len(b);
  const int32_t w = std::min(obs, ml);  // accumulated rows per head: the row blocks of the first pass
  const int32_t G = H / Hkv;
  const size_t smem = (size_t)(kRB + kKB) * (d + 4) * sizeof(float);
  {
    static std::atomic<uint64_t> smem_allowed{0};
    const purekv_status st_smem = allow_max_dynamic_smem(score_lse_kernel<T>, smem_allowed);
    if (st_smem != PUREKV_OK) return st_smem;
  }
  {
    static std::atomic<uint64_t> smem_allowed{0};
    const purekv_status st_smem = allow_max_dynamic_smem(score_colsum_kernel<T>, smem_allowed);
    if (st_smem != PUREKV_OK) return st_smem;
  }
  const float scale_log2 = scale * 1.4426950408889634f;
  dim3 g1((unsigned)((G * w + kRB - 1) / kRB), (unsigned)Hkv, (unsigned)b->n_req);
  score_lse_kernel<T><<<g1, kThreads, smem, sm>>>((const T*)q, (const T*)k, b->cu_seqlens, obs, H, Hkv, d, scale_log2,
                                                  lse2);
  PK_CUDA(cudaGetLastError());
  dim3 g2((unsigned)((ml + kKB - 1) / kKB), (unsigned)Hkv, (unsigned)b->n_req);
  score_colsum_kernel<T><<<g2, kThreads, smem, sm>>>((const T*)q, (const T*)k, b->cu_seqlens, window, obs, H, Hkv, d,
                                                     scale_log2, lse2, b->total_tokens, c_out);
  PK_CUDA(cudaGetLastError());
  return PUREKV_OK;
}

// Average pooling of the scores along the key axis (the pooled observation window of App. A.1's policies): each
// non-recent key takes the mean over `pool` positions centred on it, positions outside the non-recent segment
// counting as zero.  grid (key blocks of 256 over the longest request, n_kv_heads, n_req).
__global__ void __launch_bounds__(256) score_pool_kernel(const float* __restrict__ c_in, const int32_t* __restrict__ cu_seqlens,
                                                         int32_t window, int32_t pool, int64_t n_tokens,
                                                         float* __restrict__ c_out) {
  const int32_t r = blockIdx.z, g = blockIdx.y, j = blockIdx.x * 256 + threadIdx.x;
  const int32_t base = cu_seqlens[r], len = cu_seqlens[r + 1] - base;
  if (j >= len) return;
  const int32_t nr = len - min(window, len), half = pool / 2;
  const float* in = c_in + (int64_t)g * n_tokens + base;
  float sum = 0.f;
  if (j < nr)
    for (int32_t jj = max(0, j - half); jj <= min(nr - 1, j + half); ++jj) sum += in[jj];
  c_out[(int64_t)g * n_tokens + base + j] = sum / (float)(2 * half + 1);
}

// the last `obs` rows of every request are accumulated; < 0 or beyond the longest request: all rows
static int32_t obs_stride(const purekv_batch* b, int32_t obs_rows) {
  const int32_t ml = std::max(max_len(b), 1);
  return (obs_rows < 0 || obs_rows > ml) ? ml : std::max(obs_rows, 1);
}

// floats of log-sum-exp values per (request, head, accumulated row), plus (max, sum) pairs per 64-key block for
// the tensor-core path
static size_t score_ws_floats(const purekv_batch* batch, int32_t obs, int32_t n_q_heads) {
  const size_t rows = (size_t)batch->n_req * n_q_heads * (size_t)std::max(obs, 1);
  const size_t n_kb = ((size_t)max_len(batch) + kMmaKeys - 1) / kMmaKeys;
  return ((rows + 63) & ~(size_t)63) + rows * 2 * n_kb;
}

}  // namespace purekv

using namespace purekv;

extern "C" size_t purekv_score_ws_bytes(const purekv_batch* batch, int32_t window, int32_t n_q_heads) {
  if (!batch || window < 0 || n_q_heads < 0 || !batch->h_cu_seqlens) return 0;
  return score_ws_floats(batch, window, n_q_heads) * sizeof(float) + 256;
}

extern "C" size_t purekv_score_ex_ws_bytes(const purekv_batch* batch, int32_t obs_rows, int32_t pool, int32_t n_q_heads,
                                           int32_t n_kv_heads) {
  if (!batch || n_q_heads < 0 || n_kv_heads < 0 || !batch->h_cu_seqlens) return 0;
  size_t floats = score_ws_floats(batch, obs_stride(batch, obs_rows), n_q_heads);
  if (pool > 1) floats += (((size_t)n_kv_heads * batch->total_tokens) + 63) & ~(size_t)63;  // the scores before pooling
  return floats * sizeof(float) + 256;
}

// Common body of the score entry points: `obs_rows` accumulated rows (Eq. 2: the window), then pooling.
static purekv_status score_impl(const char* who, const void* q, const void* k, float* c_out, const purekv_batch* batch,
                                int32_t window, int32_t obs_rows, int32_t pool, int32_t n_q_heads, int32_t n_kv_heads,
                                int32_t head_dim, purekv_dtype dtype, float softmax_scale, void* ws, size_t ws_bytes,
                                size_t ws_need, void* stream) {
  purekv_status st = check_batch(batch, true);
  if (st != PUREKV_OK) return st;
  if (batch->total_tokens == 0 || batch->n_req == 0) return PUREKV_OK;  // empty batch: nothing to do
  PK_REQUIRE(q && k && c_out, PUREKV_ERR_INVALID_ARG, "%s: null pointer", who);
  PK_REQUIRE(n_q_heads >= 1 && n_kv_heads >= 1 && n_q_heads % n_kv_heads == 0, PUREKV_ERR_INVALID_ARG,
             "n_q_heads %d must be a positive multiple of n_kv_heads %d", n_q_heads, n_kv_heads);
  PK_REQUIRE(window >= 1, PUREKV_ERR_INVALID_ARG, "window must be >= 1");
  PK_REQUIRE(pool >= 1 && pool % 2 == 1, PUREKV_ERR_INVALID_ARG, "pool %d must be odd and >= 1", pool);
  PK_REQUIRE(head_dim >= 4 && head_dim % 4 == 0 && head_dim <= 256, PUREKV_ERR_UNSUPPORTED,
             "head_dim %d: need a multiple of 4 up to 256", head_dim);
  PK_REQUIRE(dtype == PUREKV_BF16 || dtype == PUREKV_FP32, PUREKV_ERR_INVALID_ARG, "unknown dtype");
  PK_REQUIRE(n_kv_heads <= 65535 && batch->n_req <= 65535, PUREKV_ERR_UNSUPPORTED, "too many heads or requests");
  PK_REQUIRE(ws && ws_bytes >= ws_need, PUREKV_ERR_WORKSPACE, "%s: workspace of %zu bytes is too small (need %zu)", who,
             ws_bytes, ws_need);
  const int32_t obs = obs_stride(batch, obs_rows);
  float* lse2 = (float*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
  float* c_raw = pool > 1 ? lse2 + score_ws_floats(batch, obs, n_q_heads) : c_out;  // scores before pooling
  const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)head_dim);
  cudaStream_t sm = (cudaStream_t)stream;
  // One launch when a cluster holds the longest request and the accumulated rows are not the whole of a long one (every block
  // of rows costs a cluster barrier, and rows before a CTA's keys are multiplied for nothing), and that is the faster form.
  const int32_t ml = max_len(batch), row_blocks = ((n_q_heads / n_kv_heads) * obs + kMmaRows - 1) / kMmaRows;
  bool launched = false;
  if (dtype == PUREKV_BF16 && head_dim % 16 == 0 && head_dim <= 128 && ml <= kClusterMax * 2 * kCtaKeys &&
      row_blocks <= kClusterRowBlocks && pool / 2 <= kPoolHalfMax)
    st = launch_score_cluster(q, k, c_out, batch, window, obs, pool, n_q_heads, n_kv_heads, head_dim, scale, sm, &launched);
  if (dtype == PUREKV_FP32 && ml <= kClusterMax * kKB && row_blocks <= kClusterRowBlocks && pool / 2 <= kKB / 2 &&
      ((uintptr_t)q | (uintptr_t)k) % 16 == 0)
    st = launch_score_cluster_f32((const float*)q, (const float*)k, c_out, batch, window, obs, pool, n_q_heads, n_kv_heads,
                                  head_dim, scale, sm, &launched);
  if (st != PUREKV_OK || launched) return st;  // (a device that cannot place one such cluster takes the separate kernels)
  if (dtype == PUREKV_BF16 && head_dim % 16 == 0)
    st = launch_score_mma(q, k, c_raw, batch, window, obs, n_q_heads, n_kv_heads, head_dim, scale, lse2, sm);
  else if (dtype == PUREKV_BF16)
    st = launch_score<__nv_bfloat16>(q, k, c_raw, batch, window, obs, n_q_heads, n_kv_heads, head_dim, scale, lse2, sm);
  else
    st = launch_score<float>(q, k, c_raw, batch, window, obs, n_q_heads, n_kv_heads, head_dim, scale, lse2, sm);
  if (st != PUREKV_OK || pool == 1) return st;
  dim3 grid((unsigned)((max_len(batch) + 255) / 256), (unsigned)n_kv_heads, (unsigned)batch->n_req);
  score_pool_kernel<<<grid, 256, 0, sm>>>(c_raw, batch->cu_seqlens, window, pool, batch->total_tokens, c_out);
  PK_CUDA(cudaGetLastError());
  return PUREKV_OK;
}

extern "C" purekv_status purekv_lowlayer_score(const void* q, const void* k, float* c_out, const purekv_batch* batch,
                                               int32_t window, int32_t n_q_heads, int32_t n_kv_heads,
                                               int32_t head_dim, purekv_dtype dtype, float softmax_scale, void* ws,
                                               size_t ws_bytes, void* stream) {
  if (batch && batch->h_cu_seqlens && window >= 1 && n_q_heads >= 1)
    return score_impl("purekv_lowlayer_score", q, k, c_out, batch, window, window, 1, n_q_heads, n_kv_heads, head_dim, dtype,
                      softmax_scale, ws, ws_bytes, purekv_score_ws_bytes(batch, window, n_q_heads), stream);
  return score_impl("purekv_lowlayer_score", q, k, c_out, batch, window, window, 1, n_q_heads, n_kv_heads, head_dim, dtype,
                    softmax_scale, ws, ws_bytes, 0, stream);
}

extern "C" purekv_status purekv_lowlayer_score_ex(const void* q, const void* k, float* c_out, const purekv_batch* batch,
                                                  int32_t window, int32_t obs_rows, int32_t pool, int32_t n_q_heads,
                                                  int32_t n_kv_heads, int32_t head_dim, purekv_dtype dtype,
                                                  float softmax_scale, void* ws, size_t ws_bytes, void* stream) {
  const size_t need = (batch && batch->h_cu_seqlens && n_q_heads >= 1 && n_kv_heads >= 1)
                          ? purekv_score_ex_ws_bytes(batch, obs_rows, pool, n_q_heads, n_kv_heads) : 0;
  return score_impl("purekv_lowlayer_score_ex", q, k, c_out, batch, window, obs_rows, pool, n_q_heads, n_kv_heads, head_dim,
                    dtype, softmax_scale, ws, ws_bytes, need, stream);
}

// Device address of the static scratch array on the current device; resolved on the first call per device.
static purekv_status noalloc_scratch(float** out) {
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static float* ptrs[kMaxDevices] = {};
  int dev = -1;
  PK_CUDA(cudaGetDevice(&dev));
  PK_REQUIRE(dev >= 0 && dev < kMaxDevices, PUREKV_ERR_UNSUPPORTED, "device ordinal %d is beyond %d", dev, kMaxDevices);
  std::lock_guard<std::mutex> lock(mu);
  if (!ptrs[dev]) {
    float* p = nullptr;
    PK_CUDA(cudaGetSymbolAddress((void**)&p, g_noalloc_score_scratch));
    PK_REQUIRE(p != nullptr, PUREKV_ERR_CUDA, "cudaGetSymbolAddress returned a null scratch address");
    ptrs[dev] = p;
  }
  *out = ptrs[dev];
  return PUREKV_OK;
}

extern "C" purekv_status purekv_lowlayer_score_noalloc(const void* q, const void* k, float* c_out,
                                                       const purekv_batch* batch, int32_t window, int32_t n_q_heads,
                                                       int32_t n_kv_heads, int32_t head_dim, purekv_dtype dtype,
                                                       float softmax_scale, void* stream) {
  purekv_status st = check_batch(batch, true);
  if (st != PUREKV_OK) return st;
  if (batch->total_tokens == 0 || batch->n_req == 0) return PUREKV_OK;  // empty batch: nothing to do
  PK_REQUIRE(window >= 1 && n_q_heads >= 1, PUREKV_ERR_INVALID_ARG, "window and n_q_heads must be >= 1");
  const size_t need = (purekv_score_ws_bytes(batch, window, n_q_heads) - 256) / sizeof(float);
  PK_REQUIRE(need <= kNoallocScoreFloats, PUREKV_ERR_WORKSPACE,
             "purekv_lowlayer_score_noalloc: this problem needs %zu scratch values, the built-in scratch holds %zu; "
             "use purekv_lowlayer_score with a caller-provided workspace",
             need, kNoallocScoreFloats);
  float* scratch = nullptr;
  if ((st = noalloc_scratch(&scratch)) != PUREKV_OK) return st;
  // The scratch needs no clearing: every entry that a later kernel of the call reads is written earlier in the call.
  return purekv_lowlayer_score(q, k, c_out, batch, window, n_q_heads, n_kv_heads, head_dim, dtype, softmax_scale,
                               scratch, (kNoallocScoreFloats + 64) * sizeof(float), stream);
}
