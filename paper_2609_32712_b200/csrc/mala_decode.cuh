// Split-KV decode ("Fused decoding execution"): the persistent split kernel lives in
// mala_decode_split.cuh; this file holds the normalizer-aware merge of the split partials, the
// workspace layout and the launch code.
#pragma once
#include <cuda_runtime.h>

#include "../../include/mala.h"
#include "mala_decode_split.cuh"
#include "mala_decode_fp8.cuh"
#include "tensor_map.h"

namespace mala {

// lse = log sum_s exp(lse_s), o = sum_s exp(lse_s - lse) o_s; one block of four warps per (b, token, query head).
// Bound by the latency of the partials' loads, so they are spread out: the log-normalizers are read by the whole block at
// once, and each warp accumulates every fourth split, a 16-byte load per lane and four splits in flight, before the warps'
// sums meet in shared memory.  With one thread per column walking the splits (21.6 us for 256 rows x 128 splits, 10 us for
// 512 x 28) a step took 629 and 93.4 us (8 x 131072 keys; four tokens over 4 x 16389 keys), now 624 and 87.8.
// Launched as a dependent of the split kernel: it may be resident before that kernel has finished and waits here (and reads
// past the L1, which may hold lines from before).
template <int D>
__global__ void __launch_bounds__(128)
decode_merge_kernel(const float* __restrict__ o_part, const float* __restrict__ lse_part, __nv_bfloat16* __restrict__ o,
                    int64_t o_sb, int64_t o_sn, int64_t o_sh, float* __restrict__ lse_out, int Sq, int Hq,
                    int num_splits, int d) {   // d <= D: columns of o
  constexpr int L4 = D / 4;                      // float4 per partial: one or two per lane, or half a warp per partial
  constexpr int V = L4 > 32 ? L4 / 32 : 1, PER = L4 < 32 ? 32 / L4 : 1;   // vectors per lane, partials per warp step
  __shared__ float red[4];
  __shared__ __align__(16) float sum[4 * PER][D];
  const int bh = blockIdx.x, h = bh % Hq, tok = (bh / Hq) % Sq, b = bh / (Hq * Sq), lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int sub = lane / (32 / PER), col = lane % (32 / PER);
  const float* lp = lse_part + (size_t)bh * num_splits;
  const float4* op = reinterpret_cast<const float4*>(o_part + (size_t)bh * num_splits * D) + col;
  wait_for_primary();
  float mx = -INFINITY;
  for (int s = threadIdx.x; s < num_splits; s += 128) mx = fmaxf(mx, __ldcg(lp + s));
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
  if (lane == 0) red[w] = mx;
  __syncthreads();
  mx = fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
  float Z = 0.f;
  float4 acc[V];
#pragma unroll
  for (int v = 0; v < V; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int s0 = w * PER + sub; s0 < num_splits; s0 += 16 * PER) {
    float ls[4];
    float4 x[4][V];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int s = s0 + u * 4 * PER;
      ls[u] = s < num_splits ? __ldcg(lp + s) : -INFINITY;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < V; ++v) {
        x[u][v] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ls[u] != -INFINITY) x[u][v] = __ldcg(op + (size_t)(s0 + u * 4 * PER) * L4 + v * 32);
      }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float f = ls[u] != -INFINITY ? exp2f((ls[u] - mx) * 1.4426950408889634f) : 0.f;
      Z += f;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        acc[v].x += f * x[u][v].x; acc[v].y += f * x[u][v].y; acc[v].z += f * x[u][v].z; acc[v].w += f * x[u][v].w;
      }
    }
  }
#pragma unroll
  for (int v = 0; v < V; ++v) *reinterpret_cast<float4*>(&sum[w * PER + sub][(v * 32 + col) * 4]) = acc[v];
  __syncthreads();                               // (red has been read by everyone; the columns are in place)
  float Zw = Z;
  if constexpr (PER > 1) Zw += __shfl_xor_sync(0xffffffffu, Zw, 16);
  if (lane == 0) red[w] = Zw;
  __syncthreads();
  Z = (red[0] + red[1]) + (red[2] + red[3]);
  // (a sequence without keys has no split with mass: its output is 0 and its log-normalizer -inf; so it is with a
  // normalizer that is not a number, whose sums must not reach the output)
  const bool any = Z > 0.f;
  const float inv = any ? 1.f / Z : 0.f;
  for (int c = threadIdx.x; c < d; c += 128) {
    float t = 0.f;
#pragma unroll
    for (int x = 0; x < 4 * PER; ++x) t += sum[x][c];
    o[b * o_sb + tok * o_sn + h * o_sh + c] = __float2bfloat16(any ? t * inv : 0.f);
  }
  if (lse_out && threadIdx.x == 0) lse_out[bh] = any ? mx + logf(Z) : -INFINITY;
}

// The same for up to 32 splits, one warp per (b, token, query head) and eight of them per block.  With few splits the
// block above is bound by its own latency -- three barriers, the log-normalizers read twice, three warps without a split --
// and thousands of rows take many rounds of such blocks.  Here nothing crosses between warps, the log-normalizers are read
// once (lane s: split s) and the first partials are requested along with them.  16416 rows of one split, 128 columns: 7.5 us
// (12.6 MB of partials and outputs), 23 with the block above, 18 with a thread per column.
template <int D>
__global__ void __launch_bounds__(256)
decode_merge_few_kernel(const float* __restrict__ o_part, const float* __restrict__ lse_part, __nv_bfloat16* __restrict__ o,
                        int64_t o_sb, int64_t o_sn, int64_t o_sh, float* __restrict__ lse_out, int rows, int Sq, int Hq,
                        int num_splits, int d) {
  constexpr uint32_t kAll = 0xffffffffu;
  constexpr int L4 = D / 4, V = L4 > 32 ? L4 / 32 : 1, PER = L4 < 32 ? 32 / L4 : 1;   // (as above)
  const int bh = blockIdx.x * 8 + (threadIdx.x >> 5), h = bh % Hq, tok = (bh / Hq) % Sq, b = bh / (Hq * Sq);
  const int lane = threadIdx.x & 31, sub = lane / (32 / PER), col = lane % (32 / PER);
  if (bh >= rows) return;
  const float4* op = reinterpret_cast<const float4*>(o_part + (size_t)bh * num_splits * D) + col;
  wait_for_primary();
  const float ls = lane < num_splits ? __ldcg(lse_part + (size_t)bh * num_splits + lane) : -INFINITY;
  float mx = 0.f, wt = 0.f, Z = 0.f;
  float4 acc[V];
#pragma unroll
  for (int v = 0; v < V; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int s0 = 0; s0 < num_splits; s0 += 4 * PER) {
    float4 x[4][V];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int s = s0 + u * PER + sub;
        x[u][v] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s < num_splits) x[u][v] = __ldcg(op + (size_t)s * L4 + v * 32);
      }
    if (s0 == 0) {
      mx = ls;
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kAll, mx, m));
      wt = ls != -INFINITY ? exp2f((ls - mx) * 1.4426950408889634f) : 0.f;
      Z = wt;
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) Z += __shfl_xor_sync(kAll, Z, m);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float f = __shfl_sync(kAll, wt, (s0 + u * PER + sub) & 31);
      if (f != 0.f) {                            // (an empty split's partial is not read into the sums)
#pragma unroll
        for (int v = 0; v < V; ++v) {
          acc[v].x += f * x[u][v].x; acc[v].y += f * x[u][v].y; acc[v].z += f * x[u][v].z; acc[v].w += f * x[u][v].w;
        }
      }
    }
  }
  const bool any = Z > 0.f;                      // (as above)
  const float inv = any ? 1.f / Z : 0.f;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if constexpr (PER > 1) {
      acc[v].x += __shfl_xor_sync(kAll, acc[v].x, 16); acc[v].y += __shfl_xor_sync(kAll, acc[v].y, 16);
      acc[v].z += __shfl_xor_sync(kAll, acc[v].z, 16); acc[v].w += __shfl_xor_sync(kAll, acc[v].w, 16);
    }
    if (!any) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (sub == 0 && (v * 32 + col) * 4 < d)
      *reinterpret_cast<uint2*>(o + b * o_sb + tok * o_sn + h * o_sh + (v * 32 + col) * 4) =
          make_uint2(pack_bf16x2(acc[v].x * inv, acc[v].y * inv), pack_bf16x2(acc[v].z * inv, acc[v].w * inv));
  }
  if (lse_out && lane == 0) lse_out[bh] = any ? mx + logf(Z) : -INFINITY;
}

// The merge as a programmatic dependent of the split kernel before it on the stream (which has let it go ahead): its
// launch latency passes while the split kernel still runs.
inline int launch_decode_merge(int D, int rows, const float* o_part, const float* lse_part, mala_tout o, int64_t o_sn,
                               float* lse_opt, int Sq, int Hq, int num_splits, int d, cudaStream_t stream) {
  // Up to twelve splits (three rounds of four loads) a warp per row is the faster form at every number of rows; a step of
  // 128 / 4096 rows with one tile per split takes 7.9 / 16.3 us instead of 8.6 / 20.1 (one split), 12.2 / 101.9 instead
  // of 12.4 / 106.1 (twelve), 12.4 / 133.5 instead of 12.4 / 136.8 (sixteen) and 17.9 instead of 17.2 (32 splits, 128 rows).
  if (num_splits <= 12) {
    auto few = D == 256 ? decode_merge_few_kernel<256> : D == 128 ? decode_merge_few_kernel<128> : decode_merge_few_kernel<64>;
    return launch_dependent(few, dim3((unsigned)((rows + 7) / 8)), dim3(256), stream, o_part, lse_part, (__nv_bfloat16*)o.p,
                            o.sb, o_sn, o.sh, lse_opt, rows, Sq, Hq, num_splits, d) == cudaSuccess ? MALA_OK : MALA_ERR_CUDA;
  }
  auto kernel = D == 256 ? decode_merge_kernel<256> : D == 128 ? decode_merge_kernel<128> : decode_merge_kernel<64>;
  return launch_dependent(kernel, dim3((unsigned)rows), dim3(128), stream, o_part, lse_part, (__nv_bfloat16*)o.p, o.sb, o_sn,
                          o.sh, lse_opt, Sq, Hq, num_splits, d) == cudaSuccess ? MALA_OK : MALA_ERR_CUDA;
}

inline size_t decode_align256(size_t x) { return (x + 255) & ~(size_t)255; }

// (B: sequences x new tokens per sequence)
inline size_t decode_workspace_bytes(int B, int Hq, int d, int S) {   // d: the padded head size
  return decode_align256((size_t)B * Hq * S * d * sizeof(float)) + decode_align256((size_t)B * Hq * S * sizeof(float));
}

inline bool decode_set_attributes() {
  bool ok = true;
#define MALA_DEC_ATTR(DENSE, GP, MULTI, SCHED) \
  ok = ok && cudaFuncSetAttribute(mala_decode_split_kernel<DENSE, GP, MULTI, 128, SCHED>, cudaFuncAttributeMaxDynamicSharedMemorySize, DecCfg::kSmemBytes) == cudaSuccess; \
  ok = ok && cudaFuncSetAttribute(mala_decode_split_kernel<DENSE, GP, MULTI, 64, SCHED>, cudaFuncAttributeMaxDynamicSharedMemorySize, DecCfg::kSmemBytes) == cudaSuccess; \
  ok = ok && cudaFuncSetAttribute(mala_decode_split_kernel<DENSE, GP, MULTI, 256, SCHED>, cudaFuncAttributeMaxDynamicSharedMemorySize, DecCfgT<256>::kSmemBytes) == cudaSuccess;
#define MALA_DEC_ATTR_S(GP, SCHED) MALA_DEC_ATTR(false, GP, false, SCHED) MALA_DEC_ATTR(true, GP, false, SCHED) MALA_DEC_ATTR(false, GP, true, SCHED) MALA_DEC_ATTR(true, GP, true, SCHED)
#define MALA_DEC_ATTR_GP(GP) MALA_DEC_ATTR_S(GP, false) MALA_DEC_ATTR_S(GP, true)
  MALA_DEC_ATTR_GP(1) MALA_DEC_ATTR_GP(2) MALA_DEC_ATTR_GP(4) MALA_DEC_ATTR_GP(8) MALA_DEC_ATTR_GP(16)
#define MALA_F8_ATTR1(DENSE, ...) \
  ok = ok && cudaFuncSetAttribute(mala_decode_fp8_kernel<DENSE, __VA_ARGS__>, cudaFuncAttributeMaxDynamicSharedMemorySize, DecF8Cfg<2, DENSE>::kSmemBytes) == cudaSuccess;
#define MALA_F8_ATTR(DENSE, GP) MALA_F8_ATTR1(DENSE, GP, false) MALA_F8_ATTR1(DENSE, GP, false, 2, false, true)
#define MALA_F8_ATTR_S(DENSE, GP, SCHED) \
  MALA_F8_ATTR1(DENSE, GP, true, 2, false, false, SCHED) MALA_F8_ATTR1(DENSE, GP, true, 2, true, false, SCHED)
#define MALA_F8_ATTR_GP(GP) \
  MALA_F8_ATTR(false, GP) MALA_F8_ATTR_S(false, GP, false) MALA_F8_ATTR_S(false, GP, true) \
  MALA_F8_ATTR(true, GP) MALA_F8_ATTR_S(true, GP, false) MALA_F8_ATTR_S(true, GP, true)
  MALA_F8_ATTR_GP(1) MALA_F8_ATTR_GP(2) MALA_F8_ATTR_GP(4) MALA_F8_ATTR_GP(8)
#undef MALA_F8_ATTR_GP
#undef MALA_F8_ATTR_S
#undef MALA_F8_ATTR1
#undef MALA_F8_ATTR
#undef MALA_DEC_ATTR_GP
#undef MALA_DEC_ATTR_S
#undef MALA_DEC_ATTR
  return ok;
}

// A cache held in pages: kc / vc are [num_pages, page_size, Hkv, d] (sb = page stride), sequence b keeps its keys
// 128*x .. in page block_table[b * bt_stride + x / (page_size / 128)], and holds seqlens[b] <= Nk keys.
struct DecPaging {
  const int* block_table;   // null: one contiguous cache per sequence
  const int* seqlens;       // null: every sequence holds Nk keys
  int bt_stride, page_size, num_pages;
};

// Launches the split kernel and the merge on `stream`.  o_part / lse_part: caller-provided scratch of
// decode_workspace_bytes() bytes in total (o_part first).  Nk: the longest cache (the splits are laid out for it).
inline int decode_launch_with_scratch(mala_tin q, mala_tin kc, mala_tin vc, mala_tout o, float* lse_opt,
                                      const mala_stats* st, int B, int Hq, int Hkv, int Nk, int d, float scale,
                                      float tau, int num_splits, float* o_part, float* lse_part, int* status,
                                      cudaStream_t stream, const DecPaging* pg = nullptr, int Sq = 1) {
  if (!head_size_ok(d, 256)) return MALA_ERR_UNSUPPORTED;
  const int D = padded_head_size(d);
  const int G = Hq / Hkv;
  if (Sq < 1 || G * Sq > 16 || Sq > Nk) return MALA_ERR_UNSUPPORTED;
  const bool paged = pg && pg->block_table;
  // pages of whole tiles, or 8, 16, 32 or 64 keys (a tile is then put together from several pages)
  if (paged && (pg->page_size < 8 || (pg->page_size % 128 != 0 && 128 % pg->page_size != 0) || pg->num_pages <= 0 ||
                pg->bt_stride <= 0))
    return MALA_ERR_UNSUPPORTED;
  const int box_rows = paged && pg->page_size < 128 ? pg->page_size : 128;
  const int per = (Nk + num_splits - 1) / num_splits;
  const int tps = (per + 127) / 128;
  if ((long long)B * Hkv * num_splits > 0x7fffffffLL) return MALA_ERR_UNSUPPORTED;

  CUtensorMap tq, tk, tv;
  // q [B,Sq,Hq,d]: one box of the group's G heads x Sq tokens
  if (!make_tensor_map_q_rows(&tq, q.p, B, Sq, Hq, d, q.sb, Sq > 1 ? q.sn : 0, q.sh, G) ||
      !make_tensor_map_bnhd(&tk, kc.p, paged ? pg->num_pages : B, paged ? pg->page_size : Nk, Hkv, d, kc.sb, kc.sn,
                            kc.sh, box_rows) ||
      !make_tensor_map_bnhd(&tv, vc.p, paged ? pg->num_pages : B, paged ? pg->page_size : Nk, Hkv, d, vc.sb, vc.sn,
                            vc.sh, box_rows))
    return MALA_ERR_TENSOR_MAP;

  DecParams p;
  p.o_part = o_part; p.lse_part = lse_part;
  p.retained = st ? st->retained_per_block : nullptr;
  p.bitmask = st ? st->tile_bitmask : nullptr;
  p.totals = st ? (unsigned long long*)st->totals : nullptr;
  p.status = status;
  p.seqlens = pg ? pg->seqlens : nullptr;
  p.block_table = paged ? pg->block_table : nullptr;
  p.bt_stride = paged ? pg->bt_stride : 0;
  p.tpp = paged && pg->page_size >= 128 ? pg->page_size / 128 : 1;
  p.ppt = 128 / box_rows;
  p.prows = box_rows;
  p.Sq = Sq;
  p.B = B; p.Hq = Hq; p.Hkv = Hkv; p.Nk = Nk; p.tps = tps; p.num_splits = num_splits; p.words = (tps + 31) / 32;
  p.n_items = B * Hkv * num_splits;
  p.by_splits.set((uint32_t)num_splits);
  p.by_hkv.set((uint32_t)Hkv);
  p.by_tps.set((uint32_t)p.tps);
  p.scale_log2 = scale * 1.4426950408889634f;
  p.log2_tau = tau > 0.f ? log2f(tau) : -INFINITY;
  if (p.bitmask &&
      cudaMemsetAsync(p.bitmask, 0, (size_t)B * Hkv * num_splits * p.words * sizeof(uint32_t), stream) != cudaSuccess)
    return MALA_ERR_CUDA;

  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
    return MALA_ERR_CUDA;
  const int grid = p.n_items < sms ? p.n_items : sms;   // persistent: one CTA per SM
  const bool sched = p.seqlens && decode_sched_fits(B, p.n_items, grid, 1, D == 256 ? DecCfgT<256>::kSchedItems : DecCfg::kSchedItems);
  const int R = G * Sq;   // rows of a work item
#define MALA_DEC_LAUNCH3(DENSE, GP, MULTI, SCHED)                                                                           \
  {                                                                                                                  \
    if (D == 256) mala_decode_split_kernel<DENSE, GP, MULTI, 256, SCHED><<<grid, DecCfg::kThreads, DecCfgT<256>::kSmemBytes, stream>>>(tq, tk, tv, p); \
    else if (D == 128) mala_decode_split_kernel<DENSE, GP, MULTI, 128, SCHED><<<grid, DecCfg::kThreads, DecCfg::kSmemBytes, stream>>>(tq, tk, tv, p); \
    else mala_decode_split_kernel<DENSE, GP, MULTI, 64, SCHED><<<grid, DecCfg::kThreads, DecCfg::kSmemBytes, stream>>>(tq, tk, tv, p);           \
  }
#define MALA_DEC_LAUNCH2(DENSE, GP, SCHED)            \
  {                                                   \
    if (Sq > 1) MALA_DEC_LAUNCH3(DENSE, GP, true, SCHED) \
    else MALA_DEC_LAUNCH3(DENSE, GP, false, SCHED)    \
  }
#define MALA_DEC_LAUNCH1(GP, SCHED)                   \
  {                                                   \
    if (tau == 0.f) MALA_DEC_LAUNCH2(true, GP, SCHED) \
    else MALA_DEC_LAUNCH2(false, GP, SCHED)           \
  }
#define MALA_DEC_LAUNCH(GP)                           \
  {                                                   \
    if (sched) MALA_DEC_LAUNCH1(GP, true)           \
    else MALA_DEC_LAUNCH1(GP, false)                  \
  }
  if (R <= 1) MALA_DEC_LAUNCH(1)
  else if (R <= 2) MALA_DEC_LAUNCH(2)
  else if (R <= 4) MALA_DEC_LAUNCH(4)
  else if (R <= 8) MALA_DEC_LAUNCH(8)
  else MALA_DEC_LAUNCH(16)
#undef MALA_DEC_LAUNCH
#undef MALA_DEC_LAUNCH1
#undef MALA_DEC_LAUNCH2
#undef MALA_DEC_LAUNCH3
  if (cudaGetLastError() != cudaSuccess) return MALA_ERR_CUDA;
  return launch_decode_merge(D, B * Sq * Hq, o_part, lse_part, o, Sq > 1 ? o.sn : 0, lse_opt, Sq, Hq, num_splits, d, stream);
}

// Decode over an e4m3 cache with one fp32 scale per (sequence, KV head, 128-key tile): kc / vc are 8-bit [B,Nk,Hkv,d]
// views (strides in elements), kscale / vscale fp32 [B,Hkv,ceil(Nk/128)].  Up to four query heads per KV head.
// pg != null: kc / vc are [num_pages, page_size, Hkv, d] (page_size a multiple of 128, or 16, 32 or 64), the scales
// [num_pages, Hkv, max(1, page_size/128)], and Nk = bt_stride * page_size lays out the splits.
inline int decode_fp8_launch(mala_tin q, mala_tin kc, mala_tin vc, const float* kscale, const float* vscale, mala_tout o,
                             float* lse_opt, const mala_stats* st, int B, int Hq, int Hkv, int Nk, int d, float scale,
                             float tau, int num_splits, void* ws, int* status, cudaStream_t stream,
                             const DecPaging* pg = nullptr, int Sq = 1) {
  const int G = Hq / Hkv;
  const int R = G * Sq;   // rows of a work item
  if (Sq < 1 || R > 8 || Sq > Nk || d % 16 != 0 || d > 128 || d < 16) return MALA_ERR_UNSUPPORTED;
  if (Sq > 1 && pg) return MALA_ERR_UNSUPPORTED;   // (several tokens per step: contiguous caches only)
  const bool small = pg && pg->page_size < 128;
  if (pg && !(pg->page_size % 128 == 0 || pg->page_size == 16 || pg->page_size == 32 || pg->page_size == 64))
    return MALA_ERR_UNSUPPORTED;
  const int box_rows = small ? pg->page_size : 128;
  const int per = (Nk + num_splits - 1) / num_splits;
  const int tps = (per + 127) / 128;
  if ((long long)B * Hkv * num_splits > 0x7fffffffLL || (long long)B * Hkv * ((Nk + 127) / 128) > 0x7fffffffLL)
    return MALA_ERR_UNSUPPORTED;
  CUtensorMap tq, tk, tv;
  if (!make_tensor_map_q_rows(&tq, q.p, B, Sq, Hq, d, q.sb, Sq > 1 ? q.sn : 0, q.sh, G) ||
      !make_tensor_map_u8_bnhd(&tk, kc.p, pg ? pg->num_pages : B, pg ? pg->page_size : Nk, Hkv, d, kc.sb, kc.sn, kc.sh, box_rows) ||
      !make_tensor_map_u8_bnhd(&tv, vc.p, pg ? pg->num_pages : B, pg ? pg->page_size : Nk, Hkv, d, vc.sb, vc.sn, vc.sh, box_rows))
    return MALA_ERR_TENSOR_MAP;
  DecF8Params p;
  p.block_table = pg ? pg->block_table : nullptr;
  p.seqlens = pg ? pg->seqlens : nullptr;
  p.num_pages = pg ? pg->num_pages : 0;
  p.max_pages = pg ? pg->bt_stride : 0;
  p.tpp = (pg && !small) ? pg->page_size / 128 : 1;
  p.by_tpp.set((uint32_t)p.tpp);
  p.ppt = 128 / box_rows;
  p.prows = box_rows;
  p.Sq = Sq;
  p.o_part = (float*)ws;
  p.lse_part = (float*)((uint8_t*)ws + decode_align256((size_t)B * Sq * Hq * num_splits * 128 * sizeof(float)));
  p.retained = st ? st->retained_per_block : nullptr;
  p.bitmask = st ? st->tile_bitmask : nullptr;
  p.totals = st ? (unsigned long long*)st->totals : nullptr;
  p.status = status;
  p.kscale = kscale; p.vscale = vscale;
  p.B = B; p.Hq = Hq; p.Hkv = Hkv; p.Nk = Nk; p.tps = tps; p.num_splits = num_splits; p.words = (tps + 31) / 32;
  p.n_items = B * Hkv * num_splits; p.nt = (Nk + 127) / 128;
  p.by_splits.set((uint32_t)num_splits);
  p.by_hkv.set((uint32_t)Hkv);
  p.by_tps.set((uint32_t)p.tps);
  p.scale_log2 = scale * 1.4426950408889634f;
  p.log2_tau = tau > 0.f ? log2f(tau) : -INFINITY;
  if (p.bitmask &&
      cudaMemsetAsync(p.bitmask, 0, (size_t)B * Hkv * num_splits * p.words * sizeof(uint32_t), stream) != cudaSuccess)
    return MALA_ERR_CUDA;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
    return MALA_ERR_CUDA;
  const int grid = p.n_items < sms ? p.n_items : sms;
  const bool sched = p.seqlens && decode_sched_fits(B, p.n_items, grid, 2, DecF8Cfg<2, false>::kSchedItems);   // (two streams)
#define MALA_F8_LAUNCH1(DENSE, GP, ...) \
  mala_decode_fp8_kernel<DENSE, GP, __VA_ARGS__><<<grid, DecF8Cfg<2, DENSE, (GP > 4)>::kThreads, DecF8Cfg<2, DENSE>::kSmemBytes, stream>>>(tq, tk, tv, p)
#define MALA_F8_LAUNCH2(DENSE, GP, SCHED)                                  \
  do {                                                                     \
    if (Sq > 1) MALA_F8_LAUNCH1(DENSE, GP, false, 2, false, true);         \
    else if (small) MALA_F8_LAUNCH1(DENSE, GP, true, 2, true, false, SCHED); \
    else if (pg) MALA_F8_LAUNCH1(DENSE, GP, true, 2, false, false, SCHED); \
    else MALA_F8_LAUNCH1(DENSE, GP, false);                                \
  } while (0)
#define MALA_F8_LAUNCH(GP)                                                 \
  do {                                                                     \
    if (tau == 0.f && sched) MALA_F8_LAUNCH2(true, GP, true);              \
    else if (tau == 0.f) MALA_F8_LAUNCH2(true, GP, false);                 \
    else if (sched) MALA_F8_LAUNCH2(false, GP, true);                      \
    else MALA_F8_LAUNCH2(false, GP, false);                                \
  } while (0)
  if (R <= 1) MALA_F8_LAUNCH(1);
  else if (R <= 2) MALA_F8_LAUNCH(2);
  else if (R <= 4) MALA_F8_LAUNCH(4);
  else MALA_F8_LAUNCH(8);
#undef MALA_F8_LAUNCH
#undef MALA_F8_LAUNCH2
#undef MALA_F8_LAUNCH1
  if (cudaGetLastError() != cudaSuccess) return MALA_ERR_CUDA;
  return launch_decode_merge(128, B * Sq * Hq, p.o_part, p.lse_part, o, Sq > 1 ? o.sn : 0, lse_opt, Sq, Hq, num_splits, d,
                             stream);
}

inline int decode_launch(mala_tin q, mala_tin kc, mala_tin vc, mala_tout o, float* lse_opt, const mala_stats* st, int B,
                         int Hq, int Hkv, int Nk, int d, float scale, float tau, int num_splits, void* ws, int* status,
                         cudaStream_t stream, const DecPaging* pg = nullptr, int Sq = 1) {
  float* o_part = (float*)ws;
  float* lse_part =
      (float*)((uint8_t*)ws + decode_align256((size_t)B * Sq * Hq * num_splits * padded_head_size(d) * sizeof(float)));
  return decode_launch_with_scratch(q, kc, vc, o, lse_opt, st, B, Hq, Hkv, Nk, d, scale, tau, num_splits, o_part,
                                    lse_part, status, stream, pg, Sq);
}

}  // namespace mala
