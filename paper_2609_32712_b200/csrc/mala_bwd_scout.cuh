// First pass of the MALA backward (Algorithm 2): the offline test of Eq. 4 for every legal tile, and nothing else.
//
// The backward test of a tile depends only on its scores and on the saved log-normalizers, not on any other tile, so
// the retained support of a key block can be found before any gradient work starts.  This kernel does that at the rate
// the tensor pipe forms the scores.  One CTA per (two or four key blocks, query head, batch) keeps the K tiles in shared memory
// and streams the head's Q tiles through a ring; a Q tile and a pair of key blocks make one MMA batch S = Q_i [K_j; K_j+1]^T of
// shape 128 x 256 into one of two TMEM buffers of 256 columns, and four warpgroups -- one per key block of a buffer -- read and
// test their score tile while the other buffer is being formed.  The queries are the rows: a thread owns one, and the test of its
// 128 scores is one comparison of their largest (max_e (s_e c2) >= bq <=> some s_e c2 >= bq; fma is monotone).
//
// Bound by the tensor pipe: 512 clk per tile.  Why this shape: a 128 x 128 MMA takes the whole bandwidth of shared memory and
// leaves none for the copies that refill the ring, a 128 x 256 MMA three quarters; a Q tile serves four score tiles, with 16 bytes of
// copies per clk and SM.  (With the keys as rows and pairs of Q tiles as columns it serves two, and every column has a threshold of
// its own: 8192 tokens, 16 / 4 heads of 128 columns, a third of the tiles retained: 157 us, now 98; 131072 tokens, 8 / 2 heads: 9.4
// and 8.9 ms, where the 1.55 PFLOP/s of tested tiles are what the power limit allows.)
// Nothing waits for a vote: a warp that finds a retained entry sets the tile's bit in a shared-memory copy of
// the row's mask, and the row is written out when the head's last tile has been tested.  The second pass
// (mala_bwd_kernel in its list mode) then visits the retained tiles only and runs the dense tile pipeline on them.
//
// Rows that retain everything gain nothing from a first pass (their scores would be formed twice), so the rows of a
// CTA are sampled first: two tiles of every sixteen.  If all of them are retained, for every key block of the CTA, the head's rows
// are left to the one-pass kernel (mala_bwd_kernel without the list, restricted to such heads), which tests and works tile by tile.
//
// Output, per (batch, query head, key block j): the row's mask (bit i set iff tile (j, i) is retained; rows padded to
// a multiple of four words) and its number of set bits, or an empty mask and the count kScoutDirectRow for a row that
// is left to the one-pass kernel.
//
// Warp roles (640 threads): warp 0 TMA producer (K once, Q ring), warp 1 UMMA issuer, warps 2-3 idle, warps 4-19 the four test
// groups (thread = query row).
#pragma once
#include <cuda_runtime.h>

#include "../../include/mala.h"
#include "sm100_ptx.cuh"
#include "tensor_map.h"

namespace mala {

constexpr uint32_t kScoutDirectRow = 0xffffffffu;   // row_count of a row left to the one-pass kernel
// Two tiles of every sixteen of a row are sampled first in rows of at least 32 tiles, in calls with at least 96 query blocks (192 with
// 64 columns).  Below that the rows that retain everything go with the list: one kernel with one tail instead of two, and every
// tile tested, against a kernel that tests as it goes (whole backward, 16 / 4 heads, sampled / not: 8192 tokens, every tile retained
// 1.07 / 0.99 ms, a third 0.45 / 0.47; 16384 tokens 3.42 / 3.69, 1.43 / 1.43; 64 columns, 16384 tokens, 8 heads 1.35 / 1.16).
constexpr int kScoutSampleStride = 16;
constexpr int kScoutSampleMinTiles = 32;

struct ScoutParams {
  const float* bq;            // [B,Hq,Np] lse2 + log2(tau / L_q); +inf on padding rows
  uint32_t* mask;             // [B,Hq,Tk,wpad] (packed sequences: B entries as well)
  uint32_t* row_count;        // [B,Hq,Tk]
  uint32_t* tel_retained;     // telemetry (may be null): [B,Hq,Tk]
  uint32_t* tel_bitmask;      // telemetry (may be null): [B,Hq,Tk,words], zero-filled by the host
  unsigned long long* totals; // telemetry (may be null)
  int* status;
  int B, Hq, Hkv, N, Np, T, words, wpad, causal;
  int Nk, Tk, koff, qshift;
  const int* cu;
  const int* cu_k;
  int sample;                 // sample the rows first and leave the ones that retain everything to the one-pass kernel
  float scale_log2;
  int by_size;                // see block_place
  int pairs, stages;          // key blocks of a CTA / 2 (1 or 2); Q tiles in the ring (2 or 3)
};

template <int D>
struct ScoutCfg {
  static constexpr int kPanels = D / 64;
  static constexpr int kTileBytes = 128 * D * 2;
  static constexpr int kPairBytes = 2 * kTileBytes;                      // two K tiles: panels of 256 rows
  static constexpr int kThreads = 640;
  static constexpr int kMaxSmem = 232448 - 1024;                         // (static: the barriers, rounded up)
  static constexpr int bytes(int pairs, int stages, int wpad) {
    return pairs * kPairBytes + stages * kTileBytes + 2 * pairs * wpad * 4 + 1024;
  }
};

// The sequence of Q tiles of a CTA, the same for every role: the sampled ones, then -- unless the sampled votes have left the
// head to the one-pass kernel (`sync` returns after *direct has been written) -- the others.  body(i) returns false to stop.
template <class Body, class Sync>
__device__ __forceinline__ bool scout_for_each_tile(int i0, int T, bool sampling, const volatile int* direct, Body body, Sync sync) {
  if (sampling) {
    for (int i = i0; i < T; i += ((i - i0) % kScoutSampleStride == 0) ? 1 : kScoutSampleStride - 1)
      if (!body(i)) return false;
    if (!sync()) return false;
    if (*direct) return true;
  }
  for (int i = i0; i < T; ++i) {
    if (sampling && ((i - i0) % kScoutSampleStride) < 2) continue;
    if (!body(i)) return false;
  }
  return true;
}

template <int D>
__global__ void __launch_bounds__(640, 1)
mala_bwd_scout_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                      const ScoutParams p) {
  using Cfg = ScoutCfg<D>;
  constexpr int PAN = Cfg::kPanels;
  const int KB = 2 * p.pairs, QS = p.stages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sK = smem;                               // [pair][panel][256 rows][128 B]
  uint8_t* sQ = sK + p.pairs * Cfg::kPairBytes;     // Q ring
  uint32_t* rowmask = (uint32_t*)(sQ + QS * Cfg::kTileBytes);   // [key block][wpad]

  __shared__ uint64_t k_full, q_full[3], q_empty[3], s_full[2], s_empty[2], fin_bar, phase_bar;
  __shared__ int direct_s;                          // the head is left to the one-pass kernel
  __shared__ uint32_t tmem_base_s;
  __shared__ int early_exit;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const BlockPlace place = block_place(p.by_size);
  const int ja = KB * place.x, h = place.y, b = place.z;
  const int hkv = h / (p.Hq / p.Hkv);
  // this sequence (the geometry of mala_bwd_kernel)
  const int row0 = p.cu ? __ldg(p.cu + b) : 0;
  const int Nq = p.cu ? __ldg(p.cu + b + 1) - row0 : p.N;
  const int krow0 = p.cu_k ? __ldg(p.cu_k + b) : row0;
  const int Nkeys = p.cu_k ? __ldg(p.cu_k + b + 1) - krow0 : (p.cu ? Nq : p.Nk);
  const int koff = p.cu_k ? (p.causal ? (Nkeys - Nq) / 128 : 0) : p.koff;
  const int qshift = p.cu_k ? (p.causal ? (Nkeys - Nq) % 128 : 0) : p.qshift;
  const int T = p.cu ? (Nq + qshift + 127) / 128 : p.T;
  const int bz = p.cu ? 0 : b;
  const int prow0 = p.cu ? ((row0 + (p.cu_k ? 384 : 128) * b) / 128) * 128 : 0;
  const int Tk_seq = p.cu ? (Nkeys + 127) / 128 : p.Tk;                      // key blocks of this sequence
  const bool none = p.cu_k && (Nq <= 0 || (p.causal && Nkeys < Nq));         // (no defined tile at all)
  const int nkb = none ? 0 : min(KB, Tk_seq - ja);                           // key blocks of this CTA (<= 0: none)
  // tile (i, j) is legal from i = first(j) on
  auto first = [&](int j) -> int { return p.causal ? max(j - koff, 0) : 0; };
  const int i0 = first(ja);
  const int ni = nkb > 0 ? T - i0 : 0;
  const bool sampling = p.sample && ni >= kScoutSampleMinTiles;
  const size_t out_row = ((size_t)b * p.Hq + h) * p.Tk + ja;
  const int wpad = p.wpad;
  int* status = p.status;
  if (ni <= 0) {   // key blocks without queries: empty rows
    for (int kb = 0; kb < KB && ja + kb < p.Tk; ++kb) {
      for (int x = tid; x < wpad; x += blockDim.x) p.mask[(out_row + kb) * wpad + x] = 0u;
      if (tid == 0) {
        p.row_count[out_row + kb] = 0u;
        if (p.tel_retained) p.tel_retained[out_row + kb] = 0u;
      }
    }
    return;
  }

  if (tid == 0) {
    early_exit = (*(volatile int*)status != 0);
    direct_s = 0;
    mbar_init(&k_full, 1);
    for (int s = 0; s < 3; ++s) { mbar_init(&q_full[s], 1); mbar_init(&q_empty[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&s_full[s], 1); mbar_init(&s_empty[s], 8); }
    mbar_init(&fin_bar, 1); mbar_init(&phase_bar, 1);
    mbar_fence_init();
  }
  for (int x = tid; x < KB * wpad; x += blockDim.x) rowmask[x] = 0u;
  __syncthreads();
  if (early_exit) return;
  if (warp == 0) { tmem_alloc(&tmem_base_s, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tb = tmem_base_s;
  // An MMA batch per pair of key blocks and Q tile, where the pair has a legal tile.  Batch m goes to TMEM buffer m & 1.
  auto batches = [&](int i) -> int { return (nkb > 2 && i >= first(ja + 2)) ? 2 : 1; };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK);
      mbar_arrive_expect_tx(&k_full, nkb * Cfg::kTileBytes);
      for (int kb = 0; kb < nkb; ++kb)
        for (int pn = 0; pn < PAN; ++pn)
          tma_load_4d(sK + (kb >> 1) * Cfg::kPairBytes + pn * 32768 + (kb & 1) * 16384, &tmK, &k_full, pn * 64, krow0 + (ja + kb) * 128, hkv, bz);
      int s = 0;
      uint32_t par = 1;
      scout_for_each_tile(i0, T, sampling, &direct_s, [&](int i) -> bool {
        if (!mbar_wait(&q_empty[s], par, status)) return false;
        mbar_arrive_expect_tx(&q_full[s], Cfg::kTileBytes);
        for (int pn = 0; pn < PAN; ++pn)   // (rows before and past the tensor read as zeros)
          tma_load_4d(sQ + s * Cfg::kTileBytes + pn * 16384, &tmQ, &q_full[s], pn * 64, row0 + i * 128 - qshift, h, bz);
        if (++s == QS) { s = 0; par ^= 1; }
        return true;
      }, [&]() -> bool { return mbar_wait(&phase_bar, 0, status); });
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ UMMA issuer (warp-uniform issue loop)
    const uint32_t leader = elect_one();
    constexpr uint32_t idesc = make_idesc_bf16(128, 256, false, false);
    const uint64_t dK0 = make_smem_desc(smem_u32(sK), 16, 1024);
    const uint64_t dQ0 = make_smem_desc(smem_u32(sQ), 16, 1024);
    bool ok = mbar_wait_warp(&k_full, 0, status);
    int s = 0, m = 0;
    uint32_t par = 0;
    if (ok) scout_for_each_tile(i0, T, sampling, &direct_s, [&](int i) -> bool {
      if (!mbar_wait_warp(&q_full[s], par, status)) return false;
      const uint64_t dQ = desc_advance(dQ0, s * Cfg::kTileBytes);
      const int nb = batches(i);
      for (int pr = 0; pr < nb; ++pr, ++m) {
        const int buf = m & 1;
        if (!mbar_wait_warp(&s_empty[buf], ((m >> 1) & 1) ^ 1, status)) return false;   // the buffer's previous batch has been read
        tc_fence_after();
        const uint64_t dK = desc_advance(dK0, pr * Cfg::kPairBytes);
#pragma unroll
        for (int k = 0; k < D / 16; ++k)
          mma_ss(tmem_addr(tb, 0, buf * 256), desc_advance(dQ, (k >> 2) * 16384 + (k & 3) * 32),
                 desc_advance(dK, (k >> 2) * 32768 + (k & 3) * 32), idesc, k > 0, leader);
        if (leader) tc_commit(&s_full[buf]);
      }
      if (leader) tc_commit(&q_empty[s]);
      if (++s == QS) { s = 0; par ^= 1; }
      return true;
    }, [&]() -> bool { return mbar_wait_warp(&phase_bar, 0, status); });
    __syncwarp();
    if (leader) tc_commit(&fin_bar);
    mbar_wait_warp(&fin_bar, 0, status);
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ test groups: group g takes the key block g & 1 of the
    // pair of the batches in buffer g >> 1
    const int g = (warp - 4) >> 2, buf = g >> 1, hf = g & 1;
    const uint32_t lane_base = (uint32_t)(warp & 3) * 32u;
    const int rl = (int)lane_base + lane;
    const float c2 = p.scale_log2;
    const int st = tid - 128;                      // 0 .. 511 among the test threads
    const float* bq = p.bq + ((size_t)bz * p.Hq + h) * p.Np + (size_t)prow0 + rl;
    bool ok = true;                                // (a warp whose wait failed goes on through the barriers below)
    int use = 0;                                   // batches this group's buffer has held (parity of its barriers)
    int m = 0;
    scout_for_each_tile(i0, T, sampling, &direct_s, [&](int i) -> bool {
      const int nb = batches(i);
      for (int pr = 0; pr < nb; ++pr, ++m) {
        if ((m & 1) != buf || !ok) continue;
        const int kb = 2 * pr + hf, j = ja + kb;
        const bool legal = kb < nkb && i >= first(j);
        const float need = legal ? __ldg(bq + (size_t)i * 128) : INFINITY;   // (in flight while the scores are waited for)
        ok = mbar_wait_warp(&s_full[buf], use & 1, status);
        ++use;
        if (!ok) continue;
        tc_fence_after();
        bool vote = false;
        if (legal) {
          // keys that this row may see: up to its own on the diagonal tile, up to the last one in the ragged last block
          int lim = min(128, Nkeys - j * 128);
          if (p.causal && i + koff == j) lim = min(lim, rl + 1);
          const bool cut = __any_sync(0xffffffffu, lim < 128);
          float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t sa[32], sb[32];
            tmem_ld_x32(tmem_addr(tb, lane_base, buf * 256 + hf * 128 + c * 64), sa);
            tmem_ld_x32(tmem_addr(tb, lane_base, buf * 256 + hf * 128 + c * 64 + 32), sb);
            tmem_wait_ld();
            if (cut) {
              const uint32_t ninf = 0xff800000u;
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                if (c * 64 + e >= lim) sa[e] = ninf;
                if (c * 64 + 32 + e >= lim) sb[e] = ninf;
              }
            }
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              m0 = max3(m0, __uint_as_float(sa[e]), __uint_as_float(sa[e + 1]));
              m1 = max3(m1, __uint_as_float(sb[e]), __uint_as_float(sb[e + 1]));
              m2 = max3(m2, __uint_as_float(sa[e + 2]), __uint_as_float(sa[e + 3]));
              m3 = max3(m3, __uint_as_float(sb[e + 2]), __uint_as_float(sb[e + 3]));
            }
          }
          vote = fmaf(fmaxf(max3(m0, m1, m2), m3), c2, -need) >= 0.f;   // Eq. 4 (padding rows: need = +inf)
        }
        const bool any = __any_sync(0xffffffffu, vote);
        tc_fence_before();
        __syncwarp();       // (all lanes' reads of the buffer stand before the arrival)
        if (lane == 0) {
          mbar_arrive(&s_empty[buf]);
          if (any) atomicOr(&rowmask[kb * wpad + (i >> 5)], 1u << (i & 31));
        }
      }
      return true;
    }, [&]() -> bool {
      // all sampled tiles have been tested once the sixteen warps meet here: if every one of them is retained, the head is left to
      // the one-pass kernel
      asm volatile("bar.sync 1, 512;" ::: "memory");
      if (st < 32) {
        int got = 0, want = 0;
        for (int x = st; x < KB * wpad; x += 32) got += __popc(rowmask[x]);
        for (int i = i0 + st * kScoutSampleStride; i < T; i += 32 * kScoutSampleStride)
          for (int e = i; e < min(i + 2, T); ++e)
            for (int kb = 0; kb < nkb; ++kb) want += e >= first(ja + kb);
        for (int sft = 16; sft > 0; sft >>= 1) {
          got += __shfl_xor_sync(0xffffffffu, got, sft);
          want += __shfl_xor_sync(0xffffffffu, want, sft);
        }
        if (st == 0) *(volatile int*)&direct_s = (got == want);
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");
      if (st == 0) mbar_arrive(&phase_bar);
      return true;
    });
    // every tile has been tested once the sixteen warps meet here: the rows go out, one warp per row
    asm volatile("bar.sync 1, 512;" ::: "memory");
    const int kb = st >> 5, j = ja + kb;
    if (kb < KB && j < p.Tk) {
      const bool direct = sampling && direct_s != 0;
      uint32_t pop = 0;
      for (int x = lane; x < wpad; x += 32) {
        const uint32_t wv = direct ? 0u : rowmask[kb * wpad + x];
        p.mask[(out_row + kb) * wpad + x] = wv;
        if (!direct && p.tel_bitmask && x < p.words) p.tel_bitmask[(out_row + kb) * p.words + x] = wv;
        pop += __popc(wv);
      }
      for (int sft = 16; sft > 0; sft >>= 1) pop += __shfl_xor_sync(0xffffffffu, pop, sft);
      if (lane == 0) {
        p.row_count[out_row + kb] = direct ? kScoutDirectRow : pop;
        if (!direct) {
          if (p.tel_retained) p.tel_retained[out_row + kb] = pop;
          if (p.totals && kb < nkb) {
            atomicAdd(&p.totals[0], (unsigned long long)pop);
            atomicAdd(&p.totals[1], (unsigned long long)max(T - first(j), 0));
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tb, 512);
}

}  // namespace mala
