// MALA forward (Algorithm 1) for sm_100a, one query block per CTA: head sizes above 128, and small calls (see fwd_impl).
//
// What bounds a block alone is the chain of its tiles: test, exponentials, test, ...  So everything else runs beside
// that chain.  There are two score buffers (TMEM: S_0, S_1 of 128 columns, O of up to 256): the scores of tile u + 1
// are formed while tile u is in the softmax path, P of tile u overwrites the half of S_(u & 1) that its own threads have
// read, and S_(u & 1) is refilled behind O += P V in tensor-pipe order.  And the softmax path of the one block has all
// eight softmax warps, two threads per query row (keys 0-63 and 64-127 of the tile), two warps per scheduler: the
// exponentials then run at the rate of the exponential unit (1065 clk per tile; one thread per row: 1280).
// The two threads of a row hand each other their maxima and (for Eq. 3) sums as letters in shared memory, without a barrier.
//
// K and V tiles lie in rings of slots of up to 128 columns (32 KB): with 256 columns a tile is two slots, and the copy of one half
// runs while the MMAs of the other do.  V of a tile is fetched once the tile before it has been retained (while MMAs read
// shared memory a copy takes longer than the exponentials), or else on demand, after its own vote.
//
// 16 / 4 heads of 256 columns, 8192 tokens, every tile retained: 426 us dense and 456 with the test; 727 and 757 with one score
// buffer, one thread per row and a stage of a whole tile each for K and V (a quarter of the tiles retained: 334, 519).  There the
// MMAs take 2048 of the 2390 clk per tile until the power limit sets in; with 64 and 128 columns the chain of 2100-2800 clk per tile is the bound.
//
// Warp roles (384 threads): warp 0 K copies (and Q), warp 1 UMMA issuer, warp 2 V copies, warp 3 idle, warps 4-7 / 8-11 the
// softmax threads of the tile's first / second 64 keys.  All synchronisation is by mbarriers and polls with bounded waits.
#pragma once
#include "mala_fwd.cuh"

namespace mala {

template <int D>
struct FwdOneCfg {
  static constexpr int kCols = D < 128 ? D : 128;         // columns of a slot
  static constexpr int kSub = D / kCols;                  // slots of a tile
  static constexpr int kPan = kCols / 64;                 // 64-column panels of a slot
  static constexpr int kSlotBytes = 128 * kCols * 2;
  static constexpr int kKSlots = D > 128 ? 2 : 3, kVSlots = 3;
  static constexpr int kTiles = (kSub + kKSlots + kVSlots) * kSlotBytes;
  static constexpr int kSmemBytes = kTiles + 2560;        // + FwdOneCtl
  static constexpr int kThreads = 384;
};

// A letter: 8 bytes of shared memory with one writer and one reader, (row maximum, sum); empty while the first word is kNoLetter.
// The writer waits until it is empty, the reader until it is not, and empties it; both waits are bounded, and the outcome is the
// same in all lanes of the (converged) warp.
constexpr uint32_t kNoLetter = 0xffffffffu;
template <bool kFull>
__device__ __forceinline__ bool letter_wait(const volatile uint64_t* at, uint64_t& w, int* status) {
  long long t0 = 0;
  for (uint32_t it = 1;; ++it) {
    w = *at;
    if (__all_sync(0xffffffffu, ((uint32_t)w != kNoLetter) == kFull)) return true;
    if ((it & 0xff) == 0) {
      const long long now = clock64();
      if (t0 == 0) t0 = now;
      const bool late = now - t0 > kWaitLimitCycles;
      if (late) atomicCAS(status, 0, kDevTimeout);
      if (__any_sync(0xffffffffu, late || *(volatile int*)status != 0)) return false;
    }
  }
}
// (`before`: what the writer read there a while ago, so that the usual case waits for nothing)
__device__ __forceinline__ bool letter_put(volatile uint64_t* at, uint64_t before, float mx, float sum, int* status) {
  if (!__all_sync(0xffffffffu, (uint32_t)before == kNoLetter) && !letter_wait<false>(at, before, status)) return false;
  const uint32_t w = __float_as_uint(mx);
  *at = ((uint64_t)__float_as_uint(sum) << 32) | (w == kNoLetter ? 0x7fffffffu : w);   // (a NaN either way)
  return true;
}
__device__ __forceinline__ bool letter_get(volatile uint64_t* at, float& mx, float& sum, int* status) {
  uint64_t w;
  if (!letter_wait<true>(at, w, status)) return false;
  mx = __uint_as_float((uint32_t)w);
  sum = __uint_as_float((uint32_t)(w >> 32));
  *at = ~0ull;
  return true;
}

// Barriers and letters, behind the tiles in the dynamic shared memory (with 256 columns the tiles leave 3 KB)
struct FwdOneCtl {
  uint64_t q_full, k_full[3], k_empty[3], v_full[3], v_empty[3], v_ask[2], s_full[2], vote_bar[2], p_full[2][2], pv_done, fin_bar;
  uint64_t letter[2][128];                       // [half that writes][row]: row maxima of a tile, sums of the retained tiles before it
  uint32_t tmem_base;
  int flag[4], v_tile[2], early_exit;
};

template <int D, bool kDense, bool kSmall = false>
__global__ void __launch_bounds__(384, 1)
mala_fwd_one_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const FwdParams p) {
  using Cfg = FwdOneCfg<D>;
  constexpr int KS = Cfg::kKSlots, VS = Cfg::kVSlots, SUB = Cfg::kSub, PAN = Cfg::kPan, SLOT = Cfg::kSlotBytes;
  constexpr uint32_t kColO = 256;
  static_assert(sizeof(FwdOneCtl) <= 2560 && KS <= 3 && VS <= 3, "");
  extern __shared__ __align__(1024) uint8_t smem[];   // (no static shared memory: the tiles start on a 1024-byte boundary)
  uint8_t* sQ = smem;
  uint8_t* sK = sQ + SUB * SLOT;
  uint8_t* sV = sK + KS * SLOT;

  FwdOneCtl& ctl = *reinterpret_cast<FwdOneCtl*>(smem + Cfg::kTiles);
  uint64_t &q_full = ctl.q_full, &pv_done = ctl.pv_done, &fin_bar = ctl.fin_bar;
  uint64_t *k_full = ctl.k_full, *k_empty = ctl.k_empty, *v_full = ctl.v_full, *v_empty = ctl.v_empty, *s_full = ctl.s_full,
           *v_ask = ctl.v_ask, *vote_bar = ctl.vote_bar;
  uint64_t (*p_full)[2] = ctl.p_full;
  int *flag = ctl.flag, *v_tile = ctl.v_tile;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = p.Hq / p.Hkv;
  const BlockPlace place = block_place(p.by_size);
  const int sp = p.num_splits > 1 ? place.z % p.num_splits : 0;
  const int b = p.num_splits > 1 ? place.z / p.num_splits : place.z;
  const int h = place.y, hkv = h / G;
  // this sequence: the geometry of mala_fwd_kernel
  const int row0 = p.cu ? __ldg(p.cu + b) : 0;
  const int Nq = p.cu ? __ldg(p.cu + b + 1) - row0 : p.N;
  const bool own_keys = p.cu_k || p.block_table;
  const int krow0 = p.cu_k ? __ldg(p.cu_k + b) : row0;
  const int Nkeys = p.block_table ? min(__ldg(p.seqlens_k + b), p.bt_stride * (p.ppt > 1 ? p.prows : p.tpp * 128))
                                  : (p.cu_k ? __ldg(p.cu_k + b + 1) - krow0 : (p.cu ? Nq : p.Nk));
  if (own_keys && (Nkeys <= 0 || (p.causal && Nkeys < Nq))) return;
  const int koff = own_keys ? (p.causal ? (Nkeys - Nq) / 128 : 0) : p.koff;
  const int qshift = own_keys ? (p.causal ? (Nkeys - Nq) % 128 : 0) : p.qshift;
  const int Tr = p.cu ? (Nq + qshift + 127) / 128 : p.Tr;
  const int Tk = p.cu ? (Nkeys + 127) / 128 : p.Tk;
  const int bz = p.cu ? 0 : b;
  // longest blocks first: of this head and sequence, or (by_size) of all of them
  const int i = (p.by_size ? (int)gridDim.x : Tr) - 1 - place.x;
  if (i < 0 || i >= Tr) return;
  const int dI = p.causal ? i + koff : Tk - 1;       // newest key block with a legal key
  int jlo = 0, jhi = Tk - 1;                         // key blocks of this CTA
  if (p.num_splits > 1) {
    jlo = sp * p.tps;
    jhi = min(Tk, jlo + p.tps) - 1;
    if (jlo > dI) return;                            // no legal key in the range (the merge knows)
  }
  const int j0 = min(dI, jhi);                       // step u = 0 .. U-1 visits key block j0 - u
  const int U = j0 - jlo + 1;
  int* status = p.status;

  // One slot of key block jt: columns sub * 128 .. of its 128 rows.  All lanes of the warp call this; pages smaller than a
  // tile: lane x issues copies of the pages x / PAN, + 32 / PAN, ... of panel x % PAN.
  auto load_slot = [&](uint8_t* dst, const CUtensorMap* tm, uint64_t* bar, int jt, int sub) {
    if (lane == 0) mbar_arrive_expect_tx(bar, SLOT);
    __syncwarp();
    if (kSmall) {
      const int pn = lane % PAN;
      for (int c = lane / PAN; c < p.ppt; c += 32 / PAN) {
        const int pg = jt * p.ppt + c;
        const int outer = pg < p.bt_stride ? __ldg(p.block_table + (size_t)b * p.bt_stride + pg) : -1;
        tma_load_4d(dst + pn * 16384 + c * p.prows * 128, tm, bar, (sub * PAN + pn) * 64, 0, hkv, outer);
      }
    } else if (lane == 0) {
      int row = krow0 + jt * 128, outer = p.cu ? 0 : b;
      if (p.block_table) {
        const int pg = jt / p.tpp;
        outer = __ldg(p.block_table + (size_t)b * p.bt_stride + pg);
        row = (jt - pg * p.tpp) * 128;
      }
      for (int pn = 0; pn < PAN; ++pn) tma_load_4d(dst + pn * 16384, tm, bar, (sub * PAN + pn) * 64, row, hkv, outer);
    }
  };

  if (tid == 0) {
    ctl.early_exit = (*(volatile int*)status != 0);
    mbar_init(&q_full, 1);
    for (int s = 0; s < KS; ++s) { mbar_init(&k_full[s], 1); mbar_init(&k_empty[s], 1); }
    for (int s = 0; s < VS; ++s) { mbar_init(&v_full[s], 1); mbar_init(&v_empty[s], 1); }
    for (int x = 0; x < 2; ++x) {
      mbar_init(&v_ask[x], 1); mbar_init(&s_full[x], 1); mbar_init(&vote_bar[x], 8); mbar_init(&p_full[x][0], 8); mbar_init(&p_full[x][1], 8);
    }
    mbar_init(&pv_done, 1); mbar_init(&fin_bar, 1);
    flag[0] = flag[1] = flag[2] = flag[3] = 0;
    mbar_fence_init();
  }
  if (tid < 256) ctl.letter[tid >> 7][tid & 127] = ~0ull;
  __syncthreads();
  if (ctl.early_exit) return;
  if (warp == 0) { tmem_alloc(&ctl.tmem_base, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tb = ctl.tmem_base;

  if (warp == 0) {
    // ------------------------------------------------------------------ Q, then K of every tile
    if (lane == 0) {
      tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK);
      mbar_arrive_expect_tx(&q_full, SUB * SLOT);
      // (the first block of a chunk that starts inside a tile begins before row 0: those rows read as zeros)
      for (int pn = 0; pn < SUB * PAN; ++pn)
        tma_load_4d(sQ + pn * 16384, &tmQ, &q_full, pn * 64, row0 + i * 128 - qshift, h, bz);
    }
    int s = 0, issued = 0;
    uint32_t par = 1;
    bool ok = true;
    for (int n = 0; n < U * SUB && ok; ++n) {
      ok = mbar_wait_warp(&k_empty[s], par, status);
      if (!ok) break;
      load_slot(sK + s * SLOT, &tmK, &k_full[s], j0 - n / SUB, n % SUB);
      issued = n + 1;
      if (++s == KS) { s = 0; par ^= 1; }
    }
    if (!ok) {   // (no copy may be in flight when the CTA exits)
      mbar_wait_warp(&q_full, 0, status);
      for (int n = max(issued - KS, 0); n < issued; ++n) mbar_wait_warp(&k_full[n % KS], (n / KS) & 1, status);
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ V of every tile (dense) or of those that the issuer asks for, in turn
    if (lane == 0) tma_prefetch_desc(&tmV);
    int s = 0, issued = 0;
    uint32_t par = 1;
    bool ok = true;
    for (int r = 0; ok; ++r) {
      int u = r;
      if (!kDense) {
        ok = mbar_wait_warp(&v_ask[r & 1], (r >> 1) & 1, status);
        if (!ok) break;
        u = __shfl_sync(0xffffffffu, *(volatile int*)&v_tile[r & 1], 0);
      }
      if (u < 0 || u >= U) break;
      for (int sub = 0; sub < SUB && ok; ++sub) {
        ok = mbar_wait_warp(&v_empty[s], par, status);
        if (!ok) break;
        load_slot(sV + s * SLOT, &tmV, &v_full[s], j0 - u, sub);
        ++issued;
        if (++s == VS) { s = 0; par ^= 1; }
      }
    }
    if (!ok)
      for (int n = max(issued - VS, 0); n < issued; ++n) mbar_wait_warp(&v_full[n % VS], (n / VS) & 1, status);
  } else if (warp == 1) {
    // ------------------------------------------------------------------ UMMA issuer (warp-uniform, one elected lane issues)
    const uint32_t leader = elect_one();
    constexpr uint32_t idesc_qk = make_idesc_bf16(128, 128, false, false);
    constexpr uint32_t idesc_pv = make_idesc_bf16(128, Cfg::kCols, false, true);
    const uint64_t dQ = make_smem_desc(smem_u32(sQ), 16, 1024);
    const uint64_t dK0 = make_smem_desc(smem_u32(sK), 16, 1024);
    const uint64_t dV0 = make_smem_desc(smem_u32(sV), 16384, 1024);
    int s = 0, vs = 0;
    uint32_t kpar = 0, vpar = 0;
    auto issue_qk = [&](int u) -> bool {   // S_(u & 1) = Q K^T
#pragma unroll
      for (int sub = 0; sub < SUB; ++sub) {
        if (!mbar_wait_warp(&k_full[s], kpar, status)) return false;
        tc_fence_after();
        const uint64_t dK = desc_advance(dK0, s * SLOT);
#pragma unroll
        for (int k = 0; k < Cfg::kCols / 16; ++k) {
          const uint32_t off = (k >> 2) * 16384 + (k & 3) * 32;
          mma_ss(tmem_addr(tb, 0, (u & 1) * 128), desc_advance(dQ, sub * SLOT + off), desc_advance(dK, off), idesc_qk, sub > 0 || k > 0, leader);
        }
        if (leader) tc_commit(&k_empty[s]);
        if (++s == KS) { s = 0; kpar ^= 1; }
      }
      if (leader) tc_commit(&s_full[u & 1]);
      return true;
    };
    bool ok = mbar_wait_warp(&q_full, 0, status);
    if (ok) ok = issue_qk(0);
    if (ok && U > 1) ok = issue_qk(1);
    int r = 0;                       // retained tiles so far
    // V copies asked for.  Asking for one more than the two that v_tile holds follows the end of an earlier one's copy.
    int asks = 0, ahead = -1;        // ahead: the tile whose V was asked for before its vote (still in the ring), or -1
    auto ask_v = [&](int u) {
      if (leader) { *(volatile int*)&v_tile[asks & 1] = u; mbar_arrive(&v_ask[asks & 1]); }
      ++asks;
    };
    auto drop_v = [&]() -> bool {    // a V tile that came for a tile which was skipped: its slots go back once it is there
      for (int sub = 0; sub < SUB; ++sub) {
        if (!mbar_wait_warp(&v_full[vs], vpar, status)) return false;
        if (leader) mbar_arrive(&v_empty[vs]);
        if (++vs == VS) { vs = 0; vpar ^= 1; }
      }
      ahead = -1;
      return true;
    };
    uint32_t ppar = 0;               // bit x: parity of p_full[x] for the next retained tile in buffer x
    for (int u = 0; u < U && ok; ++u) {
      const int x = u & 1;
      bool retain = true;
      if (!kDense) {
        ok = mbar_wait_warp(&vote_bar[x], (u >> 1) & 1, status);
        if (!ok) break;
        retain = __shfl_sync(0xffffffffu, *(volatile int*)&flag[u & 3], 0) != 0;
        if (retain) {
          if (ahead >= 0 && ahead != u) { ok = drop_v(); if (!ok) break; }
          if (ahead != u) ask_v(u);
          ahead = -1;
          if (u + 1 < U) { ask_v(u + 1); ahead = u + 1; }
        }
      }
      if (retain) {
        // P arrives in two pieces, the first 32 keys of either half of the tile before the others (the MMAs keep the order of the
        // keys, in which mala_fwd_kernel adds them too)
#pragma unroll
        for (int piece = 0; piece < 2; ++piece) {
          int vsp = vs;
          uint32_t vparp = vpar;
          ok = mbar_wait_warp(&p_full[x][piece], (ppar >> x) & 1, status);
          if (!ok) break;
#pragma unroll
          for (int sub = 0; sub < SUB; ++sub) {
            if (piece == 0) {
              ok = mbar_wait_warp(&v_full[vsp], vparp, status);
              if (!ok) break;
            }
            tc_fence_after();
            const uint64_t dV = desc_advance(dV0, vsp * SLOT);
#pragma unroll
            for (int k = piece * 2; k < (piece ? 8 : 2); ++k)
              mma_ts(tmem_addr(tb, 0, kColO + sub * 128), tmem_addr(tb, 0, x * 128 + (k >> 2) * 64 + (k & 3) * 8), desc_advance(dV, k * 2048), idesc_pv,
                     k > 0 ? 1u : (r > 0 ? 1u : 0u), leader);
            if (piece == 1 && leader) tc_commit(&v_empty[vsp]);
            if (++vsp == VS) { vsp = 0; vparp ^= 1; }
          }
          if (!ok) break;
          if (piece == 1) { vs = vsp; vpar = vparp; }
        }
        if (!ok) break;
        if (leader) tc_commit(&pv_done);
        ppar ^= 1u << x;
        ++r;
      }
      if (u + 2 < U) ok = issue_qk(u + 2);   // behind this tile's PV in the tensor pipe: the score buffer is free
    }
    if (!kDense && ok && ahead >= 0) ok = drop_v();
    if (!kDense && ok) ask_v(-1);
    __syncwarp();
    if (leader) tc_commit(&fin_bar);
    mbar_wait_warp(&fin_bar, 0, status);
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ softmax: two threads per query row
    const int half = (warp - 4) >> 2;
    const uint32_t lane_base = (uint32_t)(warp & 3) * 32u;
    const int rl = (int)lane_base + lane;
    const int prow_ = i * 128 + rl;                   // row counted in whole blocks from the first block's start
    const int row = prow_ - qshift;
    const bool valid = row >= 0 && row < Nq;
    const float c2 = p.scale_log2;
    const float Lq = p.causal ? (float)(prow_ + 1 + koff * 128) : (float)Nkeys;   // visible keys
    const float theta = kDense ? -INFINITY : (p.log2_tau - log2f(Lq));
    const bool mask_first = j0 == dI;
    float m_ref = -INFINITY, l = 0.f;                 // l: this thread's keys only
    float lg = -INFINITY;                             // m_ref + log2(l of the row)
    int r = 0;
    volatile uint64_t *out_box = &ctl.letter[half][rl], *in_box = &ctl.letter[half ^ 1][rl];
    bool fresh = false;                               // the tile before was retained: `lg` is out of date
    bool ok = true;
    uint32_t bm_bits = 0;
    int bm_word = -1;
    const bool stat_thread = warp == 4 && lane == 0;
    const size_t stat_row = (size_t)(b * p.Hq + h) * p.Tr + i;
    uint32_t* bm_row = p.bitmask ? p.bitmask + stat_row * p.words : nullptr;

    for (int t = 0; t < U; ++t) {
      const int x = t & 1, j = j0 - t;
      ok = mbar_wait_warp(&s_full[x], (t >> 1) & 1, status);
      if (!ok) break;
      tc_fence_after();
      const uint32_t colS = (uint32_t)x * 128u + (uint32_t)half * 64u;
      uint32_t s0[32], s1[32];
      tmem_ld_x32(tmem_addr(tb, lane_base, colS), s0);
      tmem_ld_x32(tmem_addr(tb, lane_base, colS + 32), s1);
      const uint64_t before = *out_box;
      tmem_wait_ld();
      if (t == 0 && mask_first) {   // the newest legal tile: causal diagonal and / or the ragged end of the keys
        const int lim = (p.causal ? rl : (Nkeys - 1 - j * 128)) - half * 64;
        const uint32_t ninf = 0xff800000u;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          if (e > lim) s0[e] = ninf;
          if (e + 32 > lim) s1[e] = ninf;
        }
      }
      float mx[4];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        mx[c] = max3(__uint_as_float(s0[c]), __uint_as_float(s0[c + 2]), __uint_as_float(s0[c + 4]));
        mx[c + 2] = max3(__uint_as_float(s1[c]), __uint_as_float(s1[c + 2]), __uint_as_float(s1[c + 4]));
      }
#pragma unroll
      for (int e = 6; e < 30; e += 4)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          mx[c] = max3(mx[c], __uint_as_float(s0[e + c]), __uint_as_float(s0[e + c + 2]));
          mx[c + 2] = max3(mx[c + 2], __uint_as_float(s1[e + c]), __uint_as_float(s1[e + c + 2]));
        }
      float mt = fmaxf(max3(mx[0], mx[1], fmaxf(__uint_as_float(s0[30]), __uint_as_float(s0[31]))),
                       max3(mx[2], mx[3], fmaxf(__uint_as_float(s1[30]), __uint_as_float(s1[31])))) * c2;
      // the row's maximum, and its normalizer after the tile before, from both threads of the row: at once where the test
      // needs the new normalizer, else only if the tile is retained
      ok = letter_put(out_box, before, mt, l, status);
      if (!ok) break;
      if (kDense || fresh) {
        float other, sum;
        ok = letter_get(in_box, other, sum, status);
        if (!ok) break;
        mt = fmaxf(mt, other);
        if (!kDense) lg = m_ref + __log2f(half ? sum + l : l + sum);
      }
      bool retain = true;
      if (!kDense) {
        // Eq. 3: skip iff rowmax - (m + log l) < log(tau / L) for every valid row (nothing retained yet: lg = -inf)
        const bool any = __any_sync(0xffffffffu, valid && !((mt - lg) - theta < 0.f));
        tc_fence_before();
        __syncwarp();       // (a vote orders no memory: all lanes' letters and reads of the scores stand before the arrival)
        if (lane == 0) {
          if (any) *(volatile int*)&flag[t & 3] = 1;
          if (warp == 4) *(volatile int*)&flag[(t + 2) & 3] = 0;   // (last read for tile t - 2, next set for tile t + 2)
          mbar_arrive(&vote_bar[x]);
        }
        // A warp that found a retaining row knows the outcome and goes straight on.
        if (!any) {
          ok = mbar_wait_warp(&vote_bar[x], (t >> 1) & 1, status);
          if (!ok) break;
          retain = __all_sync(0xffffffffu, (*(volatile int*)&flag[t & 3]) != 0);
        }
        if (!retain) {
          if (!fresh) *in_box = ~0ull;        // (both halves have voted behind their letters, so it is there)
          fresh = false;
          continue;
        }
        if (!fresh) {
          float other, sum;
          ok = letter_get(in_box, other, sum, status);
          if (!ok) break;
          mt = fmaxf(mt, other);
        }
      }
      if (stat_thread && bm_row) {
        if ((j >> 5) != bm_word) {
          if (bm_word >= 0) {
            if (p.num_splits > 1) atomicOr(&bm_row[bm_word], bm_bits);   // (ranges share words of the row)
            else bm_row[bm_word] = bm_bits;
          }
          bm_word = j >> 5;
          bm_bits = 0;
        }
        bm_bits |= 1u << (j & 31);
      }
      // Lazy rescaling: the reference maximum only moves when the row maximum grew by more than 2^8.  The PV before may
      // still be running then: it has to be over first.
      const bool need_any = __any_sync(0xffffffffu, r > 0 && mt > m_ref + 8.f);
      if (r == 0) {
        m_ref = mt;
      } else if (need_any) {
        ok = mbar_wait_warp(&pv_done, (r - 1) & 1, status);
        if (!ok) break;
        tc_fence_after();
        const float m_new = fmaxf(m_ref, mt);
        const float alpha = fast_exp2(m_ref - m_new);
        l *= alpha;
        m_ref = m_new;
#pragma unroll
        for (int cc = 0; cc < D / 64; ++cc) {
          uint32_t o[32];
          tmem_ld_x32(tmem_addr(tb, lane_base, kColO + half * (D / 2) + cc * 32), o);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
          tmem_st_x32(tmem_addr(tb, lane_base, kColO + half * (D / 2) + cc * 32), o);
        }
      }
      // P = exp2(s * c2 - m_ref), row sum in fp32 before the bf16 cast, P over this thread's own scores
      const float nm = -m_ref;
      float sum0 = 0.f, sum1 = 0.f, sum2 = 0.f, sum3 = 0.f;
#define MALA_P_PIECE(SRC, PIECE)                                                       \
      {                                                                                \
        uint32_t pk[16];                                                               \
        _Pragma("unroll") for (int e = 0; e < 8; ++e) {                                \
          const float p0 = fast_exp2(fmaf(__uint_as_float(SRC[4 * e]), c2, nm));        \
          const float p1 = fast_exp2(fmaf(__uint_as_float(SRC[4 * e + 1]), c2, nm));    \
          const float p2 = fast_exp2(fmaf(__uint_as_float(SRC[4 * e + 2]), c2, nm));    \
          const float p3 = fast_exp2(fmaf(__uint_as_float(SRC[4 * e + 3]), c2, nm));    \
          sum0 += p0; sum1 += p1; sum2 += p2; sum3 += p3;                              \
          pk[2 * e] = pack_bf16x2(p0, p1);                                             \
          pk[2 * e + 1] = pack_bf16x2(p2, p3);                                         \
        }                                                                              \
        tmem_st_x16(tmem_addr(tb, lane_base, colS + (PIECE) * 16), pk);                \
        tmem_wait_st();                                                                \
        tc_fence_before();                                                             \
        __syncwarp();                                                                  \
        if (lane == 0) mbar_arrive(&p_full[x][PIECE]);                                 \
      }
      MALA_P_PIECE(s0, 0)
      MALA_P_PIECE(s1, 1)
#undef MALA_P_PIECE
      l += (sum0 + sum1) + (sum2 + sum3);
      fresh = true;
      ++r;
    }

    if (ok) {
      // finalize once every PV has retired: O <- O / l, lse <- m + log l
      float other, sum;
      ok = letter_put(out_box, 0, 0.f, l, status);
      if (ok) ok = letter_get(in_box, other, sum, status);
      l = half ? sum + l : l + sum;
    }
    if (ok) ok = mbar_wait_warp(&fin_bar, 0, status);
    if (ok) {
      tc_fence_after();
      const float inv = 1.f / l;
      const bool parts = p.num_splits > 1;             // one range of the keys: normalised fp32 partial and its log-normalizer
      const size_t prow = (((size_t)b * p.Hq + h) * p.num_splits + sp) * p.N + row;
      __nv_bfloat16* orow = p.o + (int64_t)bz * p.o_sb + (int64_t)(row0 + row) * p.o_sn + (int64_t)h * p.o_sh;
#pragma unroll
      for (int cc = 0; cc < D / 64; ++cc) {
        const int col = half * (D / 2) + cc * 32;
        uint32_t o[32];
        tmem_ld_x32(tmem_addr(tb, lane_base, kColO + col), o);
        tmem_wait_ld();
        if (!valid) continue;
        if (parts) {
#pragma unroll
          for (int v = 0; v < 8; ++v)
            if (col + v * 4 < p.d)
              *reinterpret_cast<float4*>(p.o_part + prow * D + col + v * 4) =
                make_float4(__uint_as_float(o[4 * v]) * inv, __uint_as_float(o[4 * v + 1]) * inv,
                            __uint_as_float(o[4 * v + 2]) * inv, __uint_as_float(o[4 * v + 3]) * inv);
        } else {
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            uint4 w;
            w.x = pack_bf16x2(__uint_as_float(o[8 * v + 0]) * inv, __uint_as_float(o[8 * v + 1]) * inv);
            w.y = pack_bf16x2(__uint_as_float(o[8 * v + 2]) * inv, __uint_as_float(o[8 * v + 3]) * inv);
            w.z = pack_bf16x2(__uint_as_float(o[8 * v + 4]) * inv, __uint_as_float(o[8 * v + 5]) * inv);
            w.w = pack_bf16x2(__uint_as_float(o[8 * v + 6]) * inv, __uint_as_float(o[8 * v + 7]) * inv);
            if (col + v * 8 < p.d) *reinterpret_cast<uint4*>(orow + col + v * 8) = w;
          }
        }
      }
      if (valid && half == 0) {
        const float out = (m_ref + log2f(l)) * 0.6931471805599453f;
        if (parts) p.lse_part[prow] = out;
        else p.lse[p.cu ? (size_t)h * p.total + row0 + row : ((size_t)b * p.Hq + h) * p.N + row] = out;
      }
      if (stat_thread) {   // (several ranges add to the same telemetry rows)
        if (bm_row && bm_word >= 0) {
          if (parts) atomicOr(&bm_row[bm_word], bm_bits);
          else bm_row[bm_word] = bm_bits;
        }
        if (p.retained) {
          if (parts) atomicAdd(&p.retained[stat_row], (uint32_t)r);
          else p.retained[stat_row] = (uint32_t)r;
        }
        if (p.totals) {
          atomicAdd(&p.totals[0], (unsigned long long)r);
          atomicAdd(&p.totals[1], (unsigned long long)U);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  // (the merge waits for this grid's end all the same; let go at the kernel's start, its waiting blocks slowed the kernel)
  release_dependents();
  if (warp == 0) tmem_dealloc(tb, 512);
}

}  // namespace mala
