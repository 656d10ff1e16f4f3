// Order in which the persistent decode kernels take their work items.
//
// A work item is one split of one (sequence, KV head); the splits are laid out for the longest sequence, so a shorter one
// has fewer full splits, one partial split and empty ones.  Taken in the order of their numbers (one item per lane of work
// and round), the lanes' loads follow whatever lengths happen to fall on them: 32 sequences of 4000 .. 16000 keys in 4 splits
// left the busiest CTA with 1.74 times the mean of the K tiles (KV head slowest) or 1.33 times (KV head fastest).  Here the
// items are ordered by size -- the full splits, then the partial ones from the largest down, then the empty ones -- and
// dealt out back and forth (round k left to right, round k + 1 right to left): 1.05 times.  (Of the K tiles; how many V
// tiles its heads retain is not known here.)  The step takes 166 us instead of 241 (bf16, pages of 16 keys); 16 sequences of
// 10000 .. 40000 keys in e4m3 152 instead of 201.  Every CTA works its list out for itself from the lengths, so nothing has
// to be set up before the launch or kept after it.
#pragma once
#include <stdint.h>

namespace mala {

// Division of a 32-bit number by a divisor known at launch, as a multiplication and shifts (Granlund and Montgomery's
// round-up method for an invariant divisor; every role works out for
// itself which sequence, KV head and split a work item is; hardware has no integer divide, and the few dozen
// dependent instructions of an emulated one would sit on the per-tile chain of the softmax threads).
struct FastDiv {
  uint32_t d, mul, sh;
  __host__ void set(uint32_t divisor) {
    d = divisor;
    uint32_t l = 0;
    while ((1ull << l) < divisor) ++l;
    sh = l;
    mul = (uint32_t)(((1ull << 32) * ((1ull << l) - divisor)) / divisor + 1);
  }
  __device__ __forceinline__ uint32_t div(uint32_t n) const {
    if (d == 1u) return n;
    const uint32_t t = __umulhi(mul, n);
    return (t + ((n - t) >> 1)) >> (sh - 1u);
  }
};

constexpr int kSchedBatch = 256;     // sequences
constexpr int kSchedMaxItem = 65535; // item numbers are kept in 16 bits; this one marks the end

// Whether a call whose B sequences have lengths of their own takes this order (more than one round of items, and the tables
// fit) on `grid` CTAs that work on per_cta items at a time and have room for list_size entries.  Sequences of one length keep
// the order of the item numbers: nothing is gained by size, and dealt back and forth a lane meets the same few KV heads
// again and again (22 sequences of 15754 keys, 64 / 8 heads: 219 us in the order of the numbers, 234 dealt out; 18 of 36027,
// two tokens: 341 and 359).  So do more than 256 sequences, whose many rounds even out by themselves and whose tables
// take 1-2 us of the step: 128 sequences of up to 1024 keys 86 us ordered, 91 not (bf16; e4m3 53 and 58), 256 of them
// 149.9 and 150.0 (87.5 and 86.3), 512 of them 273.5 and 265.3 (166.9 and 160.2).
inline bool decode_sched_fits(int B, long long n_items, int grid, int per_cta, int list_size) {
  const long long lanes = (long long)grid * per_cta;
  return n_items > grid && B <= kSchedBatch && n_items < kSchedMaxItem && (n_items + lanes - 1) / lanes * per_cta <= list_size;
}

// Fills list[round * PER + k] with the item of lane k * gridDim.x + blockIdx.x in that round (item (b * splits + split) *
// Hkv + hkv; kSchedMaxItem: none).  Called by all threads of the block; `tmp`: kSchedTmpBytes of shared memory; the caller
// synchronises the block before the list is read.
// A latency in front of the step's first copy, so the work is linear in the batch, 32 sequences per warp: running counts of
// the full and the empty splits by scans, and the partial splits ranked by counting them in up to 32 classes of size (the
// tiles themselves up to 33 tiles per split), in the order of the sequences inside a class, so that every CTA finds the same
// order.  Ranking every sequence against every other, with a division per pair, took the step with 512 sequences of up to
// 512 keys, 8 / 2 heads, from 56 to 113 us (bf16) and 256 of up to 1024 keys from 57 to 65 (now 50).
constexpr int kSchedChunks = kSchedBatch / 32;
constexpr int kSchedTmpBytes = kSchedBatch * 6 + kSchedChunks * 33 * 4 + 32 * 4;
template <int PER, int kThreads>
__device__ __forceinline__ void decode_schedule(uint16_t* list, void* tmp, const int* seqlens, int B, int Hkv,
                                                const FastDiv& by_hkv, const FastDiv& by_tps, int splits, int tps, int Nk,
                                                int n_items) {
  static_assert(kThreads / 32 >= kSchedChunks, "a warp for every 32 sequences");
  constexpr uint32_t kAll = 0xffffffffu;
  uint32_t* to = reinterpret_cast<uint32_t*>(tmp);           // [b] full (low half) and empty (high half) splits of 0 .. b
  int* count = reinterpret_cast<int*>(to + kSchedBatch);     // [chunk][class] partial splits; then those of chunks before
  int* before = count + kSchedChunks * 32;                   // [class] partial splits of larger classes
  uint32_t* total = reinterpret_cast<uint32_t*>(before + 32);   // [chunk] like `to`: of the chunk, then of those before it
  uint16_t* part = reinterpret_cast<uint16_t*>(total + kSchedChunks);   // [r] sequence with the r-th largest partial split
  const int c = threadIdx.x >> 5, x = threadIdx.x & 31, b0 = threadIdx.x, chunks = (B + 31) / 32;
  // running counts of inclusive sums over the lanes
  auto scan = [&](uint32_t v) {
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
      const uint32_t y = __shfl_up_sync(kAll, v, m);
      if (x >= m) v += y;
    }
    return v;
  };
  uint32_t run = 0;
  int cls = 32, pos = 0;                                     // class 0: the largest; 32: no partial split
  if (c < chunks) {
    if (b0 < B) {
      const int shift = max(0, 27 - __clz(max(0, tps - 2)));   // (tps - 2) >> shift <= 31
      const int t = (min(Nk, max(0, __ldg(seqlens + b0))) + 127) / 128, f = (int)by_tps.div((uint32_t)t), r = t - f * tps;
      run = (uint32_t)f | (uint32_t)(splits - f - (r > 0 ? 1 : 0)) << 16;
      if (r > 0) cls = 31 - ((r - 1) >> shift);
    }
    run = scan(run);
    if (x == 31) total[c] = run;
    const uint32_t same = __match_any_sync(kAll, cls);
    pos = __popc(same & ((1u << x) - 1u));
    count[c * 32 + x] = 0;
    __syncwarp();
    if (cls < 32 && pos == 0) count[c * 32 + cls] = __popc(same);
  }
  __syncthreads();
  if (c == 0) {                                              // (lane: class)
    uint32_t sum = 0;
    for (int y = 0; y < chunks; ++y) {
      const int n = count[y * 32 + x];
      count[y * 32 + x] = (int)sum;
      sum += n;
    }
    before[x] = (int)(scan(sum) - sum);
  } else if (c == 1) {                                       // (lane: chunk)
    const uint32_t n = x < chunks ? total[x] : 0u, sum = scan(n);
    if (x < chunks) total[x] = sum - n;
  }
  __syncthreads();
  if (b0 < B) {
    to[b0] = run + total[c];
    if (cls < 32) part[before[cls] + count[c * 32 + cls] + pos] = (uint16_t)b0;
  }
  __syncthreads();
  const int n_full = (int)(to[B - 1] & 0xffffu), n_part = B * splits - n_full - (int)(to[B - 1] >> 16);
  // splits of one kind (half of `to`: 0 full, 16 empty) of the sequences 0 .. b, and the first sequence with more than v
  auto count_to = [&](int half, int b) { return b < 0 ? 0 : (int)((to[b] >> half) & 0xffffu); };
  auto find = [&](int half, int v) {
    int lo = 0, hi = B - 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (count_to(half, mid) > v) hi = mid; else lo = mid + 1;
    }
    return lo;
  };
  const int lanes = PER * (int)gridDim.x, rounds = (n_items + lanes - 1) / lanes;
  for (int e = threadIdx.x; e < rounds * PER; e += kThreads) {
    const int round = e / PER, lane = (e - round * PER) * (int)gridDim.x + (int)blockIdx.x;
    const int at = round * lanes + ((round & 1) ? lanes - 1 - lane : lane);
    int item = kSchedMaxItem;
    if (at < n_items) {
      int s = (int)by_hkv.div((uint32_t)at), b, split;
      const int hkv = at - s * Hkv;
      if (s < n_full) {
        b = find(0, s);
        split = s - count_to(0, b - 1);
      } else if (s < n_full + n_part) {
        b = part[s - n_full];
        split = count_to(0, b) - count_to(0, b - 1);
      } else {
        s -= n_full + n_part;
        b = find(16, s);
        split = splits - (count_to(16, b) - s);
      }
      item = (b * splits + split) * Hkv + hkv;
    }
    list[e] = (uint16_t)item;
  }
}

}  // namespace mala
