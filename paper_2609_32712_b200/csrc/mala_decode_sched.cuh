// Order in which the persistent decode kernels take their work items.
//
// A work item is one split of one (sequence, KV head); the splits are laid out for the longest sequence, so a shorter one
// has fewer full splits, one partial split and empty ones (and even sequences of one length leave the last splits empty
// where the split count does not divide their tiles: 129 tiles in 28 splits of 5).  Taken in the order of their numbers (one item per lane of
// work and round), the lanes' loads follow whatever lengths happen to fall on them: 32 sequences of 4000 .. 16000 keys in
// 4 splits left the busiest CTA with 1.74 times the mean (KV head slowest) or 1.33 times (KV head fastest).  Here the items
// are ordered by size -- the full splits, then the partial ones from the largest down, then the empty ones -- and dealt
// out back and forth (round k left to right, round k + 1 right to left): 1.05 times, and the step takes 165 us instead of 241 (bf16, pages of 16 keys);
// 16 sequences of 10000 .. 40000 keys in e4m3 152 instead of 201; 8 sequences of 131072 keys, where only the order of the
// heads changes, 573 instead of 616.  Every CTA works its list out for
// itself from the lengths (seqlens null: all of Nk keys), so nothing has to be set up before the launch or kept after it.
#pragma once
#include <stdint.h>

namespace mala {

// Division of a 32-bit number by a divisor known at launch, as a multiplication and shifts (every role works out for
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

constexpr int kSchedBatch = 512;     // sequences; the tables take 3 * 512 words of shared memory not yet in use
constexpr int kSchedMaxItem = 65535; // item numbers are kept in 16 bits; this one marks the end

// Whether a call with B sequences takes this order (more than one round of items, and the tables fit) on `grid` CTAs that work on per_cta items at a time and have room
// for list_size entries.
inline bool decode_sched_fits(int B, long long n_items, int grid, int per_cta, int list_size) {
  const long long lanes = (long long)grid * per_cta;
  return n_items > grid && B <= kSchedBatch && n_items < kSchedMaxItem && (n_items + lanes - 1) / lanes * per_cta <= list_size;
}

// Fills list[round * PER + k] with the item of lane k * gridDim.x + blockIdx.x in that round (item (b * splits + split) *
// Hkv + hkv; kSchedMaxItem: none).  Called by all threads of the block; `tmp`: 3 * kSchedBatch ints; the caller
// synchronises the block before the list is read.
template <int PER, int kThreads>
__device__ __forceinline__ void decode_schedule(uint16_t* list, int* tmp, const int* seqlens, int B, int Hkv, int splits,
                                                int tps, int Nk, int n_items) {
  constexpr int X = (kSchedBatch + kThreads - 1) / kThreads;
  int* full_to = tmp;                    // [b] full splits of the sequences 0 .. b
  int* part = tmp + kSchedBatch;         // [b] tiles of sequence b, then [r] sequence with the r-th largest partial split
  int* empty_to = tmp + 2 * kSchedBatch; // [b] empty splits of the sequences 0 .. b
  for (int b = threadIdx.x; b < B; b += kThreads) part[b] = ((seqlens ? min(Nk, max(0, __ldg(seqlens + b))) : Nk) + 127) / 128;
  __syncthreads();
  int full_n[X], empty_n[X], rank_n[X];
#pragma unroll
  for (int x = 0; x < X; ++x) {
    const int b = x * kThreads + threadIdx.x;
    full_n[x] = empty_n[x] = 0;
    rank_n[x] = -1;
    if (b < B) {
      const int rem = part[b] % tps;
      int rank = 0;
      for (int y = 0; y < B; ++y) {
        const int t = part[y], f = t / tps, r = t - f * tps;
        if (y <= b) { full_n[x] += f; empty_n[x] += splits - f - (r > 0 ? 1 : 0); }
        if (r > rem || (r == rem && y < b)) ++rank;
      }
      if (rem > 0) rank_n[x] = rank;
    }
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < X; ++x) {
    const int b = x * kThreads + threadIdx.x;
    if (b < B) {
      full_to[b] = full_n[x];
      empty_to[b] = empty_n[x];
      if (rank_n[x] >= 0) part[rank_n[x]] = b;
    }
  }
  __syncthreads();
  const int n_full = full_to[B - 1], n_part = B * splits - n_full - empty_to[B - 1];
  // first sequence whose running count exceeds v
  auto find = [&](const int* to, int v) {
    int lo = 0, hi = B - 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (to[mid] > v) hi = mid; else lo = mid + 1;
    }
    return lo;
  };
  const int lanes = PER * (int)gridDim.x, rounds = (n_items + lanes - 1) / lanes;
  for (int e = threadIdx.x; e < rounds * PER; e += kThreads) {
    const int round = e / PER, lane = (e - round * PER) * (int)gridDim.x + (int)blockIdx.x;
    const int pos = round * lanes + ((round & 1) ? lanes - 1 - lane : lane);
    int item = kSchedMaxItem;
    if (pos < n_items) {
      int s = pos / Hkv, b, split;
      const int hkv = pos - s * Hkv;
      if (s < n_full) {
        b = find(full_to, s);
        split = s - (b > 0 ? full_to[b - 1] : 0);
      } else if (s < n_full + n_part) {
        b = part[s - n_full];
        split = full_to[b] - (b > 0 ? full_to[b - 1] : 0);
      } else {
        s -= n_full + n_part;
        b = find(empty_to, s);
        split = splits - (empty_to[b] - s);
      }
      item = (b * splits + split) * Hkv + hkv;
    }
    list[e] = (uint16_t)item;
  }
}

}  // namespace mala
