// Block-wide selection of the k best (key, id) pairs, best first: larger key, then
// lower id. One block of a power of two of threads; k <= 1024.
//
// The pairs are read through a functor, so a row of scores, a merged list and a
// table in shared memory are selected by the same code. Rows of up to kCap pairs
// are sorted outright. Longer rows are narrowed first: a 2048-bin histogram finds the
// bin that holds the k-th best, and the pairs above it and in it remain -- until they
// fit the sort. The first round bins the score itself in equal steps, which spreads
// cosines and set similarities so well that a row is usually read twice (histogram,
// gather). Later rounds bin the 11 highest of the bits on which the remaining pairs
// differ (found by AND / OR over them), so equal leading bits cost nothing and keys
// that are all equal go straight on to their ids: any values end in at most nine.
// A byte-wise radix select with an ordered compaction, before this, read a row five
// or nine times: merging 1,000 rows of 12,000 took 297 us against 82, 16 rows of 2,000
// 47 us against 11 (where the call on the host is what is timed).
#pragma once
#include "gift_internal.cuh"

namespace gift {
namespace sel {

constexpr int kBins = 2048;  // 11 bits
constexpr int kCap = 2048;   // pairs that are sorted; at least twice the largest k
constexpr unsigned kAll = 0xffffffffu;

struct Smem {
  unsigned long long key[kCap];
  uint32_t id[kCap];
  int hist[kBins];
  int wsum[32];
  uint32_t bits[6];  // AND, OR of the remaining pairs' key (high, low word) and ~id
  int count, bin, above, in_bin;
};

// Bin of a score for the first round, from its order-preserving key: 2,000 equal steps over [0, 1], where
// cosines and set similarities lie, 47 over [-1, 0], the rest at the ends. Not decreasing in the key.
__device__ __forceinline__ int score_bin(uint32_t key) {
  if (key >= 0xBF800000u) return kBins - 1;  // f2key(1): 1 and above
  if (key <= 0x407FFFFFu) return 0;          // f2key(-1): -1 and below
  const float v = key2f(key);
  return v >= 0.f ? 47 + (int)(v * 2000.f) : (int)((v + 1.f) * 46.f);
}

// "a before b"
__device__ __forceinline__ bool before(unsigned long long ka, uint32_t ia, unsigned long long kb, uint32_t ib) {
  return ka > kb || (ka == kb && ia < ib);
}

// The strides 32 .. 1 (or size / 2 .. 1) of a bitonic sort's step `size` on the 64 pairs from
// `base` on, two per lane in registers: 24 instructions a stride and no shared memory, where a
// stride through shared memory takes 50 and its latency.
struct Two {
  unsigned long long k0, k1;
  uint32_t i0, i1;
};
__device__ __forceinline__ void sort_step64(Two& x, int base, int size) {
  const int lane = threadIdx.x & 31;
  const int e0 = base + lane, e1 = e0 + 32;
  int stride = min(32, size >> 1);
  if (stride == 32) {
    const bool up = (e0 & size) == 0;
    if (up ? before(x.k1, x.i1, x.k0, x.i0) : before(x.k0, x.i0, x.k1, x.i1)) {
      const unsigned long long k = x.k0;
      const uint32_t i = x.i0;
      x.k0 = x.k1;
      x.i0 = x.i1;
      x.k1 = k;
      x.i1 = i;
    }
    stride = 16;
  }
  for (; stride > 0; stride >>= 1) {
    const bool lower = (lane & stride) == 0;
    const unsigned long long k0 = __shfl_xor_sync(kAll, x.k0, stride), k1 = __shfl_xor_sync(kAll, x.k1, stride);
    const uint32_t i0 = __shfl_xor_sync(kAll, x.i0, stride), i1 = __shfl_xor_sync(kAll, x.i1, stride);
    if (before(k0, i0, x.k0, x.i0) == (lower == ((e0 & size) == 0))) {
      x.k0 = k0;
      x.i0 = i0;
    }
    if (before(k1, i1, x.k1, x.i1) == (lower == ((e1 & size) == 0))) {
      x.k1 = k1;
      x.i1 = i1;
    }
  }
}

// Bitonic sort, best first, of the first P (a power of two, at least 64) pairs; starts
// and ends with a barrier
__device__ __forceinline__ void sort_pairs(unsigned long long* key, uint32_t* id, int P) {
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31;
  auto steps64 = [&](int first, int last) {
    for (int base = 64 * w; base < P; base += 64 * nw) {
      Two x{key[base + lane], key[base + 32 + lane], id[base + lane], id[base + 32 + lane]};
      for (int size = first; size <= last; size <<= 1) sort_step64(x, base, size);
      key[base + lane] = x.k0;
      key[base + 32 + lane] = x.k1;
      id[base + lane] = x.i0;
      id[base + 32 + lane] = x.i1;
    }
  };
  __syncthreads();
  steps64(2, 64);
  __syncthreads();
  for (int size = 128; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 32; stride >>= 1) {
      for (int t = threadIdx.x; t < P / 2; t += blockDim.x) {
        const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
        const bool up = (lo & size) == 0;
        const unsigned long long kl = key[lo], kh = key[hi];
        const uint32_t il = id[lo], ih = id[hi];
        if (up ? before(kh, ih, kl, il) : before(kl, il, kh, ih)) {
          key[lo] = kh;
          key[hi] = kl;
          id[lo] = ih;
          id[hi] = il;
        }
      }
      __syncthreads();
    }
    steps64(size, size);
    __syncthreads();
  }
}

// pads the first `have` pairs to a power of two and sorts them
__device__ __forceinline__ void sort_have(Smem& sm, int have) {
  int P = 64;
  while (P < have) P <<= 1;
  for (int t = have + threadIdx.x; t < P; t += blockDim.x) {
    sm.key[t] = 0ull;
    sm.id[t] = 0xffffffffu;
  }
  sort_pairs(sm.key, sm.id, P);
}

// f(valid, key, id) for every i < n, Get::kAhead reads in flight; every lane of a warp
// calls f the same number of times
template <class Get, class F>
__device__ __forceinline__ void for_pairs(const Get& get, int64_t n, const F& f) {
  constexpr int U = Get::kAhead;
  const int T = blockDim.x;
  for (int64_t base = 0; base < n; base += U * T) {
    unsigned long long key[U];
    uint32_t id[U];
    bool ok[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int64_t i = base + j * T + threadIdx.x;
      ok[j] = i < n && get(i, key[j], id[j]);
    }
#pragma unroll
    for (int j = 0; j < U; ++j)
      if (base + j * T < n) f(ok[j], key[j], id[j]);
  }
}

// appends the pairs with take to sm.key / sm.id (at most kCap)
__device__ __forceinline__ void append(Smem& sm, bool take, unsigned long long key, uint32_t id) {
  const int lane = threadIdx.x & 31;
  const unsigned m = __ballot_sync(kAll, take);
  if (!m) return;
  int base = 0;
  if (lane == 0) base = atomicAdd(&sm.count, __popc(m));
  base = __shfl_sync(kAll, base, 0);
  const int at = base + __popc(m & ((1u << lane) - 1u));
  if (take && at < kCap) {
    sm.key[at] = key;
    sm.id[at] = id;
  }
}

// exclusive prefix sum of one int per thread over the block
__device__ __forceinline__ int block_prefix(Smem& sm, int v) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kAll, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sm.wsum[w] = x;
  __syncthreads();
  if (w == 0) {
    const int y = lane < nw ? sm.wsum[lane] : 0;
    int z = y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int q = __shfl_up_sync(kAll, z, o);
      if (lane >= o) z += q;
    }
    if (lane < nw) sm.wsum[lane] = z - y;
  }
  __syncthreads();
  const int r = x - v + sm.wsum[w];
  __syncthreads();
  return r;
}

// The k best of the n pairs get(i) (`valid` of them valid; n when every one is), left
// sorted in sm.key / sm.id; returns how many there are (min(k, valid)). Ends with a
// barrier. Ids are distinct. get.score(key) is the key's score word.
template <class Get>
__device__ int select(Smem& sm, const Get& get, int64_t n, int64_t valid, int k) {
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
  int bin0 = 0;                             // the remaining pairs have score_bin == bin0 (first round), ...
  unsigned long long mk = 0ull, pk = 0ull;  // ... (key & mk) == pk ...
  uint32_t ml = 0u, pl = 0u;                // ... and (~id & ml) == pl (later rounds)
  bool binned = false;
  int64_t above = 0, in_bin = valid;        // pairs above them, and how many remain
  bool equal = false;                       // the remaining pairs are copies of one pair
  auto remains = [&](unsigned long long key, uint32_t id) {
    return (!binned || score_bin(Get::score(key)) == bin0) && (key & mk) == pk && (~id & ml) == pl;
  };
  // counts d (-1: none) of the warp's lanes: lanes that share a bin by one atomic as long as the groups found are of
  // four or more (scores of a few bins, or a row that few shapes reach), and the rest one each (256 rows of 200,000
  // scores of 400 classes: 775 us with one group, 738)
  auto count_bin = [&](int d) {
    unsigned m = __ballot_sync(kAll, d >= 0);
    if (!m) return;
    int group;
    do {
      const int lead = __ffs(m) - 1, d0 = __shfl_sync(kAll, d, lead);
      const unsigned same = __ballot_sync(kAll, d == d0);
      group = __popc(same);
      if (lane == lead) atomicAdd(&sm.hist[d0], group);
      m &= ~same;
    } while (m && group >= 4);
    if (m >> lane & 1u) atomicAdd(&sm.hist[d], 1);
  };
  // the bin of the k-th best (threads own runs of bins, best bin first) -> sm.bin, sm.above, sm.in_bin
  auto find_bin = [&]() {
    __syncthreads();
    const int per = kBins / T;
    int own = 0;
    for (int j = 0; j < per; ++j) own += sm.hist[kBins - 1 - (tid * per + j)];
    const int pre = block_prefix(sm, own);
    const int need = (int)(k - above);
    if (pre < need && need <= pre + own) {
      int cum = pre, b = kBins - 1 - tid * per;
      while (cum + sm.hist[b] < need) cum += sm.hist[b--];
      sm.bin = b;
      sm.above = cum;
      sm.in_bin = sm.hist[b];
    }
    __syncthreads();
    above += sm.above;
    in_bin = sm.in_bin;
  };
  auto clear = [&]() {
    for (int b = tid; b < kBins; b += T) sm.hist[b] = 0;
    if (tid < 6) sm.bits[tid] = (tid & 1) ? 0u : 0xffffffffu;
    if (tid == 0) sm.count = 0;
    __syncthreads();
  };
  clear();
  if (valid > max(256, 2 * k)) {  // also where a sort would hold all: one of fewer pairs is cheaper
    for_pairs(get, n, [&](bool ok, unsigned long long key, uint32_t) {
      count_bin(ok ? score_bin(Get::score(key)) : -1);
    });
    find_bin();
    binned = true;
    bin0 = sm.bin;
  }
  while (above + in_bin > kCap) {
    __syncthreads();
    clear();
    uint32_t a0 = kAll, o0 = 0u, a1 = kAll, o1 = 0u, a2 = kAll, o2 = 0u;
    for_pairs(get, n, [&](bool ok, unsigned long long key, uint32_t id) {
      if (ok && remains(key, id)) {
        const uint32_t h = (uint32_t)(key >> 32), l = (uint32_t)key;
        a0 &= h;
        o0 |= h;
        a1 &= l;
        o1 |= l;
        a2 &= ~id;
        o2 |= ~id;
      }
    });
    a0 = __reduce_and_sync(kAll, a0);
    o0 = __reduce_or_sync(kAll, o0);
    a1 = __reduce_and_sync(kAll, a1);
    o1 = __reduce_or_sync(kAll, o1);
    a2 = __reduce_and_sync(kAll, a2);
    o2 = __reduce_or_sync(kAll, o2);
    if (lane == 0) {
      atomicAnd(&sm.bits[0], a0);
      atomicOr(&sm.bits[1], o0);
      atomicAnd(&sm.bits[2], a1);
      atomicOr(&sm.bits[3], o1);
      atomicAnd(&sm.bits[4], a2);
      atomicOr(&sm.bits[5], o2);
    }
    __syncthreads();
    const unsigned long long kand = ((unsigned long long)sm.bits[0] << 32) | sm.bits[2];
    const unsigned long long kdiff = kand ^ (((unsigned long long)sm.bits[1] << 32) | sm.bits[3]);
    const uint32_t iand = sm.bits[4], idiff = iand ^ sm.bits[5];
    if (kdiff == 0ull && idiff == 0u) {
      equal = true;
      mk = ~0ull;
      pk = kand;
      ml = kAll;
      pl = iand;
      break;
    }
    const bool by_key = kdiff != 0ull;
    const int top = by_key ? 63 - __clzll((long long)kdiff) : 31 - __clz((int)idiff);
    const int shift = max(0, top - 10);
    for_pairs(get, n, [&](bool ok, unsigned long long key, uint32_t id) {
      // bits above `top` are common, so a digit's unused high bits are too
      count_bin(ok && remains(key, id)
                    ? (int)((by_key ? key >> shift : (unsigned long long)(~id >> shift)) & (kBins - 1))
                    : -1);
    });
    find_bin();
    if (by_key) {
      mk = ~0ull << shift;
      pk = (kand & (top == 63 ? 0ull : ~0ull << (top + 1))) |
           ((unsigned long long)(sm.bin & ((2u << (top - shift)) - 1u)) << shift);
    } else {
      mk = ~0ull;
      pk = kand;
      ml = kAll << shift;
      pl = (iand & (top == 31 ? 0u : kAll << (top + 1))) | ((uint32_t)(sm.bin & ((2u << (top - shift)) - 1u)) << shift);
    }
  }
  // gather (sm.count is 0)
  if (mk == 0ull && !equal) {
    for_pairs(get, n, [&](bool ok, unsigned long long key, uint32_t id) {
      append(sm, ok && (!binned || score_bin(Get::score(key)) >= bin0), key, id);
    });
  } else {
    for_pairs(get, n, [&](bool ok, unsigned long long key, uint32_t id) {
      const unsigned long long x = key & mk;
      const int c = binned ? score_bin(Get::score(key)) - bin0 : 0;
      append(sm, ok && (c > 0 || (c == 0 && (x > pk || (x == pk && (equal ? (~id & ml) > pl : (~id & ml) >= pl))))),
             key, id);
    });
  }
  if (equal) {  // then as many of the copies as fit
    __syncthreads();
    for_pairs(get, n, [&](bool ok, unsigned long long key, uint32_t id) {
      append(sm, ok && remains(key, id), key, id);
    });
  }
  __syncthreads();
  const int have = min(sm.count, kCap);
  __syncthreads();
  sort_have(sm, have);
  return min(have, k);
}

}  // namespace sel
}  // namespace gift
