// Second inverted file (Fig. 3) and context re-ranking (Eqs. 7, 8, 13, 14).
//
// Build: every database shape p, matched as a query, gives its first k1
// neighbours N_k1(p) (itself included) with memberships F_p[i] = S(x_p, x_i)
// (Eq. 7). The pairs (p, i) are transposed by a stable counting sort keyed
// by i: entry i lists every p with F_p[i] != 0 in ascending p, with the
// membership as uint32 fixed point round(S * 2^31); ||F_p||_1 is the sum of
// p's k1 fixed-point memberships (uint64, exact).
//
// Re-rank: F_q comes from the first k1 candidates of the query. For each
// non-zero F_q[i] the entry i is walked and min(F_q[i], F_p[i]) is added to
// p's numerator (Eq. 13, integer atomics: exact and order-free). Then
// S' = num / (||F_q||_1 + ||F_p||_1 - num) (Eq. 14) in FP32, and the final
// order (S' desc, S desc, id asc) is a top-k over 64-bit keys
// (key(S') << 32 | key(S)) with ties to the lower id. One block per query does it
// all in shared memory (k_rerank_reach), or, for long walks of few queries and on
// caller-provided scratch, kernels over dense rows of all shapes (dense_rerank).
//
// Two measures (Sec. 2.4, Eqs. 9-11): a block per shape (database or query)
// gathers the activations that make up its two contextual activations — its
// own Eq. 7 rows, or the Eq. 7 rows of its first k2 neighbours under the same
// measure (Eq. 10) or the other one (Eq. 11) — as (id, measure, source) keys,
// sorts them in shared memory, sums each (id, measure) group in source order
// and divides by k2, and fuses the two measures per id with the generalised
// mean of Eq. 9. The database activations are transposed into a second
// inverted file of their own; a query's activation is walked through it as in
// the one-measure re-rank.
#include <cmath>

#include "gift_internal.cuh"
#include "select.cuh"

namespace gift {

namespace {

__device__ __forceinline__ uint32_t member_fix(float S) {
  const float c = fminf(fmaxf(S, 0.f), 1.f);
  return __float2uint_rn(c * 2147483648.0f);
}

__global__ void k_sif_keys(const int32_t* __restrict__ nbr_ids, int64_t n, int32_t N, int32_t* keys,
                           int* bad) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t id = nbr_ids[i];
  if (id < 0 || id >= N) {
    atomicExch(bad, 1);
    keys[i] = 0;
  } else {
    keys[i] = id;
  }
}

__global__ void k_sif_fill(const int32_t* __restrict__ perm, int64_t n, int k1,
                           const float* __restrict__ nbr_scores, int32_t* __restrict__ ids,
                           uint32_t* __restrict__ mem) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int32_t pair = perm[e];
  ids[e] = pair / k1;
  mem[e] = member_fix(nbr_scores[pair]);
}

__global__ void k_sif_card(const float* __restrict__ nbr_scores, int32_t N, int k1,
                           unsigned long long* __restrict__ card) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  unsigned long long c = 0;
  for (int r = 0; r < k1; ++r) c += member_fix(nbr_scores[p * k1 + r]);
  card[p] = c;
}

// ---------------------------------------------------------------- what a query's walk will take
// Found when an inverted file is built, by walking it from some of its own shapes, whose rows are what queries bring
constexpr int kSamples = 64;
constexpr int kSampleBits = 1 << 18;
constexpr int kSampleCoords = 128;  // of a row, spread over it; and a warp walks so many pairs, which fill any table if their
constexpr int kSamplePairs = 8192;  // shapes differ (a whole row of 1,000 long entries took 190 us)
struct Sample {
  unsigned long long pairs;   // shapes in the entries of the coordinates looked at
  unsigned long long coords;  // those coordinates
  int row;                    // all coordinates of the row
  int blank;                  // bits that no shape's hash sets
};

// block j: row j N / samples of `rows` [N, ld], cnt[.] (null: ld) coordinates; longest[0]: the longest entry (zeroed)
__global__ __launch_bounds__(512) void k_walk_sample(const int32_t* __restrict__ rows, int ld,
                                                     const int32_t* __restrict__ cnt, int32_t N, int samples,
                                                     const int64_t* __restrict__ off, const int32_t* __restrict__ ids,
                                                     Sample* __restrict__ out, int* __restrict__ longest) {
  __shared__ uint32_t bits[kSampleBits / 32];
  __shared__ unsigned long long pairs, coords;
  __shared__ int blank;
  const int t = threadIdx.x, T = blockDim.x, lane = t & 31;
  if (t == 0) {
    pairs = coords = 0ull;
    blank = 0;
  }
  for (int i = t; i < kSampleBits / 32; i += T) bits[i] = 0u;
  __syncthreads();
  int most = 0;
  for (int64_t i = (int64_t)blockIdx.x * T + t; i < N; i += (int64_t)gridDim.x * T)
    most = max(most, (int)(off[i + 1] - off[i]));
  most = __reduce_max_sync(0xffffffffu, most);
  if (lane == 0) atomicMax(longest, most);
  const int64_t p = (int64_t)blockIdx.x * N / samples;
  const int n = cnt ? cnt[p] : ld;
  const int looked = min(n, kSampleCoords);
  int64_t walked = 0;
  for (int j = t >> 5; j < looked; j += T >> 5) {
    const int32_t i = rows[p * ld + (int64_t)j * n / looked];
    if (i < 0 || i >= N) continue;
    const int64_t e0 = off[i], e1 = off[i + 1];
    if (lane == 0) {
      atomicAdd(&pairs, (unsigned long long)(e1 - e0));
      atomicAdd(&coords, 1ull);
    }
    const int64_t to = min(e1, e0 + max((int64_t)0, kSamplePairs - walked));
    walked += e1 - e0;
    for (int64_t e = e0 + lane; e < to; e += 32) {
      const uint32_t h = (uint32_t)ids[e] * 2654435761u >> 14;
      atomicOr(bits + (h >> 5), 1u << (h & 31u));
    }
  }
  __syncthreads();
  int own = 0;
  for (int i = t; i < kSampleBits / 32; i += T) own += 32 - __popc(bits[i]);
  own = __reduce_add_sync(0xffffffffu, own);
  if (lane == 0) atomicAdd(&blank, own);
  __syncthreads();
  if (t == 0) out[blockIdx.x] = Sample{pairs, coords, n, blank};
}

WalkStats walk_stats(const int32_t* rows, int ld, const int32_t* cnt, int32_t N, const int64_t* off, const int32_t* ids,
                     Scratch& sc, cudaStream_t s) {
  const int n = std::min(N, kSamples);
  Sample* d = sc.get<Sample>(kSamples);
  int* longest = sc.get<int>(1);
  GIFT_CUDA(cudaMemsetAsync(longest, 0, sizeof(int), s));
  k_walk_sample<<<(unsigned)n, 512, 0, s>>>(rows, ld, cnt, N, n, off, ids, d, longest);
  GIFT_LAUNCHED("k_walk_sample");
  Sample h[kSamples];
  WalkStats w;
  GIFT_CUDA(cudaMemcpyAsync(h, d, n * sizeof(Sample), cudaMemcpyDeviceToHost, s));
  GIFT_CUDA(cudaMemcpyAsync(&w.longest, longest, sizeof(int), cudaMemcpyDeviceToHost, s));
  GIFT_CUDA(cudaStreamSynchronize(s));
  double pairs = 0., coords = 0., rows_coords = 0., reach = 0.;
  for (int j = 0; j < n; ++j) {
    pairs += (double)h[j].pairs;
    coords += (double)h[j].coords;
    rows_coords += h[j].row;
    reach += std::min<double>(N, -(double)kSampleBits * std::log(std::max(h[j].blank, 1) / (double)kSampleBits));
  }
  w.coords = rows_coords / n;
  w.met = coords > 0. ? pairs / coords : 0.;
  w.reach = reach / n;
  return w;
}

// ---------------------------------------------------------------- re-rank of one query per block
// A query reaches few shapes: its candidates and the shapes in its k1 S-IF entries, a few
// thousand (shape, membership) pairs however large the database. One block takes one query and
// keeps the numerators and the tie-break scores in shared memory: a table with a row per shape
// where all N fit, a hash table of the reached shapes otherwise. It walks the entries (a warp
// per entry), turns the rows into ranking keys, selects the top-k and writes it -- nothing of
// the size of the database is cleared, written or scanned in global memory. What is left is a
// few dependent global reads (candidate, entry offsets, entry), then shared-memory passes.
// Measured, whole calls (256 queries, k1 = 50, 200,000 shapes): 552 us with dense [B, N] rows in
// global memory and six launches, 28 us here; two measures, 1,000 queries, 12,000 shapes: 756 and
// 240 us, 180 of them this kernel (a query there adds some 55,000 pairs).
//
// Unreached shapes all have the key (S' = 0, S = -inf). Where they are needed (fewer reached
// shapes than the top-k) they follow in id order. A hash table that overflows (a query that
// reaches more shapes than its slots) is given up, and the block walks again into a row of
// the whole database in global memory. Without such a row (no memory for one, or entries too short
// to fill the slots but unluckily placed) it goes over the database in ranges of as many shapes
// as its table holds, merging each range's best with those before. (Ranges alone, after a walk that went
// on in a full table, took 29.7 ms where rows take 5.5 now and dense rows 8.9: 256 queries, 200,000 shapes,
// k1 = 1,000.)
struct ReachArgs {
  int32_t N;                     // shapes
  const int32_t* cand_ids;       // [B, n_cand]
  const float* cand_scores;
  int n_cand;
  int k1;                        // F_q: the first k1 candidates (act_ids null), or
  const int32_t* act_ids;        // [B, act_ld] the non-zero coordinates of the activation,
  const uint32_t* act_mem;       //   their fixed-point values,
  const int32_t* act_cnt;        //   [B] how many, and
  const unsigned long long* act_norm;  // [B] their sum
  int act_ld;
  const int64_t* off;            // the inverted file and the shapes' norms
  const int32_t* ids;
  const uint32_t* mem;
  const unsigned long long* card;
  int topk;
  int32_t* out_ids;              // [B, topk]
  float* out_sprime;
  int table_bytes;               // dynamic shared memory
  int hash;                      // 1: hash table first; 0: one range when all shapes fit, else as after an overflow
  unsigned long long* win_key;   // [B, topk] the best of the ranges gone over so far
  uint32_t* win_id;
  unsigned long long* num;       // [B, N] numerators and tie-break scores of queries that no table holds,
  float* S;                      //   or null (ranges of shapes)
};
__host__ __device__ __forceinline__ int reach_coords(const ReachArgs& a) { return a.act_ids ? a.act_ld : a.k1; }

// coordinate r of query b's activation: its shape (-1: none) and fixed-point value (0: nothing to add)
__device__ __forceinline__ int32_t reach_coord(const ReachArgs& a, int b, int r, uint32_t& fq) {
  const int64_t at = (int64_t)b * (a.act_ids ? a.act_ld : a.n_cand) + r;
  const int32_t i = a.act_ids ? a.act_ids[at] : a.cand_ids[at];
  fq = 0;
  if (i < 0 || i >= a.N) return -1;
  fq = a.act_ids ? a.act_mem[at] : member_fix(a.cand_scores[at]);
  return i;
}

constexpr int kReachProbes = 64;  // slots tried before a hash table counts as full
constexpr uint32_t kNoKey = 0u;   // high key word of a row that is not reached (a real one is >= 0x80000000)

__device__ __forceinline__ uint32_t reach_slot(int32_t id, int slots) {
  return __umulhi((uint32_t)id * 2654435761u, (uint32_t)slots);
}

// row of a range's o-th shape: shapes of a class often sit at a fixed stride, whose multiples would fall in a few of
// the 32 banks (stride 40: four), so the low five bits are mixed with the next five; its own inverse
__device__ __forceinline__ int reach_row(int o) { return o ^ ((o >> 5) & 31); }

// exact 64-bit sum in two native 32-bit words
__device__ __forceinline__ void reach_add(uint32_t* lo, uint32_t* hi, int at, uint32_t v) {
  const uint32_t old = atomicAdd(lo + at, v);
  if (old > ~v) atomicAdd(hi + at, 1u);
}

// every pair of the query's entries: f(shape, min(F_q[i], F_p[i])); a lane fetches what one
// coordinate needs, then the warp reads the 32 coordinates' entries in turn
template <class F>
__device__ __forceinline__ void reach_walk(const ReachArgs& a, int b, const F& f) {
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31;
  const int cnt = a.act_ids ? a.act_cnt[b] : a.k1;
  for (int r0 = w; r0 < cnt; r0 += nw * 32) {
    const int r = r0 + nw * lane;
    int64_t e0 = 0;
    int len = 0;
    uint32_t fq = 0;
    if (r < cnt) {
      const int32_t i = reach_coord(a, b, r, fq);
      if (fq) {
        e0 = a.off[i];
        len = (int)(a.off[i + 1] - e0);
      }
    }
    for (int j = 0; j < 32 && r0 + nw * j < cnt; ++j) {
      const int64_t ej = __shfl_sync(0xffffffffu, e0, j);
      const int nj = __shfl_sync(0xffffffffu, len, j);
      const uint32_t fj = __shfl_sync(0xffffffffu, fq, j);
      for (int e = lane; e < nj; e += 128) {
        int32_t id[4];
        uint32_t m[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool in = e + 32 * u < nj;
          id[u] = in ? a.ids[ej + e + 32 * u] : 0;
          m[u] = in ? a.mem[ej + e + 32 * u] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (m[u]) f(id[u], min(fj, m[u]));
      }
    }
  }
}

// ranking key of shape p: (S' of Eqs. 13 and 14, S)
__device__ __forceinline__ unsigned long long reach_key(unsigned long long nm, unsigned long long fq_norm,
                                                        const unsigned long long* card, int32_t p, float s) {
  float sp = 0.f;
  if (nm > 0) sp = __fdiv_rn(__ull2float_rn(nm), __ull2float_rn(fq_norm + card[p] - nm));
  return ((unsigned long long)f2key(sp) << 32) | (unsigned long long)f2key(s);
}

// id of row i of the table: its own (hash) or the range's; then the winners of earlier ranges
struct ReachRows {
  static constexpr int kAhead = 4;
  static __device__ __forceinline__ uint32_t score(unsigned long long key) { return (uint32_t)(key >> 32); }
  const uint32_t* lo;
  const uint32_t* hi;
  const int32_t* hid;   // hash: the row's id
  int32_t r0;           // range: the first id
  int rows;
  const unsigned long long* wkey;
  const uint32_t* wid;
  __device__ __forceinline__ bool operator()(int64_t i, unsigned long long& key, uint32_t& id) const {
    if (i >= rows) {
      key = wkey[i - rows];
      id = wid[i - rows];
      return true;
    }
    const uint32_t h = hi[i];
    key = ((unsigned long long)h << 32) | lo[i];
    id = hid ? (uint32_t)hid[i] : (uint32_t)(r0 + reach_row((int)i));
    return h != kNoKey;
  }
};

struct DenseRows {  // a query's row of every shape, in global memory
  static constexpr int kAhead = 4;
  static __device__ __forceinline__ uint32_t score(unsigned long long key) { return (uint32_t)(key >> 32); }
  const unsigned long long* num;
  const float* S;
  const unsigned long long* card;
  unsigned long long fq_norm;
  __device__ __forceinline__ bool operator()(int64_t i, unsigned long long& key, uint32_t& id) const {
    key = reach_key(__ldcg(num + i), fq_norm, card, (int32_t)i, __ldcg(S + i));
    id = (uint32_t)i;
    return true;
  }
};

struct ReachList {  // listed rows
  static constexpr int kAhead = 4;
  static __device__ __forceinline__ uint32_t score(unsigned long long key) { return (uint32_t)(key >> 32); }
  ReachRows rows;
  const int32_t* list;
  __device__ __forceinline__ bool operator()(int64_t i, unsigned long long& key, uint32_t& id) const {
    return rows(list[i], key, id);
  }
};
constexpr int kReachList = 2048;

// table of N shapes in one range, rows rounded up to the 32 that reach_row mixes
__host__ __device__ __forceinline__ int64_t reach_rows_bytes(int64_t N) { return (N + 31) / 32 * 32 * 12; }

template <bool ROWS>
__global__ __launch_bounds__(1024) void k_rerank_reach(const ReachArgs a) {
  extern __shared__ __align__(16) uint32_t table[];
  __shared__ sel::Smem sm;
  __shared__ unsigned long long s_norm;
  __shared__ int32_t list[kReachList];
  __shared__ int s_flag, s_end, s_listed;
  const int b = blockIdx.x, t = threadIdx.x, T = blockDim.x;
  const int32_t* cid = a.cand_ids + (int64_t)b * a.n_cand;
  const float* csc = a.cand_scores + (int64_t)b * a.n_cand;
  if (t == 0) {
    s_norm = a.act_ids ? a.act_norm[b] : 0ull;
    s_flag = 0;
    s_listed = 0;
  }
  __syncthreads();
  if (!a.act_ids)
    for (int base = t - (t & 31); base < a.k1; base += T) {  // a warp's sum, then one 64-bit atomic
      const int c = base + (t & 31);
      unsigned long long f = c < a.k1 && cid[c] >= 0 && cid[c] < a.N ? member_fix(csc[c]) : 0u;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
      if ((t & 31) == 0) atomicAdd(&s_norm, f);
    }
  const int need = min(a.topk, a.N);
  int take = 0;

  // rows of the table: numerator (two words), S, and the id of a hash slot
  bool hashed = a.hash != 0;
  const bool one = reach_rows_bytes(a.N) <= a.table_bytes;
  const int W = (one ? (a.N + 31) : a.table_bytes / 12) & ~31;  // shapes of a range
  int rows = hashed ? a.table_bytes / 16 : W;
  uint32_t* lo = table;
  uint32_t* hi = lo + rows;
  float* S = reinterpret_cast<float*>(hi + rows);
  int32_t* hid = reinterpret_cast<int32_t*>(S + rows);
  auto reached = [&](int i) { return (lo[i] | hi[i]) != 0u || S[i] != -INFINITY; };
  auto numerator = [&](int i) { return ((unsigned long long)hi[i] << 32) | lo[i]; };

  if (hashed) {
    for (int i = t; i < rows; i += T) {
      lo[i] = 0u;
      hi[i] = 0u;
      S[i] = -INFINITY;
      hid[i] = -1;
    }
    __syncthreads();
    bool full = false;  // a lane that found none adds no more (a stop of the whole walk, asked for at every entry,
                        // cost walks of 1,000 entries 7%)
    auto slot_of = [&](int32_t id) {  // the shape's slot, taken if it has none; -1: none left near
      uint32_t h = reach_slot(id, rows);
      for (int n = 0; n < kReachProbes; ++n) {
        int32_t cur = *reinterpret_cast<volatile int32_t*>(hid + h);
        if (cur == -1) cur = atomicCAS(hid + h, -1, id);
        if (cur == -1 || cur == id) return (int)h;
        if (++h == (uint32_t)rows) h = 0;
      }
      s_flag = 1;
      full = true;
      return -1;
    };
    for (int c = t; c < a.n_cand; c += T)
      if (cid[c] >= 0 && cid[c] < a.N) {
        const int at = slot_of(cid[c]);
        if (at >= 0) S[at] = csc[c];
      }
    reach_walk(a, b, [&](int32_t id, uint32_t v) {
      if (full) return;
      const int at = slot_of(id);
      if (at >= 0) reach_add(lo, hi, at, v);
    });
    __syncthreads();
    hashed = s_flag == 0;
    if (!hashed) {  // the table overflowed
      rows = W;
      hi = lo + rows;
      S = reinterpret_cast<float*>(hi + rows);
    }
  }
  const bool dense = ROWS && !hashed, ranges = !hashed && !one && !dense;
  if (ROWS && dense) {  // a row of every shape
    unsigned long long* num = a.num + (int64_t)b * a.N;
    float* Sg = a.S + (int64_t)b * a.N;
    for (int64_t i = t; i < a.N; i += T) {
      num[i] = 0ull;
      Sg[i] = -INFINITY;
    }
    __syncthreads();
    for (int c = t; c < a.n_cand; c += T)
      if (cid[c] >= 0 && cid[c] < a.N) Sg[cid[c]] = csc[c];
    reach_walk(a, b, [&](int32_t id, uint32_t v) { atomicAdd(num + id, (unsigned long long)v); });
    __syncthreads();
    take = sel::select(sm, DenseRows{num, Sg, a.card, s_norm}, a.N, a.N, need);
  }
  for (int64_t r0 = 0; !hashed && !dense && r0 < a.N; r0 += W) {
    const int n = (int)min((int64_t)W, a.N - r0);
    __syncthreads();
    for (int i = t; i < rows; i += T) {
      lo[i] = 0u;
      hi[i] = 0u;
      S[i] = -INFINITY;
    }
    __syncthreads();
    for (int c = t; c < a.n_cand; c += T)
      if (cid[c] >= r0 && cid[c] < r0 + n) S[reach_row((int)(cid[c] - r0))] = csc[c];
    reach_walk(a, b, [&](int32_t id, uint32_t v) {
      if (id >= r0 && id < r0 + n) reach_add(lo, hi, reach_row((int)(id - r0)), v);
    });
    __syncthreads();
    if (!ranges) break;
    // every shape of the range, reached or not, against the winners of the ranges before
    for (int i = t; i < rows; i += T) {
      const int o = reach_row(i);
      const unsigned long long key = o < n ? reach_key(numerator(i), s_norm, a.card, (int32_t)r0 + o, S[i]) : 0ull;
      hi[i] = (uint32_t)(key >> 32);  // kNoKey past the range
      lo[i] = (uint32_t)key;
    }
    __syncthreads();
    unsigned long long* wkey = a.win_key + (int64_t)b * a.topk;
    uint32_t* wid = a.win_id + (int64_t)b * a.topk;
    const int win = take;
    take = sel::select(sm, ReachRows{lo, hi, nullptr, (int32_t)r0, rows, wkey, wid}, rows + win, n + win, need);
    for (int i = t; i < take; i += T) {
      wkey[i] = sm.key[i];
      wid[i] = sm.id[i];
    }
    __syncthreads();
  }

  if (!ranges && !dense) {
    // the reached rows, listed first, so that their keys' reads of the norms go out together
    const int lane = t & 31;
    for (int base = 0; base < rows; base += T) {
      const int i = base + t;
      const bool in = i < rows && reached(i);
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (!m) continue;
      int at = 0;
      if (lane == 0) at = atomicAdd(&s_listed, __popc(m));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
      if (in && at < kReachList) list[at] = i;
    }
    __syncthreads();
    const int M = s_listed;
    const bool listed = M <= kReachList;
    const int32_t* ids = hashed ? hid : nullptr;
    // their keys in place (of every row where the list is full)
    auto set_key = [&](int i) {
      const unsigned long long key =
          reached(i) ? reach_key(numerator(i), s_norm, a.card, ids ? ids[i] : reach_row(i), S[i]) : 0ull;
      hi[i] = (uint32_t)(key >> 32);
      lo[i] = (uint32_t)key;
    };
    if (listed) {
      for (int j = t; j < M; j += T) set_key(list[j]);
      __syncthreads();
      take = sel::select(sm, ReachList{ReachRows{lo, hi, ids, 0, rows, nullptr, nullptr}, list}, M, M, need);
    } else {
      for (int i = t; i < rows; i += T) set_key(i);
      __syncthreads();
      take = sel::select(sm, ReachRows{lo, hi, ids, 0, rows, nullptr, nullptr}, rows, M, need);
    }
    if (take < need) {  // the unreached shapes of the lowest ids fill up (listed: M < need; other rows hold zeros)
      const unsigned long long none = ((unsigned long long)f2key(0.f) << 32) | (unsigned long long)f2key(-INFINITY);
      for (int64_t c0 = 0; c0 < a.N && take < need; c0 += T) {
        const int64_t id = c0 + t;
        bool free = id < a.N;
        if (free && !hashed) {
          free = hi[reach_row((int)id)] == kNoKey;
        } else if (free) {
          uint32_t h = reach_slot((int32_t)id, rows);
          for (int n = 0; n < kReachProbes && hid[h] != -1; ++n) {
            if (hid[h] == (int32_t)id) {
              free = hi[h] == kNoKey;
              break;
            }
            if (++h == (uint32_t)rows) h = 0;
          }
        }
        const int at = take + sel::block_prefix(sm, free ? 1 : 0);
        if (free && at < need) {
          sm.key[at] = none;
          sm.id[at] = (uint32_t)id;
        }
        if (t == T - 1) s_end = at + (free ? 1 : 0);
        __syncthreads();
        take = min(need, s_end);
        __syncthreads();
      }
      sel::sort_have(sm, take);
    }
  }
  for (int i = t; i < a.topk; i += T) {
    const bool ok = i < take;
    a.out_ids[(int64_t)b * a.topk + i] = ok ? (int32_t)sm.id[i] : -1;
    a.out_sprime[(int64_t)b * a.topk + i] = ok ? key2f((uint32_t)(sm.key[i] >> 32)) : -INFINITY;
  }
}

// ---------------------------------------------------------------- re-rank on dense rows
// Five kernels over [B, N] rows in global memory: a query's walk spreads over as many blocks as it has
// coordinates.
inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
size_t dense_bytes(int32_t B, int32_t N, int32_t topk) {
  const size_t BN = (size_t)B * (size_t)N;
  return align256(BN * 8) + align256(BN * 4) + align256((size_t)B * 8) + align256(BN * 8) +
         align256((size_t)B * (size_t)topk * 8);
}

// ||F_q||_1 per query and the dense S row of the candidates (-inf elsewhere)
__global__ void k_rerank_prep(const ReachArgs a, float* __restrict__ Srow, unsigned long long* __restrict__ fq_norm) {
  const int b = blockIdx.x;
  __shared__ unsigned long long tot;
  if (threadIdx.x == 0) tot = 0;
  __syncthreads();
  for (int t = threadIdx.x; t < a.n_cand; t += blockDim.x) {
    const int32_t id = a.cand_ids[(int64_t)b * a.n_cand + t];
    const float sc = a.cand_scores[(int64_t)b * a.n_cand + t];
    if (id >= 0 && id < a.N) {
      Srow[(int64_t)b * a.N + id] = sc;
      if (t < a.k1) atomicAdd(&tot, (unsigned long long)member_fix(sc));
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) fq_norm[b] = a.act_ids ? a.act_norm[b] : tot;
}

// a block per (query, coordinate): walk its entry
constexpr int kWalkBlocks = 4096;  // per query (then each takes every so many)
__global__ __launch_bounds__(128) void k_rerank_walk(const ReachArgs a, unsigned long long* __restrict__ num) {
  const int b = blockIdx.x, cnt = a.act_ids ? a.act_cnt[b] : a.k1;
  unsigned long long* row = num + (int64_t)b * a.N;
  for (int r = blockIdx.y; r < cnt; r += gridDim.y) {
    uint32_t fq;
    const int32_t i = reach_coord(a, b, r, fq);
    if (fq == 0) continue;
    const int64_t e1 = a.off[i + 1];
    for (int64_t e = a.off[i] + threadIdx.x; e < e1; e += blockDim.x) {
      const uint32_t m = a.mem[e];
      if (m) atomicAdd(row + a.ids[e], (unsigned long long)min(fq, m));
    }
  }
}

__global__ void k_rerank_keys(const unsigned long long* __restrict__ num,
                              const unsigned long long* __restrict__ fq_norm,
                              const unsigned long long* __restrict__ card, const float* __restrict__ Srow,
                              int32_t B, int32_t N, unsigned long long* __restrict__ keys) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)B * N) return;
  const int b = (int)(idx / N);
  const int p = (int)(idx % N);
  keys[idx] = reach_key(num[idx], fq_norm[b], card, p, Srow[idx]);
}

__global__ void k_keys_to_sprime(const unsigned long long* __restrict__ keys, int64_t n,
                                 float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = keys[i] == 0ull ? -INFINITY : key2f((uint32_t)(keys[i] >> 32));
}

__global__ void k_fill_f32(float* p, int64_t n, float v) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

// scratch: dense_bytes(B, N, topk), cleared and filled here, so nothing depends on what it held before
void dense_rerank(const ReachArgs& a, int32_t B, uint8_t* p, cudaStream_t s) {
  const int64_t BN = (int64_t)B * a.N;
  unsigned long long* num = reinterpret_cast<unsigned long long*>(p);
  p += align256((size_t)BN * 8);
  float* Srow = reinterpret_cast<float*>(p);
  p += align256((size_t)BN * 4);
  unsigned long long* fqn = reinterpret_cast<unsigned long long*>(p);
  p += align256((size_t)B * 8);
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(p);
  p += align256((size_t)BN * 8);
  unsigned long long* kout = reinterpret_cast<unsigned long long*>(p);
  GIFT_CUDA(cudaMemsetAsync(num, 0, BN * 8, s));
  k_fill_f32<<<(unsigned)cdiv(BN, 256), 256, 0, s>>>(Srow, BN, -INFINITY);
  GIFT_LAUNCHED("k_fill_f32");
  k_rerank_prep<<<(unsigned)B, 256, 0, s>>>(a, Srow, fqn);
  GIFT_LAUNCHED("k_rerank_prep");
  k_rerank_walk<<<dim3((unsigned)B, (unsigned)std::min(reach_coords(a), kWalkBlocks)), 128, 0, s>>>(a, num);
  GIFT_LAUNCHED("k_rerank_walk");
  k_rerank_keys<<<(unsigned)cdiv(BN, 256), 256, 0, s>>>(num, fqn, a.card, Srow, B, a.N, keys);
  GIFT_LAUNCHED("k_rerank_keys");
  topk_rows_u64(reinterpret_cast<const uint64_t*>(keys), B, a.N, a.topk, a.out_ids, reinterpret_cast<uint64_t*>(kout), s);
  k_keys_to_sprime<<<(unsigned)cdiv((int64_t)B * a.topk, 256), 256, 0, s>>>(kout, (int64_t)B * a.topk, a.out_sprime);
  GIFT_LAUNCHED("k_keys_to_sprime");
}

// ---------------------------------------------------------------- which of the two
constexpr int kHalf = 71680, kWhole = 188416;  // bytes of a table: two blocks share an SM, or one has it

// Re-rank of B queries whose activations have `coords` coordinates; w: what a walk from the inverted file's own shapes
// takes (their number of coordinates is w.coords). heavy: many entries per query whatever w says.
//
// Table and block: two blocks of 512 threads share an SM while a table takes at most kHalf (70 KB): all N up to 5,952
// shapes, or 4,480 hash slots, which the shapes a query reaches should leave a quarter empty. Heavier walks (of more
// than twice those slots of pairs) take a whole SM's table of up to 15,680 shapes, which spares them the probing.
//
// One block's walk takes 0.24 to 0.6 ns a pair by its threads, however many SMs stand idle; on dense rows a query's
// coordinates spread over the SMs, at a price in launches and in passes over all N shapes: they take over where the
// walks are long and the queries few (both sides in microseconds, from the figures below), and where a query reaches
// more shapes than a table holds, unless every SM has a query to walk. Measured, whole calls in us (one block, dense
// rows; neighbours drawn from all shapes unless said):
//   200,000 shapes, k1 =    50, 1 query     62   187        12,000 shapes, k1 = 1,000,     1 query     267    115
//   200,000, k1 = 200 in classes, 64        61   316        12,000, k1 = 1,000,           64           278    357
//   200,000, k1 = 1,000,          1      1,034   276        12,000, two measures, k2 = 40, 1         2,811    337
//   200,000, k1 = 1,000,        256      5,264 8,853        12,000, two measures, k2 = 40, 64        2,471  2,203
void rerank_queries(ReachArgs& a, int B, double coords, const WalkStats& w, bool heavy, Scratch& sc, cudaStream_t s) {
  const int sms = device_sm_count();
  const int64_t rows = reach_rows_bytes(a.N);
  const double pairs = a.n_cand + coords * w.met;
  const double reach = std::min<double>(a.N, a.n_cand + w.reach * std::max(1., coords / std::max(1., w.coords)));
  heavy = heavy || pairs > 2 * (kHalf / 16);
  int threads = 512;
  if (rows <= kHalf || (heavy && rows <= kWhole)) {
    a.hash = 0;
    a.table_bytes = (int)rows;
    threads = a.N <= 1024 ? 256 : rows <= kHalf ? 512 : 1024;
  } else {
    a.hash = 1;
    a.table_bytes = !heavy && reach * 16 * 4 / 3 <= kHalf ? kHalf : kWhole;
    threads = a.table_bytes == kHalf ? 512 : 1024;
  }
  bool dense = false;
  const bool over = a.hash && rows > a.table_bytes && reach * 16 * 4 / 3 > a.table_bytes;  // more than a table holds
  if (over) {
    a.hash = 0;
    dense = B < sms;
  } else {
    const double one = (double)cdiv(B, (int64_t)sms * (a.table_bytes <= kHalf ? 2 : 1)) *
                       (25 + (threads == 1024 ? 0.24e-3 : threads == 512 ? 0.29e-3 : 0.6e-3) * pairs);
    // (a pair's sum is in DRAM where the rows are larger than L2)
    const double pair = (double)B * a.N * 8 > 100e6 ? 24e-6 : 3.4e-6;
    dense = 50 + 0.75e-3 * a.N + B * (1e-5 * a.N + pair * pairs) < one;
  }
  if (dense) {
    uint8_t* p = nullptr;
    try {
      p = sc.get<uint8_t>(dense_bytes(B, a.N, a.topk));
    } catch (const Error&) {  // no memory for them: a block per query
    }
    if (p) {
      dense_rerank(a, B, p, s);
      return;
    }
  }
  // Rows for queries that no table holds, at most 2 GB of them at a time. Where entries are too short for a walk to
  // overflow a hash table by much, and the ranges that would follow are few, none are kept ready.
  a.num = nullptr;
  int per = B;
  const double most = a.n_cand + (double)reach_coords(a) * w.longest;
  const int slots = a.table_bytes / 16, range = a.table_bytes / 12;
  if (rows > a.table_bytes && (over || most > 8 * slots || (most > slots / 2 && a.N > 64 * range))) {
    per = (int)std::min<int64_t>(B, std::max<int64_t>(1, ((int64_t)2 << 30) / ((int64_t)a.N * 12)));
    try {
      a.num = sc.get<unsigned long long>((size_t)per * a.N + ((size_t)per * a.N + 1) / 2);
      a.S = reinterpret_cast<float*>(a.num + (size_t)per * a.N);
    } catch (const Error&) {  // no memory for them: ranges of shapes
      per = B;
    }
  }
  if (!a.num) {
    a.win_key = sc.get<unsigned long long>((size_t)B * a.topk);
    a.win_id = sc.get<uint32_t>((size_t)B * a.topk);
  }
  // the largest table, whatever this call takes: calls of several threads set the same value
  const auto kernel = a.num ? k_rerank_reach<true> : k_rerank_reach<false>;  // (without rows: less code to fetch)
  GIFT_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWhole));
  for (int b0 = 0; b0 < B; b0 += per) {
    kernel<<<(unsigned)std::min(per, B - b0), threads, a.table_bytes, s>>>(a);
    GIFT_LAUNCHED("k_rerank_reach");
    a.cand_ids += (int64_t)per * a.n_cand;
    a.cand_scores += (int64_t)per * a.n_cand;
    if (a.act_ids) {
      a.act_ids += (int64_t)per * a.act_ld;
      a.act_mem += (int64_t)per * a.act_ld;
      a.act_cnt += per;
      a.act_norm += per;
    }
    a.out_ids += (int64_t)per * a.topk;
    a.out_sprime += (int64_t)per * a.topk;
  }
}

// ---------------------------------------------------------------- two measures
constexpr int kAcaT = 256;
constexpr int kAcaMaxP = 4096;  // sorted pairs per shape (shared memory: 16 B each)

struct AcaRowArgs {
  int mode, k1, k2, cap, nmax, P;
  float alpha;
  int32_t N;
  const int32_t* db_ids[2];  // [N, k1] ranked neighbours of every database shape, per measure
  const float* db_sc[2];     // [N, k1] their scores
  const int32_t* nb[2];      // ranking of this row under measure l (row stride ld)
  const float* own_sc[2];    // scores aligned with nb (mode 0)
  int64_t ld;
  int32_t* out_ids;          // [rows, cap] ascending ids of the non-zero coordinates
  uint32_t* out_mem;         // [rows, cap] fixed-point activation
  int32_t* out_cnt;          // [rows]
  unsigned long long* out_norm;  // [rows] ||F||_1, fixed point
};

__device__ __forceinline__ float gen_mean(float a, float b, float alpha) {
  if (alpha == 0.5f) {
    const float r = 0.5f * (sqrtf(a) + sqrtf(b));
    return r * r;
  }
  if (alpha == 1.f) return 0.5f * (a + b);
  const float m = 0.5f * (powf(a, alpha) + powf(b, alpha));
  return m > 0.f ? powf(m, 1.f / alpha) : 0.f;
}

__global__ __launch_bounds__(kAcaT) void k_aca_rows(const AcaRowArgs a) {
  extern __shared__ __align__(16) uint8_t sm[];
  uint64_t* key = reinterpret_cast<uint64_t*>(sm);
  float* val = reinterpret_cast<float*>(key + a.P);
  int* pos = reinterpret_cast<int*>(val + a.P);
  __shared__ int part[kAcaT];
  __shared__ unsigned long long norm;
  const int64_t r = blockIdx.x;
  const int tid = threadIdx.x;
  if (tid == 0) norm = 0ull;
  // gather: measure l occupies [l * nmax, (l + 1) * nmax)
  for (int t = tid; t < a.P; t += kAcaT) {
    uint64_t k = ~0ull;
    float v = 0.f;
    if (t < 2 * a.nmax) {
      const int l = t / a.nmax, u = t % a.nmax;
      int32_t id = -1;
      if (a.mode == 0) {
        id = a.nb[l][r * a.ld + u];
        v = a.own_sc[l][r * a.ld + u];
      } else {
        const int src_l = a.mode == 1 ? l : 1 - l;
        const int32_t src = a.nb[src_l][r * a.ld + u / a.k1];
        if (src >= 0 && src < a.N) {
          id = a.db_ids[l][(int64_t)src * a.k1 + u % a.k1];
          v = a.db_sc[l][(int64_t)src * a.k1 + u % a.k1];
        }
      }
      if (id >= 0 && id < a.N) k = ((uint64_t)(uint32_t)id << 32) | ((uint64_t)l << 31) | (uint64_t)u;
    }
    key[t] = k;
    val[t] = v;
  }
  __syncthreads();
  // bitonic sort of (key, val), ascending
  for (int size = 2; size <= a.P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = tid; t < a.P; t += kAcaT) {
        const int o = t ^ stride;
        if (o > t) {
          const bool up = (t & size) == 0;
          const uint64_t x = key[t], y = key[o];
          if ((x > y) == up) {
            key[t] = y;
            key[o] = x;
            const float tv = val[t];
            val[t] = val[o];
            val[o] = tv;
          }
        }
      }
      __syncthreads();
    }
  }
  // heads of id groups, block-wide exclusive scan over each thread's consecutive chunk
  const int per = a.P / kAcaT;
  const int c0 = tid * per;
  int cnt = 0;
  for (int t = c0; t < c0 + per; ++t) {
    const uint64_t k = key[t];
    const bool head = k != ~0ull && (t == 0 || (key[t - 1] >> 32) != (k >> 32));
    pos[t] = head ? 1 : 0;
    cnt += head;
  }
  part[tid] = cnt;
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int i = 0; i < kAcaT; ++i) {
      const int c = part[i];
      part[i] = run;
      run += c;
    }
    a.out_cnt[r] = run;
  }
  __syncthreads();
  int o = part[tid];
  unsigned long long sum = 0ull;
  const float div = a.mode == 0 ? 1.f : (float)a.k2;
  for (int t = c0; t < c0 + per; ++t) {
    if (!pos[t]) continue;
    const uint64_t id = key[t] >> 32;
    float s0 = 0.f, s1 = 0.f;
    for (int e = t; e < a.P && key[e] != ~0ull && (key[e] >> 32) == id; ++e) {
      if ((key[e] >> 31) & 1ull) s1 += val[e];
      else s0 += val[e];
    }
    const uint32_t m = member_fix(gen_mean(s0 / div, s1 / div, a.alpha));
    a.out_ids[r * a.cap + o] = (int32_t)id;
    a.out_mem[r * a.cap + o] = m;
    sum += m;
    ++o;
  }
#pragma unroll
  for (int k = 16; k > 0; k >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, k);
  if ((tid & 31) == 0) atomicAdd(&norm, sum);  // (64-bit atomics in shared memory are loops: one per warp)
  __syncthreads();
  if (tid == 0) a.out_norm[r] = norm;
}

__global__ void k_aca_keys(const int32_t* __restrict__ ids, const int32_t* __restrict__ cnt, int32_t N, int cap,
                           int32_t* __restrict__ keys) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)N * cap) return;
  const int64_t p = e / cap;
  keys[e] = (e % cap) < cnt[p] ? ids[e] : N;
}

__global__ void k_aca_fill(const int32_t* __restrict__ perm, int64_t n, int cap, const uint32_t* __restrict__ mem_rows,
                           int32_t* __restrict__ ids, uint32_t* __restrict__ mem) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int32_t slot = perm[e];
  ids[e] = slot / cap;
  mem[e] = mem_rows[slot];
}

void launch_aca_rows(AcaRowArgs& a, int64_t rows, cudaStream_t s) {
  a.nmax = a.mode == 0 ? a.k1 : a.k2 * a.k1;
  int P = 2 * kAcaT;
  while (P < 2 * a.nmax) P <<= 1;
  GIFT_REQUIRE(P <= kAcaMaxP, "k2 * k1 (or k1 without augmentation) exceeds 2048");
  a.P = P;
  a.cap = 2 * a.nmax;
  const size_t smem = (size_t)P * 16;
  GIFT_CUDA(cudaFuncSetAttribute(k_aca_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  if (rows <= 0) return;
  k_aca_rows<<<(unsigned)rows, kAcaT, smem, s>>>(a);
  GIFT_LAUNCHED("k_aca_rows");
}

}  // namespace

template <class T>
T* Aca::alloc(size_t n) {
  void* p = nullptr;
  const size_t bytes = std::max<size_t>(n * sizeof(T), 16);
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    fail(GIFT_ENOMEM, "allocation of " + std::to_string(bytes) + " bytes failed");
  }
  owned.push_back(p);
  device_bytes += bytes;
  return static_cast<T*>(p);
}

Aca::~Aca() {
  for (void* p : owned) cudaFree(p);
}

void aca_build(Aca& a, Scratch& sc, cudaStream_t s) {
  const int32_t N = a.N;
  AcaRowArgs r{};
  r.mode = a.mode;
  r.k1 = a.k1;
  r.k2 = a.k2;
  r.alpha = a.alpha;
  r.N = N;
  for (int l = 0; l < 2; ++l) {
    r.db_ids[l] = a.m[l]->row_ids;
    r.db_sc[l] = a.m[l]->row_sc;
    r.nb[l] = a.m[l]->row_ids;  // a database shape's own ranking
    r.own_sc[l] = a.m[l]->row_sc;
  }
  r.ld = a.k1;
  r.nmax = a.mode == 0 ? a.k1 : a.k2 * a.k1;
  r.cap = 2 * r.nmax;
  const int64_t slots = (int64_t)N * r.cap;
  r.out_ids = sc.get<int32_t>(slots);
  r.out_mem = sc.get<uint32_t>(slots);
  r.out_cnt = sc.get<int32_t>(N);
  a.card = a.alloc<unsigned long long>(N);
  r.out_norm = a.card;
  launch_aca_rows(r, N, s);
  a.cap = r.cap;
  // transpose: entry i lists every p with a non-zero coordinate i, ascending p (stable sort by i)
  int32_t* keys = sc.get<int32_t>(slots);
  k_aca_keys<<<(unsigned)cdiv(slots, 256), 256, 0, s>>>(r.out_ids, r.out_cnt, N, r.cap, keys);
  GIFT_LAUNCHED("k_aca_keys");
  int32_t* perm = sc.get<int32_t>(slots);
  int32_t* skeys = sc.get<int32_t>(slots);
  stable_sort_by_key(keys, slots, N + 1, perm, skeys, sc, s);
  int64_t* off_all = sc.get<int64_t>((size_t)N + 2);
  bin_offsets(skeys, slots, N + 1, off_all, s);
  int64_t pairs = 0;
  GIFT_CUDA(cudaMemcpyAsync(&pairs, off_all + N, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  GIFT_CUDA(cudaStreamSynchronize(s));
  a.pairs = pairs;
  a.off = a.alloc<int64_t>((size_t)N + 1);
  GIFT_CUDA(cudaMemcpyAsync(a.off, off_all, ((size_t)N + 1) * 8, cudaMemcpyDeviceToDevice, s));
  a.ids = a.alloc<int32_t>((size_t)std::max<int64_t>(pairs, 1));
  a.mem = a.alloc<uint32_t>((size_t)std::max<int64_t>(pairs, 1));
  if (pairs > 0) {
    k_aca_fill<<<(unsigned)cdiv(pairs, 256), 256, 0, s>>>(perm, pairs, r.cap, r.out_mem, a.ids, a.mem);
    GIFT_LAUNCHED("k_aca_fill");
  }
  a.walks = walk_stats(r.out_ids, r.cap, r.out_cnt, N, a.off, a.ids, sc, s);
}

void aca_rerank(const Aca& a, const int32_t* cand1, const float* sc1, const int32_t* cand2, const float* sc2,
                int32_t B, int32_t n_cand, int32_t topk, int32_t* out_ids, float* out_sprime, Scratch& sc,
                cudaStream_t s) {
  const int32_t N = a.N;
  AcaRowArgs r{};
  r.mode = a.mode;
  r.k1 = a.k1;
  r.k2 = a.k2;
  r.alpha = a.alpha;
  r.N = N;
  for (int l = 0; l < 2; ++l) {
    r.db_ids[l] = a.m[l]->row_ids;
    r.db_sc[l] = a.m[l]->row_sc;
  }
  r.nb[0] = cand1;
  r.nb[1] = cand2;
  r.own_sc[0] = sc1;
  r.own_sc[1] = sc2;
  r.ld = n_cand;
  r.nmax = a.mode == 0 ? a.k1 : a.k2 * a.k1;
  r.cap = 2 * r.nmax;
  r.out_ids = sc.get<int32_t>((size_t)B * r.cap);
  r.out_mem = sc.get<uint32_t>((size_t)B * r.cap);
  r.out_cnt = sc.get<int32_t>(B);
  r.out_norm = sc.get<unsigned long long>(B);
  launch_aca_rows(r, B, s);
  ReachArgs g{};
  g.N = N;
  g.cand_ids = cand1;
  g.cand_scores = sc1;  // S^(1) breaks ties
  g.n_cand = n_cand;
  g.k1 = a.k1;
  g.act_ids = r.out_ids;
  g.act_mem = r.out_mem;
  g.act_cnt = r.out_cnt;
  g.act_norm = r.out_norm;
  g.act_ld = r.cap;
  g.off = a.off;
  g.ids = a.ids;
  g.mem = a.mem;
  g.card = a.card;
  g.topk = topk;
  g.out_ids = out_ids;
  g.out_sprime = out_sprime;
  rerank_queries(g, B, (double)a.pairs / N, a.walks, true, sc, s);
}

void sif_build(Index& ix, const int32_t* nbr_ids, const float* nbr_scores, Scratch& sc, cudaStream_t s) {
  const int32_t N = ix.sif_n;
  const int k1 = ix.k1;
  const int64_t n = (int64_t)N * k1;
  int32_t* keys = sc.get<int32_t>(n);
  int* bad = sc.get<int>(1);
  GIFT_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), s));
  k_sif_keys<<<(unsigned)cdiv(n, 256), 256, 0, s>>>(nbr_ids, n, N, keys, bad);
  GIFT_LAUNCHED("k_sif_keys");
  int32_t* perm = sc.get<int32_t>(n);
  int32_t* skeys = sc.get<int32_t>(n);
  stable_sort_by_key(keys, n, N, perm, skeys, sc, s);
  bin_offsets(skeys, n, N, ix.sif_off, s);
  k_sif_fill<<<(unsigned)cdiv(n, 256), 256, 0, s>>>(perm, n, k1, nbr_scores, ix.sif_ids, ix.sif_mem);
  GIFT_LAUNCHED("k_sif_fill");
  k_sif_card<<<(unsigned)cdiv(N, 256), 256, 0, s>>>(nbr_scores, N, k1,
                                                      reinterpret_cast<unsigned long long*>(ix.sif_card));
  GIFT_LAUNCHED("k_sif_card");
  int h_bad = 0;
  GIFT_CUDA(cudaMemcpyAsync(&h_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  const WalkStats w = walk_stats(nbr_ids, k1, nullptr, N, ix.sif_off, ix.sif_ids, sc, s);
  if (h_bad) fail(GIFT_EINVAL, "S-IF build: a database shape has fewer than k1 neighbours");
  ix.sif_walks = w;
}

namespace {

ReachArgs sif_args(const Index& ix, const int32_t* cand_ids, const float* cand_scores, int32_t n_cand, int32_t k1,
                   int32_t topk, int32_t* out_ids, float* out_sprime) {
  ReachArgs g{};
  g.N = ix.sif_n;
  g.cand_ids = cand_ids;
  g.cand_scores = cand_scores;
  g.n_cand = n_cand;
  g.k1 = k1;
  g.off = ix.sif_off;
  g.ids = ix.sif_ids;
  g.mem = ix.sif_mem;
  g.card = reinterpret_cast<const unsigned long long*>(ix.sif_card);
  g.topk = topk;
  g.out_ids = out_ids;
  g.out_sprime = out_sprime;
  return g;
}

}  // namespace

void sif_rerank(const Index& ix, const int32_t* cand_ids, const float* cand_scores, int32_t B, int32_t n_cand,
                int32_t k1, int32_t topk, int32_t* out_ids, float* out_sprime, Scratch& sc, cudaStream_t s) {
  ReachArgs g = sif_args(ix, cand_ids, cand_scores, n_cand, k1, topk, out_ids, out_sprime);
  rerank_queries(g, B, k1, ix.sif_walks, false, sc, s);
}

size_t sif_rerank_scratch_bytes(int32_t B, int32_t N, int32_t topk) { return dense_bytes(B, N, topk); }

// The re-rank on scratch the caller provides (no allocation): the dense rows, whatever the walks are
void sif_rerank_into(const Index& ix, const int32_t* cand_ids, const float* cand_scores, int32_t B, int32_t n_cand,
                     int32_t k1, int32_t topk, int32_t* out_ids, float* out_sprime, void* scratch,
                     size_t scratch_bytes, cudaStream_t s) {
  GIFT_REQUIRE(dense_bytes(B, ix.sif_n, topk) <= scratch_bytes, "re-rank scratch too small");
  dense_rerank(sif_args(ix, cand_ids, cand_scores, n_cand, k1, topk, out_ids, out_sprime), B,
               static_cast<uint8_t*>(scratch), s);
}

}  // namespace gift
