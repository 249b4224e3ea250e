// Top-k selections: one block per row (select.cuh), ordered by (value desc, index or id asc).
//
// Values become order-preserving unsigned keys (larger value -> larger key). Rows that are sorted
// outright (up to 2,048 pairs) take one thread per pair of the sort. Longer ones take as many threads as
// keep the chip full (about 64 registers each): 256 where there are rows for four blocks on every SM (their
// barriers cost least), 512 where some SMs get a second row, 1,024 where a row has an SM to itself and its loads
// are what the narrowing passes wait for.
#include "gift_internal.cuh"
#include "select.cuh"

namespace gift {

namespace {

constexpr int kMaxK = 1024;

// threads for each of B rows of n pairs: a power of two in [64, 1024]
int row_threads(int64_t n, int B) {
  const int sms = device_sm_count();
  const int most = n <= sel::kCap ? 1024 : B >= 4 * sms ? 256 : B > sms ? 512 : 1024;
  int t = 64;
  while (t < most && 2 * (int64_t)t < n) t <<= 1;
  return t;
}

struct ScoreRow {
  static constexpr int kAhead = 8;
  static __device__ __forceinline__ uint32_t score(unsigned long long key) { return (uint32_t)key; }
  const float* s;
  __device__ __forceinline__ bool operator()(int64_t i, unsigned long long& key, uint32_t& id) const {
    key = f2key(s[i]);
    id = (uint32_t)i;
    return true;
  }
};

__global__ __launch_bounds__(1024) void k_topk(const float* __restrict__ scores, int64_t n, int k,
                                               int32_t* __restrict__ ids_out, float* __restrict__ val_out, int* err) {
  dep_begin();
  __shared__ sel::Smem sm;
  const int64_t b = blockIdx.x;
  if (b == 0 && threadIdx.x == 0) report_wait(err);
  const int take = sel::select(sm, ScoreRow{scores + b * n}, n, n, k);
  for (int t = threadIdx.x; t < k; t += blockDim.x) {
    const bool ok = t < take;
    ids_out[b * k + t] = ok ? (int32_t)sm.id[t] : -1;
    if (val_out) val_out[b * k + t] = ok ? key2f((uint32_t)sm.key[t]) : -INFINITY;
  }
}

struct KeyRow {
  static constexpr int kAhead = 4;
  static __device__ __forceinline__ uint32_t score(unsigned long long key) { return (uint32_t)(key >> 32); }
  const unsigned long long* s;
  __device__ __forceinline__ bool operator()(int64_t i, unsigned long long& key, uint32_t& id) const {
    key = s[i];
    id = (uint32_t)i;
    return true;
  }
};

__global__ __launch_bounds__(1024) void k_topk_keys(const unsigned long long* __restrict__ keys, int64_t n, int k,
                                                    int32_t* __restrict__ ids_out,
                                                    unsigned long long* __restrict__ key_out) {
  __shared__ sel::Smem sm;
  const int64_t b = blockIdx.x;
  const int take = sel::select(sm, KeyRow{keys + b * n}, n, n, k);
  for (int t = threadIdx.x; t < k; t += blockDim.x) {
    const bool ok = t < take;
    ids_out[b * k + t] = ok ? (int32_t)sm.id[t] : -1;
    key_out[b * k + t] = ok ? sm.key[t] : 0ull;
  }
}

// (id, score) pairs of a merged row; id < 0 marks an empty one
struct PairRow {
  static constexpr int kAhead = 8;
  static __device__ __forceinline__ uint32_t score(unsigned long long key) { return (uint32_t)key; }
  const int32_t* ids;
  const float* s;
  __device__ __forceinline__ bool operator()(int64_t i, unsigned long long& key, uint32_t& id) const {
    const int32_t v = ids[i];
    key = f2key(s[i]);
    id = (uint32_t)v;
    return v >= 0;
  }
};

__global__ __launch_bounds__(1024) void k_merge_rows(const int32_t* __restrict__ ids, const float* __restrict__ scores,
                                                     int64_t n, int k, int32_t* __restrict__ ids_out,
                                                     float* __restrict__ val_out) {
  __shared__ sel::Smem sm;
  __shared__ int s_valid;
  const int64_t b = blockIdx.x;
  const PairRow row{ids + b * n, scores + b * n};
  if (threadIdx.x == 0) s_valid = 0;
  __syncthreads();
  int own = 0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) own += row.ids[i] >= 0 ? 1 : 0;
  if (own) atomicAdd(&s_valid, own);
  __syncthreads();
  const int take = sel::select(sm, row, n, s_valid, k);
  for (int t = threadIdx.x; t < k; t += blockDim.x) {
    const bool ok = t < take;
    ids_out[b * k + t] = ok ? (int32_t)sm.id[t] : -1;
    val_out[b * k + t] = ok ? key2f((uint32_t)sm.key[t]) : -INFINITY;
  }
}

// rows of (id, score): sort by (score desc, id asc) and keep k; mode_ids: by id asc, invalid ids last
__global__ __launch_bounds__(1024) void k_sort_candidates(const int32_t* __restrict__ ids,
                                                          const float* __restrict__ scores, int r, int k,
                                                          int32_t* __restrict__ ids_out,
                                                          float* __restrict__ scores_out, int mode_ids, int* err) {
  dep_begin();
  if (blockIdx.x == 0 && threadIdx.x == 0) report_wait(err);
  __shared__ unsigned long long s_key[kMaxK];
  __shared__ uint32_t s_id[kMaxK];
  const int64_t b = blockIdx.x;
  int P = 64;
  while (P < r) P <<= 1;
  for (int t = threadIdx.x; t < P; t += blockDim.x) {
    int32_t id = t < r ? ids[b * r + t] : -1;
    if (id < 0) id = 0x7fffffff;
    s_id[t] = (uint32_t)id;
    s_key[t] = id == 0x7fffffff ? 0ull : mode_ids ? 1ull : (unsigned long long)f2key(scores[b * r + t]);
  }
  sel::sort_pairs(s_key, s_id, P);
  for (int t = threadIdx.x; t < k; t += blockDim.x) {
    const int64_t o = b * k + t;
    const bool ok = t < r && s_id[t] != 0x7fffffffu;
    ids_out[o] = ok ? (int32_t)s_id[t] : -1;
    if (scores_out) scores_out[o] = ok ? key2f((uint32_t)s_key[t]) : -INFINITY;
  }
}

}  // namespace

void merge_topk_rows(const int32_t* ids, const float* scores, int32_t B, int64_t n, int32_t k, int32_t* ids_out,
                     float* scores_out, cudaStream_t s) {
  if (B <= 0 || k <= 0) return;
  GIFT_REQUIRE(k <= kMaxK, "top-k is limited to 1024");
  GIFT_REQUIRE(n < (int64_t)INT32_MAX, "row too long for top-k");
  k_merge_rows<<<(unsigned)B, row_threads(n, B), 0, s>>>(ids, scores, n, k, ids_out, scores_out);
  GIFT_LAUNCHED("k_merge_rows");
}

void topk_rows_f32(const float* scores, int32_t B, int64_t n, int32_t k, int32_t* ids_out, float* val_out,
                   cudaStream_t s, int* err) {
  if (B <= 0 || k <= 0) return;
  GIFT_REQUIRE(k <= kMaxK, "top-k is limited to 1024");
  GIFT_REQUIRE(n < (int64_t)INT32_MAX, "row too long for top-k");
  launch_dep(k_topk, dim3((unsigned)B), dim3(row_threads(n, B)), 0, s, scores, n, k, ids_out, val_out, err);
  GIFT_LAUNCHED("k_topk");
}

void topk_rows_u64(const uint64_t* keys, int32_t B, int64_t n, int32_t k, int32_t* ids_out,
                   uint64_t* key_out, cudaStream_t s) {
  if (B <= 0 || k <= 0) return;
  GIFT_REQUIRE(k <= kMaxK, "top-k is limited to 1024");
  GIFT_REQUIRE(n < (int64_t)INT32_MAX, "row too long for top-k");
  k_topk_keys<<<(unsigned)B, row_threads(n, B), 0, s>>>(reinterpret_cast<const unsigned long long*>(keys), n, k, ids_out,
                                                     reinterpret_cast<unsigned long long*>(key_out));
  GIFT_LAUNCHED("k_topk_keys");
}

void sort_candidates(const int32_t* ids, const float* scores, int32_t B, int32_t r, int32_t k,
                     int32_t* ids_out, float* scores_out, cudaStream_t s, int* err) {
  if (B <= 0 || k <= 0) return;
  GIFT_REQUIRE(r <= kMaxK, "candidate rows are limited to 1024");
  launch_dep(k_sort_candidates, dim3((unsigned)B), dim3(row_threads(r, B)), 0, s, ids, scores, r, k, ids_out,
             scores_out, 0, err);
  GIFT_LAUNCHED("k_sort_candidates");
}

void sort_ids_rows(const int32_t* ids, int32_t B, int32_t r, int32_t* out, cudaStream_t s) {
  if (B <= 0 || r <= 0) return;
  GIFT_REQUIRE(r <= kMaxK, "candidate rows are limited to 1024");
  launch_dep(k_sort_candidates, dim3((unsigned)B), dim3(row_threads(r, B)), 0, s, ids, nullptr, r, r, out, nullptr, 1,
             nullptr);
  GIFT_LAUNCHED("k_sort_ids");
}

}  // namespace gift
