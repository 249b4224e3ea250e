// Host side of the engine GEMM (instantiations of GemmPolicy).
#include "tc_gemm.cuh"

namespace gift {

namespace {

// C (+)= the sum of the parts' results, in part order; n4 float4s per row of N
__global__ void k_add_parts(const float* __restrict__ part, int parts, int64_t pstride, int64_t M, int64_t N,
                            float* __restrict__ C, int64_t ldc, int accumulate) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M * N) return;
  float v = part[i];
  for (int p = 1; p < parts; ++p) v += part[p * pstride + i];
  float* dst = C + i / N * ldc + i % N;
  *dst = accumulate ? *dst + v : v;
}

// Parts of the reduction for `items` tiles on `units` SMs or pairs: the fewest rounds of k-blocks, an item costing
// about six k-blocks of its own (fill and drain), each part's result a write and a read more (in k-blocks of half a
// microsecond at 4 TB/s) and their sum a launch. 512 x 4,096 with K = 262,144: 32 pair tiles for 76 pairs in seven
// parts, 1.88 ms (one SM per tile, 128 tiles) -> 1.24; seven GEMMs of a 24-query step, whose weight gradient was four tiles:
// 132 us -> 74.
int split_parts(int64_t items, int units, int nkb, int64_t results, double& cost) {
  int best = 1;
  cost = (double)cdiv(items, (int64_t)units) * (nkb + 6);
  for (int p = 2; p <= 32 && nkb / p >= 4; ++p) {
    const double c = (double)cdiv(items * p, (int64_t)units) * ((double)nkb / p + 6) + 6 + p * results * 8 / 2.0e6;
    if (c < 0.95 * cost) {
      cost = c;
      best = p;
    }
  }
  return best;
}

template <int SPLIT>
void run_gemm(const CUtensorMap& tA, const CUtensorMap& tB, const CUtensorMap& tA2, const CUtensorMap& tB2, int64_t M,
              int64_t N, int K, float* C, int64_t ldc, int accumulate, int* err, cudaStream_t s, Scratch* split) {
  GemmPolicy<SPLIT> p;
  p.M = M;
  p.N = N;
  p.nkb = (int)cdiv(K, tc::kTK);
  p.C = C;
  p.ldc = ldc;
  p.accumulate = accumulate;
  p.row_major = cdiv(M, tc::kTM) >= cdiv(N, 128);
  const int sms = device_sm_count(), pairs = tc::pair_clusters<GemmPolicy<SPLIT>>();
  const int64_t items = cdiv(M, tc::kTM) * cdiv(N, 128), pair_items = cdiv(M, 256) * cdiv(N, 256);
  bool pair = tc::pair_wins(items, pair_items, sms, pairs);
  if (split) {
    double t1 = 0, t2 = 0;
    const int p1 = split_parts(items, sms, p.nkb, M * N, t1), p2 = split_parts(pair_items, pairs, p.nkb, M * N, t2);
    pair = 1.4 * t2 < t1;
    p.parts = pair ? p2 : p1;
  }
  if (p.parts > 1) {
    p.C = split->get<float>((size_t)p.parts * M * N);
    p.ldc = N;
    p.pstride = M * N;
    p.accumulate = 0;
  }
  if (pair)
    tc::launch_pair(tA, tB, tA2, tB2, p, err, pair_items * p.parts, s);
  else
    tc::launch_engine(tA, tB, tA2, tB2, p, err, (int)std::min<int64_t>(sms, items * p.parts), s);
  if (p.parts > 1) {
    k_add_parts<<<(unsigned)cdiv(M * N, 256), 256, 0, s>>>(p.C, p.parts, p.pstride, M, N, C, ldc, accumulate);
    GIFT_LAUNCHED("k_add_parts");
  }
}

}  // namespace

void gemm_tc(const __nv_bfloat16* a_hi, const __nv_bfloat16* a_lo, int64_t M, int64_t a_rows_alloc, int64_t lda,
             const __nv_bfloat16* b_hi, const __nv_bfloat16* b_lo, int64_t N, int64_t b_rows_alloc, int64_t ldb, int K,
             float* C, int64_t ldc, int accumulate, int* err, cudaStream_t s, Scratch* split) {
  if (M <= 0 || N <= 0) return;
  GIFT_REQUIRE(a_lo != nullptr || b_lo == nullptr, "gemm_tc: a two-part B needs a two-part A");
  const CUtensorMap tA = make_tmap_bf16(a_hi, a_rows_alloc, K, tc::kTM, lda);
  const CUtensorMap tB = make_tmap_bf16(b_hi, b_rows_alloc, K, 128, ldb);
  if (a_lo && b_lo) {
    const CUtensorMap tA2 = make_tmap_bf16(a_lo, a_rows_alloc, K, tc::kTM, lda);
    const CUtensorMap tB2 = make_tmap_bf16(b_lo, b_rows_alloc, K, 128, ldb);
    run_gemm<3>(tA, tB, tA2, tB2, M, N, K, C, ldc, accumulate, err, s, split);
  } else if (a_lo) {
    const CUtensorMap tA2 = make_tmap_bf16(a_lo, a_rows_alloc, K, tc::kTM, lda);
    run_gemm<2>(tA, tB, tA2, tB, M, N, K, C, ldc, accumulate, err, s, split);
  } else {
    run_gemm<1>(tA, tB, tA, tB, M, N, K, C, ldc, accumulate, err, s, split);
  }
}

}  // namespace gift
