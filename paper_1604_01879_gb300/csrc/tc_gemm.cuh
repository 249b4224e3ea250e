// Plain GEMM on the tcgen05 engine: C[M, N] (+)= A[M, K] * B[N, K]^T with
// A, B K-major BF16 (SPLIT = 1), two-part BF16 (SPLIT = 3: hi*hi + hi*lo +
// lo*hi, FP32-level), or a two-part A with a B exact in BF16 (SPLIT = 2:
// hi*b + lo*b), FP32 output. The reduction runs in chunks of at most 16
// k-blocks, each accumulated in its own TMEM buffer and summed in FP32 by the
// epilogue (bounds the steps that feed one tensor-core accumulator).
// Work items run along the longer side: with more row tiles than column
// tiles they run row-tile-major, so the CTAs working at the same time share
// each A tile (read from memory once) and all of B; otherwise column-tile-
// major, sharing the B tile.
#pragma once
#include "tc_pair.cuh"

namespace gift {

template <int SPLIT_>
struct GemmPolicy {
  static constexpr int TN = 128, NBUF = 4, STAGES = SPLIT_ == 1 ? 6 : SPLIT_ == 2 ? 4 : 3, SPLIT = SPLIT_, EB = 2;
  static constexpr bool REPORT = true;
  static constexpr int kTurn = 20;  // row pitch of a turned piece: 16-byte rows, bank groups apart
  static constexpr int kWarpSmem = 32 * kTurn * 4;
  int64_t M, N;
  int nkb;
  float* C;
  int64_t ldc;
  int accumulate;
  bool row_major;  // item order: row tile slow (true) or column tile slow
  // parts > 1: the reduction is cut in so many parts, items of a part together, each with its own result at
  // C + part * pstride (added up in part order by k_add_parts)
  int parts = 1;
  int64_t pstride = 0;
  struct Item {
    int64_t r0, c0;
    int nr, nc;
    int part;
  };
  struct Ctx {
    float sum[TN];
  };
  __device__ __forceinline__ int64_t n_mt() const { return cdiv(M, tc::kTM); }
  __device__ __forceinline__ int64_t total() const { return n_mt() * cdiv(N, TN) * parts; }
  __device__ __forceinline__ Item decode(int64_t item) const {
    Item it;
    const int64_t mt = n_mt(), nt = cdiv(N, TN);
    it.part = (int)(item / (mt * nt));
    item -= it.part * (mt * nt);
    const int64_t ct = row_major ? item % nt : item / mt, rt = row_major ? item / nt : item % mt;
    it.r0 = rt * tc::kTM;
    it.c0 = ct * TN;
    it.nr = (int)min((int64_t)tc::kTM, M - it.r0);
    it.nc = (int)min((int64_t)TN, N - it.c0);
    return it;
  }
  // chunks bound the MMA steps feeding one accumulator (about 192, 3 products
  // x 4 sub-steps per k-block), however long the reduction (the weight
  // gradient reduces over every database view); short reductions use one chunk
  __device__ __forceinline__ int part_kb(int part) const { return (int)((int64_t)nkb * part / parts); }
  __device__ __forceinline__ int nchunks(const Item& it) const {
    const int want = ((part_kb(it.part + 1) - part_kb(it.part)) * 12 + 191) / 192;
    return want < 1 ? 1 : want;
  }
  __device__ __forceinline__ void chunk(const Item& it, int c, int& br, int& kb0, int& kb1) const {
    const int n = nchunks(it), p0 = part_kb(it.part), len = part_kb(it.part + 1) - p0;
    br = (int)it.c0;
    kb0 = p0 + (int)((int64_t)len * c / n);
    kb1 = p0 + (int)((int64_t)len * (c + 1) / n);
  }
  __device__ __forceinline__ int a_row(const Item& it) const { return (int)it.r0; }
  // pair form: 256 x 256 tiles in the same order, a CTA's epilogue part takes 128 x 128 of them
  static constexpr int TN_PAIR = 256;
  __device__ __forceinline__ int64_t total_pair() const {
    return cdiv(M, (int64_t)256) * cdiv(N, (int64_t)256) * parts;
  }
  __device__ __forceinline__ Item decode_pair(int64_t item) const {
    const int64_t mt = cdiv(M, (int64_t)256), nt = cdiv(N, (int64_t)256);
    const int part = (int)(item / (mt * nt));
    item -= part * (mt * nt);
    const int64_t ct = row_major ? item % nt : item / mt, rt = row_major ? item / nt : item % mt;
    return Item{rt * 256, ct * 256, (int)min((int64_t)256, M - rt * 256), (int)min((int64_t)256, N - ct * 256), part};
  }
  __device__ __forceinline__ Item sub(const Item& w, int rank, int part) const {
    return Item{w.r0 + 128 * rank, w.c0 + 128 * part, min(128, max(0, w.nr - 128 * rank)),
                min(128, max(0, w.nc - 128 * part)), w.part};
  }
  __device__ __forceinline__ void epi_begin(const Item&, Ctx& x, int, int, uint8_t*) const {
#pragma unroll
    for (int j = 0; j < TN; ++j) x.sum[j] = 0.f;
  }
  __device__ __forceinline__ void epi_chunk(const Item&, int, uint32_t taddr, Ctx& x, int, uint8_t*) const {
#pragma unroll
    for (int pc = 0; pc < TN / 32; ++pc) {
      uint32_t r[32];
      tc::tmem_ld32(taddr + pc * 32, r);
      tc::tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 32; ++j) x.sum[pc * 32 + j] += __uint_as_float(r[j]);
    }
  }
  // A thread holds a row, so storing straight from its registers touches 32 rows per instruction and half of each
  // 32-byte sector. The warp turns 32 x 16 pieces in shared memory and stores eight whole 64-byte row pieces per
  // instruction instead (262,144 x 4,096, K = 512, two products, 4.3 GB of results: 2.2 ms before, 1.45 now).
  __device__ __forceinline__ void epi_end(const Item& it, Ctx& x, int m, uint8_t* ws) const {
    float* t = reinterpret_cast<float*>(ws);  // [32][kTurn]
    const int lane = threadIdx.x & 31, m0 = m - lane;
    float* out = C + it.part * pstride;
    const bool vec = (ldc % 4) == 0 && ((it.c0 % 4) == 0) && (reinterpret_cast<uintptr_t>(out) % 16) == 0;
#pragma unroll
    for (int pc = 0; pc < TN / 16; ++pc) {
      if (pc * 16 >= it.nc) break;  // warp-uniform
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 16; j += 4)
        *reinterpret_cast<float4*>(t + lane * kTurn + j) =
            make_float4(x.sum[pc * 16 + j], x.sum[pc * 16 + j + 1], x.sum[pc * 16 + j + 2], x.sum[pc * 16 + j + 3]);
      __syncwarp();
      const int q = (lane & 3) * 4, c = pc * 16 + q;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = i * 8 + (lane >> 2);
        if (m0 + r >= it.nr || c >= it.nc) continue;
        float4 v = *reinterpret_cast<const float4*>(t + r * kTurn + q);
        float* dst = out + (it.r0 + m0 + r) * ldc + it.c0 + c;
        if (vec && c + 4 <= it.nc) {
          if (accumulate) {
            const float4 o = *reinterpret_cast<const float4*>(dst);
            v.x += o.x;
            v.y += o.y;
            v.z += o.z;
            v.w += o.w;
          }
          *reinterpret_cast<float4*>(dst) = v;
        } else {
          const float e[4] = {v.x, v.y, v.z, v.w};
          for (int k = 0; k < 4 && c + k < it.nc; ++k) dst[k] = accumulate ? dst[k] + e[k] : e[k];
        }
      }
    }
  }
};

// Two-part (SPLIT 3), two-part A with one-part B (SPLIT 2, b_lo null) or
// one-part (SPLIT 1, both lo parts null) BF16 operands; a_rows_alloc /
// b_rows_alloc are the rows the tensor maps cover (rows past M or N read as
// zeros); lda / ldb are row pitches in elements (0 = K): C[M, N] (+)= A * B^T. With `split` the
// reduction may be cut in parts where the tiles alone would leave SMs idle (another order of sums).
void gemm_tc(const __nv_bfloat16* a_hi, const __nv_bfloat16* a_lo, int64_t M, int64_t a_rows_alloc, int64_t lda,
             const __nv_bfloat16* b_hi, const __nv_bfloat16* b_lo, int64_t N, int64_t b_rows_alloc, int64_t ldb, int K,
             float* C, int64_t ldc, int accumulate, int* err, cudaStream_t s, Scratch* split = nullptr);

}  // namespace gift
