// Quantiser c(x) = argmin_k ||x - b_k||^2 with multiple assignment (Sec. 2.3).
//
// Coarse stage (tensor cores): score_k = x.b_k - ||b_k||^2 / 2 (argmax of the
// score is argmin of the distance) from two-part BF16 operands (x = hi + lo,
// three products, FP32 accumulate). A work item is 128 rows x one chunk of 256
// codewords; the chunks of one row tile are consecutive items, so the CTAs
// that run them at the same time share the row tile through L2. The epilogue
// keeps each row's 16 best coarse scores of its chunk.
// Refine stage (CUDA cores, one warp per row): every codeword whose coarse
// score lies within 2E of the ma-th best over all chunks is a candidate, where
// E bounds the coarse error:
//   E = 2^-12 (||x|| max_k ||b_k|| + max_k ||b_k||^2 / 2),
// about five times the representation bound of the split (3 * 2^-16 relative
// per product) plus the measured accumulation error. When a chunk's 16th kept
// score is still a candidate, that chunk may hold more, and the row takes the
// exact pass over every codeword. A single candidate with ma = 1 is the code
// without further work; otherwise the candidates' squared distances are
// evaluated in FP32, which decides when the gaps exceed twice its error bound, and
// else in two-float (~2^-44 relative) arithmetic; the ma smallest by
// (distance, index) are the codes. Results equal an exact evaluation except
// where distances tie to ~1e-13.
#include "gift_internal.cuh"
#include "tc_pair.cuh"

namespace gift {

namespace {

constexpr unsigned kFull = 0xffffffffu;
// coarse scores kept per row and chunk of tn codewords: the best 16, or all 32 (which spares the epilogue its
// insertions, most of a small item's time)
__host__ __device__ constexpr int kept_scores(int tn) { return tn == 32 ? 32 : 16; }
constexpr int kMaxParts = 8;   // parts of the reduction
constexpr int kPartsK = 1024;  // codewords of a vocabulary whose reduction is taken in parts

// TN_: codewords per chunk. 256 where the (row tile, chunk) items fill the SMs; with few rows 64 or 32, whose more
// items run on more SMs at once with more stages in flight: an item's time is a chain of D / 64 k-blocks, 1.7 us each
// with two stages of 96 KB, 0.6 us with five of 40 KB (108 rows, D = 4096, K = 512: 110 us against 44, and the refine
// 52 against 20 with a block per row).
template <int TN_>
struct AssignPolicy {
  static constexpr int TN = TN_, NBUF = 2, SPLIT = 3, EB = 2;
  static constexpr int STAGES = TN_ == 256 ? 2 : TN_ == 128 ? 3 : TN_ == 64 ? 4 : 5;
  static constexpr int kT = kept_scores(TN_);
  static constexpr bool kAll = kT == TN_;
  static constexpr int kWarpSmem = TN * 4;
  int64_t n;          // rows
  int K;
  int nch;            // codeword chunks of TN
  int nkb;
  int parts = 1;      // parts of the reduction, each an item of its own (kAll only)
  const float* half_sq;
  float* cval;        // [n, nch, kT] best coarse scores of each chunk, descending; parts > 1: [parts, n, nch, kT] products
  int32_t* cidx;      // [n, nch, kT] their codewords (0x7fffffff: none)
  struct Item {
    int64_t r0;
    int nr;
    int c;
    int part;
  };
  struct Ctx {
    float val[kT];
    int idx[kT];
  };
  __device__ __forceinline__ int64_t total() const { return cdiv(n, tc::kTM) * nch * (kAll ? parts : 1); }
  __device__ __forceinline__ Item decode(int64_t item) const {
    Item it;
    it.part = 0;
    if constexpr (kAll) {
      it.part = (int)(item % parts);
      item /= parts;
    }
    it.r0 = (item / nch) * tc::kTM;
    it.c = (int)(item % nch);
    it.nr = (int)min((int64_t)tc::kTM, n - it.r0);
    return it;
  }
  __device__ __forceinline__ int nchunks(const Item&) const { return 1; }
  __device__ __forceinline__ void chunk(const Item& it, int, int& br, int& kb0, int& kb1) const {
    br = it.c * TN;
    kb0 = kAll ? nkb * it.part / parts : 0;
    kb1 = kAll ? nkb * (it.part + 1) / parts : nkb;
  }
  __device__ __forceinline__ int a_row(const Item& it) const { return (int)it.r0; }
  __device__ __forceinline__ void epi_begin(const Item&, Ctx& x, int, int, uint8_t*) const {
#pragma unroll
    for (int t = 0; t < kT; ++t) {
      x.val[t] = -INFINITY;
      x.idx[t] = 0x7fffffff;
    }
  }
  __device__ __forceinline__ void epi_chunk(const Item& it, int, uint32_t taddr, Ctx& x, int, uint8_t* ws) const {
    float* hs = reinterpret_cast<float*>(ws);
    const int lane = threadIdx.x & 31;
    const int c = it.c;
    for (int j = lane; j < TN; j += 32) {
      const int k = c * TN + j;
      hs[j] = k < K ? half_sq[k] : INFINITY;
    }
    __syncwarp();
    if constexpr (kAll) {
      uint32_t r[32];
      tc::tmem_ld32(taddr, r);
      tc::tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        x.val[j] = __uint_as_float(r[j]) - (parts > 1 ? 0.f : hs[j]);
        x.idx[j] = c * TN + j < K ? c * TN + j : 0x7fffffff;
      }
      __syncwarp();
      return;
    }
    const int npieces = min(TN, K - c * TN + 31) >> 5;
    for (int pc = 0; pc < npieces; ++pc) {
      uint32_t r[32];
      tc::tmem_ld32(taddr + pc * 32, r);
      tc::tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const float s = __uint_as_float(r[j]) - hs[pc * 32 + j];
        if (s > x.val[kT - 1]) {  // strict: an equal later index never displaces an earlier one
          x.val[kT - 1] = s;
          x.idx[kT - 1] = c * TN + pc * 32 + j;
#pragma unroll
          for (int t = kT - 1; t > 0; --t) {
            if (x.val[t] > x.val[t - 1]) {
              const float tv = x.val[t];
              x.val[t] = x.val[t - 1];
              x.val[t - 1] = tv;
              const int ti = x.idx[t];
              x.idx[t] = x.idx[t - 1];
              x.idx[t - 1] = ti;
            }
          }
        }
      }
    }
    __syncwarp();
  }
  __device__ __forceinline__ void epi_end(const Item& it, Ctx& x, int m, uint8_t*) const {
    if (m >= it.nr) return;
    const int64_t o = (((kAll ? it.part * n : 0) + it.r0 + m) * nch + it.c) * kT;
    if constexpr (kAll) {
#pragma unroll
      for (int t = 0; t < kT; t += 4) {
        *reinterpret_cast<float4*>(cval + o + t) = make_float4(x.val[t], x.val[t + 1], x.val[t + 2], x.val[t + 3]);
        if (parts == 1)
          *reinterpret_cast<int4*>(cidx + o + t) = make_int4(x.idx[t], x.idx[t + 1], x.idx[t + 2], x.idx[t + 3]);
      }
      return;
    }
#pragma unroll
    for (int t = 0; t < kT; ++t) {
      cval[o + t] = x.val[t];
      cidx[o + t] = x.idx[t];
    }
  }
};

// The same on pairs of SMs: 256 rows x 256 codewords per item, each epilogue part keeping the best scores of its
// 128 codewords as a chunk of its own (16,384 rows, D = 4096, K = 4,096: 972 us one SM per item, 825 in pairs; tiles of
// 128 columns, which fill a last round better, load as many bytes per product as one SM's and were no faster).
struct PairAssignPolicy : AssignPolicy<128> {
  static constexpr int TN_PAIR = 256;
  __device__ __forceinline__ int64_t total_pair() const { return cdiv(this->n, (int64_t)256) * ((this->nch + 1) / 2); }
  __device__ __forceinline__ Item decode_pair(int64_t item) const {
    const int cols = (this->nch + 1) / 2;
    Item it;
    it.r0 = item / cols * 256;
    it.c = 2 * (int)(item % cols);
    it.nr = (int)min((int64_t)256, this->n - it.r0);
    return it;
  }
  __device__ __forceinline__ Item sub(const Item& w, int rank, int part) const {
    const bool in = w.c + part < this->nch;  // (no last half chunk: no rows to write)
    return Item{w.r0 + 128 * rank, in ? min(128, max(0, w.nr - 128 * rank)) : 0, w.c + part};
  }
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// the two-float distances ||x - b||^2 of up to kBatch candidates at once: each chunk
// of the row is read once and compared with every candidate. WPR warps share a
// row (warp `sub` takes every WPR-th 128 elements; their sums are added in warp order
// through `part`, and all of the block's threads call this together).
constexpr int kBatch = 8;
struct DfPart {
  float hi[8], lo[8];
};
template <int WPR>
__device__ void dist_df_batch(const float* __restrict__ x, const float* __restrict__ cb, const int (&kc)[kBatch],
                              int n, int D, int lane, int sub, DfPart* part, float (&ohi)[kBatch],
                              float (&olo)[kBatch]) {
  float hi[kBatch], lo[kBatch];
#pragma unroll
  for (int c = 0; c < kBatch; ++c) {
    hi[c] = 0.f;
    lo[c] = 0.f;
  }
#pragma unroll(WPR == 1 ? 1 : 2)
  for (int d = (sub * 32 + lane) * 4; d < D; d += 128 * WPR) {
    const float4 xv = *reinterpret_cast<const float4*>(x + d);
    const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
    for (int c = 0; c < kBatch; ++c) {
      if (c >= n) break;
      const float4 bv = *reinterpret_cast<const float4*>(cb + (int64_t)kc[c] * D + d);
      const float bs[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float s2, e;
        two_sum(xs[q], -bs[q], s2, e);  // x - b = s2 + e exactly
        const float p = s2 * s2;
        float pe = fmaf(s2, s2, -p);    // s2^2 = p + pe exactly
        pe = fmaf(2.f * s2, e, pe);     // + 2 s2 e (e^2 is below 2^-48 s2^2)
        float t, te;
        two_sum(hi[c], p, t, te);
        hi[c] = t;
        lo[c] += te + pe;
      }
    }
  }
#pragma unroll
  for (int c = 0; c < kBatch; ++c) {
    if (c >= n) break;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h2 = __shfl_xor_sync(kFull, hi[c], o);
      const float l2 = __shfl_xor_sync(kFull, lo[c], o);
      float t, te;
      two_sum(hi[c], h2, t, te);
      hi[c] = t;
      lo[c] = lo[c] + l2 + te;
    }
  }
  if constexpr (WPR > 1) {
    __syncthreads();  // part may still be read from the call before
    if (lane == 0)
#pragma unroll
      for (int c = 0; c < kBatch; ++c) {
        part[sub].hi[c] = hi[c];
        part[sub].lo[c] = lo[c];
      }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kBatch; ++c) {
      if (c >= n) break;
      hi[c] = part[0].hi[c];
      lo[c] = part[0].lo[c];
#pragma unroll
      for (int w = 1; w < WPR; ++w) {
        float t, te;
        two_sum(hi[c], part[w].hi[c], t, te);
        hi[c] = t;
        lo[c] = lo[c] + part[w].lo[c] + te;
      }
    }
  }
#pragma unroll
  for (int c = 0; c < kBatch; ++c) {
    if (c >= n) break;
    float t, te;
    two_sum(hi[c], lo[c], t, te);
    ohi[c] = t;
    olo[c] = te;
  }
}

// the same in plain FP32: relative error below (D / 32 + 8) 2^-24, a chain of D / 32 additions per lane and a tree, and
// where squares underflow 2^-150 for each of them
template <int WPR>
__device__ void dist_f32_batch(const float* __restrict__ x, const float* __restrict__ cb, const int (&kc)[kBatch],
                               int n, int D, int lane, int sub, DfPart* part, float (&out)[kBatch]) {
#pragma unroll
  for (int c = 0; c < kBatch; ++c) out[c] = 0.f;
#pragma unroll 2
  for (int d = (sub * 32 + lane) * 4; d < D; d += 128 * WPR) {
    const float4 xv = *reinterpret_cast<const float4*>(x + d);
#pragma unroll
    for (int c = 0; c < kBatch; ++c) {
      if (c >= n) break;
      const float4 bv = *reinterpret_cast<const float4*>(cb + (int64_t)kc[c] * D + d);
      const float s0 = xv.x - bv.x, s1 = xv.y - bv.y, s2 = xv.z - bv.z, s3 = xv.w - bv.w;
      out[c] = fmaf(s0, s0, out[c]);
      out[c] = fmaf(s1, s1, out[c]);
      out[c] = fmaf(s2, s2, out[c]);
      out[c] = fmaf(s3, s3, out[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < kBatch; ++c) {
    if (c >= n) break;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) out[c] += __shfl_xor_sync(kFull, out[c], o);
  }
  if constexpr (WPR > 1) {
    __syncthreads();  // part may still be read from the call before
    if (lane == 0)
#pragma unroll
      for (int c = 0; c < kBatch; ++c) part[sub].hi[c] = out[c];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kBatch; ++c) {
      if (c >= n) break;
      out[c] = part[0].hi[c];
#pragma unroll
      for (int w = 1; w < WPR; ++w) out[c] += part[w].hi[c];
    }
  }
}

__device__ __forceinline__ bool df_less(float ah, float al, int ak, float bh, float bl, int bk) {
  if (ah != bh) return ah < bh;
  if (al != bl) return al < bl;
  return ak < bk;
}

// warp-wide best entry of (value desc, position asc) strictly after the key
// (pv, pp) in that order; positions index the row's nch * kT kept entries, those with no codeword left out
__device__ __forceinline__ void next_best(const float* __restrict__ v, const int32_t* __restrict__ id, int tot,
                                          int K, float pv, int pp, int lane, float& bv, int& bp) {
  bv = -INFINITY;
  bp = 0x7fffffff;
  for (int e = lane; e < tot; e += 32) {
    const float x = v[e];
    if ((unsigned)id[e] >= (unsigned)K) continue;
    const bool after = x < pv || (x == pv && e > pp);
    if (after && (x > bv || (x == bv && e < bp))) {
      bv = x;
      bp = e;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(kFull, bv, o);
    const int op = __shfl_xor_sync(kFull, bp, o);
    if (ov > bv || (ov == bv && op < bp)) {
      bv = ov;
      bp = op;
    }
  }
}

// WPR: warps per row, 1, or 8 (a block per row) where the rows are few: a row's distances are then eight times
// shorter chains of dependent reads. (A warp per row: four blocks on an SM, 64 registers; 76 without that bound, 1% of a
// k-means call.)
template <int WPR>
__global__ __launch_bounds__(256, WPR == 1 ? 4 : 1) void k_assign_refine(const float* __restrict__ X, int64_t n, int D,
                                                       const float* __restrict__ cb, int K, int ma,
                                                       const float* __restrict__ cval,
                                                       const int32_t* __restrict__ cidx, int nch, int tn, int kT,
                                                       const float* __restrict__ x_inv, float bmax_host,
                                                       const float* __restrict__ bmax_dev, int parts,
                                                       const float* __restrict__ half_sq,
                                                       int32_t* __restrict__ codes, int* err) {
  dep_begin();
  if (blockIdx.x == 0 && threadIdx.x == 0) report_wait(err);
  __shared__ DfPart part[8];
  __shared__ float sval[WPR > 1 ? kPartsK : 1];
  __shared__ int32_t sidx[WPR > 1 ? kPartsK : 1];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = w % WPR;
  const int64_t r = (int64_t)blockIdx.x * (8 / WPR) + w / WPR;
  if (r >= n) return;  // (with a block per row every warp decides everything alike)
  const float* x = X + r * (int64_t)D;
  const int tot = nch * kT;
  const float* v = cval + r * tot;
  const int32_t* id = cidx + r * tot;
  if constexpr (WPR > 1) {
    if (parts > 1) {  // the scores of all codewords (tot <= kPartsK), from their products' parts in order
      for (int k = threadIdx.x; k < tot; k += 256) {
        float p[kMaxParts];
#pragma unroll
        for (int i = 0; i < kMaxParts; ++i) p[i] = i < parts ? v[i * n * tot + k] : 0.f;
        float x = p[0];
#pragma unroll
        for (int i = 1; i < kMaxParts; ++i) x += p[i];
        sval[k] = k < K ? x - half_sq[k] : -INFINITY;
        sidx[k] = k < K ? k : 0x7fffffff;
      }
      __syncthreads();
      v = sval;
      id = sidx;
    }
  }
  // the ma-th best coarse score over all chunks
  float thr = INFINITY;
  int tp = -1, found = 0;
  for (int a = 0; a < ma; ++a) {
    float bv;
    int bp;
    next_best(v, id, tot, K, thr, tp, lane, bv, bp);
    if (bp == 0x7fffffff) break;
    thr = bv;
    tp = bp;
    ++found;
  }
  const float bmax = bmax_dev ? *bmax_dev : bmax_host;
  const float xi = x_inv[r];
  const float xn = xi > 0.f ? 1.0001f / xi : 0.f;
  const float E = 2.44140625e-4f * (xn * bmax + 0.5f * bmax * bmax) + 1e-30f;
  const float lim = thr - 2.f * E;
  // a chunk whose last kept score is a candidate may hold more candidates
  bool full = xi == 0.f || found < ma;  // (fewer kept scores than ma only with non-finite inputs)
  for (int c = lane; c < nch; c += 32) {
    const int e = c * kT + kT - 1;
    if ((unsigned)id[e] < (unsigned)K && v[e] >= lim && min(tn, K - c * tn) > kT) full = true;
  }
  full = __any_sync(kFull, full);
  if (!full && ma == 1) {
    // a single candidate is the nearest codeword: the true nearest always lies in
    // the window, and so would any codeword at an equal true distance
    int cnt = 0, only = 0x7fffffff;
    for (int base = 0; base < tot; base += 32) {
      const int e = base + lane;
      const int kk = e < tot ? id[e] : 0x7fffffff;
      const bool take = e < tot && (unsigned)kk < (unsigned)K && v[e] >= lim;
      const unsigned m = __ballot_sync(kFull, take);
      if (m && cnt == 0) only = __shfl_sync(kFull, kk, __ffs(m) - 1);
      cnt += __popc(m);
    }
    if (cnt == 1) {
      if (lane == 0 && sub == 0) codes[r] = only;
      return;
    }
  }
  float H[GIFT_MAX_MA], Lo[GIFT_MAX_MA];
  int Kx[GIFT_MAX_MA];
#pragma unroll
  for (int a = 0; a < GIFT_MAX_MA; ++a) {
    H[a] = INFINITY;
    Lo[a] = 0.f;
    Kx[a] = 0x7fffffff;
  }
  auto insert = [&](float h, float l, int k) {  // into the ascending list of the ma best (registers, unrolled)
    if (df_less(h, l, k, H[GIFT_MAX_MA - 1], Lo[GIFT_MAX_MA - 1], Kx[GIFT_MAX_MA - 1])) {
      H[GIFT_MAX_MA - 1] = h;
      Lo[GIFT_MAX_MA - 1] = l;
      Kx[GIFT_MAX_MA - 1] = k;
#pragma unroll
      for (int t = GIFT_MAX_MA - 1; t > 0; --t) {
        if (df_less(H[t], Lo[t], Kx[t], H[t - 1], Lo[t - 1], Kx[t - 1])) {
          const float th = H[t], tl = Lo[t];
          const int tk = Kx[t];
          H[t] = H[t - 1];
          Lo[t] = Lo[t - 1];
          Kx[t] = Kx[t - 1];
          H[t - 1] = th;
          Lo[t - 1] = tl;
          Kx[t - 1] = tk;
        }
      }
    }
  };
  bool batched = false;
  if (!full) {
    // up to kBatch candidates: one pass over the row for all of them
    int kc[kBatch];
    int n = 0;
#pragma unroll
    for (int c = 0; c < kBatch; ++c) kc[c] = 0;
    for (int base = 0; base < tot; base += 32) {
      const int e = base + lane;
      const int kk = e < tot ? id[e] : 0x7fffffff;
      unsigned m = __ballot_sync(kFull, e < tot && (unsigned)kk < (unsigned)K && v[e] >= lim);
      while (m) {
        const int j = __ffs(m) - 1;
        m &= m - 1;
        const int k = __shfl_sync(kFull, kk, j);
#pragma unroll
        for (int c = 0; c < kBatch; ++c)
          if (c == n) kc[c] = k;
        ++n;
      }
    }
    if (n <= kBatch) {
      // plain FP32 distances decide where their order is beyond their error (nearly always: the window is some
      // thirty times wider), at an eighth of the two-float instructions
      float dv[kBatch];
      int kv[kBatch];
      dist_f32_batch<WPR>(x, cb, kc, n, D, lane, sub, part, dv);
#pragma unroll
      for (int c = 0; c < kBatch; ++c) {
        kv[c] = kc[c];
        if (c >= n) dv[c] = INFINITY;
      }
#pragma unroll
      for (int i = 0; i < kBatch; ++i)
#pragma unroll
        for (int c = i & 1; c + 1 < kBatch; c += 2)
          if (dv[c + 1] < dv[c]) {
            const float td = dv[c];
            dv[c] = dv[c + 1];
            dv[c + 1] = td;
            const int tk = kv[c];
            kv[c] = kv[c + 1];
            kv[c + 1] = tk;
          }
      // twice the error bound on either side of every gap that the codes' order rests on (1e-40: D 2^-150 up to D = 2^16)
      const float eps = (float)(D / 32 + 16) * 1.1920929e-7f;
      bool clear = true;
#pragma unroll
      for (int c = 0; c + 1 < kBatch; ++c)
        if (c < ma && c + 1 < n) clear = clear && dv[c + 1] - dv[c] > fmaf(eps, dv[c + 1] + dv[c], 1e-40f);
      if (clear) {
        if (lane < ma && sub == 0) {
          int out = kv[0];
#pragma unroll
          for (int a = 1; a < kBatch; ++a)
            if (a == lane) out = kv[a];
          codes[r * ma + lane] = out;
        }
        return;
      }
      float hh[kBatch], ll[kBatch];
      dist_df_batch<WPR>(x, cb, kc, n, D, lane, sub, part, hh, ll);
#pragma unroll
      for (int c = 0; c < kBatch; ++c)
        if (c < n) insert(hh[c], ll[c], kc[c]);
      batched = true;
    }
  }
  const int nscan = batched ? 0 : full ? K : tot;
  for (int base = 0; base < nscan; base += 32) {
    const int e = base + lane;
    bool take;
    int kk;
    if (full) {
      take = e < K;
      kk = e;
    } else {
      kk = e < tot ? id[e] : 0x7fffffff;
      take = e < tot && (unsigned)kk < (unsigned)K && v[e] >= lim;
    }
    unsigned mask = __ballot_sync(kFull, take);
    while (mask) {
      const int j = __ffs(mask) - 1;
      mask &= mask - 1;
      const int k = __shfl_sync(kFull, kk, j);
      float hh[kBatch], ll[kBatch];
      int kc[kBatch];
#pragma unroll
      for (int c = 0; c < kBatch; ++c) kc[c] = k;
      dist_df_batch<WPR>(x, cb, kc, 1, D, lane, sub, part, hh, ll);
      insert(hh[0], ll[0], k);
    }
  }
  if (lane < ma && sub == 0) {
    int out = Kx[0];
#pragma unroll
    for (int a = 1; a < GIFT_MAX_MA; ++a)
      if (a == lane) out = Kx[a];
    // (no codeword is near a row that is not finite: any code of the vocabulary, for the lists are indexed by it)
    codes[r * ma + lane] = (unsigned)out < (unsigned)K ? out : lane;
  }
}

// hi = bf16(x), lo = bf16(x - hi), row-major [n, D]
__global__ void k_split_rows(const float* __restrict__ X, int64_t n, int D, __nv_bfloat16* __restrict__ hi,
                             __nv_bfloat16* __restrict__ lo) {
  dep_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // index of a float4
  if (i >= n * (D / 4)) return;
  const float4 v = reinterpret_cast<const float4*>(X)[i];
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y);
  const __nv_bfloat162 b = __floats2bfloat162_rn(v.z, v.w);
  reinterpret_cast<__nv_bfloat162*>(hi)[2 * i] = a;
  reinterpret_cast<__nv_bfloat162*>(hi)[2 * i + 1] = b;
  const float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
  reinterpret_cast<__nv_bfloat162*>(lo)[2 * i] = __floats2bfloat162_rn(v.x - fa.x, v.y - fa.y);
  reinterpret_cast<__nv_bfloat162*>(lo)[2 * i + 1] = __floats2bfloat162_rn(v.z - fb.x, v.w - fb.y);
}

// the same and 1 / ||x|| of each row (0 for a zero row) from one read; warp per row, the norm's terms added as
// k_row_invnorm adds them
__global__ __launch_bounds__(256) void k_split_norm(const float* __restrict__ X, int64_t n, int D,
                                                    __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                                    float* __restrict__ inv) {
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= n) return;
  const float4* p = reinterpret_cast<const float4*>(X + row * (int64_t)D);
  uint2* h = reinterpret_cast<uint2*>(hi + row * (int64_t)D);
  uint2* l = reinterpret_cast<uint2*>(lo + row * (int64_t)D);
  float acc = 0.f;
  for (int base = lane; base < (D >> 2); base += 32 * 8) {
    float4 x[8];  // eight reads in flight
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (base + 32 * k < (D >> 2)) x[k] = p[base + 32 * k];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = base + 32 * k;
      if (i >= (D >> 2)) break;
      const float4 v = x[k];
      acc = fmaf(v.x, v.x, acc);
      acc = fmaf(v.y, v.y, acc);
      acc = fmaf(v.z, v.z, acc);
      acc = fmaf(v.w, v.w, acc);
      const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
      const float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
      const __nv_bfloat162 c = __floats2bfloat162_rn(v.x - fa.x, v.y - fa.y);
      const __nv_bfloat162 d = __floats2bfloat162_rn(v.z - fb.x, v.w - fb.y);
      h[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
      l[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&c), *reinterpret_cast<const uint32_t*>(&d));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
  if (lane == 0) inv[row] = acc > 0.f ? 1.0f / sqrtf(acc) : 0.f;
}

}  // namespace

void split_rows_bf16(const float* X, int64_t n, int D, __nv_bfloat16* hi, __nv_bfloat16* lo, cudaStream_t s) {
  if (n <= 0) return;
  const int64_t n4 = n * (D / 4);
  launch_dep(k_split_rows, dim3((unsigned)cdiv(n4, 256)), dim3(256), 0, s, X, n, D, hi, lo);
  GIFT_LAUNCHED("k_split_rows");
}

SplitRows split_for_assign(const float* X, int64_t n, int D, float* inv, Scratch& sc, cudaStream_t s) {
  SplitRows r;
  const int64_t rows_alloc = n + tc::kTM;  // one box of padding rows
  r.hi = sc.get<__nv_bfloat16>((size_t)rows_alloc * D);
  r.lo = sc.get<__nv_bfloat16>((size_t)rows_alloc * D);
  if (n <= 0) return r;
  k_split_norm<<<(unsigned)cdiv(n, 8), 256, 0, s>>>(X, n, D, r.hi, r.lo, inv);
  GIFT_LAUNCHED("k_split_norm");
  return r;
}

void assign_codes(const Index& ix, const float* X, int64_t n, int ma, int32_t* codes, Scratch& sc, cudaStream_t s,
                  const float* x_inv, KernelClock* kc, const SplitRows* parts, const float* cb_max) {
  if (n <= 0) return;
  const int K = ix.prm.n_codewords, D = ix.prm.dim;
  GIFT_REQUIRE(ma >= 1 && ma <= GIFT_MAX_MA && ma <= K, "multiple assignment must be in [1, min(8, K)]");
  const int64_t chunk = std::min<int64_t>(n, kAssignChunk);
  const int64_t rows_alloc = chunk + tc::kTM;  // one box of padding rows
  GIFT_REQUIRE(!parts || n <= chunk, "a two-part copy made before covers one pass");
  __nv_bfloat16* hi = parts ? parts->hi : sc.get<__nv_bfloat16>((size_t)rows_alloc * D);
  __nv_bfloat16* lo = parts ? parts->lo : sc.get<__nv_bfloat16>((size_t)rows_alloc * D);
  const int sms = device_sm_count();
  // Codewords per item: 256 where that leaves an item for every SM (one pass over the rows), fewer otherwise.
  const int64_t row_tiles = cdiv(chunk, (int64_t)tc::kTM), full = row_tiles * cdiv(K, 256);
  int tn = 256;
  bool pair = false;
  if (full >= sms || K > 16384) {
    // Full SMs: pairs of them, where their rounds, each 0.85 of the others' time (measured), take less; for vocabularies
    // of 1,025 to 16,384 in any case, whose items keep their best scores sooner from 128 columns (1,300 rows, D = 256, K =
    // 16,384: 277 us in pairs, 342 one SM per item). Beyond, the refine's read of twice as many kept scores costs more.
    const int64_t items = cdiv(chunk, (int64_t)256) * cdiv(K, 256);
    pair = (K > 1024 && K <= 16384) ||
           0.85 * cdiv(items, (int64_t)tc::pair_clusters<PairAssignPolicy>()) < cdiv(full, (int64_t)sms);
  } else if (K > 4096 || (K > 192 && 3 * full >= sms)) {
    // Pairs too where a third of the SMs has items or the vocabulary is large: the refine reads 16 scores of every 64
    // codewords otherwise, which takes longer than the narrower items save (130 rows, D = 256, K = 16,384: 96 us in pairs,
    // 116 in items of 256, 183 of 64; 3,000 rows, D = 64, K = 1,100: 76, 96, 101; 20 rows, K = 4,096: 74, 85, 64)
    pair = true;
  } else {
    // all scores of items of 32 go to the refine: for small vocabularies, or one round of them (700 rows, D = 4096,
    // K = 1,024: 166 us in two rounds of 32, 120 in items of 64)
    tn = K > 1024 || row_tiles * cdiv(K, 64) >= sms || (K > 512 && row_tiles * cdiv(K, 32) > sms) ? 64 : 32;
  }
  if (pair) tn = 128;  // chunks of kept scores
  const int nch = (int)cdiv(K, tn), kT = kept_scores(tn);
  // Few items: their chains of k-blocks in parts, as long as a part keeps four k-blocks and finds a free SM; the
  // refine's block of a row adds the parts up (108 rows, D = 4096, K = 512: 16 items in 44 us, in eight parts 10;
  // the refine, which then reads its scores from shared memory, 30 and 27)
  const int nkb = (int)cdiv(D, tc::kTK);
  int cuts = 1;
  if (tn == 32 && n <= chunk && n < 8 * sms && nch * tn <= kPartsK)
    cuts = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)kMaxParts, nkb / 4, sms / (row_tiles * nch)}));
  float* cval = sc.get<float>((size_t)chunk * nch * kT * cuts);
  int32_t* cidx = sc.get<int32_t>((size_t)chunk * nch * kT);
  float* inv = nullptr;
  if (!x_inv) {
    inv = sc.get<float>(n);
    launch_row_invnorm(X, n, D, inv, s);
    x_inv = inv;
  }
  const CUtensorMap tB = make_tmap_bf16(ix.cb_hi, ix.cb_rows_alloc, D, tn);
  const CUtensorMap tB2 = make_tmap_bf16(ix.cb_lo, ix.cb_rows_alloc, D, tn);
  for (int64_t r0 = 0; r0 < n; r0 += chunk) {
    const int64_t m = std::min(chunk, n - r0);
    if (!parts) split_rows_bf16(X + r0 * D, m, D, hi, lo, s);
    const CUtensorMap tA = make_tmap_bf16(hi, rows_alloc, D, tc::kTM);
    const CUtensorMap tA2 = make_tmap_bf16(lo, rows_alloc, D, tc::kTM);
    const int grid = (int)std::min<int64_t>(sms, cdiv(m, tc::kTM) * nch * cuts);
    auto coarse = [&](auto p, auto launch) {
      p.n = m;
      p.K = K;
      p.nch = nch;
      p.nkb = nkb;
      p.parts = cuts;
      p.half_sq = ix.cb_half_sq;
      p.cval = cval;
      p.cidx = cidx;
      launch(p);
    };
    auto single = [&](const auto& p) { tc::launch_engine(tA, tB, tA2, tB2, p, ix.d_err, grid, s); };
    auto paired = [&](const auto& p) {  // (B boxes of half the pair's columns: tn)
      tc::launch_pair(tA, tB, tA2, tB2, p, ix.d_err, cdiv(m, (int64_t)256) * cdiv(nch, 2), s);
    };
    if (kc) kc->begin(0);
    if (pair) coarse(PairAssignPolicy{}, paired);
    else if (tn == 256) coarse(AssignPolicy<256>{}, single);
    else if (tn == 64) coarse(AssignPolicy<64>{}, single);
    else coarse(AssignPolicy<32>{}, single);
    if (kc) {
      kc->end(0);
      kc->assign_rows += m;
    }
    // A block that is resident while the coarse stage ends finds the SM's memory given to that stage's shared memory, and
    // little of it left as L1: where a row's kept scores are more than fit there, which its warps go over several
    // times, it waits for its launch instead (20 rows, D = 64, K = 65,536: 197 us so launched, 164 plainly).
    auto refine = [&](auto kernel, int64_t blocks) {
      const bool early = (int64_t)nch * kT * 8 <= 16 * 1024;
      auto go = [&](auto... a) {
        if (early) launch_dep(kernel, dim3((unsigned)blocks), dim3(256), 0, s, a...);
        else kernel<<<(unsigned)blocks, 256, 0, s>>>(a...);
      };
      go(X + r0 * D, m, D, (const float*)ix.codebook, K, ma, (const float*)cval, (const int32_t*)cidx, nch, tn, kT,
         x_inv + r0, ix.cb_max_norm, cb_max, cuts, (const float*)ix.cb_half_sq, codes + r0 * ma,
         ix.d_err);
    };
    if (m >= 8 * sms) refine(k_assign_refine<1>, cdiv(m, 8));
    else refine(k_assign_refine<8>, m);
    GIFT_LAUNCHED("k_assign_refine");
  }
}

}  // namespace gift
