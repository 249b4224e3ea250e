// Per-call plan of an F-IF batch (device buffers in the call's scratch).
#pragma once
#include "gift_internal.cuh"

namespace gift {

struct FifPlan {
  // inputs
  int64_t nv = 0;                 // query views in the batch
  int ma = 1;                     // assignments per view
  int32_t B = 0;                  // queries
  const float* q = nullptr;       // [nv, D] FP32 query views
  const float* q_inv = nullptr;   // [nv]
  const int32_t* q_code = nullptr;// [nv * ma]
  const int32_t* qoff = nullptr;  // [B+1] device
  const int32_t* vquery = nullptr;// [nv] query of each view
  unsigned long long* stats = nullptr;  // optional [8]: scanned bytes, pairs, rescore bytes, then the
                                        // rescore's items, kept items, candidate pairs, candidate rows,
                                        // rows of kept items
  KernelClock* kc = nullptr;            // optional kernel timing
  // derived
  int64_t nslots = 0;
  int32_t* skeys = nullptr;       // [nslots] codeword of each slot (ascending)
  int64_t* boff = nullptr;        // [K+1] slots of codeword k
  int32_t* slot_view = nullptr;   // [nslots]
  int32_t* view_slot = nullptr;   // [nv * ma]
  int64_t* runbase = nullptr;     // [nslots + 1] first table cell of each slot; [nslots] = cells in use
  int64_t upper_items = 0;        // bound on the number of scan work items, whatever the tiles
  int64_t table_upper = 0;        // bound on the table cells
  // slot-ordered two-part BF16 query rows, made by the first tensor-core pass
  // that needs them and reused by the next (scan, then rescore)
  mutable __nv_bfloat16* slot_hi = nullptr;
  mutable __nv_bfloat16* slot_lo = nullptr;
  mutable const int64_t* class_woff = nullptr;  // work offsets of every slot class (k_scan_tc.cu), made by the scan
};

// Work items of the batch's touched lists: offsets [K+1] per spec (exclusive, the last is the total). A spec takes
// tiles of tn entries x ts slots; cls > 0: only the lists of that slot class. All specs in one launch, a block each.
constexpr int kMaxSpecs = 6;
struct WorkSpecs {
  int n = 0;
  int sms = 0, pairs = 0;  // > 0: specs 0 and 1 are the same work one SM or one pair of SMs per item, and the slower
                           // one's offsets are all zero (tc::pair_wins, decided where the item counts are)
  int cls[kMaxSpecs], tn[kMaxSpecs], ts[kMaxSpecs];
  void add(int c, int n_, int s) {
    cls[n] = c;
    tn[n] = n_;
    ts[n++] = s;
  }
};
// `fold`: with at most so many items of slot-column classes altogether they all take the smallest class that holds
// their lists (0: never)
int64_t* plan_work(const Index& ix, const FifPlan& P, const WorkSpecs& specs, int64_t fold, Scratch& sc,
                   cudaStream_t s);
// slot classes: lists of up to 16, 32, 64, 80 slots (slot columns), more (slot rows, 128)
__host__ __device__ constexpr int slot_class(int64_t M) {
  return M <= 16 ? 16 : M <= 32 ? 32 : M <= 64 ? 64 : M <= 80 ? 80 : 128;
}

void fif_plan(const Index& ix, FifPlan& P, Scratch& sc, cudaStream_t s);
// clear the table cells the batch uses (runbase[nslots] of them; the table is
// allocated for table_upper)
void fif_zero_table(const FifPlan& P, uint32_t* table, cudaStream_t s);
void fif_scan(const Index& ix, const FifPlan& P, uint32_t* table, bool rescore,
              const int32_t* cand_sorted, int R, Scratch& sc, cudaStream_t s);
// tcgen05 scan of a BF16 or E4M3 store (rescore: two-part BF16, candidates only;
// table32 non-null: a BF16 store with its two-part rows scanned at FP32 level over
// every touched pair, which fills `table32` with the maxima of every run: the
// candidates and their scores both come from it, with no separate rescore)
void fif_scan_tc(const Index& ix, const FifPlan& P, uint32_t* table, bool rescore, const int32_t* cand_sorted,
                 int R, Scratch& sc, cudaStream_t s, uint32_t* table32 = nullptr);
// counts of the candidate work of a batch (stats [3..7]) without running the
// rescore: for the FP32-level pass over every touched pair of a BF16 store
void fif_rescore_stats(const Index& ix, const FifPlan& P, const int32_t* cand_sorted, int R, Scratch& sc,
                       cudaStream_t s);
void fif_combine(const Index& ix, const FifPlan& P, const uint32_t* table, float* S_dense,
                 const int32_t* cand_sorted, int R, float* cand_score, Scratch& sc, cudaStream_t s);

}  // namespace gift
