// Fold (periodic search) pieces shared by the single-curve and batch paths.
#pragma once

#include <vector>

#include "nu_internal.cuh"

namespace nu {

// Node record of the single-event grid: depth, sigma = sqrt(var) (NaN when
// any of depth/var/gain is not finite or var <= 0), gain, and ig = 1/(gap to
// the next epoch) (NaN when there is no next epoch or the gap exceeds the
// limit).  Interpolating with a NaN anywhere yields a NaN sigma, which is how
// an epoch is dropped.
template <typename T> struct __align__(4 * sizeof(T)) Node4 {
    T d, s, l, ig;
};

// Node record of the exact path: the Node4 fields plus the differences to the
// next epoch's depth, sigma and gain (NaN when the next epoch is missing or
// invalid), so that an event is one record load and three FMAs. 
template <typename T> struct __align__(8 * sizeof(T)) Node8 {
    T d, s, l, ig, dd, ds, dl, pad;
};

// Screening record, one per (duration, epoch i): the FP32
// values and slopes of the interval [t0_i, t0_{i+1}], wsc = 2^-22 dt/gap (the
// weight per unit of the 2^-22-slot position difference), and flags = 1 when
// the interval is outside the screen's error model (epochs closer than dt/4,
// end sigmas more than a factor 3 apart, or values whose FP32 sums could
// overflow): a cell with an event there is evaluated exactly.  s is NaN on an
// invalid interval.
struct __align__(32) ScreenRec {
    float d, s, l, dd, ds, dl, wsc;
    unsigned flags;
};

// Byte layout of the exact path's per-(duration, epoch) arrays for n epochs:
// Node8 records, then (where the cells are screened) screening records and
// pairs of fixed-point epoch positions.
struct ExactLayout {
    size_t off_screen, off_vpos, total;
};
inline ExactLayout exact_layout(int64_t n, int n_D, bool fp64, bool screen = true) {
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    ExactLayout L;
    const size_t node = al((size_t)n * n_D * 8 * (fp64 ? 8 : 4));
    L.off_screen = node;
    L.off_vpos = node + (screen ? al((size_t)n * n_D * sizeof(ScreenRec)) : 0);
    L.total = L.off_vpos + (screen ? al((size_t)n * 16) : 0);
    return L;
}

// Geometry of one light curve of a batch fold.
struct FoldSeg {
    int64_t s_off;      // first epoch (= first sample) in the packed arrays
    int64_t n_t0;
    double t_ref, t_last;
    int64_t n_bucket, bucket_off;
    int64_t n_slots, rec_off;
    int use_slots;
    int screen;         // FP32 screening of the exact path allowed for this curve
    int64_t srec_off;   // FP64 path: first slot-indexed screening record
    unsigned long long ulast;   // slot path: the last epoch's position, 24.40 slots
    int64_t tab_off;    // first entry of the curve's filter tables
    int64_t g_off;      // first word of its G table
    int64_t pair_off;   // first entry of its S and Q tables (durations in pairs)
    unsigned long long uspan;   // screened curves: the last epoch's position, 24.40 slots
};

// ---- filter tables (see filter.cuh) and the lists of the cell kernels
__host__ __device__ inline int64_t filter_slots(int64_t n_slots) { return (n_slots + 7) / 8 * 8; }
// Durations of G's group gi (eight, the last group one, two, four or eight), and
// the numbers of all groups per slot.
__host__ __device__ inline int filter_width(int n_D, int gi) {
    const int r = n_D - 8 * gi;
    return r >= 5 ? 8 : (r >= 3 ? 4 : r);
}
__host__ __device__ inline int filter_cols(int n_D) {
    const int last = (n_D - 1) / 8;
    return 8 * last + filter_width(n_D, last);
}

// Tables of all curves; rows of filter_slots(n_slots) per duration from
// tab_off on (in rows' entries), G from g_off on (in words).  Where scratch is
// short only L and G are there (S, Q, gB, Z and vmax null), in small calls of the
// slot path L alone: the fold then bounds by gains.  All null: no tables.
struct FilterTab {
    uint2* S;
    float* gB;
    float* L;
    unsigned* Z;      // per slot (largest, smallest) Delta v as FP16 (source of Q)
    uint2* Q;
    float* G;
    unsigned* vmax;   // per (curve, duration): max 1/s^2 (float bits)
};

struct FilterLayout {
    size_t S, gB, L, Z, Q, G, vmax, total;
};
inline FilterLayout filter_layout(int64_t entries, int64_t pairs, int64_t words, int64_t rows,
                                  bool gains_only = false) {
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t all = gains_only ? 0 : 1;
    FilterLayout F;
    F.S = 0;
    F.Q = F.S + all * al((size_t)pairs * 8);
    F.gB = F.Q + all * al((size_t)pairs * 8);
    F.Z = F.gB + all * al((size_t)entries * 4);
    F.vmax = F.Z + all * al((size_t)entries * 4);
    F.L = F.vmax + all * al((size_t)rows * 4);
    F.G = F.L + al((size_t)entries * 4);
    F.total = F.G + al((size_t)words * 4);
    return F;
}
inline FilterTab filter_tab(char* p, const FilterLayout& F, bool gains_only = false) {
    if (gains_only)
        return FilterTab{nullptr, nullptr, (float*)(p + F.L), nullptr, nullptr,
                         (float*)(p + F.G), nullptr};
    return FilterTab{(uint2*)(p + F.S), (float*)(p + F.gB), (float*)(p + F.L),
                     (unsigned*)(p + F.Z), (uint2*)(p + F.Q), (float*)(p + F.G),
                     (unsigned*)(p + F.vmax)};
}

struct FoldCand {
    long long item;        // output index (curve * n_P + period); -1: none
    unsigned j;            // phase
    int d;                 // duration
    double lnp, Dl, s2;    // written by k_cand_eval
};
struct SlotBest {          // slot path: the best cell of an item
    float lnp, Dl, s2;
    unsigned j;
    int d;                 // -1: none, -2: invalid period
};

struct PeriodConst;
size_t period_const_bytes();

// Device scratch of the batch fold.
struct FoldScratch {
    void* nodes;            // exact-path records (exact_layout of all samples)
    int* bucket;            // bucket tables
    Node4<float>* rec;      // mixed slot records
    ScreenRec* srec;        // FP64 slot-indexed screening records
    int* slot_of;           // FP64: slot of every sample
    unsigned* reg;          // two words per curve (zeroed by the prep)
    unsigned long long* peak;  // per curve, the key of its largest gain
    PeriodConst* ptab;      // per period, its curve-independent constants
    FilterTab tab;
    FoldCand* cand;         // cells left for k_cand_eval (cap entries)
    unsigned long long cap;
    unsigned long long* n_cand;
    unsigned* list;         // list of the block items and its counters (n_cand behind)
    unsigned* n_list;
    int2* range;            // per item: its candidates
    struct ItemConst* items;   // per item: constants of the screen
    SlotBest* sbest;        // per item of the slot path
    int64_t pass;           // items per pass (the lists' room); 0: one pass without lists
};

// Host side of the batch fold: per-curve layout and launches.
struct FoldBatch {
    std::vector<FoldSeg> segs;
    int64_t n_bucket_total = 0, n_rec_total = 0, n_srec_total = 0;
    int64_t n_tab_total = 0;     // entries of the filter tables
    int64_t n_pair_total = 0;    // of those with durations in pairs
    int64_t n_g_total = 0;       // words of their G tables
    bool any_slots = false, any_exact = false;
    // What the scratch holds beside the records: 2 filter tables, and lists for the
    // items of a pass; 1 neither (every cell is screened, survivors evaluated in
    // place); 0 nor the screen's records of the mixed irregular path (every cell
    // is evaluated).
    int level = 2;
};
// Bytes of the batch fold's scratch; with a base, *fs receives its pointers.  The
// lists take 230 bytes per (curve, period) item, so that a large batch goes
// through them in passes of 2^22 items (1 GB) at most.
constexpr int64_t BATCH_PASS = 1ll << 22;
size_t fold_scratch(const FoldBatch& fb, int64_t n_total, int n_lc, int n_D, int64_t n_P,
                    bool fp64, char* base, FoldScratch* fs);

void plan_fold_batch(const std::vector<int64_t>& s_off, const std::vector<double>& t_first,
                     const std::vector<double>& t_last, const std::vector<int>& irregular,
                     bool fp64, double dt, double gap_factor, int n_D, int level,
                     FoldBatch& fb);

// Enqueues the fold's preparation kernels; returns the first error of an
// enqueued memset (the launches are checked by the caller) and the number of
// kernels launched in *n_launched.
cudaError_t launch_fold_prep(const FoldBatch& fb, const FoldSeg* segs_dev,
                             const int64_t* s_off_dev, int n_seg, int64_t n_total, bool fp64,
                             const double* t, const void* depth, const void* var,
                             const void* gain, int n_D, double dt, double gap_factor,
                             const FoldScratch& fs, cudaStream_t st, int* n_launched);

// Enqueues the fold of the first n_seg curves; side: a stream of the caller's for
// the block items.  Returns the number of kernels launched, and the first error
// of an enqueued memset in *err.
int launch_fold_batch(const FoldBatch& fb, const FoldSeg* segs_dev, int n_seg,
                      int64_t n_total, bool fp64, const double* t, const FoldScratch& fs,
                      int n_D, double dt, double gap_factor, const double* periods,
                      int64_t n_P, double* Q, double* T0, int* Didx, double* dep,
                      double* sig, double* lnp, cudaStream_t st, cudaStream_t side,
                      cudaError_t* err);

int launch_slots_test(const double* t, const int64_t* s_off_dev, int n_seg, int64_t n_total,
                      double dt, int* irregular, cudaStream_t st);

}  // namespace nu
