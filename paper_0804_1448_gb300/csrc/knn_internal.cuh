// knn_internal.cuh -- declarations shared by the kernel files of the library.
//
// The search (Sec. 2.1 of Garcia, Debreuve, Barlaud, "Fast k Nearest Neighbor
// Search using GPU") runs as three stages, all on the GPU:
//   1. select   -- a fused distance + per-query top-c kernel: each tile of the
//                  n x m distance matrix is produced on chip and consumed at
//                  once by a per-query selection; only c candidates per query
//                  (and per reference split) reach global memory.  The CUDA-core
//                  form (knn_cc.cu) computes float32 distances from coordinate
//                  differences; the tensor-core form (knn_tc.cu) computes the
//                  cross term q.r with tcgen05 and ranks by ||r||^2 - 2 q.r.
//                  A float32 Euclidean search takes the tensor-core form on
//                  pairs of bf16 words, whose answers the finalize certifies;
//                  the queries it cannot certify take the CUDA-core form.
//                  Manhattan and Chebyshev searches likewise filter on CUDA
//                  cores first (knn_diff.cu).
//   2. finalize -- per query: exact float32 distances of the candidates, a sort
//                  by (distance, index), a float64 re-check of candidates whose
//                  float32 distances are within rounding of each other, and the
//                  k outputs (knn_finalize.cu).  Queries whose candidate set
//                  cannot be certified complete are queued for stage 3.
//   3. fallback -- exact float64 distances to every reference and an exact
//                  radix selection, for the queued queries only (rare: it needs
//                  more near-equal distances than there are spare candidates).
#pragma once

#include <atomic>
#include <cstdint>
#include <cuda_runtime.h>

namespace knn {

// Opt kernel KERN in to `smem` bytes of dynamic shared memory, once per
// device and size: cudaFuncSetAttribute costs host time on every call (tens
// of microseconds in front of an idle GPU), and the setting persists.
template <auto KERN>
cudaError_t allow_smem(size_t smem) {
    constexpr int kDevs = 64;
    static std::atomic<size_t> done[kDevs];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const bool tracked = dev >= 0 && dev < kDevs;
    if (tracked && smem <= done[dev].load(std::memory_order_relaxed)) return cudaSuccess;
    err = cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (err == cudaSuccess && tracked) {
        size_t cur = done[dev].load(std::memory_order_relaxed);
        while (smem > cur && !done[dev].compare_exchange_weak(cur, smem)) {
        }
    }
    return err;
}

// The kernels of one search run one after another on one stream, each set up
// while its predecessor still runs (programmatic dependent launch): a kernel
// calls chain_begin() before it touches memory, which waits until everything
// before it on the stream is done.  Every kernel that launch_chained launches
// calls it, on every path that reads or writes memory; the first kernel of a
// search is launched plainly, so a search waits for whatever the caller's stream
// holds.  Searches with device buffers are chained: n = m = 1200, d = 8 (three
// kernels) 32.5 -> 22.6 us, n = 4999, m = 20011, d = 50 116 -> 92.  Those with
// host buffers are not (chain = false): the parts of a large one share the SMs
// from two streams.
// No kernel lets its successor in early (griddepcontrol.launch_dependents): its
// CTAs would settle, waiting, on whatever SMs have room first, several on one,
// and keep the other streams' kernels out.  With it the 4096 queries of m =
// 20000, d = 96 that the exact fallback takes cost 73 ms instead of 38, n = 2000,
// m = 9600, d = 64 in tf32 58 us instead of 48, and two handles searching at once
// (n = 1024, m = 100000, d = 64, bf16) 69 us a search instead of 47; what it saves
// is about 1 us a kernel where every grid is many waves long (n = m = 38400, d =
// 96, bf16: 541 against 546 us).
__device__ __forceinline__ void chain_begin() {
#ifdef __CUDA_ARCH__
    asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}
template <typename... P, typename... A>
cudaError_t launch_chained(bool chain, void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                           cudaStream_t st, const A&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

enum Metric : int { kL2 = 0, kL1 = 1, kLinf = 2 };

constexpr uint64_t kEmptyKey = ~0ull;  // sentinel for an empty candidate slot

// Order-preserving map float -> uint32 (total order on non-NaN floats).
__host__ __device__ __forceinline__ uint32_t ord_f32(float x) {
#ifdef __CUDA_ARCH__
    uint32_t b = __float_as_uint(x);
#else
    uint32_t b;
    __builtin_memcpy(&b, &x, 4);
#endif
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__host__ __device__ __forceinline__ float unord_f32(uint32_t o) {
    uint32_t b = (o & 0x80000000u) ? (o & 0x7fffffffu) : ~o;
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    __builtin_memcpy(&x, &b, 4);
    return x;
#endif
}

// Candidate key: (distance, index) packed so that unsigned comparison is the
// lexicographic order of the pair (smaller distance first, then smaller index).
__host__ __device__ __forceinline__ uint64_t make_key(float dist, uint32_t idx) {
    return (static_cast<uint64_t>(ord_f32(dist)) << 32) | idx;
}
__host__ __device__ __forceinline__ uint32_t key_idx(uint64_t key) {
    return static_cast<uint32_t>(key & 0xffffffffu);
}
__host__ __device__ __forceinline__ float key_dist(uint64_t key) {
    return unord_f32(static_cast<uint32_t>(key >> 32));
}

// Where the candidates of one search live: n queries x S reference splits x c.
// Split s covers references [s*chunk, min(m, (s+1)*chunk)).
struct CandidateSet {
    uint64_t* keys;   // [n][S][c]
    int64_t n;
    int32_t S;
    int32_t c;
    int64_t chunk;
    int32_t exact;    // 1: key distances are float32 distances of the metric
                      //    (completeness can be certified); 0: ranking scores
    int32_t* clear;   // a counter the select sets to zero (the search's queue), or null
    int32_t chain;    // launch the select of a queue in the search's chain (launch_chained)
};

// Per-query lists of references that passed the tensor-core filter (S lists
// per query: one per reference split and epilogue column group).  A key is
// (code, index) with code in [0, 0xffff] falling linearly with the
// low-precision score (smaller code = nearer).  counts may exceed cap,
// meaning the list overflowed.
struct HitLists {
    const uint64_t* keys;   // [n][S][cap]
    const int32_t* counts;  // [n][S]
    int32_t S;
    int32_t cap;
    int32_t c;              // keep (at least) the best c before the exact re-rank
    // float32 searches, whose answers are certified (else null): [n].
    // Operand pairs: every reference is at least bound - 2 acc away (squared),
    // acc < 0 for those not listed; the keys' high word is 0x7f800000 minus the
    // bits of acc.  Differences: those not listed are farther than bound; the
    // high word is the bits of the distance.
    const float* bound;
};

// The queries one pass left to the next: list[0 .. *count).  A pass over a
// queue does nothing while it holds `direct` queries or fewer (an argument of
// each pass): those go straight to the exact fallback.
struct QueryQueue {
    int32_t* list;    // null: the pass covers every query
    int32_t* count;
};
// How many queued queries the exact fallback spreads over the GPU, given its
// scratch slots (the others take one CTA each); and the most that a queue may
// send it at once.
inline int32_t fallback_spread(int32_t slots) { return slots >= 2 ? slots / 2 : 0; }
constexpr int kDirectMost = 32;

struct FinalizeArgs {
    int32_t use_hits;       // 0: candidates come from `cand`; 1: from `hits`
    HitLists hits;
    const float* Q;
    const float* R;
    int64_t n, m;
    int32_t d, k;
    int32_t metric;
    CandidateSet cand;
    float* dist_out;
    int32_t* idx_out;
    int32_t* fallback_count;   // device counter of queued queries
    int32_t* fallback_list;    // [n] query ids
    QueryQueue from;           // list: only these queries, candidate row i being that of
                               // the queue's i-th; null: all n
    int32_t leave;             // 1: fallback_list is the next pass's queue, not the exact
                               // fallback's (its queries are not counted as such)
    int32_t direct;            // `from`: queues up to this long are not finished here
    unsigned long long* recheck_counter;
    unsigned long long* fallback_total;
    unsigned long long* fallback_reason;   // [4]: short list, overflow, wide cut, uncertified
    int32_t* fb_done;                      // fallback chunk counters to zero, or null
    int32_t fb_slots;
    int32_t chain;                         // launch in the search's chain (launch_chained)
    // rounding bounds for this d, set by launch_finalize: float32 distance
    // (relative), its near-tie window as a float, and the float-float window
    double rel;
    float relf;
    float ffw;
};

// ---- launchers (return cudaSuccess or the launch error) -------------------

// CUDA-core fused distance + top-c.  Writes cand (exact = 1).
// from.list: only the queue's queries, candidate row i being that
// of its i-th, and none while there are no more than `direct`.
cudaError_t launch_cc_select(const float* Q, int64_t n, const float* R, int64_t m, int32_t d,
                             int32_t metric, const CandidateSet& cand, cudaStream_t st,
                             int* launches, const QueryQueue& from = QueryQueue{},
                             int32_t direct = 0);

// Manhattan and Chebyshev searches with a pilot threshold and hit lists
// (knn_diff.cu), one list per query and split.
struct DiffPlan {
    int32_t rows;        // queries per CTA: 128, 64 or 16 (0: rows too long)
    int32_t tiles;       // 128-reference tiles of the set
    int32_t tps;         // tiles per split
    int32_t S;           // reference splits
    int32_t stride;      // pilot samples every stride-th tile of the set
    int32_t spt;         // sampled tiles per pilot CTA
    int32_t pS;          // pilot CTAs per query tile
    int32_t G;           // pilot group maxima per query (groups of 32 references)
    int32_t cprime;      // order statistic of the group maxima used as threshold
    int32_t cap;         // list capacity per (query, split)
    bool pilot;          // there are groups enough for the order statistic
    bool chain;          // launch in the search's chain (launch_chained)
};
DiffPlan diff_plan(int64_t n, int64_t m, int32_t d, int32_t c, int num_sms);
cudaError_t launch_diff_pilot(const DiffPlan& p, const float* Q, int64_t n, const float* R, int64_t m,
                              int32_t d, int32_t metric, uint32_t* gmax, cudaStream_t st, int* launches);
// Also clears the two counters.
cudaError_t launch_diff_threshold(const DiffPlan& p, const uint32_t* gmax, int64_t n, float* thr,
                                  int32_t* count0, int32_t* count1, cudaStream_t st, int* launches);
cudaError_t launch_diff_filter(const DiffPlan& p, const float* Q, int64_t n, const float* R, int64_t m,
                               int32_t d, int32_t metric, const float* thr, uint64_t* lists,
                               int32_t* counts, cudaStream_t st, int* launches);

// The largest c launch_cc_select supports.
int cc_max_candidates();

// Float32 select for small reference sets (knn_small.cu): one warp per query
// holds all m distances in shared memory and selects exactly a set of keys
// that holds its c_need nearest and that no key left out precedes, of at most
// cand.c (>= c_need) keys, the unused slots empty.  Writes cand with S = 1
// split of the whole set (exact = 1).  Available when small_select_fits(m, d):
// m up to kSmallSelectMaxM and the shared memory (small_select_smem) within
// one CTA's.  kSmallSelectSpare: the spare slots a search plans beyond c_need.
constexpr int64_t kSmallSelectMaxM = 4096;
constexpr int kSmallSelectSpare = 16;
// Tensor-core searches whose pilot runs still take the small-set select while
// ceil(n / 8) * m * d / SMs (an SM's share of its distance products) is below this.
constexpr double kSmallSelectShare = 2.2e5;
size_t small_select_smem(int64_t m, int32_t d);
bool small_select_fits(int64_t m, int32_t d);
cudaError_t launch_small_select(const float* Q, int64_t n, const float* R, int64_t m, int32_t d,
                                int32_t metric, int32_t c_need, const CandidateSet& cand,
                                cudaStream_t st, int* launches);

// Reference splits S of the float32 search and their length *chunk (a
// multiple of 128): among the S with every split at least 8c long and S*c
// within max_pool, and at least two CTAs per SM where that is possible, the
// one with the least estimated time, the CTAs resident on an SM sharing its
// throughput (so a partly filled last wave of CTAs costs what its busiest SM
// holds).
int cc_plan_splits(int64_t n, int64_t m, int32_t c, int num_sms, int max_pool, int64_t* chunk);

cudaError_t launch_finalize(const FinalizeArgs& a, cudaStream_t st, int* launches);
int finalize_max_pool();   // largest S*c one finalize pass handles

// Whitening for the Mahalanobis distance (knn_whiten.cu): Y = X L for rows
// of X (rows x d), L the d x d lower-triangular Cholesky factor of the inverse
// covariance (row-major float32); compensated accumulation, one rounding.
size_t whiten_smem_bytes(int32_t d);
cudaError_t launch_whiten(const float* X, int64_t rows, int32_t d, const float* L, float* Y,
                          cudaStream_t st, int* launches);

// One bounded mbarrier wait that nothing completes: raises *error_flag after
// limit_ns (the failure path of every device-side wait, exercised on purpose).
cudaError_t launch_wait_probe(int32_t* error_flag, uint64_t limit_ns, cudaStream_t st);
// One tile of bf16 MMA steps (knn_selftest_mma): D[128][256] = the first `steps`
// (1 to 4) steps of 16 columns of A[128][64] times B[256][64], one after another.
cudaError_t launch_mma_probe(const float* A, const float* B, int32_t steps, float* D,
                             int32_t* error_flag, cudaStream_t st);

// Self-join rows: the n x (k+1) result of searching R against itself, minus
// each row's own index (or its last entry), into n x k outputs.
cudaError_t launch_drop_self(const float* din, const int32_t* iin, int64_t n, int32_t k, float* dout,
                             int32_t* iout, cudaStream_t st, int* launches);   // chained

// Exact float64 pass for the queued queries.  scratch holds slots*m doubles;
// done holds `slots` counters, zeroed by the finalize that runs before (its
// FinalizeArgs::fb_done / fb_slots).  The first slots/2 queued queries have
// their float32 key pass spread over the GPU; the rest take one CTA each.
cudaError_t launch_fallback(const FinalizeArgs& a, double* scratch, int32_t slots, int32_t* done,
                            cudaStream_t st, int* launches);

// ---- tensor-core path (knn_tc.cu) -----------------------------------------

// kPair: float32 rows as pairs of bf16 words (the float32 search's own filter).
enum LowPrecision : int { kTF32 = 1, kBF16 = 2, kPair = 3 };

// Row length (elements) of the low-precision operand copies: d coordinates,
// four augmentation words (norm halves, threshold halves), zero padded to a
// whole number of 32-byte MMA K steps.
int tc_padded_dim(int32_t d, int prec);

// Launch plan of the pilot and filter passes for one search.
struct TcPlan {
    int32_t mt;          // 128-query tiles per CTA (1)
    int32_t kb;          // 128-byte K blocks per operand row (the last one maybe in part)
    int32_t ksteps;      // 32-byte MMA K steps that carry data
    int32_t rb;          // references per tile (MMA N = 256)
    int32_t kbs;         // K blocks per TMA stage (kb, or 1 for long rows)
    int32_t groups;      // hit lists per (query, split): one per epilogue column group
    int32_t stages;      // reference-stage ring depth
    int32_t S;           // reference splits
    int64_t chunk;       // references per split (multiple of rb)
    int32_t stride;      // pilot samples every stride-th stage
    int32_t spt;         // pilot tile slots per split
    int32_t G;           // pilot group maxima per query
    int32_t gsize;       // references per pilot group (32, or 16 / 8 when every tile is sampled)
    int32_t cprime;      // order statistic of the group maxima used as threshold
    int32_t pilot;       // 0: no pilot, every reference is appended
    int32_t cap;         // list capacity per (query, split, column group)
    int32_t raw;         // filter stages hit values as float32 (else 16-bit codes)
    int32_t hs;          // operand pairs: K steps of the upper words
    int64_t tiles;       // operand pairs: reference tiles of the set
    int64_t m_set;       // operand pairs: references of the set
    size_t smem_filter;
    bool chain;          // launch in the search's chain (launch_chained)
};
// smem_limit: the dynamic shared memory an item may use (the persistent batch
// kernel keeps some for itself); force_chunk > 0: split the references into
// pieces of about this length (rounded to whole tiles) instead of choosing the
// split count by how full the last wave of CTAs is.
TcPlan tc_plan(int64_t n, int64_t m, int32_t d, int32_t kp, int prec, int32_t c, int num_sms,
               size_t smem_limit = 232448, int64_t force_chunk = 0);

// Per-query scale of the 16-bit hit codes (a power of two B > |acc|): the
// largest squared reference norm (float bits, set by launch_prepare_ref) and
// the queries' B, set by launch_tc_threshold once t is known, or by
// launch_prepare_query for t = 0 when qscale is passed there (no threshold).
struct HitScale {
    const uint32_t* rmax2;
    float* qscale;   // [n]
};

// Operand pairs (rows of up to kPairMaxD coordinates): both copies of a search
// in one launch, the queries' squared norms (less twice their remainders), and
// its two queue counters cleared.  R_lp holds whole tiles, pair_tiles(m) of them.
constexpr int64_t kPairTile = 256;
inline int64_t pair_tiles(int64_t m) { return (m + kPairTile - 1) / kPairTile; }
bool pair_rows_fit(int32_t d);
// How many candidates the filter must keep for the k nearest of m references
// to be certified (more than m: hopeless).
int64_t pair_candidates(int64_t m, int32_t d, int32_t k);
cudaError_t launch_prepare_pair(const float* R, int64_t m, const float* centre, const float* Q,
                                int64_t n, int32_t d, int32_t kp, void* R_lp, void* Q_lp,
                                float* qnorm, int32_t* count0, int32_t* count1, cudaStream_t st,
                                int* launches);
// The centre [d] that the pairs' coordinates are taken relative to: once per
// reference set.
cudaError_t launch_centre(const float* R, int64_t m, int32_t d, float* centre, cudaStream_t st,
                          int* launches);

// Reference copy [r, -||r||^2/2 (hi, lo), 1, 1, 0..], float32 norms and their maximum.
cudaError_t launch_prepare_ref(const float* R, int64_t m, int32_t d, int32_t kp, int prec,
                               void* R_lp, float* norms, uint32_t* rmax2, cudaStream_t st,
                               int* launches);
// Query copy [q, 1, 1, 0, 0, 0..] (threshold words filled by the threshold pass);
// when Q_copy is given, the float32 rows are also written there (Q may then be
// host memory the GPU reads directly).  *clear is set to zero.
cudaError_t launch_prepare_query(const float* Q, int64_t n, int32_t d, int32_t kp, int prec,
                                 void* Q_lp, const HitScale& qs, float* Q_copy, int32_t* clear,
                                 cudaStream_t st, int* launches);
cudaError_t launch_tc_pilot(const TcPlan& p, const void* Q_lp, int64_t n, const void* R_lp,
                            int64_t m, int32_t kp, int prec, uint32_t* gmax, int32_t* error_flag,
                            cudaStream_t st, int* launches);
cudaError_t launch_tc_threshold(const TcPlan& p, const uint32_t* gmax, int64_t n, int32_t d,
                                int32_t kp, int prec, void* Q_lp, const HitScale& qs,
                                cudaStream_t st, int* launches);
cudaError_t launch_tc_filter(const TcPlan& p, const void* Q_lp, int64_t n, const void* R_lp,
                             int64_t m, int32_t kp, int prec, uint64_t* lists, int32_t* counts,
                             const float* qscale, int32_t* error_flag, cudaStream_t st,
                             int* launches);

}  // namespace knn
