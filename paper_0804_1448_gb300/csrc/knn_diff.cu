// knn_diff.cu -- Manhattan and Chebyshev searches on CUDA cores: pilot,
// threshold and filter, as the tensor-core forms run them, on distances from
// float32 coordinate differences.
//
// The distances are those of knn_cc.cu, coordinate 0 first, one rounding per
// operation.  What differs is the selection: knn_cc.cu keeps a heap per query
// and reference split, filled anew in every split by one thread per query, and
// passes every tile of distances through shared memory to it -- at n = 3001,
// m = 30011, d = 33, k = 10 more than half of the 0.73 ms.  Here a first pass over a sample
// of the references gives every query a threshold that at least c' of them
// meet, and the main pass compares the distances in registers with it (one
// three-input minimum per two of them) and appends the few that pass to the
// query's list: 0.34 ms, and 2.45 ms in place of 2.88 at n = m = 19200, d = 80,
// where the differences' additions set the pace (two per coordinate, 45 of the
// 64 coordinates a clock that an SM's float pipes could add).  Two-lane
// subtractions, which save issue slots but run on one of the two pipes, were
// slower (2.93 against 2.88 ms in the heap form).  The finalize takes the lists, and certifies each answer: a
// reference that was not listed is farther than the threshold.
//
// A CTA owns ROWS queries, whose coordinates stay in shared memory, and streams
// tiles of kTM references in stages of kDK coordinates, copied asynchronously
// kRing - 1 stages ahead.  Reference i of tile g is row i T + g of the set (T
// tiles in all): every tile is an evenly spaced sample of it, so a set stored
// in some order gives the pilot's sample and the splits the same shares as a
// shuffled one.
#include <algorithm>
#include <cmath>

#include "tc_device.cuh"

namespace knn {
namespace {

constexpr int kThreads = 256;
constexpr int kDK = 16;    // coordinates per stage
constexpr int kTM = 128;   // references per tile
constexpr int kRing = 4;   // stages in shared memory
constexpr int kRST = kTM + 4;
constexpr int kGroupsPerTile = kTM / 32;

// TY x TX threads, each an RR (queries) x CN (references) micro-tile whose
// references come in groups of G consecutive columns; MINB CTAs per SM.
template <int ROWS>
struct Shape;
template <>
struct Shape<128> {
    static constexpr int TY = 16, TX = 16, RR = 8, CN = 8, G = 4, MINB = 2;
};
template <>
struct Shape<64> {
    static constexpr int TY = 16, TX = 16, RR = 4, CN = 8, G = 4, MINB = 3;
};
template <>
struct Shape<16> {
    static constexpr int TY = 4, TX = 64, RR = 4, CN = 2, G = 2, MINB = 3;
};

__host__ __device__ constexpr int padded_d(int d) { return (d + 3) / 4 * 4; }

template <int ROWS>
constexpr size_t smem_bytes(int d) {
    return sizeof(float) * (static_cast<size_t>(padded_d(d)) * (ROWS + 4) +
                            static_cast<size_t>(kRing) * kDK * kRST + ROWS) +
           sizeof(int) * ROWS;
}

// Copy 4 bytes, or store zero when !ok.
__device__ __forceinline__ void cp_async4(float* smem, const float* gmem, bool ok) {
    const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(s), "l"(gmem), "r"(ok ? 4 : 0)
                 : "memory");
}

__device__ __forceinline__ float max3_abs(float x, float y, float z) {
    float r;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(x), "f"(y), "f"(z));
    return r;
}
__device__ __forceinline__ float min3(float x, float y, float z) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(x), "f"(y), "f"(z));
    return r;
}

struct DiffArgs {
    const float* Q;
    const float* R;
    int64_t n, m;
    int32_t d;
    int32_t tiles;        // of the whole set (the row stride of a tile)
    int32_t tps;          // tiles per split
    int32_t S;
    int32_t stride;       // pilot: every stride-th tile
    int32_t spt;          // pilot: sampled-tile slots per split
    int32_t G;            // pilot: group maxima per query (S * spt * kGroupsPerTile)
    uint32_t* gmax;       // pilot: [n][G] order-mapped -distance, 0 = no group
    const float* thr;     // filter: [n]
    uint64_t* lists;      // filter: [n][S][cap], keys (distance bits, index)
    int32_t* counts;      // filter: [n][S] (may exceed cap: overflow)
    int32_t cap;
};

template <int METRIC, int ROWS, bool PILOT>
__global__ void __launch_bounds__(kThreads, Shape<ROWS>::MINB) diff_kernel(DiffArgs a) {
    using S = Shape<ROWS>;
    static_assert(S::TY * S::TX == kThreads && S::TY * S::RR == ROWS && S::TX * S::CN == kTM, "shape");
    constexpr int QST = ROWS + 4;
    constexpr int RPT = kTM * kDK / kThreads;
    constexpr float kInf = __builtin_huge_valf();
    extern __shared__ __align__(16) float sm[];
    chain_begin();
    const int d = a.d, dp = padded_d(d);
    float* Qs = sm;                                    // [dp][QST]
    float* Rs = Qs + static_cast<size_t>(dp) * QST;    // [kRing][kDK][kRST]
    float* thr = Rs + kRing * kDK * kRST;              // [ROWS]
    int* cnt = reinterpret_cast<int*>(thr + ROWS);     // [ROWS]

    const int tid = threadIdx.x;
    const int ty = tid / S::TX, tx = tid % S::TX;
    const int64_t qbase = static_cast<int64_t>(blockIdx.x) * ROWS;
    const int split = blockIdx.y;
    const int g0 = split * a.tps;
    const int stride = PILOT ? a.stride : 1;
    const int tiles_here = min(a.tps, a.tiles - g0);
    const int nt = (tiles_here + stride - 1) / stride;
    const int stages = (d + kDK - 1) / kDK;
    const int steps = nt * stages;

    // stage h: coordinates 16 (h % stages) .. + 15 of tile h / stages
    const int ft = tid % kDK, fr = tid / kDK;   // this thread's coordinate and first row
    auto issue = [&](int h) {
        if (h < steps) {
            const int64_t g = g0 + static_cast<int64_t>(h / stages) * stride;
            const int t = (h % stages) * kDK + ft;
            float* dst = Rs + (h % kRing) * (kDK * kRST) + ft * kRST;
#pragma unroll
            for (int u = 0; u < RPT; ++u) {
                const int r = fr + u * (kThreads / kDK);
                const int64_t j = static_cast<int64_t>(r) * a.tiles + g;
                const bool ok = j < a.m && t < d;
                cp_async4(dst + r, a.R + (ok ? j * d + t : 0), ok);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
#pragma unroll
    for (int h = 0; h < kRing - 1; ++h) issue(h);
    for (int e = tid; e < ROWS * dp; e += kThreads) {
        const int r = e / dp, t = e % dp;
        const int64_t q = qbase + r;
        Qs[t * QST + r] = (q < a.n && t < d) ? a.Q[q * d + t] : 0.f;
    }
    if (!PILOT) {
        for (int r = tid; r < ROWS; r += kThreads) {
            thr[r] = qbase + r < a.n ? a.thr[qbase + r] : -1.f;   // distances are >= 0: none pass
            cnt[r] = 0;
        }
    }

    float acc[S::RR][S::CN];
#pragma unroll
    for (int i = 0; i < S::RR; ++i)
#pragma unroll
        for (int j = 0; j < S::CN; ++j) acc[i][j] = 0.f;

    for (int h = 0; h < steps; ++h) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing - 2) : "memory");
        __syncthreads();   // stage h is in place, and stage h - 1 is read
        issue(h + kRing - 1);
        const int dbase = (h % stages) * kDK;
        const float* qs = Qs + static_cast<size_t>(dbase) * QST + ty * S::RR;
        const float* rs = Rs + (h % kRing) * (kDK * kRST) + tx * S::G;
        auto load_q = [&](float (&qv)[S::RR], int t) {
#pragma unroll
            for (int i = 0; i < S::RR; i += 4) {
                const float4 q4 = *reinterpret_cast<const float4*>(qs + t * QST + i);
                qv[i] = q4.x; qv[i + 1] = q4.y; qv[i + 2] = q4.z; qv[i + 3] = q4.w;
            }
        };
        auto load_r = [&](float (&rv)[S::CN], int t) {
#pragma unroll
            for (int g = 0; g < S::CN / S::G; ++g) {
                const float* src = rs + t * kRST + g * S::TX * S::G;
                if constexpr (S::G == 4) {
                    const float4 r4 = *reinterpret_cast<const float4*>(src);
                    rv[g * 4 + 0] = r4.x; rv[g * 4 + 1] = r4.y;
                    rv[g * 4 + 2] = r4.z; rv[g * 4 + 3] = r4.w;
                } else {
                    const float2 r2 = *reinterpret_cast<const float2*>(src);
                    rv[g * 2 + 0] = r2.x; rv[g * 2 + 1] = r2.y;
                }
            }
        };
        auto four = [&](int t0) {
            if constexpr (METRIC == kLinf) {
#pragma unroll
                for (int t = t0; t < t0 + 4; t += 2) {
                    float qa[S::RR], qb[S::RR], ra[S::CN], rb[S::CN];
                    load_q(qa, t);
                    load_q(qb, t + 1);
                    load_r(ra, t);
                    load_r(rb, t + 1);
#pragma unroll
                    for (int i = 0; i < S::RR; ++i)
#pragma unroll
                        for (int j = 0; j < S::CN; ++j)
                            acc[i][j] = max3_abs(acc[i][j], qa[i] - ra[j], qb[i] - rb[j]);
                }
            } else {
#pragma unroll
                for (int t = t0; t < t0 + 4; ++t) {
                    float qv[S::RR], rv[S::CN];
                    load_q(qv, t);
                    load_r(rv, t);
#pragma unroll
                    for (int i = 0; i < S::RR; ++i)
#pragma unroll
                        for (int j = 0; j < S::CN; ++j) acc[i][j] += fabsf(qv[i] - rv[j]);
                }
            }
        };
        // whole stages unrolled; a row's last one as many coordinates as it has,
        // in fours (both operands are zero beyond d)
        if (d - dbase >= kDK) {
#pragma unroll
            for (int t0 = 0; t0 < kDK; t0 += 4) four(t0);
        } else {
            for (int t0 = 0; t0 < d - dbase; t0 += 4) four(t0);
        }
        if (h % stages != stages - 1) continue;

        // a tile is complete
        const int slot = h / stages;
        const int64_t g = g0 + static_cast<int64_t>(slot) * stride;
        auto col_of = [&](int j) { return (j / S::G) * (S::TX * S::G) + tx * S::G + j % S::G; };
        const int64_t last = (a.m - 1 - g) / a.tiles;   // columns beyond it hold no reference
        if (last < kTM - 1) {
#pragma unroll
            for (int j = 0; j < S::CN; ++j)
                if (col_of(j) > last)
#pragma unroll
                    for (int i = 0; i < S::RR; ++i) acc[i][j] = kInf;
        }
        float least[S::RR];
#pragma unroll
        for (int i = 0; i < S::RR; ++i) {
            float x = acc[i][0];
#pragma unroll
            for (int j = 1; j + 1 < S::CN; j += 2) x = min3(x, acc[i][j], acc[i][j + 1]);
            least[i] = fminf(x, acc[i][S::CN - 1]);
        }
        if (PILOT) {
            // groups of 32 references: the columns of 32 / CN neighbouring threads
            constexpr int LPG = 32 / S::CN;
#pragma unroll
            for (int i = 0; i < S::RR; ++i) {
                float x = least[i];
#pragma unroll
                for (int o = LPG / 2; o > 0; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
                const int64_t q = qbase + ty * S::RR + i;
                if (tx % LPG == 0 && q < a.n)
                    a.gmax[q * a.G + (static_cast<int64_t>(split) * a.spt + slot) * kGroupsPerTile +
                           tx / LPG] = x < kInf ? ord_f32(-x) : 0u;
            }
        } else {
#pragma unroll
            for (int i = 0; i < S::RR; ++i) {
                const int row = ty * S::RR + i;
                const float lim = thr[row];
                if (least[i] <= lim) {
                    uint64_t* list = a.lists + ((qbase + row) * a.S + split) * static_cast<int64_t>(a.cap);
#pragma unroll
                    for (int j = 0; j < S::CN; ++j) {
                        if (acc[i][j] <= lim && acc[i][j] < kInf) {
                            const int at = atomicAdd(&cnt[row], 1);
                            if (at < a.cap)
                                list[at] = (static_cast<uint64_t>(__float_as_uint(acc[i][j])) << 32) |
                                           static_cast<uint32_t>(col_of(j) * static_cast<int64_t>(a.tiles) + g);
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < S::RR; ++i)
#pragma unroll
            for (int j = 0; j < S::CN; ++j) acc[i][j] = 0.f;
    }
    if (PILOT) {
        // the group slots of tiles this split does not have
        for (int e = tid; e < ROWS * (a.spt - nt) * kGroupsPerTile; e += kThreads) {
            const int row = e / ((a.spt - nt) * kGroupsPerTile), s = e % ((a.spt - nt) * kGroupsPerTile);
            if (qbase + row < a.n)
                a.gmax[(qbase + row) * a.G +
                       (static_cast<int64_t>(split) * a.spt + nt) * kGroupsPerTile + s] = 0u;
        }
    } else {
        __syncthreads();
        for (int r = tid; r < ROWS; r += kThreads)
            if (qbase + r < a.n) a.counts[(qbase + r) * a.S + split] = cnt[r];
    }
}

// One warp per query: the distance that at least cprime sampled references
// meet.  It also clears the search's two queue counters.
template <int VPL>
__global__ void diff_threshold_kernel(const uint32_t* __restrict__ gmax, int64_t n, int32_t G,
                                      int32_t cprime, float* __restrict__ thr,
                                      int32_t* __restrict__ count0, int32_t* __restrict__ count1) {
    chain_begin();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *count0 = 0;
        *count1 = 0;
    }
    const int64_t q = static_cast<int64_t>(blockIdx.x) * (blockDim.x / 32) + threadIdx.x / 32;
    if (q >= n) return;
    const int lane = threadIdx.x % 32;
    const float t = -unord_f32(order_statistic<VPL>(gmax + q * G, G, cprime, lane));
    if (lane == 0) thr[q] = t;
}

template <int METRIC, int ROWS>
cudaError_t launch_shape(const DiffArgs& a, bool pilot, bool chain, cudaStream_t st) {
    const size_t smem = smem_bytes<ROWS>(a.d);
    const dim3 grid(static_cast<unsigned>((a.n + ROWS - 1) / ROWS), static_cast<unsigned>(a.S));
    cudaError_t err = pilot ? allow_smem<diff_kernel<METRIC, ROWS, true>>(smem)
                            : allow_smem<diff_kernel<METRIC, ROWS, false>>(smem);
    if (err != cudaSuccess) return err;
    if (!pilot) return launch_chained(chain, diff_kernel<METRIC, ROWS, false>, grid, dim3(kThreads), smem, st, a);
    diff_kernel<METRIC, ROWS, true><<<grid, kThreads, smem, st>>>(a);   // a search's first kernel
    return cudaGetLastError();
}

template <int METRIC>
cudaError_t launch_metric(const DiffArgs& a, int rows, bool pilot, bool chain, cudaStream_t st) {
    if (rows == 128) return launch_shape<METRIC, 128>(a, pilot, chain, st);
    if (rows == 64) return launch_shape<METRIC, 64>(a, pilot, chain, st);
    return launch_shape<METRIC, 16>(a, pilot, chain, st);
}

DiffArgs base_args(const DiffPlan& p, const float* Q, int64_t n, const float* R, int64_t m, int32_t d) {
    DiffArgs a{};
    a.Q = Q;
    a.R = R;
    a.n = n;
    a.m = m;
    a.d = d;
    a.tiles = p.tiles;
    a.tps = p.tps;
    a.S = p.S;
    a.stride = p.stride;
    a.spt = p.spt;
    a.G = p.G;
    a.cap = p.cap;
    return a;
}

}  // namespace

DiffPlan diff_plan(int64_t n, int64_t m, int32_t d, int32_t c, int num_sms) {
    DiffPlan p{};
    // the queries' coordinates of two 128-row CTAs fit an SM up to d = 128
    if (d > 128 || m > (1ll << 31) - 256) return p;
    p.rows = n > 64 ? 128 : (n > 16 ? 64 : 16);
    const int per_sm = p.rows == 128 ? Shape<128>::MINB : Shape<64>::MINB;
    p.tiles = static_cast<int32_t>((m + kTM - 1) / kTM);
    const int64_t qtiles = (n + p.rows - 1) / p.rows;
    const int64_t slots = static_cast<int64_t>(per_sm) * num_sms;
    // splits: CTAs run in waves of `slots`, each wave as long as its tiles plus
    // about one for its start; the fewest splits within 2% of the shortest
    auto tps_of = [&](int64_t s) { return (p.tiles + s - 1) / s; };
    auto cost = [&](int64_t s) {
        const int64_t ctas = qtiles * ((p.tiles + tps_of(s) - 1) / tps_of(s));
        const int64_t sms = num_sms;
        const int64_t rounds = (ctas / slots) * per_sm + (ctas % slots + sms - 1) / sms;
        return static_cast<double>(std::max<int64_t>(rounds, per_sm)) * static_cast<double>(tps_of(s) + 1);
    };
    const int64_t s_cap = std::max<int64_t>(1, std::min<int64_t>(512, p.tiles / 4));
    double best = cost(1);
    for (int64_t s = 2; s <= s_cap; ++s) best = std::min(best, cost(s));
    int64_t S = 1;
    while (S < s_cap && cost(S) > 1.02 * best) ++S;
    p.tps = static_cast<int32_t>(tps_of(S));
    p.S = static_cast<int32_t>((p.tiles + p.tps - 1) / p.tps);
    // pilot: one tile in 32 (the CUDA cores pay for it in full, the extra hits
    // cost little), at most about 1024 groups per query, denser until the order
    // statistic has groups to spare (the c' of the tensor-core pilot)
    int stride = 32;
    while (static_cast<int64_t>(p.tiles) * kGroupsPerTile / stride > 1024) stride *= 2;
    for (;; stride /= 2) {
        p.stride = stride;
        // its own split of the sampled tiles: one CTA per sampled tile while all
        // of them fit the GPU at once
        const int64_t sampled = (p.tiles + stride - 1) / stride;
        p.spt = static_cast<int32_t>(std::min(sampled, (qtiles * sampled + slots - 1) / slots));
        p.pS = static_cast<int32_t>((sampled + p.spt - 1) / p.spt);
        p.G = p.pS * p.spt * kGroupsPerTile;
        const double lambda = static_cast<double>(c) * static_cast<double>(sampled) / p.tiles;
        p.cprime = sampled == p.tiles ? c : static_cast<int>(std::ceil(lambda + 4.0 * std::sqrt(lambda) + 4.0));
        const int64_t groups = sampled * kGroupsPerTile;
        p.pilot = groups >= p.cprime + 8 && p.G <= 2048;
        if (p.pilot) {
            // as in tc_plan: 2.5 times the mean per list plus 48
            const double pg = static_cast<double>(p.cprime) / static_cast<double>(groups);
            const double f = 1.0 - std::pow(1.0 - pg, 1.0 / 32.0);
            const int64_t cap = static_cast<int64_t>(std::ceil(2.5 * static_cast<double>(m) * f / p.S)) + 48;
            p.cap = static_cast<int32_t>(std::min<int64_t>((cap + 31) / 32 * 32, static_cast<int64_t>(p.tps) * kTM));
        }
        if (p.pilot || stride == 1 || p.G > 2048) break;
    }
    return p;
}

cudaError_t launch_diff_pilot(const DiffPlan& p, const float* Q, int64_t n, const float* R, int64_t m,
                              int32_t d, int32_t metric, uint32_t* gmax, cudaStream_t st, int* launches) {
    DiffArgs a = base_args(p, Q, n, R, m, d);
    a.tps = p.spt * p.stride;
    a.S = p.pS;
    a.gmax = gmax;
    if (launches) ++*launches;
    return metric == kL1 ? launch_metric<kL1>(a, p.rows, true, p.chain, st) : launch_metric<kLinf>(a, p.rows, true, p.chain, st);
}

cudaError_t launch_diff_threshold(const DiffPlan& p, const uint32_t* gmax, int64_t n, float* thr,
                                  int32_t* count0, int32_t* count1, cudaStream_t st, int* launches) {
    const unsigned grid = static_cast<unsigned>((n + 7) / 8);
    const int vpl = (p.G + 31) / 32;
    if (launches) ++*launches;
    if (vpl > 64) return cudaErrorInvalidValue;
    return launch_chained(p.chain, vpl <= 4    ? diff_threshold_kernel<4>
                          : vpl <= 16 ? diff_threshold_kernel<16>
                                      : diff_threshold_kernel<64>,
                          dim3(grid), dim3(256), 0, st, gmax, n, p.G, p.cprime, thr, count0, count1);
}

cudaError_t launch_diff_filter(const DiffPlan& p, const float* Q, int64_t n, const float* R, int64_t m,
                               int32_t d, int32_t metric, const float* thr, uint64_t* lists,
                               int32_t* counts, cudaStream_t st, int* launches) {
    DiffArgs a = base_args(p, Q, n, R, m, d);
    a.thr = thr;
    a.lists = lists;
    a.counts = counts;
    if (launches) ++*launches;
    return metric == kL1 ? launch_metric<kL1>(a, p.rows, false, p.chain, st) : launch_metric<kLinf>(a, p.rows, false, p.chain, st);
}

}  // namespace knn
