// Vocabulary-wide tail of a step: temperature softmax statistics, the accept / reject scan,
// residual renormalise-and-resample or bonus draw, and the draft's "sample from q, export q".
// (Section "Speculative Sampling", Figure 2: the target model passes or refuses each draft token in
// turn and generates one token itself.)  No host round-trip: everything a decision
// needs stays on the device.
//
// A sequence's rows are worked on by a thread-block cluster of kTailCluster CTAs of 32 warps (one SM alone is issue-
// and latency-bound on a 50 K-entry row).  Warp g of the cluster owns the contiguous piece [g * per, (g + 1) * per)
// of every row and its lanes take consecutive entries of it, kStep / 32 loads in flight per lane (1, 4 or 8: what the
// vocabulary fills); what the warps find meets once in shared memory and once, through distributed shared memory, across
// the cluster, always combined in the same order.  What bounds it is instruction issue on the cluster's few SMs and that
// chain of exchanges, not the bytes: hence one kernel per verification, which carries the statistics of ALL rows of a
// sequence through one exchange (one sequence, 5 rows of 32000: 20.8 us a call back to back with a cluster per row and a
// second launch for the draw, 12.3 so), as long as the rows that follow one another cost less than a second launch.
#pragma once
#include <cooperative_groups.h>

#include "common.cuh"

namespace ssd {

namespace cg = cooperative_groups;

constexpr int kTailThreads = 1024;
constexpr int kTailWarps = kTailThreads / 32;
constexpr int kTailCluster = 8;
constexpr int kTailMaxRows = kMaxRowsPerSeq;

struct RowStat {
    float mx;      // max logit of the row
    float z;       // sum exp((l - mx) / T)
    int32_t amax;  // argmax (lowest index among maxima)
    int32_t pad;
};

// p_j of a row from its statistics; the one place this is computed, so the rows exported for
// inspection are bit-identical to the rows the decisions use.
__device__ __forceinline__ float prob_of(float logit, const RowStat &st, float inv_t, int j) {
    if (inv_t == 0.f) return j == st.amax ? 1.f : 0.f;  // greedy: one-hot at the argmax
    return expf((logit - st.mx) * inv_t) / st.z;
}

// Restriction of a row to its most probable tokens (top-k, then top-p on what top-k kept): token j stays iff
// its probability is >= thr, and the kept ones are divided by their mass.  mass == 0 means "no restriction".
struct RowFilter {
    float thr;
    float mass;
};
__device__ __forceinline__ float prob_f(float logit, const RowStat &st, const RowFilter &f, float inv_t, int j) {
    const float pr = prob_of(logit, st, inv_t, j);
    if (f.mass == 0.f || inv_t == 0.f) return pr;  // (a one-hot row is its own restriction)
    return pr >= f.thr ? pr / f.mass : 0.f;
}

// Warp `g` of `pieces` warps owns this piece [lo, hi) of a row of V entries: whole lane rows.
__device__ __forceinline__ void row_piece(int V, int pieces, int g, int &lo, int &hi) {
    const int per = (((V + pieces - 1) / pieces) + 31) & ~31;
    lo = min(V, g * per);
    hi = min(V, lo + per);
}
__device__ __forceinline__ void tail_piece(int V, int rank, int &lo, int &hi) {
    row_piece(V, kTailCluster * kTailWarps, rank * kTailWarps + (int)(threadIdx.x >> 5), lo, hi);
}
// Entries base + lane, base + lane + 32, ... of the piece; `fill` where it has ended.
template <int IT>
__device__ __forceinline__ void tail_load(const float *row, int base, int hi, float fill, float (&l)[IT]) {
    const int j = base + (int)(threadIdx.x & 31);
    if (base + 32 * IT <= hi) {
#pragma unroll
        for (int u = 0; u < IT; ++u) l[u] = __ldcg(row + j + 32 * u);
    } else {
#pragma unroll
        for (int u = 0; u < IT; ++u) l[u] = j + 32 * u < hi ? __ldcg(row + j + 32 * u) : fill;
    }
}

// (max, argmax, sum of exp relative to the max) of a part of a row
struct PartStat {
    float mx;
    int am;
    double s;
};
// The statistics of W parts held by the W lanes of a group (W = 32: the warps of a CTA, else the CTAs of a cluster).
template <int W>
__device__ __forceinline__ PartStat join_parts(PartStat a, float inv_t) {
    float m = a.mx;
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    int am = a.mx == m ? a.am : 0x7fffffff;
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) am = min(am, __shfl_xor_sync(0xffffffffu, am, o));
    double s = 0.0;
    if (inv_t != 0.f) {
        s = a.mx > -INFINITY ? a.s * (double)expf((a.mx - m) * inv_t) : a.s;  // (nothing, or NaN)
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    PartStat r;
    r.mx = m;
    r.am = am;
    r.s = s;
    return r;
}
__device__ __forceinline__ RowStat row_stat(const PartStat &t) {
    RowStat st;
    st.mx = t.mx;
    st.z = (float)t.s;
    st.amax = t.am;
    st.pad = 0;
    return st;
}

struct StatSmem {
    PartStat warp[kTailMaxRows][kTailWarps];  // of this CTA's warps
    PartStat cta[kTailMaxRows];               // of this CTA, read by the others
    RowStat row[kTailMaxRows];
};

// Statistics of `rows` rows (row pitch V) by the whole cluster, left in ss->row of every CTA.  Where a piece fits one
// step (hi - lo <= 32 IT) `l` returns its entries of the last row.
template <int IT>
__device__ __forceinline__ void cluster_stats(const float *logits, int rows, int V, float inv_t, StatSmem *ss,
                                              cg::cluster_group &cl, float (&l)[IT]) {
    constexpr int kStep = 32 * IT;
    const int rank = (int)cl.block_rank(), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int lo, hi;
    tail_piece(V, rank, lo, hi);
    const bool one = hi - lo <= kStep;
    float nx[IT];
    tail_load<IT>(logits, lo, hi, -INFINITY, nx);
    for (int r = 0; r < rows; ++r) {
        const float *lg = logits + (size_t)r * V;
#pragma unroll
        for (int u = 0; u < IT; ++u) l[u] = nx[u];
        if (r + 1 < rows) tail_load<IT>(lg + V, lo, hi, -INFINITY, nx);  // the next row, under this one's arithmetic
        float mx = -INFINITY;
        int at = lo;  // the step that the lane's first maximum lies in
        for (int b = lo;;) {
            float m = l[0];
#pragma unroll
            for (int u = 1; u < IT; ++u) m = fmaxf(m, l[u]);
            if (m > mx) { mx = m; at = b; }
            b += kStep;
            if (b >= hi) break;
            tail_load<IT>(lg, b, hi, -INFINITY, l);
        }
        const float m = warp_max_redux(mx);
        int am = 0x7fffffff;
        if (mx == m && m > -INFINITY) {
            float x[IT];
#pragma unroll
            for (int u = 0; u < IT; ++u) x[u] = l[u];
            if (!one) tail_load<IT>(lg, at, hi, -INFINITY, x);
#pragma unroll
            for (int u = IT - 1; u >= 0; --u)
                if (x[u] == m) am = at + 32 * u + lane;  // the lowest index
        }
        am = __reduce_min_sync(0xffffffffu, am);
        double s = 0.0;
        if (inv_t != 0.f) {
            float part = 0.f;
            if (!one) tail_load<IT>(lg, lo, hi, -INFINITY, l);
            const float ref = m > -INFINITY ? m : 0.f;  // (a piece of NaNs has no maximum, but they reach the row's sum)
            for (int b = lo;;) {
#pragma unroll
                for (int u = 0; u < IT; ++u) part += expf((l[u] - ref) * inv_t);  // exp(-inf) = 0
                b += kStep;
                if (b >= hi) break;
                tail_load<IT>(lg, b, hi, -INFINITY, l);
            }
            s = warp_sum((double)part);
        }
        if (lane == 0) {
            PartStat t;
            t.mx = m;
            t.am = am;
            t.s = s;
            ss->warp[r][warp] = t;
        }
    }
    __syncthreads();
    for (int r = warp; r < rows; r += kTailWarps) {
        const PartStat t = join_parts<32>(ss->warp[r][lane], inv_t);
        if (lane == 0) ss->cta[r] = t;
    }
    cl.sync();
    for (int i = threadIdx.x; i < ((rows * kTailCluster + 31) & ~31); i += kTailThreads) {
        const int r = min(i / kTailCluster, rows - 1);
        const PartStat t = join_parts<kTailCluster>(*cl.map_shared_rank(&ss->cta[r], i % kTailCluster), inv_t);
        if (i % kTailCluster == 0 && i / kTailCluster < rows) ss->row[r] = row_stat(t);
    }
    __syncthreads();
}

// ---- top-k / top-p ---------------------------------------------------------------------------------
// The threshold of a restriction: the largest probability value t such that the tokens with p >= t number at least top_k,
// or - of those that top-k kept - weigh at least top_p of their mass; if no t reaches it, the smallest value there is.
// Tokens equal to the threshold all stay.
//
// Probabilities are >= 0, so their fp32 bit patterns order like the values.  A token's key is its pattern's distance
// below the largest one's.  First pass: 1024 bins of 2^18 keys, 32 to a factor of two, so that a softmax row spreads over
// hundreds of them (bins of the pattern's top eight bits put a whole row into a dozen: the histogram's atomic operations
// queue up on a few addresses); the bins are walked from the top, and two or three more passes refine the one that the
// target falls into.  A bin holds a count and the tokens' mass in units of 2^-62, in three native 32-bit words: integer
// sums do not depend on their order and are finer than an fp64 running sum.  A thread joins consecutive tokens of one bin
// before it touches the histogram (a row of equal values, or the tail of a peaked one, is one bin).  The first histogram
// is kept: with the tokens that top-k took off its bin put aside, it is top-p's first pass too.
//
// A row is a cluster of TWO CTAs, its probabilities computed once and kept in their shared memory (up to kFilterCache of
// them each): the histograms of two CTAs are joined with three remote loads per thread, where eight CTAs took 9 us per
// pass for it and left most of 48 rows waiting for SMs.
// 8 sequences x 6 rows x 50304 entries, top-k 50 and top-p 0.9, whole call: 565 us with byte-wide bins and fp64 atomics on
// eight CTAs, 193 with these bins on eight, 53 on two.
constexpr int kBins = 1024;
constexpr int kFilterCluster = 2;
constexpr int kFilterCache = 44 * 1024;     // probabilities a CTA keeps (176 KB)
constexpr int kFilterBatch = 8;
constexpr double kMassUnit = 4611686018427387904.0;  // 2^62
// Up to kPickK tokens the threshold is found among candidates instead of by histograms over the row: the k-th largest of a CTA's
// 1024 threads' maxima is a lower bound of the k-th largest logit, and some 2 k tokens of the two CTAs reach it (at k = 96 about
// 195 of the 256 that there is room for; beyond 96 ever more rows would not fit).  A pass of the histograms computes a
// probability, its mass in fp64 and a bin for every entry of the row, 4-10 us each; picking compares every entry once.
// Same counts and masses of the same tokens (integers, so in any order): the same bits.  Rows with more than kPickMax candidates
// (ties, a run of large entries in one warp's piece), without a finite sum or with a bound below 1e-30 go the general way; what
// lies below a bound is not counted there, which pays for the search.
// us a call, histograms / picked, top-p 0.9 and rows exported: 8 sequences x 6 rows x 50304 entries, k = 1 53.5 / 24.9, 20 28.9,
// 50 28.9, 96 31.0 (the same around -100 and 300); 17 x 12 rows of 32000, k = 50, 103.7 / 52.4.  Rows that go back to the histograms:
// constant 67.8 / 63.7, 30 finite entries 78.1 / 73.2, a NaN 57.1 / 55.5, sorted 59.3 / 57.5, 300 equal maxima 57.5 / 57.5
// (17 x 12 rows of 32000 111.4 / 117.0).
constexpr int kPickK = 96, kPickMax = 256;
struct FilterHist {
    unsigned cnt[kBins], mlo[kBins], mhi[kBins];
};
struct FilterSmem {
    PartStat warp[kTailWarps], cta;
    FilterHist hist[3];         // [0] the first pass; [1], [2] in turn for the others, so that a pass needs one cluster barrier
    unsigned wcnt[kTailWarps];
    unsigned long long wmass[kTailWarps];
    int first, last;            // first bin that meets the target, last bin that holds anything
    unsigned above_cnt;         // of the chosen bin: what lies above it, and its own mass
    unsigned long long above_mass, sel_mass;
    // few tokens to keep: per warp the bits that are set in all and in any of its threads' maxima, the largest of these and the
    // smallest that reaches the bound; the bound and how many of the CTA's maxima reach it; its candidates, both CTAs' together with their
    // masses, the thresholds' patterns and what weighs at least as much
    unsigned key_and[kTailWarps], key_or[kTailWarps], key_top[kTailWarps], key_low[kTailWarps];
    float low;
    int n_low, n_cand;
    float cand[kPickMax];
    float all[kPickMax];
    unsigned long long all_mass[kPickMax];
    unsigned best[2];
    unsigned long long best_mass[2];
};
__host__ __device__ constexpr size_t filter_smem(int V) {  // dynamic shared memory: the CTA's probabilities
    const size_t n = (size_t)((V + kFilterCluster - 1) / kFilterCluster) + 32 * kTailWarps;
    return n <= (size_t)kFilterCache ? n * 4 : 0;
}

__device__ __forceinline__ void bin_add(FilterHist &h, int bin, unsigned c, unsigned long long m) {
    if (c == 0) return;
    atomicAdd(&h.cnt[bin], c);
    const unsigned lo = (unsigned)m, old = atomicAdd(&h.mlo[bin], lo);
    const unsigned hi = (unsigned)(m >> 32) + (old + lo < old ? 1u : 0u);
    if (hi) atomicAdd(&h.mhi[bin], hi);
}

// What a search has narrowed its threshold down to: the keys [d_lo, d_lo + 2^width) and what lies above them.
struct KeyRange {
    unsigned d_lo;
    int width;
    unsigned above_cnt;
    unsigned long long above_mass, sel_mass;
};

// Choose the first bin (thread = bin, holding count c and mass m) that `met(inclusive count, inclusive mass)` holds at.
template <typename MetFn>
__device__ __forceinline__ int choose_bin(unsigned c, unsigned long long m, MetFn met, FilterSmem *fs, KeyRange &kr) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned ci = c;              // inclusive sums over the bins, from the largest keys down
    unsigned long long mi = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned tc = __shfl_up_sync(0xffffffffu, ci, o);
        const unsigned long long tm = __shfl_up_sync(0xffffffffu, mi, o);
        if (lane >= o) { ci += tc; mi += tm; }
    }
    if (lane == 31) { fs->wcnt[warp] = ci; fs->wmass[warp] = mi; }
    if (tid == 0) { fs->first = kBins; fs->last = -1; }
    __syncthreads();
    unsigned wc = lane < warp ? fs->wcnt[lane] : 0u;
    unsigned long long wm = lane < warp ? fs->wmass[lane] : 0ull;
    wc = __reduce_add_sync(0xffffffffu, wc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wm += __shfl_xor_sync(0xffffffffu, wm, o);
    ci += wc;
    mi += wm;
    const unsigned met_mask = __ballot_sync(0xffffffffu, c > 0 && met(kr.above_cnt + ci, kr.above_mass + mi));
    const unsigned any_mask = __ballot_sync(0xffffffffu, c > 0);
    if (lane == 0) {
        if (met_mask) atomicMin(&fs->first, tid + __ffs(met_mask) - 1);
        if (any_mask) atomicMax(&fs->last, tid + 31 - __clz(any_mask));
    }
    __syncthreads();
    const int sel = fs->first < kBins ? fs->first : max(fs->last, 0);  // (out of reach: keep everything there is)
    if (tid == sel) {
        fs->above_cnt = kr.above_cnt + ci - c;
        fs->above_mass = kr.above_mass + mi - m;
        fs->sel_mass = m;
    }
    __syncthreads();
    kr.above_cnt = fs->above_cnt;
    kr.above_mass = fs->above_mass;
    kr.sel_mass = fs->sel_mass;
    return sel;
}

// grid (kFilterCluster rows, B): statistics, restriction and p row of the rows that a restriction applies to.
struct FilterArgs {
    const float *logits;  // [B, M, V]
    int M, V;
    const int32_t *n_eff; // null: every row, grid.x = kFilterCluster M; else only row n_eff[b] - 1 of sequence b
    float inv_t;
    int top_k;
    float top_p;
    RowStat *stats;       // [B, grid.x / kFilterCluster]
    RowFilter *filt;
    float *p_out;         // [B, M, V] or null
};
inline bool filter_picks(const FilterArgs &a) {
    return a.top_k > 0 && a.top_k <= kPickK && a.top_k < a.V && a.inv_t > 0.f && filter_smem(a.V) > 0;
}
// PICK: with the search among candidates in front (see kPickK); without it, nothing of it is in the general way's way.
template <bool PICK>
__global__ void __cluster_dims__(kFilterCluster, 1, 1) __launch_bounds__(kTailThreads) row_filter_kernel(FilterArgs a) {
    extern __shared__ float fcache[];
    __shared__ FilterSmem sm;
    FilterSmem *fs = &sm;
    cg::cluster_group cl = cg::this_cluster();
    constexpr int IT = kFilterBatch, kStep = 32 * IT;
    const int b = blockIdx.y, i = blockIdx.x / kFilterCluster, V = a.V, n_rows = gridDim.x / kFilterCluster;
    const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float inv_t = a.inv_t;
    const size_t row = (size_t)b * a.M + (a.n_eff ? max(a.n_eff[b] - 1, 0) : i);
    const float *lg = a.logits + row * V;
    int lo, hi;
    row_piece(V, kFilterCluster * kTailWarps, rank * kTailWarps + warp, lo, hi);
    const bool cached = PICK || filter_smem(V) > 0;
    int cta_lo, unused;
    row_piece(V, kFilterCluster * kTailWarps, rank * kTailWarps, cta_lo, unused);
    float *mine = fcache - cta_lo;   // entry j of the row at mine[j]

    // ---- statistics; the logits stay in shared memory ----
    float mx = -INFINITY;
    int at = 0x7fffffff;
    for (int base = lo; base < hi; base += kStep) {
        float x[IT];
        tail_load<IT>(lg, base, hi, -INFINITY, x);
#pragma unroll
        for (int u = 0; u < IT; ++u) {
            const int j = base + 32 * u + lane;
            if (x[u] > mx) { mx = x[u]; at = j; }
            if (cached && j < hi) mine[j] = x[u];
        }
    }
    auto entry = [&](int j) { return cached ? mine[j] : __ldcg(lg + j); };
    int n_low = 0;
    if constexpr (PICK) {
        // The bound, from the order-preserving patterns of the threads' maxima: the largest if it is there top_k times; else, from the
        // top, the bits in which they differ at all, until little more than top_k of them reach it.  So it is as close wherever
        // the logits lie: on the patterns' upper halves, rows around 300 had too many candidates.
        const bool any = mx > -INFINITY;
        const unsigned bits = __float_as_uint(mx), key = any ? bits ^ ((bits >> 31) ? 0xffffffffu : 0x80000000u) : 0u;
        const unsigned wa = __reduce_and_sync(0xffffffffu, any ? key : 0xffffffffu), wo = __reduce_or_sync(0xffffffffu, key);
        const unsigned wt = __reduce_max_sync(0xffffffffu, key);
        if (lane == 0) { fs->key_and[warp] = wa; fs->key_or[warp] = wo; fs->key_top[warp] = wt; }
        unsigned bound = 0xffffffffu;
        n_low = __syncthreads_count(any);
        if (n_low >= a.top_k) {
            bound = __reduce_max_sync(0xffffffffu, fs->key_top[lane]);
            const int n_top = __syncthreads_count(key == bound);
            if (n_top >= a.top_k) {
                n_low = n_top;
            } else {
                bound = __reduce_and_sync(0xffffffffu, fs->key_and[lane]);
                unsigned rest = bound ^ __reduce_or_sync(0xffffffffu, fs->key_or[lane]);
                const int enough = a.top_k + (a.top_k >> 5) + 2;
#pragma unroll 1
                while (rest && n_low > enough) {
                    const unsigned bit = 0x80000000u >> __clz(rest);
                    rest ^= bit;
                    const int n = __syncthreads_count(key >= (bound | bit));
                    if (n >= a.top_k) { bound |= bit; n_low = n; }
                }
            }
        }
        const unsigned wl = __reduce_min_sync(0xffffffffu, any && key >= bound ? key : 0xffffffffu);
        if (lane == 0) fs->key_low[warp] = wl;
    }
    {
        const float m = warp_max_redux(mx);
        const int am = __reduce_min_sync(0xffffffffu, mx == m ? at : 0x7fffffff);
        float part = 0.f;
        const float ref = m > -INFINITY ? m : 0.f;  // (as in cluster_stats)
        for (int j = lo + lane; j < hi; j += 32) part += expf((entry(j) - ref) * inv_t);
        const double s = warp_sum((double)part);
        if (lane == 0) {
            PartStat t;
            t.mx = m;
            t.am = am;
            t.s = s;
            fs->warp[warp] = t;
        }
    }
    for (int k = tid; k < 2 * 3 * kBins; k += kTailThreads) reinterpret_cast<unsigned *>(fs->hist)[k] = 0;
    __syncthreads();
    if (warp == 0) {
        const PartStat t = join_parts<32>(fs->warp[lane], inv_t);
        if (lane == 0) fs->cta = t;
        if constexpr (PICK) {
            const unsigned k = __reduce_min_sync(0xffffffffu, fs->key_low[lane]);
            if (lane == 0) {
                fs->low = k == 0xffffffffu ? -INFINITY : __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu));
                fs->n_low = n_low;
                fs->n_cand = 0;
                fs->best[0] = fs->best[1] = 0;
            }
        }
    }
    cl.sync();
    const RowStat st = row_stat(join_parts<kFilterCluster>(*cl.map_shared_rank(&fs->cta, lane % kFilterCluster), inv_t));
    const unsigned kmax = __float_as_uint(prob_of(st.mx, st, inv_t, st.amax));
    auto mass_of = [](float p) { return __double2ull_rz((double)fminf(p, 2.f) * kMassUnit); };
    auto write_stats = [&](const RowFilter &f) {
        if (rank == 0 && tid == 0) {
            a.stats[(size_t)b * n_rows + i] = st;
            a.filt[(size_t)b * n_rows + i] = f;
        }
    };
    const bool use_k = PICK || (a.top_k > 0 && a.top_k < V), use_p = a.top_p > 0.f && a.top_p < 1.f;
    float cut = -INFINITY;  // entries whose exponent lies below it are out whatever the search finds
    if constexpr (PICK) {
        const FilterSmem *o = cl.map_shared_rank(fs, rank ^ 1);
        const float low = fmaxf(fs->low, o->low);
        // (an entry 1e-4 below the bound in the exponent has the smaller probability whatever the roundings)
        if (low > -INFINITY && st.z > 0.f && st.z < INFINITY && prob_of(low, st, inv_t, -1) >= 1e-30f) cut = (low - st.mx) * inv_t - 1e-4f;
        const int n_min = (fs->low == low ? fs->n_low : 0) + (o->low == low ? o->n_low : 0);
        int n = kPickMax + 1;
        if (cut > -INFINITY && n_min <= kPickMax) {  // (the same on both CTAs)
            for (int base = lo; base < hi; base += 128) {
                float x[4];
                bool some = false;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int j = base + 32 * u + lane;
                    x[u] = j < hi ? mine[j] : -INFINITY;
                    some |= (x[u] - st.mx) * inv_t >= cut;
                }
                if (some) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if ((x[u] - st.mx) * inv_t >= cut) {
                            const int at_ = atomicAdd(&fs->n_cand, 1);
                            if (at_ < kPickMax) fs->cand[at_] = prob_of(x[u], st, inv_t, base + 32 * u + lane);
                        }
                    }
                }
            }
            cl.sync();
            n = fs->n_cand + o->n_cand;
        }
        const FilterSmem *o0 = cl.map_shared_rank(fs, 0), *o1 = cl.map_shared_rank(fs, 1);
        if (n <= kPickMax) {
            const int n0 = o0->n_cand;
            float v = 0.f;
            if (tid < n) {
                v = tid < n0 ? o0->cand[tid] : o1->cand[tid - n0];
                fs->all[tid] = v;
                fs->all_mass[tid] = mass_of(v);
            }
            __syncthreads();
            int c = 0;                  // tokens at least as probable, and their mass
            unsigned long long m = 0;
            if (tid < n) {
                for (int j = 0; j < n; ++j)
                    if (fs->all[j] >= v) { ++c; m += fs->all_mass[j]; }
                if (c >= a.top_k) atomicMax(&fs->best[0], __float_as_uint(v));
            }
            __syncthreads();
            RowFilter f;
            f.thr = __uint_as_float(fs->best[0]);
            if (tid < n && v == f.thr) fs->best_mass[0] = m;  // (the same value by whoever holds it)
            __syncthreads();
            const unsigned long long kept = fs->best_mass[0];
            unsigned long long mass = kept;
            if (use_p) {
                const unsigned long long target = __double2ull_ru((double)a.top_p * (double)kept);
                if (tid < n && v >= f.thr && m >= target) atomicMax(&fs->best[1], __float_as_uint(v));
                __syncthreads();
                f.thr = __uint_as_float(fs->best[1]);
                if (tid < n && v == f.thr) fs->best_mass[1] = m;
                __syncthreads();
                mass = fs->best_mass[1];
            }
            f.mass = (float)((double)mass / kMassUnit);
            write_stats(f);
            if (a.p_out) {
                float *p = a.p_out + row * V;
                for (int j = lo + lane; j < hi; j += 32) {
                    const float x = mine[j];
                    float out = 0.f;
                    if ((x - st.mx) * inv_t >= cut) {
                        const float pr = prob_of(x, st, inv_t, j);
                        out = pr < f.thr ? 0.f : pr / f.mass;
                    }
                    p[j] = out;
                }
            }
            cl.sync();  // nobody leaves while its shared memory is read
            return;
        }
    }

    // ---- histogram of the keys in [d_lo, d_lo + bins << shift) with p >= p_min (open_end: the last bin takes all beyond) ----
    auto count = [&](FilterHist &h, unsigned d_lo, int shift, int bins, bool open_end, float p_min, bool first) {
        int bin = -1;
        unsigned c = 0;
        unsigned long long m = 0;
        for (int j = lo + lane; j < hi; j += 32) {
            float p;
            if (first || !cached) {
                const float x = entry(j);
                if constexpr (PICK) {
                    if ((x - st.mx) * inv_t < cut) {  // (below the threshold, whatever it is: never counted, exported as zero)
                        mine[j] = 0.f;
                        continue;
                    }
                }
                p = prob_of(x, st, inv_t, j);
                if (cached) mine[j] = p;
            } else {
                p = mine[j];
            }
            if (!(p >= p_min)) continue;   // (a NaN is not looked at)
            const unsigned bits = __float_as_uint(p), d = bits < kmax ? kmax - bits : 0u;
            if (d < d_lo) continue;
            unsigned k = (d - d_lo) >> shift;
            if (k >= (unsigned)bins) {
                if (!open_end) continue;
                k = bins - 1;
            }
            if ((int)k != bin) {
                bin_add(h, bin, c, m);
                bin = (int)k;
                c = 0;
                m = 0;
            }
            ++c;
            m += mass_of(p);
        }
        bin_add(h, bin, c, m);
    };
    auto joined = [&](int h, unsigned &c, unsigned long long &m) {  // this thread's bin over the cluster
        c = 0;
        m = 0;
#pragma unroll
        for (int r = 0; r < kFilterCluster; ++r) {
            const FilterHist *o = cl.map_shared_rank(&fs->hist[h], r);
            c += o->cnt[tid];
            m += (unsigned long long)o->mlo[tid] + ((unsigned long long)o->mhi[tid] << 32);
        }
    };
    int turn = 0;
    auto refine = [&](KeyRange &kr, float p_min, auto met) {  // down to one key
        while (kr.width > 0) {
            const int shift = max(0, kr.width - 10), h = 1 + (turn & 1);
            ++turn;
            count(fs->hist[h], kr.d_lo, shift, 1 << (kr.width - shift), false, p_min, false);
            cl.sync();
            unsigned c;
            unsigned long long m;
            joined(h, c, m);
            for (int k = tid; k < 3 * kBins; k += kTailThreads) reinterpret_cast<unsigned *>(&fs->hist[3 - h])[k] = 0;  // (read by all before the barrier above)
            const int sel = choose_bin(c, m, met, fs, kr);
            kr.d_lo += (unsigned)sel << shift;
            kr.width = shift;
        }
    };
    constexpr int kShift0 = 18;
    auto range_of = [&](int sel, KeyRange &kr) {
        kr.d_lo = (unsigned)sel << kShift0;
        kr.width = sel == kBins - 1 ? 30 : kShift0;
    };
    count(fs->hist[0], 0u, kShift0, kBins, true, 0.f, true);
    cl.sync();
    unsigned c0;
    unsigned long long m0;
    joined(0, c0, m0);

    RowFilter f;
    f.thr = 0.f;
    f.mass = 0.f;
    double mass = 0.0;
    unsigned long long kept = ~0ull;  // mass of what top-k keeps
    if (use_k) {
        const unsigned want = (unsigned)a.top_k;
        auto met = [&](unsigned c, unsigned long long) { return c >= want; };
        KeyRange kr = {0u, 0, 0u, 0ull, 0ull};
        const int sel = choose_bin(c0, m0, met, fs, kr);
        const unsigned long long above = kr.above_mass;
        range_of(sel, kr);
        refine(kr, 0.f, met);
        f.thr = __uint_as_float(kmax - min(kr.d_lo, kmax));
        kept = kr.above_mass + kr.sel_mass;
        mass = (double)kept / kMassUnit;
        // top-p looks at what is left: whole bins above the chosen one, a part of it
        if (tid == sel) m0 = kept - above;
        if (tid > sel) { c0 = 0; m0 = 0; }
    }
    if (use_p) {
        if (kept == ~0ull) {  // (everything: the sum over the bins, once more through the exchange words)
            unsigned long long w = m0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (lane == 0) fs->wmass[warp] = w;
            __syncthreads();
            kept = 0;
            for (int k = 0; k < kTailWarps; ++k) kept += fs->wmass[k];
            __syncthreads();
        }
        const unsigned long long target = __double2ull_ru((double)a.top_p * (double)kept);
        auto met = [&](unsigned, unsigned long long m) { return m >= target; };
        KeyRange kr = {0u, 0, 0u, 0ull, 0ull};
        const int sel = choose_bin(c0, m0, met, fs, kr);
        range_of(sel, kr);
        refine(kr, f.thr, met);
        f.thr = __uint_as_float(kmax - min(kr.d_lo, kmax));
        mass = (double)(kr.above_mass + kr.sel_mass) / kMassUnit;
    }
    f.mass = (float)mass;
    write_stats(f);
    if (a.p_out) {
        float *p = a.p_out + row * V;
        // (as prob_f; a row without mass is one of NaNs.  A test for that in the loop cost 2 of 36 us, 15 rows of 32000)
        const float thr = f.mass == 0.f ? 0.f : f.thr, kept_mass = f.mass == 0.f ? 1.f : f.mass;
        for (int j = lo + lane; j < hi; j += 32) {
            const float pr = cached ? mine[j] : prob_of(__ldcg(lg + j), st, inv_t, j);
            p[j] = pr < thr ? 0.f : pr / kept_mass;
        }
    }
    cl.sync();  // nobody leaves while its shared memory is read
}

// The unrestricted counterpart, a cluster of eight per row: grid (kTailCluster M, B).  Taken where one cluster per sequence would
// walk the rows for longer than a second launch costs (see rows_apart in the host code).
template <int IT>
__global__ void __cluster_dims__(kTailCluster, 1, 1) __launch_bounds__(kTailThreads) row_stats_kernel(FilterArgs a) {
    __shared__ StatSmem ss;
    cg::cluster_group cl = cg::this_cluster();
    const int i = blockIdx.x / kTailCluster, b = blockIdx.y, V = a.V, rank = (int)cl.block_rank(), lane = threadIdx.x & 31;
    const size_t row = (size_t)b * a.M + i;
    const float *lg = a.logits + row * V;
    float l[IT];
    cluster_stats<IT>(lg, 1, V, a.inv_t, &ss, cl, l);
    const RowStat st = ss.row[0];
    if (rank == 0 && threadIdx.x == 0) {
        a.stats[row] = st;
        a.filt[row].thr = a.filt[row].mass = 0.f;
    }
    if (a.p_out) {
        int lo, hi;
        tail_piece(V, rank, lo, hi);
        const bool one = hi - lo <= 32 * IT;
        float *p = a.p_out + row * V;
        for (int base = lo; base < hi; base += 32 * IT) {
            if (!one) tail_load<IT>(lg, base, hi, 0.f, l);
#pragma unroll
            for (int k = 0; k < IT; ++k) {
                const int j = base + lane + 32 * k;
                if (j < hi) p[j] = prob_of(l[k], st, a.inv_t, j);
            }
        }
    }
    cl.sync();  // nobody leaves while its shared memory is read
}

// ---- inverse-CDF draw -------------------------------------------------------------------------------
struct DrawSmem {
    double tot[kTailWarps], incl[kTailWarps];  // the warps' sums, and their running sums
    double cta[2];              // this CTA's total, by draw (a kernel draws at most twice)
    float w[32 * 8];            // the owner warp's entries, handed from its load order to index order
};

// Inverse-CDF draw over V weights >= 0 by the whole cluster: the smallest j whose inclusive prefix sum (fp64, pieces in
// index order) exceeds u * S.  `weights(base, w)` gives the piece's weights from `base` on, 0 beyond its end; it is
// called again by the warp whose piece the draw falls into.  That warp is found without a vote: piece boundaries are the
// same fp64 numbers on both sides (a piece ends where the next one starts), so exactly one piece holds u * S.  Inside it
// a zero-weight index is never drawn; if rounding leaves no index, the piece's largest with weight > 0 is taken.
// Outside [0, 1) no piece holds u * S: below 0 the first index with weight > 0 is drawn, from 1 on (and for a NaN, or an
// infinite S) the last one.
// Returns the index in every lane of that warp and -1 elsewhere; *total = S everywhere (S <= 0: nothing was drawn).
template <int IT, typename WeightFn>
__device__ __forceinline__ int cluster_draw(WeightFn weights, int V, float u, DrawSmem *ds, cg::cluster_group &cl, int slot,
                                            double *total) {
    constexpr int kStep = 32 * IT;
    const int rank = (int)cl.block_rank(), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int lo, hi;
    tail_piece(V, rank, lo, hi);
    double sum = 0.0;
    float w[IT];
    for (int b = lo; b < hi; b += kStep) {
        weights(b, w);
#pragma unroll
        for (int k = 0; k < IT; ++k) sum += (double)w[k];
    }
    sum = warp_sum(sum);
    if (lane == 0) ds->tot[warp] = sum;
    __syncthreads();
    // Piece boundaries as running sums in index order: what one warp takes for its end is bit for bit the next one's beginning.
    if (warp == 0) {
        double T = 0.0;
#pragma unroll
        for (int k = 0; k < kTailWarps; ++k)
            if (k <= lane) T += ds->tot[k];
        ds->incl[lane] = T;
        if (lane == 31) ds->cta[slot] = T;
    }
    cl.sync();
    const double w_beg = warp ? ds->incl[warp - 1] : 0.0, w_end = ds->incl[warp];
    const double one_cta = lane < kTailCluster ? *cl.map_shared_rank(&ds->cta[slot], lane) : 0.0;
    double c_beg = 0.0, S = 0.0;
#pragma unroll
    for (int k = 0; k < kTailCluster; ++k) {
        if (k == rank) c_beg = S;
        S += __shfl_sync(0xffffffffu, one_cta, k);
    }
    *total = S;
    if (!(S > 0.0)) return -1;
    const double beg = c_beg + w_beg, end = c_beg + w_end;  // (the last warp's end is c_beg + T, where the next CTA begins)
    double target = (double)u * S;
    bool owner;
    if (target < S) {
        target = target < 0.0 ? 0.0 : target;
        owner = beg <= target && target < end;
    } else {  // (the same in all threads of the cluster) the last piece that weighs anything, walked to its end
        const unsigned warps = __ballot_sync(0xffffffffu, ds->tot[lane] > 0.0), ctas = __ballot_sync(0xffffffffu, one_cta > 0.0);
        owner = __clz(ctas) == 31 - rank && __clz(warps) == 31 - warp;
        target = INFINITY;
    }
    if (!owner) return -1;  // the same in all lanes
    double run = beg;
    int hit = -1, last = -1;
    for (int b = lo; b < hi && hit < 0; b += kStep) {
        weights(b, w);
#pragma unroll
        for (int k = 0; k < IT; ++k) ds->w[32 * k + lane] = w[k];
        __syncwarp();
        float v[IT];
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            v[k] = ds->w[IT * lane + k];
            s += (double)v[k];
        }
        double si = s;  // inclusive over the lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, si, o);
            if (lane >= o) si += t;
        }
        double r = run + (si - s);
        int mine = 0x7fffffff, tail = -1;
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            r += (double)v[k];
            if (v[k] > 0.f) {
                tail = b + IT * lane + k;
                if (mine == 0x7fffffff && r > target) mine = tail;
            }
        }
        mine = __reduce_min_sync(0xffffffffu, mine);
        last = max(last, __reduce_max_sync(0xffffffffu, tail));
        if (mine != 0x7fffffff) hit = mine;
        run += __shfl_sync(0xffffffffu, si, 31);
        __syncwarp();
    }
    return hit >= 0 ? hit : last;
}

struct VerifyArgs {
    const float *logits;    // [B, K+1, V]
    int K, V;
    const int32_t *rows;    // [B, K+1]: pending, x~_1..x~_K
    const float *q;         // [B, K, V]
    const float *u;         // [B, K+1]
    float inv_t;            // 1/T, 0 = greedy
    int32_t *n_accepted;    // [B]
    int32_t *next_token;
    int next_stride;
    float *p_debug;         // [B, K+1, V] or null
    int32_t *keep;          // [B] or null: n_accepted + 1 for kv_commit
    const RowStat *stats;   // [B, K+1], only under a restriction of the target rows (q arrives already restricted)
    const RowFilter *filt;
};

// grid (kTailCluster B), one cluster per sequence: row statistics (given by row_filter_kernel under a restriction), accept
// scan, then residual / bonus draw.
template <bool kGiven, int IT>
__global__ void __cluster_dims__(kTailCluster, 1, 1) __launch_bounds__(kTailThreads) verify_kernel(VerifyArgs a) {
    __shared__ StatSmem ss;
    __shared__ DrawSmem ds;
    __shared__ int s_acc;
    cg::cluster_group cl = cg::this_cluster();
    constexpr int kStep = 32 * IT;
    const int b = blockIdx.x / kTailCluster, K = a.K, V = a.V, lane = threadIdx.x & 31;
    const float *logits = a.logits + (size_t)b * (K + 1) * V;
    const RowFilter none = {0.f, 0.f};
    const float inv_t = a.inv_t;
    // what the accept scan needs of row i, in lane i of warp 0: on its way under the statistics
    float xl = 0.f, xq = 0.f, xu = 0.f;
    int x = 0;
    if (threadIdx.x < K) {
        x = max(0, min(a.rows[b * (K + 1) + 1 + lane], V - 1));
        xl = __ldcg(logits + (size_t)lane * V + x);
        xq = __ldcg(a.q + ((size_t)b * K + lane) * V + x);
        xu = a.u[b * (K + 1) + lane];
    }
    const float u = a.u[b * (K + 1) + K];
    if (kGiven) {
        for (int i = threadIdx.x; i <= K; i += kTailThreads) ss.row[i] = a.stats[b * (K + 1) + i];
        __syncthreads();
    } else {
        float l[IT];
        cluster_stats<IT>(logits, K + 1, V, inv_t, &ss, cl, l);
    }
    if (threadIdx.x < 32) {  // (every CTA of the cluster takes the same few steps)
        bool ok = false;
        if (lane < K) {
            const float px = prob_f(xl, ss.row[lane], kGiven ? a.filt[b * (K + 1) + lane] : none, inv_t, x);
            ok = __fmul_rn(xu, xq) < px;  // accept with probability min(1, p/q): u * q < p, one fp32 rounding of the product
        }
        const unsigned refused = ~__ballot_sync(0xffffffffu, ok);  // (K <= 31: lane K always refuses)
        if (lane == 0) s_acc = min(K, __ffs(refused) - 1);
    }
    __syncthreads();
    const int acc = s_acc;
    const float *lg = logits + (size_t)acc * V;
    const RowStat rs = ss.row[acc];
    const RowFilter rf = kGiven ? a.filt[b * (K + 1) + acc] : none;
    const int rank = (int)cl.block_rank();
    int lo, hi;
    tail_piece(V, rank, lo, hi);
    double S = 0.0;
    int y = -1;
    auto p_weights = [&](int base, float (&w)[IT]) {
        tail_load<IT>(lg, base, hi, 0.f, w);
#pragma unroll
        for (int k = 0; k < IT; ++k) w[k] = base + lane + 32 * k < hi ? prob_f(w[k], rs, rf, inv_t, base + lane + 32 * k) : 0.f;
    };
    if (acc < K) {
        const float *qr = a.q + ((size_t)b * K + acc) * V;
        y = cluster_draw<IT>(
            [&](int base, float (&w)[IT]) {
                float qv[IT];
                tail_load<IT>(qr, base, hi, 0.f, qv);
                p_weights(base, w);
#pragma unroll
                for (int k = 0; k < IT; ++k) w[k] = fmaxf(0.f, __fsub_rn(w[k], qv[k]));
            },
            V, u, &ds, cl, 0, &S);
    }
    if (!(S > 0.0))  // all accepted: bonus from p_{K+1}; or an all-zero residual: fall back to p
        y = cluster_draw<IT>(p_weights, V, u, &ds, cl, 1, &S);
    const bool first = rank == 0 && threadIdx.x == 0;
    if (!(S > 0.0) && first) y = rs.amax;  // a row whose probabilities all vanished (non-finite logits)
    if (y >= 0 && lane == 0) a.next_token[(size_t)b * a.next_stride] = y;
    if (first) {
        a.n_accepted[b] = acc;
        if (a.keep) a.keep[b] = acc + 1;
    }
    if (!kGiven && a.p_debug) {
        for (int i = 0; i <= K; ++i) {
            const RowStat st = ss.row[i];
            const float *row = logits + (size_t)i * V;
            float *p = a.p_debug + ((size_t)b * (K + 1) + i) * V;
            for (int base = lo; base < hi; base += kStep) {
                float l[IT];
                tail_load<IT>(row, base, hi, 0.f, l);
#pragma unroll
                for (int k = 0; k < IT; ++k)
                    if (base + lane + 32 * k < hi) p[base + lane + 32 * k] = prob_of(l[k], st, inv_t, base + lane + 32 * k);
            }
        }
    }
    cl.sync();  // nobody leaves while its shared memory is read
}

struct DraftTailArgs {
    const float *logits;  // [B, M, V] rows of the draft forward
    int M, V;
    const int32_t *n_eff; // [B] rows fed per sequence (the last one is sampled)
    float inv_t;
    const float *u; int u_stride;
    int32_t *token_out; int token_stride;
    float *q_out; size_t q_stride;
    const RowStat *stats; // [B], only under a restriction: of the sampled rows, from row_filter_kernel
    const RowFilter *filt;
    int32_t *len;         // [B] committed lengths: the fed rows are committed here
    unsigned long long *mailbox; unsigned seq;  // see report_len
};

__device__ __forceinline__ void report_len(unsigned long long *mailbox, int b, unsigned seq, int len);

// grid (kTailCluster B), one cluster per sequence: q = softmax(last row / T), exported; x~ = inverse-CDF(q, u); the fed
// rows become part of the cache
template <bool kGiven, int IT>
__global__ void __cluster_dims__(kTailCluster, 1, 1) __launch_bounds__(kTailThreads) draft_tail_kernel(DraftTailArgs a) {
    __shared__ StatSmem ss;
    __shared__ DrawSmem ds;
    cg::cluster_group cl = cg::this_cluster();
    constexpr int kStep = 32 * IT;
    const int b = blockIdx.x / kTailCluster, rank = (int)cl.block_rank(), lane = threadIdx.x & 31;
    const int fed = a.n_eff[b], row = max(fed - 1, 0);
    const float u = a.u[(size_t)b * a.u_stride];
    const float *lg = a.logits + ((size_t)b * a.M + row) * a.V;
    int lo, hi;
    tail_piece(a.V, rank, lo, hi);
    float l[IT];
    RowStat st;
    RowFilter fl = {0.f, 0.f};
    if (kGiven) {
        tail_load<IT>(lg, lo, hi, 0.f, l);
        st = a.stats[b];
        fl = a.filt[b];
    } else {
        cluster_stats<IT>(lg, 1, a.V, a.inv_t, &ss, cl, l);
        st = ss.row[0];
    }
    float *q = a.q_out + (size_t)b * a.q_stride;
    const bool one = hi - lo <= kStep;
    for (int base = lo; base < hi; base += kStep) {
        if (!one) tail_load<IT>(lg, base, hi, 0.f, l);
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            const int j = base + lane + 32 * k;
            l[k] = j < hi ? prob_f(l[k], st, fl, a.inv_t, j) : 0.f;
            if (j < hi) q[j] = l[k];
        }
    }
    double S;
    int y = cluster_draw<IT>(
        [&](int base, float (&w)[IT]) {
            if (one) {
#pragma unroll
                for (int k = 0; k < IT; ++k) w[k] = l[k];
            } else {
                tail_load<IT>(q, base, hi, 0.f, w);  // (written by this very lane)
            }
        },
        a.V, u, &ds, cl, 0, &S);
    const bool first = rank == 0 && threadIdx.x == 0;
    if (!(S > 0.0) && first) y = st.amax;
    if (y >= 0 && lane == 0) a.token_out[(size_t)b * a.token_stride] = y;
    if (first) {
        const int n = a.len[b] + fed;  // fed is what the forward's set-up found to fit
        a.len[b] = n;
        report_len(a.mailbox, b, a.seq, n);
    }
    cl.sync();  // nobody leaves while its shared memory is read
}

// ---------------- cache length bookkeeping ----------------
// Every kernel that changes a committed length reports it to the host through the sequence's word of mapped host
// memory, tagged with the host's number of the operation: (seq << 32) | length.  The host plans attention splits
// from an upper bound of the lengths; with these words the bound follows the real lengths without a
// synchronisation (it adds what the operations queued behind `seq` can add at most).
__device__ __forceinline__ void report_len(unsigned long long *mailbox, int b, unsigned seq, int len) {
    if (mailbox) *reinterpret_cast<volatile unsigned long long *>(mailbox + b) = ((unsigned long long)seq << 32) | (unsigned)len;
}
// Keep n_keep[b] more rows.  A length that would pass the capacity S is clamped and recorded as
// SSD_E_CAPACITY in the sticky status word: rows that no forward wrote must not become context.
__global__ void kv_commit_kernel(int32_t *len, const int32_t *n_keep, int B, int S, int32_t *status,
                                 unsigned long long *mailbox, unsigned seq) {
    const int b = threadIdx.x;
    if (b < B) {
        int v = len[b] + max(0, n_keep[b]);
        if (v > S) {
            v = S;
            set_status(status, -3);
        }
        len[b] = v;
        report_len(mailbox, b, seq, v);
    }
}
__global__ void kv_commit_rows_kernel(int32_t *len, const int32_t *n_eff, int B, unsigned long long *mailbox,
                                      unsigned seq) {
    const int b = threadIdx.x;
    if (b < B) {
        const int v = len[b] + n_eff[b];   // n_eff is what the forward's set-up found to fit
        len[b] = v;
        report_len(mailbox, b, seq, v);
    }
}
__global__ void kv_rollback_kernel(int32_t *len, const int32_t *new_len, int B, unsigned long long *mailbox,
                                   unsigned seq) {
    const int b = threadIdx.x;
    if (b < B) {
        const int v = max(0, min(len[b], new_len[b]));
        len[b] = v;
        report_len(mailbox, b, seq, v);
    }
}
// The cache of a layer-skip draft from its target's: both were empty and the target has been fed, so the draft's layers hold
// the target's first layers' keys and values.  The host knows that from its bounds; a sequence whose lengths say otherwise
// (someone wrote the slab) is left as it is, and the draft's status says SSD_E_ARG.
// grid (16-row blocks of the longest prompt, H, 2 B layers), 16-byte pieces.
__global__ void __launch_bounds__(256) kv_adopt_kernel(const uint8_t *src, uint8_t *dst, const int32_t *src_len, const int32_t *dst_len,
                                                       int max_tokens, int B, int src_S, int dst_S, int row_bytes) {
    const int plane = blockIdx.z, b = (plane >> 1) % B;   // plane = (layer B + b) 2 + K|V
    if (dst_len[b] != 0 || src_len[b] > max_tokens) return;
    const int rows = min(min(src_len[b], dst_S) - (int)blockIdx.x * 16, 16);
    if (rows <= 0) return;
    const size_t head = (size_t)plane * gridDim.y + blockIdx.y;
    const uint4 *s = reinterpret_cast<const uint4 *>(src + (head * src_S + (size_t)blockIdx.x * 16) * row_bytes);
    uint4 *d = reinterpret_cast<uint4 *>(dst + (head * dst_S + (size_t)blockIdx.x * 16) * row_bytes);
    for (int i = threadIdx.x; i < rows * row_bytes / 16; i += 256) d[i] = s[i];
}
// ... and its lengths (one block of 64 threads)
__global__ void kv_adopt_len_kernel(const int32_t *src_len, const int32_t *src_status, int32_t *len, int32_t *status, int max_tokens,
                                    int B, int S, unsigned long long *mailbox, unsigned seq) {
    const int b = threadIdx.x;
    if (b == 0 && *src_status != 0) set_status(status, *src_status);
    if (b < B) {
        const bool empty = len[b] == 0 && src_len[b] <= max_tokens;
        if (!empty) set_status(status, -1);
        const int v = empty ? min(src_len[b], S) : len[b];
        len[b] = v;
        report_len(mailbox, b, seq, v);
    }
}
// chunk c of a prompt pass: rows fed per sequence = clamp(n_tokens - c*C, 0, C)
__global__ void prefill_rows_kernel(const int32_t *n_tokens, int chunk, int C, int32_t *n_rows, int B) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) n_rows[b] = max(0, min(C, n_tokens[b] - chunk * C));
}

struct AdvanceArgs {
    int32_t *tlen, *dlen;  // target / draft committed lengths (dlen may be null)
    int32_t *rows;         // [B, K+1]
    int K, B;
    const int32_t *n_accepted, *next_token;
    int next_stride;
    int32_t *out_tokens; int out_cap; int32_t *out_count;
    int32_t *draft_in, *draft_n_in;
    unsigned long long *t_mailbox, *d_mailbox;  // see report_len
    unsigned t_seq, d_seq;
};

__device__ __forceinline__ void spec_advance_one(const AdvanceArgs &a, int b) {
    const int K = a.K;
    int acc = max(0, min(a.n_accepted[b], K));
    const int y = a.next_token[(size_t)b * a.next_stride];
    int32_t *row = a.rows + (size_t)b * (K + 1);
    const int n = a.tlen[b] + 1;  // committed tokens before this iteration
    if (a.out_tokens && a.out_count) {
        int c = a.out_count[b];
        for (int i = 0; i < acc; ++i, ++c)
            if (c < a.out_cap) a.out_tokens[(size_t)b * a.out_cap + c] = row[1 + i];
        if (c < a.out_cap) a.out_tokens[(size_t)b * a.out_cap + c] = y;
        a.out_count[b] = c + 1;
    } else if (a.out_count) {
        a.out_count[b] += acc + 1;
    }
    if (a.draft_in && a.draft_n_in) {
        if (acc == K && K > 0) {
            a.draft_in[2 * b] = row[K];
            a.draft_in[2 * b + 1] = y;
            a.draft_n_in[b] = 2;
        } else {
            a.draft_in[2 * b] = y;
            a.draft_in[2 * b + 1] = y;
            a.draft_n_in[b] = 1;
        }
    }
    const int t_new = n + acc;
    a.tlen[b] = t_new;
    report_len(a.t_mailbox, b, a.t_seq, t_new);
    if (a.dlen) {
        const int d_new = min(a.dlen[b], K > 0 ? min(n + acc, n + K - 1) : n + acc);
        a.dlen[b] = d_new;
        report_len(a.d_mailbox, b, a.d_seq, d_new);
    }
    row[0] = y;
}
__global__ void spec_advance_kernel(AdvanceArgs a) {  // one block of 64 threads
    if ((int)threadIdx.x < a.B) spec_advance_one(a, threadIdx.x);
}

}  // namespace ssd
