// The whole decoder forward of a small fp32 model as ONE cooperative kernel.
//
// Such a model (a few layers of a few hundred columns) sits in L2; a pass over it is a chain of tiny dependent steps and
// nothing else: as one launch per step (47 of them for a four-layer pass, 17 for a one-layer draft step) each cost 3-13 us
// of launch, ramp and a single exposed trip to L2.  Here a step is a phase of 2-4 us between grid barriers, and there are
// fewer of them: the norm of a row block is taken by every CTA that multiplies it, biases, activation and the residual
// add ride in the epilogues, rotary and the cache append belong to the attention item.  Per sequential layer: qkv |
// attention | out-projection | MLP in + activation | MLP out; per parallel-residual layer: qkv + MLP in | attention |
// out-projection + MLP out.
//   * projections: a warp owns an output column and holds eight activation rows' sums; the rows sit in shared memory, the
//     first 1024 weights of the warp's first column are fetched into registers BEFORE the barrier in front of the phase;
//   * attention: one CTA per (sequence, head): four lanes per position for the scores, a thread per (head column, position
//     group) for P V; the CTA appends the pass's keys / values itself, so nothing else has to wait for them.
// Generation with the four-layer 256-wide model (K = 4, 16 iterations): 13.7 ms as one launch per step, 5.3 as one
// per forward.
// Results as the stepwise path's up to fp32 summation order.  Every barrier wait is bounded.
#pragma once
#include "attention.cuh"
#include "common.cuh"
#include "gemm.cuh"
#include "persistent.cuh"
#include "rowops.cuh"

namespace ssd {

constexpr int kFfThreads = 512, kFfWarps = kFfThreads / 32;
constexpr int kFfRows = 8;              // activation rows a warp sums at a time, query rows an attention item walks its positions for
constexpr int kFfMaxLayers = 32;        // (their tensors' addresses ride in the kernel parameters)
constexpr int kFfMaxSmem = 200 * 1024;
constexpr int kFfChunk = 256;           // positions per attention step
// An item walks its positions alone (6.5 us per 256 of them and layer at head 64, 20 at head 128, half as much again per further
// block of eight rows); beyond this many the stepwise path, which splits them over CTAs, is the faster form.  What the one kernel
// saves elsewhere grows with the rows of the pass and with the width.  us a layer, one kernel / stepwise: head 128, d 512, one
// row at 700 positions 91 / 92, at 1000 117 / 97; five rows at 1000 128 / 147; head 64, d 64, nine rows at 700 89 / 99, at
// 1300 122 / 104.
// (From 32 items on the split path's share of an SM is no smaller.)
inline int ff_max_ctx(int d, int Dh, int H, int B, int M) {
    if (B * H >= 32) return 1536;
    const double one = 64.0 / Dh * (1280.0 + (d > 256 ? 0.5 * (d - 256) : 0.0)), per_row = 30.0 + 0.3 * d * 64.0 / Dh;
    const double most = (one + per_row * (B * M - 1)) / (1.0 + 0.6 * ((M - 1) / kFfRows));
    return most < 1536.0 ? (int)most : 1536;
}

struct FfLayer {
    const float *ln1_g, *ln1_b, *w_qkv, *b_qkv, *w_o, *b_o, *ln2_g, *ln2_b, *w_in, *b_in, *w_out, *b_out;
};
struct FfParams {
    int n_layers, d, H, Dh, F, V, norm_kind, swiglu, parallel, rotary_dim, learned_pos, pos_limit;
    float eps, rotary_base, scale;
    double inv_d;  // 1 / d
    int B, M, R, S;
    const int32_t *tokens; int tok_stride;
    const int32_t *n_rows;
    const float *tok_emb, *pos_emb, *lnf_g, *lnf_b, *w_lm;
    float *cache; size_t layer_elems;
    const int32_t *len;
    int32_t *status;
    RowInfo ri;
    float *x, *qkv, *ao, *act, *logits;
    unsigned *gbar;      // see leave_grid
    long long wait_cycles;
    int want_logits;
    unsigned long long *trace;  // optional: CTA 0 stamps the global timer at the start, after every grid barrier and at the end
    FfLayer layer[kFfMaxLayers];
};

// dynamic shared memory of a pass
inline size_t ff_smem(int d, int F, int M, int Dh) {
    const size_t gemm = (size_t)kFfRows * (d > F ? d : F) * 4;
    const size_t groups = kFfThreads / Dh;
    const size_t attn = ((size_t)M * Dh + (size_t)kFfRows * kFfChunk + 3 * (size_t)kFfRows + groups * kFfRows * Dh) * 4;
    return gemm > attn ? gemm : attn;
}

__device__ __forceinline__ void ff_stamp(const FfParams &p, unsigned i) {
    if (p.trace && blockIdx.x == 0 && threadIdx.x == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        p.trace[i] = t;
        p.trace[i + 1] = 0;
    }
}
// All threads of the grid; false (everywhere in the CTA) once a wait has run out.
__device__ __forceinline__ bool ff_sync(const FfParams &p, unsigned &epoch, volatile int *ok) {
    ++epoch;
    __syncthreads();
    if (threadIdx.x == 0) {
        red_release_add(p.gbar, 1u);  // (one release and one acquire: the CTA barriers pass them on)
        const unsigned target = epoch * gridDim.x;
        if (ld_acquire(p.gbar) < target) {
            const long long t0 = clock64();
            while (ld_acquire(p.gbar) < target) {
                if (clock64() - t0 > p.wait_cycles) {
                    set_status(p.status, kTimeoutCode);
                    *ok = 0;
                    break;
                }
            }
        }
        ff_stamp(p, epoch);
    }
    __syncthreads();
    return *ok != 0;
}

// A warp's weights on their way: 1024 / NF entries of each of NF columns' rows (columns `cols` apart; those from n_end on
// are read as the last one and dropped by the caller).
template <int NF>
__device__ __forceinline__ void ff_fetch(const float *W, int n, int cols, int n_end, int K4, int k0, float4 (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < NF; ++j) {
        const float4 *w = reinterpret_cast<const float4 *>(W) + (size_t)min(n + j * cols, n_end - 1) * K4;
#pragma unroll
        for (int i = 0; i < 8 / NF; ++i) {
            const int k = k0 + lane + 32 * i;
            v[j * (8 / NF) + i] = k < K4 ? __ldg(w + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}
// acc[j][r] = sum_k w_j[k] x[r][k] for NF columns and the `rows` staged rows; `v` holds the columns' first entries (and is used
// up).  A staged row is read once for all NF columns: shared-memory reads bound the small projections.
template <int NF>
__device__ __forceinline__ void ff_dot(const float *W, int n, int cols, int n_end, int K4, const float4 *xs, int rows, float4 (&v)[8],
                                       float (&acc)[NF][kFfRows]) {
    const int lane = threadIdx.x & 31;
    constexpr int KC = 8 / NF;
#pragma unroll
    for (int j = 0; j < NF; ++j)
#pragma unroll
        for (int r = 0; r < kFfRows; ++r) acc[j][r] = 0.f;
    for (int k0 = 0;;) {
#pragma unroll
        for (int r = 0; r < kFfRows; ++r) {
            if (r < rows) {
#pragma unroll
                for (int i = 0; i < KC; ++i) {
                    const int k = k0 + lane + 32 * i;
                    if (k < K4) {
                        const float4 x = xs[(size_t)r * K4 + k];
#pragma unroll
                        for (int j = 0; j < NF; ++j) {
                            const float4 w = v[j * KC + i];
                            acc[j][r] = fmaf(w.x, x.x, fmaf(w.y, x.y, fmaf(w.z, x.z, fmaf(w.w, x.w, acc[j][r]))));
                        }
                    }
                }
            }
        }
        k0 += 32 * KC;
        if (k0 >= K4) break;
        ff_fetch<NF>(W, n, cols, n_end, K4, k0, v);
    }
}
// the sums over the warp: lane 4 r (and its three neighbours) returns row r's
__device__ __forceinline__ float ff_reduce(float (&a)[kFfRows]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 4; h > 0; h >>= 1) {
        const bool up = lane & (4 * h);
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const float send = up ? a[j] : a[j + h], keep = up ? a[j + h] : a[j];
            a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
        }
    }
    float v = a[0];
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}

// Rows 8 rb .. of the residual stream, normalised, into xs [8][d]: a warp per row, everything it needs (row, gain, bias) on
// its way together; rows of up to 256 columns stay in registers, wider ones are read again.  `embed`: they are embedding rows
// (and their owner starts the residual stream with them).
__device__ __forceinline__ void ff_stage_norm(const FfParams &p, int rb, bool embed, const float *g, const float *b, float *xs) {
    constexpr int NR = 2;  // float4 per lane held in registers
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = rb * kFfRows + warp, d4 = p.d / 4;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    if (warp < kFfRows) {
        float4 *xr = reinterpret_cast<float4 *>(xs) + (size_t)warp * d4;
        if (r >= p.R) {
            for (int i = lane; i < d4; i += 32) xr[i] = zero;
        } else {
            const float4 *x4 = reinterpret_cast<const float4 *>(p.x + (size_t)r * p.d), *q4 = nullptr;
            if (embed) {
                const int bs = r / p.M, j = r % p.M;
                int n = p.n_rows ? p.n_rows[bs] : p.M;
                n = max(0, min(n, p.M));
                const int len = p.len[bs];
                const bool fits = len + n <= p.S && (p.pos_limit == 0 || len + n <= p.pos_limit);
                int pos = len + j, lim = p.S - 1;
                if (p.pos_limit && p.pos_limit - 1 < lim) lim = p.pos_limit - 1;
                pos = min(pos, lim);
                int tok = fits && j < n ? p.tokens[(size_t)bs * p.tok_stride + j] : 0;  // rows that are not fed read nothing
                tok = max(0, min(tok, p.V - 1));
                x4 = reinterpret_cast<const float4 *>(p.tok_emb + (size_t)tok * p.d);
                if (p.learned_pos) q4 = reinterpret_cast<const float4 *>(p.pos_emb + (size_t)pos * p.d);
            }
            auto entry = [&](int i) {
                float4 v = __ldcg(x4 + i);
                if (q4) {
                    const float4 w = __ldg(q4 + i);
                    v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
                }
                return v;
            };
            const float4 *g4 = reinterpret_cast<const float4 *>(g), *b4 = reinterpret_cast<const float4 *>(b);
            float4 x[NR], gv[NR], bv[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                const int i = lane + 32 * k;
                x[k] = i < d4 ? entry(i) : zero;
                gv[k] = i < d4 ? __ldg(g4 + i) : zero;
                bv[k] = i < d4 && b ? __ldg(b4 + i) : zero;
            }
            double s1 = 0.0, s2 = 0.0;
            auto add = [&](const float4 &v) {
                s1 += ((double)v.x + (double)v.y) + ((double)v.z + (double)v.w);
                s2 += ((double)v.x * v.x + (double)v.y * v.y) + ((double)v.z * v.z + (double)v.w * v.w);
            };
#pragma unroll
            for (int k = 0; k < NR; ++k) add(x[k]);
            for (int i = lane + 32 * NR; i < d4; i += 32) add(entry(i));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            }
            const double mean = p.norm_kind == 0 ? s1 * p.inv_d : 0.0;
            double var = s2 * p.inv_d - mean * mean;
            if (var < 0.0) var = 0.0;
            const double rstd = rsqrt(var + (double)p.eps);
            const bool owner = embed && (int)blockIdx.x == r % (int)gridDim.x;
            auto emit = [&](int i, const float4 &v, const float4 &gg, const float4 &bb) {
                float4 y;
                y.x = (float)(((double)v.x - mean) * rstd * (double)gg.x + (double)bb.x);
                y.y = (float)(((double)v.y - mean) * rstd * (double)gg.y + (double)bb.y);
                y.z = (float)(((double)v.z - mean) * rstd * (double)gg.z + (double)bb.z);
                y.w = (float)(((double)v.w - mean) * rstd * (double)gg.w + (double)bb.w);
                xr[i] = y;
                if (owner) reinterpret_cast<float4 *>(p.x + (size_t)r * p.d)[i] = v;
            };
#pragma unroll
            for (int k = 0; k < NR; ++k)
                if (lane + 32 * k < d4) emit(lane + 32 * k, x[k], gv[k], bv[k]);
            for (int i = lane + 32 * NR; i < d4; i += 32) emit(i, entry(i), __ldg(g4 + i), b ? __ldg(b4 + i) : zero);
        }
    }
    __syncthreads();
}
// rows 8 rb .. of a [R, K] buffer into xs [8][K]
__device__ __forceinline__ void ff_stage(const FfParams &p, int rb, const float *src, int K, float *xs) {
    const int K4 = K / 4, rows = min(kFfRows, p.R - rb * kFfRows);
    const float4 *s4 = reinterpret_cast<const float4 *>(src + (size_t)rb * kFfRows * K);
    float4 *d4 = reinterpret_cast<float4 *>(xs);
#pragma unroll 4
    for (int i = threadIdx.x; i < kFfRows * K4; i += kFfThreads)
        d4[i] = i < rows * K4 ? __ldcg(s4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
}

// Attention of one (sequence, head): rotary, append, then scores, softmax and P V for eight rows at a time (their sums live in
// registers: arrays for all 32 rows a pass may have went through the stack, 50 us per 256 positions where eight rows take 8).
__device__ __forceinline__ void ff_attention(const FfParams &p, int layer, int item, bool append_only, float *smem) {
    const int b = item / p.H, h = item % p.H, Dh = p.Dh, d = p.d, M = p.M, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = p.ri.n_eff[b], len = p.len[b], r0 = b * M, half = p.rotary_dim / 2;
    float *qs = smem, *sc = qs + M * Dh, *fac = sc + kFfRows * kFfChunk, *run_m = fac + kFfRows, *run_l = run_m + kFfRows, *red = run_l + kFfRows;
    float *kc = p.cache + (size_t)layer * p.layer_elems + ((size_t)(b * 2) * p.H + h) * p.S * Dh;
    float *vc = kc + (size_t)p.H * p.S * Dh;
    for (int i = tid; i < M * Dh; i += kFfThreads) {
        const int m = i / Dh, e = i % Dh, r = r0 + m;
        const float *row = p.qkv + (size_t)r * 3 * d + h * Dh;
        float q = __ldcg(row + e), k = __ldcg(row + d + e);
        if (e < p.rotary_dim) {
            const int j = e < half ? e : e - half, o = e < half ? e + half : e - half;
            const float c = __ldcg(p.ri.rope_cos + (size_t)r * half + j), s = __ldcg(p.ri.rope_sin + (size_t)r * half + j);
            const float qo = __ldcg(row + o), ko = __ldcg(row + d + o);
            q = e < half ? q * c - qo * s : qo * s + q * c;
            k = e < half ? k * c - ko * s : ko * s + k * c;
        }
        qs[i] = q * p.scale;
        if (m < n) {
            kc[(size_t)(len + m) * Dh + e] = k;
            vc[(size_t)(len + m) * Dh + e] = __ldcg(row + 2 * d + e);
        }
    }
    if (append_only) return;
    const int groups = kFfThreads / Dh, ge = tid % Dh, gi = tid / Dh;
#pragma unroll 1
    for (int m0 = 0; m0 < M; m0 += kFfRows) {
    const int rows = min(kFfRows, M - m0), nb = max(0, min(n - m0, kFfRows)), end = nb > 0 ? len + m0 + nb : 0;
    if (tid < kFfRows) { run_m[tid] = -INFINITY; run_l[tid] = 0.f; }
    float o[kFfRows];
#pragma unroll
    for (int m = 0; m < kFfRows; ++m) o[m] = 0.f;
    __syncthreads();  // (the first time:) the appended rows are read back through the cache
    for (int t0 = 0; t0 < end; t0 += kFfChunk) {
        const int np = min(kFfChunk, end - t0);
        // scores: four lanes per position, each a quarter of the head in 16-byte pieces
        for (int pp = tid >> 2; pp < ((np + 7) & ~7); pp += kFfThreads / 4) {
            const int quarter = tid & 3;
            float s[kFfRows];
#pragma unroll
            for (int m = 0; m < kFfRows; ++m) s[m] = 0.f;
            if (pp < np) {
                const float4 *k4 = reinterpret_cast<const float4 *>(kc + (size_t)(t0 + pp) * Dh);
#pragma unroll 4
                for (int i = quarter; i < Dh / 4; i += 4) {
                    const float4 k = k4[i];
#pragma unroll
                    for (int m = 0; m < kFfRows; ++m) {
                        if (m < nb) {
                            const float4 q = reinterpret_cast<const float4 *>(qs + (m0 + m) * Dh)[i];
                            s[m] = fmaf(q.x, k.x, fmaf(q.y, k.y, fmaf(q.z, k.z, fmaf(q.w, k.w, s[m]))));
                        }
                    }
                }
            }
#pragma unroll
            for (int m = 0; m < kFfRows; ++m) {
                if (m < nb) {
                    float v = s[m];
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    if (quarter == (m & 3) && pp < np) sc[m * kFfChunk + pp] = t0 + pp <= len + m0 + m ? v : -INFINITY;
                }
            }
        }
        __syncthreads();
        for (int m = warp; m < nb; m += kFfWarps) {  // running softmax statistics: one warp per row
            float v[kFfChunk / 32], mx = run_m[m];
            const float old = mx;
#pragma unroll
            for (int i = 0; i < kFfChunk / 32; ++i) {
                v[i] = lane + 32 * i < np ? sc[m * kFfChunk + lane + 32 * i] : -INFINITY;
                mx = fmaxf(mx, v[i]);
            }
            mx = warp_max(mx);
            float sum = 0.f;
#pragma unroll
            for (int i = 0; i < kFfChunk / 32; ++i) {
                const float e = mx > -INFINITY ? __expf(v[i] - mx) : 0.f;
                if (lane + 32 * i < np) sc[m * kFfChunk + lane + 32 * i] = e;
                sum += e;
            }
            sum = warp_sum(sum);
            if (lane == 0) {
                const float f = mx > -INFINITY ? __expf(old - mx) : 1.f;  // 0 on the first non-empty step
                fac[m] = f;
                run_m[m] = mx;
                run_l[m] = run_l[m] * f + sum;
            }
        }
        __syncthreads();
        if (gi < groups) {
#pragma unroll
            for (int m = 0; m < kFfRows; ++m)
                if (m < nb) o[m] *= fac[m];
#pragma unroll 4
            for (int pp = gi; pp < np; pp += groups) {
                const float v = vc[(size_t)(t0 + pp) * Dh + ge];
#pragma unroll
                for (int m = 0; m < kFfRows; ++m)
                    if (m < nb) o[m] = fmaf(sc[m * kFfChunk + pp], v, o[m]);
            }
        }
        __syncthreads();  // the scores are overwritten by the next step
    }
    if (gi < groups) {
#pragma unroll
        for (int m = 0; m < kFfRows; ++m)
            if (m < nb) red[(gi * kFfRows + m) * Dh + ge] = o[m];
    }
    __syncthreads();
    for (int i = tid; i < rows * Dh; i += kFfThreads) {
        const int m = i / Dh, e = i % Dh;
        float v = 0.f;
        if (m < nb) {
            for (int k = 0; k < groups; ++k) v += red[(k * kFfRows + m) * Dh + e];
            const float L = run_l[m];
            v = L > 0.f ? v / L : 0.f;
        }
        p.ao[(size_t)(r0 + m0 + m) * d + h * Dh + e] = v;
    }
    __syncthreads();
    }
}

// The steps of a pass.  Sequential layer: qkv | attention | out-projection | MLP in | MLP out; parallel-residual layer: qkv, MLP in |
// attention | out-projection, MLP out (a bar is a grid barrier); at the end the LM head.  One loop over them, so that staging
// and projection exist once in the code: a phase runs a few hundred instructions per warp, and fetching them would cost more.
enum { FS_QKV = 0, FS_ATTN, FS_O, FS_IN, FS_OUT, FS_LM };
struct FfStep {
    const float *W, *bias, *src;  // projection: weights, bias, operand rows (null: the norm of the residual stream with g, b)
    const float *g, *b;
    int N, K4, kind;
    bool barrier;                 // behind it
};
__device__ __forceinline__ FfStep ff_step(const FfParams &p, int i) {
    FfStep s;
    const int l = i / 5, e = i % 5;
    if (l >= p.n_layers) {
        s.kind = FS_LM;
        s.W = p.w_lm; s.bias = nullptr; s.src = nullptr; s.g = p.lnf_g; s.b = p.lnf_b; s.N = p.V; s.K4 = p.d / 4; s.barrier = false;
        return s;
    }
    const FfLayer &L = p.layer[l];
    s.kind = !p.parallel ? e : e == 0 ? FS_QKV : e == 1 ? FS_IN : e == 2 ? FS_ATTN : e == 3 ? FS_O : FS_OUT;
    s.barrier = !(p.parallel && (e == 0 || e == 3));
    s.K4 = p.d / 4; s.src = nullptr; s.g = s.b = nullptr; s.W = nullptr; s.bias = nullptr; s.N = 0;
    if (s.kind == FS_QKV) { s.W = L.w_qkv; s.bias = L.b_qkv; s.g = L.ln1_g; s.b = L.ln1_b; s.N = 3 * p.d; }
    if (s.kind == FS_O) { s.W = L.w_o; s.bias = L.b_o; s.src = p.ao; s.N = p.d; }
    if (s.kind == FS_IN) { s.W = L.w_in; s.bias = L.b_in; s.g = L.ln2_g; s.b = L.ln2_b; s.N = p.F; }
    if (s.kind == FS_OUT) { s.W = L.w_out; s.bias = L.b_out; s.src = p.act; s.N = p.d; s.K4 = p.F / 4; }
    return s;
}
// one projected value to where the step wants it
__device__ __forceinline__ void ff_out(const FfParams &p, const FfStep &s, int n, int row, float v) {
    if (s.bias) v += __ldg(s.bias + n);
    if (s.kind == FS_QKV) p.qkv[(size_t)row * 3 * p.d + n] = v;
    else if (s.kind == FS_IN) p.act[(size_t)row * p.F + n] = gelu_erf(v);
    else if (s.kind == FS_LM) p.logits[(size_t)row * p.V + n] = v;
    else {  // the residual stream: this thread owns the entry in both projections that add to it
        float *x = p.x + (size_t)row * p.d + n;
        *x = __ldcg(x) + v;
    }
}

__device__ __forceinline__ void ff_forward(const FfParams &p, float *xs, volatile int &ok) {
    const float4 *xs4 = reinterpret_cast<const float4 *>(xs);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r8 = lane >> 2;
    const int blocks = (p.R + kFfRows - 1) / kFfRows;
    const int gw = blockIdx.x * kFfWarps + warp, nw = gridDim.x * kFfWarps;  // this warp's columns: gw, gw + nw, ...
    unsigned epoch = 0;
    if (threadIdx.x == 0) ok = 1;

    // Four columns at a time where a warp has several and their rows are short; gate and up together for SwiGLU; else one.
    float4 pre[8];
    auto columns = [&](const FfStep &s) { return s.kind == FS_IN && p.swiglu ? 2 : s.N > nw && s.K4 <= 64 ? 4 : 1; };
    auto fetch = [&](const FfStep &s, int n) {
        const int nf = columns(s);
        if (n >= s.N) return;
        if (nf == 4) ff_fetch<4>(s.W, n, nw, s.N, s.K4, 0, pre);
        else if (nf == 2) ff_fetch<2>(s.W, n, p.F, 2 * p.F, s.K4, 0, pre);
        else ff_fetch<1>(s.W, n, nw, s.N, s.K4, 0, pre);
    };

    ff_stamp(p, 0);
    FfStep s = ff_step(p, 0);
    fetch(s, gw);
    // row bookkeeping and the rotary table (read behind the first barrier)
    {
        const int half = p.rotary_dim / 2;
        for (int r = blockIdx.x; r < p.R; r += gridDim.x) {
            const int b = r / p.M, j = r % p.M;
            int n = p.n_rows ? p.n_rows[b] : p.M;
            n = max(0, min(n, p.M));
            const int len = p.len[b];
            if (!(len + n <= p.S && (p.pos_limit == 0 || len + n <= p.pos_limit))) {
                n = 0;
                if (threadIdx.x == 0) set_status(p.status, -3);
            }
            int pos = len + j, lim = p.S - 1;
            if (p.pos_limit && p.pos_limit - 1 < lim) lim = p.pos_limit - 1;
            pos = min(pos, lim);
            if (threadIdx.x == 0) {
                p.ri.seq[r] = b;
                p.ri.pos[r] = pos;
                p.ri.valid[r] = j < n;
                if (j == 0) p.ri.n_eff[b] = n;
            }
            for (int i = threadIdx.x; i < half; i += kFfThreads) {
                double sn, c;
                sincos((double)pos * exp2(-2.0 * i / p.rotary_dim * log2((double)p.rotary_base)), &sn, &c);
                p.ri.rope_cos[(size_t)r * half + i] = (float)c;
                p.ri.rope_sin[(size_t)r * half + i] = (float)sn;
            }
        }
    }
    const int steps = 5 * p.n_layers + 1;
#pragma unroll 1
    for (int i = 0; i < steps; ++i) {
        const bool last = i >= 5 * (p.n_layers - 1) && !p.want_logits;  // of the last layer only the keys and values are wanted
        bool fetched = true;                                            // this warp's first columns
        if (s.kind == FS_ATTN) {
            for (int item = blockIdx.x; item < p.B * p.H; item += gridDim.x) ff_attention(p, i / 5, item, last, xs);
            if (last) return;
        } else if (!(last && s.kind == FS_IN)) {
#pragma unroll 1
            for (int rb = 0; rb < blocks; ++rb) {
                __syncthreads();  // the staged rows of before have been read
                if (s.src) ff_stage(p, rb, s.src, 4 * s.K4, xs);
                else ff_stage_norm(p, rb, i < 5 && (s.kind == FS_QKV || p.parallel), s.g, s.b, xs);
                const int rows = min(kFfRows, p.R - rb * kFfRows), row = rb * kFfRows + r8, nf = columns(s);
                const bool writes = (lane & 3) == 0 && r8 < rows;
#pragma unroll 1
                for (int n = gw; n < s.N; n += nf == 4 ? 4 * nw : nw) {
                    if (!fetched) fetch(s, n);
                    fetched = false;
                    if (nf == 4) {
                        float acc[4][kFfRows];
                        ff_dot<4>(s.W, n, nw, s.N, s.K4, xs4, rows, pre, acc);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float v = ff_reduce(acc[j]);
                            if (writes && n + j * nw < s.N) ff_out(p, s, n + j * nw, row, v);
                        }
                    } else if (nf == 1) {
                        float acc[1][kFfRows];
                        ff_dot<1>(s.W, n, nw, s.N, s.K4, xs4, rows, pre, acc);
                        const float v = ff_reduce(acc[0]);
                        if (writes) ff_out(p, s, n, row, v);
                    } else {
                        float acc[2][kFfRows];
                        ff_dot<2>(s.W, n, p.F, 2 * p.F, s.K4, xs4, rows, pre, acc);
                        const float g = ff_reduce(acc[0]) + (s.bias ? __ldg(s.bias + n) : 0.f);
                        const float u = ff_reduce(acc[1]) + (s.bias ? __ldg(s.bias + p.F + n) : 0.f);
                        if (writes) p.act[(size_t)row * p.F + n] = silu(g) * u;
                    }
                }
                fetched = false;
            }
        }
        const bool barrier = s.barrier;
        if (i + 1 < steps) {
            s = ff_step(p, i + 1);
            if (s.kind != FS_ATTN) fetch(s, gw);  // ahead of the barrier
        }
        if (barrier && !ff_sync(p, epoch, &ok)) return;
    }
    ff_stamp(p, epoch + 1);
}

// (The same kernel as one cluster of 16 CTAs, with the cluster's hardware barrier instead of the counter in L2, gains what the
// barriers cost and loses it again to 16 SMs' share of the projections: 124 us for four layers and 5 rows against 128 on 64
// CTAs, 31 against 30 for one layer and one row.)
__global__ void __launch_bounds__(kFfThreads, 1) forward_f32_kernel(const __grid_constant__ FfParams p) {
    extern __shared__ __align__(16) float ff_smem_[];
    __shared__ volatile int ok;
    ff_forward(p, ff_smem_, ok);
    __syncthreads();
    if (threadIdx.x == 0) leave_grid(p.gbar);
}

}  // namespace ssd
