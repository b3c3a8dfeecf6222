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
// Generation with the four-layer 256-wide model (K = 4, 16 iterations): 13.2 ms as one launch per step, 6.5 as one
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
constexpr int kFfRows = 8;              // activation rows a warp sums at a time
constexpr int kFfMaxLayers = 32;        // (their tensors' addresses ride in the kernel parameters)
constexpr int kFfMaxSmem = 200 * 1024;
constexpr int kFfChunk = 256;           // positions per attention step
// An item walks its positions alone: beyond this many the stepwise path's split over CTAs is the faster form
// (a 256-position step costs about 3 us, the split path's three launches about 20).
constexpr int kFfMaxCtx = 1536;

struct FfLayer {
    const float *ln1_g, *ln1_b, *w_qkv, *b_qkv, *w_o, *b_o, *ln2_g, *ln2_b, *w_in, *b_in, *w_out, *b_out;
};
struct FfParams {
    int n_layers, d, H, Dh, F, V, norm_kind, swiglu, parallel, rotary_dim, learned_pos, pos_limit;
    float eps, rotary_base, scale;
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
inline size_t ff_smem(int d, int F, int parallel, int M, int Dh) {
    const size_t gemm = (size_t)kFfRows * (parallel ? d + F : (d > F ? d : F)) * 4;
    const size_t groups = kFfThreads / Dh;
    const size_t attn = ((size_t)M * Dh + (size_t)M * kFfChunk + 3 * (size_t)M + groups * M * Dh) * 4;
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
    __syncthreads();
    ++epoch;
    if (threadIdx.x == 0) {
        __threadfence();
        red_release_add(p.gbar, 1u);
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
        __threadfence();
        ff_stamp(p, epoch);
    }
    __syncthreads();
    return *ok != 0;
}

// the first 1024 entries of a weight row
__device__ __forceinline__ void ff_fetch(const float4 *w, int K4, float4 (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = lane + 32 * i < K4 ? __ldg(w + lane + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
}
// sum_k w[k] x[r][k] for the eight staged rows; `v` holds the first 1024 entries of w (and is used up)
__device__ __forceinline__ void ff_dot(const float4 *w, int K4, const float4 *xs, float4 (&v)[8], float (&acc)[kFfRows]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < kFfRows; ++r) acc[r] = 0.f;
    for (int k0 = 0;;) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = k0 + lane + 32 * i;
            if (k0 + 32 * i >= K4) break;
            if (k < K4) {
#pragma unroll
                for (int r = 0; r < kFfRows; ++r) {
                    const float4 x = xs[(size_t)r * K4 + k];
                    acc[r] = fmaf(v[i].x, x.x, acc[r]);
                    acc[r] = fmaf(v[i].y, x.y, acc[r]);
                    acc[r] = fmaf(v[i].z, x.z, acc[r]);
                    acc[r] = fmaf(v[i].w, x.w, acc[r]);
                }
            }
        }
        k0 += 256;
        if (k0 >= K4) break;
        ff_fetch(w + k0, K4 - k0, v);
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

// Rows 8 rb .. of the residual stream, normalised, into xs [8][d]: a warp per row.  `embed`: they are embedding rows
// (and their owner starts the residual stream with them).
__device__ __forceinline__ void ff_stage_norm(const FfParams &p, int rb, bool embed, const float *g, const float *b, float *xs) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = rb * kFfRows + warp, d = p.d;
    if (warp < kFfRows) {
        float *xr = xs + (size_t)warp * d;
        if (r >= p.R) {
            for (int i = lane; i < d; i += 32) xr[i] = 0.f;
        } else {
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
                const float4 *e = reinterpret_cast<const float4 *>(p.tok_emb + (size_t)tok * d);
                const float4 *q = p.learned_pos ? reinterpret_cast<const float4 *>(p.pos_emb + (size_t)pos * d) : nullptr;
                for (int i = lane; i < d / 4; i += 32) {
                    float4 v = __ldg(e + i);
                    if (q) {
                        const float4 w = __ldg(q + i);
                        v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
                    }
                    reinterpret_cast<float4 *>(xr)[i] = v;
                    if ((int)blockIdx.x == r % (int)gridDim.x) reinterpret_cast<float4 *>(p.x + (size_t)r * d)[i] = v;
                }
            } else {
                const float4 *x4 = reinterpret_cast<const float4 *>(p.x + (size_t)r * d);
#pragma unroll 4
                for (int i = lane; i < d / 4; i += 32) reinterpret_cast<float4 *>(xr)[i] = __ldcg(x4 + i);
            }
            __syncwarp();
            double s1 = 0.0, s2 = 0.0;
            for (int i = lane; i < d; i += 32) {
                const double v = (double)xr[i];
                s1 += v;
                s2 += v * v;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            }
            const double mean = p.norm_kind == 0 ? s1 / d : 0.0;
            double var = s2 / d - mean * mean;
            if (var < 0.0) var = 0.0;
            const double rstd = rsqrt(var + (double)p.eps);
            for (int i = lane; i < d; i += 32) {
                double y = ((double)xr[i] - mean) * rstd * (double)__ldg(g + i);
                if (b) y += (double)__ldg(b + i);
                xr[i] = (float)y;
            }
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

// What a CTA will read behind the next barrier and nobody writes before it: into L1, under the wait.
__device__ __forceinline__ void ff_prefetch_norm(const FfParams &p, const float *g, const float *b) {
    for (int i = threadIdx.x * 32; i < p.d; i += kFfThreads * 32) {
        prefetch_l1(g + i);
        if (b) prefetch_l1(b + i);
    }
}
__device__ __forceinline__ void ff_prefetch_cache(const FfParams &p, int layer, int item) {
    if (item >= p.B * p.H) return;
    const int b = item / p.H, h = item % p.H, n = min(p.len[b], kFfChunk) * p.Dh;  // (the committed positions of the first step)
    const float *kc = p.cache + (size_t)layer * p.layer_elems + ((size_t)(b * 2) * p.H + h) * p.S * p.Dh, *vc = kc + (size_t)p.H * p.S * p.Dh;
    for (int i = threadIdx.x * 32; i < n; i += kFfThreads * 32) {
        prefetch_l1(kc + i);
        prefetch_l1(vc + i);
    }
}

// Attention of one (sequence, head): rotary, append, scores, softmax, P V.  MR bounds the rows per sequence.
template <int MR>
__device__ __forceinline__ void ff_attention(const FfParams &p, int layer, int item, bool append_only, float *smem) {
    const int b = item / p.H, h = item % p.H, Dh = p.Dh, d = p.d, M = p.M, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = p.ri.n_eff[b], len = p.len[b], r0 = b * M, half = p.rotary_dim / 2;
    float *qs = smem, *sc = qs + M * Dh, *fac = sc + M * kFfChunk, *run_m = fac + M, *run_l = run_m + M, *red = run_l + M;
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
    if (tid < M) { run_m[tid] = -INFINITY; run_l[tid] = 0.f; }
    const int groups = kFfThreads / Dh, ge = tid % Dh, gi = tid / Dh;
    float o[MR];
#pragma unroll
    for (int m = 0; m < MR; ++m) o[m] = 0.f;
    const int end = len + n;
    __syncthreads();  // the appended rows are read back through the cache
    for (int t0 = 0; t0 < end; t0 += kFfChunk) {
        const int np = min(kFfChunk, end - t0);
        // scores: four lanes per position, each a quarter of the head in 16-byte pieces
        for (int pp = tid >> 2; pp < ((np + 7) & ~7); pp += kFfThreads / 4) {
            const int quarter = tid & 3;
            float s[MR];
#pragma unroll
            for (int m = 0; m < MR; ++m) s[m] = 0.f;
            if (pp < np) {
                const float4 *k4 = reinterpret_cast<const float4 *>(kc + (size_t)(t0 + pp) * Dh);
#pragma unroll 4
                for (int i = quarter; i < Dh / 4; i += 4) {
                    const float4 k = k4[i];
#pragma unroll
                    for (int m = 0; m < MR; ++m) {
                        if (m < n) {
                            const float4 q = reinterpret_cast<const float4 *>(qs + m * Dh)[i];
                            s[m] = fmaf(q.x, k.x, fmaf(q.y, k.y, fmaf(q.z, k.z, fmaf(q.w, k.w, s[m]))));
                        }
                    }
                }
            }
#pragma unroll
            for (int m = 0; m < MR; ++m) {
                if (m < n) {
                    float v = s[m];
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    if (quarter == (m & 3) && pp < np) sc[m * kFfChunk + pp] = t0 + pp <= len + m ? v : -INFINITY;
                }
            }
        }
        __syncthreads();
        for (int m = warp; m < n; m += kFfWarps) {  // running softmax statistics: one warp per row
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
            for (int m = 0; m < MR; ++m)
                if (m < n) o[m] *= fac[m];
#pragma unroll 4
            for (int pp = gi; pp < np; pp += groups) {
                const float v = vc[(size_t)(t0 + pp) * Dh + ge];
#pragma unroll
                for (int m = 0; m < MR; ++m)
                    if (m < n) o[m] = fmaf(sc[m * kFfChunk + pp], v, o[m]);
            }
        }
        __syncthreads();  // the scores are overwritten by the next step
    }
    if (gi < groups) {
#pragma unroll
        for (int m = 0; m < MR; ++m)
            if (m < n) red[((size_t)gi * M + m) * Dh + ge] = o[m];
    }
    __syncthreads();
    for (int i = tid; i < M * Dh; i += kFfThreads) {
        const int m = i / Dh, e = i % Dh;
        float v = 0.f;
        if (m < n) {
            for (int k = 0; k < groups; ++k) v += red[((size_t)k * M + m) * Dh + e];
            const float L = run_l[m];
            v = L > 0.f ? v / L : 0.f;
        }
        p.ao[(size_t)(r0 + m) * d + h * Dh + e] = v;
    }
    __syncthreads();
}

template <int MR>
__device__ __forceinline__ void ff_forward(const FfParams &p, float *xs, volatile int &ok) {
    const float4 *xs4 = reinterpret_cast<const float4 *>(xs);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r8 = lane >> 2;
    const int d = p.d, F = p.F, d4 = d / 4, F4 = F / 4, blocks = (p.R + kFfRows - 1) / kFfRows;
    const int gw = blockIdx.x * kFfWarps + warp, nw = gridDim.x * kFfWarps;  // this warp's first column, and the stride
    unsigned epoch = 0;
    if (threadIdx.x == 0) ok = 1;

    float4 pre[8];
    auto fetch = [&](const float *W, int N, int K4) {  // of the next phase's first column
        if (gw < N) ff_fetch(reinterpret_cast<const float4 *>(W + (size_t)gw * K4 * 4), K4, pre);
    };
    // out(n, row in block, value) for every column n of W [N, K] and the staged rows
    auto project = [&](const float *W, int N, int K4, const float4 *x4, bool fetched, auto out) {
        for (int n = gw; n < N; n += nw) {
            const float4 *w = reinterpret_cast<const float4 *>(W + (size_t)n * K4 * 4);
            if (!fetched || n != gw) ff_fetch(w, K4, pre);
            float acc[kFfRows];
            ff_dot(w, K4, x4, pre, acc);
            const float v = ff_reduce(acc);
            if ((lane & 3) == 0) out(n, r8, v);
        }
    };
    auto mlp_in = [&](const FfLayer &L, int rb, bool fetched) {
        if (!p.swiglu) {
            project(L.w_in, F, d4, xs4, fetched, [&](int n, int r, float v) {
                if (rb * kFfRows + r < p.R) p.act[(size_t)(rb * kFfRows + r) * F + n] = gelu_erf(v + (L.b_in ? __ldg(L.b_in + n) : 0.f));
            });
        } else {
            for (int n = gw; n < F; n += nw) {
                const float4 *wg = reinterpret_cast<const float4 *>(L.w_in + (size_t)n * d), *wu = wg + (size_t)F * d4;
                if (!fetched || n != gw) ff_fetch(wg, d4, pre);
                float acc[kFfRows];
                ff_dot(wg, d4, xs4, pre, acc);
                ff_fetch(wu, d4, pre);
                const float gv = ff_reduce(acc) + (L.b_in ? __ldg(L.b_in + n) : 0.f);
                ff_dot(wu, d4, xs4, pre, acc);
                const float uv = ff_reduce(acc) + (L.b_in ? __ldg(L.b_in + F + n) : 0.f);
                const int r = rb * kFfRows + r8;
                if ((lane & 3) == 0 && r < p.R) p.act[(size_t)r * F + n] = silu(gv) * uv;
            }
        }
    };
    auto add_to_x = [&](int rb, int n, int r, float v, const float *bias) {
        const int row = rb * kFfRows + r;
        if (row < p.R) {
            float *x = p.x + (size_t)row * d + n;
            *x = __ldcg(x) + (v + (bias ? __ldg(bias + n) : 0.f));
        }
    };

    ff_stamp(p, 0);
    fetch(p.layer[0].w_qkv, 3 * d, d4);
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
                double s, c;
                sincos((double)pos * exp2(-2.0 * i / p.rotary_dim * log2((double)p.rotary_base)), &s, &c);
                p.ri.rope_cos[(size_t)r * half + i] = (float)c;
                p.ri.rope_sin[(size_t)r * half + i] = (float)s;
            }
        }
    }
    for (int l = 0; l < p.n_layers; ++l) {
        const FfLayer &L = p.layer[l];
        const bool last = l + 1 == p.n_layers && !p.want_logits;  // only its keys and values are wanted
        for (int rb = 0; rb < blocks; ++rb) {
            if (rb) __syncthreads();
            ff_stage_norm(p, rb, l == 0, L.ln1_g, L.ln1_b, xs);
            project(L.w_qkv, 3 * d, d4, xs4, rb == 0, [&](int n, int r, float v) {
                if (rb * kFfRows + r < p.R) p.qkv[(size_t)(rb * kFfRows + r) * 3 * d + n] = v + (L.b_qkv ? __ldg(L.b_qkv + n) : 0.f);
            });
            if (p.parallel && !last) {
                __syncthreads();
                ff_stage_norm(p, rb, l == 0, L.ln2_g, L.ln2_b, xs);
                mlp_in(L, rb, false);
            }
        }
        ff_prefetch_cache(p, l, blockIdx.x);
        if (!ff_sync(p, epoch, &ok)) return;
        for (int item = blockIdx.x; item < p.B * p.H; item += gridDim.x) ff_attention<MR>(p, l, item, last, xs);
        if (last) return;
        fetch(L.w_o, d, d4);
        if (!ff_sync(p, epoch, &ok)) return;
        if (p.parallel) {
            float *xf = xs + (size_t)kFfRows * d;
            for (int rb = 0; rb < blocks; ++rb) {
                if (rb) __syncthreads();
                ff_stage(p, rb, p.ao, d, xs);
                ff_stage(p, rb, p.act, F, xf);
                for (int n = gw; n < d; n += nw) {
                    const float4 *wo = reinterpret_cast<const float4 *>(L.w_o + (size_t)n * d), *wf = reinterpret_cast<const float4 *>(L.w_out + (size_t)n * F);
                    if (rb || n != gw) ff_fetch(wo, d4, pre);
                    float acc[kFfRows];
                    ff_dot(wo, d4, xs4, pre, acc);
                    ff_fetch(wf, F4, pre);
                    const float av = ff_reduce(acc);
                    ff_dot(wf, F4, reinterpret_cast<const float4 *>(xf), pre, acc);
                    const float fv = ff_reduce(acc) + (L.b_out ? __ldg(L.b_out + n) : 0.f);
                    if ((lane & 3) == 0) add_to_x(rb, n, r8, av + fv, L.b_o);
                }
            }
        } else {
            for (int rb = 0; rb < blocks; ++rb) {
                if (rb) __syncthreads();
                ff_stage(p, rb, p.ao, d, xs);
                project(L.w_o, d, d4, xs4, rb == 0, [&](int n, int r, float v) { add_to_x(rb, n, r, v, L.b_o); });
            }
            fetch(L.w_in, F, d4);
            ff_prefetch_norm(p, L.ln2_g, L.ln2_b);
            if (!ff_sync(p, epoch, &ok)) return;
            for (int rb = 0; rb < blocks; ++rb) {
                if (rb) __syncthreads();
                ff_stage_norm(p, rb, false, L.ln2_g, L.ln2_b, xs);
                mlp_in(L, rb, rb == 0);
            }
            fetch(L.w_out, d, F4);
            if (!ff_sync(p, epoch, &ok)) return;
            for (int rb = 0; rb < blocks; ++rb) {
                if (rb) __syncthreads();
                ff_stage(p, rb, p.act, F, xs);
                project(L.w_out, d, F4, xs4, rb == 0, [&](int n, int r, float v) { add_to_x(rb, n, r, v, L.b_out); });
            }
        }
        if (l + 1 < p.n_layers) {
            fetch(p.layer[l + 1].w_qkv, 3 * d, d4);
            ff_prefetch_norm(p, p.layer[l + 1].ln1_g, p.layer[l + 1].ln1_b);
        } else {
            fetch(p.w_lm, p.V, d4);
            ff_prefetch_norm(p, p.lnf_g, p.lnf_b);
        }
        if (!ff_sync(p, epoch, &ok)) return;
    }
    for (int rb = 0; rb < blocks; ++rb) {
        if (rb) __syncthreads();
        ff_stage_norm(p, rb, false, p.lnf_g, p.lnf_b, xs);
        project(p.w_lm, p.V, d4, xs4, rb == 0, [&](int n, int r, float v) {
            if (rb * kFfRows + r < p.R) p.logits[(size_t)(rb * kFfRows + r) * p.V + n] = v;
        });
    }
    ff_stamp(p, epoch + 1);
}

template <int MR>
__global__ void __launch_bounds__(kFfThreads, 1) forward_f32_kernel(const __grid_constant__ FfParams p) {
    extern __shared__ __align__(16) float ff_smem_[];
    __shared__ volatile int ok;
    ff_forward<MR>(p, ff_smem_, ok);
    __syncthreads();
    if (threadIdx.x == 0) leave_grid(p.gbar);
}

}  // namespace ssd
