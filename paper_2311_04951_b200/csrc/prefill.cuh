// Prompt pass over many rows at once (Section "KV Caching", Figure 1: the pass that fills the cache before
// sampling starts).  With hundreds or thousands of rows per forward the linear layers are compute-bound: this
// file holds the two kernels that differ from the few-row path - a tiled tcgen05 GEMM over 128 activation rows
// x 256 weight rows per CTA, and a causal attention over row tiles whose keys / values all sit in the cache -
// with the norm and the rotary / append / query steps at memory speed; set-up and embedding are the stepwise path's kernels,
// which take any number of rows.
//
// prefill_gemm_kernel:  out[r, n] += sum_k (Xhi[r, k] + Xlo[r, k]) * W[n, k]
//   * output tiles of 128 rows x 256 columns, dealt round-robin to one CTA per SM; 320 threads: warp 0 = TMA
//     producer, warp 1 = MMA issuer, warps 2-9 = epilogue (a tensor-memory lane quadrant and half of the columns each:
//     with four warps the 128 x 256 GELUs of a tile took longer than the next tile's products: 929 us where eight take
//     690, 8184 rows x 2560 -> 10240); two accumulators in tensor memory (2 x 256 columns), so a tile's epilogue runs under the next tile's products;
//   * a stage of the shared-memory ring = the activation rows' hi tile and lo tile (128 rows x 64 k, bf16) and
//     the weight tile (256 rows x 64 k), all by 2-D tensor-map copies with the 128-byte swizzle, 64 KB;
//   * per stage eight tcgen05.mma (M = 128, N = 256, K = 16): four k-steps with the hi tile, four with the lo
//     tile, into ONE fp32 accumulator in tensor memory: W hi + W lo is the fp32-activation product to ~2^-17,
//     the same arithmetic as the few-row path (the price is half the tensor throughput);
//   * the tile is owned by this CTA alone (no split over k), so the epilogue writes accumulator + bias over the
//     output, adds them to it (the residual stream), or - the MLP's input projection - applies the activation and writes the
//     next projection's bf16 hi / lo operand, all with plain loads and stores under the next tile's products.  For SwiGLU a
//     weight tile is 128 gate rows and the 128 up rows of the same columns.  (8184 rows x 2560 -> 10240: 690 us; with the
//     fp32 pre-activations written and read back by a kernel of its own 640 + 138.)
// Every wait is bounded; on time-out the kernel records SSD_E_TIMEOUT, drains its copies and returns.
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "gemm.cuh"
#include "persistent.cuh"
#include "rowops.cuh"

namespace ssd {

constexpr int kPfTileM = 128, kPfTileN = 256, kPfStages = 3;
constexpr int kPfABytes = kPfTileM * kTileK * 2;            // 16 KB: one of hi / lo
constexpr int kPfWBytes = kPfTileN * kTileK * 2;            // 32 KB
constexpr int kPfStageBytes = 2 * kPfABytes + kPfWBytes;    // 64 KB
constexpr int kPfEpiWarps = 8, kPfThreads = 64 + 32 * kPfEpiWarps;
constexpr size_t kPfSmem = 1024 + (size_t)kPfStages * kPfStageBytes + 256;  // + barriers, TMEM slot, abort flag

// eight values as bf16 hi + lo, 16 bytes each
__device__ __forceinline__ void split_hilo8(const float (&y)[8], uint4 &hi, uint4 &lo) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 hv = __floats2bfloat162_rn(y[2 * i], y[2 * i + 1]);
        h[i] = *reinterpret_cast<const uint32_t *>(&hv);
        l[i] = pack_bf16x2(y[2 * i] - __low2float(hv), y[2 * i + 1] - __high2float(hv));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

enum { PF_WRITE = 0,   // out = X W^T + bias
       PF_ADD,         // out += X W^T + bias (the residual stream)
       PF_GELU,        // act = GELU(X W^T + bias), as bf16 hi + lo
       PF_SWIGLU };    // act = SiLU(gate) * up
struct PfGemmArgs {
    float *out;         // [R, ldo] fp32
    const float *bias;  // [N] or null
    int mode;           // PF_*
    int ldo, N, Kd, R;  // N = output columns (SwiGLU: half of W's rows)
    __nv_bfloat16 *act_hi, *act_lo;  // PF_GELU / PF_SWIGLU: [R, N] row-major
    long long wait_cycles;  // bound of every wait that takes work
    int32_t *status;
};

__global__ void __launch_bounds__(kPfThreads, 1)
prefill_gemm_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmXhi,
                    const __grid_constant__ CUtensorMap tmXlo, const PfGemmArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + (size_t)kPfStages * kPfStageBytes);
    uint64_t *empty = full + kPfStages;
    uint64_t *acc_full = empty + kPfStages;  // [2]
    uint64_t *acc_empty = acc_full + 2;      // [2]
    uint32_t *tmem_slot = (uint32_t *)(acc_empty + 2);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kchunks = (a.Kd + kTileK - 1) / kTileK;
    const int cols = a.mode == PF_SWIGLU ? kPfTileN / 2 : kPfTileN;  // output columns of a tile
    const int tiles_m = (a.R + kPfTileM - 1) / kPfTileM, tiles_n = (a.N + cols - 1) / cols;
    const int n_tiles = tiles_m * tiles_n;
    // this CTA's tiles: blockIdx.x, + gridDim.x, ...; row tiles vary fastest, so the CTAs that run together share
    // weight tiles in L2 (the activations of all rows stay there anyway)

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "n"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < kPfStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&acc_full[i], 1);
            mbar_init(&acc_empty[i], kPfEpiWarps);  // one arrival per epilogue warp
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    int issued = 0;  // stage fills issued by the producer thread
    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            for (int tile = blockIdx.x; ok && tile < n_tiles; tile += gridDim.x) {
                const int m0 = (tile % tiles_m) * kPfTileM, n0 = (tile / tiles_m) * cols;
                for (int kc = 0; kc < kchunks; ++kc, ++issued) {
                    const int s = issued % kPfStages;
                    if (*abort_flag ||
                        (issued >= kPfStages && !mbar_wait_limit(&empty[s], ((issued / kPfStages) - 1) & 1, a.wait_cycles))) {
                        ok = false;
                        break;
                    }
                    uint8_t *st = smem + (size_t)s * kPfStageBytes;
                    mbar_expect_tx(&full[s], kPfStageBytes);
                    tma_load_2d(st, &tmXhi, kc * kTileK, m0, &full[s]);
                    tma_load_2d(st + kPfABytes, &tmXlo, kc * kTileK, m0, &full[s]);
                    tma_load_2d(st + 2 * kPfABytes, &tmW, kc * kTileK, n0, &full[s]);
                    if (a.mode == PF_SWIGLU)  // (the map's box is 128 rows: gate above, up here)
                        tma_load_2d(st + 2 * kPfABytes + kPfWBytes / 2, &tmW, kc * kTileK, a.N + n0, &full[s]);
                }
            }
            if (!ok) {
                set_status(a.status, kTimeoutCode);
                *abort_flag = 1;
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = umma_idesc_bf16(kPfTileM, kPfTileN);
            bool ok = true;
            int it = 0, j = 0;
            for (int tile = blockIdx.x; ok && tile < n_tiles; tile += gridDim.x, ++j) {
                const int buf = j & 1;
                if (j >= 2 && !mbar_wait_limit(&acc_empty[buf], ((j >> 1) - 1) & 1, 4 * a.wait_cycles)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d_tmem = tmem + (uint32_t)(buf * kPfTileN);
                for (int kc = 0; kc < kchunks; ++kc, ++it) {
                    const int s = it % kPfStages;
                    if (*abort_flag || !mbar_wait_limit(&full[s], (it / kPfStages) & 1, a.wait_cycles)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t st = smem_u32(smem + (size_t)s * kPfStageBytes);
                    const uint64_t hi = umma_desc_sw128(st), lo = umma_desc_sw128(st + kPfABytes), w = umma_desc_sw128(st + 2 * kPfABytes);
#pragma unroll
                    for (int ks = 0; ks < kTileK / 16; ++ks) tc_mma_bf16(d_tmem, hi + 2 * ks, w + 2 * ks, idesc, (kc | ks) ? 1u : 0u);
#pragma unroll
                    for (int ks = 0; ks < kTileK / 16; ++ks) tc_mma_bf16(d_tmem, lo + 2 * ks, w + 2 * ks, idesc, 1u);
                    tc_commit(&empty[s]);
                }
                if (ok) tc_commit(&acc_full[buf]);
            }
            if (!ok) {
                set_status(a.status, kTimeoutCode);
                *abort_flag = 1;
            }
        }
        __syncwarp();
    } else {
        // epilogue: accumulator row r sits in tensor-memory lane r; warp w reaches lanes 32 (w % 4) ..
        const int quad = warp & 3, part = (warp - 2) >> 2;
        const bool vec = ((uintptr_t)a.out & 15) == 0 && (a.ldo & 3) == 0 && (!a.bias || ((uintptr_t)a.bias & 15) == 0);
        int j = 0;
        for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++j) {
            const int buf = j & 1;
            const int m0 = (tile % tiles_m) * kPfTileM, n0 = (tile / tiles_m) * cols;
            const int row = m0 + quad * 32 + lane;
            // (the wait ends early once another role has given up)
            bool landed = false;
            {
                const long long t0 = clock64();
                while (!(landed = mbar_try_wait(&acc_full[buf], (j >> 1) & 1))) {
                    if (*abort_flag || clock64() - t0 > 8 * a.wait_cycles) break;
                }
            }
            if (!__all_sync(0xffffffffu, landed)) {  // (the tensor-memory loads are warp-wide)
                set_status(a.status, kTimeoutCode);
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            if (a.mode >= PF_GELU) {
                const uint32_t acc = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * kPfTileN);
                const size_t orow = (size_t)row * a.N + n0;
#pragma unroll 1
                for (int cb = part * (cols / 64); cb < (part + 1) * (cols / 64); ++cb) {
                    if (n0 + cb * 32 >= a.N) break;
                    float v[32], u[32];
                    tc_ld_32(acc + cb * 32, v);
                    if (a.mode == PF_SWIGLU) tc_ld_32(acc + kPfTileN / 2 + cb * 32, u);
                    if (row < a.R) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {   // eight columns: 16 bytes of hi, 16 bytes of lo (N is a multiple of 8)
                            const int c0 = n0 + cb * 32 + 8 * i;
                            if (c0 >= a.N) break;
                            float y[8], bg[8] = {}, bu[8] = {};
                            if (a.bias) {
#pragma unroll
                                for (int e = 0; e < 8; ++e) bg[e] = __ldg(a.bias + c0 + e);
                                if (a.mode == PF_SWIGLU) {
#pragma unroll
                                    for (int e = 0; e < 8; ++e) bu[e] = __ldg(a.bias + a.N + c0 + e);
                                }
                            }
                            if (a.mode == PF_GELU) {
#pragma unroll
                                for (int e = 0; e < 8; ++e) y[e] = gelu_erf(v[8 * i + e] + bg[e]);
                            } else {
#pragma unroll
                                for (int e = 0; e < 8; ++e) y[e] = silu(v[8 * i + e] + bg[e]) * (u[8 * i + e] + bu[e]);
                            }
                            uint4 hv, lv;
                            split_hilo8(y, hv, lv);
                            *reinterpret_cast<uint4 *>(a.act_hi + orow + cb * 32 + 8 * i) = hv;
                            *reinterpret_cast<uint4 *>(a.act_lo + orow + cb * 32 + 8 * i) = lv;
                        }
                    }
                }
            } else {
                float *orow = a.out + (size_t)row * a.ldo + n0;
#pragma unroll 1
                for (int cb = part * (kPfTileN / 64); cb < (part + 1) * (kPfTileN / 64); ++cb) {
                    if (n0 + cb * 32 >= a.N) break;
                    float v[32];
                    tc_ld_32(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * kPfTileN + cb * 32), v);
                    if (row < a.R) {
                        if (vec && n0 + cb * 32 + 31 < a.N) {
                            if (a.bias) {
#pragma unroll
                                for (int i = 0; i < 8; ++i) {
                                    const float4 bv = __ldg(reinterpret_cast<const float4 *>(a.bias + n0 + cb * 32 + 4 * i));
                                    v[4 * i] += bv.x; v[4 * i + 1] += bv.y; v[4 * i + 2] += bv.z; v[4 * i + 3] += bv.w;
                                }
                            }
                            if (a.mode == PF_ADD) {
                                float4 o[8];
#pragma unroll
                                for (int i = 0; i < 8; ++i) o[i] = *reinterpret_cast<const float4 *>(orow + cb * 32 + 4 * i);
#pragma unroll
                                for (int i = 0; i < 8; ++i) {
                                    v[4 * i] += o[i].x; v[4 * i + 1] += o[i].y; v[4 * i + 2] += o[i].z; v[4 * i + 3] += o[i].w;
                                }
                            }
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                *reinterpret_cast<float4 *>(orow + cb * 32 + 4 * i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                        } else {
                            for (int i = 0; i < 32; ++i) {
                                const int col = n0 + cb * 32 + i;
                                if (col < a.N) {
                                    float y = v[i] + (a.bias ? a.bias[col] : 0.f);
                                    if (a.mode == PF_ADD) y += orow[cb * 32 + i];
                                    orow[cb * 32 + i] = y;
                                }
                            }
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);  // this warp has read its part of the buffer
        }
        tc_fence_before();
    }
    __syncthreads();
    if (warp == 0) {
        if (lane == 0 && *abort_flag)  // error path only: copies that may still land in this CTA's shared memory
            for (int i = (issued > kPfStages ? issued - kPfStages : 0); i < issued; ++i) mbar_wait(&full[i % kPfStages], (i / kPfStages) & 1);
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512) : "memory");
    }
}

// Row norm for the many-row pass: one CTA of 256 threads per row, the row held in registers (float4 per thread,
// up to 8192 columns; wider rows are re-read), statistics in fp64 in one exchange, one or two outputs (bf16 hi + lo, row-major)
// from the same statistics.  The mean is subtracted as an fp32 pair, so a large common offset costs nothing; the rest is fp32
// arithmetic (the result is split to 16 bits next): converting each value to fp64 and back took most of the kernel.
// Memory-bound: 8184 x 2560, two outputs, 252 MB: 109 us with the values in fp64 and two exchanges, 64 so.
struct PfNormArgs {
    const float *x;
    int d, kind;  // 0 LayerNorm, 1 RMSNorm
    float eps;
    int n_norms;
    const float *g[2], *b[2];
    __nv_bfloat16 *hi[2], *lo[2];
};
__device__ __forceinline__ void store_hilo4(__nv_bfloat16 *hi, __nv_bfloat16 *lo, size_t idx, float4 y) {
    const __nv_bfloat162 h01 = __floats2bfloat162_rn(y.x, y.y), h23 = __floats2bfloat162_rn(y.z, y.w);
    const __nv_bfloat162 l01 = __floats2bfloat162_rn(y.x - __low2float(h01), y.y - __high2float(h01));
    const __nv_bfloat162 l23 = __floats2bfloat162_rn(y.z - __low2float(h23), y.w - __high2float(h23));
    uint2 hv, lv;
    hv.x = *reinterpret_cast<const uint32_t *>(&h01); hv.y = *reinterpret_cast<const uint32_t *>(&h23);
    lv.x = *reinterpret_cast<const uint32_t *>(&l01); lv.y = *reinterpret_cast<const uint32_t *>(&l23);
    *reinterpret_cast<uint2 *>(hi + idx) = hv;
    *reinterpret_cast<uint2 *>(lo + idx) = lv;
}
__global__ void __launch_bounds__(256) prefill_norm_kernel(const PfNormArgs a) {  // d % 4 == 0
    __shared__ double red[16];
    const int r = blockIdx.x, q4 = a.d >> 2;
    const float4 *x4 = reinterpret_cast<const float4 *>(a.x + (size_t)r * a.d);
    float4 v[8];
    double s = 0.0, ss = 0.0;
    auto add = [&](const float4 &w) {
        s += ((double)w.x + (double)w.y) + ((double)w.z + (double)w.w);
        ss += ((double)w.x * w.x + (double)w.y * w.y) + ((double)w.z * w.z + (double)w.w * w.w);
    };
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int i = threadIdx.x + 256 * k;
        v[k] = i < q4 ? x4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (256 * k < q4) add(v[k]);
    for (int i = threadIdx.x + 2048; i < q4; i += 256) add(x4[i]);
    s = warp_sum(s);
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = s;
        red[8 + (threadIdx.x >> 5)] = ss;
    }
    __syncthreads();
    s = ss = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        s += red[w];
        ss += red[8 + w];
    }
    const double mean = a.kind == 0 ? s / a.d : 0.0;
    const double var = ss / a.d - mean * mean;
    const float mu = (float)mean, mu_lo = (float)(mean - (double)mu), rs = (float)rsqrt((var > 0.0 ? var : 0.0) + (double)a.eps);
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        if (n >= a.n_norms) break;
        const float4 *g4 = reinterpret_cast<const float4 *>(a.g[n]);
        const float4 *b4 = reinterpret_cast<const float4 *>(a.b[n]);
        auto emit = [&](int i, const float4 &w) {
            const float4 g = __ldg(g4 + i);
            const float4 bb = b4 ? __ldg(b4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 y;
            y.x = ((w.x - mu) - mu_lo) * rs * g.x + bb.x;
            y.y = ((w.y - mu) - mu_lo) * rs * g.y + bb.y;
            y.z = ((w.z - mu) - mu_lo) * rs * g.z + bb.z;
            y.w = ((w.w - mu) - mu_lo) * rs * g.w + bb.w;
            store_hilo4(a.hi[n], a.lo[n], (size_t)r * a.d + 4 * (size_t)i, y);
        };
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (threadIdx.x + 256 * k < q4) emit(threadIdx.x + 256 * k, v[k]);
        for (int i = threadIdx.x + 2048; i < q4; i += 256) emit(i, x4[i]);
    }
}

// Rotary, the cache append and the attention kernels' queries: eight columns of one row per thread (16-byte loads and stores).
// prefill_append_kernel puts keys and values into the cache in its bf16, prefill_query_kernel scales the queries to log2 units
// and makes a bf16 hi / lo operand of them.  grid (ceil(2 d / 8 / 256), rows) and (ceil(d / 8 / 256), rows).
// Memory-bound: 8184 rows x 7680, 419 MB: 121 us in one kernel with a column per thread, 60 + 31 so.
struct PfAppendArgs {
    const float *qkv;                // [R, 3 d]
    __nv_bfloat16 *q_hi, *q_lo;      // [R, d]
    __nv_bfloat16 *cache;            // this layer's slab [B][2][H][S][Dh]
    int d, H, Dh, S, rotary_dim;
    float q_scale;
    RowInfo ri;
};
__device__ __forceinline__ void load8(const float *p, float (&v)[8]) {  // p 16-byte aligned
    const float4 u = *reinterpret_cast<const float4 *>(p), w = *reinterpret_cast<const float4 *>(p + 4);
    v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
    v[4] = w.x; v[5] = w.y; v[6] = w.z; v[7] = w.w;
}
// eight columns of row r from `src` (the head's column e first), turned by the row's position
__device__ __forceinline__ void load8_rotary(const PfAppendArgs &a, const float *src, int r, int e, int rotary_dim, float (&x)[8]) {
    load8(src, x);
    if (e < rotary_dim) {
        const int half = rotary_dim >> 1;
        const float *cos_r = a.ri.rope_cos + (size_t)r * half, *sin_r = a.ri.rope_sin + (size_t)r * half;
        if ((half & 7) == 0) {  // the eight columns lie on one side of the split, their partners are eight columns too
            const bool low = e < half;
            const int j = low ? e : e - half;
            float o[8], cs[8], sn[8];
            load8(low ? src + half : src - half, o);
            load8(cos_r + j, cs);
            load8(sin_r + j, sn);
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = low ? x[i] * cs[i] - o[i] * sn[i] : o[i] * sn[i] + x[i] * cs[i];
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (e + i >= rotary_dim) break;
                const bool low = e + i < half;
                const int j = low ? e + i : e + i - half;
                const float o = low ? src[i + half] : src[i - half];
                x[i] = low ? x[i] * cos_r[j] - o * sin_r[j] : o * sin_r[j] + x[i] * cos_r[j];
            }
        }
    }
}
__global__ void __launch_bounds__(256) prefill_append_kernel(const PfAppendArgs a) {
    const int r = blockIdx.y, c = (blockIdx.x * 256 + threadIdx.x) * 8;
    if (c >= 2 * a.d || !a.ri.valid[r]) return;
    const int is_v = c >= a.d ? 1 : 0, col = c - is_v * a.d, h = col / a.Dh, e = col % a.Dh;
    float x[8];
    load8_rotary(a, a.qkv + (size_t)r * 3 * a.d + a.d + c, r, e, is_v ? 0 : a.rotary_dim, x);
    const size_t plane = ((size_t)a.ri.seq[r] * 2 + is_v) * a.H + h;
    *reinterpret_cast<uint4 *>(a.cache + (plane * a.S + a.ri.pos[r]) * a.Dh + e) =
        make_uint4(pack_bf16x2(x[0], x[1]), pack_bf16x2(x[2], x[3]), pack_bf16x2(x[4], x[5]), pack_bf16x2(x[6], x[7]));
}
__global__ void __launch_bounds__(256) prefill_query_kernel(const PfAppendArgs a) {
    const int r = blockIdx.y, c = (blockIdx.x * 256 + threadIdx.x) * 8;
    if (c >= a.d) return;
    float x[8];
    load8_rotary(a, a.qkv + (size_t)r * 3 * a.d + c, r, c % a.Dh, a.rotary_dim, x);
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] *= a.q_scale;
    uint4 hi, lo;
    split_hilo8(x, hi, lo);
    *reinterpret_cast<uint4 *>(a.q_hi + (size_t)r * a.d + c) = hi;
    *reinterpret_cast<uint4 *>(a.q_lo + (size_t)r * a.d + c) = lo;
}

// prefill_attn_kernel: causal attention of 64 query rows of one (sequence, head) over the cache, which already
// holds this pass's keys / values (the append kernel has run).  Four warps of 16 rows each; K / V chunks of 64
// positions go through two cp.async buffers shared by the four warps; per warp and chunk
//   S [16 x 64] = Q (bf16 hi + lo) K^T,   running max / sum in registers (base-2 exponentials),
//   O [16 x Dh] += P (bf16 hi + lo) V,
// on mma.sync tiles (m16n8k16).  Taken for caches of 2^31 (layer, sequence, K | V, head, position) rows or more, which the
// tensor-core form's map cannot address.  Row m of the sequence sees positions <= len + m.  The result goes to the out-projection
// operand as bf16 hi + lo, row-major; rows that are not fed get zeros.
constexpr int kPaRows = 64, kPaThreads = 128, kPaChunk = 64;
inline size_t prefill_attn_smem(int Dh) {
    return (size_t)2 * kPaRows * (Dh + 8) * 2 + (size_t)2 * 2 * kPaChunk * (Dh + 8) * 2;
}

struct PfAttnArgs {
    const __nv_bfloat16 *q_hi, *q_lo;  // [B * M, d] position-encoded queries, in log2 units
    const __nv_bfloat16 *cache;  // this layer's slab [B][2][H][S][Dh]
    const int32_t *len;          // [B] committed lengths
    const int32_t *n_eff;        // [B] rows fed per sequence
    __nv_bfloat16 *out_hi, *out_lo;  // [B * M, d]
    int M, H, Dh, S, d;
};

__global__ void __launch_bounds__(kPaThreads) prefill_attn_kernel(const PfAttnArgs a) {
    extern __shared__ __align__(16) uint8_t pa_smem[];
    const int mt = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int Dh = a.Dh, pitch = Dh + 8;
    const uint32_t pitchB = (uint32_t)pitch * 2u;
    __nv_bfloat16 *Qhi = reinterpret_cast<__nv_bfloat16 *>(pa_smem);
    __nv_bfloat16 *Qlo = Qhi + kPaRows * pitch;
    __nv_bfloat16 *KV = Qlo + kPaRows * pitch;  // buffer i: K at KV + i * 2 * 64 * pitch, V 64 * pitch later
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int nk = Dh >> 4, vpr = Dh >> 3;
    const int len = a.len[b], n = a.n_eff[b];
    const int m_base = mt * kPaRows, r0 = b * a.M;
    const int rows_fed = max(0, min(kPaRows, n - m_base));
    const int p_end = rows_fed > 0 ? min(len + m_base + rows_fed, a.S) : 0;  // positions any row of this tile sees
    const int n_chunks = (p_end + kPaChunk - 1) / kPaChunk;
    const __nv_bfloat16 *kc = a.cache + ((size_t)(b * 2) * a.H + h) * a.S * Dh;
    const __nv_bfloat16 *vc = kc + (size_t)a.H * a.S * Dh;

    auto load_chunk = [&](int c) {
        __nv_bfloat16 *Kb = KV + (size_t)(c & 1) * 2 * kPaChunk * pitch, *Vb = Kb + kPaChunk * pitch;
        const int t0 = c * kPaChunk;
        for (int i = tid; i < kPaChunk * vpr; i += kPaThreads) {
            const int pp = i / vpr, v8 = i % vpr, pos = t0 + pp;
            __nv_bfloat16 *dk = Kb + pp * pitch + v8 * 8, *dv = Vb + pp * pitch + v8 * 8;
            if (pos < p_end) {
                cp_async16(dk, kc + (size_t)pos * Dh + v8 * 8);
                cp_async16(dv, vc + (size_t)pos * Dh + v8 * 8);
            } else {  // masked positions: P is 0 there, and 0 x these zeros stays 0
                *reinterpret_cast<uint4 *>(dk) = make_uint4(0, 0, 0, 0);
                *reinterpret_cast<uint4 *>(dv) = make_uint4(0, 0, 0, 0);
            }
        }
        cp_async_commit();
    };
    if (n_chunks > 0) load_chunk(0);
    // Q rows of this tile
    for (int i = tid; i < kPaRows * vpr; i += kPaThreads) {
        const int ml = i / vpr, v8 = i % vpr, m = m_base + ml;
        uint4 hv = make_uint4(0, 0, 0, 0), lv = hv;
        if (m < n) {
            const size_t off = (size_t)(r0 + m) * a.d + h * Dh + v8 * 8;
            hv = *reinterpret_cast<const uint4 *>(a.q_hi + off);
            lv = *reinterpret_cast<const uint4 *>(a.q_lo + off);
        }
        *reinterpret_cast<uint4 *>(Qhi + ml * pitch + v8 * 8) = hv;
        *reinterpret_cast<uint4 *>(Qlo + ml * pitch + v8 * 8) = lv;
    }

    float o[16][4];
#pragma unroll
    for (int j = 0; j < 16; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
    const int row_lo = m_base + 16 * warp;           // this warp's rows: row_lo + g, row_lo + g + 8
    const int warp_end = len + row_lo + 15;           // last position any of them sees

    for (int c = 0; c < n_chunks; ++c) {
        if (c + 1 < n_chunks) load_chunk(c + 1); else cp_async_commit();
        cp_async_wait<1>();
        __syncthreads();  // chunk c (and, first time, Q) is in shared memory
        const int t0 = c * kPaChunk;
        if (t0 <= warp_end && row_lo < n) {
            const __nv_bfloat16 *Kb = KV + (size_t)(c & 1) * 2 * kPaChunk * pitch, *Vb = Kb + kPaChunk * pitch;
            float s[8][4];
#pragma unroll
            for (int j = 0; j < 8; ++j) s[j][0] = s[j][1] = s[j][2] = s[j][3] = 0.f;
            const uint32_t qa = smem_u32(Qhi) + (uint32_t)(16 * warp + (lane & 15)) * pitchB + (uint32_t)(lane >> 4) * 16u;
            const uint32_t ql = qa + (uint32_t)kPaRows * pitchB;
            const uint32_t ka = smem_u32(Kb) + (uint32_t)((lane & 7) + 8 * (lane >> 4)) * pitchB + (uint32_t)((lane >> 3) & 1) * 16u;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                if (ks < nk) {
                    uint32_t a0, a1, a2, a3, c0, c1, c2, c3;
                    ldmatrix_x4(qa + ks * 32, a0, a1, a2, a3);
                    ldmatrix_x4(ql + ks * 32, c0, c1, c2, c3);
#pragma unroll
                    for (int j2 = 0; j2 < 4; ++j2) {  // 16 positions: (0-7: k lo, k hi), (8-15: k lo, k hi)
                        uint32_t k0, k1, k2, k3;
                        ldmatrix_x4(ka + (uint32_t)(16 * j2) * pitchB + ks * 32, k0, k1, k2, k3);
                        mma_bf16(s[2 * j2], a0, a1, a2, a3, k0, k1);
                        mma_bf16(s[2 * j2], c0, c1, c2, c3, k0, k1);
                        mma_bf16(s[2 * j2 + 1], a0, a1, a2, a3, k2, k3);
                        mma_bf16(s[2 * j2 + 1], c0, c1, c2, c3, k2, k3);
                    }
                }
            }
            // mask, running max / sum (rows g and g + 8)
#pragma unroll
            for (int hrow = 0; hrow < 2; ++hrow) {
                const int m = row_lo + g + 8 * hrow;
                const int last = m < n ? len + m : -1;  // last visible position
                float mx = -INFINITY;
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int pos = t0 + 8 * j + 2 * t + e;
                        const float v = pos <= last ? s[j][2 * hrow + e] : -INFINITY;
                        s[j][2 * hrow + e] = v;
                        mx = fmaxf(mx, v);
                    }
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                const float m_new = fmaxf(m_run[hrow], mx);
                float f = 1.f, sum = 0.f;
                if (m_new > -INFINITY) {
                    f = exp2f(m_run[hrow] - m_new);  // 0 on the first non-empty block
#pragma unroll
                    for (int j = 0; j < 8; ++j)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float pv = exp2f(s[j][2 * hrow + e] - m_new);
                            s[j][2 * hrow + e] = pv;
                            sum += pv;
                        }
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) s[j][2 * hrow] = s[j][2 * hrow + 1] = 0.f;
                }
                m_run[hrow] = m_new;
                l_run[hrow] = l_run[hrow] * f + sum;  // this thread's share; lanes are summed at the end
#pragma unroll
                for (int j = 0; j < 16; ++j) { o[j][2 * hrow] *= f; o[j][2 * hrow + 1] *= f; }
            }
            // O += P V: k = 16 positions per step, n = the head's columns
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                uint32_t ph[4], pl[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {  // a0: (row g, k 2t..) a1: (row g+8, ..) a2: (row g, k 8+2t..) a3: (row g+8, ..)
                    const int j = 2 * kk + (q >> 1), hrow = q & 1;
                    const float x0 = s[j][2 * hrow], x1 = s[j][2 * hrow + 1];
                    const __nv_bfloat162 hv = __floats2bfloat162_rn(x0, x1);
                    ph[q] = *reinterpret_cast<const uint32_t *>(&hv);
                    pl[q] = pack_bf16x2(x0 - __low2float(hv), x1 - __high2float(hv));
                }
                const uint32_t va = smem_u32(Vb) + (uint32_t)(16 * kk + (lane & 15)) * pitchB;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    if (j < 2 * nk) {
                        uint32_t b0, b1;
                        ldmatrix_x2_trans(va + j * 16, b0, b1);
                        mma_bf16(o[j], ph[0], ph[1], ph[2], ph[3], b0, b1);
                        mma_bf16(o[j], pl[0], pl[1], pl[2], pl[3], b0, b1);
                    }
                }
            }
        }
        __syncthreads();  // everyone is done with this buffer before it is refilled
    }
    cp_async_wait<0>();
    // output: rows g, g + 8 of this warp; columns 8 j + 2 t, + 1
#pragma unroll
    for (int hrow = 0; hrow < 2; ++hrow) {
        float L = l_run[hrow];
        L += __shfl_xor_sync(0xffffffffu, L, 1);
        L += __shfl_xor_sync(0xffffffffu, L, 2);
        const int m = row_lo + g + 8 * hrow;
        if (m >= a.M) continue;
        const float inv = (m < n && L > 0.f) ? 1.f / L : 0.f;
        const size_t base = (size_t)(r0 + m) * a.d + h * Dh + 2 * t;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            if (j < 2 * nk) {
                const float y0 = o[j][2 * hrow] * inv, y1 = o[j][2 * hrow + 1] * inv;
                const __nv_bfloat162 hv = __floats2bfloat162_rn(y0, y1);
                const __nv_bfloat162 lv = __floats2bfloat162_rn(y0 - __low2float(hv), y1 - __high2float(hv));
                *reinterpret_cast<__nv_bfloat162 *>(a.out_hi + base + 8 * j) = hv;
                *reinterpret_cast<__nv_bfloat162 *>(a.out_lo + base + 8 * j) = lv;
            }
        }
    }
}

// prefill_attn_tc_kernel: the same causal attention on the 5th-generation tensor core, 128 query rows
// of one (sequence, head) per CTA, 128 positions per chunk, scores, probabilities and output in tensor memory:
//   S [128 rows x 128 positions] = Q (bf16 hi + lo, in log2 units) x K chunk^T, both straight from TMA copies into
//                                  128-byte-swizzled tiles: 2 x Dh / 16 MMAs of K = 16 head dims;
//   two threads (warps w and w + 4, 64 positions each) share query row r = tensor-memory lane r: they read its row of S, keep
//   the row's running maximum (exchanged once per chunk) and their share of its sum in registers, and write P = exp2(S - max) back over the same
//   columns as packed bf16 hi and lo (per group of 32 positions: 16 columns hi, 16 columns lo);
//   O [128 rows x 128 head dims] += P (hi, then lo: the A operand read from tensor memory) x V chunk (the B operand,
//                                  head dims contiguous: MN-major): 2 x 8 MMAs of K = 16 positions.
// A tile is one or two panels of 64 head dims; the copies fill a shorter head up with zeros (K, V), which only P V multiplies.
// V rows past the last visible position are whatever the cache holds there: they are cleared in the tile, for 0 x NaN is not 0.
// Head 80, 8 x 1023 tokens: 458 us a layer on warp-level
// MMAs, 241 here.
// S is double-buffered (256 columns) so that the scores of chunk c + 1 are computed while the threads work on chunk
// c; O takes 128 columns.  The running maximum is only raised when a chunk exceeds it by more than 2^8 (the sums and
// O absorb the factor), so that rescaling O - a read and a write of the thread's half of the columns - is rare.
// Bound by the softmax arithmetic's latency: with one thread per row (one warp per scheduler) 8 x 1023 rows of head 80 took
// 335 us a layer, with two 241.
// Warp 8 issues the MMAs, warp 9 the Q, K and V copies (two stages of K and V).  Every wait is bounded.
constexpr int kPtRows = 128, kPtChunk = 128, kPtThreads = 320;
constexpr int kPtPanel = 128 * 128;                  // 64 head dims of 128 rows
constexpr int kPtTile = 2 * kPtPanel;                // room of a Q (hi or lo), K or V tile
constexpr size_t kPtSmem = 1024 + 6 * kPtTile + 256 + 4 * 128 * 4; // Q hi, Q lo, two K and two V chunks; barriers; maxima by chunk parity
constexpr float kPtMaxSlack = 8.f;

struct PtAttnArgs {
    const int32_t *len;          // [B] committed lengths
    const int32_t *n_eff;        // [B] rows fed per sequence
    __nv_bfloat16 *out_hi, *out_lo;  // [B * M, d]
    int M, H, Dh, S, d;
    int kv_row0;                 // first row of this layer in the cache seen as rows of one head
    long long wait_cycles;
    int32_t *status;
};

// 32 columns of this thread's lane; completion is awaited by tc_wait_st
__device__ __forceinline__ void tc_st_32u_nowait(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n" ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]) : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// D[tmem] (+)= A[tmem] x B[smem descriptor]
__device__ __forceinline__ void tc_mma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n" ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__global__ void __launch_bounds__(kPtThreads, 1)
prefill_attn_tc_kernel(const __grid_constant__ CUtensorMap tmKV, const __grid_constant__ CUtensorMap tmQhi,
                       const __grid_constant__ CUtensorMap tmQlo, const PtAttnArgs a) {
    extern __shared__ uint8_t pt_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)pt_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *qhi = smem, *qlo = smem + kPtTile, *kring = smem + 2 * kPtTile, *vring = kring + 2 * kPtTile;
    uint64_t *bars = (uint64_t *)(vring + 2 * kPtTile);
    uint64_t *k_full = bars, *k_free = bars + 2, *v_full = bars + 4, *v_free = bars + 6, *s_full = bars + 8;
    // By chunk parity, like the score buffers: S of chunk c + 1 is issued before P V of chunk c, so a warp may be a whole
    // chunk ahead of the slowest one.  With one barrier its arrival for c + 1 would count for c, and its wait for P V of
    // the last chunk would pass on the phase before the previous chunk's.
    uint64_t *p_ready = bars + 10, *o_done = bars + 12;
    uint64_t *q_full = bars + 14;
    uint32_t *tmem_slot = (uint32_t *)(bars + 15);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    volatile float *row_x = (volatile float *)(bars + 32);  // [chunk parity][half][row]: what the two threads of a row exchange

    const int Dh = a.Dh, panels = Dh > 64 ? 2 : 1;
    // the longest row tiles first: a CTA's time goes with the positions its rows see
    const int mt = (int)gridDim.x - 1 - (int)blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int len = a.len[b], n = a.n_eff[b];
    const int m_base = mt * kPtRows, r0 = b * a.M;
    const int rows_fed = max(0, min(kPtRows, n - m_base));
    if (rows_fed == 0) {  // nothing fed in this tile: zeros for its rows
        for (int i = tid; i < kPtRows * (Dh / 8); i += kPtThreads) {
            const int m = m_base + i / (Dh / 8);
            if (m < a.M) {
                const size_t off = (size_t)(r0 + m) * a.d + h * Dh + (i % (Dh / 8)) * 8;
                *reinterpret_cast<uint4 *>(a.out_hi + off) = make_uint4(0, 0, 0, 0);
                *reinterpret_cast<uint4 *>(a.out_lo + off) = make_uint4(0, 0, 0, 0);
            }
        }
        return;
    }
    const int p_end = min(len + m_base + rows_fed, a.S);  // positions any row of this tile sees
    const int n_chunks = (p_end + kPtChunk - 1) / kPtChunk;
    const int krow0 = a.kv_row0 + ((b * 2) * a.H + h) * a.S, vrow0 = krow0 + a.H * a.S;

    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "n"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < 10; ++i) mbar_init(&bars[i], 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&p_ready[i], 256);
            mbar_init(&o_done[i], 1);
        }
        mbar_init(q_full, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t tS = tmem, tO = tmem + 256;  // S / P of chunk c at tS + 128 (c & 1)
    auto wait = [&](uint64_t *bar, uint32_t parity) {  // keeps every role's control flow intact once anything has timed out
        if (*abort_flag) return;
        const long long t0 = clock64();
        while (!mbar_try_wait(bar, parity)) {
            if (*abort_flag) return;
            if (clock64() - t0 > a.wait_cycles) {
                set_status(a.status, kTimeoutCode);
                *abort_flag = 1;
                return;
            }
        }
    };

    if (warp == 9) {
        if (lane == 0) {
            int issued_k = 0, issued_v = 0;
            auto copy = [&](uint8_t *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
                mbar_expect_tx(bar, panels * kPtPanel);
                for (int i = 0; i < panels; ++i) tma_load_2d(dst + i * kPtPanel, map, x + 64 * i, y, bar);
            };
            mbar_expect_tx(q_full, 2 * panels * kPtPanel);
            for (int i = 0; i < panels; ++i) {
                tma_load_2d(qhi + i * kPtPanel, &tmQhi, h * Dh + 64 * i, r0 + m_base, q_full);
                tma_load_2d(qlo + i * kPtPanel, &tmQlo, h * Dh + 64 * i, r0 + m_base, q_full);
            }
            for (int c = 0; c < n_chunks && !*abort_flag; ++c) {
                const int s = c & 1;
                if (c >= 2) wait(&k_free[s], ((c >> 1) - 1) & 1);
                if (*abort_flag) break;
                copy(kring + s * kPtTile, &tmKV, 0, krow0 + c * kPtChunk, &k_full[s]);
                ++issued_k;
                if (c >= 2) wait(&v_free[s], ((c >> 1) - 1) & 1);
                if (*abort_flag) break;
                copy(vring + s * kPtTile, &tmKV, 0, vrow0 + c * kPtChunk, &v_full[s]);
                ++issued_v;
            }
            // no copy is in flight into this CTA's shared memory when it ends, whichever role has given up meanwhile
            mbar_wait(q_full, 0);
            for (int c = max(0, issued_k - 2); c < issued_k; ++c) mbar_wait(&k_full[c & 1], (c >> 1) & 1);
            for (int c = max(0, issued_v - 2); c < issued_v; ++c) mbar_wait(&v_full[c & 1], (c >> 1) & 1);
        }
        __syncwarp();
    } else if (warp == 8) {
        if (lane == 0) {
            const uint32_t idS = umma_idesc_bf16(128, 128), idO = umma_idesc_bf16(128, 64 * panels) | (1u << 16);  // B of P V: MN-major
            auto issue_s = [&](int c) {
                const int s = c & 1;
                wait(&k_full[s], (c >> 1) & 1);
                if (*abort_flag) return;
                tc_fence_after();
                const uint32_t ka = smem_u32(kring + s * kPtTile), qa = smem_u32(qhi);
                for (int part = 0; part < 2; ++part)  // hi, then lo
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {  // k = 16 head dims per step; panel ks / 4
                        if (16 * ks >= Dh) break;
                        const uint32_t off = (ks >> 2) * kPtPanel + (ks & 3) * 32;
                        tc_mma_bf16(tS + 128 * s, umma_desc(qa + part * kPtTile + off, 16, 1024), umma_desc(ka + off, 16, 1024), idS,
                                    (part | ks) ? 1u : 0u);
                    }
                tc_commit(&s_full[s]);
                tc_commit(&k_free[s]);
            };
            wait(q_full, 0);
            issue_s(0);
            for (int c = 0; c < n_chunks && !*abort_flag; ++c) {
                const int s = c & 1;
                if (c + 1 < n_chunks) issue_s(c + 1);
                wait(&p_ready[s], (c >> 1) & 1);
                wait(&v_full[s], (c >> 1) & 1);
                if (*abort_flag) break;
                tc_fence_after();
                const uint32_t va = smem_u32(vring + s * kPtTile), tP = tS + 128 * s;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)  // k = 16 positions per step: two 8-row groups of the V tile; P hi
                    tc_mma_bf16_ta(tO, tP + 32 * (ks >> 1) + 8 * (ks & 1), umma_desc(va + ks * 2048, kPtPanel, 1024), idO, (c | ks) ? 1u : 0u);
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)  // P lo
                    tc_mma_bf16_ta(tO, tP + 32 * (ks >> 1) + 16 + 8 * (ks & 1), umma_desc(va + ks * 2048, kPtPanel, 1024), idO, 1u);
                tc_commit(&o_done[s]);
                tc_commit(&v_free[s]);
            }
        }
        __syncwarp();
    } else {
        // ---------------- softmax and output: two threads per query row = tensor-memory lane ----------------
        const int row = tid & 127, half = tid >> 7;
        const int m = m_base + row;
        const int last = m < n ? len + m : -1;  // last visible position
        const uint32_t lane_sel = (uint32_t)((warp & 3) * 32) << 16;
        auto exchange = [&](int parity, float x) {  // the other thread's x (a barrier for the two warps of a lane quadrant)
            row_x[(parity * 2 + half) * 128 + row] = x;
            asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp & 3)) : "memory");
            return row_x[(parity * 2 + (half ^ 1)) * 128 + row];
        };
        float m_run = -INFINITY, l_run = 0.f;
        for (int c = 0; c < n_chunks; ++c) {
            const uint32_t tSc = tS + 128 * (c & 1) + lane_sel + 64 * half;
            const int pos0 = c * kPtChunk;
            wait(&s_full[c & 1], (c >> 1) & 1);
            tc_fence_after();
            float v[64];  // the thread's scores, kept in registers for both passes
            tc_ld_64(tSc, v);
            const int seen = last - (pos0 + 64 * half);  // the last of them that the row sees
            if (!__all_sync(0xffffffffu, seen >= 63)) {
#pragma unroll
                for (int i = 0; i < 64; ++i) v[i] = i <= seen ? v[i] : -INFINITY;
            }
            float mc = v[0], mc1 = v[1], mc2 = v[2], mc3 = v[3];
#pragma unroll
            for (int i = 4; i < 64; i += 4) {
                mc = fmaxf(mc, v[i]);
                mc1 = fmaxf(mc1, v[i + 1]);
                mc2 = fmaxf(mc2, v[i + 2]);
                mc3 = fmaxf(mc3, v[i + 3]);
            }
            mc = fmaxf(fmaxf(mc, mc1), fmaxf(mc2, mc3));
            mc = fmaxf(mc, exchange(c & 1, mc));
            const float m_new = (mc > m_run + kPtMaxSlack || m_run == -INFINITY) ? fmaxf(m_run, mc) : m_run;
            const float f = m_new > -INFINITY ? exp2f(m_run - m_new) : 1.f;  // 0 on the first non-empty chunk
            const float m_ref = m_new > -INFINITY ? m_new : 0.f;             // (all masked: every p is exp2(-inf) = 0)
            float sum = 0.f, sum1 = 0.f;
#pragma unroll
            for (int g = 0; g < 2; ++g) {  // P: per 32 positions 16 columns hi, 16 lo
                uint32_t w[32];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float p0 = exp2f(v[32 * g + 2 * i] - m_ref), p1 = exp2f(v[32 * g + 2 * i + 1] - m_ref);
                    sum += p0;
                    sum1 += p1;
                    const __nv_bfloat162 hv = __floats2bfloat162_rn(p0, p1);
                    w[i] = *reinterpret_cast<const uint32_t *>(&hv);
                    w[16 + i] = pack_bf16x2(p0 - __low2float(hv), p1 - __high2float(hv));
                }
                tc_st_32u_nowait(tSc + 32 * g, w);
            }
            tc_wait_st();
            sum += sum1;
            l_run = l_run * f + sum;
            m_run = m_new;
            // the accumulated O row moves to the new maximum, once P V of the previous chunk has written it; the
            // tensor-memory loads and stores are warp-wide, so the warp goes together (f = 1 where nothing moved)
            if (c > 0 && __any_sync(0xffffffffu, f != 1.f)) {
                wait(&o_done[(c - 1) & 1], ((c - 1) >> 1) & 1);
                tc_fence_after();
#pragma unroll 1
                for (int g = half * panels; g < (half + 1) * panels; ++g) {  // its half of the columns, 32 at a time
                    float o[32];
                    tc_ld_32(tO + lane_sel + 32 * g, o);
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] *= f;
                    tc_st_32(tO + lane_sel + 32 * g, o);
                }
            }
            if (pos0 + kPtChunk > p_end) {  // (the last chunk)
                wait(&v_full[c & 1], (c >> 1) & 1);
                if (pos0 + row >= p_end && half < panels && !*abort_flag)
                    for (int i = 0; i < 8; ++i)  // (the swizzle stays within a row's 128 bytes)
                        *reinterpret_cast<uint4 *>(vring + (c & 1) * kPtTile + half * kPtPanel + row * 128 + i * 16) =
                            make_uint4(0, 0, 0, 0);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            tc_fence_before();
            mbar_arrive(&p_ready[c & 1]);
        }
        wait(&o_done[(n_chunks - 1) & 1], ((n_chunks - 1) >> 1) & 1);
        tc_fence_after();
        {
            const float l = l_run + exchange(n_chunks & 1, l_run);
            const bool store = m < a.M && !*abort_flag;  // (the loads are warp-wide: every lane takes them)
            const float inv = (m < n && l > 0.f) ? 1.f / l : 0.f;
            const size_t base = (size_t)(r0 + (store ? m : 0)) * a.d + h * Dh;
#pragma unroll 1
            for (int g = half * panels; g < (half + 1) * panels; ++g) {
                if (32 * g >= Dh) break;
                float o[32];
                tc_ld_32(tO + lane_sel + 32 * g, o);
                if (store) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {  // eight head dims: 16 bytes of hi, 16 bytes of lo
                        if (32 * g + 8 * i >= Dh) break;
                        float y[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) y[e] = o[8 * i + e] * inv;
                        uint4 hv, lv;
                        split_hilo8(y, hv, lv);
                        *reinterpret_cast<uint4 *>(a.out_hi + base + 32 * g + 8 * i) = hv;
                        *reinterpret_cast<uint4 *>(a.out_lo + base + 32 * g + 8 * i) = lv;
                    }
                }
            }
        }
        tc_fence_before();
    }
    __syncthreads();
    if (warp == 8) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512) : "memory");
    }
}

}  // namespace ssd
