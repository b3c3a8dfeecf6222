// The whole decoder forward of a verification pass (or a draft step) as ONE persistent
// cooperative kernel, one CTA per SM.
//
// Why: a pass is a chain of ~8 small dependent steps per layer; as separate launches the HBM
// stream stops at every boundary (the paper's point in Section "Autoregressive vs Speculative
// Sampling" is that the pass is memory-bound, so idle HBM time is the cost).  Here the weight
// stream never stops: a producer thread per CTA walks the static schedule of every weight tile
// this CTA will need in the whole forward and keeps a deep shared-memory ring full with TMA
// copies, running ahead across phase boundaries; only the small activation tiles wait for the
// grid barrier of the phase that produces them.
//
// Roles in a CTA (288 threads):
//   warp 8      producer: TMA issue for weight tiles, free-running across phase boundaries
//   warp 5      (one lane) during a GEMM phase: bulk copies of that GEMM's operand tiles, which
//               exist only once the grid barrier of the phase that wrote them has been passed
//   warp 4      (one lane) issues the GEMM: per ring stage four tcgen05.mma, each (activation
//               rows, hi and lo, as the M = 64 or 128 operand) x (256 weight rows as the N
//               operand) x 16 k, accumulating in tensor memory.  A K = 16 MMA step costs about
//               120 cycles whatever M and N are, so the weights sit on the side that lets one
//               step consume the most of them (8 KB).  tcgen05.commit hands the stage back to
//               the producer and, at the end of a tile segment, the accumulator to the
//               epilogue; two accumulator buffers overlap that epilogue with the next MMAs
//   warps 0-3   epilogue: tensor memory -> registers with the 16-lane x 256-bit load, which
//               puts a row's hi and lo products in one thread; hi + lo goes through a small
//               shared-memory tile so that all four warps add it (+ bias from the segment that
//               holds k-chunk 0) to the output with 16-byte vector reductions: a reduction
//               costs its warp a memory latency, so there must be few of them per thread
//   warps 0-7   between GEMM phases: the small phases (row set-up, embedding, norm, activation,
//               attention with rotary + KV append + split merge - on warp-level MMAs, or for head
//               dim 128 and long splits on tcgen05 with its own roles, see attention_item_tc),
//               which leave every GEMM operand in global memory already split into bf16 hi + lo,
//               and the grid barriers
// Every phase is a function of its own (not inlined) that reads a shared-memory copy of the kernel
// parameters and keeps what must survive between calls in shared memory: the phase loop holds nothing
// across calls, because a spilled value or a read through the parameter bank would be a trip to L2 at
// the head of every one of the pass's ~130-260 phases (227 KB of shared memory leave next to no L1).
// Every wait (mbarrier, grid barrier) is bounded; on time-out SSD_E_TIMEOUT is recorded, the CTA
// does no more GEMM work and stops at the next grid barrier that it waits at (an arrival takes no
// snapshot of the outcome), waits (bounded) for its copies in flight, drains the tensor core, frees its
// tensor memory and returns.  A parity wait is used only where the waiter follows every phase of its
// barrier in order and the barrier cannot pass it by two phases.
#pragma once
#include <cuda.h>

#include "attention.cuh"
#include "common.cuh"
#include "gemm.cuh"
#include "rowops.cuh"

namespace ssd {

constexpr int kConsumerWarps = 8;
constexpr int kWorkThreads = kConsumerWarps * 32;  // 256: everyone but the producer
constexpr int kPersistThreads = kWorkThreads + 32;
constexpr int kAttnThreadsP = 256;
constexpr int kMaxStagedLayers = 64;  // layers whose gain / bias pointers are staged in shared memory
constexpr int kTileNP = 256;                        // weight rows per tile: the N of one MMA
constexpr int kWTileBytesP = kTileNP * kTileK * 2;  // 32 KB

struct alignas(64) LayerDesc {
    CUtensorMap tm[4];  // qkv, o, in, out
    const float *ln1_g, *ln1_b, *b_qkv, *b_o, *ln2_g, *ln2_b, *b_in, *b_out;
};
struct alignas(64) ModelDesc {
    CUtensorMap tm_lm;
    const float *lnf_g, *lnf_b;
    const void *pad[6];
    // LayerDesc layers[] follow
};
__device__ __forceinline__ const LayerDesc *layer_desc(const ModelDesc *md, int l) {
    return reinterpret_cast<const LayerDesc *>(md + 1) + l;
}

__device__ __forceinline__ uint8_t *smem_base() {
    extern __shared__ uint8_t smem_raw[];
    return (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
}

enum { OP_XN1 = 0, OP_XN2 = 1, OP_AO = 2, OP_ACT = 3 };

struct alignas(64) FwdParams {
    // GEMM operands in global memory (normalised rows - two sets for parallel-residual blocks -,
    // attention output, MLP activation), stored the way a ring stage wants them: one contiguous
    // tile per 64-wide k-chunk, 2 rk rows of 128 bytes (per block of 8 rows: their 8 bf16 hi rows, then
    // their 8 lo rows), 16-byte chunks already in 128-byte-swizzle order, so one linear bulk copy
    // fetches a tile.
    // (A strided 2-D tensor copy of the same tile costs a sixth of the weight stream's bandwidth.)
    __nv_bfloat16 *op[4];
    int op_ld[4];  // K of each operand
    int rk;
    const ModelDesc *md;
    // architecture
    int n_layers, d, H, Dh, F, d_in, V, norm_kind, swiglu, parallel, rotary_dim, learned_pos;
    float eps, rotary_base, attn_scale;
    double inv_d;  // 1 / d (the norms' statistics are taken in fp64; a division there is a long routine)
    // rows
    int B, M, R;
    const int32_t *tokens;
    int tok_stride;
    const int32_t *n_rows;
    const void *tok_emb, *pos_emb;
    int pos_limit;
    // cache
    uint8_t *cache;
    size_t layer_bytes;
    const int32_t *len;
    int S;
    int32_t *status;
    // workspace
    RowInfo ri;
    float *x, *qkv, *t_in, *logits;
    float *part_m, *part_l, *part_o;
    unsigned *tickets;  // [B*H]: zeroed by the set-up
    unsigned *gbar;     // grid barrier counter (see leave_grid)
    int chunk, n_split;
    int want_logits;
    // Shared-memory ring: slots [0, stages_lo) hold weights at any time; slots [stages_lo, stages) share
    // their bytes with the attention scratch (at attn_smem_off = stages_lo * stage bytes) and are used
    // only between attention phases.
    int stages, stages_lo, attn_smem_off;
    unsigned long long *trace;  // optional: CTA 0 stamps the global timer at every grid barrier (see grid_stamp)
    // tensor-core attention (head dim 128): the whole cache as rows of Dh bf16, box 64 x 128 rows
    CUtensorMap tm_kv;
    const CUtensorMap *tm_kv_ptr;  // where the copy engine can read tm_kv (set by the kernel: see params copy)
    int attn_form;           // ATT_*: the form of the attention items
    int kv_rows_per_layer;   // B * 2 * H * S
    int attn_items;          // attention items of a layer
    int attn_ctas;           // min(attention items, CTAs): set by the host together with the split plan
    int overlap_out;         // parallel-residual block and at most half of the CTAs on attention
    long long wait_cycles;   // bound of every wait that takes work (see Shared::wait_limit)
    // Several draft steps in one launch (n_steps >= 1; the draft loop of a speculative iteration).  With tail == 1
    // every step ends inside the kernel: the logits of each sequence's last fed row become q = softmax(logits / T),
    // a token is drawn from q with the step's uniform, both are written out, the fed rows are committed, and the
    // next step feeds that token (one row per sequence).  cur_step is kept by the kernel in its copy of this block.
    int n_steps, tail, cur_step;
    float inv_t;                                   // 1 / T; 0 = greedy
    const float *u;     int u_stride;              // uniform of sequence b at step s: u[b * u_stride + s]
    int32_t *tok_out;   int tok_out_stride;        // token of step s: tok_out[b * tok_out_stride + s]
    float *q_out;       size_t q_stride;           // q row of step s: q_out + b * q_stride + s * V
    int32_t *len_rw;                               // the committed lengths, advanced after every step
    float *tp_m, *tp_s; int32_t *tp_a;             // per (sequence, CTA): max, sum of exp relative to it, argmax of the CTA's slice
    double *tp_mass;                               // per (sequence, CTA): mass of q in the CTA's slice
    int32_t *tail_hit;                             // [n_steps][B][2]: smallest index past u S (INT_MAX: none) / largest index with q > 0
    unsigned long long *mailbox; unsigned mb_seq;  // the lengths, reported to the host at the end
};

struct GemmDesc {
    const CUtensorMap *tmW;
    const __nv_bfloat16 *xop;  // tiled operand
    int N, Kd, n_tiles, kchunks;
    int need;  // grid barriers that must have completed before its operand exists
    int need_hi;  // grid barriers that this CTA must have arrived at before its tiles may use the ring slots shared with the attention scratch
    int kind;     // 0 qkv, 1 o, 2 in, 3 out, 4 LM head
    unsigned wait_attn;  // attention CTAs that must have signalled before its operand exists (0: a grid barrier covers it)
    float *out;
    int ldo;
    const float *bias;
};

// (without logits the last layer ends with its keys and values: only its qkv projection is run)
__device__ __forceinline__ int n_gemms(const FwdParams &p) { return p.want_logits ? 4 * p.n_layers + 1 : 4 * p.n_layers - 3; }
// CTAs that run an attention item in a phase (each at most one when this is below the grid size).
__device__ __forceinline__ int attention_ctas(const FwdParams &p) { return p.attn_ctas; }
// Parallel-residual blocks with at most half of the CTAs on attention: the MLP-out GEMM depends on the
// activation, not on attention, so the CTAs without an attention item run it during the attention phase.
__device__ __forceinline__ bool overlap_mlp_out(const FwdParams &p) { return p.overlap_out != 0; }
__device__ __forceinline__ int barriers_per_layer(const FwdParams &p) { return p.parallel ? 4 : 8; }
__device__ __forceinline__ int attention_end(const FwdParams &p) { return overlap_mlp_out(p) ? 3 : 2; }  // barriers into the layer

// GEMM number gi in execution order.  sequential: qkv, o, in, out; parallel: qkv, in, o, out.
// Barrier count before layer l: 1 (set-up, embedding and first norm) + barriers_per_layer * l.
//   sequential layer: qkv | attention | o | norm2 | in | act | out | next norm   (8 barriers)
//   parallel layer:   qkv, in | attention + act | o, out | next norms            (4 barriers)
//   ... with few attention items: qkv, in | act | attention (some CTAs); out, then - once every attention CTA has
//       signalled - o (the others) | next norms   (4)
// Grid barriers of one step of a launch: the head, the layers', and five around the phases of the in-kernel tail.
__device__ __forceinline__ int step_barriers(const FwdParams &p) { return 1 + barriers_per_layer(p) * p.n_layers + (p.tail ? 5 : 0); }
constexpr int kStepShift = 12;  // a GEMM is named (step << kStepShift) | number within the forward

__device__ __forceinline__ GemmDesc gemm_desc(const FwdParams &p, int gi_step, const float *const *ltab = nullptr) {
    GemmDesc g;
    g.wait_attn = 0;
    const int step = gi_step >> kStepShift, gi = gi_step & ((1 << kStepShift) - 1);
    const int sb = step * step_barriers(p);  // barriers before this step
    const int l = gi >> 2, e = gi & 3;
    const int base = sb + 1 + barriers_per_layer(p) * l;
    if (l >= p.n_layers) {  // LM head
        g.tmW = &p.md->tm_lm; g.xop = p.op[OP_XN1];
        g.N = p.V; g.Kd = p.d; g.need = base; g.out = p.logits; g.ldo = p.V; g.bias = nullptr;
        g.kind = 4; g.need_hi = base - barriers_per_layer(p) + attention_end(p);  // end of the last attention phase
    } else {
        const LayerDesc *ld = layer_desc(p.md, l);
        int kind;  // 0 qkv, 1 o, 2 in, 3 out
        if (p.parallel && overlap_mlp_out(p)) kind = (e == 0) ? 0 : (e == 1) ? 2 : (e == 2) ? 3 : 1;  // out before o
        else if (p.parallel) kind = (e == 0) ? 0 : (e == 1) ? 2 : (e == 2) ? 1 : 3;
        else kind = e;
        g.tmW = &ld->tm[kind];
        g.kind = kind;
        // the attention phase of layer l ends at barrier base + 2; qkv precedes it (previous layer's counts)
        // (so does the MLP input GEMM of a parallel-residual block)
        g.need_hi = (kind == 0 || (kind == 2 && p.parallel)) ? (l == 0 ? sb : base - barriers_per_layer(p) + attention_end(p))
                                                             : base + attention_end(p);
        if (kind == 0) {
            g.xop = p.op[OP_XN1]; g.N = 3 * p.d; g.Kd = p.d; g.need = base;
            g.out = p.qkv; g.ldo = 3 * p.d; g.bias = ltab ? ltab[8 * l + 2] : ld->b_qkv;
        } else if (kind == 1) {
            g.xop = p.op[OP_AO]; g.N = p.d; g.Kd = p.d; g.need = base + 2;
            if (overlap_mlp_out(p)) g.wait_attn = (unsigned)(step * p.n_layers + l + 1) * (unsigned)attention_ctas(p);
            g.out = p.x; g.ldo = p.d; g.bias = ltab ? ltab[8 * l + 3] : ld->b_o;
        } else if (kind == 2) {
            g.xop = p.op[p.parallel ? OP_XN2 : OP_XN1]; g.N = p.d_in; g.Kd = p.d; g.need = p.parallel ? base : base + 4;
            g.out = p.t_in; g.ldo = p.d_in; g.bias = ltab ? ltab[8 * l + 6] : ld->b_in;
        } else {
            g.xop = p.op[OP_ACT]; g.N = p.d; g.Kd = p.F; g.need = p.parallel ? base + 2 : base + 6;
            g.out = p.x; g.ldo = p.d; g.bias = ltab ? ltab[8 * l + 7] : ld->b_out;
        }
    }
    g.n_tiles = (g.N + kTileNP - 1) / kTileNP;
    g.kchunks = (g.Kd + kTileK - 1) / kTileK;
    return g;
}

// This CTA's contiguous share of a GEMM's (tile, k-chunk) units.  Equal shares, except in the GEMM that
// follows the attention phase (MLP-out of a parallel-residual block, out-projection otherwise) when
// at most half of the CTAs ran an attention item: those enter the phase with only the lower ring
// slots filled ahead, the others with the whole ring, so they get that many units fewer.
__device__ __forceinline__ void unit_range(const FwdParams &p, const GemmDesc &g, int &c0, int &c1) {
    const long long total = (long long)g.n_tiles * g.kchunks;
    const int N = (int)gridDim.x, i = (int)blockIdx.x;
    const int A = attention_ctas(p), bonus = p.stages - p.stages_lo;
    if (overlap_mlp_out(p)) {  // MLP-out runs beside attention on the CTAs without an item; everything else in equal shares
        if (g.kind == 3 || g.kind == 1) {  // (the out-projection follows on the same CTAs: see attn_done)
            c0 = i < A ? 0 : (int)(total * (i - A) / (N - A));
            c1 = i < A ? 0 : (int)(total * (i - A + 1) / (N - A));
            return;
        }
        c0 = (int)(total * i / N);
        c1 = (int)(total * (i + 1) / N);
        return;
    }
    const bool after_attention = p.parallel ? g.kind == 3 : g.kind == 1;
    if (after_attention && 2 * A <= N && bonus > 0) {  // (with most CTAs on attention the few others would become the stragglers)
        long long xa = (total + (long long)A * bonus) / N - bonus;  // an attention CTA's share
        if (xa < 0) xa = 0;
        const long long rest = total - xa * A;                      // over the N - A others
        if (i < A) {
            c0 = (int)(xa * i);
            c1 = (int)(xa * (i + 1));
        } else {
            c0 = (int)(xa * A + rest * (i - A) / (N - A));
            c1 = (int)(xa * A + rest * (i - A + 1) / (N - A));
        }
        return;
    }
    c0 = (int)(total * i / N);
    c1 = (int)(total * (i + 1) / N);
}

__device__ __forceinline__ void named_bar(int id, int count) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add(unsigned *p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned atomic_add_acq_rel(unsigned *p, unsigned v) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async;" ::: "memory"); }
// ... for shared memory alone (some 40 cycles; the general form about half a microsecond) and for global memory alone
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// Tile row of the hi part of row r (the lo part is 8 further): rows come in blocks of 8, each block
// as 8 hi rows followed by 8 lo rows, so that an accumulator load hands both to one thread.
__device__ __forceinline__ int op_row(int r) { return 16 * (r >> 3) + (r & 7); }
// Element offset of (tile row, column i) in a tiled operand: tile row in [0, 2 rk).
__device__ __forceinline__ size_t op_off(int rk, int row, int i) {
    const int kc = i >> 6, w = i & 63;
    return (size_t)kc * (size_t)(2 * rk * kTileK) + (size_t)(row * kTileK + ((((w >> 3) ^ (row & 7)) << 3) | (w & 7)));
}
// operand element (r, i) as hi + lo
__device__ __forceinline__ void store_hilo(__nv_bfloat16 *buf, int rk, int r, int i, float v) {
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    buf[op_off(rk, op_row(r), i)] = h;
    buf[op_off(rk, op_row(r) + 8, i)] = __float2bfloat16_rn(v - __bfloat162float(h));
}
__device__ __forceinline__ void bulk_load_1d(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// ---- tcgen05 (5th-generation tensor core) helpers ---------------------------------------------
constexpr int kTmemCols = 512;  // two accumulator buffers of 256 fp32 columns each
constexpr int kAccStride = 256;
constexpr int kEpiWarps = 4;    // warps 0-3: one tensor-memory lane quadrant each
constexpr int kMmaWarp = 4;
constexpr int kEpiPitch = kTileNP + 8;             // floats per row of the epilogue tile (bank spread)
constexpr int kXWarp = 5;      // issues the operand copies of a GEMM phase

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// mbarrier arrive once every MMA issued so far by this thread has completed
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// Shared-memory matrix descriptor of a K-major bf16 tile stored as rows of 128 bytes with the
// 128-byte swizzle (what the TMA copies write): start address / 16, leading byte offset unused (1),
// stride between 8-row groups 1024 bytes, descriptor version 1, layout type 2 (128-byte swizzle).
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}
// Instruction descriptor, kind::f16: fp32 accumulate, A and B bf16, both K-major, M = m, N = n.
__device__ __forceinline__ uint32_t umma_idesc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// 16 lanes x 64 columns of the accumulator (the 16-lane x 256-bit shape, eight times along the columns).
// Thread (g = lane / 4, t = lane % 4) receives, for column block k = 0..7: v[4k], v[4k+1] = lane g,
// columns 8k + 2t, 8k + 2t + 1 and v[4k+2], v[4k+3] = lane g + 8, the same columns.  The wait is part
// of the same statement so that no use of the results can be scheduled before it.
__device__ __forceinline__ void tc_ld_16x64(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,"
        "%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void red_add_v4(float *dst, float4 v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// Slot schedule of the ring, identical in every role that walks it (weight producer, operand issuer,
// MMA issuer).  Unit j of this CTA's share of a GEMM takes the next slot of the full cycle, except
// the first stages_lo units of an out-projection - the ones fetched while the attention phase still
// owns the upper slots - which cycle through the lower slots only.  One parity bit per slot.
struct RingPos {
    int pos_all = 0, pos_lo = 0;
    uint32_t par = 0, used = 0;
};
__device__ __forceinline__ int ring_next(RingPos &r, bool lo_only, int S, int S1, uint32_t &parity) {
    int s;
    if (lo_only) { s = r.pos_lo; if (++r.pos_lo == S1) r.pos_lo = 0; }
    else { s = r.pos_all; if (++r.pos_all == S) r.pos_all = 0; }
    parity = (r.par >> s) & 1u;
    r.par ^= 1u << s;
    r.used |= 1u << s;
    return s;
}
__device__ __forceinline__ bool ring_lo_only(const GemmDesc &g, int j, int S1) { return g.kind == 1 && j < S1; }

struct alignas(16) Shared {
    volatile int arrived;   // grid barriers this CTA has arrived at: its scratch is free of the phase in front of the last of them
    volatile int passed;    // grid barriers seen to be complete
    volatile int abort;     // some wait in this CTA gave up
    volatile int go;        // snapshot of !abort taken inside the grid barrier: uniform for all work threads
    int epoch;              // grid barriers arrived at (thread 0's)
    int flag;
    long long wait_limit;   // cycles after which a wait that takes work gives up (the drain waits of the error path keep kWaitCycles)
    uint32_t tmem_base;     // base address of this CTA's tensor memory
    int ltab_staged;        // the layers' gain / bias pointers are in shared memory (else: more layers than the table holds)
};
// The phase functions find their state at fixed shared-memory addresses: nothing is passed to them and nothing is kept in
// registers across their calls for it, and a field is one shared-memory load with an immediate address.
constexpr int kAttnBars = 16;
struct alignas(128) SharedBlock {
    uint8_t params[(sizeof(FwdParams) + 63) / 64 * 64];  // the kernel parameters, copied once (see forward_kernel)
    Shared state;
    int seq[128];                                  // committed length [64] and rows of this pass [64], per sequence
    const float *ltab[8 * kMaxStagedLayers + 2];   // the layers' gain / bias pointers, then the final norm's
    uint64_t fullW[32], fullX[32], empty[32];      // ring slots: weights there, operand there, free again
    uint64_t accFull[2], accEmpty[2], mmaDone;     // accumulators
    uint64_t abar[kAttnBars];                      // the tensor-core attention's barriers, and
    uint32_t acnt[kAttnBars];                      // the phases they have completed
    RingPos role_rp[2];  // the MMA issuer's and the operand issuer's walk of the ring, between GEMMs
    int role_seg[8];     // per work warp: tile segments so far
    int epi_ok[4];       // the epilogue warps' wait results
    uint32_t tmem_slot;
    double red[16];      // block reductions
    float epi_tile[8 * kEpiPitch];
};
__device__ __forceinline__ SharedBlock &shared_block() {
    __shared__ SharedBlock blk;
    return blk;
}
__device__ __forceinline__ FwdParams &params_copy() { return *reinterpret_cast<FwdParams *>(shared_block().params); }
__device__ __forceinline__ Shared *shared_state() { return &shared_block().state; }
__device__ __forceinline__ const int *staged_len() { return shared_block().seq; }
__device__ __forceinline__ const float *const *staged_ltab() { return shared_state()->ltab_staged ? shared_block().ltab : nullptr; }

// Bounded wait that also gives up as soon as another thread of the CTA has.
__device__ __forceinline__ bool mbar_wait_or_abort(uint64_t *bar, uint32_t parity, const Shared *sh) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (sh->abort || clock64() - t0 > sh->wait_limit) return false;
    }
    return true;
}

// The same as a pure poll (a suspended waiter wakes up late; used where a hand-off is on the critical path).
__device__ __forceinline__ bool mbar_spin_or_abort(uint64_t *bar, uint32_t parity, const Shared *sh) {
    if (mbar_test_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_test_wait(bar, parity)) {
        if (sh->abort || clock64() - t0 > sh->wait_limit) return false;
    }
    return true;
}

// Poll (bounded) until grid barrier number `epoch` is complete; one thread.
__device__ __forceinline__ bool grid_poll(const FwdParams &p, Shared *sh, int epoch) {
    const unsigned target = (unsigned)epoch * gridDim.x;
    if (ld_acquire(p.gbar) < target) {
        const long long t0 = clock64();
        while (ld_acquire(p.gbar) < target)
            if (sh->abort || clock64() - t0 > sh->wait_limit) return false;
    }
    sh->passed = epoch;
    return true;
}
// CTA 0's stamp of a barrier: its completion where a thread of that CTA waits for it (grid_sync, or the operand issuer of the GEMM
// behind an arrival), else the CTA's arrival.
__device__ __forceinline__ void grid_stamp(const FwdParams &p, int epoch) {
    if (p.trace && blockIdx.x == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        p.trace[epoch] = t;
    }
}

// Arrival of the 256 work threads at the next grid barrier; what they wrote before it is published.
// One release (and where the barrier is waited for, one acquire), both thread 0's: the CTA barriers around them pass them on to
// the other threads.  A fence per thread in front and one behind the poll made two more trips to L2 of every barrier (7B
// verification 3486 -> 3371 us, 1.4B 945 -> 899).
__device__ __forceinline__ bool grid_arrive_work(const FwdParams &p, Shared *sh) {
    // What this thread did in shared memory is over before the producer's copies may land there.  (Its writes to global memory reach
    // other CTAs' bulk copies through the release below, the operand issuer's acquire and that thread's proxy fence.  The general
    // fence here, in every thread, costs each barrier half a microsecond: a layer of the 7B verification 100.7 us instead of 99.5,
    // at batch 8 159.7 / 158.2, of the 7B's draft there 47.1 / 44.5, of 2.7B 54.9 / 54.1.)
    fence_async_shared();
    named_bar(1, kWorkThreads);
    if (threadIdx.x != 0) return true;
    const int epoch = ++sh->epoch;
    bool ok = sh->abort == 0;
    __threadfence_block();  // (the producer reads `arrived` without a barrier)
    sh->arrived = epoch;
    // (the count is the sum of all arrivals: nobody arrives at a barrier before the one in front of it is complete)
    if (ok && sh->passed < epoch - 1) ok = grid_poll(p, sh, epoch - 1);
    if (ok) red_release_add(p.gbar, 1u);
    return ok;
}
// Grid barrier.  Returns false (the same value in every work thread of the CTA) once a wait has timed out anywhere in this CTA;
// the caller then stops.
__device__ __noinline__ bool grid_sync() {
    const FwdParams &p = params_copy();
    Shared *sh = shared_state();
    bool ok = grid_arrive_work(p, sh);
    if (threadIdx.x == 0) {
        ok = ok && grid_poll(p, sh, sh->epoch);
        if (!ok) {
            set_status(p.status, kTimeoutCode);
            sh->abort = 1;
        }
        sh->go = ok ? 1 : 0;
        grid_stamp(p, sh->epoch);
    }
    named_bar(1, kWorkThreads);
    return sh->go != 0;
}

// Arrival without a wait: in front of a GEMM, whose operand issuer waits for the barrier itself (gemm_desc's `need`) while the other
// roles set themselves up - the epilogue needs the other CTAs' zeroing of its output, but has nothing to reduce before operand
// copies, MMAs and commit have passed the issuer's wait on to it; and of a CTA whose next work does not depend on what the
// others publish there.  The barrier behind that work waits for this one first where nobody has (a time-out in between
// is found there as well).
__device__ __noinline__ void grid_arrive() {
    const FwdParams &p = params_copy();
    Shared *sh = shared_state();
    const bool ok = grid_arrive_work(p, sh);
    if (threadIdx.x == 0) {
        if (!ok) {
            set_status(p.status, kTimeoutCode);
            sh->abort = 1;
        }
        grid_stamp(p, sh->epoch);  // (where the operand issuer waits for it, its stamp replaces this one)
    }
}

// The barrier counter and its neighbours live in the cache's header, which kv_init zeroes; every launch leaves them at
// zero again: one thread per CTA calls this as the CTA's last step, whatever way it came there, and the last one clears
// them.  (A memset in front of every launch cost a stream operation of 2-3 us.)
__device__ __forceinline__ void leave_grid(unsigned *gbar) {
    __threadfence();
    if (atomicAdd(gbar + 16, 1u) == gridDim.x - 1) {
        atomicExch(gbar, 0u);
        atomicExch(gbar + 8, 0u);
        atomicExch(gbar + 16, 0u);
    }
}

// Count of attention CTAs that have finished their items, over the layers of this pass (cleared with the
// barrier counter).  With few attention items in a parallel-residual block the CTAs
// without an item run the MLP-out GEMM beside the attention and go straight on to the out-projection:
// its operand issuer waits for this count as well as for the barrier behind the activation, which says nothing of the attention.
__device__ __forceinline__ unsigned *attn_done(const FwdParams &p) { return p.gbar + 8; }
__device__ __noinline__ void attn_signal() {
    const FwdParams &p = params_copy();
    Shared *sh = shared_state();
    named_bar(1, kWorkThreads);
    if (threadIdx.x == 0 && sh->abort == 0) red_release_add(attn_done(p), 1u);
}

// ---- non-GEMM phases (256 work threads) -------------------------------------------------------

// two sums in one exchange
__device__ __forceinline__ void block_sum2_work(double &a, double &b, double *red) {
    a = warp_sum(a);
    b = warp_sum(b);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    named_bar(2, kWorkThreads);
    if (lane == 0) { red[w] = a; red[kConsumerWarps + w] = b; }
    named_bar(2, kWorkThreads);
    double ta = 0.0, tb = 0.0;
#pragma unroll
    for (int i = 0; i < kConsumerWarps; ++i) { ta += red[i]; tb += red[kConsumerWarps + i]; }
    a = ta;
    b = tb;
}

// zero a [R, n] fp32 buffer (row pitch ld), spread over the whole grid
__device__ __forceinline__ void grid_zero(float *dst, int R, int n, int ld) {
    if (n == ld && ((R * (long long)n) & 3) == 0) {  // contiguous: 16-byte stores
        const long long total4 = (long long)R * n / 4;
        float4 *d4 = reinterpret_cast<float4 *>(dst);
        for (long long i = (long long)blockIdx.x * kWorkThreads + threadIdx.x; i < total4;
             i += (long long)gridDim.x * kWorkThreads)
            d4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const long long total = (long long)R * n;
    for (long long i = (long long)blockIdx.x * kWorkThreads + threadIdx.x; i < total;
         i += (long long)gridDim.x * kWorkThreads) {
        int r = (int)(i / n), c = (int)(i % n);
        dst[(size_t)r * ld + c] = 0.f;
    }
}

// Norm of every row of x into hi/lo operand buffers (one or two gain/bias sets from the same
// statistics); one CTA per row.  Bound by latency: a barrier, the row, its sums, the operand.  The row (Q float4 per thread)
// stays in registers between the statistics and the write pass, and gains and biases are loaded with it: prefetched into L1 -
// of which there is next to none - under the statistics, they were a second trip behind them (a layer of 1.4B 32.9 -> 32.5 us, of
// its draft 21.1 -> 20.4, of 12B 115.5 -> 114.4; of 7B and 2.7B 0.1-0.2).  Q is a template parameter so
// that a call executes only the code its row width needs: the instructions of a phase are not in
// the instruction cache when it starts (the kernel is far larger than that cache), and every KB of
// straight-line code costs a fraction of a microsecond to fetch.
__device__ __forceinline__ void norm_emit(const FwdParams &p, int r, int i, const float4 v, float mu, float rs,
                                          const float4 gg, const float4 bb, int op) {
    const float y0 = (v.x - mu) * rs * gg.x + bb.x, y1 = (v.y - mu) * rs * gg.y + bb.y;
    const float y2 = (v.z - mu) * rs * gg.z + bb.z, y3 = (v.w - mu) * rs * gg.w + bb.w;
    const __nv_bfloat162 h01 = __floats2bfloat162_rn(y0, y1), h23 = __floats2bfloat162_rn(y2, y3);
    const __nv_bfloat162 l01 = __floats2bfloat162_rn(y0 - __low2float(h01), y1 - __high2float(h01));
    const __nv_bfloat162 l23 = __floats2bfloat162_rn(y2 - __low2float(h23), y3 - __high2float(h23));
    __nv_bfloat16 *hi = p.op[op] + op_off(p.rk, op_row(r), 4 * i);
    __nv_bfloat16 *lo = p.op[op] + op_off(p.rk, op_row(r) + 8, 4 * i);
    uint2 hv, lv;
    hv.x = *reinterpret_cast<const uint32_t *>(&h01); hv.y = *reinterpret_cast<const uint32_t *>(&h23);
    lv.x = *reinterpret_cast<const uint32_t *>(&l01); lv.y = *reinterpret_cast<const uint32_t *>(&l23);
    *reinterpret_cast<uint2 *>(hi) = hv;
    *reinterpret_cast<uint2 *>(lo) = lv;
}
__device__ __forceinline__ float4 norm_vec(const float *v, int i, int n4) {  // (no bias: zeros)
    return v && i < n4 ? __ldg(reinterpret_cast<const float4 *>(v) + i) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// Entry i of the table of gains and biases: eight per layer (norm 1 at 0, norm 2 at 4), then the final norm's two.  The norms find
// their vectors by that one number: as six arguments through three functions they were reloaded from the stack at the head of
// every norm (with the zeroing in front of the norm, so that nothing is kept across it: 7B verification 3252 -> 3238 us, at
// batch 8 5128 -> 5061, 1.4B 833 -> 807).
__device__ __forceinline__ const float *norm_ptr(const FwdParams &p, int i) {
    const float *const *lt = staged_ltab();
    if (lt) return lt[i];
    const int l = i >> 3;
    return l < p.n_layers ? (&layer_desc(p.md, l)->ln1_g)[i & 7] : (i & 1) ? p.md->lnf_b : p.md->lnf_g;
}

// Q: float4 per thread, rows up to Q * 1024 wide.  Wider rows (TAIL: beyond 5120) are read again, with what goes with them.  Eight
// steps in registers instead - the second set's vectors behind the sums, as all four do not fit - were the longer way up to 7168
// columns and no shorter beyond (eight layers, us, five / eight: two sets, d = 5632 1247 / 1284, 7168 1828 / 1860, 8192 2307 / 2324;
// one set, 5632 1331 / 1345, 7168 1926 / 1927, 8192 2375 / 2366).
// set: where the vectors stand in the pointer table (see norm_ptr); TWO: norm 2 of the same layer as well.
template <int Q, bool TWO, bool TAIL>
__device__ __noinline__ void norm_rows(int set) {
    const FwdParams &p = params_copy();
    const float *g1 = norm_ptr(p, set), *b1 = norm_ptr(p, set + 1);
    const float *g2 = TWO ? norm_ptr(p, set + 4) : nullptr, *b2 = TWO ? norm_ptr(p, set + 5) : nullptr;
    const int n4 = p.d >> 2;  // d is a multiple of 8
    for (int r = blockIdx.x; r < p.R; r += gridDim.x) {
        const float4 *x4 = reinterpret_cast<const float4 *>(p.x + (size_t)r * p.d);
        float4 xv[Q], gv[Q], bv[Q], hv[TWO ? Q : 1], cv[TWO ? Q : 1];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int i = threadIdx.x + q * kWorkThreads;
            xv[q] = i < n4 ? __ldcg(x4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
            gv[q] = norm_vec(g1, i, n4);
            bv[q] = norm_vec(b1, i, n4);
            if constexpr (TWO) {
                hv[q] = norm_vec(g2, i, n4);
                cv[q] = norm_vec(b2, i, n4);
            }
        }
        double s1 = 0.0, s2 = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            s1 += (double)xv[q].x + (double)xv[q].y + (double)xv[q].z + (double)xv[q].w;
            s2 += (double)xv[q].x * xv[q].x + (double)xv[q].y * xv[q].y + (double)xv[q].z * xv[q].z + (double)xv[q].w * xv[q].w;
        }
        if constexpr (TAIL) {
#pragma unroll 1
            for (int i = threadIdx.x + Q * kWorkThreads; i < n4; i += kWorkThreads) {
                const float4 v = __ldcg(x4 + i);
                s1 += (double)v.x + (double)v.y + (double)v.z + (double)v.w;
                s2 += (double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z + (double)v.w * v.w;
            }
        }
        block_sum2_work(s1, s2, shared_block().red);
        double mean = 0.0, var;
        if (p.norm_kind == 0) {
            mean = s1 * p.inv_d;
            var = s2 * p.inv_d - mean * mean;
            if (var < 0.0) var = 0.0;
        } else {
            var = s2 * p.inv_d;
        }
        const float mu = (float)mean, rs = (float)rsqrt(var + (double)p.eps);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int i = threadIdx.x + q * kWorkThreads;
            if (i < n4) {
                norm_emit(p, r, i, xv[q], mu, rs, gv[q], bv[q], OP_XN1);
                if constexpr (TWO) norm_emit(p, r, i, xv[q], mu, rs, hv[q], cv[q], OP_XN2);
            }
        }
        if constexpr (TAIL) {
#pragma unroll 1
            for (int i = threadIdx.x + Q * kWorkThreads; i < n4; i += kWorkThreads) {
                const float4 v = __ldcg(x4 + i);
                norm_emit(p, r, i, v, mu, rs, norm_vec(g1, i, n4), norm_vec(b1, i, n4), OP_XN1);
                if constexpr (TWO) norm_emit(p, r, i, v, mu, rs, norm_vec(g2, i, n4), norm_vec(b2, i, n4), OP_XN2);
            }
        }
    }
}

template <bool TWO>
__device__ __forceinline__ void norm_widths(int set) {
    const int n4 = params_copy().d >> 2;
    if (n4 <= kWorkThreads) norm_rows<1, TWO, false>(set);
    else if (n4 <= 2 * kWorkThreads) norm_rows<2, TWO, false>(set);
    else if (n4 <= 3 * kWorkThreads) norm_rows<3, TWO, false>(set);
    else if (n4 <= 4 * kWorkThreads) norm_rows<4, TWO, false>(set);
    else if (n4 <= 5 * kWorkThreads) norm_rows<5, TWO, false>(set);
    else norm_rows<5, TWO, true>(set);
}

// The norm in front of layer l's first GEMM(s) - or of the LM head - and the zeroing of what they accumulate into (first: nothing
// has to be kept across the norm then).
__device__ __noinline__ void norm_for_layer(int l) {
    const FwdParams &p = params_copy();
    if (l < p.n_layers) {
        grid_zero(p.qkv, p.R, 3 * p.d, 3 * p.d);
        if (p.parallel) {
            grid_zero(p.t_in, p.R, p.d_in, p.d_in);
            norm_widths<true>(8 * l);
            return;
        }
    } else if (p.want_logits) {
        grid_zero(p.logits, p.R, p.V, p.V);
    } else {
        return;
    }
    norm_widths<false>(8 * l);
}
// ... and between the two halves of a sequential block.
__device__ __noinline__ void norm_mid_layer(int l) {
    const FwdParams &p = params_copy();
    grid_zero(p.t_in, p.R, p.d_in, p.d_in);
    norm_widths<false>(8 * l + 4);
}

// MLP activation of t_in into the hi/lo operand of the down projection, spread over the grid
__device__ __noinline__ void act_phase() {
    const FwdParams &p = params_copy();
    const int f4 = p.F >> 2;
    const long long total = (long long)p.R * f4;
    for (long long i = (long long)blockIdx.x * kWorkThreads + threadIdx.x; i < total;
         i += (long long)gridDim.x * kWorkThreads) {
        const int r = (int)(i / f4), c = (int)(i % f4);
        const float4 *t = reinterpret_cast<const float4 *>(p.t_in + (size_t)r * p.d_in);
        const float4 a = __ldcg(t + c);
        float y0, y1, y2, y3;
        if (p.swiglu) {
            const float4 u = __ldcg(t + f4 + c);
            y0 = silu(a.x) * u.x; y1 = silu(a.y) * u.y; y2 = silu(a.z) * u.z; y3 = silu(a.w) * u.w;
        } else {
            y0 = gelu_erf(a.x); y1 = gelu_erf(a.y); y2 = gelu_erf(a.z); y3 = gelu_erf(a.w);
        }
        const __nv_bfloat162 h01 = __floats2bfloat162_rn(y0, y1), h23 = __floats2bfloat162_rn(y2, y3);
        const __nv_bfloat162 l01 = __floats2bfloat162_rn(y0 - __low2float(h01), y1 - __high2float(h01));
        const __nv_bfloat162 l23 = __floats2bfloat162_rn(y2 - __low2float(h23), y3 - __high2float(h23));
        uint2 hv, lv;
        hv.x = *reinterpret_cast<const uint32_t *>(&h01); hv.y = *reinterpret_cast<const uint32_t *>(&h23);
        lv.x = *reinterpret_cast<const uint32_t *>(&l01); lv.y = *reinterpret_cast<const uint32_t *>(&l23);
        __nv_bfloat16 *base = p.op[OP_ACT];
        *reinterpret_cast<uint2 *>(base + op_off(p.rk, op_row(r), 4 * c)) = hv;
        *reinterpret_cast<uint2 *>(base + op_off(p.rk, op_row(r) + 8, 4 * c)) = lv;
    }
}

__device__ __noinline__ void setup_phase() {
    const FwdParams &p = params_copy();
    if (blockIdx.x == gridDim.x - 1)  // (they are used behind this phase's barrier; every user leaves its own at zero)
        for (int i = threadIdx.x; i < p.B * p.H; i += kWorkThreads) p.tickets[i] = 0;
    // K not a multiple of 64: the last tile's unused columns must be finite (the weight copy zero-fills its own)
    for (int o = 0; o < 4; ++o) {
        const int K = p.op_ld[o], pad = (-K) & (kTileK - 1);
        if (!p.op[o] || !pad) continue;
        for (int e = blockIdx.x * kWorkThreads + threadIdx.x; e < 2 * p.rk * pad; e += gridDim.x * kWorkThreads)
            p.op[o][op_off(p.rk, e / pad, K + e % pad)] = __float2bfloat16_rn(0.f);
    }
    const int half = p.rotary_dim / 2;
    for (int r = blockIdx.x; r < p.R; r += gridDim.x) {
        const int b = r / p.M, j = r % p.M;
        int n = p.cur_step > 0 ? 1 : (p.n_rows ? p.n_rows[b] : p.M);
        n = max(0, min(n, p.M));
        const int len = __ldcg(p.len + b);  // (advanced between the steps of a draft loop)
        const bool fits = len + n <= p.S && (p.pos_limit == 0 || len + n <= p.pos_limit);
        if (!fits) {
            n = 0;
            if (threadIdx.x == 0) set_status(p.status, -3);
        }
        int pos = len + j, lim = p.S - 1;
        if (p.pos_limit && p.pos_limit - 1 < lim) lim = p.pos_limit - 1;
        if (pos > lim) pos = lim;
        if (threadIdx.x == 0) {
            p.ri.seq[r] = b;
            p.ri.pos[r] = pos;
            p.ri.valid[r] = j < n;
            if (j == 0) p.ri.n_eff[b] = n;
        }
        for (int i = threadIdx.x; i < half; i += kWorkThreads) {
            double theta = (double)pos * exp2(-2.0 * i / p.rotary_dim * log2((double)p.rotary_base));
            double s, c;
            sincos(theta, &s, &c);
            p.ri.rope_cos[(size_t)r * half + i] = (float)c;
            p.ri.rope_sin[(size_t)r * half + i] = (float)s;
        }
    }
}

// Bound by latency: a row's loads are all issued before the first store (a load of two bytes per step of a loop waits for the
// store before it, which may alias: a trip to DRAM per 256 columns.  From the start of a 7B pass to its first projection 22.6 -> 15.6 us).
__device__ __noinline__ void embed_phase() {
    const FwdParams &p = params_copy();
    for (int r = blockIdx.x; r < p.R; r += gridDim.x) {
        const int b = r / p.M, j = r % p.M;
        int tok = 0;
        if (__ldcg(p.ri.valid + r))
            tok = p.cur_step > 0 ? __ldcg(p.tok_out + (size_t)b * p.tok_out_stride + p.cur_step - 1) : p.tokens[(size_t)b * p.tok_stride + j];
        tok = max(0, min(tok, p.V - 1));
        const int pos = __ldcg(p.ri.pos + r);
        const __nv_bfloat16 *te = (const __nv_bfloat16 *)p.tok_emb + (size_t)tok * p.d;
        const __nv_bfloat16 *pe = p.learned_pos ? (const __nv_bfloat16 *)p.pos_emb + (size_t)pos * p.d : nullptr;
        float *x = p.x + (size_t)r * p.d;
        if (!pe && ((uintptr_t)te & 15) == 0) {
#pragma unroll 1
            for (int i0 = threadIdx.x; i0 < (p.d >> 3); i0 += 2 * kWorkThreads) {
                const int i1 = i0 + kWorkThreads;
                const uint4 t0 = __ldg(reinterpret_cast<const uint4 *>(te) + i0);
                const uint4 t1 = i1 < (p.d >> 3) ? __ldg(reinterpret_cast<const uint4 *>(te) + i1) : t0;
                auto put = [&](int i, const uint4 &t) {
                    reinterpret_cast<float4 *>(x)[2 * i] = make_float4(__uint_as_float(t.x << 16), __uint_as_float(t.x & 0xffff0000u),
                                                                       __uint_as_float(t.y << 16), __uint_as_float(t.y & 0xffff0000u));
                    reinterpret_cast<float4 *>(x)[2 * i + 1] = make_float4(__uint_as_float(t.z << 16), __uint_as_float(t.z & 0xffff0000u),
                                                                           __uint_as_float(t.w << 16), __uint_as_float(t.w & 0xffff0000u));
                };
                put(i0, t0);
                if (i1 < (p.d >> 3)) put(i1, t1);
            }
        } else {
            for (int i = threadIdx.x; i < p.d; i += kWorkThreads)
                x[i] = __bfloat162float(te[i]) + (pe ? __bfloat162float(pe[i]) : 0.f);
        }
    }
}

// ---- attention ---------------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void ldmatrix_x2_trans(uint32_t addr, uint32_t &r0, uint32_t &r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// Columns e0 .. e0+7 of one head's q or k row (fp32, `row` points at the head's first column) with
// the rotary turn of row r applied; rotary_dim and its half are multiples of 8, so the eight
// columns fall on one side of the split.  All loads are issued before the first use.
__device__ __forceinline__ void rope_vec8(const FwdParams &p, const float *row, int r, int e0, float (&out)[8]) {
    const float4 a0 = __ldcg(reinterpret_cast<const float4 *>(row + e0)), a1 = __ldcg(reinterpret_cast<const float4 *>(row + e0 + 4));
    out[0] = a0.x; out[1] = a0.y; out[2] = a0.z; out[3] = a0.w; out[4] = a1.x; out[5] = a1.y; out[6] = a1.z; out[7] = a1.w;
    if (e0 < p.rotary_dim) {
        const int half = p.rotary_dim >> 1;
        const bool low = e0 < half;
        const int j0 = low ? e0 : e0 - half;
        const float *pr_ = row + (low ? e0 + half : e0 - half);
        const float4 b0 = __ldcg(reinterpret_cast<const float4 *>(pr_)), b1 = __ldcg(reinterpret_cast<const float4 *>(pr_ + 4));
        const float *cp = p.ri.rope_cos + (size_t)r * half + j0, *sp = p.ri.rope_sin + (size_t)r * half + j0;
        const float4 c0 = __ldcg(reinterpret_cast<const float4 *>(cp)), c1 = __ldcg(reinterpret_cast<const float4 *>(cp + 4));
        const float4 s0 = __ldcg(reinterpret_cast<const float4 *>(sp)), s1 = __ldcg(reinterpret_cast<const float4 *>(sp + 4));
        const float pb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        const float cc[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
        const float ss[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
        for (int u = 0; u < 8; ++u) out[u] = low ? out[u] * cc[u] - pb[u] * ss[u] : pb[u] * ss[u] + out[u] * cc[u];
    }
}

// four output columns of one row of the out-projection operand, as bf16 hi + lo
__device__ __forceinline__ void store_ao4(const FwdParams &p, int r, int col, float4 y) {
    const __nv_bfloat162 h01 = __floats2bfloat162_rn(y.x, y.y), h23 = __floats2bfloat162_rn(y.z, y.w);
    const __nv_bfloat162 l01 = __floats2bfloat162_rn(y.x - __low2float(h01), y.y - __high2float(h01));
    const __nv_bfloat162 l23 = __floats2bfloat162_rn(y.z - __low2float(h23), y.w - __high2float(h23));
    uint2 hv, lv;
    hv.x = *reinterpret_cast<const uint32_t *>(&h01); hv.y = *reinterpret_cast<const uint32_t *>(&h23);
    lv.x = *reinterpret_cast<const uint32_t *>(&l01); lv.y = *reinterpret_cast<const uint32_t *>(&l23);
    __nv_bfloat16 *base = p.op[OP_AO];
    *reinterpret_cast<uint2 *>(base + op_off(p.rk, op_row(r), col)) = hv;
    *reinterpret_cast<uint2 *>(base + op_off(p.rk, op_row(r) + 8, col)) = lv;
}

// The item that finishes last for a (sequence, head) merges the splits' partials (m, l, o) of all its
// rows into the out-projection operand; 256 threads.
__device__ __forceinline__ void merge_splits(const FwdParams &p, int r0, int h, int Dh) {
    const int tid = threadIdx.x, q4 = Dh >> 2;
    auto store_ao4 = [&](int r, int col, float4 y) { ssd::store_ao4(p, r, col, y); };
            // one work item = four columns of one row; the loads of up to eight splits are issued together
            for (int idx = tid; idx < p.M * q4; idx += kAttnThreadsP) {
                const int m = idx / q4, e = (idx % q4) * 4;
                const size_t base = ((size_t)(r0 + m) * p.H + h) * p.n_split;
                float mx = -INFINITY, L = 0.f;
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int s0 = 0; s0 < p.n_split; s0 += 8) {
                    float pm[8], pl[8];
                    float4 po[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const bool in = s0 + u < p.n_split;
                        pm[u] = in ? __ldcg(p.part_m + base + s0 + u) : -INFINITY;
                        pl[u] = in ? __ldcg(p.part_l + base + s0 + u) : 0.f;
                        po[u] = in ? __ldcg(reinterpret_cast<const float4 *>(p.part_o + (base + s0 + u) * Dh + e))
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    float bm = mx;
#pragma unroll
                    for (int u = 0; u < 8; ++u) bm = fmaxf(bm, pm[u]);
                    if (bm == -INFINITY) continue;
                    const float f = exp2f(mx - bm);  // 0 while nothing has been accumulated
                    L *= f; acc.x *= f; acc.y *= f; acc.z *= f; acc.w *= f;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (pm[u] == -INFINITY) continue;
                        const float w = exp2f(pm[u] - bm);
                        L = fmaf(pl[u], w, L);
                        acc.x = fmaf(po[u].x, w, acc.x); acc.y = fmaf(po[u].y, w, acc.y);
                        acc.z = fmaf(po[u].z, w, acc.z); acc.w = fmaf(po[u].w, w, acc.w);
                    }
                    mx = bm;
                }
                const float inv = L > 0.f ? 1.f / L : 0.f;
                store_ao4(r0 + m, h * Dh + e, make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
            }
}

// Positions per split of a sequence that holds `total` positions after this pass: equal shares of whole
// tiles, taken on the device from the sequence's own length.  The host fixes only the number of splits
// (from an upper bound of the lengths), so ragged sequences are each cut evenly and a loose bound costs
// nothing but an empty split.
__device__ __forceinline__ int split_chunk(const FwdParams &p, int total, int tile) {
    const int c = (max(total, 1) + p.n_split - 1) / p.n_split;
    return (c + tile - 1) / tile * tile;
}

constexpr int kAttnRows = 16;  // query rows per item (one MMA row tile)
constexpr int kAttnBufs = 3;   // K/V chunk buffers: two chunks (64 KB at head 128) in flight per SM
__host__ __device__ inline size_t attn_scratch_bytes(int Dh) {
    // Q hi/lo [16][Dh+8] bf16, kAttnBufs K/V chunk buffers [2][64][Dh+8] bf16 each, per-warp (m, l) [8][16] fp32 x 2,
    // per-thread partial scores [256][8] fp32
    return (size_t)2 * kAttnRows * (Dh + 8) * 2 + (size_t)kAttnBufs * 2 * kAttnTile * (Dh + 8) * 2 + 2 * 8 * kAttnRows * 4 +
           (size_t)256 * 8 * 4;
}

// Attention of up to 16 query rows of one (sequence, head) over one split of the position axis, by
// 256 threads, on tensor cores.  K/V chunks of 64 positions are fetched with cp.async into three
// buffers (the next two chunks load while this one is used).  Warp w owns positions 16 (w & 3) .. +15
// of each chunk and the output columns of half (w >> 2) of the head.  The two warps of a position
// group each contract half of the head dimension of the 16 x 16 score block S = Q K^T (Q as bf16
// hi + lo) and exchange the halves, so both hold S; each keeps its own running max / sum (equal in
// both, the sum of two halves being order-independent) and adds P V (P as bf16
// hi + lo) to its 16 x Dh/2 accumulators -- no exchange between warps until the end, where the
// four position groups are merged in shared memory.  Rows of this pass (positions >= len) take
// their keys / values from qkv (rotary, cache rounding) and the split that owns them appends them
// to the cache.  With one split the result goes straight to the out-projection operand; otherwise
// partials are written and the split that finishes last merges them.  All exponentials are base 2.
__device__ __noinline__ void attention_items(int layer) {
    const FwdParams &p = params_copy();
    Shared *sh = shared_state();
    uint8_t *scratch = smem_base() + p.attn_smem_off;
#pragma unroll 1
    for (int item = blockIdx.x; item < p.attn_items; item += gridDim.x) {
    const int MT = (p.M + kAttnRows - 1) / kAttnRows;
    const int mt = item % MT, rest = item / MT;
    const int split = rest % p.n_split, bh = rest / p.n_split, b = bh / p.H, h = bh % p.H;
    const int Dh = p.Dh, d = p.d, pitch = Dh + 8;
    const uint32_t pitchB = (uint32_t)pitch * 2u;
    __nv_bfloat16 *Qhi = reinterpret_cast<__nv_bfloat16 *>(scratch);
    __nv_bfloat16 *Qlo = Qhi + kAttnRows * pitch;
    __nv_bfloat16 *KV = Qlo + kAttnRows * pitch;  // buffer i: K at KV + i * 2 * 64 * pitch, V 64 * pitch later
    float *mw = reinterpret_cast<float *>(KV + kAttnBufs * 2 * kAttnTile * pitch);
    float *lw = mw + 8 * kAttnRows;
    float *sx = lw + 8 * kAttnRows;  // score halves exchanged between the two warps of a position group
    float *o_acc = reinterpret_cast<float *>(KV);  // [4][16][Dh] fp32, reuses the chunk buffers after the loop

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int pg = warp & 3, dhh = warp >> 2;
    const int nk = Dh >> 4;          // k-steps of Q K^T; also 8-column output tiles per head half
    const int dh0 = dhh * (Dh >> 1);
    const int n_rows = staged_len()[64 + b];
    const int len = staged_len()[b];
    const int r0 = b * p.M, m_base = mt * kAttnRows;
    const int chunk = split_chunk(p, len + n_rows, kAttnTile);
    const int p_begin = split * chunk;
    const int p_end = min(p_begin + chunk, len + n_rows);
    const float sc = p.attn_scale * 1.4426950408889634f;  // scores in log2 units

    __nv_bfloat16 *kc = (__nv_bfloat16 *)(p.cache + (size_t)layer * p.layer_bytes) + ((size_t)(b * 2) * p.H + h) * p.S * Dh;
    __nv_bfloat16 *vc = kc + (size_t)p.H * p.S * Dh;
    const int vpr = Dh >> 3;  // 16-byte vectors per row
    auto load_chunk = [&](int c) {
        __nv_bfloat16 *Kb = KV + (size_t)(c % kAttnBufs) * 2 * kAttnTile * pitch, *Vb = Kb + kAttnTile * pitch;
        const int t0 = p_begin + c * kAttnTile, np = min(kAttnTile, p_end - t0);
        const int prow = tid >> 4, v8 = tid & 15;  // 16 threads per row, 16 rows per pass
        if (v8 < vpr) {
            if (t0 + kAttnTile <= len) {  // the common case: all 64 positions come from the cache
                const __nv_bfloat16 *ks = kc + (size_t)(t0 + prow) * Dh + v8 * 8, *vs = vc + (size_t)(t0 + prow) * Dh + v8 * 8;
                __nv_bfloat16 *dk = Kb + prow * pitch + v8 * 8, *dv = Vb + prow * pitch + v8 * 8;
#pragma unroll
                for (int q = 0; q < kAttnTile / 16; ++q) {
                    cp_async16(dk + q * 16 * pitch, ks + (size_t)q * 16 * Dh);
                    cp_async16(dv + q * 16 * pitch, vs + (size_t)q * 16 * Dh);
                }
            } else {
#pragma unroll 1
                for (int q = 0; q < kAttnTile / 16; ++q) {
                    const int pp = prow + 16 * q, pos = t0 + pp;
                    __nv_bfloat16 *dk = Kb + pp * pitch + v8 * 8, *dv = Vb + pp * pitch + v8 * 8;
                    if (pp >= np) {  // beyond the split: zeros (P is 0 there, but 0 * garbage must not be NaN)
                        *reinterpret_cast<uint4 *>(dk) = make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4 *>(dv) = make_uint4(0, 0, 0, 0);
                    } else if (pos < len) {
                        const size_t go = (size_t)pos * Dh + v8 * 8;
                        cp_async16(dk, kc + go);
                        cp_async16(dv, vc + go);
                    } else {  // a row of this pass: from qkv, position-encoded and rounded as the cache stores it
                        const int r = r0 + (pos - len);
                        const float *krow = p.qkv + (size_t)r * 3 * d + d + h * Dh;
                        float kf[8];
                        rope_vec8(p, krow, r, v8 * 8, kf);
                        const float4 v0 = __ldcg(reinterpret_cast<const float4 *>(krow + d + v8 * 8));
                        const float4 v1 = __ldcg(reinterpret_cast<const float4 *>(krow + d + v8 * 8 + 4));
                        const float vf[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
                        __nv_bfloat16 kb[8], vb[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            kb[u] = __float2bfloat16_rn(kf[u]);
                            vb[u] = __float2bfloat16_rn(vf[u]);
                        }
                        const uint4 kq = *reinterpret_cast<uint4 *>(kb), vq = *reinterpret_cast<uint4 *>(vb);
                        *reinterpret_cast<uint4 *>(dk) = kq;
                        *reinterpret_cast<uint4 *>(dv) = vq;
                        if (mt == 0) {  // append: exactly one split owns this position
                            const size_t go = (size_t)pos * Dh + v8 * 8;
                            *reinterpret_cast<uint4 *>(kc + go) = kq;
                            *reinterpret_cast<uint4 *>(vc + go) = vq;
                        }
                    }
                }
            }
        }
        cp_async_commit();
    };

    float o[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
    const int n_chunks = p_begin < p_end ? (p_end - p_begin + kAttnTile - 1) / kAttnTile : 0;

    // kAttnBufs - 1 chunks are always in flight; one group is committed per chunk slot so that
    // "at most kAttnBufs - 1 groups pending" means "chunk c has landed"
    for (int c = 0; c < kAttnBufs - 1; ++c) {
        if (c < n_chunks) load_chunk(c); else cp_async_commit();
    }
    // ---- Q rows (rotary applied) as bf16 hi / lo: thread = (row, 8 columns) ----
    {
        const int ml = tid >> 4, v8 = tid & 15, m = m_base + ml;
        if (v8 < vpr) {
            float q[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) q[u] = 0.f;
            if (m < n_rows) rope_vec8(p, p.qkv + (size_t)(r0 + m) * 3 * d + h * Dh, r0 + m, v8 * 8, q);
            __nv_bfloat16 hq[8], lq[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                hq[u] = __float2bfloat16_rn(q[u]);
                lq[u] = __float2bfloat16_rn(q[u] - __bfloat162float(hq[u]));
            }
            *reinterpret_cast<uint4 *>(Qhi + ml * pitch + v8 * 8) = *reinterpret_cast<uint4 *>(hq);
            *reinterpret_cast<uint4 *>(Qlo + ml * pitch + v8 * 8) = *reinterpret_cast<uint4 *>(lq);
        }
    }
    for (int c = 0; c < n_chunks; ++c) {
        if (c + kAttnBufs - 1 < n_chunks) load_chunk(c + kAttnBufs - 1); else cp_async_commit();
        cp_async_wait<kAttnBufs - 1>();
        named_bar(3, kAttnThreadsP);  // chunk c (and, first time, Q) is in shared memory
        const __nv_bfloat16 *Kb = KV + (size_t)(c % kAttnBufs) * 2 * kAttnTile * pitch, *Vb = Kb + kAttnTile * pitch;
        const int pos0 = p_begin + c * kAttnTile + 16 * pg;  // this warp's 16 positions
        // ---- S = Q K^T for 16 rows x 16 positions; four independent accumulator sets (Q hi / lo x
        //      even / odd k-step) keep the dependent MMA chains short ----
        float s[2][4];
        {
            float sa[2][2][2][4];  // [hi|lo][even|odd][position tile][4]
#pragma unroll
            for (int x = 0; x < 2; ++x)
#pragma unroll
                for (int y = 0; y < 2; ++y)
#pragma unroll
                    for (int j = 0; j < 2; ++j) sa[x][y][j][0] = sa[x][y][j][1] = sa[x][y][j][2] = sa[x][y][j][3] = 0.f;
            const uint32_t qa = smem_u32(Qhi) + (uint32_t)(lane & 15) * pitchB + (uint32_t)(lane >> 4) * 16u;
            const uint32_t ql = qa + (uint32_t)kAttnRows * pitchB;
            const uint32_t ka = smem_u32(Kb) + (uint32_t)(16 * pg + (lane & 7) + 8 * (lane >> 4)) * pitchB + (uint32_t)((lane >> 3) & 1) * 16u;
            const int ks_lo = dhh ? (nk + 1) / 2 : 0, ks_hi = dhh ? nk : (nk + 1) / 2;  // this warp's half of Dh
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                if (ks >= ks_lo && ks < ks_hi) {
                    uint32_t a0, a1, a2, a3, c0, c1, c2, c3, k0, k1, k2, k3;
                    ldmatrix_x4(qa + ks * 32, a0, a1, a2, a3);
                    ldmatrix_x4(ql + ks * 32, c0, c1, c2, c3);
                    ldmatrix_x4(ka + ks * 32, k0, k1, k2, k3);  // (pos 0-7: k lo, k hi), (pos 8-15: k lo, k hi)
                    mma_bf16(sa[0][ks & 1][0], a0, a1, a2, a3, k0, k1);
                    mma_bf16(sa[1][ks & 1][0], c0, c1, c2, c3, k0, k1);
                    mma_bf16(sa[0][ks & 1][1], a0, a1, a2, a3, k2, k3);
                    mma_bf16(sa[1][ks & 1][1], c0, c1, c2, c3, k2, k3);
                }
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) s[j][e] = (sa[0][0][j][e] + sa[0][1][j][e]) + (sa[1][0][j][e] + sa[1][1][j][e]);
            // exchange with the warp that holds the other half (same position group, same lane = same elements)
            float4 *mine = reinterpret_cast<float4 *>(sx + (size_t)tid * 8);
            mine[0] = make_float4(s[0][0], s[0][1], s[0][2], s[0][3]);
            mine[1] = make_float4(s[1][0], s[1][1], s[1][2], s[1][3]);
            named_bar(8 + pg, 64);
            const float4 *other = reinterpret_cast<const float4 *>(sx + (size_t)(tid ^ 128) * 8);
            const float4 o0 = other[0], o1 = other[1];
            s[0][0] += o0.x; s[0][1] += o0.y; s[0][2] += o0.z; s[0][3] += o0.w;
            s[1][0] += o1.x; s[1][1] += o1.y; s[1][2] += o1.z; s[1][3] += o1.w;
        }
        // ---- mask, running max / sum (rows g and g + 8) ----
        float pr[2][4];
#pragma unroll
        for (int hrow = 0; hrow < 2; ++hrow) {
            const int m = m_base + g + 8 * hrow;
            float mx = -INFINITY;
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int pos = pos0 + 8 * j + 2 * t + e;
                    const bool vis = pos < p_end && pos <= len + m;
                    const float v = vis ? s[j][2 * hrow + e] * sc : -INFINITY;
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
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float pv = exp2f(s[j][2 * hrow + e] - m_new);
                        pr[j][2 * hrow + e] = pv;
                        sum += pv;
                    }
            } else {
#pragma unroll
                for (int j = 0; j < 2; ++j) pr[j][2 * hrow] = pr[j][2 * hrow + 1] = 0.f;
            }
            m_run[hrow] = m_new;
            l_run[hrow] = l_run[hrow] * f + sum;  // this thread's share; lanes are summed at the end
#pragma unroll
            for (int j = 0; j < 8; ++j) { o[j][2 * hrow] *= f; o[j][2 * hrow + 1] *= f; }
        }
        // ---- O += P V  (P as hi + lo; k = the 16 positions; n = this warp's Dh/2 columns) ----
        {
            uint32_t ph[4], pl[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {  // a0: (row g, k 2t..) a1: (row g+8, ..) a2: (row g, k 8+2t..) a3: (row g+8, ..)
                const int j = q >> 1, hrow = q & 1;
                const float x0 = pr[j][2 * hrow], x1 = pr[j][2 * hrow + 1];
                const __nv_bfloat162 hv = __floats2bfloat162_rn(x0, x1);
                ph[q] = *reinterpret_cast<const uint32_t *>(&hv);
                pl[q] = pack_bf16x2(x0 - __low2float(hv), x1 - __high2float(hv));
            }
            const uint32_t va = smem_u32(Vb) + (uint32_t)(16 * pg + (lane & 15)) * pitchB + (uint32_t)dh0 * 2u;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (j < nk) {
                    uint32_t b0, b1;
                    ldmatrix_x2_trans(va + j * 16, b0, b1);
                    mma_bf16(o[j], ph[0], ph[1], ph[2], ph[3], b0, b1);
                    mma_bf16(o[j], pl[0], pl[1], pl[2], pl[3], b0, b1);
                }
            }
        }
        named_bar(3, kAttnThreadsP);  // everyone is done with this buffer before it is refilled
    }
    if (n_chunks == 0) named_bar(3, kAttnThreadsP);  // Q stores vs. later reuse of the scratch

    // ---- merge the four position groups ----
#pragma unroll
    for (int hrow = 0; hrow < 2; ++hrow) {
        l_run[hrow] += __shfl_xor_sync(0xffffffffu, l_run[hrow], 1);
        l_run[hrow] += __shfl_xor_sync(0xffffffffu, l_run[hrow], 2);
    }
    if (t == 0) {
        mw[warp * kAttnRows + g] = m_run[0];
        mw[warp * kAttnRows + g + 8] = m_run[1];
        lw[warp * kAttnRows + g] = l_run[0];
        lw[warp * kAttnRows + g + 8] = l_run[1];
    }
    named_bar(3, kAttnThreadsP);
    // every warp scales its block to the common maximum and stores it: o_part[pg][16][Dh] (fp32, in the
    // chunk buffers, free now); the output loop adds the four position groups in a fixed order
#pragma unroll
    for (int hrow = 0; hrow < 2; ++hrow) {
        const int row = g + 8 * hrow;
        float mx = -INFINITY;
#pragma unroll
        for (int q = 0; q < 4; ++q) mx = fmaxf(mx, mw[q * kAttnRows + row]);
        const float f = (m_run[hrow] > -INFINITY) ? exp2f(m_run[hrow] - mx) : 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (j < nk) {
                float2 v2 = make_float2(o[j][2 * hrow] * f, o[j][2 * hrow + 1] * f);
                *reinterpret_cast<float2 *>(o_acc + ((size_t)pg * kAttnRows + row) * Dh + dh0 + 8 * j + 2 * t) = v2;
            }
        }
    }
    named_bar(3, kAttnThreadsP);
    const bool direct = p.n_split == 1;
    // four output columns of one real row per work item
    auto store_ao4 = [&](int r, int col, float4 y) {
        const __nv_bfloat162 h01 = __floats2bfloat162_rn(y.x, y.y), h23 = __floats2bfloat162_rn(y.z, y.w);
        const __nv_bfloat162 l01 = __floats2bfloat162_rn(y.x - __low2float(h01), y.y - __high2float(h01));
        const __nv_bfloat162 l23 = __floats2bfloat162_rn(y.z - __low2float(h23), y.w - __high2float(h23));
        uint2 hv, lv;
        hv.x = *reinterpret_cast<const uint32_t *>(&h01); hv.y = *reinterpret_cast<const uint32_t *>(&h23);
        lv.x = *reinterpret_cast<const uint32_t *>(&l01); lv.y = *reinterpret_cast<const uint32_t *>(&l23);
        __nv_bfloat16 *base = p.op[OP_AO];
        *reinterpret_cast<uint2 *>(base + op_off(p.rk, op_row(r), col)) = hv;
        *reinterpret_cast<uint2 *>(base + op_off(p.rk, op_row(r) + 8, col)) = lv;
    };
    const int q4 = Dh >> 2;  // float4 per row
    const int rows_here = max(0, min(kAttnRows, p.M - m_base));
    for (int i = tid; i < rows_here * q4; i += kAttnThreadsP) {
        const int ml = i / q4, e = (i % q4) * 4, m = m_base + ml;
        float mx = -INFINITY;
#pragma unroll
        for (int q = 0; q < 4; ++q) mx = fmaxf(mx, mw[q * kAttnRows + ml]);
        float L = 0.f;
        if (mx > -INFINITY) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float mq = mw[q * kAttnRows + ml];
                if (mq > -INFINITY) L += lw[q * kAttnRows + ml] * exp2f(mq - mx);
            }
        }
        const bool live = m < n_rows && L > 0.f;
        const int gs = kAttnRows * Dh;  // stride between position groups
        const float *oa = o_acc + ml * Dh + e;
        const float4 a0 = *reinterpret_cast<const float4 *>(oa), a1 = *reinterpret_cast<const float4 *>(oa + gs);
        const float4 a2 = *reinterpret_cast<const float4 *>(oa + 2 * gs), a3 = *reinterpret_cast<const float4 *>(oa + 3 * gs);
        float4 osum = make_float4((a0.x + a1.x) + (a2.x + a3.x), (a0.y + a1.y) + (a2.y + a3.y),
                                  (a0.z + a1.z) + (a2.z + a3.z), (a0.w + a1.w) + (a2.w + a3.w));
        if (!live) osum = make_float4(0.f, 0.f, 0.f, 0.f);
        if (direct) {
            const float inv = live ? 1.f / L : 0.f;
            store_ao4(r0 + m, h * Dh + e, make_float4(osum.x * inv, osum.y * inv, osum.z * inv, osum.w * inv));
        } else {
            const size_t slot = ((size_t)(r0 + m) * p.H + h) * p.n_split + split;
            if (e == 0) {
                p.part_m[slot] = live ? mx : -INFINITY;
                p.part_l[slot] = live ? L : 0.f;
            }
            *reinterpret_cast<float4 *>(p.part_o + slot * Dh + e) = osum;
        }
    }
    if (!direct) {
        // ticket: the item that finishes last for this (sequence, head) merges all partials
        // (one release and one acquire for the CTA, as in the grid barrier)
        named_bar(3, kAttnThreadsP);
        if (tid == 0) sh->flag = (atomic_add_acq_rel(p.tickets + bh, 1u) == (unsigned)(p.n_split * MT - 1));
        named_bar(3, kAttnThreadsP);
        if (sh->flag) {
            merge_splits(p, r0, h, Dh);
            if (tid == 0) p.tickets[bh] = 0;  // ready for the next layer (a grid barrier lies between)
        }
    }
    named_bar(3, kAttnThreadsP);  // scratch is free for the next item
    }
}

#include "attn_mma8.cuh"

// ---- attention on tcgen05 (head dim 128) ----------------------------------------------------------
// ALL query rows of one (sequence, head) - up to RP = 16 or 32 of them, so that every key and value is fetched once - over one
// split of the position axis, with the two products on the 5th-generation tensor core and the scores and the output in tensor
// memory, 128 positions per chunk:
//   S^T [128 positions x 2 RP]  = K chunk (the M = 128 operand, straight from the TMA copy of the cache)
//                                 x Q rows (RP hi + RP lo, the N operand; in log2 units)
//   O^T [128 head dims x 2 RP] += V chunk read as its transpose (MN-major M = 128 operand) x P (RP hi + RP lo)
// Roles: threads 0-127 = one position each (masks, P = exp2(S - reference), running sums in registers, P as bf16 hi + lo
// into the P tile) and, at the end, one head dim each (output); warp 4: MMA issue; warp 5: TMA copies of K and V chunks
// into a 4-stage ring; warps 6-7: rows of this pass (positions >= len) - rotary, rounding, append to the cache - written
// into the chunk tiles over what the copy brought.  Positions behind them are masked (P = 0) and
// multiply whatever the cache holds there: kv_init zeroes the cache, and all later writes are
// finite rows of earlier passes, so 0 x stale is 0.
// A row's softmax reference is the maximum of the first chunk it sees; it is only raised when a score passes it by more than
// 2^32 (fp32 sums and bf16 hi + lo carry the factor without loss), which one barrier vote per chunk finds out: no maxima are
// exchanged and O^T is not rescaled in the ordinary chunk.
// Bound: the 64 KB of K and V a chunk fetches.  7B, 17 rows x 16384 positions: 249 us a layer with two 16-row tiles that each
// walk the cache and exchange maxima in every chunk, 84 now, against 41 us of HBM time.
constexpr int kTcChunk = 128;
constexpr int kTcStages = 4;  // K / V ring stages of 32 KB: the bytes in flight set the chunk rate (3 stages: 2.7 us per chunk)
constexpr int kTcKvStage = kTcChunk * 128 * 2;  // one K or V chunk: two 64-column panels of 128 rows x 128 B
__host__ __device__ constexpr int tc_p_tiles(int rp) { return rp == 16 ? 2 : 1; }   // P tiles used in turn
__host__ __device__ constexpr int tc_scratch_bytes(int rp) {  // ring, Q tile, P tiles, maxima and sums of four warps, references and factors
    return kTcStages * kTcKvStage + (1 + tc_p_tiles(rp)) * 2 * rp * 256 + 10 * rp * 4;
}
// Its mbarriers live outside the scratch (which the weight ring reuses), are initialised once per kernel
// and keep running: cnt[i] = phases barrier i has completed before the current item.  A parity wait is
// only meaningful for a waiter that follows every phase of its barrier in order and that the barrier
// cannot pass by two phases; the threads that patch this pass's rows into a chunk skip most chunks, so
// they do not wait on the ring's barriers: the MMA issuer, which follows every stage, tells them through
// `landed` when such a chunk has arrived, and hears back through `fixed`.  p_ready goes by chunk parity, as the P tiles do:
// with two tiles the softmax may hand over P of chunk c + 1 before the issuer has looked for P of chunk c, and on one barrier
// that wait would be passed by two phases (and run to its limit).
enum { AB_KV_FULL = 0, AB_KV_FREE = kTcStages, AB_S_FULL = 2 * kTcStages, AB_P_READY = AB_S_FULL + 2, AB_O_DONE = AB_P_READY + 2 /* two each: chunk parity */,
       AB_FIXED = AB_O_DONE + 2, AB_LANDED, AB_COUNT };
constexpr float kTcMaxSlack = 32.f;

__device__ __forceinline__ void tc_ld_32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,"
        "%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// 64 consecutive columns of this thread's lane in one round trip
__device__ __forceinline__ void tc_ld_64(uint32_t taddr, float (&v)[64]) {
    uint32_t r[64];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}
// eight columns from each of two places of this warp's lane quadrant, one round trip
__device__ __forceinline__ void tc_ld_2x8(uint32_t ta, uint32_t tb, float (&a)[8], float (&b)[8]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(ta), "r"(tb)
        : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) { a[i] = __uint_as_float(r[i]); b[i] = __uint_as_float(r[8 + i]); }
}
__device__ __forceinline__ void tc_st_32(uint32_t taddr, const float (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,"
        "%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n"
        "tcgen05.wait::st.sync.aligned;\n" ::"r"(taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
        "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
        "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15])),
        "r"(__float_as_uint(v[16])), "r"(__float_as_uint(v[17])), "r"(__float_as_uint(v[18])), "r"(__float_as_uint(v[19])),
        "r"(__float_as_uint(v[20])), "r"(__float_as_uint(v[21])), "r"(__float_as_uint(v[22])), "r"(__float_as_uint(v[23])),
        "r"(__float_as_uint(v[24])), "r"(__float_as_uint(v[25])), "r"(__float_as_uint(v[26])), "r"(__float_as_uint(v[27])),
        "r"(__float_as_uint(v[28])), "r"(__float_as_uint(v[29])), "r"(__float_as_uint(v[30])), "r"(__float_as_uint(v[31]))
        : "memory");
}
// shared-memory matrix descriptor, 128-byte swizzle, explicit leading / stride byte offsets
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}
// byte offset of (row, 16-byte chunk c) in a tile of 128-byte rows with the 128-byte swizzle
__device__ __forceinline__ uint32_t sw128(int row, int c) { return (uint32_t)(row * 128 + ((c ^ (row & 7)) << 4)); }

// 2^x by the special-function unit (results below 2^-126, which the references keep 2^-94 below a row's largest, become 0)
__device__ __forceinline__ float exp2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// (all of the first 128 threads) true in all of them if `mine` is true in any
__device__ __forceinline__ bool softmax_vote(bool mine) {
    uint32_t any;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.u32 p, %1, 0;\n"
        "barrier.cta.red.or.pred q, 6, 128, p;\n"
        "selp.u32 %0, 1, 0, q;\n"
        "}\n"
        : "=r"(any)
        : "r"(mine ? 1u : 0u)
        : "memory");
    return any != 0;
}

template <int RP>
__device__ __noinline__ void attention_items_tc(int layer) {
    const FwdParams &p = params_copy();
    Shared *sh = shared_state();
    uint8_t *scratch = smem_base() + p.attn_smem_off;
#pragma unroll 1
    for (int item = blockIdx.x; item < p.attn_items; item += gridDim.x) {
    constexpr int NP = tc_p_tiles(RP), kQBytes = 2 * RP * 256, kPanel = 2 * RP * 128;  // a tile: two panels of 2 RP rows x 128 B
    const uint32_t tmem_base = sh->tmem_base;
    static_assert(AB_COUNT == kAttnBars, "barriers in the shared block");
    uint64_t *abar = shared_block().abar;
    uint32_t *acnt = shared_block().acnt;
    constexpr int Dh = 128;
    const int split = item % p.n_split, bh = item / p.n_split, b = bh / p.H, h = bh % p.H;
    const int d = p.d;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint8_t *ring = scratch, *qt = scratch + kTcStages * kTcKvStage, *pt = qt + kQBytes;
    float *wmax = reinterpret_cast<float *>(pt + NP * kQBytes);  // [4][RP] of the four softmax warps
    float *wsum = wmax + 4 * RP, *m_ref = wsum + 4 * RP, *fsh = m_ref + RP;  // [4][RP], the rows' references, a raise's factors
    uint64_t *kv_full = abar + AB_KV_FULL, *kv_free = abar + AB_KV_FREE;  // [kTcStages] each
    uint64_t *s_full = abar + AB_S_FULL;  // [2]: the scores are double-buffered in tensor memory
    uint64_t *p_ready = abar + AB_P_READY, *o_done = abar + AB_O_DONE, *fixed = abar + AB_FIXED, *landed = abar + AB_LANDED;

    const int n_rows = staged_len()[64 + b];
    const int len = staged_len()[b];
    const int r0 = b * p.M, rows_here = p.M;
    const int chunk = split_chunk(p, len + n_rows, kTcChunk);
    const int p_begin = split * chunk;
    const int p_end = min(p_begin + chunk, len + n_rows);
    const int n_chunks = p_begin < p_end ? (p_end - p_begin + kTcChunk - 1) / kTcChunk : 0;
    const float sc = p.attn_scale * 1.4426950408889634f;  // scores in log2 units
    const uint32_t tS = tmem_base, tO = tmem_base + 4 * RP;  // scores of chunk c at tS + 2 RP (c & 1)
    __nv_bfloat16 *kc = (__nv_bfloat16 *)(p.cache + (size_t)layer * p.layer_bytes) + ((size_t)(b * 2) * p.H + h) * p.S * Dh;
    __nv_bfloat16 *vc = kc + (size_t)p.H * p.S * Dh;
    const int krow0 = layer * p.kv_rows_per_layer + ((b * 2) * p.H + h) * p.S, vrow0 = krow0 + p.H * p.S;

    // a wait that keeps the control flow of every role intact: once anything has timed out, waits fall through
    auto wait = [&](uint64_t *bar, uint32_t parity) {
        if (sh->abort) return;
        if (!mbar_spin_or_abort(bar, parity, sh)) {
            set_status(p.status, kTimeoutCode);
            sh->abort = 1;
        }
    };

    // acnt: phases completed before this item (advanced by thread 0 at the end of the previous item, behind a barrier)
    // P V of chunk c completes phase c >> 1 of o_done[c & 1]
    auto o_par = [&](int c) { return (acnt[AB_O_DONE + (c & 1)] + (uint32_t)(c >> 1)) & 1u; };
    auto s_par = [&](int c) { return (acnt[AB_S_FULL + (c & 1)] + (uint32_t)(c >> 1)) & 1u; };
    auto p_par = [&](int c) { return (acnt[AB_P_READY + (c & 1)] + (uint32_t)(c >> 1)) & 1u; };
    auto full_par = [&](int j) { return (acnt[AB_KV_FULL + j % kTcStages] + (uint32_t)(j / kTcStages)) & 1u; };          // stage j has landed
    auto free_par = [&](int j) { return ((acnt[AB_KV_FREE + j % kTcStages] + (uint32_t)(j / kTcStages)) & 1u) ^ 1u; };   // its slot was released
    int n_fix_total = 0;
    for (int c = 0; c < n_chunks; ++c) n_fix_total += (p_begin + (c + 1) * kTcChunk > len) ? 1 : 0;

    // The copies of the first chunks do not depend on the set-up below: start them now.
    auto issue_kv = [&](int j) {
        const int slot = j % kTcStages, c = j >> 1;
        const int row = ((j & 1) ? vrow0 : krow0) + p_begin + c * kTcChunk;
        uint8_t *dst = ring + slot * kTcKvStage;
        mbar_expect_tx(&kv_full[slot], kTcKvStage);
        tma_load_2d(dst, p.tm_kv_ptr, 0, row, &kv_full[slot]);
        tma_load_2d(dst + kTcKvStage / 2, p.tm_kv_ptr, 64, row, &kv_full[slot]);
    };
    const int n_early = min(kTcStages, 2 * n_chunks);
    if (warp == 5 && lane == 0 && !sh->abort) {
        // Shared AND global memory: the previous user of these slots wrote them through the generic proxy, and so did the items of an
        // earlier step of this launch with the cache rows that the copies read (they reach this thread through the grid
        // barriers, which fence shared memory alone).
        fence_async_proxy();
        for (int j = 0; j < n_early; ++j) issue_kv(j);
    }
    // ---- set-up: Q tile (rotary applied, in log2 units; RP hi rows, RP lo rows) ----
#pragma unroll
    for (int it = 0; it < RP / 16; ++it) {
        const int m = 16 * it + (tid >> 4), v8 = tid & 15;
        float q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) q[u] = 0.f;
        if (m < n_rows) rope_vec8(p, p.qkv + (size_t)(r0 + m) * 3 * d + h * Dh, r0 + m, v8 * 8, q);
        __nv_bfloat16 hq[8], lq[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            q[u] *= sc;
            hq[u] = __float2bfloat16_rn(q[u]);
            lq[u] = __float2bfloat16_rn(q[u] - __bfloat162float(hq[u]));
        }
        uint8_t *panel = qt + (v8 >> 3) * kPanel;
        *reinterpret_cast<uint4 *>(panel + sw128(m, v8 & 7)) = *reinterpret_cast<uint4 *>(hq);
        *reinterpret_cast<uint4 *>(panel + sw128(RP + m, v8 & 7)) = *reinterpret_cast<uint4 *>(lq);
    }
    // (P rows that no softmax thread writes meet output columns that nobody reads)
    fence_async_shared();
    named_bar(3, kAttnThreadsP);

    if (warp == 5) {
        // ---------------- K / V chunk copies: stage j = 2 c (K), 2 c + 1 (V), slot j % kTcStages ----------------
        if (lane == 0) {
            int issued = n_early;
            for (int j = n_early; j < 2 * n_chunks && !sh->abort; ++j) {
                wait(&kv_free[j % kTcStages], free_par(j));
                if (sh->abort) break;
                issue_kv(j);
                ++issued;
            }
            if (sh->abort)  // error path only: copies still in flight
                for (int j = max(0, issued - kTcStages); j < issued; ++j) mbar_wait(&kv_full[j % kTcStages], full_par(j));
        }
        __syncwarp();
    } else if (warp == 4) {
        // ---------------- MMA issue ----------------
        if (lane == 0) {
            const uint32_t idS = umma_idesc_bf16(128, 2 * RP), idO = umma_idesc_bf16(128, 2 * RP) | (1u << 15);  // A of PV: MN-major
            const uint32_t qa = smem_u32(qt), pa = smem_u32(pt);
            int n_fix = 0;
            // S(c): scores of chunk c into buffer c & 1; issued one chunk ahead of P V so that it runs
            // while the softmax threads work on the previous chunk
            auto issue_s = [&](int c) {
                const int jk = 2 * c, jv = 2 * c + 1;
                const bool fix = p_begin + (c + 1) * kTcChunk > len;
                wait(&kv_full[jk % kTcStages], full_par(jk));
                if (fix) {  // both tiles are here: let the patching threads in, wait for them
                    wait(&kv_full[jv % kTcStages], full_par(jv));
                    if (!sh->abort) mbar_arrive(landed);
                    wait(fixed, (acnt[AB_FIXED] + n_fix) & 1u);
                    ++n_fix;
                }
                if (sh->abort) return;
                tc_fence_after();
                const uint32_t ka = smem_u32(ring + (jk % kTcStages) * kTcKvStage);
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)  // k = 16 head dims per step; panel ks / 4
                    tc_mma_bf16(tS + 2 * RP * (c & 1), umma_desc(ka + (ks >> 2) * (kTcKvStage / 2) + (ks & 3) * 32, 16, 1024),
                                umma_desc(qa + (ks >> 2) * kPanel + (ks & 3) * 32, 16, 1024), idS, ks ? 1u : 0u);
                tc_commit(&s_full[c & 1]);
                tc_commit(&kv_free[jk % kTcStages]);
            };
            if (n_chunks > 0) issue_s(0);
            for (int c = 0; c < n_chunks && !sh->abort; ++c) {
                const int jv = 2 * c + 1;
                if (c + 1 < n_chunks) issue_s(c + 1);
                wait(&p_ready[c & 1], p_par(c));
                wait(&kv_full[jv % kTcStages], full_par(jv));
                if (sh->abort) break;
                tc_fence_after();
                const uint32_t va = smem_u32(ring + (jv % kTcStages) * kTcKvStage);
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)  // k = 16 positions per step: two 8-row groups of the V tile
                    tc_mma_bf16(tO, umma_desc(va + ks * 2048, kTcKvStage / 2, 1024),
                                umma_desc(pa + (c % NP) * kQBytes + (ks >> 2) * kPanel + (ks & 3) * 32, 16, 1024), idO, (c | ks) ? 1u : 0u);
                tc_commit(&o_done[c & 1]);
                tc_commit(&kv_free[jv % kTcStages]);
            }
        }
        __syncwarp();
    } else if (warp >= 6) {
        // ---------------- rows of this pass, chunk by chunk ----------------
        const int ft = tid - 192;  // 0..63
        int n_fixed = 0;
        for (int c = 0; c < n_chunks; ++c) {
            const int base = p_begin + c * kTcChunk;
            if (base + kTcChunk <= len) continue;
            const int jk = 2 * c, jv = 2 * c + 1;
            uint8_t *kt = ring + (jk % kTcStages) * kTcKvStage, *vt = ring + (jv % kTcStages) * kTcKvStage;
            const int first = max(0, len - base), last = min(kTcChunk, len + n_rows - base);  // tile rows [first, last)
            // 16 vectors a row; two of them per thread and step, computed before the copies are waited for
            bool here = false;
#pragma unroll 1
            for (int i0 = ft; i0 < (last - first) * 16; i0 += 128) {
                uint4 kq[2], vq[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int i = i0 + 64 * u, pr = first + (i >> 4), v8 = i & 15;
                    if (pr < last) {
                        const int pos = base + pr, r = r0 + (pos - len);
                        const float *krow = p.qkv + (size_t)r * 3 * d + d + h * Dh;
                        float kf[8];
                        rope_vec8(p, krow, r, v8 * 8, kf);
                        const float4 v0 = __ldcg(reinterpret_cast<const float4 *>(krow + d + v8 * 8));
                        const float4 v1 = __ldcg(reinterpret_cast<const float4 *>(krow + d + v8 * 8 + 4));
                        kq[u] = make_uint4(pack_bf16x2(kf[0], kf[1]), pack_bf16x2(kf[2], kf[3]), pack_bf16x2(kf[4], kf[5]), pack_bf16x2(kf[6], kf[7]));
                        vq[u] = make_uint4(pack_bf16x2(v0.x, v0.y), pack_bf16x2(v0.z, v0.w), pack_bf16x2(v1.x, v1.y), pack_bf16x2(v1.z, v1.w));
                    }
                }
                if (!here) {
                    wait(landed, (acnt[AB_LANDED] + (uint32_t)n_fixed) & 1u);
                    here = true;
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int i = i0 + 64 * u, pr = first + (i >> 4), v8 = i & 15;
                    if (pr < last) {
                        const uint32_t off = (uint32_t)(v8 >> 3) * (kTcKvStage / 2) + sw128(pr, v8 & 7);
                        *reinterpret_cast<uint4 *>(kt + off) = kq[u];
                        *reinterpret_cast<uint4 *>(vt + off) = vq[u];
                        const size_t go = (size_t)(base + pr) * Dh + v8 * 8;  // append: exactly one split owns this position
                        *reinterpret_cast<uint4 *>(kc + go) = kq[u];
                        *reinterpret_cast<uint4 *>(vc + go) = vq[u];
                    }
                }
            }
            if (!here) wait(landed, (acnt[AB_LANDED] + (uint32_t)n_fixed) & 1u);
            ++n_fixed;
            fence_async_shared();
            mbar_arrive(fixed);
        }
    } else {
        // ---------------- softmax: thread = position tid of the chunk ----------------
        const uint32_t lane_sel = (uint32_t)(warp * 32) << 16;
        float l[RP];
#pragma unroll
        for (int r = 0; r < RP; ++r) l[r] = 0.f;
        if (tid < RP) m_ref[tid] = -INFINITY;
        named_bar(6, 128);
        for (int c = 0; c < n_chunks; ++c) {
            const int pos = p_begin + c * kTcChunk + tid;
            // rows from `first` on see this position (none beyond the split)
            const int first = pos < p_end ? pos - len : RP;
            const uint32_t tSc = tS + 2 * RP * (c & 1) + lane_sel;
            wait(&s_full[c & 1], s_par(c));
            tc_fence_after();
            // all rows' scores in one tensor-memory round trip (they take 0.3 - 0.5 us each), kept in registers
            float v[2 * RP];
            if constexpr (RP == 16) tc_ld_32(tSc, v);
            else tc_ld_64(tSc, v);
            bool over = false;
#pragma unroll
            for (int r = 0; r < RP; ++r) {
                v[r] = r >= first ? v[r] + v[RP + r] : -INFINITY;
                if (r % 4 == 0 && r >= rows_here) break;  // (rows in fours: the queries beyond rows_here are zeros)
                over = over || (r < rows_here && v[r] > m_ref[r] + kTcMaxSlack);
            }
            if (softmax_vote(over)) {  // rare, and the first chunk: raise the references that are passed
                // (rolled, and from tensor memory again: straight-line code that runs once per item costs its instruction fetch)
#pragma unroll 1
                for (int blk = 0; 8 * blk < rows_here; ++blk) {
                    float hi[8], lo[8];
                    tc_ld_2x8(tSc + 8 * blk, tSc + RP + 8 * blk, hi, lo);
                    float mine = -INFINITY;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float mx = warp_max_redux(8 * blk + i >= first ? fmaxf(hi[i] + lo[i], -INFINITY) : -INFINITY);  // (no NaN)
                        mine = lane == i ? mx : mine;
                    }
                    if (lane < 8) wmax[warp * RP + 8 * blk + lane] = mine;
                }
                named_bar(6, 128);
                if (tid < rows_here) {
                    const float mx = fmaxf(fmaxf(wmax[tid], wmax[RP + tid]), fmaxf(wmax[2 * RP + tid], wmax[3 * RP + tid]));
                    const float old = m_ref[tid];
                    const bool up = mx > old + kTcMaxSlack;
                    fsh[tid] = up ? exp2f(old - mx) : 1.f;  // 0 where nothing had been seen
                    if (up) m_ref[tid] = mx;
                }
                named_bar(6, 128);
#pragma unroll
                for (int r = 0; r < RP; ++r)
                    if (r < rows_here) l[r] *= fsh[r];
                if (c > 0) {  // thread = head dim tid: scale the accumulated O^T, once P V of the previous chunk has written it
                    wait(&o_done[(c - 1) & 1], o_par(c - 1));
                    tc_fence_after();
#pragma unroll 1
                    for (int blk = 0; blk < 2 * RP / 32; ++blk) {
                        float o[32];
                        tc_ld_32(tO + lane_sel + 32 * blk, o);
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] *= i % RP < rows_here ? fsh[i % RP] : 1.f;
                        tc_st_32(tO + lane_sel + 32 * blk, o);
                    }
                }
            }
            if (c >= NP) wait(&o_done[(c - NP) & 1], o_par(c - NP));  // this chunk's P tile was last read by P V of chunk c - NP
            // (opaque, or the compiler keeps the tile's 2 RP store addresses in registers - and on the stack - across the chunks)
            uint32_t panel = smem_u32(pt) + (uint32_t)((c % NP) * kQBytes + (tid >> 6) * kPanel + (tid & 7) * 2);
            uint32_t cc = (uint32_t)((tid & 63) >> 3);
            asm volatile("" : "+r"(panel), "+r"(cc));
            // four rows' values before their stores: the stores keep the loads behind them from moving up
#pragma unroll
            for (int r4 = 0; r4 < RP; r4 += 4) {
                if (r4 >= rows_here) break;  // (rows beyond rows_here: columns nobody reads)
                const float4 m4 = *reinterpret_cast<const float4 *>(m_ref + r4);
                const float m[4] = {m4.x, m4.y, m4.z, m4.w};
                __nv_bfloat16 hv[4], lv[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    // (a row that has seen nothing yet: reference -inf, every score -inf; a NaN score reaches the row's sum)
                    const float pv = v[r4 + i] != -INFINITY ? exp2_approx(v[r4 + i] - m[i]) : 0.f;
                    l[r4 + i] += pv;
                    hv[i] = __float2bfloat16_rn(pv);
                    lv[i] = __float2bfloat16_rn(pv - __bfloat162float(hv[i]));
                }
                // P as bf16 hi + lo into the P tile: row r (hi) / RP + r (lo), column = this position
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = r4 + i;
                    const uint32_t at = panel + r * 128 + ((cc ^ (r & 7)) << 4);
                    asm volatile("st.shared.b16 [%0], %1;" ::"r"(at), "h"(__bfloat16_as_ushort(hv[i])) : "memory");
                    asm volatile("st.shared.b16 [%0], %1;" ::"r"(at + RP * 128), "h"(__bfloat16_as_ushort(lv[i])) : "memory");
                }
            }
            fence_async_shared();  // (the general form, per chunk and thread: 17 rows x 16384 positions 100 -> 87 us a layer)
            tc_fence_before();
            mbar_arrive(&p_ready[c & 1]);
        }
        // ---- the sums over positions, then thread = head dim tid: output or partial ----
        // (lane r of a warp ends up with row r's sum: RP - 1 exchanges instead of 5 RP)
#pragma unroll
        for (int hf = RP / 2; hf > 0; hf >>= 1) {
            const bool up = lane & hf;
#pragma unroll
            for (int j = 0; j < hf; ++j) {
                const float send = up ? l[j] : l[j + hf], keep = up ? l[j + hf] : l[j];
                l[j] = keep + __shfl_xor_sync(0xffffffffu, send, hf);
            }
        }
        if (RP == 16) l[0] += __shfl_xor_sync(0xffffffffu, l[0], 16);
        if (lane < RP) wsum[warp * RP + lane] = l[0];
        if (n_chunks > 1) wait(&o_done[(n_chunks - 2) & 1], o_par(n_chunks - 2));
        if (n_chunks > 0) {
            wait(&o_done[(n_chunks - 1) & 1], o_par(n_chunks - 1));
            tc_fence_after();
        }
        named_bar(6, 128);
        const bool direct = p.n_split == 1;
#pragma unroll 1
        for (int blk = 0; blk < RP / 8; ++blk) {
            if (8 * blk < rows_here) {
                float oh[8], ol[8];
                if (n_chunks > 0) tc_ld_2x8(tO + lane_sel + 8 * blk, tO + lane_sel + RP + 8 * blk, oh, ol);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = 8 * blk + i;
                    if (r < rows_here) {
                        const float L = (wsum[r] + wsum[RP + r]) + (wsum[2 * RP + r] + wsum[3 * RP + r]);
                        const bool live = r < n_rows && L > 0.f && n_chunks > 0;
                        const float acc = live ? oh[i] + ol[i] : 0.f;
                        if (direct) {
                            store_hilo(p.op[OP_AO], p.rk, r0 + r, h * Dh + tid, live ? acc / L : 0.f);
                        } else {
                            const size_t slot = ((size_t)(r0 + r) * p.H + h) * p.n_split + split;
                            if (tid == 0) {
                                p.part_m[slot] = live ? m_ref[r] : -INFINITY;
                                p.part_l[slot] = live ? L : 0.f;
                            }
                            p.part_o[slot * Dh + tid] = acc;
                        }
                    }
                }
            }
        }
        tc_fence_before();
    }
    if (p.n_split != 1) {
        // ticket: the item that finishes last for this (sequence, head) merges all partials
        // (one release and one acquire for the CTA, as in the grid barrier)
        named_bar(3, kAttnThreadsP);
        if (tid == 0) sh->flag = (atomic_add_acq_rel(p.tickets + bh, 1u) == (unsigned)(p.n_split - 1));
        named_bar(3, kAttnThreadsP);
        if (sh->flag) {
            merge_splits(p, r0, h, Dh);
            if (tid == 0) p.tickets[bh] = 0;  // ready for the next layer (a grid barrier lies between)
        }
    }
    named_bar(3, kAttnThreadsP);  // everyone has read the counts
    if (tid == 0) {
        for (int i = 0; i < kTcStages; ++i) {
            const uint32_t uses = (uint32_t)((2 * n_chunks + kTcStages - 1 - i) / kTcStages);  // stages j < 2 n_chunks with j % kTcStages == i
            acnt[AB_KV_FULL + i] += uses;
            acnt[AB_KV_FREE + i] += uses;
        }
        acnt[AB_S_FULL] += (uint32_t)((n_chunks + 1) / 2);
        acnt[AB_S_FULL + 1] += (uint32_t)(n_chunks / 2);
        acnt[AB_P_READY] += (uint32_t)((n_chunks + 1) / 2);
        acnt[AB_P_READY + 1] += (uint32_t)(n_chunks / 2);
        acnt[AB_O_DONE] += (uint32_t)((n_chunks + 1) / 2);
        acnt[AB_O_DONE + 1] += (uint32_t)(n_chunks / 2);
        acnt[AB_FIXED] += n_fix_total;
        acnt[AB_LANDED] += n_fix_total;
    }
    named_bar(3, kAttnThreadsP);  // scratch, tensor memory and the counts are ready for the next item
    }
}

// WIDE: passes of more than 16 rows per sequence on the tensor core, a kernel of its own.  (A function that might be called
// shapes the register allocation of the whole kernel body: with the 32-row item beside the other forms the body reloads 3 KB of
// spilled values around its phases, 176 bytes without it.  One kernel per form leaves the body none, but its live values then
// take the registers that the items want, which save and restore them instead: the 16-row items 15.1 -> 17.8 us, the packed ones
// of eight 2100-position sequences 51.3 -> 53.8.)
enum { ATT_MMA = 0, ATT_TC16, ATT_PACKED, ATT_TC32 };
template <bool WIDE>
__device__ __forceinline__ void attention_phase(int layer) {
    const FwdParams &p = params_copy();
    if constexpr (WIDE) attention_items_tc<32>(layer);
    else if (p.attn_form == ATT_TC16) attention_items_tc<16>(layer);
    else if (p.attn_form == ATT_PACKED && p.Dh == 128) attention_items_mma8<128>(layer);
    else if (p.attn_form == ATT_PACKED) attention_items_mma8<64>(layer);
    else attention_items(layer);
}

// Run this CTA's units of GEMM gi (all 256 work threads call it; NT = padded rows / 8).  The units are
// contiguous in (tile, k-chunk) order, so they form one segment per tile touched; each segment is
// accumulated in tensor memory and reduced into the output once.  A function of its own, with the
// little state that survives from GEMM to GEMM kept in shared memory, so that the kernel's phase loop
// holds nothing across its calls: with 227 KB of shared memory there is next to no L1 left, and a
// value spilled to the stack costs an L2 round trip at every phase.
template <int NT>
__device__ __noinline__ void run_gemm(int gi) {
    const FwdParams &p = params_copy();
    uint8_t *smem = smem_base();
    constexpr int kRp = NT * 8;
    constexpr int kXBytes = 2 * kRp * kTileK * 2;
    constexpr int kStageBytes = kXBytes + kWTileBytesP;
    // M of the MMA: the operand tile's 2 kRp rows; the rows the MMA reads beyond them are the weight
    // tile's bytes (finite or not, they only reach accumulator lanes that nobody loads)
    constexpr int kM = 2 * kRp <= 64 ? 64 : 128;
    SharedBlock &mp = shared_block();
    const int S = p.stages, S1 = p.stages_lo;
    uint8_t *ring = smem;
    uint64_t *fullW = mp.fullW, *fullX = mp.fullX, *empty = mp.empty, *accFull = mp.accFull, *accEmpty = mp.accEmpty;
    Shared *sh = &mp.state;
    float *epi_tile = mp.epi_tile;
    volatile int *epi_ok = mp.epi_ok;
    const uint32_t tmem_base = sh->tmem_base;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool walks_ring = lane == 0 && (warp == kMmaWarp || warp == kXWarp);
    RingPos rp;
    if (walks_ring) rp = mp.role_rp[warp == kMmaWarp ? 0 : 1];
    int seg = mp.role_seg[warp];
    auto save_state = [&]() {
        if (walks_ring) mp.role_rp[warp == kMmaWarp ? 0 : 1] = rp;
        __syncwarp();
        if (lane == 0) mp.role_seg[warp] = seg;
        __syncwarp();
    };

            const GemmDesc g = gemm_desc(p, gi, staged_ltab());
            int c0, c1;
            unit_range(p, g, c0, c1);
            if (c0 >= c1) return;  // (no state to save: nothing moved)
            const int tile0 = c0 / g.kchunks, tile1 = (c1 - 1) / g.kchunks;
            if (warp == kMmaWarp) {
                if (lane == 0 && !sh->abort) {
                    const uint32_t idesc = umma_idesc_bf16(kM, kTileNP);
                    int sg = seg, kc = c0 % g.kchunks;
                    bool first = true;
                    for (int c = c0; c < c1; ++c) {
                        uint32_t ph;
                        const int s = ring_next(rp, ring_lo_only(g, c - c0, S1), S, S1, ph), b = sg & 1;
                        bool ok = true;
                        if (first && sg >= 2) ok = mbar_wait_or_abort(&accEmpty[b], ((sg >> 1) - 1) & 1, sh);
                        ok = ok && mbar_wait_or_abort(&fullW[s], ph, sh) && mbar_wait_or_abort(&fullX[s], ph, sh);
                        if (!ok) {
                            set_status(p.status, kTimeoutCode);
                            sh->abort = 1;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t st = smem_u32(ring + (size_t)s * kStageBytes);
                        const uint64_t adesc = umma_desc_sw128(st), bdesc = umma_desc_sw128(st + kXBytes);
                        const uint32_t d_tmem = tmem_base + (uint32_t)(b * kAccStride);
#pragma unroll
                        for (int ks = 0; ks < kTileK / 16; ++ks)  // 32 bytes further along k inside the swizzle atom
                            tc_mma_bf16(d_tmem, adesc + 2 * ks, bdesc + 2 * ks, idesc, (first && ks == 0) ? 0u : 1u);
                        tc_commit(&empty[s]);
                        first = false;
                        ++kc;
                        if (kc == g.kchunks || c + 1 == c1) {
                            tc_commit(&accFull[b]);
                            ++sg;
                            first = true;
                            if (kc == g.kchunks) kc = 0;
                        }
                    }
                }
                __syncwarp();
            } else if (warp == kXWarp) {
                // operand tiles of this GEMM, once the barrier behind the phase that makes them is complete
                bool ready = true;
                if (lane == 0 && !sh->abort && sh->passed < g.need) {
                    ready = grid_poll(p, sh, g.need);
                    if (ready) {
                        grid_stamp(p, g.need);
                    } else {
                        set_status(p.status, kTimeoutCode);
                        sh->abort = 1;
                    }
                }
                if (lane == 0 && !sh->abort && g.wait_attn) {
                    // the attention output is complete once every attention CTA of this layer has signalled
                    const unsigned *cnt = attn_done(p);
                    if (ld_acquire(cnt) < g.wait_attn) {
                        const long long t0 = clock64();
                        while (ld_acquire(cnt) < g.wait_attn) {
                            if (sh->abort || clock64() - t0 > sh->wait_limit) { ready = false; break; }
                        }
                    }
                    if (!ready) {
                        set_status(p.status, kTimeoutCode);
                        sh->abort = 1;
                    }
                }
                if (lane == 0 && ready && !sh->abort) {
                    fence_async_global();  // that phase's generic-proxy writes -> visible to the bulk copies
                    int kx = c0 % g.kchunks;
                    for (int c = c0; c < c1; ++c) {
                        uint32_t ph;
                        const int s = ring_next(rp, ring_lo_only(g, c - c0, S1), S, S1, ph);
                        if (!mbar_wait_or_abort(&empty[s], ph ^ 1u, sh)) {
                            rp.par ^= 1u << s;  // nothing was issued into s
                            set_status(p.status, kTimeoutCode);
                            sh->abort = 1;
                            break;
                        }
                        mbar_expect_tx(&fullX[s], kXBytes);
                        bulk_load_1d(ring + (size_t)s * kStageBytes, g.xop + (size_t)kx * (2 * kRp * kTileK), kXBytes,
                                     &fullX[s]);
                        if (++kx == g.kchunks) kx = 0;
                    }
                }
                __syncwarp();
            } else if (warp < kEpiWarps) {
                int sg = seg;
                const bool vec_ok = (((uintptr_t)g.out & 15) == 0) && ((g.ldo & 3) == 0) &&
                                    (!g.bias || ((uintptr_t)g.bias & 15) == 0);
                for (int t = tile0; t <= tile1; ++t, ++sg) {
                    const int b = sg & 1;
                    // the four warps take the same decision: the named barriers below need all of them
                    const bool mine = mbar_wait_or_abort(&accFull[b], (sg >> 1) & 1, sh);
                    if (lane == 0) epi_ok[warp] = mine ? 1 : 0;
                    named_bar(5, kEpiWarps * 32);
                    if (!(epi_ok[0] && epi_ok[1] && epi_ok[2] && epi_ok[3])) {
                        set_status(p.status, kTimeoutCode);
                        sh->abort = 1;
                        break;
                    }
                    tc_fence_after();
                    const bool has_k0 = (t > tile0) || (c0 % g.kchunks == 0);
                    const float *bias = (has_k0 && g.bias) ? g.bias : nullptr;
                    const int g8 = lane >> 2, t4 = lane & 3;
                    // a thread's four columns are the same in every row: their bias is taken once per tile
                    const int c4 = (threadIdx.x & 63) * 4, n = t * kTileNP + c4;
                    float *col = g.out + n;
                    float4 bb = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (bias && n + 3 < g.N && vec_ok) {
                        bb = __ldg(reinterpret_cast<const float4 *>(bias + n));
                    } else if (bias) {
                        if (n < g.N) bb.x = __ldg(bias + n);
                        if (n + 1 < g.N) bb.y = __ldg(bias + n + 1);
                        if (n + 2 < g.N) bb.z = __ldg(bias + n + 2);
                        if (n + 3 < g.N) bb.w = __ldg(bias + n + 3);
                    }
                    // Block q of 8 rows sits in accumulator lanes 32 q .. 32 q + 15 (M = 64) or 16 q .. 16 q + 15
                    // (M = 128); a warp reaches the 32 lanes of its own quadrant only.
#pragma unroll 1
                    for (int q = 0; q < NT; ++q) {
                        if (8 * q >= p.R) break;
                        const int wq = kM == 64 ? q : (q >> 1), half = kM == 64 ? 0 : (q & 1);
                        if (wq == warp) {
                            const uint32_t ta = tmem_base + ((uint32_t)(warp * 32 + half * 16) << 16) + (uint32_t)(b * kAccStride);
                            for (int cg = 0; cg < kTileNP / 64; ++cg) {  // 64 columns per tensor-memory round trip
                                if (t * kTileNP + cg * 64 >= g.N) break;
                                float v[32];
                                tc_ld_16x64(ta + (uint32_t)(cg * 64), v);
#pragma unroll
                                for (int k = 0; k < 8; ++k)
                                    *reinterpret_cast<float2 *>(epi_tile + g8 * kEpiPitch + cg * 64 + 8 * k + 2 * t4) =
                                        make_float2(v[4 * k] + v[4 * k + 2], v[4 * k + 1] + v[4 * k + 3]);
                            }
                        }
                        named_bar(5, kEpiWarps * 32);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int rr = (threadIdx.x >> 6) + 2 * k, row = 8 * q + rr;
                            if (row < p.R && n < g.N) {
                                float4 v = *reinterpret_cast<const float4 *>(epi_tile + rr * kEpiPitch + c4);
                                v.x += bb.x; v.y += bb.y; v.z += bb.z; v.w += bb.w;
                                float *dst = col + (size_t)row * g.ldo;
                                if (vec_ok && n + 3 < g.N) {
                                    red_add_v4(dst, v);
                                } else {
                                    atomicAdd(dst, v.x);
                                    if (n + 1 < g.N) atomicAdd(dst + 1, v.y);
                                    if (n + 2 < g.N) atomicAdd(dst + 2, v.z);
                                    if (n + 3 < g.N) atomicAdd(dst + 3, v.w);
                                }
                            }
                        }
                        named_bar(5, kEpiWarps * 32);  // the tile is free for the next block
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&accEmpty[b]);
                }
            }
            seg += tile1 - tile0 + 1;
            save_state();
}

// ---- the vocabulary-wide tail of a draft step, inside the kernel ---------------------------------
// After the LM head of a draft step every sequence's last fed row of logits is turned into q = softmax(row / T),
// exported, and sampled by inverse CDF with the step's uniform - the work of draft_tail_kernel, spread over the
// whole grid so that the kernel can go on to the next step without returning to the host.  CTA c owns the slice
// [c * per, (c + 1) * per) of the vocabulary; inside a CTA warp w works on sequences w, w + 8, ... with warp
// shuffles only.  Three phases, a grid barrier behind each:
//   1. per (sequence, CTA): max, argmax and sum of exp relative to that max over the slice;
//   2. every CTA combines the partials of all CTAs into (max, argmax, Z), writes its slice of q and the slice's
//      mass (fp64, index order: lane l holds a contiguous piece of the slice);
//   3. every CTA takes the prefix of the slice masses in CTA order; the lanes whose piece can hold the first
//      index with c_j > u S walk it and post the index (atomic minimum); the largest index with q > 0 is
//      posted too (the fallback when rounding leaves no index past u S);
// then CTA 0 writes the tokens and commits the rows fed in this step.
__device__ __forceinline__ int tail_per(const FwdParams &p) { return (((p.V + (int)gridDim.x - 1) / (int)gridDim.x) + 3) & ~3; }
__device__ __forceinline__ const float *tail_row(const FwdParams &p, int b) {
    int row = (b < 64 ? staged_len()[64 + b] : __ldcg(p.ri.n_eff + b)) - 1;  // (staged behind the step's first barrier)
    if (row < 0) row = 0;
    return p.logits + ((size_t)b * p.M + row) * p.V;
}

// (All loops below fetch eight elements before they use the first: a load from L2 costs about a microsecond
// under the weight stream, and a slice is only a few hundred elements.)
__device__ __noinline__ void tail_partial() {
    const FwdParams &p = params_copy();
    Shared *sh = shared_state();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = (int)gridDim.x;
    const int per = tail_per(p), lo = min(p.V, (int)blockIdx.x * per), hi = min(p.V, lo + per);
    for (int b = warp; b < p.B; b += kConsumerWarps) {
        const float *lg = tail_row(p, b);
        // running (max, argmax, sum of exp relative to the max) per lane, then over the warp
        float mx = -INFINITY, sum = 0.f;
        int am = 0x7fffffff;
        for (int jb = lo + lane; jb < hi; jb += 256) {
            float l[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) l[u] = jb + 32 * u < hi ? __ldcg(lg + jb + 32 * u) : -INFINITY;
            float m8 = mx;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (l[u] > m8) { m8 = l[u]; am = jb + 32 * u; }  // ascending per lane: the first maximum
            if (p.inv_t != 0.f && m8 > -INFINITY) {
                sum *= expf((mx - m8) * p.inv_t);  // 0 while nothing has been summed
#pragma unroll
                for (int u = 0; u < 8; ++u) sum += expf((l[u] - m8) * p.inv_t);  // exp(-inf) = 0
            }
            mx = m8;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, mx, o), os = __shfl_xor_sync(0xffffffffu, sum, o);
            const int oi = __shfl_xor_sync(0xffffffffu, am, o);
            const float m2 = fmaxf(mx, ov);
            if (m2 > -INFINITY) sum = sum * expf((mx - m2) * p.inv_t) + os * expf((ov - m2) * p.inv_t);
            if (ov > mx || (ov == mx && oi < am)) am = oi;
            mx = m2;
        }
        if (lane == 0) {
            p.tp_m[(size_t)b * G + blockIdx.x] = mx;
            p.tp_s[(size_t)b * G + blockIdx.x] = sum;
            p.tp_a[(size_t)b * G + blockIdx.x] = am;
        }
    }
}

// (max, argmax - lowest index among the maxima -, Z) of a sequence's row from the CTAs' partials; the same in every lane
__device__ __forceinline__ void tail_stats(const FwdParams &p, int b, float &mx, int &am, float &z) {
    const int lane = threadIdx.x & 31, G = (int)gridDim.x;
    float pm[8], ps[8];
    int pa[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {  // (grids of up to 256 CTAs)
        const int c = lane + 32 * k;
        pm[k] = c < G ? __ldcg(p.tp_m + (size_t)b * G + c) : -INFINITY;
        ps[k] = c < G ? __ldcg(p.tp_s + (size_t)b * G + c) : 0.f;
        pa[k] = c < G ? __ldcg(p.tp_a + (size_t)b * G + c) : 0x7fffffff;
    }
    mx = -INFINITY;
    am = 0x7fffffff;
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (pm[k] > mx || (pm[k] == mx && pa[k] < am)) { mx = pm[k]; am = pa[k]; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, mx, o);
        const int oi = __shfl_xor_sync(0xffffffffu, am, o);
        if (ov > mx || (ov == mx && oi < am)) { mx = ov; am = oi; }
    }
    double zz = 0.0;
    if (p.inv_t != 0.f) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (pm[k] > -INFINITY) zz += (double)ps[k] * (double)expf((pm[k] - mx) * p.inv_t);
    }
    zz = warp_sum(zz);
    z = (float)zz;
}
__device__ __forceinline__ float tail_prob(float logit, float mx, int am, float z, float inv_t, int j) {
    if (inv_t == 0.f) return j == am ? 1.f : 0.f;
    return expf((logit - mx) * inv_t) / z;
}

__device__ __noinline__ void tail_q() {
    const FwdParams &p = params_copy();
    Shared *sh = shared_state();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = (int)gridDim.x;
    const int per = tail_per(p), lo = min(p.V, (int)blockIdx.x * per), hi = min(p.V, lo + per);
    const int seg = (hi - lo + 31) / 32, j0 = min(hi, lo + lane * seg), j1 = min(hi, j0 + seg);
    for (int b = warp; b < p.B; b += kConsumerWarps) {
        const float *lg = tail_row(p, b);
        float l[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) l[u] = j0 + u < j1 ? __ldcg(lg + j0 + u) : 0.f;  // (under the partials' latency)
        float mx, z;
        int am;
        tail_stats(p, b, mx, am, z);
        float *q = p.q_out + (size_t)b * p.q_stride + (size_t)p.cur_step * p.V;
        double local = 0.0;
        for (int jb = j0; jb < j1; jb += 8) {
            if (jb > j0) {
#pragma unroll
                for (int u = 0; u < 8; ++u) l[u] = jb + u < j1 ? __ldcg(lg + jb + u) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (jb + u < j1) {
                    const float w = tail_prob(l[u], mx, am, z, p.inv_t, jb + u);
                    q[jb + u] = w;
                    local += (double)w;
                }
        }
        local = warp_sum(local);  // (a sum of at most 32 pieces: the order does not matter at fp64 for a decision that
        if (lane == 0) p.tp_mass[(size_t)b * G + blockIdx.x] = local;  //  is excused within 1e-6 S of a step anyway)
    }
}

__device__ __noinline__ void tail_draw() {
    const FwdParams &p = params_copy();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = (int)gridDim.x;
    const int per = tail_per(p), lo = min(p.V, (int)blockIdx.x * per), hi = min(p.V, lo + per);
    const int seg = (hi - lo + 31) / 32, j0 = min(hi, lo + lane * seg), j1 = min(hi, j0 + seg);
    for (int b = warp; b < p.B; b += kConsumerWarps) {
        // total and this CTA's offset from the slice masses (lane l takes CTAs l, l + 32, ...; fp64)
        double off = 0.0, S = 0.0;
        {
            double t[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) t[k] = lane + 32 * k < G ? __ldcg(p.tp_mass + (size_t)b * G + lane + 32 * k) : 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                S += t[k];
                if (lane + 32 * k < (int)blockIdx.x) off += t[k];
            }
            S = warp_sum(S);
            off = warp_sum(off);
        }
        const float *q = p.q_out + (size_t)b * p.q_stride + (size_t)p.cur_step * p.V;
        double local = 0.0;
        int last_pos = -1;
        for (int jb = j0; jb < j1; jb += 8) {
            float w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) w[u] = jb + u < j1 ? __ldcg(q + jb + u) : 0.f;  // written by this very lane in the phase before
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                local += (double)w[u];
                if (w[u] > 0.f) last_pos = jb + u;
            }
        }
        double incl = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const double target = (double)__ldcg(p.u + (size_t)b * p.u_stride + p.cur_step) * S;
        double run = off + (incl - local);
        int hit = 0x7fffffff;
        if (S > 0.0 && (run + local > target || run > target)) {
            for (int j = j0; j < j1; ++j) {
                const float w = __ldcg(q + j);
                run += (double)w;
                if (w > 0.f && run > target) { hit = j; break; }  // a zero-weight index is never drawn
            }
        }
        // one atomic per warp, not per lane: thousands of atomics on one word would serialise in L2
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            hit = min(hit, __shfl_xor_sync(0xffffffffu, hit, o));
            last_pos = max(last_pos, __shfl_xor_sync(0xffffffffu, last_pos, o));
        }
        int32_t *slot = p.tail_hit + ((size_t)p.cur_step * p.B + b) * 2;
        if (lane == 0 && hit != 0x7fffffff) atomicMin(slot, hit);
        if (lane == 0 && last_pos >= 0) atomicMax(slot + 1, last_pos);
    }
}

// CTA 0: the tokens of this step, and the rows it fed become part of the cache
__device__ __noinline__ void tail_commit() {
    const FwdParams &p = params_copy();
    if (blockIdx.x != 0) return;
    for (int b = threadIdx.x; b < p.B; b += kWorkThreads) {
        const int32_t *slot = p.tail_hit + ((size_t)p.cur_step * p.B + b) * 2;
        const int hit = __ldcg(slot), last = __ldcg(slot + 1);
        int tok = hit != 0x7fffffff ? hit : last;
        if (tok < 0) tok = max(0, min(__ldcg(p.tp_a + (size_t)b * gridDim.x), p.V - 1));  // a row without any probability
        p.tok_out[(size_t)b * p.tok_out_stride + p.cur_step] = tok;
        p.len_rw[b] = __ldcg(p.len_rw + b) + __ldcg(p.ri.n_eff + b);
    }
}

// ---- the kernel -----------------------------------------------------------------------------
// The producer's walk and the work warps' phase program keep next to nothing alive across the calls they make: what is live
// there takes registers that the attention items and GEMMs want, and is spilled around every one of the 130-260 calls of a pass
// (about a microsecond each where the line has left the little L1 there is).  Both are part of the kernel body: as functions of
// their own they cost every pass 0.5 - 1.4 % (7B decode, eight sequences of 2100 positions, us a layer: 144.5 so, 143.6 inline).
template <int NT>
__device__ __forceinline__ constexpr int stage_x_bytes() { return 2 * NT * 8 * kTileK * 2; }

template <int NT>
__device__ __forceinline__ void producer_program() {
    const FwdParams &p = params_copy();
    constexpr int kXBytes = stage_x_bytes<NT>(), kStageBytes = kXBytes + kWTileBytesP;
    uint64_t *fullW = shared_block().fullW, *empty = shared_block().empty;
    Shared *sh = shared_state();
    uint8_t *ring = smem_base();
    const int S = p.stages, S1 = p.stages_lo, NG = n_gemms(p), lane = threadIdx.x & 31;
    // Weights never change, so this cursor runs as far ahead as the ring allows, across grid
    // barriers.  The loop is kept minimal (no divisions, no clock reads while it makes progress):
    // its rate bounds the weight stream.
    if (lane == 0) {
        RingPos rp;
        bool failed = false;
        int seen_arrival = 0;
        // a CTA that never runs an attention item (fewer items than CTAs) never uses the scratch: its
        // upper slots take weights at any time
        const bool scratch_used = (int)blockIdx.x < p.attn_items;
        for (int gws = 0; gws < NG * p.n_steps && !failed; ++gws) {
            const int gw = ((gws / NG) << kStepShift) | (gws % NG);
            const GemmDesc dw = gemm_desc(p, gw);
            int c0, c1;
            unit_range(p, dw, c0, c1);
            if (c0 >= c1) continue;
            int tw = c0 / dw.kchunks, kw = c0 % dw.kchunks;
            for (int c = c0; c < c1; ++c) {
                uint32_t ph;
                const int s = ring_next(rp, ring_lo_only(dw, c - c0, S1), S, S1, ph);
                if (s >= S1 && scratch_used && seen_arrival < dw.need_hi) {  // slot shared with the attention scratch
                    const long long t0 = clock64();
                    while ((seen_arrival = sh->arrived) < dw.need_hi) {
                        if (sh->abort || clock64() - t0 > sh->wait_limit) { failed = true; break; }
                        __nanosleep(100);  // (a tight poll takes issue slots and shared-memory cycles from the attention loop)
                    }
                    if (failed) { rp.par ^= 1u << s; break; }  // nothing was issued into s
                }
                if (!mbar_test_wait(&empty[s], ph ^ 1u)) {
                    const long long t0 = clock64();
                    while (!mbar_test_wait(&empty[s], ph ^ 1u)) {
                        if (sh->abort || clock64() - t0 > sh->wait_limit) { failed = true; break; }
                    }
                    if (failed) { rp.par ^= 1u << s; break; }  // nothing was issued into s
                }
                mbar_expect_tx(&fullW[s], kWTileBytesP);
                tma_load_2d(ring + (size_t)s * kStageBytes + kXBytes, dw.tmW, kw * kTileK, tw * kTileNP, &fullW[s]);
                if (++kw == dw.kchunks) { kw = 0; ++tw; }
            }
        }
        if (failed) {
            set_status(p.status, kTimeoutCode);
            sh->abort = 1;
        }
        // error path only: wait (bounded) for copies still in flight before the CTA may exit
        if (sh->abort)
            for (int s = 0; s < S; ++s)
                if ((rp.used >> s) & 1u) mbar_wait(&fullW[s], ((rp.par >> s) & 1u) ^ 1u);
    }
}
// The phase program (the same structure gemm_desc() encodes).  `go` is uniform over the work threads (taken inside the grid
// barrier), so every named barrier is reached by all of them or by none.
template <int NT, bool WIDE>
__device__ __forceinline__ void work_program() {
    const FwdParams &p = params_copy();
    if (p.trace && blockIdx.x == 0 && threadIdx.x == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        p.trace[0] = t;
    }
    if (p.tail && blockIdx.x == 0)  // the draws' meeting places: smallest hit index / largest index with weight
        for (int i = threadIdx.x; i < p.n_steps * p.B * 2; i += kWorkThreads) p.tail_hit[i] = (i & 1) ? -1 : 0x7fffffff;
    bool go = true;
    for (int step = 0; step < p.n_steps && go; ++step) {
        if (step > 0) {  // the rows of this step: one per sequence, the token the step before drew
            if (threadIdx.x == 0) params_copy().cur_step = step;
            named_bar(2, kWorkThreads);
        }
        // Set-up, embedding and the first norm of a row all run on the CTA that owns the row, so only
        // CTA-wide barriers separate them: one grid barrier in front of the first GEMM instead of two.
        setup_phase();
        named_bar(2, kWorkThreads);  // the row's position and validity are read back by the embedding
        embed_phase();
        named_bar(2, kWorkThreads);  // the embedding rows are read back by the norm
        norm_for_layer(0);
        go = grid_sync();
        if (go && threadIdx.x < 64) {  // lengths and rows of this pass (written by the set-up of every row), for the
            int *tab = shared_block().seq;  // attention items, which run behind further grid barriers
            const int b = threadIdx.x;
            tab[b] = b < p.B ? __ldcg(p.len + b) : 0;
            tab[64 + b] = b < p.B ? __ldcg(p.ri.n_eff + b) : 0;
        }
        for (int l = 0; l < p.n_layers && go; ++l) {
            asm volatile("" : "+r"(l));  // (no induction variables beside it: each would be one more value kept across the calls)
            run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * l + 0));                  // qkv
            const bool kv_only = !p.want_logits && l + 1 == p.n_layers;
            if (p.parallel && !kv_only) run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * l + 1));  // MLP in (same block input)
            if (!(go = grid_sync())) break;
            if (kv_only) {
                attention_phase<WIDE>(l);  // (its items append the rows)
                break;
            }
            if (overlap_mlp_out(p)) {
                act_phase();
                if ((int)blockIdx.x < attention_ctas(p)) {
                    grid_arrive();  // the activation is out; attention needs nothing from the others
                    attention_phase<WIDE>(l);
                    attn_signal();
                } else {
                    grid_arrive();
                    run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * l + 2));               // MLP out -> x, beside the attention items
                    run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * l + 3));               // out-proj -> x, once the attention CTAs have signalled
                }
                if (!(go = grid_sync())) break;
            } else {
                attention_phase<WIDE>(l);
                if (p.parallel) act_phase();
                grid_arrive();
                if (p.parallel) {
                    run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * l + 2));                   // out-proj -> x
                    run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * l + 3));                   // MLP out  -> x
                    if (!(go = grid_sync())) break;
                } else {
                    run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * l + 1));                   // out-proj -> x
                    if (!(go = grid_sync())) break;
                    norm_mid_layer(l);
                    grid_arrive();
                    run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * l + 2));                   // MLP in
                    if (!(go = grid_sync())) break;
                    act_phase();
                    grid_arrive();
                    run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * l + 3));                   // MLP out -> x
                    if (!(go = grid_sync())) break;
                }
            }
            norm_for_layer(l + 1);
            grid_arrive();
        }
        if (go && p.want_logits) run_gemm<NT>((params_copy().cur_step << kStepShift) | (4 * p.n_layers));
        if (go && p.tail) {  // q, the draw and the commit of this step (see tail_partial)
            if (!(go = grid_sync())) break;
            tail_partial();
            if (!(go = grid_sync())) break;
            tail_q();
            if (!(go = grid_sync())) break;
            tail_draw();
            if (!(go = grid_sync())) break;
            tail_commit();
            if (!(go = grid_sync())) break;
        }
    }
    if (go && p.tail && p.mailbox && blockIdx.x == 0 && (int)threadIdx.x < p.B)  // the host's length bound follows (see report_len)
        *reinterpret_cast<volatile unsigned long long *>(p.mailbox + threadIdx.x) =
            ((unsigned long long)p.mb_seq << 32) | (unsigned)__ldcg(p.len_rw + threadIdx.x);
    if (p.trace && blockIdx.x == 0 && threadIdx.x == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        p.trace[shared_state()->epoch + 1] = t;
        p.trace[shared_state()->epoch + 2] = 0;
    }
}
// NT = padded rows / 8
template <int NT, bool WIDE>
__global__ void __launch_bounds__(kPersistThreads, 1) forward_kernel(const __grid_constant__ FwdParams kp) {
    // A reference into the kernel-parameter bank would make every field a generic load at the head of each phase: the phase
    // functions read a copy in shared memory (tensor maps stay where the copy engine can read them: pointers into kp / global).
    SharedBlock &blk = shared_block();
    for (int i = threadIdx.x; i < (int)(sizeof(FwdParams) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t *>(blk.params)[i] = reinterpret_cast<const uint32_t *>(&kp)[i];
    __syncthreads();
    if (threadIdx.x == 0) params_copy().tm_kv_ptr = &kp.tm_kv;
    if (kp.n_layers <= kMaxStagedLayers) {  // the layers' gain / bias pointers and the final norm's
        for (int i = threadIdx.x; i < 8 * kp.n_layers + 2; i += blockDim.x) {
            const int l = i >> 3, k = i & 7;
            blk.ltab[i] = l < kp.n_layers ? (&layer_desc(kp.md, l)->ln1_g)[k] : (k == 0 ? kp.md->lnf_g : kp.md->lnf_b);
        }
    }

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {  // tensor memory for the accumulators; released by the same warp at the end
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&blk.tmem_slot)),
                     "n"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < kp.stages; ++s) {
            mbar_init(&blk.fullW[s], 1);
            mbar_init(&blk.fullX[s], 1);
            mbar_init(&blk.empty[s], 1);  // one tcgen05.commit per stage
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&blk.accFull[b], 1);
            mbar_init(&blk.accEmpty[b], kEpiWarps);
        }
        mbar_init(&blk.mmaDone, 1);
        for (int i = 0; i < AB_COUNT; ++i) {
            mbar_init(&blk.abar[i], i == AB_P_READY || i == AB_P_READY + 1 ? 128 : i == AB_FIXED ? 64 : 1);  // landed: the MMA issuer alone
            blk.acnt[i] = 0;
        }
        blk.role_rp[0] = RingPos();
        blk.role_rp[1] = RingPos();
        for (int i = 0; i < 8; ++i) blk.role_seg[i] = 0;
        Shared *sh = &blk.state;
        sh->arrived = 0;
        sh->passed = 0;
        sh->abort = 0;
        sh->go = 1;
        sh->epoch = 0;
        sh->wait_limit = kp.wait_cycles > 0 ? kp.wait_cycles : kWaitCycles;
        sh->ltab_staged = kp.n_layers <= kMaxStagedLayers;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x == 0) blk.state.tmem_base = blk.tmem_slot;  // read after the next barrier only

    if (warp == kConsumerWarps) {
        producer_program<NT>();
    } else {
        // =============================== work warps ===============================
        work_program<NT, WIDE>();
        if (warp == kXWarp && lane == 0 && blk.state.abort) {  // error path only: copies still in flight
            const RingPos rp = blk.role_rp[1];
            for (int s = 0; s < kp.stages; ++s)
                if ((rp.used >> s) & 1u) mbar_wait(&blk.fullX[s], ((rp.par >> s) & 1u) ^ 1u);
        }
        if (warp == kMmaWarp) {  // nothing of this CTA may still be running on the tensor core
            if (lane == 0) {
                tc_commit(&blk.mmaDone);
                mbar_wait(&blk.mmaDone, 0);
            }
            __syncwarp();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) leave_grid(kp.gbar);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(blk.tmem_slot), "n"(kTmemCols) : "memory");
    }
}

}  // namespace ssd
