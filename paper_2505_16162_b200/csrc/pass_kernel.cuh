// One decoder pass as ONE persistent kernel (sm_100a): one CTA per SM, launched cooperatively.
//
// The pass is a list of operations (embedding, the linear maps of the retained sublayers, KV-cache attention,
// LM head, arg-max) that every CTA walks in the same order.  Inside a CTA the producer warp walks the list on
// its own and streams the weights of every linear map into the shared-memory ring as fast as stages free up:
// weights do not depend on activations, so it runs ahead across operation boundaries.  The eight consumer
// warps execute the operations; between operations that depend on each other they meet all other CTAs at a
// grid-wide barrier (a monotonic counter in global memory).  While consumers wait there - or work through an
// attention operation, which reads the KV cache with plain loads - the ring keeps filling with the next linear
// map's weights, so the HBM stream does not stop at operation boundaries.
//
// Sublayers the skip mask leaves out are simply absent from the list: none of their weights is ever touched.
//
// Every wait is bounded.  A barrier or ring wait that gives up raises a device-wide abort word; every CTA then
// falls through the rest of the list without waiting or touching memory, and the host reports a timeout.
#pragma once
#include "linear_presplit.cuh"

namespace knnssd {
namespace pass {

using stream::LinPhase;
using stream::Ring;
using stream::NCW;

constexpr int MAXM = 16;           // rows per pass this kernel handles
constexpr int BLKM = 8;            // rows per tensor-core row block (linear maps take two blocks at once, an attention task has one)
constexpr int SEGP = 64;           // attention: positions per segment (fixed absolute boundaries)
constexpr unsigned BAR_SPIN_LIMIT = 4000000u;

enum { OP_EMBED = 0, OP_LINEAR = 1, OP_ATTN = 2, OP_HIDDEN = 3, OP_ARGMAX = 4, OP_ATTN_MERGE = 5 };
constexpr int MERGE_ROWS = 3;      // tasks with at least this many (row, head) pairs leave the merge to a separate operation

struct alignas(16) Op {
    int type;
    int barrier_after;   // 1: all CTAs meet before the next operation starts
    int is_head;         // OP_LINEAR: the LM head (runs on rows head_row0.. only)
    int layer;
    LinPhase lin;        // OP_LINEAR; OP_EMBED and OP_ATTN use its ys / next_gain / ss_out fields for their output
    bf16_t *kc, *vc;     // OP_ATTN: this layer's cache [n_kv_heads][max_seq][head_dim]
};
constexpr int OP_SLOTS_AT = 256;   // where the ring's bytes for barriers hold the operation at work and the one behind it
static_assert(OP_SLOTS_AT + 2 * sizeof(Op) <= stream::BAR_BYTES && 2 * stream::WS * 8 + 16 <= OP_SLOTS_AT, "two operations beside the ring's barriers");

struct Model {           // what does not change from pass to pass
    const bf16_t *tok_embed;
    const float *final_norm;
    float rms_eps;
    int d_model, H, Hkv, hd, vocab, max_seq, n_seg_max;
    const double *inv_freq;    // [hd/2]
    float *x, *logits, *hfinal;
    bf16_t *q;                 // [MAXM][H][2 terms][hd] rotated, hi and lo
    float2 *rope_cs;           // [grid][MAXM][hd/2]: one copy per CTA, written and read by that CTA only
    float *part_o;             // [MAXM][H][n_seg_max][hd]
    float2 *part_ml;           // [MAXM][H][n_seg_max]
    int *attn_cnt;             // [MAXM][H], zero between passes
    float *amax_v;             // [MAXM][grid]
    int *amax_i;
    int *amax_cnt;             // [1], zero between passes
    const DeviceState *state;
    unsigned long long *bar;   // grid barrier counter (monotonic)
    int *gabort;               // device-wide abort word
    int *err;
    unsigned long long *trace; // optional [n_ops][2] nanosecond stamps of CTA 0 (work done, barrier passed); nullptr = off
};

struct Params {
    const Op *ops;
    int n_ops;
    int M;                     // rows of this pass (1..MAXM)
    const int *tok;            // [M] token ids (device)
    int pos_off;               // first row sits at position state->len + pos_off
    int head_row0;             // rows >= head_row0 get logits and an arg-max (== M: none)
    int *argmax_out;           // [M - head_row0]
    int want_hidden;
    int out_row0;              // row of the logits / hidden-state buffers that this pass's row 0 goes to
    unsigned long long bar_base;   // value of *bar when this launch starts
    int merge_op;              // the attention partials are merged by the separate merge operation (merge_rows_separately)
    unsigned long long *stamp; // if given: when the pass began (pinned host memory)
    unsigned bar_spin_limit;   // polls a grid-barrier wait may take before the pass is aborted (0 = BAR_SPIN_LIMIT)
};

// Whether a pass of M rows merges its attention partials in the separate operation: when an attention task carries
// at least MERGE_ROWS (row, head) pairs.
__host__ __device__ inline bool merge_rows_separately(int M, int G) { return M * G >= MERGE_ROWS; }

// ---- grid-wide barrier among the consumer warps of all CTAs -----------------------------------------------
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Called by all 256 consumer threads.  Returns false once the pass has been aborted.  meanwhile(): what the CTA has to do for itself, done
// between its arrival and the wait for the others.
template <typename F>
__device__ __forceinline__ bool grid_barrier(const Model &md, const Ring &r, unsigned long long target, int tid, bool alive,
                                             unsigned spin_limit, F meanwhile) {
    asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory");
    if (tid == 0 && alive) {
        __threadfence();                       // cumulative: covers the writes of the CTA's other threads ordered by the bar.sync
        atomicAdd(md.bar, 1ULL);
    }
    meanwhile();
    if (tid == 0 && alive) {
        unsigned spins = 0;
        while (ld_acquire_u64(md.bar) < target) {
            // the abort words are looked at every 64 polls: a second trip to L2 per poll doubled the time between polls
            // (8 layers of the 13B widths, one row: 0.6255 -> 0.6237 ms)
            if ((spins & 63u) == 63u && (*r.abort_flag || *reinterpret_cast<volatile int *>(md.gabort))) { *r.abort_flag = 1; break; }
            if (++spins > spin_limit) {
                *r.abort_flag = 1;
                atomicExch(md.gabort, 1);
                atomicExch(md.err, 7);
                break;
            }
            __nanosleep(20);
        }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory");
    return alive && !*r.abort_flag;
}

// What runs once a pass is kept out of line: inlined, it shifted the registers and the code of the linear maps by up to 1 % of a pass.
// ---- embedding gather ----------------------------------------------------------------------------------------
__device__ __noinline__ void embed_phase(const Model &md, const Op &op, const Params &pr, const Ring &r, int cta, int n_cta,
                                            int tid) {
    if (tid == 0) *r.pos0 = md.state->len + pr.pos_off;
    if (tid == 0 && cta == 0 && pr.stamp) *pr.stamp = globaltimer_ns();
    if (cta >= pr.M) return;                               // whole CTAs only: the named barrier below is CTA-local
    // row m = cta: residual stream in fp32, its pre-split form times the first RMSNorm's gain, its sum of squares
    const int d = md.d_model, m = cta, lane = tid & 31, warp = tid >> 5;
    int t = pr.tok[m];
    if (t < 0 || t >= md.vocab) {                          // never gather outside the table: report and read row 0 instead
        if (tid == 0) atomicExch(md.err, ERR_BAD_TOKEN);
        t = 0;
    }
    const bf16_t *row = md.tok_embed + (size_t)t * d;
    float ss = 0.f;
    constexpr int U = 10;                                  // values in flight
    for (int i0 = tid; i0 < d; i0 += U * NCW * 32) {
        float v[U], g[U];
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const int i = i0 + e * NCW * 32;
            v[e] = i < d ? bf16_bits_to_float(__ldg(row + i)) : 0.f;
            g[e] = i < d && op.lin.next_gain ? __ldg(op.lin.next_gain + i) : 1.f;
        }
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const int i = i0 + e * NCW * 32;
            if (i >= d) break;
            __stcg(md.x + (size_t)m * d + i, v[e]);
            stream::store_split(op.lin.ys, d >> 7, m, i, v[e] * g[e]);
            ss = fmaf(v[e], v[e], ss);
        }
    }
    ss = warp_sum(ss);
    if (lane == 0) r.red_ss[32 + warp] = ss;
    asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory");
    if (tid == 0) {
        float tot = 0.f;
        for (int w = 0; w < NCW; ++w) tot += r.red_ss[32 + w];
        __stcg(op.lin.ss_out + (size_t)m * n_cta, tot);
    }
    for (int c = 1 + tid; c < n_cta; c += NCW * 32) __stcg(op.lin.ss_out + (size_t)m * n_cta + c, 0.f);
}

// The (cos, sin) of all rows' rotary angles, a copy for every CTA: 148 readers of one copy would queue up at L2.  Nobody else waits for it.
__device__ __noinline__ void rope_table(const Model &md, const Params &pr, int cta, int tid) {
    const int half = md.hd >> 1, p0 = md.state->len + pr.pos_off;
    float2 *mine = md.rope_cs + (size_t)cta * MAXM * half;
    for (int idx = tid; idx < pr.M * half; idx += NCW * 32) {
        const int m = idx / half, i = idx % half;
        double s, c;
        sincos((double)(p0 + m) * md.inv_freq[i], &s, &c);
        mine[idx] = make_float2((float)c, (float)s);
    }
}

// ---- RMSNorm of the rows written out (hidden-state output) -------------------------------------------------
__device__ __noinline__ void hidden_phase(const Model &md, const Params &pr, const Ring &r, int cta, int tid) {
    if (cta >= pr.M) return;          // whole CTAs only: the named barrier below is CTA-local
    const int d = md.d_model, m = cta, lane = tid & 31, warp = tid >> 5;
    const float *xr = md.x + (size_t)m * d;
    float s = 0.f;
    for (int i = tid; i < d; i += NCW * 32) { const float v = __ldcg(xr + i); s = fmaf(v, v, s); }
    s = warp_sum(s);
    if (lane == 0) r.red_ss[warp] = s;
    asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory");
    float tot = 0.f;
    for (int w = 0; w < NCW; ++w) tot += r.red_ss[w];
    const float rinv = 1.0f / sqrtf(tot / (float)d + md.rms_eps);
    for (int i = tid; i < d; i += NCW * 32) __stcg(md.hfinal + (size_t)(pr.out_row0 + m) * d + i, __ldcg(xr + i) * rinv * md.final_norm[i]);
    asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory");
}

// ---- greedy arg-max: every CTA scans the logits that it has just made (no barrier lies between), the last one folds the partials ----
// All warps share a row's slice, two rows at a time.  Row after row behind a barrier of the grid, five rows took 7.2 us and nine 10.
__device__ __noinline__ void argmax_phase(const Model &md, const Params &pr, const Ring &r, int cta, int n_cta, int tid) {
    const int V = md.vocab, lane = tid & 31, warp = tid >> 5, rows = pr.M - pr.head_row0;
    int i0, n;
    stream::unit_range(V, cta, n_cta, i0, n);
    float *s_v = r.red;                        // [rows][NCW]
    int *s_i = reinterpret_cast<int *>(r.red + MAXM * NCW);
    int *s_last = reinterpret_cast<int *>(r.red + 2 * MAXM * NCW);
    auto fold_warp = [](float &bv, int &bi) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            argmax_fold(bv, bi, ov, oi);
        }
    };
    for (int m = 0; m < rows; m += 2) {
        const float *row0 = md.logits + (size_t)(pr.out_row0 + pr.head_row0 + m) * V + i0, *row1 = row0 + (m + 1 < rows ? V : 0);
        float v0 = -INFINITY, v1 = -INFINITY;
        int k0 = 0x7fffffff, k1 = 0x7fffffff;
#pragma unroll 5
        for (int i = tid; i < n; i += NCW * 32) {
            argmax_fold(v0, k0, __ldcg(row0 + i), i0 + i);
            argmax_fold(v1, k1, __ldcg(row1 + i), i0 + i);
        }
        fold_warp(v0, k0);
        fold_warp(v1, k1);
        if (lane == 0) { s_v[m * NCW + warp] = v0; s_i[m * NCW + warp] = k0; s_v[(m + 1) * NCW + warp] = v1; s_i[(m + 1) * NCW + warp] = k1; }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory");
    if (warp == 0) {
        if (lane < rows) {
            float bv = -INFINITY;
            int bi = 0x7fffffff;
            for (int w = 0; w < NCW; ++w) argmax_fold(bv, bi, s_v[lane * NCW + w], s_i[lane * NCW + w]);
            __stcg(md.amax_v + lane * n_cta + cta, bv);
            __stcg(md.amax_i + lane * n_cta + cta, bi);
        }
        __syncwarp();
        if (lane == 0) {
            __threadfence();
            *s_last = atomicAdd(md.amax_cnt, 1) == n_cta - 1;
        }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory");
    if (*s_last) {
        __threadfence();
        for (int m = warp; m < rows; m += NCW) {
            float bv = -INFINITY;
            int bi = 0x7fffffff;
#pragma unroll 5
            for (int b = lane; b < n_cta; b += 32) argmax_fold(bv, bi, __ldcg(md.amax_v + m * n_cta + b), __ldcg(md.amax_i + m * n_cta + b));
            fold_warp(bv, bi);
            if (lane == 0) pr.argmax_out[m] = argmax_checked(bi, V, md.err);
        }
        if (tid == 0) *md.amax_cnt = 0;
    }
}

// ---- attention over the KV cache ------------------------------------------------------------------------------
// Rows m = 0..M-1 sit at positions P0 + m; row m attends to positions [0, P0 + m], all of them in the cache: the q / k / v map before
// has put the pass's own rows there.  The context is cut at fixed absolute boundaries into segments of SEGP positions; a warp
// handles one (K/V head, segment) for eight (query head, row) pairs: it reads each K and V row of the segment once, keeps the
// segment's scores in registers, takes a plain softmax over the segment and writes an un-normalised partial (max, sum, o).  The
// partials are merged in segment order and written pre-split for the output projection, by the warp that completes the last
// segment of a (row, head) where a task has one or two of them, else by an operation of its own.

// N 32-bit words of a q, K or V row.  STREAM: K and V, which come by once per pass: first to go when L2 needs room.
template <int N, bool STREAM> __device__ __forceinline__ void ld_words(const void *p, uint32_t *w) {
    if constexpr (N == 8 && STREAM)
        asm volatile("ld.global.L1::no_allocate.L2::evict_first.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]) : "l"(p) : "memory");
    else if constexpr (N == 8)
        asm volatile("ld.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]) : "l"(p) : "memory");
    else {
        static_assert(N == 4, "16 or 32 bytes");
        const uint4 v = STREAM ? __ldcs(reinterpret_cast<const uint4 *>(p)) : __ldcg(reinterpret_cast<const uint4 *>(p));
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    }
}

// c += a . b (m16n8k16, bf16 operands, fp32 accumulation): rows 0..7 of a from (a0, a2), rows 8..15 from (a1, a3).
__device__ __forceinline__ void mma_bf16_rows(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Merge the segment partials of one (row m, head h) in segment order and write the result pre-split (one warp).  Bound by the trips to L2: in
// passes of up to 8 rows (NB = 1) the first 24 segments' outputs come along with the statistics, others follow 24 at a time.  8 layers, ms, with
// 16 at a time behind the statistics and so: 13B 1 row at 1280 positions 0.5666 / 0.5626, 5 rows 1.0243 / 1.0164; Qwen 14B 5 rows at 2304 1.125 / 1.110.
// (9 and more rows have more merges than CTAs, and lose 0.5 .. 1 % by it.)
template <int HD, int NB>
__device__ __forceinline__ void attn_merge_row(const Model &md, const Op &op, int P0, int m, int h, int lane) {
    constexpr int DPL = HD / 32, AHEAD = NB == 1 ? 24 : 16;
    const int H = md.H, d0 = DPL * lane;
    const int n_seg_m = (P0 + m + SEGP) / SEGP;
    const size_t base = ((size_t)m * H + h) * md.n_seg_max;
    float pv[AHEAD][DPL];
    auto fetch = [&](int s0) {
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
            // one vector load per segment (DPL = 4: 16 bytes, DPL = 2: 8 bytes)
            const float *src = md.part_o + (base + s0 + i) * HD + d0;
            if (DPL == 4) {
                const float4 v = s0 + i < n_seg_m ? __ldcg(reinterpret_cast<const float4 *>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
                pv[i][0] = v.x; pv[i][1] = v.y; pv[i][DPL - 2] = v.z; pv[i][DPL - 1] = v.w;
            } else {
                const float2 v = s0 + i < n_seg_m ? __ldcg(reinterpret_cast<const float2 *>(src)) : make_float2(0.f, 0.f);
                pv[i][0] = v.x; pv[i][DPL - 1] = v.y;
            }
        }
    };
    // segment statistics: lane s holds segments s and s + 32 (contexts up to 4096); fixed-order warp reductions
    const float2 ml0 = lane < n_seg_m ? __ldcg(md.part_ml + base + lane) : make_float2(-INFINITY, 0.f);
    const float2 ml1 = lane + 32 < n_seg_m ? __ldcg(md.part_ml + base + lane + 32) : make_float2(-INFINITY, 0.f);
    if (NB == 1) fetch(0);
    const float gm = warp_max(fmaxf(ml0.x, ml1.x));
    const float w0 = ml0.x == -INFINITY ? 0.f : expf(ml0.x - gm), w1 = ml1.x == -INFINITY ? 0.f : expf(ml1.x - gm);
    const float L = warp_sum(fmaf(ml1.y, w1, ml0.y * w0));
    // weighted sum of the partial outputs in segment order
    float acc[DPL];
#pragma unroll
    for (int e = 0; e < DPL; ++e) acc[e] = 0.f;
    for (int s0 = 0; s0 < n_seg_m; s0 += AHEAD) {
        if (NB > 1 || s0) fetch(s0);
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
            const int sg = s0 + i;
            const float w = __shfl_sync(0xffffffffu, sg < 32 ? w0 : w1, sg & 31);
#pragma unroll
            for (int e = 0; e < DPL; ++e) acc[e] = fmaf(pv[i][e], w, acc[e]);
        }
    }
#pragma unroll
    for (int e = 0; e < DPL; ++e) stream::store_split(op.lin.ys, (H * HD) >> 7, m, h * HD + d0 + e, acc[e] / L);
}

// Tensor-core form.  Lane (g8, t4) = (lane / 4, lane % 4).  The task's eight (query head, row) pairs are both halves of the 16-row MMA
// operand: rows 0..7 their hi terms, rows 8..15 their lo terms, so that one product does both.
//   scores  S = Q K^T   m16n8k16 bf16: the 8 columns of a tile are 8 consecutive positions (column n = g8 of the K
//           operand = position 8*nt + g8).  A dot product does not care in which order its terms are taken, so k-step
//           s pairs k-indices with words 2s, 2s + 1 of the lane's share of a row: dimensions [RUN t4, RUN t4 + RUN) of either half
//           of the head, RUN = HD / 8, 32 bytes of either (HD = 128) - whole sectors.
//   output  O += P V    m16n8k16 bf16 over pairs of tiles: k-indices 2t4, 2t4+1 stand for positions 2t4, 2t4+1 of the
//           first tile and 2t4+8, 2t4+9 for the same positions of the second - exactly the four scores the lane already
//           holds - and column n = g8 of V-tile j is dimension (HD/8)*g8 + j, so a lane reads HD/8 contiguous
//           dimensions of four V rows; an operand register (two positions of one dimension) is one byte-permute of two
//           loaded words.  p is split into two bf16 terms.
// A lane ends up with output dimensions [DL*t4, DL*t4 + DL) of row g8, DL = HD / 4.
// Bound by the chain of latencies of one task (a warp has at most a few): q and half of the segment's K and V are on their way at once.
// With the heads rotated and split by every task, the pass's own K / V rows staged beside it and K read in 16-byte pieces 64 bytes apart
// (two requests a sector), attention and what follows it up to the output projection took 16.7 us a layer of the 13B widths at 1 row and
// 1280 positions, 18.5 at 5 rows, 23.7 of the 7B widths at 9 rows and 640; so 12.3, 12.7 and 10.8.
template <int HD, int NB>
__device__ __forceinline__ void attn_phase(const Model &md, const Op &op, const Params &pr, const Ring &r, int cta, int n_cta, int warp, int lane) {
    constexpr int DL = HD / 4;         // output dimensions per lane
    constexpr int RUN = HD / 8;        // dimensions of q and K per lane and half of the head
    constexpr int NW = HD / 8;         // 32-bit words of a q or K row per lane
    constexpr int VW = HD / 16;        // 32-bit words of a V row per lane
    constexpr int VJ = HD / 8;         // V tiles (8 dimensions each)
    constexpr int HALF = HD / 2;
    constexpr int NT = SEGP / 8;       // position tiles per segment
    constexpr int KR = 4;              // tiles in flight
    const int g8 = lane >> 2, t4 = lane & 3;
    const int M = pr.M, H = md.H, Hkv = md.Hkv, G = H / Hkv;
    const int P0 = *r.pos0, Ttot = P0 + M;
    // A task = (segment, K/V head, block of 8 of the R = G M (query head of the group, row) pairs rr = hg M + m).
    const int R = M * G, nblk = (R + BLKM - 1) / BLKM;
    const int n_seg = (Ttot + SEGP - 1) / SEGP, n_tasks = Hkv * n_seg * nblk;
    const float scale = 1.0f / sqrtf((float)HD);

    for (int t = warp * n_cta + cta; t < n_tasks; t += NCW * n_cta) {
        const int blk = t % nblk, tt = t / nblk, seg = tt / Hkv, kvh = tt % Hkv;
        const int rr = min(blk * BLKM + g8, R - 1);          // this lane's pair
        const int rm = rr % M, h = kvh * G + rr / M;
        const int p_begin = seg * SEGP, p_end = min(p_begin + SEGP, Ttot);
        const bool row_live = blk * BLKM + g8 < R && P0 + rm >= p_begin;         // it exists, and sees the segment
        if (!__any_sync(0xffffffffu, row_live)) continue;
        const bf16_t *kbase = op.kc + ((size_t)kvh * md.max_seq + p_begin + g8) * HD + RUN * t4;
        const bf16_t *vbase = op.vc + ((size_t)kvh * md.max_seq + p_begin + 2 * t4) * HD + 2 * VW * g8;
        auto load_k = [&](int nt, uint32_t (&dst)[NW]) {
            if (p_begin + 8 * nt + g8 < p_end) {
                ld_words<NW / 2, true>(kbase + 8 * nt * HD, dst);
                ld_words<NW / 2, true>(kbase + 8 * nt * HD + HALF, dst + NW / 2);
            } else {
#pragma unroll
                for (int w = 0; w < NW; ++w) dst[w] = 0u;
            }
        };
        auto load_v = [&](int nt, uint32_t (&dst)[2][VW]) {
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (p_begin + 8 * nt + 2 * t4 + e < p_end) {
                    ld_words<VW, true>(vbase + (8 * nt + e) * HD, dst[e]);
                } else {
#pragma unroll
                    for (int w = 0; w < VW; ++w) dst[e][w] = 0u;
                }
        };
        uint32_t qh[NW], ql[NW], kb[KR][NW], vb[KR][2][VW];
        {
            const bf16_t *q = md.q + ((size_t)rm * H + h) * (2 * HD) + RUN * t4;
            ld_words<NW / 2, false>(q, qh);
            ld_words<NW / 2, false>(q + HALF, qh + NW / 2);
            ld_words<NW / 2, false>(q + HD, ql);
            ld_words<NW / 2, false>(q + HD + HALF, ql + NW / 2);
        }
#pragma unroll
        for (int i = 0; i < KR; ++i) load_k(i, kb[i]);
#pragma unroll
        for (int i = 0; i < KR; ++i) load_v(i, vb[i]);
        // ---- scores of pair g8, positions 8 nt + 2 t4 + {0, 1} ----
        float sc[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            uint32_t(&k)[NW] = kb[nt % KR];
            float c[4] = {};
#pragma unroll
            for (int w = 0; w < NW; w += 2) mma_bf16_rows(c, qh[w], ql[w], qh[w + 1], ql[w + 1], k[w], k[w + 1]);
            sc[nt][0] = c[2] + c[0];
            sc[nt][1] = c[3] + c[1];
            if (nt + KR < NT) load_k(nt + KR, k);
        }
        // ---- softmax over the segment (the four lanes of a pair share it) ----
        float mx = -INFINITY, lsum = 0.f;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const bool valid = row_live && p_begin + 8 * nt + 2 * t4 + e <= P0 + rm;     // causal; also excludes positions past p_end
                sc[nt][e] = valid ? sc[nt][e] * scale : -INFINITY;
                mx = fmaxf(mx, sc[nt][e]);
            }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                sc[nt][e] = sc[nt][e] == -INFINITY ? 0.f : expf(sc[nt][e] - mx);
                lsum += sc[nt][e];
            }
        lsum += __shfl_xor_sync(0xffffffffu, lsum, 1);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, 2);
        // ---- o += p V ----
        float o[VJ][4];
#pragma unroll
        for (int j = 0; j < VJ; ++j) { o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f; }
#pragma unroll
        for (int np = 0; np < NT; np += 2) {
            // k-indices 2t4, 2t4+1 stand for this lane's two positions of tile np, 2t4+8, 2t4+9 for those of tile np + 1
            uint32_t ah[2], al[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) split_pair(sc[np + i][0], sc[np + i][1], ah[i], al[i]);
#pragma unroll
            for (int j = 0; j < VJ; ++j) {
                uint32_t b[2];
#pragma unroll
                for (int i = 0; i < 2; ++i)                  // dimension j of the two positions' rows
                    b[i] = __byte_perm(vb[(np + i) % KR][0][j / 2], vb[(np + i) % KR][1][j / 2], (j & 1) ? 0x7632 : 0x5410);
                mma_bf16_rows(o[j], ah[0], al[0], ah[1], al[1], b[0], b[1]);
            }
            if (np + KR < NT) { load_v(np + KR, vb[np % KR]); load_v(np + 1 + KR, vb[(np + 1) % KR]); }
        }
        // ---- partials out (pair g8: dimensions DL*t4 + j and DL*t4 + VJ + j); the last warp of a (row, head) merges ----
        if (row_live) {
            const size_t pidx = ((size_t)rm * H + h) * md.n_seg_max + seg;
            if (t4 == 0) __stcg(md.part_ml + pidx, make_float2(mx, lsum));
            float *po = md.part_o + pidx * HD + DL * t4;
#pragma unroll
            for (int j = 0; j < VJ; j += 4) {
                __stcg(reinterpret_cast<float4 *>(po + j), make_float4(o[j][2] + o[j][0], o[j + 1][2] + o[j + 1][0], o[j + 2][2] + o[j + 2][0], o[j + 3][2] + o[j + 3][0]));
                __stcg(reinterpret_cast<float4 *>(po + VJ + j), make_float4(o[j][3] + o[j][1], o[j + 1][3] + o[j + 1][1], o[j + 2][3] + o[j + 2][1], o[j + 3][3] + o[j + 3][1]));
            }
        }
        if (pr.merge_op) continue;                            // a separate merge operation follows a grid barrier
        __threadfence();
        __syncwarp();
        bool last = false;
        if (row_live && t4 == 0) {
            const int n_seg_m = (P0 + rm + SEGP) / SEGP;                  // segments row rm sees
            last = atomicAdd(md.attn_cnt + rm * H + h, 1) == n_seg_m - 1;
        }
        const unsigned last_mask = __ballot_sync(0xffffffffu, last);     // bit 4*g set: this warp finishes the (row, head) of lane row g
        if (last_mask) {
            __threadfence();
            for (int g = 0; g < BLKM; ++g) {
                if (!((last_mask >> (4 * g)) & 1u)) continue;
                const int rg = blk * BLKM + g, mg = rg % M, hg = kvh * G + rg / M;
                attn_merge_row<HD, NB>(md, op, P0, mg, hg, lane);
                if (lane == 0) md.attn_cnt[mg * H + hg] = 0;
            }
        }
    }
}

// With several rows the warp that finishes a head last would merge all its rows one after the other; the merges
// then run as an operation of their own instead, one (row, head) per warp across the whole grid.
template <int HD, int NB>
__device__ __forceinline__ void attn_merge_phase(const Model &md, const Op &op, const Params &pr, const Ring &r, int cta, int n_cta, int warp,
                                                 int lane) {
    const int P0 = *r.pos0, jobs = pr.M * md.H;
    for (int j = warp * n_cta + cta; j < jobs; j += NCW * n_cta) attn_merge_row<HD, NB>(md, op, P0, j / md.H, j % md.H, lane);
}

// ---- the pass ---------------------------------------------------------------------------------------------------
// NB = 1: passes of up to BLKM rows; NB = 2: 9..16 rows (a kernel of its own, so that the common one stays small).
// NP > 0: the linear maps take the rows four at a time with both terms in one operand (NP = 1: passes of up to 4 rows -
// every draft step; NP = 3, 4 with NB = 2: passes of 9..12 and 13..16 rows); NP = 0: eight at a time, one operand per term.
template <int HD, int NB, int NP>
__global__ void __launch_bounds__(stream::NTHREADS, 1) pass_kernel(const __grid_constant__ Model md, const __grid_constant__ Params pr) {
    extern __shared__ __align__(128) unsigned char smem[];
    Ring r;
    stream::ring_setup(r, smem, md.err);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cta = blockIdx.x, n_cta = gridDim.x;
    int w_use = 0;
    bool alive = true;
    if (warp >= NCW) {
        stream::regs_dec<stream::regs_producer<NB, NP>()>();
        if (warp == NCW) {
            for (int i = 0; i < pr.n_ops && alive; ++i) {
                const Op &op = pr.ops[i];
                if (op.type != OP_LINEAR) continue;
                LinPhase lp = op.lin;
                lp.M = pr.M;
                lp.gb = stream::groups_per_batch<NB, NP>();
                if (op.is_head) { if (pr.head_row0 >= pr.M) continue; }
                stream::produce_linear(lp, r, cta, n_cta, lane, w_use, alive);
            }
            if (!alive) stream::producer_drain_after_abort();
        } else if (stream::scales_apart<NB, NP>()) {
#pragma unroll 1
            for (int i = 0; i < pr.n_ops; ++i) {
                const Op &op = pr.ops[i];
                if (op.type != OP_LINEAR || !op.lin.ss_in || (op.is_head && pr.head_row0 >= pr.M)) continue;
                const int row0 = op.is_head ? pr.head_row0 : 0;
                stream::scale_rows(op.lin.ss_in + (size_t)row0 * n_cta, pr.M - row0, op.lin.K, op.lin.eps, r, n_cta, warp - NCW - 1, lane);
            }
        }
        return;
    }
    stream::regs_inc<stream::regs_consumer<NB, NP>()>();
    const int tid = threadIdx.x;
    unsigned long long n_bar = 0;
    // The operation behind the one at work is on its way into shared memory: read from L2 when its turn came (a barrier leaves nothing in
    // L1), its type and then its fields took two trips of ~0.6 us, six times a layer.
    Op *slots = reinterpret_cast<Op *>(reinterpret_cast<unsigned char *>(r.full_w) + OP_SLOTS_AT);
    auto fetch_op = [&](int i) {
        if (i < pr.n_ops && tid < (int)(sizeof(Op) / 16))
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(stream::smem_u32(slots + (i & 1)) + 16 * tid),
                         "l"(reinterpret_cast<const unsigned char *>(pr.ops + i) + 16 * tid) : "memory");
    };
    auto op_arrived = [] { asm volatile("cp.async.wait_all;" ::: "memory"); };
    fetch_op(0);
    op_arrived();
    asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory");
    for (int i = 0; i < pr.n_ops; ++i) {
        const Op &op = slots[i & 1];
        fetch_op(i + 1);                       // over the operation before this one, which all have left
        bool ran = true;
        if (op.type == OP_LINEAR) {
            LinPhase lp = op.lin;
            lp.M = pr.M;
            lp.gb = stream::groups_per_batch<NB, NP>();
            if (op.is_head) {
                if (pr.head_row0 >= pr.M) ran = false;
                lp.M = pr.M - pr.head_row0;
                lp.xs += (size_t)pr.head_row0 * (lp.K >> 7) * stream::SLOT_WORDS;
                lp.ss_in += (size_t)pr.head_row0 * n_cta;
                lp.y += (size_t)(pr.out_row0 + pr.head_row0) * lp.units;
            }
            lp.rope = md.rope_cs + (size_t)cta * MAXM * (HD / 2);
            if (stream::scales_apart<NB, NP>() && ran && lp.ss_in) stream::rows_ready();
            if (ran) stream::consume_linear_pre<NB, NP>(lp, r, cta, n_cta, warp, lane, w_use, alive);
        } else if (alive) {
            if (op.type == OP_EMBED) embed_phase(md, op, pr, r, cta, n_cta, tid);
            else if (op.type == OP_ATTN) attn_phase<HD, NB>(md, op, pr, r, cta, n_cta, warp, lane);
            else if (op.type == OP_ATTN_MERGE) { if (pr.merge_op) attn_merge_phase<HD, NB>(md, op, pr, r, cta, n_cta, warp, lane); else ran = false; }
            else if (op.type == OP_HIDDEN) { if (pr.want_hidden) hidden_phase(md, pr, r, cta, tid); else ran = false; }
            else if (op.type == OP_ARGMAX) { if (pr.head_row0 < pr.M) argmax_phase(md, pr, r, cta, n_cta, tid); else ran = false; }
        }
        if (md.trace && cta == 0 && tid == 0) md.trace[2 * i] = globaltimer_ns();
        op_arrived();
        if (op.barrier_after && ran) {
            ++n_bar;
            alive = grid_barrier(md, r, pr.bar_base + n_bar * (unsigned long long)n_cta, tid, alive,
                                 pr.bar_spin_limit ? pr.bar_spin_limit : BAR_SPIN_LIMIT,
                                 [&] { if (op.type == OP_EMBED) rope_table(md, pr, cta, tid); });
        } else {
            asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory");
        }
        if (md.trace && cta == 0 && tid == 0) md.trace[2 * i + 1] = globaltimer_ns();
    }
}

}  // namespace pass
}  // namespace knnssd
