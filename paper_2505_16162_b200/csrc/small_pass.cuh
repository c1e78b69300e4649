// A decoder pass of a small model in one launch (sm_100a).
//
// Models that the streaming pass kernel does not take (fp32 weights, widths that are no multiples of 128) run kernel by kernel.
// Where a layer's weights are a few MB the work of such a kernel is a microsecond and what it costs is the way from one to
// the next: 7 launches a layer, ~4.3 us each.  Here the pass is one cooperative launch of at most one block per SM that walks the
// same operations with a grid-wide meeting between dependent ones, five a layer (six where a row's context is more than one split): the rotary embedding and the K / V rows are
// written by the warps that compute the projections (a warp owns the two units of a rotary pair), and a row whose context is one
// split leaves its attention output without a merge.  Bound by the meetings and the trips to L2 behind them.  What a block can have before a
// meeting is over - the layers' pointers, its warps' first weight rows of the next map, the gains - is on its way into shared memory
// between its arrival and the others', and the rows of a map are brought in once for all warps.  Calls, us, before and with that: fp32 tiny
// shape (4 layers, d 256) at 96 positions, 1 / 5 / 16 rows 97 / 113 / 159, 93 / 108 / 151; bf16 d 1000, two layers 118 / 150 / 250, 86 / 112 / 187.
// (The copies begun before the arrival: no gain on the tiny shape.)
//
// Rows are independent of how many the pass carries.  Every wait is bounded: a block that gives up reports to the session's error
// word and all blocks fall through to the end.
#pragma once

#include "kernels.cuh"

namespace knnssd {
namespace small {

constexpr int NT = 256, NW = NT / 32;
constexpr int MASK_WORDS = 16;                 // sublayers of at most 256 layers
constexpr unsigned POLL_LIMIT = 4000000u;      // polls of one meeting
static_assert(NT == ATT_CHUNK, "a thread per position of a split");

struct LayerW {
    const void *wq, *wk, *wv, *wo, *w_gate, *w_up, *w_down;
    const float *attn_norm, *mlp_norm;
};
struct Args {
    const LayerW *layers;                      // [n_layers], device
    const void *tok_embed, *lm_head;
    const float *final_norm;
    int n_layers, d, H, Hkv, hd, F, V, max_seq;
    float eps;
    const DeviceState *st;
    const int *tok;                            // [M] device
    int M, pos_off, head_row0, want_hidden;    // rows from head_row0 on get logits and an arg-max (== M: none)
    int *argmax_out;
    const double *inv_freq;
    float *x, *qkv, *attn, *act, *logits, *hfinal, *part_o;
    float2 *part_ml, *rope_cs;
    int n_splits;
    void *kc, *vc;                             // [layer][kv head][max_seq][hd]
    unsigned long long *stamp;                 // if given: when the pass began (pinned host memory)
    unsigned *bar, *next_bar;                  // arrivals of this launch's meetings, zero at its start; the next launch's, zeroed by this one
    int *err;
    unsigned skip[MASK_WORDS];                 // bit j: sublayer j is left out
    // A pass whose attention has launches of its own (small_attend_kernel) comes in parts: from behind the attention of layer l_from
    // (-1: from the embedding) up to that of layer l_to (n_layers: to the end).
    int l_from, l_to;
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// All blocks have come this far and see one another's writes.  target: arrivals up to and including this meeting.  meanwhile(): what a block
// does for itself between its arrival and the others'.
template <typename F> __device__ __forceinline__ bool meet_grid(const Args &a, unsigned &target, int *s_abort, F meanwhile) {
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0 && !*s_abort) {
        __threadfence();                       // cumulative: covers the writes of the block's other threads ordered by the barrier
        atomicAdd(a.bar, 1u);
    }
    meanwhile();
    if (threadIdx.x == 0 && !*s_abort) {
        unsigned polls = 0;
        while (ld_acquire_u32(a.bar) < target)
            if (++polls > POLL_LIMIT) { *s_abort = 1; atomicExch(a.err, 8); break; }
    }
    __syncthreads();
    if (!*s_abort) return true;
    asm volatile("cp.async.wait_all;" ::: "memory");      // the block leaves: its own copies have landed by then
    return false;
}

// What the blocks of this launch write is read past the read-only path, from L2.
__device__ __forceinline__ float4 ld_row4(const float *p) { return __ldcg(reinterpret_cast<const float4 *>(p)); }

// RMSNorm scales of M rows of width d, a warp per row.
__device__ __forceinline__ void norm_scales(const float *x, int M, int d, float eps, float *s_rinv) {
    const int lane = threadIdx.x & 31;
    for (int m = threadIdx.x >> 5; m < M; m += NW) {
        float s = 0.f;
#pragma unroll 4
        for (int i = 4 * lane; i < d; i += 128) {
            const float4 v = ld_row4(x + (size_t)m * d + i);
            s = fmaf(v.x, v.x, s); s = fmaf(v.y, v.y, s); s = fmaf(v.z, v.z, s); s = fmaf(v.w, v.w, s);
        }
        s = warp_sum(s);
        if (lane == 0) s_rinv[m] = 1.0f / sqrtf(s / (float)d + eps);
    }
    __syncthreads();
}

// What a block keeps in shared memory: the layers' pointers; the weight rows of every warp's first item of the next map and that map's
// gains, on their way while the grid meets; the rows of the map at work.  What does not fit is read where it lies.
constexpr int W_STAGE = 8192, G_STAGE = 8192, X_STAGE = 96 * 1024, LAYERS_STAGE = 16 * MASK_WORDS * (int)sizeof(LayerW);
constexpr int SMEM_BYTES = NW * W_STAGE + G_STAGE + X_STAGE + LAYERS_STAGE;
struct Stage {
    unsigned char *w;                          // this warp's
    float *g, *x;
    LayerW *layers;
};
enum { MAP_HEADS = 0, MAP_O = 1, MAP_GATE_UP = 2, MAP_DOWN = 3, MAP_HEAD = 4, MAP_NONE = 5 };
struct Map { int which, layer; };

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ bool skipped(const Args &a, int sublayer) { return a.skip[sublayer >> 5] >> (sublayer & 31) & 1u; }
// The first map of layer l or of the layers behind it, then the head.
__device__ __forceinline__ Map first_map(const Args &a, int l) {
    for (; l < a.n_layers; ++l) {
        if (!skipped(a, 2 * l)) return {MAP_HEADS, l};
        if (!skipped(a, 2 * l + 1)) return {MAP_GATE_UP, l};
    }
    return {a.head_row0 < a.M ? MAP_HEAD : MAP_NONE, 0};
}
__device__ __forceinline__ Map next_map(const Args &a, Map m) {
    if (m.which == MAP_HEADS) return {MAP_O, m.layer};
    if (m.which == MAP_GATE_UP) return {MAP_DOWN, m.layer};
    if (m.which == MAP_O && !skipped(a, 2 * m.layer + 1)) return {MAP_GATE_UP, m.layer};
    return first_map(a, m.layer + 1);
}
__device__ __forceinline__ int map_width(const Args &a, int which) { return which == MAP_O ? a.H * a.hd : which == MAP_DOWN ? a.F : a.d; }
__device__ __forceinline__ int map_items(const Args &a, int which) {
    return which == MAP_HEADS ? (a.H + 2 * a.Hkv) * (a.hd / 2) : which == MAP_GATE_UP ? a.F : which == MAP_HEAD ? (a.V + 1) / 2 : a.d / 2;
}
__device__ __forceinline__ const float *map_gain(const Args &a, const Stage &st, Map m) {
    return m.which == MAP_HEADS ? st.layers[m.layer].attn_norm : m.which == MAP_GATE_UP ? st.layers[m.layer].mlp_norm : m.which == MAP_HEAD ? a.final_norm : nullptr;
}
// The two weight rows of an item: the dimensions of a rotary pair, gate and up, or units 2 item and 2 item + 1.
template <typename WT> __device__ __forceinline__ void map_rows_of(const Args &a, const Stage &st, Map m, int item, const WT *&r0, const WT *&r1) {
    const LayerW &ly = st.layers[m.layer];
    if (m.which == MAP_HEADS) {
        const int half = a.hd / 2;
        int slot = item / half;
        const void *W = ly.wq;
        if (slot >= a.H) { W = ly.wk; slot -= a.H; if (slot >= a.Hkv) { W = ly.wv; slot -= a.Hkv; } }
        r0 = reinterpret_cast<const WT *>(W) + (size_t)(slot * a.hd + item % half) * a.d;
        r1 = r0 + (size_t)half * a.d;
    } else if (m.which == MAP_GATE_UP) {
        r0 = reinterpret_cast<const WT *>(ly.w_gate) + (size_t)item * a.d;
        r1 = reinterpret_cast<const WT *>(ly.w_up) + (size_t)item * a.d;
    } else {
        const int K = map_width(a, m.which), n = m.which == MAP_HEAD ? a.V : a.d;
        const WT *W = reinterpret_cast<const WT *>(m.which == MAP_HEAD ? a.lm_head : m.which == MAP_O ? ly.wo : ly.w_down);
        r0 = W + (size_t)(2 * item) * K;
        r1 = W + (size_t)min(2 * item + 1, n - 1) * K;
    }
}
template <typename WT> __device__ __forceinline__ bool weights_fit(int K) { return 2 * K * (int)sizeof(WT) <= W_STAGE; }
// Starts the copies of what the blocks know of map m before they meet.  No warp is at a map with gains when another one's are fetched.
template <typename WT> __device__ __forceinline__ void stage_map(const Args &a, const Stage &st, Map m) {
    if (m.which == MAP_NONE) return;
    const int lane = threadIdx.x & 31, K = map_width(a, m.which), item = blockIdx.x * NW + (threadIdx.x >> 5);
    __syncwarp();                                                // the rows before have been read
    if (weights_fit<WT>(K) && item < map_items(a, m.which)) {
        const WT *r0, *r1;
        map_rows_of(a, st, m, item, r0, r1);
        for (int e = lane * 16; e < K * (int)sizeof(WT); e += 512) {
            cp_async16(st.w + e, reinterpret_cast<const unsigned char *>(r0) + e);
            cp_async16(st.w + K * sizeof(WT) + e, reinterpret_cast<const unsigned char *>(r1) + e);
        }
    }
    const float *gain = map_gain(a, st, m);
    if (gain && K * (int)sizeof(float) <= G_STAGE)
        for (int i = 4 * threadIdx.x; i < K; i += 4 * NT) cp_async16(st.g + i, gain + i);
}
// Eight weights from shared memory or from where they lie.
__device__ __forceinline__ void load8_any(const float *row, int e, float (&w)[8]) {
    const float4 p = *reinterpret_cast<const float4 *>(row + e), q = *reinterpret_cast<const float4 *>(row + e + 4);
    w[0] = p.x; w[1] = p.y; w[2] = p.z; w[3] = p.w; w[4] = q.x; w[5] = q.y; w[6] = q.z; w[7] = q.w;
}
__device__ __forceinline__ void load8_any(const bf16_t *row, int e, float (&w)[8]) {
    const uint4 v = *reinterpret_cast<const uint4 *>(row + e);
    const uint32_t p[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { w[2 * i] = __uint_as_float(p[i] << 16); w[2 * i + 1] = __uint_as_float(p[i] & 0xFFFF0000u); }
}

// A linear map over M <= MT rows of width K: a warp takes items gw, gw + (warps of the grid), ..; early(item, m) fetches what row m's end
// needs, done(item, m, v0, v1, fetched) gets the products with row m, in lane m.  NORM: of the rows times the map's gain, scaled by
// their RMSNorm (every warp reads the rows whole: it sums the squares on the way, where a pass of its own over them took 0.8 us).  The
// order of a sum depends on K alone.
template <typename WT, int MT, bool NORM, typename Early, typename Done>
__device__ __forceinline__ void map_rows(const Args &a, const Stage &st, Map map, const float *x, int M, Early early, Done done) {
    const int lane = threadIdx.x & 31, K = map_width(a, map.which), n_items = map_items(a, map.which);
    const float *gain = nullptr;
    if (NORM) gain = K * (int)sizeof(float) <= G_STAGE ? st.g : map_gain(a, st, map);
    if (M * K * (int)sizeof(float) <= X_STAGE) {                 // every warp of the block reads all rows
#pragma unroll 4
        for (int i = threadIdx.x; i < M * K / 4; i += NT) cp_async16(st.x + 4 * i, x + 4 * i);
        x = st.x;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (int first = blockIdx.x * NW + (threadIdx.x >> 5), item = first; item < n_items; item += gridDim.x * NW) {
        const WT *r0, *r1;
        if (item == first && weights_fit<WT>(K)) {
            r0 = reinterpret_cast<const WT *>(st.w);
            r1 = r0 + K;
        } else {
            map_rows_of(a, st, map, item, r0, r1);
        }
        float2 fetched = make_float2(0.f, 0.f);
        if (lane < M) fetched = early(item, lane);
        float acc[2][MT], ss[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) acc[0][m] = acc[1][m] = ss[m] = 0.f;
        for (int e = 8 * lane; e < K; e += 256) {
            float w0[8], w1[8];
            load8_any(r0, e, w0);
            load8_any(r1, e, w1);
            if (NORM) {
                const float4 g0 = *reinterpret_cast<const float4 *>(gain + e), g1 = *reinterpret_cast<const float4 *>(gain + e + 4);
                const float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
                for (int j = 0; j < 8; ++j) { w0[j] *= g[j]; w1[j] *= g[j]; }
            }
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const float *xr = x + (size_t)min(m, M - 1) * K + e;
                const float4 x0 = *reinterpret_cast<const float4 *>(xr), x1 = *reinterpret_cast<const float4 *>(xr + 4);
                const float xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    acc[0][m] = fmaf(w0[j], xv[j], acc[0][m]);
                    acc[1][m] = fmaf(w1[j], xv[j], acc[1][m]);
                    if (NORM) ss[m] = fmaf(xv[j], xv[j], ss[m]);
                }
            }
        }
        float v0 = 0.f, v1 = 0.f, sq = 0.f;
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const float s0 = warp_sum(acc[0][m]), s1 = warp_sum(acc[1][m]), s2 = NORM ? warp_sum(ss[m]) : 0.f;
            if (lane == m) { v0 = s0; v1 = s1; sq = s2; }
        }
        if (NORM) {
            const float rinv = 1.0f / sqrtf(sq / (float)K + a.eps);
            v0 = __fmul_rn(v0, rinv);
            v1 = __fmul_rn(v1, rinv);
        }
        if (lane < M) done(item, lane, v0, v1, fetched);
    }
}

// Attention of one (head, row, split of ATT_CHUNK positions) by a block: a thread per position for the scores, then threads by
// dimension, the positions in NT / hd interleaved runs, whose first PRE values are fetched along with the K rows (U float4s of one at a
// time).  single: the row's context is this split, its output is written at once.
template <typename WT, int PRE, int U>
__device__ __forceinline__ void attend(const Args &a, const WT *kc, const WT *vc, int T, int head, int m, int split, bool single, float *s_p, float *s_red) {
    const int t0 = split * ATT_CHUNK;
    if (t0 >= T) return;                                     // uniform over the block
    const int nt = min(T - t0, ATT_CHUNK), tid = threadIdx.x, hd = a.hd, warp = tid >> 5, lane = tid & 31;
    const size_t row0 = (size_t)(head / (a.H / a.Hkv)) * a.max_seq + t0;
    const int runs = NT / hd, e = tid % hd, run = tid / hd;
    const WT *vr = vc + row0 * hd + e;
    WT v_pre[PRE];
#pragma unroll
    for (int i = 0; i < PRE; ++i) v_pre[i] = run + i * runs < nt ? __ldcg(vr + (size_t)(run + i * runs) * hd) : WT(0);
    const float *q = a.qkv + (size_t)m * (a.H + 2 * a.Hkv) * hd + (size_t)head * hd;
    float s = -INFINITY;
    if (tid < nt) {
        const WT *kr = kc + (row0 + tid) * hd;
        float dot = 0.f;
        if (sizeof(WT) == 4) {
#pragma unroll U
            for (int i = 0; i < hd; i += 4) {
                const float4 k4 = ld_row4(reinterpret_cast<const float *>(kr) + i), q4 = ld_row4(q + i);
                dot = fmaf(q4.x, k4.x, dot); dot = fmaf(q4.y, k4.y, dot); dot = fmaf(q4.z, k4.z, dot); dot = fmaf(q4.w, k4.w, dot);
            }
        } else {
#pragma unroll (U / 2)
            for (int i = 0; i < hd; i += 8) {
                const uint4 k8 = __ldcg(reinterpret_cast<const uint4 *>(kr + i));
                const float4 qa = ld_row4(q + i), qb = ld_row4(q + i + 4);
                const uint32_t w[4] = {k8.x, k8.y, k8.z, k8.w};
                const float qv[8] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    dot = fmaf(qv[2 * j], __uint_as_float(w[j] << 16), dot);
                    dot = fmaf(qv[2 * j + 1], __uint_as_float(w[j] & 0xFFFF0000u), dot);
                }
            }
        }
        s = __fmul_rn(dot, 1.0f / sqrtf((float)hd));
    }
    const float wm = warp_max(s);
    if (lane == 0) s_red[warp] = wm;
    __syncthreads();
    float mx = s_red[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) mx = fmaxf(mx, s_red[w]);
    const float p = tid < nt ? expf(s - mx) : 0.f;
    s_p[tid] = p;
    const float ws = warp_sum(p);
    if (lane == 0) s_red[NW + warp] = ws;
    __syncthreads();
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) sum += s_red[NW + w];
    float o = 0.f;
#pragma unroll
    for (int i = 0; i < PRE; ++i)
        if (run + i * runs < nt) o = fmaf(s_p[run + i * runs], WeightLoad<WT>::load1(v_pre + i), o);
#pragma unroll 16
    for (int t = run + PRE * runs; t < nt; t += runs) {
        const WT v = __ldcg(vr + (size_t)t * hd);
        o = fmaf(s_p[t], WeightLoad<WT>::load1(&v), o);
    }
    __syncthreads();                                         // s_p has been read
    s_p[tid] = o;
    __syncthreads();
    if (tid < hd) {
        for (int r = 1; r < runs; ++r) o += s_p[r * hd + tid];
        if (single) {
            a.attn[(size_t)m * a.H * hd + (size_t)head * hd + tid] = o / sum;
        } else {
            const size_t at = ((size_t)m * a.H + head) * a.n_splits + split;
            a.part_o[at * hd + tid] = o;
            if (tid == 0) a.part_ml[at] = make_float2(mx, sum);
        }
    }
    __syncthreads();                                         // the next task's
}

// Attention of layer l for the pass's rows, the first of them at position pos0, by all blocks of the launch.
template <typename WT, int PRE, int U> __device__ __forceinline__ void attend_rows(const Args &a, int l, int pos0, float *s_p, float *s_red) {
    const size_t layer = (size_t)l * a.Hkv * a.max_seq * a.hd;
    const WT *kc = reinterpret_cast<const WT *>(a.kc) + layer, *vc = reinterpret_cast<const WT *>(a.vc) + layer;
    const int M = a.M, n_split = (pos0 + M + ATT_CHUNK - 1) / ATT_CHUNK;      // of the pass's last row
    for (int task = blockIdx.x; task < a.H * M * n_split; task += gridDim.x)
        attend<WT, PRE, U>(a, kc, vc, pos0 + task / a.H % M + 1, task % a.H, task / a.H % M, task / (a.H * M), n_split == 1, s_p, s_red);
}

// The same as a launch of its own, for many tasks: four blocks on an SM (fp32: three, whose rows are twice as long), which hide their latencies in
// one another, where small_pass_kernel has one with everything in flight that it can.  Bit for bit what that leaves.  Passes of 5 / 9 / 16 rows
// at 8000 positions, four layers of 16 heads of 64, two blocks as in small_pass_kernel / three / four, us: bf16 611 / 894 / 1382, 474 / 676 / 1094, 453 /
// 642 / 995; fp32 491 / 728 / 1206, 462 / 695 / 1134, 471 / 685 / 1110, of 8 heads of 128 532 / 758 / 1196, 489 / 715 / 1132, 523 / 728 / 1125.
template <typename WT> __global__ void __launch_bounds__(NT, sizeof(WT) == 4 ? 3 : 4) small_attend_kernel(const __grid_constant__ Args a, int l) {
    __shared__ float s_p[NT], s_red[2 * NW];
    attend_rows<WT, sizeof(WT) == 4 ? 16 : 8, 8>(a, l, a.st->len + a.pos_off, s_p, s_red);
}

template <typename WT, int MT>
__global__ void __launch_bounds__(NT, 1) small_pass_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(16) unsigned char small_smem[];
    __shared__ float s_rinv[MT], s_p[NT], s_red[2 * NW];
    __shared__ int s_red_i[NW], s_abort;
    const int tid = threadIdx.x, M = a.M, d = a.d, hd = a.hd, half = hd / 2, slots = a.H + 2 * a.Hkv;
    unsigned met = 0;
    if (tid == 0) {
        s_abort = 0;
        if (blockIdx.x == 0) {
            *a.next_bar = 0u;
            if (a.stamp && a.l_from < 0) *a.stamp = globaltimer_ns();
        }
    }
    const int pos0 = a.st->len + a.pos_off;
    auto nothing_more = [] {};
    Stage st;
    st.w = small_smem + (tid >> 5) * W_STAGE;
    st.g = reinterpret_cast<float *>(small_smem + NW * W_STAGE);
    st.x = st.g + G_STAGE / 4;
    st.layers = reinterpret_cast<LayerW *>(st.x + X_STAGE / 4);
    for (int i = tid; i < a.n_layers * (int)(sizeof(LayerW) / 8); i += NT)
        reinterpret_cast<unsigned long long *>(st.layers)[i] = reinterpret_cast<const unsigned long long *>(a.layers)[i];
    __syncthreads();
    stage_map<WT>(a, st, a.l_from < 0 ? first_map(a, 0) : Map{MAP_O, a.l_from});

    if (a.l_from < 0) {
        // embedding rows, and (from the last block on) the rows' rotary angles, in fp64
        for (int m = blockIdx.x; m < M; m += gridDim.x) {
            int t = a.tok[m];
            if (t < 0 || t >= a.V) {                         // never gather outside the table: report and read row 0 instead
                if (tid == 0) atomicExch(a.err, ERR_BAD_TOKEN);
                t = 0;
            }
            const WT *row = reinterpret_cast<const WT *>(a.tok_embed) + (size_t)t * d;
            for (int i = tid; i < d; i += NT) a.x[(size_t)m * d + i] = WeightLoad<WT>::load1(row + i);
        }
        for (int m = gridDim.x - 1 - blockIdx.x; m < M; m += gridDim.x)
            for (int i = tid; i < half; i += NT) {
                double s, c;
                sincos((double)(pos0 + m) * a.inv_freq[i], &s, &c);
                a.rope_cs[m * half + i] = make_float2((float)c, (float)s);
            }
        if (!meet_grid(a, met, &s_abort, nothing_more)) return;
    }

    const int n_split = (pos0 + M + ATT_CHUNK - 1) / ATT_CHUNK;      // of the pass's last row
    // d is even
    auto old_pair = [&](int item, int m) { return __ldcg(reinterpret_cast<const float2 *>(a.x + (size_t)m * d + 2 * item)); };
    auto add_pair = [&](int item, int m, float v0, float v1, float2 old) {
        *reinterpret_cast<float2 *>(a.x + (size_t)m * d + 2 * item) = make_float2(old.x + v0, old.y + v1);
    };
    auto nothing = [&](int, int) { return make_float2(0.f, 0.f); };
    for (int l = max(a.l_from, 0); l < a.n_layers; ++l) {
        if (!skipped(a, 2 * l)) {
            if (l != a.l_from) {
                WT *kc = reinterpret_cast<WT *>(a.kc) + (size_t)l * a.Hkv * a.max_seq * hd, *vc = reinterpret_cast<WT *>(a.vc) + (size_t)l * a.Hkv * a.max_seq * hd;
                map_rows<WT, MT, true>(a, st, {MAP_HEADS, l}, a.x, M,
                                 [&](int item, int m) { return __ldcg(a.rope_cs + m * half + item % half); },
                                 [&](int item, int m, float p, float q, float2 c) {
                                     const int slot = item / half, i = item % half;
                                     if (slot < a.H + a.Hkv) {
                                         // the rounding is spelled out, so that it is the same in every instance of the kernel
                                         const float rp = __fmaf_rn(p, c.x, -__fmul_rn(q, c.y));
                                         q = __fmaf_rn(q, c.x, __fmul_rn(p, c.y));
                                         p = rp;
                                     }
                                     if (slot < a.H) {
                                         float *dst = a.qkv + (size_t)m * slots * hd + (size_t)slot * hd + i;
                                         dst[0] = p;
                                         dst[half] = q;
                                     } else {
                                         const bool is_k = slot < a.H + a.Hkv;
                                         WT *dst = (is_k ? kc : vc) + ((size_t)(slot - a.H - (is_k ? 0 : a.Hkv)) * a.max_seq + pos0 + m) * hd + i;
                                         WeightLoad<WT>::store1(dst, p);
                                         WeightLoad<WT>::store1(dst + half, q);
                                     }
                                 });
                if (l == a.l_to) return;
                if (!meet_grid(a, met, &s_abort, [&] { stage_map<WT>(a, st, {MAP_O, l}); })) return;
                // (32 bf16 values of V ahead of the scores cost more than they hide: eight heads of 128, four layers, at 2000 positions, 5 / 9 rows
                // 384 / 498 us a call so, 353 / 459 with 16; fp32 loses 5 % at short contexts with 16)
                attend_rows<WT, sizeof(WT) == 4 ? 32 : 16, 16>(a, l, pos0, s_p, s_red);
                if (!meet_grid(a, met, &s_abort, nothing_more)) return;
            }
            if (n_split > 1) {
                for (int task = blockIdx.x; task < a.H * M; task += gridDim.x) {
                    const int m = task / a.H, ns = (pos0 + m + ATT_CHUNK) / ATT_CHUNK;
                    if (tid < hd) {
                        const size_t at = (size_t)task * a.n_splits;     // task = m H + head
                        float mx = -INFINITY, den = 0.f, o = 0.f;
                        for (int s = 0; s < ns; ++s) mx = fmaxf(mx, __ldcg(a.part_ml + at + s).x);
                        for (int s = 0; s < ns; ++s) {
                            const float2 ml = __ldcg(a.part_ml + at + s);
                            const float w = expf(ml.x - mx);
                            den = fmaf(ml.y, w, den);
                            o = fmaf(__ldcg(a.part_o + (at + s) * hd + tid), w, o);
                        }
                        a.attn[(size_t)task * hd + tid] = o / den;
                    }
                }
                if (!meet_grid(a, met, &s_abort, nothing_more)) return;
            }
            map_rows<WT, MT, false>(a, st, {MAP_O, l}, a.attn, M, old_pair, add_pair);
            if (!meet_grid(a, met, &s_abort, [&] { stage_map<WT>(a, st, next_map(a, {MAP_O, l})); })) return;
        }
        if (!skipped(a, 2 * l + 1)) {
            map_rows<WT, MT, true>(a, st, {MAP_GATE_UP, l}, a.x, M,
                             nothing,
                             [&](int item, int m, float g, float u, float2) {
                                 a.act[(size_t)m * a.F + item] = g / (1.0f + expf(-g)) * u;
                             });
            if (!meet_grid(a, met, &s_abort, [&] { stage_map<WT>(a, st, {MAP_DOWN, l}); })) return;
            map_rows<WT, MT, false>(a, st, {MAP_DOWN, l}, a.act, M, old_pair, add_pair);
            if (!meet_grid(a, met, &s_abort, [&] { stage_map<WT>(a, st, next_map(a, {MAP_DOWN, l})); })) return;
        }
    }
    const int hm = M - a.head_row0;
    if (!a.want_hidden && hm <= 0) return;
    if (a.want_hidden && (int)blockIdx.x < M) {
        norm_scales(a.x, M, d, a.eps, s_rinv);
        for (int m = blockIdx.x; m < M; m += gridDim.x)
            for (int i = tid; i < d; i += NT) a.hfinal[(size_t)m * d + i] = __ldcg(a.x + (size_t)m * d + i) * s_rinv[m] * a.final_norm[i];
    }
    if (hm <= 0) return;
    map_rows<WT, MT, true>(a, st, {MAP_HEAD, 0}, a.x + (size_t)a.head_row0 * d, hm,
                     nothing,
                     [&](int item, int m, float v0, float v1, float2) {
                         float *dst = a.logits + (size_t)(a.head_row0 + m) * a.V + 2 * item;
                         dst[0] = v0;
                         if (2 * item + 1 < a.V) dst[1] = v1;
                     });
    if (!meet_grid(a, met, &s_abort, nothing_more)) return;
    for (int j = blockIdx.x; j < hm; j += gridDim.x) {               // arg-max of a row by a block, lowest index among equals
        const float *row = a.logits + (size_t)(a.head_row0 + j) * a.V;
        float bv = -INFINITY;
        int bi = 0x7fffffff;
#pragma unroll 4
        for (int i = tid; i < a.V; i += NT) argmax_fold(bv, bi, __ldcg(row + i), i);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            argmax_fold(bv, bi, ov, oi);
        }
        __syncthreads();
        if ((tid & 31) == 0) { s_red[tid >> 5] = bv; s_red_i[tid >> 5] = bi; }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < NW; ++w) argmax_fold(bv, bi, s_red[w], s_red_i[w]);
            a.argmax_out[j] = argmax_checked(bi, a.V, a.err);
        }
    }
}

}  // namespace small
}  // namespace knnssd
