// Prompt pass on the 5th-generation tensor cores.
//
// The prompt pass is the full model over all T prompt tokens at once (Section 4.2: the sample's last hidden vector
// comes from a pass of the model over the sample; the same pass fills the K/V cache that drafting and verification
// read).  With T in the hundreds or thousands every linear map is a real contraction [T x K] . [K x N], so it runs on
// tcgen05.mma with the accumulator in tensor memory, operands staged in shared memory by TMA:
//
//   gemm_split_kernel   Y[T][N] (+)= A[T][K] . W[N][K]^T, A given as two bf16 planes (hi + lo of the fp32
//                       activation, so that the product with the bf16 weights carries 16 mantissa bits of A, as in
//                       the decode passes), accumulator fp32.  Epilogues: store, add to the residual stream,
//                       SwiGLU of a gate tile and an up tile.
//   norm_split_kernel   the embedding rows times the first gain, as the two bf16 planes the first map reads, and their RMSNorm scales.
//   scales_kernel       the RMSNorm scales of rows that a map has added to.
//   fold_pieces_kernel  the sums of the tiles that a launch did in pieces, and their epilogue.
//   rope_kv_rows_kernel rotary embedding of q and k, K/V rows rounded to bf16 into the cache, where the contraction's epilogue
//                       has not done it.
//   attn_prompt_kernel  causal attention of 64 query rows per CTA (16 per warp) over the cached K/V, staged segment by
//                       segment in shared memory, on mma.sync (the sizes are small next to the linear maps), output
//                       written as bf16 planes for the O projection.
//
// Every wait in these kernels is bounded; a wait that gives up sets the error word and the kernel returns after
// releasing its tensor memory.
#pragma once

#include <cuda.h>

#include "linear_stream.cuh"

namespace knnssd {
namespace prefill {

using stream::mbar_init;
using stream::mbar_try_wait;
using stream::smem_u32;

constexpr int ROW_PAD = 128;                          // the activation planes' rows are padded to a multiple of this
constexpr int PAIR_UNITS = 256;                       // weight rows per tile: 128 in each CTA of a pair = lanes of its tensor memory
constexpr int TT_MAX = 256, TT_STEP = 32;             // most tokens per tile = accumulator columns; a launch picks a multiple of 32
constexpr int BOX_N = 64;                             // weight rows per TMA box
constexpr int BK = 64;                                // input columns per stage: 128 bytes of bf16 = one swizzle row
constexpr int W_BYTES = 128 * BK * 2;                 // a CTA's weight rows of a stage
// The ring of stages.  A stage is what a CTA holds of a k-block: 128 weight rows and half of the tile's token rows of either
// plane, 48 KB at 256 tokens (four stages), 28 KB at 96 (six).
constexpr int RING_BYTES = 192 * 1024;
constexpr int MAX_STAGES = 10;
__host__ __device__ constexpr int stage_bytes_of(int tt) { return W_BYTES + tt * BK * 2; }
__host__ __device__ constexpr int ring_stages(int tt) {
    return RING_BYTES / stage_bytes_of(tt) < MAX_STAGES ? RING_BYTES / stage_bytes_of(tt) : MAX_STAGES;
}
constexpr int TURN_TOKENS = 16;                       // tokens that a group of epilogue warps turns at a time (see below)
constexpr int TURN_BYTES = 2 * 2 * TURN_TOKENS * 128 * 4 + 2 * 128 * 4;      // two groups: two buffers each, and the scales of their tokens
constexpr int TMEM_COLS = 512;                        // columns of tensor memory a CTA takes: two accumulators of TT_MAX columns
constexpr int CHUNK_KB = 8;                           // k-blocks accumulated in tensor memory before the sum moves to registers
constexpr int GEMM_THREADS = 320;                     // warp 0: TMA; warp 1: MMA issue + tensor-memory owner; warps 2..9: epilogue
__host__ __device__ constexpr int gemm_smem(int tt) {          // + slack to align the tiles to 1024 bytes + barriers
    return TURN_BYTES + ring_stages(tt) * stage_bytes_of(tt) + 1024 + 256;
}
constexpr int GEMM_SMEM_MAX = TURN_BYTES + RING_BYTES + 1024 + 256;
constexpr unsigned WAIT_LIMIT = 4000000u;           // polls of one wait (a whole tile takes well under a millisecond)

enum { PF_STORE = 0, PF_ADD = 1, PF_SWIGLU = 2, PF_QKV = 3 };

struct GemmArgs {
    int T;             // live rows
    int K;             // input width, a multiple of BK
    int N;             // output units (per matrix)
    int tt;            // tokens per tile: a multiple of TT_STEP, at most TT_MAX
    float *y;          // STORE: y[t * ldy + col0 + n] = sum;  ADD: y[t * ldy + col0 + n] += sum
    int ldy, col0;
    bf16_t *out_hi;    // SWIGLU: silu(gate) * up as two bf16 planes, [t * ldo + n]
    bf16_t *out_lo;
    int ldo;
    int *err;          // set non-zero if a bounded wait gave up
    int tiles_x, tiles_y;   // token tiles and unit tiles of the launch (tile = ty tiles_x + tx)
    int box;           // weight rows per box: BOX_N, or 128 where the matrices allow it
    int whole;         // tiles [0, whole) are done whole by one pair each, the others in pieces (see Jobs below)
    float *part;       // the chunk sums of the tiles done in pieces, [tiles - whole][chunks][CTA of the pair][tt][128]: what
                       // gemm_split_kernel leaves and fold_pieces_kernel picks up
    int nA, nB;        // STORE over stacked matrices (q, k, v in one launch): units [0, nA) are rows of map tb0,
                       // [nA, nA + nB) rows of tb1, the rest rows of tb2; all multiples of BOX_N.  One matrix: nA = N
    const float *row_scale;   // if given: every sum of row t is multiplied by row_scale[t] before the epilogue (the RMSNorm
                              // scale of the row whose gain-weighted, un-normalised values the planes hold)
    // ADD, if given: what the map that reads the new rows behind an RMSNorm needs of them: y times next_gain as two planes of row length
    // N, and the sums of squares of every four of their columns, [t][N / 4] (N a multiple of 128)
    const float *next_gain;
    bf16_t *next_hi, *next_lo;
    float *ss_out;
    // PF_QKV (stacked q, k, v; head dimension 128, so that a CTA's 128 weight rows are one head): the q heads are rotated
    // and stored to y, the k heads rotated, the k and v heads rounded to bf16 into the cache rows of position pos0 + t
    const float2 *rope;    // [T][64] (cos, sin) of the rows' positions
    bf16_t *kc, *vc;       // this layer's K and V cache, [kv head][max_seq][128]
    int max_seq, pos0;
};

// What one thread of a warp issues - copies, products, commits - takes its operands in uniform registers.  Inside a branch on the lane
// the compiler has to move each of them there first (46 clocks per product of any size, 0.08 us per copy), so the warp
// runs these loops as a whole and the instructions are predicated: `one` is 1 in the thread that issues them.
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t one;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one));
    return one;
}
// A TMA load into this CTA's shared memory (dst) whose bytes are counted by a barrier of the pair's first CTA (`bar`: its address
// in the cluster's window).
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar, uint64_t policy, uint32_t one) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %6, 0;\n\t"
                 "@p cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;\n\t}" ::"r"(dst),
                 "l"(map), "r"(bar), "r"(x), "r"(y), "l"(policy), "r"(one)
                 : "memory");
}
__device__ __forceinline__ void expect_tx_if(uint32_t bar, uint32_t bytes, uint32_t one) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(bar), "r"(bytes), "r"(one) : "memory");
}

// Shared-memory operand descriptor of tcgen05.mma for a K-major tile whose rows are 128 bytes, written by TMA with the
// 128-byte swizzle: start address / 16 in bits 0..13, leading-dimension offset (unused for this layout) in 16..29,
// stride between groups of 8 rows (1024 bytes) / 16 in 32..45, descriptor version 1 in 46..47, swizzle mode 2
// (128 bytes) in 61..63.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
           ((uint64_t)2 << 61);
}
// Instruction descriptor, kind::f16: fp32 accumulator (bits 4..5 = 1), A and B bf16 (bits 7..9 and 10..12 = 1), both
// K-major (bits 15, 16 = 0), N / 8 in bits 17..22, M / 16 in bits 24..28.
__device__ __forceinline__ uint32_t umma_idesc(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// One instruction for the pair, issued by its first CTA: the 256 rows of A are 128 rows of either CTA's shared memory, the
// columns of B half of either's, at the same addresses; a CTA's tensor memory takes the sums of its own 128 rows.  a, b: the
// operands' descriptors without their constant upper halves.  The weights of a k-step meet the hi and the lo terms: FIRST reads them
// from shared memory, the product behind it takes them from where the first left them.
constexpr uint32_t DESC_UPPER = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lower(uint32_t saddr) { return (saddr >> 4) | (1u << 16); }
template <bool FIRST>
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t accumulate, uint32_t one) {
#define KNNSSD_UMMA_PAIR(COLLECT) \
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\tmov.b64 da, {%1, %6};\n\tmov.b64 db, {%2, %6};\n\t" \
                 "@q tcgen05.mma.cta_group::2.kind::f16.collector::a::" COLLECT " [%0], da, db, %3, p;\n\t}\n" \
                 ::"r"(tmem_d), "r"(a), "r"(b), "r"(idesc), "r"(accumulate), "r"(one), "r"(DESC_UPPER) : "memory")
    if (FIRST) KNNSSD_UMMA_PAIR("fill");
    else KNNSSD_UMMA_PAIR("lastuse");
#undef KNNSSD_UMMA_PAIR
}
// The barrier at this address in both CTAs gets one arrival once every MMA this thread issued before has finished.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar, uint32_t one) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}" ::"r"(bar),
                 "h"((uint16_t)3), "r"(one)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// The address of the pair's first CTA's copy of a shared-memory word.
__device__ __forceinline__ uint32_t first_cta_addr(const void *p) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(smem_u32(p)));
    return a;
}
__device__ __forceinline__ void pair_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void pair_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// 32 consecutive accumulator columns of this thread's lane (lane = 32 * (warp % 4) + lane id).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, "
        "%18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// mbar_try_wait for a barrier whose other CTA's arrivals have to be seen with what they release.
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t *b, uint32_t parity) {
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(smem_u32(b)), "r"(parity) : "memory");
    return done != 0;
}

// Bounded wait on an mbarrier phase; false once the limit is reached or another thread of the CTA has given up.
template <bool CLUSTER = false>
__device__ __forceinline__ bool pf_wait(uint64_t *b, uint32_t parity, volatile int *cta_abort, int *err, int code) {
    unsigned spins = 0;
    while (!(CLUSTER ? mbar_try_wait_cluster(b, parity) : mbar_try_wait(b, parity))) {
        if (*cta_abort) return false;
        if (++spins > WAIT_LIMIT) {
            *cta_abort = 1;
            atomicExch(err, code);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ uint32_t pack_bf16(uint32_t lo16, uint32_t hi16) { return lo16 | (hi16 << 16); }

// How a launch's work is dealt out to its pairs of CTAs (one CTA per SM).  Tiles [0, whole) go round: pair c takes tiles c,
// c + G, .., so that all pairs are at the same k-blocks of neighbouring tiles and share them through L2.  The chunks (CHUNK_KB
// k-blocks) of the tiles that are left, fewer than the pairs, are dealt out evenly, pair c of P getting chunks
// [c U / P, (c + 1) U / P): a last round that would leave most of the chip idle takes the time its work takes.
// A piece's chunk sums go to `part` one by one, and fold_pieces_kernel, launched behind, adds a tile's up from the first chunk
// to the last, the order of a tile done whole: a row's numbers do not depend on how the launch was dealt out.  No pair waits
// for another: a launch that is not cooperative may run in parts, with another stream's launch on the SMs between them.
struct Jobs {
    int G, P, cta, whole, nchunks, n_whole, r0;      // P: the pairs that get pieces, one chunk each at least
    long long units, u0, u1;
    __device__ __forceinline__ Jobs(const GemmArgs &g) : G(gridDim.x >> 1), cta(blockIdx.x >> 1), whole(g.whole) {
        nchunks = (g.K / BK + CHUNK_KB - 1) / CHUNK_KB;
        n_whole = cta < whole ? (whole - cta + G - 1) / G : 0;
        units = (long long)(g.tiles_x * g.tiles_y - whole) * nchunks;
        P = (int)min((long long)G, units);
        u0 = cta < P ? units * cta / P : 0;
        u1 = cta < P ? units * (cta + 1) / P : 0;
        r0 = (int)(u0 / nchunks);
    }
    // job i of this pair: chunks [c0, c1) of a tile; false when there is none
    __device__ __forceinline__ bool get(int i, int &tile, int &c0, int &c1) const {
        if (i < n_whole) { tile = cta + i * G; c0 = 0; c1 = nchunks; return true; }
        const int r = r0 + i - n_whole;
        const long long first = (long long)r * nchunks;
        if (first >= u1 || u0 >= u1) return false;
        tile = whole + r;
        c0 = first < u0 ? (int)(u0 - first) : 0;
        c1 = (int)min((long long)nchunks, u1 - first);
        return true;
    }
};

// First unit of a CTA's 128 weight rows (SwiGLU: 64 gate rows, then the up rows of the same 64 units).
template <int EPI> __device__ __forceinline__ int first_unit(int ty, int rank) {
    return EPI == PF_SWIGLU ? ty * (PAIR_UNITS / 2) + 64 * rank : ty * PAIR_UNITS + 128 * rank;
}

// The sum of four squares, as one order of roundings wherever it is taken.
__device__ __forceinline__ float squares(float a, float b, float c, float d) {
    return __fmaf_rn(d, d, __fmaf_rn(c, c, __fmaf_rn(a, a, __fmul_rn(b, b))));
}
// v = x g in two bf16 terms.
__device__ __forceinline__ void split_product(float x, float g, uint32_t &hi, uint32_t &lo) {
    const float v = __fmul_rn(x, g);
    hi = float_to_bf16_rne(v);
    lo = float_to_bf16_rne(v - __uint_as_float(hi << 16));
}
// RMSNorm's scale of a row.  ss: the squares of the columns 4 tid .. 4 tid + 3, 1024 further and so on, added up by 256 threads; here lanes and
// then warps are.
__device__ __forceinline__ float scale_of_row(float ss, float *part, int d, float eps) {
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += part[w];
    return 1.0f / sqrtf(tot / (float)d + eps);
}

// ADD: the old values of token t that finish_sums takes for weight rows j .. j + 3 and j + 64 .. j + 67.
template <int EPI> __device__ __forceinline__ void old_values(const GemmArgs &g, int u0, int t, int j, float4 (&x)[2]) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        x[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (EPI == PF_ADD && t < g.T && u0 + j + 64 * e < g.N) x[e] = *reinterpret_cast<const float4 *>(g.y + (size_t)t * g.ldy + g.col0 + u0 + j + 64 * e);
    }
}

// What becomes of the sums of token t for the weight rows j .. j + 3 (v[0 .. 3]) and j + 64 .. j + 67 (v[4 .. 7]) of a CTA whose
// rows start at unit u0; j is a multiple of 4 below 64.  SwiGLU: gate and up of four units; q / k / v heads: four pairs of one
// head; else units.  Products that meet a sum are rounded by themselves, whichever kernel this is part of.
// rs: the row's scale (SwiGLU, q / k / v and store; 1: none).
template <int EPI> __device__ __forceinline__ void finish_sums(const GemmArgs &g, int u0, int t, int j, float (&v)[8], const float4 (&x)[2], float rs) {
    if (EPI != PF_ADD) {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __fmul_rn(v[i], rs);
    }
    if (EPI == PF_SWIGLU) {
        if (u0 + j >= g.N) return;                       // N is a multiple of 8
        uint32_t h[4], l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = __fmul_rn(v[i] / (1.0f + expf(-v[i])), v[4 + i]);
            h[i] = float_to_bf16_rne(a);
            l[i] = float_to_bf16_rne(a - __uint_as_float(h[i] << 16));
        }
        const size_t at = (size_t)t * g.ldo + u0 + j;
        *reinterpret_cast<uint2 *>(g.out_hi + at) = make_uint2(pack_bf16(h[0], h[1]), pack_bf16(h[2], h[3]));
        *reinterpret_cast<uint2 *>(g.out_lo + at) = make_uint2(pack_bf16(l[0], l[1]), pack_bf16(l[2], l[3]));
    } else if (EPI == PF_QKV) {
        if (u0 >= g.N) return;
        if (u0 < g.nA + g.nB) {                          // a q or a k head: rotary embedding
            const float4 *cs = reinterpret_cast<const float4 *>(g.rope + (size_t)t * 64 + j);
            const float4 c0 = cs[0], c1 = cs[1];
            rotate_pair(v[0], v[4], make_float2(c0.x, c0.y));
            rotate_pair(v[1], v[5], make_float2(c0.z, c0.w));
            rotate_pair(v[2], v[6], make_float2(c1.x, c1.y));
            rotate_pair(v[3], v[7], make_float2(c1.z, c1.w));
        }
        const bool is_k = u0 < g.nA + g.nB;
        const int kvh = (u0 - g.nA - (is_k ? 0 : g.nB)) >> 7;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if (u0 < g.nA) {
                *reinterpret_cast<float4 *>(g.y + (size_t)t * g.ldy + g.col0 + u0 + j + 64 * e) = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            } else {
                bf16_t *dst = (is_k ? g.kc : g.vc) + ((size_t)kvh * g.max_seq + g.pos0 + t) * 128 + j + 64 * e;
                uint32_t w[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) w[i] = pack_bf16(float_to_bf16_rne(v[4 * e + 2 * i]), float_to_bf16_rne(v[4 * e + 2 * i + 1]));
                *reinterpret_cast<uint2 *>(dst) = make_uint2(w[0], w[1]);
            }
        }
    } else {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if (u0 + j + 64 * e >= g.N) continue;        // N is a multiple of 8
            float4 o = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            if (EPI == PF_ADD) { o.x += x[e].x; o.y += x[e].y; o.z += x[e].z; o.w += x[e].w; }
            *reinterpret_cast<float4 *>(g.y + (size_t)t * g.ldy + g.col0 + u0 + j + 64 * e) = o;
            if (EPI == PF_ADD) { v[4 * e] = o.x; v[4 * e + 1] = o.y; v[4 * e + 2] = o.z; v[4 * e + 3] = o.w; }
        }
        if (EPI == PF_ADD && g.next_gain && u0 < g.N) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float4 gn = __ldg(reinterpret_cast<const float4 *>(g.next_gain + u0 + j + 64 * e));
                const float w[4] = {gn.x, gn.y, gn.z, gn.w};
                uint32_t h[4], l[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) split_product(v[4 * e + i], w[i], h[i], l[i]);
                const size_t at = (size_t)t * g.N + u0 + j + 64 * e;
                *reinterpret_cast<uint2 *>(g.next_hi + at) = make_uint2(pack_bf16(h[0], h[1]), pack_bf16(h[2], h[3]));
                *reinterpret_cast<uint2 *>(g.next_lo + at) = make_uint2(pack_bf16(l[0], l[1]), pack_bf16(l[2], l[3]));
                g.ss_out[at >> 2] = squares(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            }
        }
    }
}

// Tiles of 256 weight rows x tt tokens, dealt out to pairs of CTAs, one CTA per SM (Jobs).  The weights are the row operand of
// the products, 128 rows in either CTA, and the tokens their columns, so that a tile takes any multiple of 32 tokens; each
// CTA brings in half of the token rows of both planes, and the pair's tensor cores read both halves.  EPI = PF_SWIGLU: a CTA's
// rows are 64 units of the gate matrix (map tb0) and the same units of the up matrix (map tb1); otherwise units of one
// matrix (tb0 = tb1).  ta covers both activation planes: rows [0, Tpad) the hi terms, rows [Tpad, 2 Tpad) the lo terms, in boxes
// of tt / 2 rows (rows past T are whatever the planes hold; they meet no live token).  Weight maps: boxes of g.box rows.
//
// Accumulation.  The tensor core adds every 16-column product into its fp32 accumulator by truncation, so a sum that
// stays in tensor memory over all of K collects an error that grows with the number of steps (measured: ~4e-5 relative
// at K = 13824, ten times the error of the decode passes' sums; through the bf16 rounding of the K/V rows it feeds,
// that showed as 2.4e-2 on the logits of a 40-layer model).  The sum over K is therefore cut into chunks of CHUNK_KB
// k-blocks: a chunk accumulates in one of two accumulators in tensor memory while the eight epilogue warps move the
// previous chunk's sum out and add it, rounded to nearest, to the running sums they keep in registers (a thread owns
// one weight row and half of the tile's tokens).  The error left is that of the short chunks plus K / (64 CHUNK_KB)
// ordinary fp32 additions.
//
// The sums of a tile done whole lie with their weight row's thread; what finishes them (rotary pairs, gate and up, rows of y)
// wants four neighbouring units of a token in one thread, so a group of four warps turns 16 tokens at a time through shared memory.
template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GEMM_THREADS, 1)
gemm_split_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb0,
                  const __grid_constant__ CUtensorMap tb1, const __grid_constant__ CUtensorMap tb2, GemmArgs g, int Tpad) {
    const int tt = g.tt, half = tt / 2, stage_bytes = stage_bytes_of(tt), stages = ring_stages(tt);
    extern __shared__ unsigned char pf_smem_raw[];
    unsigned char *turn_smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(pf_smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *smem = turn_smem + TURN_BYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + stages * stage_bytes);      // in use in the first CTA: both CTAs' boxes have landed
    uint64_t *empty = full + MAX_STAGES;          // in both: the MMAs that read the stage have finished
    uint64_t *acc_full = empty + MAX_STAGES;      // [2], in both: a chunk's sum is complete in accumulator b
    uint64_t *acc_empty = acc_full + 2;           // [2], in use in the first CTA: both CTAs' epilogue warps have moved accumulator b's sum out
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 2);
    volatile int *cta_abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31, rank = blockIdx.x & 1;   // rank: of the pair
    const Jobs jobs(g);                                              // tiles: token tile fastest (tile = ty * tiles_x + tx)
    const int nkb = g.K / BK, nchunks = jobs.nchunks;
    constexpr int EPI_WARPS = GEMM_THREADS / 32 - 2;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * EPI_WARPS); }
        *cta_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    pair_sync();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ---- TMA producer: a stage is refilled once the MMAs that read it have finished ----
        const uint32_t one = elect_one(), arms = rank == 0 ? one : 0u;
        const uint32_t ring = smem_u32(smem), full_here = smem_u32(full), full_first = first_cta_addr(full);
        const int n_box = 128 / (EPI == PF_SWIGLU ? 64 : g.box);
        uint64_t w_policy, a_policy;
        // weights that a launch reads once (one token tile) go first when L2 needs room
        if (g.tiles_x == 1) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(w_policy));
        else asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(w_policy));
        asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(a_policy));
        // a job's weight rows: the map and the row in it of either box
        const CUtensorMap *w_map[2];
        int w_row[2], t0;
        auto locate = [&](int tile) {
            const int u0 = first_unit<EPI>(tile / g.tiles_x, rank);
            t0 = (tile % g.tiles_x) * tt + rank * half;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                w_map[r] = EPI == PF_SWIGLU && r ? &tb1 : &tb0;
                w_row[r] = EPI == PF_SWIGLU ? u0 : u0 + 64 * r;
                if (EPI != PF_SWIGLU && w_row[r] >= g.nA) {          // stacked matrices: the box lies in the second or third one
                    w_map[r] = &tb1; w_row[r] -= g.nA;
                    if (w_row[r] >= g.nB) { w_map[r] = &tb2; w_row[r] -= g.nB; }
                }
            }
        };
        auto load_w = [&](int kb, int s) {
            expect_tx_if(full_here + 8 * s, 2 * stage_bytes, arms);
            tma_load_pair(ring + s * stage_bytes, w_map[0], kb * BK, w_row[0], full_first + 8 * s, w_policy, one);
            if (n_box == 2) tma_load_pair(ring + s * stage_bytes + 64 * BK * 2, w_map[1], kb * BK, w_row[1], full_first + 8 * s, w_policy, one);
        };
        auto load_a = [&](int kb, int s) {
            tma_load_pair(ring + s * stage_bytes + W_BYTES, &ta, kb * BK, t0, full_first + 8 * s, a_policy, one);
            tma_load_pair(ring + s * stage_bytes + W_BYTES + half * BK * 2, &ta, kb * BK, Tpad + t0, full_first + 8 * s, a_policy, one);
        };
        int s = 0, ahead = 0, tile, c_begin, c_end;      // s, ph: the next k-block's stage and phase
        uint32_t ph = 0;
        bool ok = true;
        // the weights are there before the kernel before this one has finished: the first stages' go out at once
        if (jobs.get(0, tile, c_begin, c_end)) {
            locate(tile);
            ahead = min(stages, min(nkb, c_end * CHUNK_KB) - c_begin * CHUNK_KB);
            for (int k = 0; k < ahead; ++k) load_w(c_begin * CHUNK_KB + k, k);
            chain_wait();
            for (int k = 0; k < ahead; ++k) load_a(c_begin * CHUNK_KB + k, k);
            s = ahead == stages ? 0 : ahead;
            ph = ahead == stages;
        }
        for (int i = 0; ok && jobs.get(i, tile, c_begin, c_end); ++i) {
            locate(tile);
            const int kb1 = min(nkb, c_end * CHUNK_KB);
            for (int kb = c_begin * CHUNK_KB + (i == 0 ? ahead : 0); kb < kb1; ++kb) {
                ok = __all_sync(0xffffffffu, pf_wait(&empty[s], ph ^ 1u, cta_abort, g.err, 21));
                if (!ok) break;
                load_w(kb, s);
                load_a(kb, s);
                if (++s == stages) { s = 0; ph ^= 1u; }
            }
        }
        if (*cta_abort) {
            // Copies in flight land in this CTA's shared memory, counted by a barrier that the other CTA may not have armed:
            // they take microseconds, the CTA stays for some milliseconds (and the other one until this one is done).
            for (int k = 0; k < 5000; ++k) __nanosleep(1000);
        }
    } else if (warp == 1) {
        chain_wait();
        if (rank == 0) {
            // ---- MMA issue: chunk c goes to accumulator c & 1; per stage 4 k-steps of 16 columns, hi and lo term ----
            bool ok = true;
            const uint32_t one = elect_one(), idesc = umma_idesc(PAIR_UNITS, tt);
            const uint32_t ring = smem_u32(smem), empty_at = smem_u32(empty), acc_full_at = smem_u32(acc_full);
            int cg = 0, s = 0;               // chunks issued so far, over all of this pair's jobs; stage and phase of the next k-block
            uint32_t ph = 0;
            for (int i = 0, tile, c_begin, c_end; ok && jobs.get(i, tile, c_begin, c_end); ++i)
            for (int c = c_begin; c < c_end && ok; ++c, ++cg) {
                const int b = cg & 1;
                ok = __all_sync(0xffffffffu, pf_wait<true>(&acc_empty[b], ((uint32_t)(cg >> 1) & 1u) ^ 1u, cta_abort, g.err, 24));
                if (!ok) break;
                tc_fence_after();
                const uint32_t acc_addr = tmem + (uint32_t)(b * TT_MAX);
                const int kb1 = min(nkb, (c + 1) * CHUNK_KB);
                for (int kb = c * CHUNK_KB; kb < kb1; ++kb) {
                    ok = __all_sync(0xffffffffu, pf_wait<true>(&full[s], ph, cta_abort, g.err, 22));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t w = desc_lower(ring + s * stage_bytes), x_hi = w + (W_BYTES >> 4), x_lo = x_hi + (half * BK * 2 >> 4);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        umma_pair<true>(acc_addr, w + 2 * k, x_hi + 2 * k, idesc, kb != c * CHUNK_KB || k != 0, one);
                        umma_pair<false>(acc_addr, w + 2 * k, x_lo + 2 * k, idesc, 1u, one);
                    }
                    umma_commit_pair(empty_at + 8 * s, one);
                    if (++s == stages) { s = 0; ph ^= 1u; }
                }
                umma_commit_pair(acc_full_at + 8 * b, one);     // on the abort path too: it releases the epilogue warps' wait
            }
            if (!ok) { umma_commit_pair(acc_full_at, one); umma_commit_pair(acc_full_at + 8, one); }
        }
    } else {
        // ---- epilogue warps: warp w reads lanes 32 (w % 4) .. + 31 of tensor memory = this CTA's weight rows; the two groups of
        //      four warps split the tile's tokens.  acc[] = this thread's running sums over the chunks, token half * hsel + i ----
        chain_wait();
        const int q = warp & 3, hsel = (warp - 2) >> 2, row = 32 * q + lane, gt = (threadIdx.x - 64) & 127;
        const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16);
        float *turn = reinterpret_cast<float *>(turn_smem) + hsel * (2 * TURN_TOKENS * 128);
        float *scales = reinterpret_cast<float *>(turn_smem) + 2 * (2 * TURN_TOKENS * 128) + hsel * 128;
        const int f_tok = gt >> 4, f_j = 4 * (gt & 15);      // what this thread finishes: tokens f_tok and f_tok + 8 of 16, rows f_j ..
        bool ok = true;
        int cg = 0;                          // chunks taken so far, over all of this pair's jobs
        int tile, c_begin, c_end;
        for (int i = 0; jobs.get(i, tile, c_begin, c_end); ++i) {
            const int t0 = (tile % g.tiles_x) * tt + hsel * half;
            const bool piece = tile >= g.whole;
            float own_scale = 1.0f;          // of the group's token gt, fetched while the first chunk is under way
            if (EPI != PF_ADD && g.row_scale && !piece && gt < half && t0 + gt < g.T) own_scale = g.row_scale[t0 + gt];
            float acc[128];
#pragma unroll
            for (int e = 0; e < 128; ++e) acc[e] = 0.f;
            for (int c = c_begin; c < c_end && ok; ++c, ++cg) {
                const int b = cg & 1;
                // the loads from tensor memory are warp-wide: the warp goes on only if all of its threads saw the accumulator
                ok = __all_sync(0xffffffffu, pf_wait(&acc_full[b], (uint32_t)(cg >> 1) & 1u, cta_abort, g.err, 23) && !*cta_abort);
                if (!ok) break;
                tc_fence_after();
                // the last group of 32 columns may reach into the other half's (or past them, inside the accumulators)
#pragma unroll
                for (int gi = 0; gi < 4; ++gi) {
                    if (32 * gi >= half) continue;
                    float v[32];
                    tmem_ld32(trow + (uint32_t)(b * TT_MAX + hsel * half + 32 * gi), v);
                    if (piece) {                             // warp-uniform
                        float *dst = g.part + (((size_t)(tile - g.whole) * nchunks + c) * 2 + rank) * (tt * 128) + (size_t)(hsel * half + 32 * gi) * 128 + row;
                        const int live = min(half, g.T - t0) - 32 * gi;
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (e < live) __stcg(dst + e * 128, v[e]);
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e) acc[32 * gi + e] += v[e];
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) pair_arrive(first_cta_addr(&acc_empty[b]));
            }
            // a group's four warps go on together or not at all: they meet in what follows
            asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, %2, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                         : "=r"(c_begin) : "r"((uint32_t)ok), "r"(1 + hsel) : "memory");
            ok = c_begin != 0;
            if (!ok) break;
            if (piece) continue;             // fold_pieces_kernel goes on from here
            if (EPI != PF_ADD) scales[gt] = own_scale;       // the group is done with the job before
            const int u0 = first_unit<EPI>(tile / g.tiles_x, rank);
            float4 x[2][2];
            old_values<EPI>(g, u0, f_tok < half ? t0 + f_tok : g.T, f_j, x[0]);
            old_values<EPI>(g, u0, f_tok + 8 < half ? t0 + f_tok + 8 : g.T, f_j, x[1]);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int i0 = TURN_TOKENS * k;
                if (i0 >= half) break;       // uniform
                float *buf = turn + (k & 1) * (TURN_TOKENS * 128);
#pragma unroll
                for (int e = 0; e < TURN_TOKENS; ++e) buf[e * 128 + row] = acc[i0 + e];
                asm volatile("barrier.cta.sync %0, 128;" ::"r"(1 + hsel) : "memory");
                float4 next[2][2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int it = i0 + TURN_TOKENS + f_tok + 8 * e;
                    old_values<EPI>(g, u0, it < half ? t0 + it : g.T, f_j, next[e]);
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int tok = f_tok + 8 * e, t = t0 + i0 + tok;
                    if (i0 + tok < half && t < g.T) {
                        const float4 lo = *reinterpret_cast<const float4 *>(buf + tok * 128 + f_j), hi = *reinterpret_cast<const float4 *>(buf + tok * 128 + 64 + f_j);
                        float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                        finish_sums<EPI>(g, u0, t, f_j, v, x[e], EPI != PF_ADD ? scales[i0 + tok] : 1.0f);
                    }
                    x[e][0] = next[e][0];
                    x[e][1] = next[e][1];
                }
            }
        }                                    // next job: its first chunks are already accumulating in tensor memory
    }
    tc_fence_before();
    __syncwarp();
    __syncthreads();
    pair_sync();                             // neither CTA's barriers and tensor memory go away before the other is done with them
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// The tiles of a launch that were done in pieces: adds up the chunk sums of each, first chunk to last, and finishes them as
// gemm_split_kernel finishes a tile done whole.  grid = (2 ceil(tt / 16), tiles - whole), 256 threads: block x has 16 tokens of one CTA's
// 128 weight rows, a thread four rows and the four 64 further on of one token.  Bound by reading the sums back from L2, which
// all SMs share here.
template <int EPI>
__global__ void __launch_bounds__(256) fold_pieces_kernel(const GemmArgs g) {
    chain_wait();
    const int r = blockIdx.y, tile = g.whole + r, rank = blockIdx.x & 1, tok = 16 * (blockIdx.x >> 1) + (threadIdx.x >> 4), j = 4 * (threadIdx.x & 15);
    const int t = (tile % g.tiles_x) * g.tt + tok, u0 = first_unit<EPI>(tile / g.tiles_x, rank);
    if (t >= g.T || u0 >= g.N) return;
    const int nchunks = (g.K / BK + CHUNK_KB - 1) / CHUNK_KB;
    const size_t stride = (size_t)2 * g.tt * (128 / 4);      // between chunks, in float4s
    const float4 *src = reinterpret_cast<const float4 *>(g.part + (((size_t)r * nchunks * 2 + rank) * g.tt + tok) * 128 + j);
    float4 x[2];
    old_values<EPI>(g, u0, t, j, x);
    const float rs = EPI != PF_ADD && g.row_scale ? g.row_scale[t] : 1.0f;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = 0.f;
    constexpr int B = 8;                                     // chunks in flight: 8 KB a warp
    for (int c0 = 0; c0 < nchunks; c0 += B) {
        float4 p[B][2];
#pragma unroll
        for (int c = 0; c < B; ++c)
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (c0 + c < nchunks) p[c][e] = __ldcg(src + (size_t)(c0 + c) * stride + 16 * e);
#pragma unroll
        for (int c = 0; c < B; ++c)
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (c0 + c < nchunks) { v[4 * e] += p[c][e].x; v[4 * e + 1] += p[c][e].y; v[4 * e + 2] += p[c][e].z; v[4 * e + 3] += p[c][e].w; }
    }
    finish_sums<EPI>(g, u0, t, j, v, x, rs);
}

// ---------------------------------------------------------------------------------------------
// Row-wise kernels around the contractions
// ---------------------------------------------------------------------------------------------

// x[t][:] = embedding row of token t (bf16 -> fp32), eight values per thread and step (d is a multiple of 8).  grid = T.
__global__ void embed_rows_kernel(const bf16_t *__restrict__ table, const int *__restrict__ tok, int d, float *__restrict__ x) {
    chain_wait();
    const bf16_t *row = table + (size_t)tok[blockIdx.x] * d;
    float *xr = x + (size_t)blockIdx.x * d;
    for (int i = threadIdx.x * 8; i < d; i += blockDim.x * 8) {
        const uint4 w = __ldg(reinterpret_cast<const uint4 *>(row + i));
        const uint32_t p[4] = {w.x, w.y, w.z, w.w};
        float4 *dst = reinterpret_cast<float4 *>(xr + i);
        dst[0] = make_float4(__uint_as_float(p[0] << 16), __uint_as_float(p[0] & 0xFFFF0000u), __uint_as_float(p[1] << 16), __uint_as_float(p[1] & 0xFFFF0000u));
        dst[1] = make_float4(__uint_as_float(p[2] << 16), __uint_as_float(p[2] & 0xFFFF0000u), __uint_as_float(p[3] << 16), __uint_as_float(p[3] & 0xFFFF0000u));
    }
}

// RMSNorm of row t (gain g, epsilon eps) for the contraction that follows: the planes hold v = x g WITHOUT the row's
// scale, hi = bf16(v) and lo = bf16(v - hi), and rinv[t] = 1 / sqrt(mean(x^2) + eps) goes to the contraction's epilogue
// (a linear map commutes with a per-row scale).  Same operands as the decode passes use: values that are exact in two
// bf16 terms - embedding rows with unit gains - stay exact.  For the embedding rows only: the maps that add to the residual stream leave
// planes and squares of the rows they have changed, and scales_kernel does the rest.  grid = T, 256 threads.
__global__ void __launch_bounds__(256) norm_split_kernel(const float *__restrict__ x, int d, const float *__restrict__ gain, float eps,
                                                         bf16_t *__restrict__ hi, bf16_t *__restrict__ lo, float *__restrict__ rinv_out) {
    chain_wait();
    __shared__ float part[8];
    const float *xr = x + (size_t)blockIdx.x * d;
    bf16_t *hr = hi + (size_t)blockIdx.x * d, *lr = lo + (size_t)blockIdx.x * d;
    float ss = 0.f;
    // one walk over the row: the planes do not depend on the row's scale
    for (int i = threadIdx.x * 4; i < d; i += 1024) {
        const float4 v = *reinterpret_cast<const float4 *>(xr + i);
        const float4 g = *reinterpret_cast<const float4 *>(gain + i);
        ss += squares(v.x, v.y, v.z, v.w);
        uint32_t h[4], l[4];
        split_product(v.x, g.x, h[0], l[0]);
        split_product(v.y, g.y, h[1], l[1]);
        split_product(v.z, g.z, h[2], l[2]);
        split_product(v.w, g.w, h[3], l[3]);
        *reinterpret_cast<uint2 *>(hr + i) = make_uint2(pack_bf16(h[0], h[1]), pack_bf16(h[2], h[3]));
        *reinterpret_cast<uint2 *>(lr + i) = make_uint2(pack_bf16(l[0], l[1]), pack_bf16(l[2], l[3]));
    }
    const float rinv = scale_of_row(ss, part, d, eps);
    if (threadIdx.x == 0) rinv_out[blockIdx.x] = rinv;
}

// rinv[t] of a row whose squares a contraction has left four columns at a time.  The order of the sum is norm_split_kernel's.  Summed by
// 128 columns in the one epilogue and slot after slot in the next one, without this launch, a scale of 5120 columns had twice the error (1.0e-7 rms
// against 64 bits for 5.1e-8), and the epilogues of long prompts took longer than the launch does (4 layers of the 7B widths, 77 / 300 / 1024
// rows: 631 / 1251 / 2980 us so, 647 / 1209 / 2918 with it).  grid = T, 256 threads.
__global__ void __launch_bounds__(256) scales_kernel(const float *__restrict__ squares4, int d, float eps, float *__restrict__ rinv_out) {
    chain_wait();
    __shared__ float part[8];
    const float *sr = squares4 + (size_t)blockIdx.x * (d / 4);
    float ss = 0.f;
#pragma unroll 5
    for (int i = threadIdx.x; i < d / 4; i += 256) ss += __ldcg(sr + i);
    const float rinv = scale_of_row(ss, part, d, eps);
    if (threadIdx.x == 0) rinv_out[blockIdx.x] = rinv;
}

// (cos, sin) of the rotary angles of rows t = 0 .. T-1 at positions pos0 + t, once per chunk: all layers and heads
// use the same table.  grid = T, hd / 2 threads.
__global__ void rope_table_kernel(const double *__restrict__ inv_freq, int pos0, float2 *__restrict__ table) {
    chain_wait();
    double sn, cs;
    sincos((double)(pos0 + (int)blockIdx.x) * inv_freq[threadIdx.x], &sn, &cs);
    table[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = make_float2((float)cs, (float)sn);
}

// Rotary embedding of the q and k heads of row t at position pos0 + t (q in place, fp32); K and V rows rounded to
// bf16 into the cache.  grid = (T, ROPE_PARTS), 256 threads: a thread walks pairs (i, i + hd / 2) of the row's H + 2 Hkv head
// slots (in one part, 77 rows of the 13B width took 13 us: 30 steps of dependent latencies, in eight 4).
constexpr int ROPE_PARTS = 8;
__global__ void __launch_bounds__(256) rope_kv_rows_kernel(float *__restrict__ qkv, int H, int Hkv, int hd,
                                                           const float2 *__restrict__ table, bf16_t *__restrict__ kc,
                                                           bf16_t *__restrict__ vc, int max_seq, int pos0) {
    chain_wait();
    const int t = blockIdx.x, half = hd / 2, pos = pos0 + t;
    float *trow = qkv + (size_t)t * (H + 2 * Hkv) * hd;
    for (int idx = blockIdx.y * 256 + threadIdx.x; idx < (H + 2 * Hkv) * half; idx += 256 * ROPE_PARTS) {
        const int slot = idx / half, i = idx % half;
        float *row = trow + (size_t)slot * hd;
        float a = row[i], b = row[i + half];
        if (slot < H + Hkv) {
            rotate_pair(a, b, table[(size_t)t * half + i]);
            if (slot < H) {
                row[i] = a;
                row[i + half] = b;
            } else {
                bf16_t *dst = kc + ((size_t)(slot - H) * max_seq + pos) * hd;
                dst[i] = float_to_bf16_rne(a);
                dst[i + half] = float_to_bf16_rne(b);
            }
        } else {
            bf16_t *dst = vc + ((size_t)(slot - H - Hkv) * max_seq + pos) * hd;
            dst[i] = float_to_bf16_rne(a);
            dst[i + half] = float_to_bf16_rne(b);
        }
    }
}

// y[t][n] = hi[t][n] + lo[t][n] (the value a pair of planes stands for).  grid = T.
__global__ void join_planes_kernel(const bf16_t *__restrict__ hi, const bf16_t *__restrict__ lo, int n, float *__restrict__ y) {
    const size_t base = (size_t)blockIdx.x * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) y[base + i] = bf16_bits_to_float(hi[base + i]) + bf16_bits_to_float(lo[base + i]);
}
// The two planes of plain fp32 rows (no norm).  grid = T.
__global__ void split_rows_kernel(const float *__restrict__ x, int n, bf16_t *__restrict__ hi, bf16_t *__restrict__ lo) {
    const size_t base = (size_t)blockIdx.x * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float v = x[base + i];
        const uint32_t h = float_to_bf16_rne(v);
        hi[base + i] = (bf16_t)h;
        lo[base + i] = float_to_bf16_rne(v - __uint_as_float(h << 16));
    }
}

// ---------------------------------------------------------------------------------------------
// Causal attention over the prompt
// ---------------------------------------------------------------------------------------------

// One CTA of four warps per (head, block of 64 consecutive prompt rows), one warp per 16 of the rows.  The CTA walks
// the positions 0 .. (its last row's position) in segments of 64: the segment's K and V rows (bf16, as cached; this
// chunk's rows are in the cache already) are brought into shared memory with 16-byte asynchronous copies, two segments
// in flight, and are read from there by all four warps with `ldmatrix` - every cached row crosses the L2 -> SM path
// once per 64 query rows.  A shared-memory row keeps its 16-byte pieces at (piece ^ (row & 7)), so the eight rows of
// an `ldmatrix` matrix fall into distinct banks.  Rows past the block's last position are filled with zeros.
//
// Arithmetic per warp: q (rotated fp32) is split into hi + lo bf16 once and stays in registers as the 16-row operand
// of m16n8k16; scores = q . K^T with the lo term added before the hi term at every k-step; the softmax of a row is a
// running maximum and sum over the segments (it differs from the softmax over all positions at once by rounding
// only); the probabilities are split into hi + lo bf16 in registers (the accumulator layout of two position tiles is
// the operand layout of one k-step) and o += p . V with V read through `ldmatrix.trans`.  fp32 accumulation.
// The exponentials are exp2 of scores scaled by log2(e) / sqrt(HD) (`ex2.approx`, 2 ulp), the bf16 splits use the
// hardware's round-to-nearest-even pair conversion.
// grid = (H, ceil(T / 64)), 128 threads, attn_smem_bytes<HD>() of dynamic shared memory; the last row blocks (longest
// walks) of all heads are scheduled first.
constexpr int ATTN_SEG = 64;
template <int HD> constexpr int attn_smem_bytes() { return 2 * 2 * ATTN_SEG * HD * 2; }      // 2 stages x (K, V)

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
    const int n = valid ? 16 : 0;                           // 0 bytes read: the 16 bytes are filled with zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t &a0, uint32_t &a1, uint32_t &a2, uint32_t &a3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(a0), "=r"(a1), "=r"(a2), "=r"(a3) : "r"(addr));
}

// c += a . b (m16n8k16, bf16 operands, fp32 accumulation); a pure function of its registers, free to be scheduled
__device__ __forceinline__ void mma_acc(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int HD>
__global__ void __launch_bounds__(128, 2) attn_prompt_kernel(const float *__restrict__ qkv, int H, int Hkv, const bf16_t *__restrict__ kc,
                                                             const bf16_t *__restrict__ vc, int max_seq, int pos0, int T,
                                                             bf16_t *__restrict__ out_hi, bf16_t *__restrict__ out_lo) {
    chain_wait();
    constexpr int SEG = ATTN_SEG, NT = SEG / 8, KS = HD / 16, VJ = HD / 8, KP = SEG / 16, RB = 64;
    constexpr int CH = HD / 8;                               // 16-byte pieces per row
    constexpr int TILE = SEG * HD * 2;                       // bytes of one K (or V) segment
    extern __shared__ __align__(128) unsigned char attn_smem[];
    const uint32_t sm0 = stream::smem_u32(attn_smem);        // stage st: K at sm0 + st * 2 TILE, V one TILE further
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g8 = lane >> 2, t4 = lane & 3;
    const int h = blockIdx.x;
    const int rb = gridDim.y - 1 - blockIdx.y;               // all heads' longest walks first, the short ones fill the tail
    const int t_first = rb * RB;
    const int p_last = pos0 + min(t_first + RB - 1, T - 1);  // the block's last position
    const int n_seg = p_last / SEG + 1;
    const int kvh = h / (H / Hkv);
    const int qstride = (H + 2 * Hkv) * HD;
    const bf16_t *kbase = kc + (size_t)kvh * max_seq * HD, *vbase = vc + (size_t)kvh * max_seq * HD;
    const float scale = 1.4426950408889634f / sqrtf((float)HD);      // scores in units of log 2: p = 2^(s - max)

    auto load_segment = [&](int seg) {
        const uint32_t kdst = sm0 + (uint32_t)(seg & 1) * 2 * TILE, vdst = kdst + TILE;
        for (int i = threadIdx.x; i < SEG * CH; i += 128) {
            const int r = i / CH, c = i % CH, p = seg * SEG + r;
            const bool ok = p <= p_last;
            const size_t off = (size_t)(ok ? p : 0) * HD + 8 * c;
            const uint32_t d = (uint32_t)(r * HD * 2 + ((c ^ (r & 7)) << 4));
            cp_async16(kdst + d, kbase + off, ok);
            cp_async16(vdst + d, vbase + off, ok);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load_segment(0);

    // ---- this warp's rows: g8 and g8 + 8 of its 16 ----
    const int w_first = t_first + 16 * warp;
    const bool warp_live = w_first < T;
    const int wp_last = pos0 + min(w_first + 15, T - 1);     // the warp's last position
    int t_row[2], p_row[2];
    bool live[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) { t_row[r] = w_first + g8 + 8 * r; live[r] = t_row[r] < T; p_row[r] = pos0 + t_row[r]; }

    // q as operand registers: k-step ks covers dimensions 16 ks .. 16 ks + 15; [0] row g8, dims 2 t4 + {0, 1};
    // [1] row g8 + 8; [2], [3] the same rows, dims + 8
    uint32_t qh[KS][4], ql[KS][4];
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = i & 1, dim = 16 * ks + 2 * t4 + 8 * (i >> 1);
            float2 v = make_float2(0.f, 0.f);
            if (live[r]) v = *reinterpret_cast<const float2 *>(qkv + (size_t)t_row[r] * qstride + (size_t)h * HD + dim);
            split_pair(v.x, v.y, qh[ks][i], ql[ks][i]);
        }

    float o[VJ][4];
#pragma unroll
    for (int j = 0; j < VJ; ++j) { o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f; }
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};   // l_run: this lane's share of the row's sum

    // ldmatrix sources of this lane.  K (plain): matrix lane / 8 = 16-byte piece (lane / 8) of the two k-steps, row
    // lane % 8 of the position tile.  V (transposed): matrices 0, 1 = positions 0-7, 8-15 of the k-step, piece j;
    // 2, 3 = the same positions, piece j + 1.
    const int k_row = lane & 7, k_piece = lane >> 3;
    const int v_row = (lane & 7) + ((lane >> 3) & 1) * 8, v_piece = lane >> 4;

    for (int seg = 0; seg < n_seg; ++seg) {
        if (seg + 1 < n_seg) {
            load_segment(seg + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const int p_begin = seg * SEG;
        if (warp_live && p_begin <= wp_last) {
            const uint32_t ks0 = sm0 + (uint32_t)(seg & 1) * 2 * TILE, vs0 = ks0 + TILE;
            // ---- scores of rows (g8: [0], [1]; g8 + 8: [2], [3]) x positions 8 nt + 2 t4 + {0, 1} ----
            // Four position tiles at a time: their products are independent, so the tensor pipe always has one to start.
            float sc[NT][4];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) { sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f; }
#pragma unroll
            for (int n0 = 0; n0 < NT; n0 += 4)
#pragma unroll
                for (int kk = 0; kk < KS; kk += 2) {
                    uint32_t b[4][4];                        // per tile: (b[0], b[1]) k-step kk; (b[2], b[3]) k-step kk + 1
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int r = 8 * (n0 + i) + k_row;
                        stream::ldmatrix_x4(ks0 + (uint32_t)(r * HD * 2) + (uint32_t)(((2 * kk + k_piece) ^ (r & 7)) << 4), b[i][0], b[i][1],
                                            b[i][2], b[i][3]);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma_acc(sc[n0 + i], ql[kk], b[i][0], b[i][1]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma_acc(sc[n0 + i], qh[kk], b[i][0], b[i][1]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma_acc(sc[n0 + i], ql[kk + 1], b[i][2], b[i][3]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma_acc(sc[n0 + i], qh[kk + 1], b[i][2], b[i][3]);
                }
            // ---- running softmax per row: new maximum, old sums and outputs rescaled ----
            const bool diagonal = p_begin + SEG - 1 > pos0 + w_first;      // some (row, position) of the tile is masked
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float mx = -INFINITY;
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int p = p_begin + 8 * nt + 2 * t4 + e;
                        float &v = sc[nt][2 * r + e];
                        v = (!diagonal || (live[r] && p <= p_row[r])) ? v * scale : -INFINITY;
                        mx = fmaxf(mx, v);
                    }
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                const float m_new = fmaxf(m_run[r], mx);
                const float f = m_run[r] == -INFINITY ? 0.f : exp2f(m_run[r] - m_new);
                m_run[r] = m_new;
                l_run[r] *= f;
                const float m_sub = m_new == -INFINITY ? 0.f : m_new;      // a row with nothing to see yet: 2^(-inf) = 0
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float &v = sc[nt][2 * r + e];
                        v = exp2f(v - m_sub);
                        l_run[r] += v;
                    }
#pragma unroll
                for (int j = 0; j < VJ; ++j) { o[j][2 * r] *= f; o[j][2 * r + 1] *= f; }
            }
            // ---- o += p V, 16 positions per k-step ----
#pragma unroll
            for (int kp = 0; kp < KP; ++kp) {
                uint32_t ah[4], al[4];     // [0], [1]: rows g8, g8 + 8, positions 16 kp + 2 t4 + {0, 1}; [2], [3]: positions + 8
#pragma unroll
                for (int i = 0; i < 4; ++i) split_pair(sc[2 * kp + (i >> 1)][2 * (i & 1)], sc[2 * kp + (i >> 1)][2 * (i & 1) + 1], ah[i], al[i]);
                const int r = 16 * kp + v_row;
                const uint32_t rowaddr = vs0 + (uint32_t)(r * HD * 2);
#pragma unroll
                for (int j = 0; j < VJ; j += 4) {
                    uint32_t b[4][2];                        // dimension tiles j .. j + 3
                    ldmatrix_x4_trans(rowaddr + (uint32_t)(((j + v_piece) ^ (r & 7)) << 4), b[0][0], b[0][1], b[1][0], b[1][1]);
                    ldmatrix_x4_trans(rowaddr + (uint32_t)(((j + 2 + v_piece) ^ (r & 7)) << 4), b[2][0], b[2][1], b[3][0], b[3][1]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma_acc(o[j + i], al, b[i][0], b[i][1]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma_acc(o[j + i], ah, b[i][0], b[i][1]);
                }
            }
        }
        __syncthreads();                                     // the stage is refilled by the next round's copies
    }

    // ---- rows g8 ([0], [1]) and g8 + 8 ([2], [3]) x dimensions 8 j + 2 t4 + {0, 1}, divided by the row's sum ----
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        float l = l_run[r];
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        if (!live[r]) continue;
        const size_t base = (size_t)t_row[r] * ((size_t)H * HD) + (size_t)h * HD + 2 * t4;
#pragma unroll
        for (int j = 0; j < VJ; ++j) {
            uint32_t hw, lw;
            split_pair(o[j][2 * r] / l, o[j][2 * r + 1] / l, hw, lw);
            *reinterpret_cast<uint32_t *>(out_hi + base + 8 * j) = hw;
            *reinterpret_cast<uint32_t *>(out_lo + base + 8 * j) = lw;
        }
    }
}

}  // namespace prefill
}  // namespace knnssd
