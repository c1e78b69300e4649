// Host side of the tensor-core prompt pass: TMA tensor maps and the launches of prefill.cuh's kernels.
#pragma once

#include "prefill.cuh"

#include <cuda_runtime.h>

namespace knnssd {
namespace prefill {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up through the runtime (the library does not link against the driver).
inline EncodeTiledFn encode_tiled_fn() {
    static const EncodeTiledFn fn = [] {                 // once, and for all threads that come meanwhile
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        const bool found = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess;
        return found ? reinterpret_cast<EncodeTiledFn>(p) : nullptr;
    }();
    return fn;
}

// Map of a row-major bf16 matrix [rows][cols] (cols a multiple of 64) read in boxes of box_rows rows x 64 columns,
// 128-byte swizzle; rows past the end read as zero.
inline bool make_map(CUtensorMap *m, const void *base, size_t rows, size_t cols, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The contraction kernels need more dynamic shared memory than the default limit; the attribute belongs to the
// current device, so it is set once per device (one process may drive several GPUs).
inline bool gemm_attrs_once() {
    static bool done[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (done[dev]) return true;
    const bool ok =
        cudaFuncSetAttribute(gemm_split_kernel<PF_STORE>, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM_MAX) == cudaSuccess &&
        cudaFuncSetAttribute(gemm_split_kernel<PF_ADD>, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM_MAX) == cudaSuccess &&
        cudaFuncSetAttribute(gemm_split_kernel<PF_SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM_MAX) == cudaSuccess &&
        cudaFuncSetAttribute(gemm_split_kernel<PF_QKV>, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM_MAX) == cudaSuccess &&
        cudaFuncSetAttribute(attn_prompt_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, attn_smem_bytes<128>()) == cudaSuccess &&
        cudaFuncSetAttribute(attn_prompt_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, attn_smem_bytes<64>()) == cudaSuccess;
    done[dev] = ok;
    return ok;
}

// Most floats of chunk sums a launch may leave in the scratch of the pieces: 72 MB of the 126 MB of L2, which they have to stay in to be
// worth it while weights and activations pass through it.
constexpr size_t MAX_SUMS = (size_t)18 << 20;

// Tokens per tile, pairs of CTAs, how many tiles are done whole (the rest in pieces), and the floats of chunk sums that the pieces leave.
struct Deal { int tt, pairs, whole; size_t sums; };

// The cheapest split of T rows into token tiles, tiles all whole or the last, incomplete round of them in pieces, by times measured
// on the 7B, 13B and Qwen 14B widths at 20 .. 1024 rows (689 launches; the choice is within 0.4 % of the best one on average,
// 13 % at worst):
//   a k-block of a tile: 0.28 + 0.0016 tt us where the copies bound it (0.41 at 96 tokens), 0.0034 tt us where the products do (0.6 .. 0.75 at
//     192, 0.72 .. 0.85 at 256: the tensor pipe at the clock that the power limit leaves); not less than the weights' bytes at 5.6 TB/s;
//   whole tiles: 7 us + rounds.  4096 x 4096 at 512 rows: 64 tiles of 128 tokens 38 us, 32 of 256 62 us.
//   pieces: 12 us for the launch and the fold behind it, and 0.2 us per MB of chunk sums.  4096 x 11008 at 77 rows: 352 pieces of 16 tiles
//     30 us, the tiles whole 56 us; at 512 rows, 256 tokens: 51 MB of sums, 146 us against 168 (128 tokens, whole: 142).
inline Deal deal_out(int T, int N, int K, bool swiglu, int n_sms) {
    const int nkb = K / BK, nchunks = (nkb + CHUNK_KB - 1) / CHUNK_KB, pairs = n_sms / 2;
    const int tiles_y = (N + (swiglu ? PAIR_UNITS / 2 : PAIR_UNITS) - 1) / (swiglu ? PAIR_UNITS / 2 : PAIR_UNITS);
    const double weights_us = (swiglu ? 4.0 : 2.0) * N * K / 5.6e6;
    Deal best{0, 0, 0, 0};
    double best_us = 0.0;
    for (int tx = (T + TT_MAX - 1) / TT_MAX, last_tt = 0; tx <= (T + TT_STEP - 1) / TT_STEP; ++tx) {
        const int tt = ((T + tx - 1) / tx + TT_STEP - 1) / TT_STEP * TT_STEP;
        if (tt == last_tt) continue;
        last_tt = tt;
        const long long tiles = (long long)((T + tt - 1) / tt) * tiles_y, last_round = tiles % pairs, units = last_round * nchunks;
        const double copy_us = 0.28 + 0.0016 * tt, mma_us = 0.0034 * tt, kb_us = mma_us > copy_us ? mma_us : copy_us;
        for (int pieces = 0; pieces < 2; ++pieces) {
            Deal d{tt, (int)(tiles < pairs ? tiles : pairs), (int)tiles, 0};
            double fixed_us = 7.0, us = (double)((tiles + pairs - 1) / pairs) * nkb * kb_us;
            if (pieces) {
                d.sums = (size_t)units * PAIR_UNITS * tt;
                if (last_round == 0 || d.sums > MAX_SUMS) continue;
                d.whole = (int)(tiles - last_round);
                d.pairs = d.whole == 0 && units < pairs ? (int)units : pairs;
                us = (double)((d.whole / pairs) * nkb + (units + d.pairs - 1) / d.pairs * CHUNK_KB) * kb_us;
                fixed_us = 12.0 + 0.8e-6 * units * PAIR_UNITS * (T < tt ? T : tt);
            }
            us = fixed_us + (us > weights_us ? us : weights_us);
            if (!best.tt || us <= best_us) { best = d; best_us = us; }
        }
    }
    return best;
}

// Whether a stacked q / k / v launch finishes the heads in its epilogue (a CTA's 128 weight rows are one head).
inline bool heads_in_epilogue(int head_dim, int nA, int nB, int N) { return head_dim == 128 && nA % 128 == 0 && nB % 128 == 0 && N % 128 == 0; }

// At least the floats of chunk sums that any launch of a prompt pass over up to `cap` rows leaves: what its scratch has to hold.  (Going
// through deal_out for every row count took a session's first call 25 ms.)
inline size_t most_sums(int cap, int d, int nq, int nkv, int d_ff, int n_sms) {
    const int units[] = {nq + 2 * nkv, d, 2 * d_ff, d}, width[] = {d, nq, d, d_ff};      // gate and up rows share a tile
    size_t most = 0;
    for (int i = 0; i < 4; ++i)
        for (int tt = TT_STEP; tt <= TT_MAX && tt < cap + TT_STEP; tt += TT_STEP) {
            const size_t tiles = (size_t)((cap + tt - 1) / tt) * ((units[i] + PAIR_UNITS - 1) / PAIR_UNITS), pairs = n_sms / 2;
            const size_t sums = (tiles < pairs ? tiles : pairs - 1) * ((width[i] / BK + CHUNK_KB - 1) / CHUNK_KB) * PAIR_UNITS * tt;
            if (sums > most) most = sums;
        }
    return most < MAX_SUMS ? most : MAX_SUMS;
}

// What the q / k / v launch needs to finish the heads in its epilogue (rotary embedding, K / V rows into the cache).
struct QkvFuse {
    const float2 *rope;    // [T][64]
    bf16_t *kc, *vc;
    int max_seq, pos0, head_dim;
};

// RMSNorms around a contraction: the scales of the rows it reads; gain, planes and squares of the rows it has added to (GemmArgs).
struct Norms {
    const float *row_scale = nullptr;
    const float *next_gain = nullptr;
    bf16_t *next_hi = nullptr, *next_lo = nullptr;
    float *ss_out = nullptr;
};

// One contraction over T rows, dealt out as `deal` says.  `planes` = the activations' planes [2][cap][K], 16-byte aligned; W0 (and W1 for
// SwiGLU: W0 = gate, W1 = up) are [N][K] bf16.  STORE with W1 and W2 given: the three matrices (nA, nB and nC rows, all
// multiples of BOX_N) are stacked along the output units, N = nA + nB + nC, one launch for q, k and v.
// `part`: room for deal.sums floats.  Returns the number of kernels launched, 0 if a tensor map could not be made.
// `fuse` (stacked q, k, v only): if the head dimension is 128 the epilogue does the rotary embedding and writes K / V to the
// cache itself; *fused says whether it did (otherwise the caller runs rope_kv_rows_kernel on y).
inline int launch_gemm(const Deal &deal, const bf16_t *planes, float *part, int cap, const void *W0, const void *W1, int N, int K, int T, int epi, float *y,
                        int ldy, int col0, bf16_t *out_hi, bf16_t *out_lo, int ldo, int *err, cudaStream_t s,
                        const void *W2 = nullptr, int nA = 0, int nB = 0, const QkvFuse *fuse = nullptr, bool *fused = nullptr,
                        const Norms &norms = Norms()) {
    if (fused) *fused = false;
    if (!gemm_attrs_once()) return 0;
    const bool stacked = epi == PF_STORE && W1 && W2;
    const bool heads = stacked && fuse && heads_in_epilogue(fuse->head_dim, nA, nB, N);
    const int box = epi != PF_SWIGLU && (!stacked || (nA % 128 == 0 && nB % 128 == 0)) ? 128 : BOX_N;
    CUtensorMap ta, tb0, tb1, tb2;
    if (!make_map(&ta, planes, 2 * (size_t)cap, (size_t)K, deal.tt / 2) || !make_map(&tb0, W0, (size_t)(stacked ? nA : N), (size_t)K, box)) return 0;
    tb1 = tb2 = tb0;
    if (epi == PF_SWIGLU && !make_map(&tb1, W1, (size_t)N, (size_t)K, box)) return 0;
    if (stacked && (!make_map(&tb1, W1, (size_t)nB, (size_t)K, box) || !make_map(&tb2, W2, (size_t)(N - nA - nB), (size_t)K, box))) return 0;
    const int per = epi == PF_SWIGLU ? PAIR_UNITS / 2 : PAIR_UNITS;
    const int tiles_x = (T + deal.tt - 1) / deal.tt, tiles_y = (N + per - 1) / per, pieces = tiles_x * tiles_y - deal.whole;
    GemmArgs g{T, K, N, deal.tt, y, ldy, col0, out_hi, out_lo, ldo, err, tiles_x, tiles_y, box, deal.whole, part, stacked ? nA : N, stacked ? nB : 0, norms.row_scale, norms.next_gain, norms.next_hi, norms.next_lo, norms.ss_out, nullptr, nullptr, nullptr, 0, 0};
    auto run = [&](auto *contract, auto *fold) {
        launch_chained(contract, dim3(2 * deal.pairs), dim3(GEMM_THREADS), gemm_smem(deal.tt), s, ta, tb0, tb1, tb2, g, cap);
        if (pieces) launch_chained(fold, dim3(2 * (deal.tt / 16), pieces), dim3(256), 0, s, g);
    };
    if (heads) {
        g.rope = fuse->rope; g.kc = fuse->kc; g.vc = fuse->vc; g.max_seq = fuse->max_seq; g.pos0 = fuse->pos0;
        run(gemm_split_kernel<PF_QKV>, fold_pieces_kernel<PF_QKV>);
        if (fused) *fused = true;
    } else if (epi == PF_STORE) run(gemm_split_kernel<PF_STORE>, fold_pieces_kernel<PF_STORE>);
    else if (epi == PF_ADD) run(gemm_split_kernel<PF_ADD>, fold_pieces_kernel<PF_ADD>);
    else run(gemm_split_kernel<PF_SWIGLU>, fold_pieces_kernel<PF_SWIGLU>);
    return pieces ? 2 : 1;
}

}  // namespace prefill
}  // namespace knnssd
