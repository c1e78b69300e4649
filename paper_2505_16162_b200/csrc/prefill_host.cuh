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
        cudaFuncSetAttribute(gemm_split_kernel<PF_STORE>, cudaFuncAttributeMaxDynamicSharedMemorySize, RING_BYTES + 1280) == cudaSuccess &&
        cudaFuncSetAttribute(gemm_split_kernel<PF_ADD>, cudaFuncAttributeMaxDynamicSharedMemorySize, RING_BYTES + 1280) == cudaSuccess &&
        cudaFuncSetAttribute(gemm_split_kernel<PF_SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, RING_BYTES + 1280) == cudaSuccess &&
        cudaFuncSetAttribute(gemm_split_kernel<PF_QKV>, cudaFuncAttributeMaxDynamicSharedMemorySize, RING_BYTES + 1280) == cudaSuccess &&
        cudaFuncSetAttribute(attn_prompt_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, attn_smem_bytes<128>()) == cudaSuccess &&
        cudaFuncSetAttribute(attn_prompt_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, attn_smem_bytes<64>()) == cudaSuccess;
    done[dev] = ok;
    return ok;
}

// Most chunk sums a launch may leave in the scratch of the pieces: PIECE_FLOATS each, 72 MB in all of the 126 MB of L2, which they
// have to stay in to be worth it while weights and activations pass through it.
constexpr int MAX_PIECES = 576;

// Columns per tile, CTAs, how many tiles are done whole (the rest in pieces), and the chunk sums that the pieces leave.
struct Deal { int bn, grid, whole, sums; };

// The cheapest of 128, 192 and 256 columns, tiles all whole or the last, incomplete round of them in pieces, by times measured
// on the 13B widths (5120 / 13824 columns in, 77 .. 1024 rows):
//   whole tiles: 8 us + rounds x k-blocks x 0.5 / 0.62 / 0.73 us - the products of a k-block take that long (both terms'
//     operands leave shared memory at ~64 bytes per clock), copies and sums run under them.  5120 units x 1024 rows, 256
//     columns: two rounds 144 us, of which the second has 12 tiles.
//   pieces: 14 us for a launch, the fold behind it and the last sums, 1.3 x the products' time (pieces are not in step, so they share
//     less through L2), and per chunk sum 0.012 us + 0.036 us per 128 KB to write and read it.  The same launch: one
//     round + 12 tiles in 120 pieces, 93 us; at 77 rows, 27 tiles in 270 pieces 29 us against 63 us.
// Sums of a layer's four maps on other widths, measured launch by launch (modelled), us at 77 / 300 / 512 / 1024 rows: 7B 163 (179), 316
// (290), 395 (383), 642 (578); 13B 213 (225), 432 (434), 548 (508), 934 (883); Qwen 14B 192 (202), 399 (390), 480 (449).
// `heads`: 256 columns let the launch finish the heads itself; else a kernel of its own does.
inline Deal deal_out(int T, int N, int K, bool swiglu, bool heads, int n_sms) {
    const int row_tiles = (T + BM - 1) / BM, nkb = K / BK, nchunks = (nkb + CHUNK_KB - 1) / CHUNK_KB;
    Deal best{0, 0, 0, 0};
    double best_us = 0.0;
    for (int bn = 128; bn <= BN_MAX; bn += 64) {
        if (swiglu && bn % 128) continue;
        const int per = swiglu ? bn / 2 : bn;
        const long long tiles = (long long)row_tiles * ((N + per - 1) / per), last_round = tiles % n_sms, units = last_round * nchunks;
        const double kb_us = bn == 256 ? 0.73 : bn == 192 ? 0.62 : 0.5, heads_us = heads && bn != 256 ? 12.0 + T * 0.02 : 0.0;
        const double round_us = nkb * kb_us;
        for (int pieces = 0; pieces < 2; ++pieces) {
            Deal d{bn, (int)(tiles < n_sms ? tiles : n_sms), (int)tiles, 0};
            double us = heads_us + 8.0 + (double)((tiles + n_sms - 1) / n_sms) * round_us;
            if (pieces) {
                if (last_round == 0 || units > MAX_PIECES) continue;
                d.whole = (int)(tiles - last_round);
                d.sums = (int)units;
                d.grid = d.whole == 0 && units < n_sms ? (int)units : n_sms;
                const long long most = (units + d.grid - 1) / d.grid;
                us = heads_us + 14.0 + (double)(d.whole / n_sms) * round_us + most * 1.3 * CHUNK_KB * kb_us +
                     units * (0.012 + 0.036 * (T < BM ? T : BM) * bn / (double)PIECE_FLOATS);
            }
            if (!best.bn || us <= best_us) { best = d; best_us = us; }
        }
    }
    return best;
}

// Rows of an activation box: a tile's worth, or what a launch of fewer rows needs (the rows a box leaves out of a tile hold
// whatever the stage held before; they meet no live row).
inline int act_box_rows(int T) { return T >= BM ? BM : (T + 7) / 8 * 8; }

// Whether a stacked q / k / v launch may finish the heads in its epilogue (it does at 256 columns).
inline bool heads_in_epilogue(int head_dim, int nA, int nB, int N) { return head_dim == 128 && nA % 128 == 0 && nB % 128 == 0 && N % 128 == 0; }

// Most chunk sums that any launch of a prompt pass over up to `cap` rows leaves: what its scratch has to hold.
inline int most_sums(int cap, int d, int nq, int nkv, int d_ff, int head_dim, int n_sms) {
    const int ldq = nq + 2 * nkv;
    const bool heads = heads_in_epilogue(head_dim, nq, nkv, ldq);
    int most = 0;
    for (int T = 1; T <= cap; ++T) {
        const int sums[] = {deal_out(T, ldq, d, false, heads, n_sms).sums, deal_out(T, d, nq, false, false, n_sms).sums,
                            deal_out(T, d_ff, d, true, false, n_sms).sums, deal_out(T, d, d_ff, false, false, n_sms).sums};
        for (int n : sums)
            if (n > most) most = n;
    }
    return most;
}

// One contraction over T rows.  `planes` = the activation map (hi rows [0, cap), lo rows [cap, 2 cap)); W0 (and W1 for
// SwiGLU: W0 = gate, W1 = up) are [N][K] bf16.  STORE with W1 and W2 given: the three matrices (nA, nB and nC rows, all
// multiples of BOX_N) are stacked along the output units, N = nA + nB + nC, one launch for q, k and v.
// `part`: scratch of PIECE_FLOATS for every chunk sum that deal_out gives the launch.  Returns the number of kernels launched, 0 if a tensor map could not be made.
// What the q / k / v launch needs to finish the heads in its epilogue (rotary embedding, K / V rows into the cache).
struct QkvFuse {
    const float2 *rope;    // [T][64]
    bf16_t *kc, *vc;
    int max_seq, pos0, head_dim;
};

// `fuse` (stacked q, k, v only): if the head dimension is 128 and the launch takes 256-column tiles, the epilogue does
// the rotary embedding and writes K / V to the cache itself; *fused says whether it did (otherwise the caller runs
// rope_kv_rows_kernel on y).
inline int launch_gemm(const CUtensorMap &planes, float *part, int cap, const void *W0, const void *W1, int N, int K, int T, int epi, float *y,
                        int ldy, int col0, bf16_t *out_hi, bf16_t *out_lo, int ldo, int *err, int n_sms, cudaStream_t s,
                        const void *W2 = nullptr, int nA = 0, int nB = 0, const QkvFuse *fuse = nullptr, bool *fused = nullptr,
                        const float *row_scale = nullptr) {
    if (fused) *fused = false;
    if (!gemm_attrs_once()) return 0;
    const bool stacked = epi == PF_STORE && W1 && W2;
    const bool heads = stacked && fuse && heads_in_epilogue(fuse->head_dim, nA, nB, N);
    const Deal deal = deal_out(T, N, K, epi == PF_SWIGLU, heads, n_sms);
    const int bn = deal.bn;
    const int per = epi == PF_SWIGLU ? bn / 2 : bn;
    const int box = per % 128 == 0 && (!stacked || (nA % 128 == 0 && nB % 128 == 0)) ? 128 : BOX_N;
    CUtensorMap tb0, tb1, tb2;
    if (!make_map(&tb0, W0, (size_t)(stacked ? nA : N), (size_t)K, box)) return 0;
    if (epi == PF_SWIGLU) {
        if (!make_map(&tb1, W1, (size_t)N, (size_t)K, box)) return 0;
        tb2 = tb1;
    } else if (stacked) {
        if (!make_map(&tb1, W1, (size_t)nB, (size_t)K, box) || !make_map(&tb2, W2, (size_t)(N - nA - nB), (size_t)K, box)) return 0;
    } else {
        tb1 = tb0;
        tb2 = tb0;
    }
    const int tiles_x = (T + BM - 1) / BM, tiles_y = (N + per - 1) / per;
    GemmArgs g{T, K, N, bn, y, ldy, col0, out_hi, out_lo, ldo, err, tiles_x, tiles_y, box, act_box_rows(T), deal.whole, part, stacked ? nA : N, stacked ? nB : 0, row_scale, nullptr, nullptr, nullptr, 0, 0};
    const dim3 grid(deal.grid);
    const int smem = gemm_smem(g.a_rows, bn);
    const int pieces = tiles_x * tiles_y - deal.whole;
    auto run = [&](auto *contract, auto *fold) {
        launch_chained(contract, grid, dim3(GEMM_THREADS), smem, s, planes, tb0, tb1, tb2, g, cap);
        if (pieces) launch_chained(fold, dim3(8 * pieces), dim3(256), 0, s, g);
    };
    if (heads && bn == 256) {
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
