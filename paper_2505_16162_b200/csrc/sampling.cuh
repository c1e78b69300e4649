// Stochastic speculative sampling on the logits of the draft and verification passes (sm_100a).
//
// The paper's set-up lists temperature 0.2 and top-p 0.85 (App. C.1) and the method is to leave the distribution of
// the generated tokens unchanged (Sec. 1, Sec. 3.1); it prints no acceptance rule for the sampled case.  The rule
// used is the one of speculative sampling with that property: p and q are the full and the draft model's next-token
// distributions after temperature and nucleus filtering; a draft d ~ q is kept with probability min(1, p(d) / q(d));
// at the first rejection the token is drawn from the normalised positive part of p - q; if every draft is kept one
// more token is drawn from p.  Random numbers are inputs (one uniform per draw), consumed through the inverse CDF in
// token-id order, so that the choices are reproducible.
//
// A row is the work of a cluster of eight blocks, each with a contiguous eighth of the ids, or, where the filter has a long row, of
// sixteen: a few passes over values that stay in shared memory, bound by the meetings between the passes (~1.5 us each: block, then
// cluster).  Every sum has a fixed order, which the row's length alone decides.
#pragma once
#include <climits>
#include <cooperative_groups.h>

#include "kernels.cuh"

namespace knnssd {
namespace sampling {

namespace cg = cooperative_groups;

constexpr int NT = 512;                    // at 1024 the meetings take twice as long (32 sums per warp to add up), at 256 long rows do
constexpr int NW = NT / 32;
constexpr int CL = 8;                      // blocks per row; the filter takes CL_WIDE for few long rows
constexpr int CL_WIDE = 16;
constexpr int NS = 32;                     // sums that one meeting adds up: one per lane, and per warp
constexpr int SLICE_MAX = 49152;           // ids per block that fit in shared memory (192 KB)

// Meeting place of the C blocks of a row, each with SL slices of it.  `slot` alternates: a block may still read the last meeting's sums
// while another already writes the next one's.
template <int C, int SL = 1> struct MeetOf {
    static constexpr int BLOCKS = C, SLICES = SL;
    float red[SL][NW][NS + 1];
    float slot[2][C * SL][NS];
};
typedef MeetOf<CL> Meet;

// A meeting: sums (MAX: maximum of v[0]) over the threads of all blocks, in a fixed order: lanes, warps, slices.  First every warp brings
// its share of each slice, then all of them join: lane j of every warp gets sum j.  `turn` counts the meetings.
template <bool MAX, typename M>
__device__ __forceinline__ void bring(M &sh, int slice, float (&v)[NS]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (MAX) {
        const float m = warp_max(v[0]);
        if (lane == 0) sh.red[slice][warp][0] = m;
    } else {
        // each step halves the sums a lane is in charge of: 31 exchanges instead of 5 for every sum
#pragma unroll
        for (int h = NS / 2, bit = 16; h >= 1; h >>= 1, bit >>= 1) {
            const bool up = lane & bit;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const float give = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
            }
        }
        sh.red[slice][warp][lane] = v[0];
    }
}
template <bool MAX, typename M>
__device__ __forceinline__ float join(M &sh, int &turn) {
    constexpr int CL = M::BLOCKS, SL = M::SLICES;
    cg::cluster_group cluster = cg::this_cluster();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, par = turn & 1;
    ++turn;
    __syncthreads();
    // lanes r NW .. r NW + NW - 1 of warp w add up sum w PW + r of the NW warps
    constexpr int PW = NS / NW;
    static_assert(CL <= NW && NW <= 32 && NS == 32, "a lane per block in every group of lanes");
#pragma unroll
    for (int slice = 0; slice < SL; ++slice) {
        float t0 = sh.red[slice][lane % NW][MAX ? 0 : warp * PW + lane / NW];
#pragma unroll
        for (int o = NW / 2; o > 0; o >>= 1) {
            const float other = __shfl_xor_sync(0xffffffffu, t0, o);
            t0 = MAX ? fmaxf(t0, other) : t0 + other;
        }
        if (lane % NW < CL && (!MAX || (warp == 0 && lane < NW)))
            cluster.map_shared_rank(&sh, lane % NW)->slot[par][cluster.block_rank() * SL + slice][MAX ? 0 : warp * PW + lane / NW] = t0;
    }
    cluster.sync();
    float t[CL * SL];
#pragma unroll
    for (int r = 0; r < CL * SL; ++r) t[r] = sh.slot[par][r][MAX ? 0 : lane];
#pragma unroll
    for (int h = CL * SL / 2; h >= 1; h >>= 1)                   // by halves: fewer roundings than one after the other
#pragma unroll
        for (int r = 0; r < h; ++r) t[r] = MAX ? fmaxf(t[r], t[r + h]) : t[r] + t[r + h];
    return t[0];
}
template <bool MAX, typename M>
__device__ __forceinline__ float meet(M &sh, int &turn, float (&v)[NS]) {
    static_assert(M::SLICES == 1, "one slice a block");
    bring<MAX>(sh, 0, v);
    return join<MAX>(sh, turn);
}

// Count over one block.
__device__ __forceinline__ int block_count(int v, int *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    int t = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) t += sh[w];
    return t;
}

// Ids per slice of a row of V cut into so many: [r S, r S + S).
__host__ __device__ __forceinline__ int slice_len(int V, int slices = CL) { return (V + slices - 1) / slices; }
// Shared memory of filtered_probs_kernel: the values of a block's slices and, where it fits as well, the candidates among them.
inline size_t probs_smem(int V, int blocks, int slices) {
    const size_t S = slice_len(V, blocks * slices), padded = (S + NT - 1) / NT * NT;
    return sizeof(float) * (slices * (S + padded) <= SLICE_MAX ? slices * (S + padded) : slices * S <= SLICE_MAX ? slices * S : 0);
}

// use(i, p[i]) for this thread's entries i = tid, tid + NT, .. below n, U of them fetched together: the rest of an unrolled loop would
// fetch one after the other.
template <int U, typename F> __device__ __forceinline__ void each_entry(const float *p, int n, F use) {
    for (int i0 = threadIdx.x; i0 < n; i0 += U * NT) {
        float y[U];
#pragma unroll
        for (int e = 0; e < U; ++e) y[e] = i0 + e * NT < n ? p[i0 + e * NT] : 0.f;
#pragma unroll
        for (int e = 0; e < U; ++e)
            if (i0 + e * NT < n) use(i0 + e * NT, y[e]);
    }
}

// probs[row] = nucleus-filtered softmax(logits[row] / temperature), renormalised.  A token is kept iff the probability
// mass of the tokens ranked before it (higher probability first, lower id first among equals) is below top_p.
// The mass above a value is a decreasing step function of the value, so the smallest kept probability x0 is found in
// the bit patterns of positive floats, 32 candidates at a time (five bits per pass; one candidate per pass, by one block
// that re-read its row from L2 each time, took 65 us for 5 rows of 32000 and 241 us for one of 152064; this takes 15 and 21).  The first pass leaves
// a few per cent of the values between its bounds; a thread keeps those of its own aside for the others.  Once no block has more than
// GATHER values left between the bounds all blocks get them all, and each finds x0 for itself: a meeting instead of five.
// Tokens whose probability equals x0 are ranked by id.  The sum of the row comes with the first pass, what is kept is scaled once at the end:
// 5 rows of 32000 and their 4 filtered after them, with the keep-or-resample round behind: 64 us a call for 54 (kernels set up under the
// end of the one before), 9 + 8 of 152064 165 for 136; one of 152064 and a draw 52 for 48.  Error against 64 bits, rms over 2200 rows: 8.1e-8 so far,
// 7.0e-8 so.
// Every thread goes through the values left twice, ~35 ns each, where a pass leaves a thirtieth of them in 2 us: rows of sixteen slices, which may
// have 512 of them, take another pass while there are more than GATHER_WIDE (one / five / nine rows of 65536 at temperature 1, top_p 0.95:
// 28 / 34 / 44 us a call with up to 512, 23 / 24 / 32 so; 48 or 160 instead of 96: the same within 1 %, 0.2 .. 2 us more in some).
// A row is cut into C SL slices; what comes out depends on their number, not on how many blocks share them.
// grid = (C, rows), NT threads, probs_smem(V, C, SL) of shared memory; rows too long for it keep their values in `probs`.
constexpr int GATHER = 32, GATHER_WIDE = 96;
template <int C, int SL> __global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(NT)
filtered_probs_kernel(const float *__restrict__ logits, int V, float inv_temperature, float top_p, float *__restrict__ probs) {
    chain_wait();
    constexpr int SLICES = C * SL;
    static_assert(SLICES <= NS, "a sum per slice");
    extern __shared__ float probs_slice[];
    __shared__ MeetOf<C, SL> sh;
    __shared__ int shi[SL][NW];
    __shared__ int s_cut;
    __shared__ float left[SLICES][GATHER];                       // the slices' values between the bounds
    __shared__ int n_left[SLICES];
    __shared__ unsigned s_x0;
    cg::cluster_group cluster = cg::this_cluster();
    const int S = slice_len(V, SLICES), padded = (S + NT - 1) / NT * NT, rank = (int)cluster.block_rank(), tid = threadIdx.x;
    const bool keeps_list = SL * (S + padded) <= SLICE_MAX;
    int turn = 0;
    // this block's slices
    int id0[SL], n[SL], n_list[SL];
    float *p[SL];                                                // a thread only ever touches its own entries, except where ids count
    float above[SL];                                             // this thread's values that lie above all candidates
#pragma unroll
    for (int k = 0; k < SL; ++k) {
        id0[k] = min(V, (rank * SL + k) * S);
        n[k] = min(V, id0[k] + S) - id0[k];
        p[k] = keeps_list ? probs_slice + k * (S + padded) : SL * S <= SLICE_MAX ? probs_slice + k * S : probs + (size_t)blockIdx.y * V + id0[k];
        n_list[k] = 0;
        above[k] = 0.f;
    }
    auto list = [&](int k) { return probs_slice + k * (S + padded) + S + tid; };
    float v[NS];
    cluster.barrier_arrive();                                    // every block has to run before another writes to its shared memory
    float m = -INFINITY;
#pragma unroll
    for (int k = 0; k < SL; ++k) {
        float *to = p[k];
        each_entry<8>(logits + (size_t)blockIdx.y * V + id0[k], n[k], [&](int i, float x) { to[i] = x; m = fmaxf(m, x); });
    }
    v[0] = m;
    cluster.barrier_wait();
#pragma unroll
    for (int k = 0; k < SL; ++k) bring<true>(sh, k, v);
    m = join<true>(sh, turn);
    // From here on the values are e = exp((x - max) / temperature), softmax before its division by the sum, which the first pass brings along:
    // a token's mass is compared with top_p times that sum.  (A pass of its own over the row for the sum and one for the division cost a
    // meeting and 2 us.)  The largest value is 1, nothing lies above it.  Below (1 - top_p) / (2 V) there is less than half of 1 - top_p of the
    // mass, which is at least 1, so what lies above that is not below top_p of it: a sum of V terms is not off by the other half
    // unless top_p is 1 to four digits.
#pragma unroll
    for (int k = 0; k < SL; ++k) {
        float *to = p[k];
        each_entry<4>(to, n[k], [&](int i, float x) { to[i] = expf((x - m) * inv_temperature); });
    }
    unsigned lo = 0u, hi = __float_as_uint(1.0f);
    if (1.0f - top_p > 1e-4f) lo = min(hi, __float_as_uint(0.5f * (1.0f - top_p) / (float)V));
    // The largest value, 1, is counted and not added: the sums are of what lies below it, so that they are not rounded at its size.
    float ones = 0.f, kept_mass = 0.f, kept_rest = 0.f;          // how often it occurs; top_p times the whole sum, and what that leaves for the rest
    auto small = [](float y) { return y == 1.f ? 0.f : y; };
    float above_hi = 0.f;                                        // the rest of all threads' values above hi
    int gathered = -1;                                           // values between the bounds, once all blocks have them
    for (bool first = true; first || hi > lo + 1u; first = false) {
        const int nc = first ? NS - 2 : NS;                      // candidates lo, lo + step, ..: lo itself only counts in the first pass, whose last
        const unsigned step = (hi - lo + nc - 1) / nc;           // sums are the row's ones and the rest of it
        float x[NS];
#pragma unroll
        for (int j = 0; j < NS; ++j) x[j] = __uint_as_float(min(hi, lo + j * step));
        const bool listed = keeps_list && !first;
#pragma unroll
        for (int k = 0; k < SL; ++k) {
#pragma unroll
            for (int j = 0; j < NS; ++j) v[j] = above[k];
            auto count = [&](float y) {
                const float r = small(y);
#pragma unroll
                for (int j = 0; j < NS - 2; ++j) v[j] += y > x[j] ? r : 0.f;
                if (first) {
                    v[NS - 2] += y == 1.f ? 1.f : 0.f;
                    v[NS - 1] += r;
                } else {
                    v[NS - 2] += y > x[NS - 2] ? r : 0.f;
                    v[NS - 1] += y > x[NS - 1] ? r : 0.f;
                }
            };
            if (listed) {                                        // hardly any thread has more than one left
#pragma unroll 1
                for (int i = 0; i < n_list[k]; ++i) count(list(k)[NT * i]);
            } else {
                each_entry<4>(p[k], n[k], [&](int, float y) { count(y); });
            }
            bring<false>(sh, k, v);
        }
        const float mass = join<false>(sh, turn);
        if (first) {
            const float rest = __shfl_sync(0xffffffffu, mass, NS - 1);
            if (!(rest == rest)) { hi = lo = __float_as_uint(2.0f); break; }     // a NaN in the row: nothing is kept of it
            ones = __shfl_sync(0xffffffffu, mass, NS - 2);
            kept_mass = fmaf(top_p, rest, top_p * ones);
            // (from 1 on nothing is left out: where the sums' rounding ends the nucleus is not searched for)
            kept_rest = top_p >= 1.0f ? INFINITY : fmaf(top_p, rest, (top_p - 1.0f) * ones);
        }
        const unsigned below = __ballot_sync(0xffffffffu, mass < kept_rest) & (first ? 0x3fffffffu : 0xffffffffu);
        int j = below ? __ffs(below) - 1 : nc;                   // the first candidate with less than top_p above it
        if (j == 0) {
            if (first) { hi = lo; above_hi = __shfl_sync(0xffffffffu, mass, 0); break; }
            j = 1;                                               // lo was ruled out before, by sums in another order
        }
        if (j < nc && lo + j * step < hi) above_hi = __shfl_sync(0xffffffffu, mass, j);
        const unsigned nhi = j < nc ? min(hi, lo + j * step) : hi;
        lo = min(hi, lo + (j - 1) * step);
        hi = nhi;
        const float xl = __uint_as_float(lo), xh = __uint_as_float(hi);
        if (first && keeps_list) {
#pragma unroll
            for (int k = 0; k < SL; ++k)
                each_entry<4>(p[k], n[k], [&](int, float y) {
                    if (y > xh) above[k] += small(y);
                    else if (y > xl) list(k)[NT * n_list[k]++] = y;
                });
        } else if (keeps_list && hi > lo + 1u) {
            // hand the values left to all blocks, in the order of slices, threads and each thread's list
            const int lane = tid & 31, warp = tid >> 5;
            int upto[SL], own[SL], all[SL];
#pragma unroll
            for (int k = 0; k < SL; ++k) {
                own[k] = 0;
                for (int i = 0; i < n_list[k]; ++i) { const float y = list(k)[NT * i]; own[k] += y > xl && y <= xh ? 1 : 0; }
                upto[k] = own[k];                                // of the warp's lanes up to this one
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, upto[k], o); if (lane >= o) upto[k] += t; }
                if (lane == 31) shi[k][warp] = upto[k];
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < SL; ++k) {
                int before = 0;
                all[k] = 0;
#pragma unroll
                for (int w = 0; w < NW; ++w) { if (w == warp) before = all[k]; all[k] += shi[k][w]; }
                int at = before + upto[k] - own[k];
                for (int i = 0; i < n_list[k]; ++i) {
                    const float y = list(k)[NT * i];
                    if (y > xl && y <= xh) { if (at < GATHER) left[rank * SL + k][at] = y; ++at; }
                }
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < SL; ++k)
                for (int t = tid; t < C * GATHER; t += NT) {
                    const int r = t / GATHER, i = t % GATHER;
                    if (r != rank && i < min(all[k], GATHER)) *cluster.map_shared_rank(&left[rank * SL + k][i], r) = left[rank * SL + k][i];
                    if (i == 0) *cluster.map_shared_rank(&n_left[rank * SL + k], r) = all[k];
                }
            cluster.sync();
            int most = 0, total = 0;
#pragma unroll
            for (int r = 0; r < SLICES; ++r) { most = max(most, n_left[r]); total += n_left[r]; }
            if (most <= GATHER && (SLICES <= CL || total <= GATHER_WIDE)) { gathered = total; break; }
            cluster.sync();                                      // nobody writes the next values while others read these counts
        }
    }
    float x0 = __uint_as_float(hi);
    float a0 = above_hi;                                         // the rest's mass above x0
    int c = 0, own_c[SL];                                        // tokens at x0: of all slices, and this thread's share of its block's
#pragma unroll
    for (int k = 0; k < SL; ++k) own_c[k] = 0;
    if (gathered >= 0) {
        // the smallest of the values left with less than top_p above it; if rounding has it that there is none, hi
        if (tid == 0) s_x0 = hi;
        __syncthreads();
        for (int t = tid; t < SLICES * GATHER; t += NT) {
            const int r = t / GATHER, i = t % GATHER;
            if (i < n_left[r]) {
                const float y = left[r][i];
                float m_above = 0.f;                             // the few small values by themselves, then one rounding at the size of the mass
                for (int q = 0; q < SLICES; ++q)
                    for (int e = 0, n_q = n_left[q]; e < n_q; ++e) { const float o = left[q][e]; m_above += o > y ? small(o) : 0.f; }
                if (y == 1.f || above_hi + m_above < kept_rest) atomicMin(&s_x0, __float_as_uint(y));
            }
        }
        __syncthreads();
        x0 = __uint_as_float(s_x0);
        float left_above = 0.f;
        for (int q = 0; q < SLICES; ++q)
            for (int e = 0, n_q = n_left[q]; e < n_q; ++e) {
                const float o = left[q][e];
                left_above += o > x0 ? small(o) : 0.f;
                if (o == x0) {
                    ++c;
#pragma unroll
                    for (int k = 0; k < SL; ++k) own_c[k] += q == rank * SL + k && tid == 0 ? 1 : 0;
                }
            }
        a0 = above_hi + left_above;
    } else {
        // rows whose values are not kept aside, and bounds that met without it
#pragma unroll
        for (int k = 0; k < SL; ++k) {
#pragma unroll
            for (int j = 0; j < NS; ++j) v[j] = 0.f;
            each_entry<4>(p[k], n[k], [&](int, float y) {
                v[0] += y > x0 ? small(y) : 0.f;
                if (y == x0) v[1] += 1.f;                        // counts are exact up to 2^24 tokens
            });
            own_c[k] = (int)v[1];
            bring<false>(sh, k, v);
        }
        const float tot = join<false>(sh, turn);
        a0 = __shfl_sync(0xffffffffu, tot, 0);
        c = (int)__shfl_sync(0xffffffffu, tot, 1);
    }
    const bool at_top = x0 == 1.f;                               // the largest value's tokens are the last ones kept
    if (at_top) a0 = 0.f;
    const float enough = at_top ? kept_mass : kept_rest;
    // tokens at exactly x0: the n-th of them by id (n = 0, 1, ..) is kept iff mass above x0 + n x0 < top_p of it all
    int nk = 1, id_cut = V;                                      // tokens at x0 with id < id_cut are kept; the first one always is
    if (c > 1) {
        nk = 0;
        for (int i = tid; i < c; i += NT) nk += (a0 + (float)i * x0 < enough) ? 1 : 0;
        nk = max(1, block_count(nk, shi[0]));
        if (nk < c) {                                            // which of them: the slice that has the nk-th is searched for its id
            // sum r of this meeting: the tokens at x0 in slice r
#pragma unroll
            for (int k = 0; k < SL; ++k) {
#pragma unroll
                for (int j = 0; j < NS; ++j) v[j] = j == rank * SL + k ? (float)own_c[k] : 0.f;
                bring<false>(sh, k, v);
            }
            const float tot = join<false>(sh, turn);
            int before = 0, holder = 0;
            for (int r = 0; r < SLICES; ++r) {
                const int cr = (int)__shfl_sync(0xffffffffu, tot, r);
                if (before + cr >= nk) { holder = r; break; }
                before += cr;
            }
#pragma unroll
            for (int k = 0; k < SL; ++k)
                if (rank * SL + k == holder) {
                    __syncthreads();
                    int jl = 0, jh = n[k];                       // smallest J with #{j < J : p_j == x0} >= nk - before
                    while (jh > jl + 1) {
                        const int jm = jl + (jh - jl) / 2;
                        int g = 0;
                        for (int i = tid; i < jm; i += NT) g += p[k][i] == x0 ? 1 : 0;
                        g = block_count(g, shi[0]);
                        if (g >= nk - before) jh = jm; else jl = jm;
                    }
                    if (tid < C) *cluster.map_shared_rank(&s_cut, tid) = id0[k] + jh;
                }
            cluster.sync();
            id_cut = s_cut;
        }
    }
    // one over what is kept in all, in two floats: a product with both is rounded once (and costs less than a division)
    const double per_z = 1.0 / ((at_top ? 0.0 : (double)ones) + (double)a0 + (double)min(nk, c) * (double)x0);
    const float z_hi = (float)per_z, z_lo = (float)(per_z - (double)z_hi);
#pragma unroll
    for (int k = 0; k < SL; ++k) {
        float *out = probs + (size_t)blockIdx.y * V + id0[k];
        each_entry<4>(p[k], n[k], [&](int i, float y) { out[i] = (y > x0 || (y == x0 && id0[k] + i < id_cut)) ? fmaf(y, z_hi, y * z_lo) : 0.f; });
    }
    cluster.sync();                                              // nobody leaves while its shared memory may still be written to
}

// Inverse CDF in token-id order: the smallest id x with w_0 + .. + w_x > u * sum(w); w_i = a_i (b == nullptr) or
// max(a_i - b_i, 0), falling back to a if that is zero everywhere.  Called by all threads of a cluster; block r has the ids
// [r S, (r + 1) S), its warp w a contiguous run of them, read 32 at a time; the block whose ids hold the crossing walks the run of the warp
// that does with all its threads.  Block 0's thread 0 returns the token (-1: no weight anywhere).
// (One block with a run of ids per thread and a serial scan of 1024 sums took 41 us for 152064 ids, the run walked by its own warp 8.5.)
struct Draw {
    Meet m;
    float warp_sum[NW], tot[4 * NW];
    int last[CL];
    int first, seen;                                             // of the ids that the block walks: where the sum crosses, the last with weight
    int token;
};
__device__ __forceinline__ int cluster_sample(const float *__restrict__ a, const float *__restrict__ b, int V, float u, Draw &sh) {
    cg::cluster_group cluster = cg::this_cluster();
    const int S = slice_len(V), rank = (int)cluster.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int run = (S + NW - 1) / NW, lim = min(V, rank * S + S);
    const int i0 = min(lim, rank * S + warp * run), i1 = min(lim, i0 + run);
    bool use_b = b != nullptr;
    int turn = 0;
    if (tid == 0) sh.token = -1;
    cluster.barrier_arrive();                                    // every block has to run before another writes to its shared memory
    for (bool first = true;; first = false) {
        auto weight = [&](int i) { return use_b ? fmaxf(a[i] - b[i], 0.f) : a[i]; };
        float w = 0.f;
        int last = -1;
#pragma unroll 8
        for (int i = i0 + lane; i < i1; i += 32) {
            const float x = weight(i);
            if (x > 0.f) last = i;
            w += x;
        }
        w = warp_sum(w);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
        if (first) cluster.barrier_wait();
        __syncthreads();
        if (lane == 0) { sh.warp_sum[warp] = w; sh.m.red[0][warp][NS] = __int_as_float(last); }
        __syncthreads();
        // sum r of the meeting: block r's weights, its warps added in order
        float v[NS], mine = 0.f;
        if (tid == 0)
            for (int k = 0; k < NW; ++k) mine += sh.warp_sum[k];
        if (warp == 0) {
            int lb = lane < NW ? __float_as_int(sh.m.red[0][lane][NS]) : -1;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lb = max(lb, __shfl_xor_sync(0xffffffffu, lb, o));
            if (lane == 0) cluster.map_shared_rank(&sh, 0)->last[rank] = lb;
        }
#pragma unroll
        for (int j = 0; j < NS; ++j) v[j] = j == rank ? mine : 0.f;
        const float per_block = meet<false>(sh.m, turn, v);
        float total = 0.f, before = 0.f, through = 0.f;
#pragma unroll
        for (int r = 0; r < CL; ++r) {
            if (r == rank) before = total;
            total += __shfl_sync(0xffffffffu, per_block, r);
            if (r == rank) through = total;
        }
        if (use_b && !(total > 0.f)) { use_b = false; continue; }
        const float target = u * total;
        if (before <= target && through > target) {              // uniform: the crossing is in this block
            // the warp whose run holds it (the last one ends where the block does); the whole block walks that run, 4 NT ids at a time
            int w = 0;
            float excl = before;
            while (w < NW - 1 && !(excl + sh.warp_sum[w] > target)) excl += sh.warp_sum[w++];
            const int j0 = min(lim, rank * S + w * run), j1 = min(lim, j0 + run);
            if (tid == 0) { sh.first = INT_MAX; sh.seen = -1; }
            __syncthreads();
            int tok = -1;
            for (int jb = j0; jb < j1 && tok < 0; jb += 4 * NT) {
                float x[4], sc[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) { const int i = jb + e * NT + tid; x[e] = i < j1 ? weight(i) : 0.f; }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    sc[e] = x[e];
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const float t = __shfl_up_sync(0xffffffffu, sc[e], o);
                        if (lane >= o) sc[e] += t;
                    }
                    if (lane == 31) sh.tot[e * NW + warp] = sc[e];
                }
                __syncthreads();
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (jb + e * NT >= j1) break;                // uniform
                    float acc = excl;                            // before this thread's warp, and before the next NT ids
#pragma unroll
                    for (int k = 0; k < NW; ++k) {
                        const float t = sh.tot[e * NW + k];
                        if (k < warp) acc += t;
                        excl += t;
                    }
                    const int i = jb + e * NT + tid;
                    if (x[e] > 0.f) {
                        if (acc + sc[e] > target) atomicMin(&sh.first, i);
                        atomicMax(&sh.seen, i);
                    }
                }
                __syncthreads();
                if (sh.first != INT_MAX) tok = sh.first;
            }
            if (tok < 0) tok = sh.seen;                          // the last id with weight, if rounding hides the crossing
            // no weight in the run: the block's sum, added at once, ends an ulp past the running sum of its warps, and the target lies between.
            // The crossing is in this block all the same: its last id with weight
            if (tok < 0)
                for (int k = 0; k < NW; ++k) tok = max(tok, __float_as_int(sh.m.red[0][k][NS]));
            if (tid == 0 && tok >= 0) atomicMax(&cluster.map_shared_rank(&sh, 0)->token, tok);
        }
        break;
    }
    cluster.sync();
    int tok = sh.token;
    if (rank == 0 && tok < 0)                                    // target rounded up to the total: the last id with weight
        for (int r = 0; r < CL; ++r) tok = max(tok, sh.last[r]);
    return tok;
}

// token <- draw from weights w[V] with the uniform *u_ptr (u_val if u_ptr is null).  One cluster.
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(NT)
sample_kernel(const float *__restrict__ w, int V, const float *__restrict__ u_ptr, float u_val, int *__restrict__ token) {
    chain_wait();
    __shared__ Draw sh;
    const int tok = cluster_sample(w, nullptr, V, u_ptr ? *u_ptr : u_val, sh);
    if (threadIdx.x == 0 && blockIdx.x == 0) *token = tok < 0 ? 0 : tok;
}

// The drafts of a round and their uniforms: on the device, or with the launch (read from pinned host memory they were a trip across the bus).
struct DeviceRound {
    const int *drafts;
    const float *u_accept, *u_final;
    __device__ __forceinline__ int draft(int j) const { return drafts[j]; }
    __device__ __forceinline__ float accept(int j) const { return u_accept[j]; }
    __device__ __forceinline__ float last() const { return *u_final; }
};
struct GivenRound {
    int drafts[16];
    float u_accept[16], u_final;
    __device__ __forceinline__ int draft(int j) const { return drafts[j]; }
    __device__ __forceinline__ float accept(int j) const { return u_accept[j]; }
    __device__ __forceinline__ float last() const { return u_final; }
};

// One verification round of speculative sampling.  p [k+1][V], q [k][V] filtered distributions, k <= 16.  out[0] = number of drafts kept,
// out[1] = the token emitted after them.  One cluster.
template <typename Round>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(NT)
spec_accept_kernel(const float *__restrict__ p, const float *__restrict__ q, const __grid_constant__ Round round, int k, int V, int *__restrict__ out) {
    chain_wait();
    __shared__ Draw sh;
    const float u_final = round.last();
    // every warp tests all drafts, one per lane: the first that is not kept ends the round
    const int lane = threadIdx.x & 31;
    bool keep = false;
    if (lane < k) {
        const int d = round.draft(lane);
        // a token outside the vocabulary is never kept
        keep = d >= 0 && d < V && round.accept(lane) * q[(size_t)lane * V + d] < p[(size_t)lane * V + d];
    }
    const unsigned lost = ~__ballot_sync(0xffffffffu, keep) & ((1u << k) - 1u);
    const int j = lost ? __ffs(lost) - 1 : k;
    const int tok = j < k ? cluster_sample(p + (size_t)j * V, q + (size_t)j * V, V, u_final, sh)
                          : cluster_sample(p + (size_t)k * V, nullptr, V, u_final, sh);
    if (threadIdx.x == 0 && blockIdx.x == 0) { out[0] = j; out[1] = tok < 0 ? 0 : tok; }
}

// The round's result into the session (one thread): res[0] = drafts kept, res[1] = the token after them; chain[1 .. k]
// the drafts.  Same bookkeeping as the greedy accept step.
__global__ void commit_sampled_kernel(int *__restrict__ chain, const int *__restrict__ res, DeviceState *__restrict__ st,
                                      int *__restrict__ out_tokens, int out_cap, int *__restrict__ accept_log, int round_idx) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int a = res[0], next = res[1];
    int p = st->produced;
    for (int j = 0; j < a && p < out_cap; ++j) out_tokens[p++] = chain[j + 1];
    if (p < out_cap) out_tokens[p++] = next;
    st->produced = p;
    st->len += a + 1;
    st->last_accept = a;
    st->last_next = next;
    chain[0] = next;
    if (accept_log) accept_log[round_idx] = a;
}

}  // namespace sampling
}  // namespace knnssd
