// Anchor construction of the pre-inference stage (Sec. 4.1): the sampled last hidden vectors of all domains are
// clustered with K-means (Lloyd's iteration, as many clusters as domains), and each cluster's k members nearest to
// its centroid become its anchors (Eq. (2): the k smallest distances minimise the sum over size-k subsets).
//
// The points are fp32 [N][d] (d = the model width, N = domains x samples per domain: 5 x 1000 in the paper's
// set-up, 100 MB at d = 5120).  Centroids and their sums are fp64.  A squared distance is formed from fp32
// differences to the fp32-rounded centroid, squared and added eight at a time in fp32, and those short sums are
// accumulated without loss in pairs of floats (fp64 only for the final reductions): a float becomes a double at 15 lanes per clock and SM
// (fp64 additions and products 58), so fp64 arithmetic for every element and cluster made the assignment 15x slower than its memory
// traffic, while this form keeps ~1e-8 relative accuracy (error of a
// distance^2 of ~1e3: ~1e-5, four orders below the gaps that decide nearest centroids and nearest members).  A round
// reads the points twice (assignment, centroid sums).  Every reduction has a fixed order, given by the sizes: results depend neither on
// timing nor on the device's share of SMs.
#pragma once

#include "kernels.cuh"

namespace knnssd {
namespace anchors {

constexpr int MAXC = 16;       // most clusters (domains)
constexpr int CHUNK = 256;     // columns of the centroids staged in shared memory per step
constexpr int MAX_WARPS = 8;   // most warps of a block of assign_kernel, two points each
constexpr int RING = 3;        // steps of columns a block of assign_kernel has in flight or in use: three blocks per SM

// What the rounds of a call leave on the device, so that several rounds can be enqueued without the host looking at the
// outcome of each: the kernels of a round do nothing once an earlier round changed no assignment.
struct Progress {
    int done;                  // a round changed nothing
    int rounds;                // assignment rounds done
    int changed[2];            // by round parity: the round changed an assignment
    int counts[2][MAXC];       // by round parity: members per cluster
};

// One 16-byte (VEC) or 4-byte piece on its way into shared memory; zeros where there is nothing to read.
template <bool VEC> __device__ __forceinline__ void copy_piece(float *dst, const float *src, bool live) {
    const unsigned to = (unsigned)__cvta_generic_to_shared(dst);
    if (VEC) {
        const int n = live ? 16 : 0;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(src), "r"(n) : "memory");
    } else {
        const int n = live ? 4 : 0;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(to), "l"(src), "r"(n) : "memory");
    }
}

// For each point: the squared distances to all n centroids, labels[p] <- the nearest centroid (lowest index among equal
// distances); the round's `changed` is set if that differs from the old label, its counts[c] incremented.  mu32 holds the
// centroids rounded to fp32, rows of stride ld (a multiple of 4).  4 .. 8 warps a block (assign_warps), grid = ceil(N / (2 warps)): a
// warp owns two points, the block shares the columns of the centroids.  Per step of 256 columns a lane holds 8 columns of each of its
// points (VEC, d % 4 == 0: two runs of four).  Points and centroids come through a ring of RING steps of asynchronous
// copies: what bounds the kernel is how much of the points is in flight (5000 x 5120: one step ahead in registers 58 us, with the ring 35) and
// the SM with most of the points (blocks of 8 warps leave 48 points on some SMs for 34 on average, of 6 warps 36: 30 us).
// NC = the cluster count rounded up to 4, 8 or 16: the per-cluster registers follow it.
template <int NC> constexpr int assign_smem(int warps) { return RING * (2 * warps + NC) * CHUNK * (int)sizeof(float); }
// Warps per block: the fewest rows for the fullest SM, blocks dealt out evenly, each with its points and all n centroids; the larger block
// among equals.  5 clusters: 5000 x 5120 six warps 67 us a round, eight 71; 300000 x 64 eight 600, six 624, five (the fewest points alone) 628.
inline int assign_warps(int N, int n, int n_sms) {
    int best = MAX_WARPS;
    long long least = -1;
    for (int w = MAX_WARPS; w >= 4; --w) {
        const long long blocks = (N + 2 * w - 1) / (2 * w), most = (blocks + n_sms - 1) / n_sms * (2 * w + n);
        if (least < 0 || most < least) { least = most; best = w; }
    }
    return best;
}
template <bool VEC, int NC>
__global__ void __launch_bounds__(256, NC <= 8 ? 3 : 2) assign_kernel(const float *__restrict__ x, int N, int d, const float *__restrict__ mu32, int ld, int n,
                                                     int parity, int *__restrict__ labels, Progress *__restrict__ pg) {
    extern __shared__ __align__(16) float as_smem[];             // [RING][pts points, then NC centroids][CHUNK]
    chain_wait();
    if (pg->done) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5, pts = 2 * warps;
    const int p0 = blockIdx.x * pts, pa = p0 + 2 * warp;
    // running sums as unevaluated pairs of floats (hi + lo, hi the rounded sum, lo the rounding errors collected by
    // the error-free two-sum): ~48 bits without touching the fp64 pipe in the loop
    float hi[2][NC], lo[2][NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) hi[0][c] = hi[1][c] = lo[0][c] = lo[1][c] = 0.f;
    auto add_pair = [](float &h, float &l, float v) {
        const float s = __fadd_rn(h, v);
        const float bb = __fsub_rn(s, h);
        l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(v, bb)));
        h = s;
    };
    const int steps = (d + CHUNK - 1) / CHUNK;
    constexpr int W = VEC ? 4 : 1;                               // columns per piece
    auto fetch = [&](int step) {
        if (step < steps) {
            const int col0 = step * CHUNK;
            float *st = as_smem + (step % RING) * (pts + NC) * CHUNK;
            // rows of this warp: its two points, and its share of the centroids
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int p = pa + q;
                const float *src = x + (size_t)min(p, N - 1) * d;
#pragma unroll
                for (int j = lane * W; j < CHUNK; j += 32 * W) {
                    const bool live = p < N && col0 + j < d;
                    copy_piece<VEC>(st + (2 * warp + q) * CHUNK + j, src + (live ? col0 + j : 0), live);
                }
            }
            for (int c = warp; c < n; c += warps)
#pragma unroll
                for (int j = lane * 4; j < CHUNK; j += 128) {
                    const bool live = col0 + j < ld;
                    copy_piece<true>(st + (pts + c) * CHUNK + j, mu32 + (size_t)c * ld + (live ? col0 + j : 0), live);
                }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");     // empty groups keep the count of groups equal to that of steps
    };
#pragma unroll
    for (int i = 0; i < RING - 1; ++i) fetch(i);
    for (int step = 0; step < steps; ++step) {
        asm volatile("cp.async.wait_group %0;" ::"n"(RING - 2) : "memory");
        __syncthreads();                                         // this step has arrived for all; the one before has been read by all
        fetch(step + RING - 1);
        const float *st = as_smem + (step % RING) * (pts + NC) * CHUNK;
        auto row = [&](int r, float (&v)[8]) {
            if (VEC) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 t = *reinterpret_cast<const float4 *>(st + r * CHUNK + h * 128 + 4 * lane);
                    v[4 * h] = t.x; v[4 * h + 1] = t.y; v[4 * h + 2] = t.z; v[4 * h + 3] = t.w;
                }
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = st[r * CHUNK + lane + 32 * i];
            }
        };
        float ca[8], cb[8];
        row(2 * warp, ca);
        row(2 * warp + 1, cb);
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (c < n) {
                // columns past the end hold zeros on both sides: they add nothing
                float m[8], sa = 0.f, sb = 0.f;
                row(pts + c, m);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float da = ca[i] - m[i], db = cb[i] - m[i];
                    sa = fmaf(da, da, sa);
                    sb = fmaf(db, db, sb);
                }
                add_pair(hi[0][c], lo[0][c], sa);
                add_pair(hi[1][c], lo[1][c], sb);
            }
    }
    double acc[2][NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) { acc[0][c] = (double)hi[0][c] + (double)lo[0][c]; acc[1][c] = (double)hi[1][c] + (double)lo[1][c]; }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int p = pa + q;
        if (p >= N) continue;                                  // warp-uniform
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (c < n) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc[q][c] += __shfl_xor_sync(0xffffffffu, acc[q][c], o);
            }
        if (lane == 0) {
            int best = 0;
            double bv = acc[q][0];
#pragma unroll
            for (int c = 1; c < NC; ++c)
                if (c < n && acc[q][c] < bv) { bv = acc[q][c]; best = c; }
            if (best != labels[p]) { labels[p] = best; atomicOr(pg->changed + parity, 1); }
            atomicAdd(pg->counts[parity] + best, 1);
        }
    }
}

// Slices of the centroid sums: at least 64 points each, at most 64 slices, and as many as keep all blocks resident (six on each of 148 SMs) if
// that is fewer: then the sorted form runs.  N and d decide, not the SMs that the process has got: the slices are the order of the
// additions, and the centroids' last bits are the same on a part of a GPU.
constexpr int SUM_BLOCKS = 6 * 148;
inline int sum_slices(int N, int d, bool &sorted) {
    int S = (N + 63) / 64;
    if (S > 64) S = 64;
    const int cols = (d + 255) / 256, most = SUM_BLOCKS / cols;
    sorted = S > most;
    return !sorted ? S : most > 1 ? most : 1;
}
// part[s][c][j] = sum of x[p][j] over the points p of slice s (S slices of `per` consecutive points) labelled c, added
// in index order.  grid = (ceil(d / 256), S), 256 threads: a thread owns one column.  Bound by the trips to memory, eight points at a
// time.  (The fp64 pipe has room: 58 additions and 15 conversions per clock and SM, measured.)
__global__ void __launch_bounds__(256) partial_sums_kernel(const float *__restrict__ x, int N, int d, const int *__restrict__ labels,
                                                           int n, int per, double *__restrict__ part, int parity,
                                                           const Progress *__restrict__ pg) {
    chain_wait();
    if (pg->done || !pg->changed[parity]) return;
    __shared__ double acc[MAXC][256];
    const int j = blockIdx.x * 256 + threadIdx.x, s = blockIdx.y;
    for (int c = 0; c < n; ++c) acc[c][threadIdx.x] = 0.0;
    const int p0 = s * per, p1 = min(N, p0 + per);
    if (j < d) {
        int p = p0;
        for (; p + 8 <= p1; p += 8) {                          // eight loads in flight, added in index order
            float v[8];
            int l[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) { v[i] = __ldg(x + (size_t)(p + i) * d + j); l[i] = labels[p + i]; }
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[l[i]][threadIdx.x] += (double)v[i];
        }
        for (; p < p1; ++p) acc[labels[p]][threadIdx.x] += (double)__ldg(x + (size_t)p * d + j);
    }
    if (j < d)
        for (int c = 0; c < n; ++c) part[((size_t)s * n + c) * d + j] = acc[c][threadIdx.x];
}

// The same where its blocks would not all be resident at once: fewer and longer slices (sum_slices), whose points are taken cluster by
// cluster - a stable sort of at most 256 of them at a time -, so that a running sum stays in a register and only goes to shared memory
// where the cluster changes.  5000 x 5120: 26 us for 32 in one and a half rounds of blocks, the call of four rounds 320 us for 341; 4000 x 4096 252
// for 258.  Where all blocks of the plain form are resident the sort only costs: 120 x 1024 106 us for 101, 1200 x 2049 157 for 150.  (The
// running sums in as much shared memory as there: another size has the SM's memory divided anew between kernels, 5 .. 7 us a round.)
constexpr int SUM_LOADS = 8;
__global__ void __launch_bounds__(256, 6) sorted_sums_kernel(const float *__restrict__ x, int N, int d, const int *__restrict__ labels,
                                                              int n, int per, double *__restrict__ part, int parity,
                                                              const Progress *__restrict__ pg) {
    chain_wait();
    if (pg->done || !pg->changed[parity]) return;
    __shared__ double sum_acc[MAXC * 256];                     // [n][256]
    __shared__ int order[256], first[MAXC + 1], in_warp[8][MAXC];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, j = blockIdx.x * 256 + tid, s = blockIdx.y;
    const int p0 = s * per, p1 = min(N, p0 + per);
    const float *col = x + min(j, d - 1);
    for (int c = 0; c < n; ++c) sum_acc[c * 256 + tid] = 0.0;
    for (int q0 = p0; q0 < p1; q0 += 256) {
        const int len = min(256, p1 - q0), l = tid < len ? labels[q0 + tid] : -1;
        unsigned mine = 0u;
        for (int c = 0; c < n; ++c) {
            const unsigned who = __ballot_sync(0xffffffffu, l == c);
            if (l == c) mine = who;
            if (lane == 0) in_warp[warp][c] = __popc(who);
        }
        __syncthreads();                                       // the counts are there, the order before has been read
        if (l >= 0) {
            int at = __popc(mine & ((1u << lane) - 1u));
            for (int c = 0; c < l; ++c)
#pragma unroll
                for (int w = 0; w < 8; ++w) at += in_warp[w][c];
            for (int w = 0; w < warp; ++w) at += in_warp[w][l];
            order[at] = q0 + tid;
        }
        if (tid <= n) {
            int at = 0;
            for (int c = 0; c < tid; ++c)
#pragma unroll
                for (int w = 0; w < 8; ++w) at += in_warp[w][c];
            first[tid] = at;
        }
        __syncthreads();
        int c = 0, end = first[1];
        double a = sum_acc[tid];
        for (int i0 = 0; i0 < len; i0 += SUM_LOADS) {
            float v[SUM_LOADS];
#pragma unroll
            for (int e = 0; e < SUM_LOADS; ++e) v[e] = __ldg(col + (size_t)order[min(i0 + e, len - 1)] * d);
#pragma unroll
            for (int e = 0; e < SUM_LOADS; ++e) {
                if (i0 + e >= len) break;                      // uniform, as are the clusters' ends
                while (i0 + e >= end) { sum_acc[c * 256 + tid] = a; ++c; a = sum_acc[c * 256 + tid]; end = first[c + 1]; }
                a += (double)v[e];
            }
        }
        sum_acc[c * 256 + tid] = a;
    }
    if (j < d)
        for (int c = 0; c < n; ++c) part[((size_t)s * n + c) * d + j] = sum_acc[c * 256 + tid];
}

// The end of a round.  If it changed an assignment: mu[c][j] = (sum over slices, in slice order, of part[s][c][j]) /
// counts[c], in mu32 rounded to fp32; a cluster without members keeps its centroid.  Otherwise the iteration is done.  Clears
// the counters of the next round.  grid = (ceil(d / 128), n), 128 threads.  Bound by the trips to L2: twenty slices in flight (44 slices of
// 5 x 5120 7.5 us; eight of 64 in flight took 9.3).
__global__ void __launch_bounds__(128) fold_centroids_kernel(const double *__restrict__ part, int n, int d, int S, double *__restrict__ mu, float *__restrict__ mu32,
                                      int ld, int parity, Progress *__restrict__ pg) {
    chain_wait();
    const bool changed = pg->changed[parity] != 0;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && !pg->done) {
        // the other blocks act on this round's `changed` and `counts` alone, which stay as they are until the next round's end
        pg->rounds += 1;
        pg->changed[parity ^ 1] = 0;
        for (int c = 0; c < MAXC; ++c) pg->counts[parity ^ 1][c] = 0;
        if (!changed) pg->done = 1;
    }
    const int j = blockIdx.x * 128 + threadIdx.x, c = blockIdx.y;
    if (!changed || j >= d || pg->counts[parity][c] == 0) return;
    double s = 0.0;
    constexpr int U = 20;                                     // loads in flight, added in slice order
    for (int i = 0; i < S; i += U) {
        double v[U];
#pragma unroll
        for (int e = 0; e < U; ++e) v[e] = i + e < S ? __ldcg(part + ((size_t)(i + e) * n + c) * d + j) : 0.0;
#pragma unroll
        for (int e = 0; e < U; ++e)
            if (i + e < S) s += v[e];
    }
    s /= (double)pg->counts[parity][c];
    mu[(size_t)c * d + j] = s;
    mu32[(size_t)c * ld + j] = (float)s;
}

// The starting centroids in both precisions (mu32's padding and the progress start at zero).  grid = (ceil(d / 256), n).
__global__ void start_centroids_kernel(const float *__restrict__ start, int d, double *__restrict__ mu, float *__restrict__ mu32, int ld) {
    const int j = blockIdx.x * 256 + threadIdx.x, c = blockIdx.y;
    if (j >= d) return;
    const float v = start[(size_t)c * d + j];
    mu[(size_t)c * d + j] = (double)v;
    mu32[(size_t)c * ld + j] = v;
}

// dist[p] = ||x_p - mu_{labels[p]}|| with every difference, square and sum in fp64 against the fp64 centroid: the
// distances Eq. (2) ranks the members by.  Points at equal distance in exact arithmetic (duplicates, or points mirrored
// about their centroid) then get equal values, so the lowest index decides among them.  One warp per point, lanes
// stride over the columns, fixed-order reduction.  Nothing happens while the rounds are
// not done and these are not the last ones.  grid = ceil(N / 8), 256 threads.
__global__ void __launch_bounds__(256) member_dist_kernel(const float *__restrict__ x, int N, int d, const double *__restrict__ mu,
                                                          const int *__restrict__ labels, double *__restrict__ dist,
                                                          const Progress *__restrict__ pg, int last) {
    chain_wait();
    if (!pg->done && !last) return;
    const int lane = threadIdx.x & 31, p = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (p >= N) return;
    const float *xr = x + (size_t)p * d;
    const double *m = mu + (size_t)labels[p] * d;
    double s = 0.0;
    auto take = [&](float v, double c) {
        const double df = (double)v - c;
        s = fma(df, df, s);
    };
    if (d % 4 == 0) {                                          // rows of both are aligned to what is read at once
        constexpr int U = 4;                                   // 512 columns in flight
        for (int j0 = 4 * lane; j0 < d; j0 += 128 * U) {
            float4 v[U];
            double2 a[U], b[U];
#pragma unroll
            for (int e = 0; e < U; ++e) {
                const int j = min(j0 + 128 * e, d - 4);
                const uint4 t = ld_stream16(xr + j);         // a point comes by once: L1 is left to the centroids
                v[e] = make_float4(__uint_as_float(t.x), __uint_as_float(t.y), __uint_as_float(t.z), __uint_as_float(t.w));
                a[e] = __ldg(reinterpret_cast<const double2 *>(m + j));
                b[e] = __ldg(reinterpret_cast<const double2 *>(m + j) + 1);
            }
#pragma unroll
            for (int e = 0; e < U; ++e)
                if (j0 + 128 * e < d) { take(v[e].x, a[e].x); take(v[e].y, a[e].y); take(v[e].z, b[e].x); take(v[e].w, b[e].y); }
        }
    } else {
#pragma unroll 8
        for (int j = lane; j < d; j += 32) take(__ldg(xr + j), __ldg(m + j));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) dist[p] = sqrt(s);
}

// Eq. (2) for cluster c = blockIdx.x: k times, the not yet taken member with the smallest (distance, index);
// out[c][r] = its index, -1 once the cluster has run out of members.  Distances are compared as the bit patterns of non-negative
// doubles.  A copy of them in shared memory (staged != 0: N words), NO_KEY for
// points that are no member or taken, serves all k searches; longer lists are read from global memory each time, taken[N]
// starting at zero.  SEL_NT threads.  Staged and k <= SEL_K: every warp takes the k first of its own points, without
// meeting the others, and one warp merges the lists (5 x 10 of 5000 points: 15 us; a meeting of the block per anchor and fp64
// comparisons 17).
constexpr int SEL_NT = 1024, SEL_STAGED = 25600, SEL_K = 32;
constexpr unsigned long long NO_KEY = ~0ull;
// The smallest (key, i) of the lanes, in every lane.
__device__ __forceinline__ void first_of_warp(unsigned long long &key, int &i) {
    const unsigned hi = (unsigned)(key >> 32), mh = __reduce_min_sync(0xffffffffu, hi);
    const unsigned lo = (unsigned)key, ml = __reduce_min_sync(0xffffffffu, hi == mh ? lo : ~0u);
    i = __reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? i : 0x7fffffff);
    key = (unsigned long long)mh << 32 | ml;
}
__global__ void __launch_bounds__(SEL_NT) select_anchors_kernel(const double *__restrict__ dist, const int *__restrict__ labels, int N, int k,
                                                                int staged, unsigned char *__restrict__ taken, int *__restrict__ out,
                                                                const Progress *__restrict__ pg, int last) {
    chain_wait();
    if (!pg->done && !last) return;
    extern __shared__ unsigned long long sel_key[];
    __shared__ unsigned long long list_key[SEL_NT / 32][SEL_K];
    __shared__ int list_i[SEL_NT / 32][SEL_K];
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (staged)
        for (int p0 = tid; p0 < N; p0 += 8 * SEL_NT) {           // eight points' loads in flight
            int l[8];
            double v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int p = min(p0 + e * SEL_NT, N - 1);
                l[e] = labels[p];
                v[e] = dist[p];
            }
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (p0 + e * SEL_NT < N) sel_key[p0 + e * SEL_NT] = l[e] == c ? (unsigned long long)__double_as_longlong(v[e]) : NO_KEY;
        }
    // this thread's first untaken point: ascending p, so the first of equals wins
    auto own_first = [&](unsigned long long &key, int &i) {
        key = NO_KEY;
        i = 0x7ffffffe;
        for (int p = tid; p < N; p += SEL_NT) {
            const unsigned long long v = staged ? sel_key[p] : (labels[p] == c && !taken[p] ? (unsigned long long)__double_as_longlong(dist[p]) : NO_KEY);
            if (v < key) { key = v; i = p; }
        }
    };
    unsigned long long key;
    int i;
    if (staged && k <= SEL_K) {
        unsigned long long own;
        int own_i;
        own_first(own, own_i);
        for (int r = 0; r < k; ++r) {
            key = own;
            i = own_i;
            first_of_warp(key, i);
            if (lane == 0) { list_key[warp][r] = key; list_i[warp][r] = i; }
            if (key != NO_KEY && i == own_i) {                   // only the owner of the point looks for its next one
                sel_key[i] = NO_KEY;
                own_first(own, own_i);
            }
        }
        __syncthreads();
        if (warp) return;
        int at = 0;                                              // lane = list
        for (int r = 0; r < k; ++r) {
            const int mine = at < k ? list_i[lane][at] : 0x7ffffffe;
            key = at < k ? list_key[lane][at] : NO_KEY;
            i = mine;
            first_of_warp(key, i);
            if (key != NO_KEY && i == mine) ++at;
            if (lane == 0) out[c * k + r] = key != NO_KEY ? i : -1;
        }
        return;
    }
    for (int r = 0; r < k; ++r) {
        own_first(key, i);
        first_of_warp(key, i);
        if (lane == 0) { list_key[warp][0] = key; list_i[warp][0] = i; }
        __syncthreads();
        if (warp == 0) {
            key = list_key[lane][0];
            i = list_i[lane][0];
            first_of_warp(key, i);
            if (lane == 0) {
                out[c * k + r] = key != NO_KEY ? i : -1;
                if (key != NO_KEY) {
                    if (staged) sel_key[i] = NO_KEY;
                    else taken[i] = 1;
                }
            }
        }
        __syncthreads();
    }
}

// What the host gets, into pinned memory, behind the ranking: the progress always, the other words (anchors, labels) and the centroids
// (out_mu, if given) once the rounds are done or the last ones have been.  (All of it copied behind every four rounds, done or not: 36.5 ms for
// 50 rounds of 300000 x 64, so 35.1.)
__global__ void __launch_bounds__(256) hand_over_kernel(const int *__restrict__ words, int n_progress, size_t n_words, int *__restrict__ host,
                                                        const double *__restrict__ mu, size_t n_mu, double *__restrict__ out_mu,
                                                        const Progress *__restrict__ pg, int last) {
    chain_wait();
    const size_t first = (size_t)blockIdx.x * 256 + threadIdx.x, stride = (size_t)gridDim.x * 256;
    const size_t n = pg->done || last ? n_words : n_progress;
    for (size_t i = first; i < n; i += stride) host[i] = words[i];
    if (out_mu && n == n_words)
        for (size_t i = first; i < n_mu; i += stride) out_mu[i] = mu[i];
}

}  // namespace anchors
}  // namespace knnssd
