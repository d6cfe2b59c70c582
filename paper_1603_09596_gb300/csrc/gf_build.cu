// gf_build.cu -- GPU forest construction (Alg. 1; Alg. 3 variance; Sec. 2.1 randomization;
// Sec. 3 "Median, variances", "Tree structure").
//
// All T trees are built together, one tree level per step.  At level l every tree has 2^l nodes;
// node a of tree t owns the positions [a n >> l, (a+1) n >> l) of the tree's point sequence, and
// every step is a stable partition of each node's positions into its two children, so each
// sequence ends as the tree's leaf permutation (leaves list their points in ascending id order
// because the sequences start as 0..n-1).
//
// Per node:
//   1. per-dimension variance of the node's points from the sums of (x - K) and (x - K)^2 with K
//      the node's first point (no cancellation), accumulated as compensated float32 pairs and
//      combined in float64, then var = (S2 - S1^2 / c) / (c - 1);
//   2. the t dimensions of largest variance, ranked by (variance desc, index asc), and the split
//      dimension s = D[u mod t] with u the node's SplitMix64 draw;
//   3. the split: points ordered by the unique 64-bit key (order-preserving bits of x_s, rk_t(id))
//      where rk_t is the tree's fmix32 permutation of the ids; the h = |left child| smallest keys
//      go left.  The h-th key is found by an 8-pass radix select; v = x_s of that key (+inf when
//      the right child is empty, which only leaf_size 1 can produce);
//   4. the stable partition.
// The split dimension needs the t largest variances only, so step 1 runs twice (per-node scope, points
// as they are): first for every dimension in 16-bit fixed point, with exact integer sums and a proven
// bound on the rounding (k_qsum, k_cand); then, in the arithmetic above, for the few dimensions that
// the bounds leave a place among the t largest (k_exact), which gives the same choice.  The integer
// sums are exact, so a right child's are its parent's minus its sibling's, and half of the points are
// read at most levels; at the root all trees hold the same points, and one of them is summed.  A
// node whose bounds leave more than CAND_MAX dimensions goes through the full-precision kernels.
// Levels whose nodes hold more than SMALL points use chunked kernels over all nodes of the level
// (the variance partial sums of the chunks are added in a fixed order, so the build is
// deterministic); deeper levels use one CTA per node that keeps the node's keys in shared memory.
#include "gf_internal.cuh"
#include "gf_device.cuh"
#include "gf_trace.cuh"

#include <algorithm>
#include <utility>
#include <vector>

namespace {

using namespace gfdev;

constexpr int NT = 256;        // threads per CTA in every build kernel
constexpr int DPT = 4;         // dimensions per thread per dimension block
constexpr int DB = NT * DPT;   // dimensions per block
constexpr int CHUNK = 2048;    // points per chunk on the chunked levels
constexpr int SMALL = 8192;    // nodes up to this size are built by one CTA
constexpr int TMAX = 64;       // largest supported t

// ---------------------------------------------------------------- random numbers
// SplitMix64 (Steele, Lea, Flood 2014) output number i of the stream starting at s0, and the
// MurmurHash3 32-bit finalizer (a bijection), from their published definitions.
__device__ __forceinline__ unsigned long long sm64_at(unsigned long long s0, unsigned long long i) {
    unsigned long long z = s0 + (i + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ unsigned fmix32(unsigned h) {
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return h;
}

struct BuildParams {
    const float *x;
    long long n;
    int d, ldx, T, t, shuffle, global_scope;
    unsigned long long seed;
    int2 *nodes;  // [T][2^L - 1]
    int nnodes;
    int *D;       // [TMAX] global top dims (global scope)
    const float *U;   // [T][d] Householder vectors, or null (trees on X itself)
    const float *W2;  // [T][n] 2 * u_t^T x_i of every point, when U is set
};

// Coordinate `dim` of point `id` as tree `tree` sees it: x itself, or its reflection (Sec. 2.2).
__device__ __forceinline__ float tree_coord(const BuildParams &P, int tree, int id, int dim) {
    const float x = __ldg(P.x + (size_t)id * P.ldx + dim);
    if (!P.U) return x;
    return reflect_coord(x, __ldg(P.W2 + (size_t)tree * P.n + id), __ldg(P.U + (size_t)tree * P.d + dim));
}

__device__ __forceinline__ unsigned long long tree_key(const BuildParams &P, int tree) {
    return sm64_at(P.seed, (unsigned long long)tree);
}

// tie-break order of point id in a tree whose key is tk
__device__ __forceinline__ unsigned rank_of(const BuildParams &P, unsigned long long tk, unsigned id) {
    return P.shuffle ? fmix32(id ^ (unsigned)sm64_at(tk, 0)) : id;
}

__device__ __forceinline__ unsigned ordered_bits(float f) {
    const unsigned u = __float_as_uint(f == 0.f ? 0.f : f);  // -0.0 reads as +0.0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float from_ordered(unsigned o) {
    return __uint_as_float((o & 0x80000000u) ? (o ^ 0x80000000u) : ~o);
}

__device__ __forceinline__ unsigned long long point_key(const BuildParams &P, unsigned long long tk, int tree,
                                                        int id, int s) {
    return ((unsigned long long)ordered_bits(tree_coord(P, tree, id, s)) << 32) | rank_of(P, tk, (unsigned)id);
}

// node geometry at level l
struct NodeGeo {
    int tree, a, j;
    long long lo, hi, mid;
};

__device__ __forceinline__ NodeGeo geo(const BuildParams &P, int l, long long seg) {
    NodeGeo g;
    g.tree = (int)(seg >> l);
    g.a = (int)(seg & ((1ll << l) - 1));
    g.j = (1 << l) - 1 + g.a;
    g.lo = ((long long)g.a * P.n) >> l;
    g.hi = ((long long)(g.a + 1) * P.n) >> l;
    g.mid = ((long long)(2 * g.a + 1) * P.n) >> (l + 1);
    return g;
}

// ---------------------------------------------------------------- variance

// Error-free transformations on float32 (Knuth's TwoSum; Dekker's product with an FMA): the
// result pair (s, e) satisfies s + e = a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Compensated sum hi + lo of float32 terms: hi is the running float32 sum, lo collects every
// rounding error of hi exactly (plus its own, second-order, rounding).
struct FF {
    float hi, lo;
};

__device__ __forceinline__ void ff_add(FF &a, float x, float xlo) {
    float s, e;
    two_sum(a.hi, x, s, e);
    a.hi = s;
    a.lo += e + xlo;
}

// Shifted sums over rows[0..cnt) for the dims dbase + tid + NT*u, u < DPT: S1 = sum (x - K),
// S2 = sum (x - K)^2 with K the node's first point.  Each difference is split exactly into
// float32 hi + lo, its square into a float32 product plus its exact FMA error (the lo^2 term is
// below 2^-48 relative and dropped), and both sums are compensated, so the relative error is of
// order cnt * 2^-48 -- float64 accuracy at float32 instruction rates (GB300's float64 rate is a
// small fraction of its float32 rate).
__device__ __forceinline__ void var_accum(const BuildParams &P, int tree, const int *__restrict__ rows,
                                          long long cnt, int krow, int dbase, double S1[DPT], double S2[DPT]) {
    float K[DPT], uu[DPT];
    int dim[DPT];
    FF s1[DPT], s2[DPT];
    const float *W2 = P.U ? P.W2 + (size_t)tree * P.n : nullptr;
#pragma unroll
    for (int u = 0; u < DPT; ++u) {
        dim[u] = dbase + threadIdx.x + NT * u;
        K[u] = dim[u] < P.d ? tree_coord(P, tree, krow, dim[u]) : 0.f;
        uu[u] = (P.U && dim[u] < P.d) ? __ldg(P.U + (size_t)tree * P.d + dim[u]) : 0.f;
        s1[u] = FF{0.f, 0.f};
        s2[u] = FF{0.f, 0.f};
    }
    auto add = [&](int u, float x) {
        float dh, dl;
        two_sum(x, -K[u], dh, dl);          // x - K = dh + dl exactly
        const float p = dh * dh;
        float pe = fmaf(dh, dh, -p);         // dh^2 = p + pe exactly
        pe = fmaf(2.f * dh, dl, pe);         // + 2 dh dl
        ff_add(s1[u], dh, dl);
        ff_add(s2[u], p, pe);
    };
    long long r = 0;
    for (; r + 4 <= cnt; r += 4) {
        float v[4][DPT], w2[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int id = __ldg(rows + r + q);
            const float *row = P.x + (size_t)id * P.ldx;
            w2[q] = W2 ? __ldg(W2 + id) : 0.f;
#pragma unroll
            for (int u = 0; u < DPT; ++u) v[q][u] = dim[u] < P.d ? __ldg(row + dim[u]) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < DPT; ++u) add(u, W2 ? reflect_coord(v[q][u], w2[q], uu[u]) : v[q][u]);
    }
    for (; r < cnt; ++r) {
        const int id = __ldg(rows + r);
        const float *row = P.x + (size_t)id * P.ldx;
        const float w2 = W2 ? __ldg(W2 + id) : 0.f;
#pragma unroll
        for (int u = 0; u < DPT; ++u) {
            const float x = dim[u] < P.d ? __ldg(row + dim[u]) : 0.f;
            add(u, W2 ? reflect_coord(x, w2, uu[u]) : x);
        }
    }
#pragma unroll
    for (int u = 0; u < DPT; ++u) {
        S1[u] = (double)s1[u].hi + (double)s1[u].lo;
        S2[u] = (double)s2[u].hi + (double)s2[u].lo;
    }
}

// Sums beyond float32's range (a spread above some 1e19) give infinities or NaN: such a variance counts
// as +inf, so that the rankings below compare values of a total order.  (With NaN among them the lanes of
// a ranking warp disagree on the winner and run out of dimensions.)
__device__ __forceinline__ double var_of(double S1, double S2, long long c) {
    if (c < 2) return 0.0;
    const double v = (S2 - S1 * S1 / (double)c) / (double)(c - 1);
    return v == v ? v : __longlong_as_double(0x7ff0000000000000ll);
}

__device__ __forceinline__ bool better(double va, int da, double vb, int db) {
    return va > vb || (va == vb && da < db);
}

// Warp 0 merges the block's variances vblk[0..nb) (dims dbase..) into the running top list
// (topv/topi, *have entries) and keeps the t best.  Called by all threads (syncs inside).
__device__ void topt_merge(const double *vblk, int nb, int dbase, double *topv, int *topi, int *have, int t) {
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const int h = *have, tot = h + nb;
        unsigned long long picked = 0ull;
        double nv[TMAX];
        int ni[TMAX];
        const int rounds = min(t, tot);
        for (int r = 0; r < rounds; ++r) {
            double bv = -1.0;
            int bd = 0x7fffffff, bslot = -1;
            for (int c = lane, k = 0; c < tot; c += 32, ++k) {
                if ((picked >> k) & 1ull) continue;
                const double v = c < h ? topv[c] : vblk[c - h];
                const int dd = c < h ? topi[c] : dbase + (c - h);
                if (bslot < 0 || better(v, dd, bv, bd)) { bv = v; bd = dd; bslot = k; }
            }
            // warp argmax over (bv, bd); lanes with no candidate carry bslot < 0
            int owner = lane;
            for (int o = 16; o > 0; o >>= 1) {
                const double ov = __shfl_xor_sync(FULL, bv, o);
                const int od = __shfl_xor_sync(FULL, bd, o);
                const int os = __shfl_xor_sync(FULL, bslot, o);
                const int ow = __shfl_xor_sync(FULL, owner, o);
                const bool take = os >= 0 && (bslot < 0 || better(ov, od, bv, bd) ||
                                              (ov == bv && od == bd && ow < owner));
                if (take) { bv = ov; bd = od; bslot = os; owner = ow; }
            }
            if (lane == owner) picked |= 1ull << bslot;
            nv[r] = bv;
            ni[r] = bd;
        }
        __syncwarp();
        if (lane == 0) {
            for (int r = 0; r < rounds; ++r) { topv[r] = nv[r]; topi[r] = ni[r]; }
            *have = rounds;
        }
    }
    __syncthreads();
}

// Split dimension of node j of a tree: top list -> D[u mod t]
__device__ __forceinline__ int pick_dim(const BuildParams &P, unsigned long long tk, int j, const int *D) {
    const unsigned long long u = sm64_at(tk, (unsigned long long)j + 1ull);
    return D[u % (unsigned long long)P.t];
}

// Stable partition of rows[0..cnt) by key < kh into out[0..h) and out[h..cnt).
__device__ void block_partition(const int *__restrict__ rows, const unsigned long long *keys, int cnt,
                                unsigned long long kh, int h, int *out, int *wcnt, int *sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (threadIdx.x == 0) { sh[0] = 0; sh[1] = 0; }
    __syncthreads();
    for (int base = 0; base < cnt; base += blockDim.x) {
        const int i = base + threadIdx.x;
        const bool in = i < cnt;
        const bool left = in && keys[i] < kh;
        const unsigned bl = __ballot_sync(FULL, left), bi = __ballot_sync(FULL, in);
        if (lane == 0) { wcnt[w] = __popc(bl); wcnt[32 + w] = __popc(bi & ~bl); }
        __syncthreads();
        int lo_l = sh[0], lo_r = sh[1];
        for (int q = 0; q < w; ++q) { lo_l += wcnt[q]; lo_r += wcnt[32 + q]; }
        const unsigned below = (1u << lane) - 1u;
        if (in) {
            const int id = rows[i];
            if (left) out[lo_l + __popc(bl & below)] = id;
            else out[h + lo_r + __popc(bi & ~bl & below)] = id;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int tl = 0, tr = 0;
            for (int q = 0; q < nw; ++q) { tl += wcnt[q]; tr += wcnt[32 + q]; }
            sh[0] += tl;
            sh[1] += tr;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- variance bounds in fixed point
//
// Coordinate j of every point as q = rint((x - low_j) / s_j) - 32500, 16 bits, s_j = range_j / 65000.
// (From the smallest value, not the middle: a dimension that spans few float32 steps has no middle to
// that precision, and q would leave 16 bits.)  Rounding moves a coordinate by at most QERR s_j (half
// a step, plus the float32 rounding of x - low_j, of the product and of 1 / s_j against s_j, together
// under 0.02 of a step at 65,000 steps), so over a node of c points the square root of
// the sum of squared deviations moves by at most QERR sqrt(c) s_j (triangle inequality), which bounds
// the variance on both sides.  What has to lie between the bounds is the variance as the full sums give
// it.  Over the up to 8192 points they add at a time, these are off by some 2^-38 of range_j^2 a point,
// a sixtieth of s_j^2 (ROUNDED allows half of it), as long as nothing under- or overflows: for range_j
// in [QLOW, QHIGH].  Below, squares may vanish altogether, but the sums stay at most c (range_j^2 + 2^-147): no
// lower bound, that upper one.  Above, nothing is known.  A level's sums read 2 bytes a coordinate instead of 4 and cost a few
// integer instructions instead of some 26 of compensated float32: 500,000 x 960, T = 32, a level took
// 15.4 ms of compensated sums (1.0e12 coordinates/s, bound by those instructions) and takes 2.1 ms of
// k_qsum over half the points (7.4 TB/s of rows, 6.8 of them from HBM: its limit) and 0.7 to 1.1 ms of the
// listed dimensions; the build with its bf16 copy and the export 174.6 -> 44.8 ms.
constexpr int CAND_MAX = 64;       // dimensions listed per node; -1: more, the node is summed in full
constexpr float QERR = 0.52f;
constexpr float QSTEPS = 65000.f;  // s_j = range_j / QSTEPS
constexpr float QLOW = 1e-16f, QHIGH = 1e14f;  // 2^-148, what a square may lose, is 0.2% of s_j^2; 2^31 range_j^2 is finite
constexpr float ROUNDED = 0.5f;
constexpr int QBIAS = 32500;       // half of them
constexpr int QCHUNK = 2048;       // points a CTA sums
// Points from which a build takes the fixed-point pass (ms without / with it, d = 128, T = 8: 1000 points
// 0.67 / 0.66, 2048 1.09 / 1.03, 5000 2.54 / 1.96; below, its launches and memory cost up to 0.1 ms).
constexpr long long QMIN = 2048;
constexpr long long QSUM_BYTES = 1ll << 30;  // sums kept for a level's nodes (and its parents')

__device__ __forceinline__ unsigned range_bits(float f) {
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// rng[j], rng[d + j]: smallest and largest value of dimension j, as ordered bits (preset ~0, 0)
__global__ void __launch_bounds__(256) k_range(const float *__restrict__ x, long long n, int d, int ldx, int rows, unsigned *rng) {
    const int j = blockIdx.y * 256 + threadIdx.x;
    if (j >= d) return;
    const long long r0 = (long long)blockIdx.x * rows, r1 = min(n, r0 + rows);
    float lo = __int_as_float(0x7f800000), hi = -lo;
#pragma unroll 8
    for (long long r = r0; r < r1; ++r) {
        const float v = __ldg(x + r * ldx + j);
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
    }
    atomicMin(rng + j, range_bits(lo));
    atomicMax(rng + d + j, range_bits(hi));
}

// qdim[j] = (low, 1 / s, s); s = 0: a constant dimension; s = -range: one below QLOW; s = +inf: one above
// QHIGH (every q the same in these three)
__global__ void k_qdim(const unsigned *__restrict__ rng, int d, float4 *qdim) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= d) return;
    const float lo = from_ordered(rng[j]), hi = from_ordered(rng[d + j]);
    const float range = hi - lo;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (range != 0.f) {
        if (range >= QLOW && range <= QHIGH) q = make_float4(lo, QSTEPS / range, range / QSTEPS, 0.f);
        else q.z = range < QLOW ? -range : __int_as_float(0x7f800000);
    }
    qdim[j] = q;
}

// xq[i][j], rows padded with zeros to ldq = round_up(d, 8).  tpr threads cover a row (or, blockIdx.y,
// a part of it), eight values each, and walk down the rows, so a dimension's (low, 1 / s) stays in
// registers and a warp reads and writes whole lines: bound by the bytes in and out (500,000 x 960:
// 1.98 ms with every thread fetching the eight dimensions' constants anew).
__global__ void __launch_bounds__(256) k_quant(const float *__restrict__ x, long long n, int d, int ldx, int ldq, int tpr,
                                               const float4 *__restrict__ qdim, short *xq) {
    const int col = threadIdx.x & (tpr - 1), grp = threadIdx.x / tpr, ngrp = 256 / tpr;
    const int j0 = (blockIdx.y * tpr + col) * 8;
    if (j0 >= ldq) return;
    float low[8], inv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float4 p = j0 + u < d ? __ldg(qdim + j0 + u) : make_float4(0.f, 0.f, 0.f, 0.f);
        low[u] = p.x;
        inv[u] = p.y;
    }
    const bool second = j0 + 4 < ldx;  // (ldx is a multiple of four, above j0)
    const long long step = (long long)gridDim.x * ngrp;
#pragma unroll 4
    for (long long i = (long long)blockIdx.x * ngrp + grp; i < n; i += step) {
        const float4 *src = reinterpret_cast<const float4 *>(x + i * ldx + j0);
        const float4 a = __ldg(src), b = second ? __ldg(src + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        unsigned w[4];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = j0 + u < d ? __float2int_rn((v[u] - low[u]) * inv[u]) - QBIAS : 0;
            if (u & 1) w[u / 2] |= (unsigned)q << 16;
            else w[u / 2] = (unsigned)q & 0xffffu;
        }
        *reinterpret_cast<uint4 *>(xq + i * ldq + j0) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// What a level's kernels do, settled on the device from the level before.
// On points whose bounds decide few nodes (a far outlier sets the step of its dimension; many dimensions
// tie) the pass, a quarter of a level's time where no sums are derived, would be spent for nothing.  After
// a level that left more than three quarters of its nodes undecided only a few nodes of a level are summed,
// until those are decided again; the host, which reads the outcome of the first level and of such probes,
// leaves the levels between probes alone.  Milliseconds, every dimension summed / the pass at every level /
// with this rule, one far outlier: 500,000 x 960, T = 32 166.1 / 187.6 / 169.8; 200,000 x 256, T = 8 27.8 /
// 31.0 / 29.2; 100,000 x 128, T = 1 4.7 / 5.9 / 5.4.  Two far points that the deep nodes leave behind, 200,000
// x 256, T = 8: 27.9 / 23.1 / 23.3.
enum QMode { Q_ALL, Q_LEFT, Q_PROBE, Q_NONE };  // every node, left ones (the right ones are derived), a few, none

constexpr int PROBE = 8;      // nodes a probe sums, but no more points than there are
constexpr int TALLY = 1024;   // nodes of a level that count (spread over all of them)
constexpr long long PROBE_OFTEN = 1ll << 28;  // coordinates times trees from which every second level is probed, else every fourth

struct QLevel {
    int tried, left;  // counted nodes summed, and those left undecided
    int sums;         // every node's sums are kept for the next level
};

__host__ __device__ inline bool q_decides(const QLevel &a) { return a.tried > 0 && 4 * a.left <= 3 * a.tried; }

struct QPlan {
    QLevel *lv;       // [levels], zeroed
    long long nodes;  // of this level
    int first, keeps, stride;  // first: no level before; keeps: a sums buffer holds the level; stride: levels between probes
};

__device__ __forceinline__ QMode q_mode(const QPlan &W, int l) {
    if (W.first) return Q_ALL;
    const QLevel a = W.lv[l - 1];
    if (!q_decides(a)) return l % W.stride == 0 ? Q_PROBE : Q_NONE;
    return W.keeps && a.sums ? Q_LEFT : Q_ALL;
}

// Whether seg is one of about `count` nodes spread over a level, from the middle of each stretch: a tree's
// first node and its last hold the outermost points.
__device__ __forceinline__ bool q_sampled(const QPlan &W, long long count, long long seg) {
    const long long step = max(1ll, W.nodes / count);
    return seg % step == step / 2;
}

// Whether k_qsum sums node seg.
__device__ __forceinline__ bool q_takes(const QPlan &W, QMode mode, int l, long long seg) {
    if (mode == Q_PROBE) return q_sampled(W, min((long long)PROBE, 1ll << l), seg);
    return mode == Q_ALL || (mode == Q_LEFT && !(seg & 1));
}

// Sums of q and q^2 over a chunk of a node, per dimension, exact.  tpr threads cover a row 16 bytes
// (eight values) each, 256 / tpr rows at a time, eight row loads in flight a thread; bound by the
// rows it reads (one level of 500,000 x 960, T = 32: half the points, 15.4 GB, 2.05 ms).
// sums[seg - node0][2][d]; several chunks a node are added with (integer, so order-independent) atomics to
// zeroed sums.
__global__ void __launch_bounds__(256) k_qsum(BuildParams P, QPlan W, int l, long long node0, int nch, int tpr,
                                              const int *__restrict__ pin, const short *__restrict__ xq, int ldq,
                                              long long *sums) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    long long *sh = reinterpret_cast<long long *>(smem_raw);  // [2][8 tpr]
    const long long idx = blockIdx.x / (unsigned)nch;
    const int ci = (int)(blockIdx.x - (unsigned)idx * (unsigned)nch);
    const long long seg = node0 + idx;
    if (!q_takes(W, q_mode(W, l), l, seg)) return;
    const NodeGeo g = geo(P, l, seg);
    const long long beg = min(g.lo + (long long)ci * QCHUNK, g.hi), end = nch == 1 ? g.hi : min(beg + QCHUNK, g.hi);
    const int *rows = pin + (size_t)g.tree * P.n;
    const int col = threadIdx.x & (tpr - 1), grp = threadIdx.x / tpr, ngrp = 256 / tpr;
    const int dbase = blockIdx.y * tpr * 8, j0 = dbase + col * 8;
    const bool live = j0 < ldq;
    int s1[8];
    long long s2[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        s1[u] = 0;
        s2[u] = 0;
    }
    const short *base = xq + (live ? j0 : 0);
    auto add = [&](const uint4 v) {
        const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int a = (int)(w[u] << 16) >> 16, b = (int)w[u] >> 16;
            s1[2 * u] += a;
            s1[2 * u + 1] += b;
            s2[2 * u] += (long long)a * a;
            s2[2 * u + 1] += (long long)b * b;
        }
    };
    constexpr int U = 8;
    long long r = beg + grp;
    for (; r + (U - 1) * ngrp < end; r += U * ngrp) {
        int id[U];
        uint4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) id[u] = __ldg(rows + r + u * ngrp);
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = __ldg(reinterpret_cast<const uint4 *>(base + (size_t)id[u] * ldq));
#pragma unroll
        for (int u = 0; u < U; ++u) add(v[u]);
    }
    for (; r < end; r += ngrp) add(__ldg(reinterpret_cast<const uint4 *>(base + (size_t)__ldg(rows + r) * ldq)));
    for (int q = ngrp - 1; q >= 0; --q) {  // the row groups add up in shared memory
        if (grp == q) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                long long *p1 = sh + col * 8 + u, *p2 = sh + tpr * 8 + col * 8 + u;
                *p1 = s1[u] + (q == ngrp - 1 ? 0 : *p1);
                *p2 = s2[u] + (q == ngrp - 1 ? 0 : *p2);
            }
        }
        __syncthreads();
    }
    long long *o = sums + (size_t)idx * 2 * P.d;
    for (int i = threadIdx.x; i < 2 * tpr * 8; i += 256) {
        const int h = i >= tpr * 8, j = dbase + i - h * tpr * 8;
        if (j >= P.d) continue;
        if (nch == 1) o[h * P.d + j] = sh[i];
        else atomicAdd(reinterpret_cast<unsigned long long *>(o + h * P.d + j), (unsigned long long)sh[i]);
    }
}

// Bounds of one dimension's sum of squared deviations over a node of c points, in units of
// (c - 1) x variance, from the sums of q and q^2: evaluated in float32 with room for its rounding
// (2^-20 of the second moment, 1e-5 of the result) and for the full sums' own.
__device__ __forceinline__ void dev_bounds(long long S1, long long S2, float c, float s, float &lo, float &hi) {
    if (s < 0.f || s > QHIGH) {
        lo = 0.f;
        hi = s < 0.f ? c * (s * s * 1.001f + 1e-37f) : __int_as_float(0x7f800000);
        return;
    }
    const float m2 = (float)S2, m1 = (float)S1;
    const float v = m2 - m1 * (m1 / c), e = m2 * 9.5367431640625e-7f, h = QERR * sqrtf(c);
    const float rl = fmaxf(sqrtf(fmaxf(v - e, 0.f)) - h, 0.f), rh = sqrtf(fmaxf(v + e, 0.f)) + h;
    lo = fmaxf(rl * rl - ROUNDED * c, 0.f) * (1.f - 1e-5f) * s * s;  // (s * s alone may vanish)
    hi = (rh * rh + ROUNDED * c) * (1.f + 1e-5f) * s * s;
}

// The dimensions that may be among the t of largest variance, per node: those whose upper bound
// reaches the t-th largest of the threads' largest lower bounds (t dimensions lie at or above that).
// Q_LEFT: an odd (right) node's sums are its parent's minus its left sibling's, and are kept.
// sums[slot], slot = blockIdx.x = seg - node0; ncand[seg] = -1: undecided, more than CAND_MAX or not summed.
__global__ void __launch_bounds__(NT) k_cand(BuildParams P, QPlan W, int l, long long node0,
                                             const float4 *__restrict__ qdim, const long long *__restrict__ parent,
                                             long long *sums, int *ncand, int *cand) {
    __shared__ float top[NT];
    __shared__ float tau;
    __shared__ int count;
    const long long seg = node0 + blockIdx.x;
    const QMode mode = q_mode(W, l);
    const bool right = mode == Q_LEFT && (seg & 1);
    if (seg == 0 && threadIdx.x == 0) W.lv[l].sums = W.keeps && mode <= Q_LEFT;
    if (!right && !q_takes(W, mode, l, seg)) {
        if (threadIdx.x == 0) ncand[seg] = -1;
        return;
    }
    const NodeGeo g = geo(P, l, seg);
    const float c = (float)(g.hi - g.lo);
    const bool counts = mode == Q_PROBE || q_sampled(W, TALLY, seg);
    if (counts && threadIdx.x == 0) atomicAdd(&W.lv[l].tried, 1);
    int *out = cand + seg * CAND_MAX;
    if (g.hi - g.lo < 2) {  // every variance is 0: the first t dimensions
        for (int r = threadIdx.x; r < P.t; r += NT) out[r] = r;
        if (threadIdx.x == 0) ncand[seg] = P.t;
        return;
    }
    long long *S = sums + (size_t)blockIdx.x * 2 * P.d;
    const long long *up = right ? parent + (size_t)(l == 1 ? 0 : seg >> 1) * 2 * P.d : nullptr;
    const long long *left = S - 2 * (size_t)P.d;
    float best = -1.f;
    for (int j = threadIdx.x; j < P.d; j += NT) {
        long long S1, S2;
        if (right) {
            S1 = up[j] - left[j];
            S2 = up[P.d + j] - left[P.d + j];
            S[j] = S1;
            S[P.d + j] = S2;
        } else {
            S1 = S[j];
            S2 = S[P.d + j];
        }
        float lo, hi;
        dev_bounds(S1, S2, c, qdim[j].z, lo, hi);
        best = fmaxf(best, lo);
    }
    top[threadIdx.x] = best;
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    int rank = 0;  // by (bound, thread)
    for (int i = 0; i < NT; ++i) rank += top[i] > best || (top[i] == best && i < (int)threadIdx.x);
    if (rank == P.t - 1) tau = best;
    __syncthreads();
    const float need = tau;
    for (int j = threadIdx.x; j < P.d; j += NT) {
        float lo, hi;
        dev_bounds(S[j], S[P.d + j], c, qdim[j].z, lo, hi);
        if (hi >= need) {
            const int at = atomicAdd(&count, 1);
            if (at < CAND_MAX) out[at] = j;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        ncand[seg] = count <= CAND_MAX ? count : -1;
        if (counts && count > CAND_MAX) atomicAdd(&W.lv[l].left, 1);
    }
}

// One dimension of var_accum over rows[0..cnt), cnt > 0, K the coordinate of krow: lane `lane` of
// the warp takes dimension `dim` (negative: none).  The points come in the same order and the sums in
// the same arithmetic, so they are var_accum's bit for bit.  Warp-wide.
__device__ __forceinline__ void var_accum_dim(const BuildParams &P, const int *__restrict__ rows, int cnt, int krow,
                                              int dim, double &S1, double &S2) {
    const int lane = threadIdx.x & 31;
    const float *xd = P.x + (dim < 0 ? 0 : dim);
    const float K = __ldg(xd + (size_t)krow * P.ldx);
    FF s1 = {0.f, 0.f}, s2 = {0.f, 0.f};
    auto add = [&](float x) {
        float dh, dl;
        two_sum(x, -K, dh, dl);
        const float p = dh * dh;
        float pe = fmaf(dh, dh, -p);
        pe = fmaf(2.f * dh, dl, pe);
        ff_add(s1, dh, dl);
        ff_add(s2, p, pe);
    };
    for (int r0 = 0; r0 < cnt; r0 += 32) {
        const int mine = r0 + lane < cnt ? __ldg(rows + r0 + lane) : krow;
        const int m = min(32, cnt - r0);
        int i = 0;
        for (; i + 8 <= m; i += 8) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = __ldg(xd + (size_t)__shfl_sync(FULL, mine, i + u) * P.ldx);
#pragma unroll
            for (int u = 0; u < 8; ++u) add(v[u]);
        }
        for (; i < m; ++i) add(__ldg(xd + (size_t)__shfl_sync(FULL, mine, i) * P.ldx));
    }
    S1 = (double)s1.hi + (double)s1.lo;
    S2 = (double)s2.hi + (double)s2.lo;
}

// The candidate of rank `want` by (variance desc, dimension asc); lane holds candidates lane and
// lane + 32 (d < 0: none).  Warp-wide.
__device__ int cand_rank(const double (&v)[2], const int (&d)[2], int want) {
    bool taken[2] = {d[0] < 0, d[1] < 0};
    int bd = -1;
    for (int r = 0; r <= want; ++r) {
        double bv = -1.0;
        bd = 0x7fffffff;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (!taken[h] && (bd == 0x7fffffff || better(v[h], d[h], bv, bd))) { bv = v[h]; bd = d[h]; }
        for (int o = 16; o > 0; o >>= 1) {
            const double ov = __shfl_xor_sync(FULL, bv, o);
            const int od = __shfl_xor_sync(FULL, bd, o);
            if (od != 0x7fffffff && (bd == 0x7fffffff || better(ov, od, bv, bd))) { bv = ov; bd = od; }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) taken[h] = taken[h] || d[h] == bd;
    }
    return bd;
}

__device__ __forceinline__ int draw_rank(const BuildParams &P, unsigned long long tk, int j) {
    return (int)(sm64_at(tk, (unsigned long long)j + 1ull) % (unsigned long long)P.t);
}

// The exact variances of a node's listed dimensions, a warp per node (nodes of at most SMALL points),
// and the node's split dimension.
__global__ void __launch_bounds__(NT) k_exact(BuildParams P, int l, long long nseg, const int *__restrict__ pin,
                                              const int *__restrict__ ncand, const int *__restrict__ cand, int *seg_s) {
    const long long seg = ((long long)blockIdx.x * NT + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (seg >= nseg) return;
    const int nc = ncand[seg];
    if (nc < 0) return;
    const NodeGeo g = geo(P, l, seg);
    const int *rows = pin + (size_t)g.tree * P.n + g.lo;
    const int cnt = (int)(g.hi - g.lo);
    double v[2] = {0.0, 0.0};
    int d[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        d[h] = lane + 32 * h < nc ? cand[seg * CAND_MAX + lane + 32 * h] : -1;
        if (32 * h < nc && cnt > 0) {
            double S1, S2;
            var_accum_dim(P, rows, cnt, rows[0], d[h], S1, S2);
            v[h] = var_of(S1, S2, cnt);
        }
    }
    const int s = cand_rank(v, d, draw_rank(P, tree_key(P, g.tree), g.j));
    if (lane == 0) seg_s[seg] = s;
}

// ---------------------------------------------------------------- small levels: CTA per node

struct SmallSmem {
    double vblk[DB];
    double topv[TMAX];
    int topi[TMAX];
    unsigned hist[256];
    int wcnt[64];
    int sh[4];
    int have;
    int s;
    int hs;
    unsigned long long pref;
};

// seg_s: the split dimensions already chosen (null: none), except for nodes of ncand < 0
__global__ void __launch_bounds__(NT) k_level_small(BuildParams P, int l, const int *__restrict__ pin,
                                                    const int *__restrict__ seg_s, const int *__restrict__ ncand,
                                                    int *pout) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallSmem &S = *reinterpret_cast<SmallSmem *>(smem_raw);
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(smem_raw + sizeof(SmallSmem));
    const NodeGeo g = geo(P, l, blockIdx.x);
    const int cnt = (int)(g.hi - g.lo), h = (int)(g.mid - g.lo);
    const int *rows = pin + (size_t)g.tree * P.n + g.lo;
    const unsigned long long tk = tree_key(P, g.tree);
    // 1-2: split dimension
    if (P.global_scope && l > 0) {
        if (threadIdx.x == 0) S.s = pick_dim(P, tk, g.j, P.D);
    } else if (seg_s && ncand[blockIdx.x] >= 0) {
        if (threadIdx.x == 0) S.s = seg_s[blockIdx.x];
    } else {
        if (threadIdx.x == 0) S.have = 0;
        for (int dbase = 0; dbase < P.d; dbase += DB) {
            double S1[DPT], S2[DPT];
            var_accum(P, g.tree, rows, cnt, rows[0], dbase, S1, S2);
#pragma unroll
            for (int u = 0; u < DPT; ++u) S.vblk[threadIdx.x + NT * u] = var_of(S1[u], S2[u], cnt);
            topt_merge(S.vblk, min(DB, P.d - dbase), dbase, S.topv, S.topi, &S.have, P.t);
        }
        if (threadIdx.x == 0) {
            S.s = pick_dim(P, tk, g.j, S.topi);
            if (P.global_scope)  // level 0 of the global scope: the root's top dims serve every node
                for (int r = 0; r < P.t; ++r) P.D[r] = S.topi[r];
        }
    }
    __syncthreads();
    const int s = S.s;
    // 3: keys, split key, split value
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) keys[i] = point_key(P, tk, g.tree, rows[i], s);
    __syncthreads();
    unsigned long long kh = ~0ull;
    float v = __int_as_float(0x7f800000);
    if (h < cnt) {
        kh = block_select(keys, cnt, h, S.hist, &S.pref, &S.hs);
        v = from_ordered((unsigned)(kh >> 32));
    }
    // 4: stable partition
    block_partition(rows, keys, cnt, kh, h, pout + (size_t)g.tree * P.n + g.lo, S.wcnt, S.sh);
    if (threadIdx.x == 0) P.nodes[(size_t)g.tree * P.nnodes + g.j] = make_int2(s, __float_as_int(v));
}

// ---------------------------------------------------------------- chunked levels

struct ChunkGeo {
    NodeGeo g;
    long long seg;
    int ci;
    long long beg, end;  // positions of the chunk (absolute within the tree's sequence)
};

__device__ __forceinline__ ChunkGeo chunk_geo(const BuildParams &P, int l, int nch, long long c) {
    ChunkGeo q;
    q.seg = c / nch;
    q.ci = (int)(c - q.seg * nch);
    q.g = geo(P, l, q.seg);
    q.beg = min(q.g.lo + (long long)q.ci * CHUNK, q.g.hi);
    q.end = min(q.beg + CHUNK, q.g.hi);
    return q;
}

// The exact partial sums of a node's listed dimensions, a warp per chunk: xpart[chunk][2][CAND_MAX].
__global__ void __launch_bounds__(NT) k_exact_chunk(BuildParams P, int l, int nch, long long nchunks, const int *__restrict__ pin,
                                                    const int *__restrict__ ncand, const int *__restrict__ cand, double *xpart) {
    const long long c = ((long long)blockIdx.x * NT + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (c >= nchunks) return;
    const ChunkGeo q = chunk_geo(P, l, nch, c);
    const int nc = ncand[q.seg], cnt = (int)(q.end - q.beg);
    const int *seq = pin + (size_t)q.g.tree * P.n;
    for (int h = 0; 32 * h < nc; ++h) {
        const int dim = lane + 32 * h < nc ? cand[q.seg * CAND_MAX + lane + 32 * h] : -1;
        double S1 = 0.0, S2 = 0.0;
        if (cnt > 0) var_accum_dim(P, seq + q.beg, cnt, seq[q.g.lo], dim, S1, S2);
        double *o = xpart + (size_t)c * 2 * CAND_MAX + 32 * h + lane;
        o[0] = S1;
        o[CAND_MAX] = S2;
    }
}

// Adds a node's chunk sums in chunk order, ranks its listed dimensions and picks the split dimension:
// a warp per node.  Level 0: tree 0's list and sums serve every tree.
__global__ void __launch_bounds__(NT) k_exact_pick(BuildParams P, int l, int nch, long long nseg, const int *__restrict__ ncand,
                                                   const int *__restrict__ cand, const double *__restrict__ xpart, int *seg_s) {
    const long long seg = ((long long)blockIdx.x * NT + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (seg >= nseg) return;
    const NodeGeo g = geo(P, l, seg);
    const long long from = l == 0 ? 0 : seg;
    const int nc = ncand[from];
    if (nc < 0) return;
    double v[2] = {0.0, 0.0};
    int d[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        d[h] = lane + 32 * h < nc ? cand[from * CAND_MAX + lane + 32 * h] : -1;
        double S1 = 0.0, S2 = 0.0;
        if (d[h] >= 0)
            for (int ci = 0; ci < nch; ++ci) {
                const double *p = xpart + ((size_t)from * nch + ci) * 2 * CAND_MAX + 32 * h + lane;
                S1 += p[0];
                S2 += p[CAND_MAX];
            }
        v[h] = var_of(S1, S2, g.hi - g.lo);
    }
    const int s = cand_rank(v, d, draw_rank(P, tree_key(P, g.tree), g.j));
    if (lane == 0) seg_s[seg] = s;
}

// variance partial sums of one chunk: part[c][0..d) = S1, part[c][d..2d) = S2
// (skip: the nodes whose split dimension is chosen already, ncand >= 0; level 0: tree 0's entry)
__global__ void __launch_bounds__(NT) k_var_partial(BuildParams P, int l, int nch, const int *__restrict__ pin,
                                                    const int *__restrict__ skip, double *part) {
    const ChunkGeo q = chunk_geo(P, l, nch, blockIdx.x);
    if (skip && skip[l == 0 ? 0 : q.seg] >= 0) return;
    const int *seq = pin + (size_t)q.g.tree * P.n;
    const int dbase = blockIdx.y * DB;
    double S1[DPT], S2[DPT];
    var_accum(P, q.g.tree, seq + q.beg, q.end - q.beg, seq[q.g.lo], dbase, S1, S2);
    double *o = part + (size_t)blockIdx.x * 2 * P.d;
#pragma unroll
    for (int u = 0; u < DPT; ++u) {
        const int dim = dbase + threadIdx.x + NT * u;
        if (dim < P.d) { o[dim] = S1[u]; o[P.d + dim] = S2[u]; }
    }
}

// add a node's chunk partials in chunk order, rank the dims, pick the split dimension
__global__ void __launch_bounds__(NT) k_var_combine(BuildParams P, int l, int nch, const int *__restrict__ skip,
                                                    const double *__restrict__ part, int *seg_s) {
    __shared__ double vblk[DB];
    __shared__ double topv[TMAX];
    __shared__ int topi[TMAX];
    __shared__ int have;
    if (skip && skip[l == 0 ? 0 : blockIdx.x] >= 0) return;
    const NodeGeo g = geo(P, l, blockIdx.x);
    const long long cnt = g.hi - g.lo;
    if (threadIdx.x == 0) have = 0;
    for (int dbase = 0; dbase < P.d; dbase += DB) {
#pragma unroll
        for (int u = 0; u < DPT; ++u) {
            const int dim = dbase + threadIdx.x + NT * u;
            double S1 = 0.0, S2 = 0.0;
            if (dim < P.d)
                for (int ci = 0; ci < nch; ++ci) {
                    const double *p = part + ((size_t)blockIdx.x * nch + ci) * 2 * P.d;
                    S1 += p[dim];
                    S2 += p[P.d + dim];
                }
            vblk[threadIdx.x + NT * u] = var_of(S1, S2, cnt);
        }
        topt_merge(vblk, min(DB, P.d - dbase), dbase, topv, topi, &have, P.t);
    }
    if (threadIdx.x == 0) {
        const unsigned long long tk = tree_key(P, g.tree);
        seg_s[blockIdx.x] = pick_dim(P, tk, g.j, topi);
        if (P.global_scope)
            for (int r = 0; r < P.t; ++r) P.D[r] = topi[r];
    }
}

// global scope below the root: s = D[u mod t]
__global__ void k_pick_global(BuildParams P, int l, long long nseg, int *seg_s) {
    const long long sg = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (sg >= nseg) return;
    const NodeGeo g = geo(P, l, sg);
    seg_s[sg] = pick_dim(P, tree_key(P, g.tree), g.j, P.D);
}

// keys of every position of every tree at level l
__global__ void k_keys(BuildParams P, int l, const int *__restrict__ pin, const int *__restrict__ seg_s,
                       unsigned long long *keys) {
    const long long tot = P.n * P.T;
    for (long long gidx = (long long)blockIdx.x * blockDim.x + threadIdx.x; gidx < tot;
         gidx += (long long)gridDim.x * blockDim.x) {
        const int tree = (int)(gidx / P.n);
        const long long p = gidx - (long long)tree * P.n;
        const long long a = ((((p + 1) << l)) - 1) / P.n;  // node owning position p
        const long long seg = ((long long)tree << l) + a;
        keys[gidx] = point_key(P, tree_key(P, tree), tree, pin[gidx], seg_s[seg]);
    }
}

// radix-select state of a node: prefix of the wanted key, its rank among the keys with that prefix
struct SelState {
    unsigned long long pref;
    int hrem;
    int active;  // 0 when the right child is empty (no split key)
};

__global__ void k_sel_init(BuildParams P, int l, long long nseg, SelState *st, unsigned *ghist) {
    const long long sg = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (sg >= nseg) return;
    const NodeGeo g = geo(P, l, sg);
    st[sg].pref = 0ull;
    st[sg].hrem = (int)(g.mid - g.lo);
    st[sg].active = g.mid < g.hi;
    for (int b = 0; b < 256; ++b) ghist[sg * 256 + b] = 0;
}

__global__ void __launch_bounds__(NT) k_sel_hist(BuildParams P, int l, int nch, int pass,
                                                 const unsigned long long *__restrict__ keys,
                                                 const SelState *__restrict__ st, unsigned *ghist) {
    __shared__ unsigned hist[256];
    const ChunkGeo q = chunk_geo(P, l, nch, blockIdx.x);
    const SelState s = st[q.seg];
    if (!s.active) return;  // uniform per CTA
    for (int b = threadIdx.x; b < 256; b += NT) hist[b] = 0;
    __syncthreads();
    const int shift = 56 - 8 * pass;
    const unsigned long long *kk = keys + (size_t)q.g.tree * P.n;
    for (long long base = q.beg; base < q.end; base += NT) {
        const long long i = base + threadIdx.x;
        bool act = false;
        unsigned bin = 0;
        if (i < q.end) {
            const unsigned long long k = kk[i];
            act = pass == 0 || ((k ^ s.pref) >> (shift + 8)) == 0ull;
            bin = (unsigned)(k >> shift) & 255u;
        }
        hist_add(hist, bin, act);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < 256; b += NT)
        if (hist[b]) atomicAdd(ghist + q.seg * 256 + b, hist[b]);
}

// one warp per node: find the bucket holding the wanted rank, extend the prefix, clear the histogram
__global__ void k_sel_pick(long long nseg, int pass, SelState *st, unsigned *ghist) {
    const long long sg = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (sg >= nseg) return;
    if (!st[sg].active) return;
    const int shift = 56 - 8 * pass;
    unsigned *hh = ghist + sg * 256;
    unsigned c[8], s = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) { c[q] = hh[8 * lane + q]; s += c[q]; }
    unsigned incl = s;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += v;
    }
    const unsigned before = incl - s;
    const unsigned hr = (unsigned)st[sg].hrem;
    const unsigned long long pref = st[sg].pref;
    __syncwarp();
    if (hr >= before && hr < incl) {
        unsigned acc = before;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (hr >= acc && hr < acc + c[q]) {
                st[sg].pref = pref | ((unsigned long long)(8 * lane + q) << shift);
                st[sg].hrem = (int)(hr - acc);
            }
            acc += c[q];
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) hh[8 * lane + q] = 0;
}

__device__ __forceinline__ unsigned long long split_key(const SelState &s) { return s.active ? s.pref : ~0ull; }

// number of left points (key < split key) per chunk
__global__ void __launch_bounds__(NT) k_part_count(BuildParams P, int l, int nch,
                                                   const unsigned long long *__restrict__ keys,
                                                   const SelState *__restrict__ st, int *lcount) {
    __shared__ int wsum[NT / 32];
    const ChunkGeo q = chunk_geo(P, l, nch, blockIdx.x);
    const unsigned long long kh = split_key(st[q.seg]);
    const unsigned long long *kk = keys + (size_t)q.g.tree * P.n;
    int c = 0;
    for (long long i = q.beg + threadIdx.x; i < q.end; i += NT) c += kk[i] < kh;
    c = __reduce_add_sync(FULL, c);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int w = 0; w < NT / 32; ++w) s += wsum[w];
        lcount[blockIdx.x] = s;
    }
}

// per node: chunk offsets of the left and right points; node record
__global__ void k_part_scan(BuildParams P, int l, int nch, long long nseg, const SelState *__restrict__ st,
                            const int *__restrict__ seg_s, const int *__restrict__ lcount, int *loff, int *roff) {
    const long long sg = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (sg >= nseg) return;
    const NodeGeo g = geo(P, l, sg);
    int accl = 0, accr = 0;
    for (int ci = 0; ci < nch; ++ci) {
        const long long c = sg * nch + ci;
        const long long beg = min(g.lo + (long long)ci * CHUNK, g.hi);
        const long long end = min(beg + CHUNK, g.hi);
        loff[c] = accl;
        roff[c] = accr;
        accl += lcount[c];
        accr += (int)(end - beg) - lcount[c];
    }
    const SelState s = st[sg];
    const float v = s.active ? from_ordered((unsigned)(s.pref >> 32)) : __int_as_float(0x7f800000);
    P.nodes[(size_t)g.tree * P.nnodes + g.j] = make_int2(seg_s[sg], __float_as_int(v));
}

__global__ void __launch_bounds__(NT) k_part_write(BuildParams P, int l, int nch, const int *__restrict__ pin,
                                                   const unsigned long long *__restrict__ keys,
                                                   const SelState *__restrict__ st, const int *__restrict__ loff,
                                                   const int *__restrict__ roff, int *pout) {
    __shared__ int wcnt[64];
    __shared__ int sh[4];
    const ChunkGeo q = chunk_geo(P, l, nch, blockIdx.x);
    const unsigned long long kh = split_key(st[q.seg]);
    const size_t toff = (size_t)q.g.tree * P.n;
    const int h = (int)(q.g.mid - q.g.lo);
    const int cnt = (int)(q.end - q.beg);
    // partition the chunk into a local view of the node's output: left part starts at
    // lo + loff, right part at lo + h + roff
    int *outL = pout + toff + q.g.lo + loff[blockIdx.x];
    int *outR = pout + toff + q.g.lo + h + roff[blockIdx.x];
    const int *rows = pin + toff + q.beg;
    const unsigned long long *kk = keys + toff + q.beg;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) { sh[0] = 0; sh[1] = 0; }
    __syncthreads();
    for (int base = 0; base < cnt; base += NT) {
        const int i = base + threadIdx.x;
        const bool in = i < cnt;
        const bool left = in && kk[i] < kh;
        const unsigned bl = __ballot_sync(FULL, left), bi = __ballot_sync(FULL, in);
        if (lane == 0) { wcnt[w] = __popc(bl); wcnt[32 + w] = __popc(bi & ~bl); }
        __syncthreads();
        int lo_l = sh[0], lo_r = sh[1];
        for (int qq = 0; qq < w; ++qq) { lo_l += wcnt[qq]; lo_r += wcnt[32 + qq]; }
        const unsigned below = (1u << lane) - 1u;
        if (in) {
            if (left) outL[lo_l + __popc(bl & below)] = rows[i];
            else outR[lo_r + __popc(bi & ~bl & below)] = rows[i];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int tl = 0, tr = 0;
            for (int qq = 0; qq < NT / 32; ++qq) { tl += wcnt[qq]; tr += wcnt[32 + qq]; }
            sh[0] += tl;
            sh[1] += tr;
        }
        __syncthreads();
    }
}

// W2[t][i] = 2 * u_t^T x_i, one warp per point and one lane per tree, summed over j ascending with
// every multiply and add rounded on its own (the order reflect_w2 uses for queries).
__global__ void k_reflect_w2(const float *__restrict__ x, int ldx, long long n, int d, int T,
                             const float *__restrict__ U, float *W2) {
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long i = warp; i < n; i += nw) {
        const float *row = x + i * ldx;
        for (int t0 = 0; t0 < T; t0 += 32) {
            const int t = t0 + lane;
            if (t < T) W2[(size_t)t * n + i] = reflect_w2(U + (size_t)t * d, row, d);
        }
    }
}

__global__ void k_iota(int *perm, long long n, int T) {
    const long long tot = n * T;
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < tot;
         g += (long long)gridDim.x * blockDim.x)
        perm[g] = (int)(g % n);
}

struct DevBuf {
    void *p = nullptr;
    ~DevBuf() { cudaFree(p); }
};

// Scratch of the fixed-point pass (k_qsum and after); without it the build takes the full-precision
// sums of every dimension.
struct QuantScratch {
    DevBuf mem;             // all of it (nine allocations and frees took 0.1 ms, half of a build of 300 points)
    unsigned *rng = nullptr;
    float4 *qdim = nullptr;
    short *xq = nullptr;
    long long *sums[2] = {nullptr, nullptr};
    int *ncand = nullptr, *cand = nullptr, *segs = nullptr;
    double *xpart = nullptr;
    QLevel *lv = nullptr;
    int ldq = 0, tpr = 8;
    long long cap = 0;      // nodes each sums buffer holds
    bool on = false;
    int first = -1;         // the first level it was taken for
    int stride = 1;         // levels between probes
    bool decides = true;    // as far as the host knows: the last level it read was decided
    bool takes(int l) const { return on && (decides || l % stride == 0); }
};

// Allocates it and makes the 16-bit copy of the points.  widest: nodes of the last level.
cudaError_t quant_prepare(QuantScratch &S, const BuildParams &P, long long widest, long long maxch, int sms, cudaStream_t st) {
    const int d = P.d;
    S.ldq = (d + 7) / 8 * 8;
    while (S.tpr < 128 && S.tpr * 8 < d) S.tpr <<= 1;
    S.cap = std::max(1ll, std::min(widest, QSUM_BYTES / (16ll * d)));
    size_t total = 0;
    auto place = [&](size_t bytes) {
        const size_t at = total;
        total += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t rng = place((size_t)d * 8), qdim = place((size_t)d * 16), xq = place((size_t)P.n * S.ldq * 2);
    const size_t sums[2] = {place((size_t)S.cap * d * 16), place((size_t)S.cap * d * 16)};
    const size_t ncand = place((size_t)widest * 4), cand = place((size_t)widest * CAND_MAX * 4), segs = place((size_t)widest * 4);
    const size_t xpart = place((size_t)maxch * 2 * CAND_MAX * 8), lv = place(32 * sizeof(QLevel));
    S.on = gf_dmalloc_if(&S.mem.p, total);
    if (!S.on) return cudaSuccess;
    char *m = (char *)S.mem.p;
    S.rng = (unsigned *)(m + rng);
    S.qdim = (float4 *)(m + qdim);
    S.xq = (short *)(m + xq);
    for (int i = 0; i < 2; ++i) S.sums[i] = (long long *)(m + sums[i]);
    S.ncand = (int *)(m + ncand);
    S.cand = (int *)(m + cand);
    S.segs = (int *)(m + segs);
    S.xpart = (double *)(m + xpart);
    S.lv = (QLevel *)(m + lv);
    S.stride = P.n * P.d * P.T >= PROBE_OFTEN ? 2 : 4;
    cudaError_t e = cudaMemsetAsync(S.lv, 0, 32 * sizeof(QLevel), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(S.rng, 0xff, (size_t)d * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(S.rng + d, 0, (size_t)d * 4, st);
    if (e != cudaSuccess) return e;
    const int rows = 256;
    k_range<<<dim3((unsigned)((P.n + rows - 1) / rows), (d + 255) / 256), 256, 0, st>>>(P.x, P.n, d, P.ldx, rows, S.rng);
    k_qdim<<<(d + 255) / 256, 256, 0, st>>>(S.rng, d, S.qdim);
    const int dblocks = (S.ldq + S.tpr * 8 - 1) / (S.tpr * 8);
    k_quant<<<dim3((unsigned)(sms * 8), dblocks), 256, 0, st>>>(P.x, P.n, d, P.ldx, S.ldq, S.tpr, S.qdim, S.xq);
    return cudaGetLastError();
}

// The candidate dimensions of every node of level l (level 0: of the points, once).
cudaError_t quant_level(QuantScratch &S, const BuildParams &P, int l, const int *seq, cudaStream_t st) {
    const long long nseg = l == 0 ? 1 : (long long)P.T << l;
    const long long cm = (P.n + (1ll << l) - 1) >> l;
    const int nch = (int)((cm + QCHUNK - 1) / QCHUNK);
    const int dblocks = (S.ldq + S.tpr * 8 - 1) / (S.tpr * 8);
    const size_t smem = (size_t)2 * S.tpr * 8 * 8;
    long long *sums = S.sums[l & 1], *parent = S.sums[(l & 1) ^ 1];
    if (S.first < 0) S.first = l;
    QPlan W;
    W.lv = S.lv;
    W.nodes = nseg;
    W.first = l == S.first;
    W.keeps = nseg <= S.cap;
    W.stride = S.stride;
    cudaError_t e = cudaSuccess;
    // (the left children's sums and the derived ones are all written before any child reads them: the left
    // ones in the first launch)
    for (long long n0 = 0; n0 < nseg && e == cudaSuccess; n0 += S.cap) {
        const long long nodes = std::min(S.cap, nseg - n0);
        if (nch > 1 && (e = cudaMemsetAsync(sums, 0, (size_t)nodes * P.d * 16, st)) != cudaSuccess) break;
        k_qsum<<<dim3((unsigned)(nodes * nch), dblocks), 256, smem, st>>>(P, W, l, n0, nch, S.tpr, seq, S.xq, S.ldq, sums);
        k_cand<<<(unsigned)nodes, NT, 0, st>>>(P, W, l, n0, S.qdim, parent, sums, S.ncand, S.cand);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && (W.first || !S.decides)) {
        QLevel got;
        e = cudaMemcpyAsync(&got, S.lv + l, sizeof got, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        S.decides = q_decides(got);
    }
    return e;
}

}  // namespace

static int build_levels(gf_forest *F, const gf_rand_params &rp, uint64_t seed, cudaStream_t st) {
    const long long n = F->n;
    const int T = F->T, L = F->L;
    DevBuf tmp, Dbuf;
    int r;
    if ((r = gf_dmalloc(&tmp.p, (size_t)T * n * 4))) return r;
    if ((r = gf_dmalloc(&Dbuf.p, TMAX * sizeof(int)))) return r;
    // sequences ping-pong so that the last level writes into F->perm
    int *bufA = (L % 2 == 0) ? F->perm : (int *)tmp.p;
    int *bufB = (L % 2 == 0) ? (int *)tmp.p : F->perm;
    k_iota<<<F->num_sms * 8, 256, 0, st>>>(bufA, n, T);
    GF_CUDA_TRY(cudaGetLastError());

    BuildParams P;
    P.x = F->x; P.n = n; P.d = F->d; P.ldx = F->ldx; P.T = T; P.t = rp.t; P.shuffle = rp.shuffle ? 1 : 0;
    P.global_scope = rp.var_scope == GF_VAR_GLOBAL; P.seed = seed; P.nodes = F->nodes;
    P.nnodes = (1 << L) - 1; P.D = (int *)Dbuf.p;
    P.U = F->U;
    P.W2 = nullptr;
    DevBuf w2buf;
    if (F->U) {  // every tree sees its reflected points (Sec. 2.2)
        if ((r = gf_dmalloc(&w2buf.p, (size_t)T * n * 4))) return r;
        k_reflect_w2<<<F->num_sms * 16, 256, 0, st>>>(F->x, F->ldx, n, F->d, T, F->U, (float *)w2buf.p);
        GF_CUDA_TRY(cudaGetLastError());
        P.W2 = (const float *)w2buf.p;
    }

    // chunked-level scratch, sized for the deepest chunked level
    int lc = -1;  // last chunked level
    for (int l = 0; l < L; ++l)
        if (((n + (1ll << l) - 1) >> l) > SMALL) lc = l;
    DevBuf part, keys, segs, sel, ghist, lcnt, loff, roff;
    long long maxch = 0, maxseg = 0;
    if (lc >= 0) {
        for (int l = 0; l <= lc; ++l) {
            const long long cm = (n + (1ll << l) - 1) >> l;
            const long long nch = (cm + CHUNK - 1) / CHUNK;
            maxch = std::max(maxch, ((long long)T << l) * nch);
            maxseg = std::max(maxseg, (long long)T << l);
        }
        if ((r = gf_dmalloc(&part.p, (size_t)maxch * 2 * F->d * sizeof(double)))) return r;
        if ((r = gf_dmalloc(&keys.p, (size_t)T * n * 8))) return r;
        if ((r = gf_dmalloc(&segs.p, (size_t)maxseg * 4))) return r;
        if ((r = gf_dmalloc(&sel.p, (size_t)maxseg * sizeof(SelState)))) return r;
        if ((r = gf_dmalloc(&ghist.p, (size_t)maxseg * 256 * 4))) return r;
        if ((r = gf_dmalloc(&lcnt.p, (size_t)maxch * 4))) return r;
        if ((r = gf_dmalloc(&loff.p, (size_t)maxch * 4))) return r;
        if ((r = gf_dmalloc(&roff.p, (size_t)maxch * 4))) return r;
    }
    int dev = 0, smem_optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t small_max = sizeof(SmallSmem) + (size_t)SMALL * 8;
    if (small_max > (size_t)smem_optin) return gf_fail(GF_EUNSUPPORTED, "build needs %zu B shared memory", small_max);
    GF_CUDA_TRY(cudaFuncSetAttribute(k_level_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)small_max));

    QuantScratch S;
    if (!F->U && !P.global_scope && L > 0 && n >= QMIN) GF_CUDA_TRY(quant_prepare(S, P, (long long)T << (L - 1), maxch, F->num_sms, st));

    const int ndb = (F->d + DB - 1) / DB;
    for (int l = 0; l < L; ++l) {
        GfRange level_range("gf_build: level");
        const long long cm = (n + (1ll << l) - 1) >> l;
        const long long nseg = (long long)T << l;
        if (cm <= SMALL) {
            const size_t smem = sizeof(SmallSmem) + (size_t)cm * 8;
            // (level 0 of a small set: every tree does its own root)
            const bool sel = S.takes(l) && l > 0;
            const int *chosen = sel ? S.ncand : nullptr;  // >= 0: the node's split dimension is in segs
            if (sel) {
                GF_CUDA_TRY(quant_level(S, P, l, bufA, st));
                k_exact<<<(unsigned)((nseg * 32 + NT - 1) / NT), NT, 0, st>>>(P, l, nseg, bufA, chosen, S.cand, S.segs);
            }
            k_level_small<<<(unsigned)nseg, NT, smem, st>>>(P, l, bufA, sel ? S.segs : nullptr, chosen, bufB);
            GF_CUDA_TRY(cudaGetLastError());
        } else {
            const int nch = (int)((cm + CHUNK - 1) / CHUNK);
            const long long nchunks = nseg * nch;
            int *seg_s = (int *)segs.p;
            SelState *ss = (SelState *)sel.p;
            unsigned *gh = (unsigned *)ghist.p;
            const unsigned gseg = (unsigned)((nseg + 255) / 256);
            if (!P.global_scope || l == 0) {
                const int *chosen = S.takes(l) ? S.ncand : nullptr;  // >= 0: the node's split dimension is in segs
                if (chosen) {
                    GF_CUDA_TRY(quant_level(S, P, l, bufA, st));
                    const long long own = l == 0 ? nch : nchunks;  // level 0: tree 0's chunks serve all
                    k_exact_chunk<<<(unsigned)((own * 32 + NT - 1) / NT), NT, 0, st>>>(
                        P, l, nch, own, bufA, chosen, S.cand, S.xpart);
                    k_exact_pick<<<(unsigned)((nseg * 32 + NT - 1) / NT), NT, 0, st>>>(
                        P, l, nch, nseg, chosen, S.cand, S.xpart, seg_s);
                }
                k_var_partial<<<dim3((unsigned)nchunks, ndb), NT, 0, st>>>(P, l, nch, bufA, chosen, (double *)part.p);
                k_var_combine<<<(unsigned)nseg, NT, 0, st>>>(P, l, nch, chosen, (const double *)part.p, seg_s);
            } else {
                k_pick_global<<<gseg, 256, 0, st>>>(P, l, nseg, seg_s);
            }
            k_keys<<<F->num_sms * 16, 256, 0, st>>>(P, l, bufA, seg_s, (unsigned long long *)keys.p);
            k_sel_init<<<gseg, 256, 0, st>>>(P, l, nseg, ss, gh);
            for (int pass = 0; pass < 8; ++pass) {
                k_sel_hist<<<(unsigned)nchunks, NT, 0, st>>>(P, l, nch, pass, (const unsigned long long *)keys.p, ss, gh);
                k_sel_pick<<<(unsigned)((nseg * 32 + 255) / 256), 256, 0, st>>>(nseg, pass, ss, gh);
            }
            k_part_count<<<(unsigned)nchunks, NT, 0, st>>>(P, l, nch, (const unsigned long long *)keys.p, ss,
                                                           (int *)lcnt.p);
            k_part_scan<<<gseg, 256, 0, st>>>(P, l, nch, nseg, ss, seg_s, (const int *)lcnt.p, (int *)loff.p,
                                              (int *)roff.p);
            k_part_write<<<(unsigned)nchunks, NT, 0, st>>>(P, l, nch, bufA, (const unsigned long long *)keys.p, ss,
                                                           (const int *)loff.p, (const int *)roff.p, bufB);
            GF_CUDA_TRY(cudaGetLastError());
        }
        std::swap(bufA, bufB);
    }
    GF_CUDA_TRY(cudaStreamSynchronize(st));
    return GF_OK;
}

static int build_any(const float *X, int64_t n, int32_t d, int32_t T, int32_t leaf_size, const gf_rand_params *rp_in,
                     uint64_t seed, const float *U_host, int32_t borrow_x, void *stream, gf_forest **out);

extern "C" int gf_build_ex(const float *X, int64_t n, int32_t d, int32_t T, int32_t leaf_size,
                           const gf_rand_params *rp_in, uint64_t seed, int32_t borrow_x, void *stream,
                           gf_forest **out) {
    return build_any(X, n, d, T, leaf_size, rp_in, seed, nullptr, borrow_x, stream, out);
}

extern "C" int gf_build_reflected(const float *X, int64_t n, int32_t d, int32_t T, int32_t leaf_size,
                                  const gf_rand_params *rp, uint64_t seed, const float *U_host,
                                  int32_t borrow_x, void *stream, gf_forest **out) {
    if (!U_host) return gf_fail(GF_EINVAL, "gf_build_reflected: U is null");
    return build_any(X, n, d, T, leaf_size, rp, seed, U_host, borrow_x, stream, out);
}

static int build_any(const float *X, int64_t n, int32_t d, int32_t T, int32_t leaf_size, const gf_rand_params *rp_in,
                     uint64_t seed, const float *U_host, int32_t borrow_x, void *stream, gf_forest **out) {
    GfRange range("gf_build");
    if (!out) return gf_fail(GF_EINVAL, "out is null");
    *out = nullptr;
    gf_rand_params rp;
    gf_rand_params_default(&rp);
    if (rp_in) rp = *rp_in;
    if (rp.householder && !U_host)
        return gf_fail(GF_EINVAL, "householder = 1 needs the per-tree vectors: use gf_build_reflected");
    if (U_host && rp.var_scope == GF_VAR_GLOBAL)
        return gf_fail(GF_EINVAL, "a global variance ranking is not defined for per-tree reflected points");
    if (rp.t < 1 || rp.t > d || rp.t > TMAX) return gf_fail(GF_EINVAL, "t=%d outside [1, min(d, %d)]", rp.t, TMAX);
    if (rp.var_scope != GF_VAR_NODE && rp.var_scope != GF_VAR_GLOBAL) return gf_fail(GF_EINVAL, "bad var_scope");
    if (n >= 1 && leaf_size >= 1) {
        const int L = depth_of(n, leaf_size);
        if (L > 0 && ((long long)T << (L - 1)) >= (1ll << 31))
            return gf_fail(GF_EUNSUPPORTED, "T * 2^(L-1) nodes per level exceeds 2^31");
    }
    cudaStream_t st = (cudaStream_t)stream;
    gf_forest *F = nullptr;
    int r = gf_forest_alloc(&F, X, n, d, T, leaf_size, borrow_x != 0, st);
    if (r) return r;
    if ((r = gf_check_finite(F->x, (int64_t)n * F->ldx, st))) { gf_forest_destroy(F); return r; }
    if (U_host && (r = gf_forest_set_U(F, U_host))) { gf_forest_destroy(F); return r; }
    if ((r = build_levels(F, rp, seed, st))) { gf_forest_destroy(F); return r; }
    *out = F;
    return GF_OK;
}

extern "C" int gf_build(const float *X, int64_t n, int32_t d, int32_t T, int32_t leaf_size,
                        const gf_rand_params *rp, uint64_t seed, gf_forest **out) {
    return gf_build_ex(X, n, d, T, leaf_size, rp, seed, 0, nullptr, out);
}
