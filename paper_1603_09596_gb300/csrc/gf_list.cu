// gf_list.cu -- the staged per-query path: the search of gf_query.cu (Alg. 2; Eq. 1; Sec. 2.3;
// Sec. 3 "Distance computation") cut into launches, so that the work of a query is not bound to one
// CTA:
//   1. the leaves of every (query, tree): gf_descend, or one warp per pair (k_list_descend, or the
//      admission's own warps), or the priority search's list;
//   2. admit: the points of a query's leaves are written to its candidate list once each (the "seen"
//      array of Sec. 2.3): through a hash set or a bitmap over the point ids in shared memory, one CTA
//      a query; where the points are too many for that, through a bitmap in device memory, a warp per
//      128 positions of a leaf;
//   3. score (k_list_score): CTAs take blocks of rows of the lists, a warp G rows at a time;
//   4. select (k_list_select): one CTA a query finds the `keep` smallest keys (distance, id), rescores
//      a screen's shortlist in float32 and writes the k nearest.
// Calls too small for five launches run the same steps in one (k_list_one).
// A row's distance is warp_dist_g's, the same arithmetic in the same order as in the other per-query
// kernels, and a key holds (distance, id), so the answers are theirs bit for bit.
//
// Why: a query that is one CTA's alone reads its rows at that CTA's rate, and its descent,
// de-duplication and sorts stand between the reads.  Here step 3 is a flat pass over all rows of the
// batch that the whole chip shares.  Microseconds a call on one GB300, the one-CTA kernels -> this:
//   1 query, 10^6 x 960, T = 32, p = 1024, bf16 (10.9k rows)         950 -> 29   (streaming)
//   199 queries, 5 10^5 x 960, T = 32, p = 512, bf16 (5.6k rows)     742 -> 324  (streaming)
//   27 queries, 5 10^4 x 512, T = 16, p = 256, float32               160 -> 30   (sort)
//   2000 queries, 2 10^5 x 10^4, T = 24, p = 32, E4M3               3173 -> 2238 (sort)
//   10^4 queries, 10^6 x 960, T = 32, p = 64, bf16 (1.24k rows)     8798 -> 3037 (sort)
//   5003 queries, 7 10^5 x 101, T = 32, p = 64, float32              890 -> 419  (sort)
// The scoring step is bound by the row loads: 9.8 TB/s of rows at 10^4 queries, of which HBM serves 3.9
// (ncu) and L2 the rest, whose register loads peak at 10.6 TB/s; 7.2 TB/s at 199 queries, 6.5 of them from
// HBM (the 0.96 GB of the copy are read almost twice: half of the repeats miss L2); E4M3 rows of 10^4
// bytes 4.8 TB/s from HBM, which is not at its limit there.
#include "gf_internal.cuh"
#include "gf_device.cuh"
#include "gf_score.cuh"

#include <algorithm>
#include <climits>

namespace {

constexpr int KEEP_MAX = 128;      // longest k or R the selection keeps (it sorts 256 group minima)
constexpr int GROUPS = 256;        // groups of keys whose minima bound the keep-th key
constexpr int SEL_BUF = 1024;      // keys at or below that bound the selection holds
constexpr int HASH_MAX = 16384;    // slots of the shared-memory hash set (at least twice the ids)
constexpr int MAP_MAX = 1800000;   // points whose bitmap fits shared memory (225,000 bytes)
constexpr int SEG = 128;           // positions of a leaf a warp admits at once (four a lane)
constexpr int ONE_MAX = 640000;    // candidates of a call that runs in one launch,
constexpr int ONE_BYTES = 768 << 10;  // and bytes of a query's rows there, with fewer queries than SMs
constexpr int ORDER_MIN = 512;     // batches from here on are walked in the order of tree 0's leaves

// The leaves of the batch: leaf[q][T] (one per tree) or the priority search's lists.
struct Leaves {
    const int *leaf;
    const unsigned *plist;
    const int *pn;
    int S;  // leaves per query
};

// The steps' launches overlap (programmatic dependent launch): a kernel may start once every CTA of the
// one before it has begun, prepares what does not depend on it, and waits here for its end.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// slot s of query q: its first position in perm and its length (0 when the query has fewer leaves)
__device__ __forceinline__ int leaf_of(const ForestView &F, const Leaves &V, long long q, int s, long long &base) {
    long long t, b;
    if (V.plist) {
        if (s >= V.pn[q]) return 0;
        const unsigned code = V.plist[q * V.S + s];
        t = code >> F.L;
        b = code & ((1u << F.L) - 1u);
    } else {
        t = s;
        b = V.leaf[q * V.S + s];
    }
    const long long lo = (b * F.n) >> F.L, hi = ((b + 1) * F.n) >> F.L;
    base = t * F.n + lo;
    return (int)(hi - lo);
}

// The leaves of trees t0 .. t0 + N - 1 (below T) that query q reaches (Eq. 1), by a whole warp: per tree
// it loads the five-level subtree below the current node at once (lane i: node i in breadth-first
// order, with the query's coordinate) and walks it in the ballot of the comparisons, so a path of L
// nodes costs ceil(L / 5) rounds of dependent loads instead of L, and the trees go level in step.
// For batches of a few thousand (query, tree) pairs, where the chip has warps to spare and the
// latency of the chain is what counts.
template <int N>
__device__ __forceinline__ void warp_descend(const ForestView &F, int t0, const float *__restrict__ q, int (&leaf)[N]) {
    const int lane = threadIdx.x & 31;
    const int lv = 31 - __clz(lane + 1);  // lane's level in the subtree (lanes 0..30)
    int j[N];
#pragma unroll
    for (int h = 0; h < N; ++h) j[h] = 0;
    for (int l0 = 0; l0 < F.L; l0 += 5) {  // (the trees are perfect: every path has L nodes)
        unsigned lefts[N];
        int2 nd[N];
        bool in[N];
#pragma unroll
        for (int h = 0; h < N; ++h) {
            const long long node = (((long long)j[h] + 1) << lv) - 1 + (lane + 1 - (1 << lv));
            in[h] = lane < 31 && node < F.nnodes && t0 + h < F.T;
            if (in[h]) nd[h] = __ldg(F.nodes + (size_t)(t0 + h) * F.nnodes + node);
        }
#pragma unroll
        for (int h = 0; h < N; ++h) {
            const bool left = in[h] && __ldg(q + nd[h].x) < __int_as_float(nd[h].y);
            lefts[h] = __ballot_sync(FULL, left);
        }
#pragma unroll
        for (int h = 0; h < N; ++h) {
            int bi = 0;
            for (int l = l0; l < min(l0 + 5, F.L); ++l) {
                const int side = (lefts[h] >> bi) & 1u ? 1 : 2;
                j[h] = 2 * j[h] + side;
                bi = 2 * bi + side;
            }
        }
    }
#pragma unroll
    for (int h = 0; h < N; ++h) leaf[h] = j[h] - F.nnodes;
}

__global__ void __launch_bounds__(128) k_list_descend(ForestView F, const float *__restrict__ Q, long long pairs,
                                                      int *leaf) {
    const long long g = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    pdl_next();
    if (g >= pairs) return;
    const long long qi = g / F.T;
    int b[1];
    warp_descend<1>(F, (int)(g - qi * F.T), Q + qi * F.d, b);
    if ((threadIdx.x & 31) == 0) leaf[g] = b[0];
}

// ---------------------------------------------------------------- admission

// Whether `id` is new to the shared-memory set, adding it.
template <bool BITS>
__device__ __forceinline__ bool seen_first(int *table, int words, int id) {
    if (BITS) {
        const int bit = 1 << (id & 31);
        return !(atomicOr(table + (id >> 5), bit) & bit);
    }
    unsigned h = ((unsigned)id * 2654435769u) >> (__clz(words) + 1);  // the hash's top log2(words) bits
    for (;;) {
        const int old = atomicCAS(table + h, -1, id);
        if (old == -1) return true;
        if (old == id) return false;
        h = (h + 1) & (unsigned)(words - 1);
    }
}

// One CTA per query: every id of its leaves is tested and set in shared memory and, when it was not
// there, written to the query's list.  BITS: a bitmap over the point ids; else a hash set (open
// addressing, linear probing; the table has at least twice as many slots as ids, so a probe ends).
// A warp has eight ids a lane in flight: of one leaf, or (SHORT: leaves of at most 64) of four.
// DESC: one leaf per tree, and the warps find the leaves themselves (a launch less).
template <bool BITS, bool SHORT, int NT, bool DESC>
__global__ void __launch_bounds__(NT) k_list_admit(ForestView F, const float *__restrict__ Q, Leaves V, long long q0, const int *__restrict__ order,
                                                   int words, int cap, unsigned long long *keys, int *cnt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *table = reinterpret_cast<int *>(smem_raw);  // [words], a multiple of four
    __shared__ int count;
    const long long w0 = blockIdx.x;
    const int none = BITS ? 0 : -1;
    for (int i = threadIdx.x; i < words / 4; i += NT) reinterpret_cast<int4 *>(table)[i] = make_int4(none, none, none, none);
    if (threadIdx.x == 0) count = 0;
    pdl_wait();
    pdl_next();
    const long long qi = order ? (long long)order[q0 + w0] : q0 + w0;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    unsigned long long *out = keys + w0 * cap;
    constexpr int PER = SHORT ? 4 : 1;  // leaves at once
    constexpr int E = 8 / PER;          // ids a lane of each
    for (int s = w * PER; s < V.S; s += NT / 32 * PER) {
        long long base[PER];
        int c[PER], longest = 0, leaf[PER];
        if (DESC) warp_descend<PER>(F, s, Q + qi * F.d, leaf);
#pragma unroll
        for (int h = 0; h < PER; ++h) {
            base[h] = 0;
            c[h] = 0;
            if (s + h < V.S) {
                if (DESC) {
                    const long long b = leaf[h], lo = (b * F.n) >> F.L;
                    base[h] = (long long)(s + h) * F.n + lo;
                    c[h] = (int)((((b + 1) * F.n) >> F.L) - lo);
                } else {
                    c[h] = leaf_of(F, V, qi, s + h, base[h]);
                }
            }
            longest = max(longest, c[h]);
        }
        for (int i0 = 0; i0 < longest; i0 += 32 * E) {
            int id[8];
            unsigned bl[8];
            int total = 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + lane + 32 * (u % E);
                id[u] = i < c[u / E] ? __ldg(F.perm + base[u / E] + i) : -1;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const bool fresh = id[u] >= 0 && seen_first<BITS>(table, words, id[u]);
                __syncwarp();
                bl[u] = __ballot_sync(FULL, fresh);
                total += __popc(bl[u]);
            }
            int at = 0;
            if (lane == 0 && total) at = atomicAdd(&count, total);
            at = __shfl_sync(FULL, at, 0);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if ((bl[u] >> lane) & 1u) out[at + __popc(bl[u] & lt)] = (unsigned)id[u];
                at += __popc(bl[u]);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) cnt[w0] = count;
}

// One warp per SEG positions of a (query, leaf): test-and-set in the query's bitmap (zeroed before).
__global__ void __launch_bounds__(256) k_list_admit_bits(ForestView F, Leaves V, long long q0, long long nq,
                                                         const int *__restrict__ order, int segs, long long nwords,
                                                         unsigned *bitmaps, int cap, unsigned long long *keys, int *cnt) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const long long g = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long per = (long long)V.S * segs, w0 = g / per;
    pdl_next();
    if (w0 >= nq) return;
    const int r = (int)(g - w0 * per), s = r / segs, p0 = (r - s * segs) * SEG;
    const long long qi = order ? (long long)order[q0 + w0] : q0 + w0;
    long long base;
    const int c = leaf_of(F, V, qi, s, base);
    if (p0 >= c) return;
    unsigned *bm = bitmaps + w0 * nwords;
    int id[4];
    bool fresh[4];
    unsigned bl[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int p = p0 + lane + 32 * u;
        id[u] = p < c ? __ldg(F.perm + base + p) : -1;
    }
    int total = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
        fresh[u] = id[u] >= 0 && !(atomicOr(bm + (id[u] >> 5), 1u << (id[u] & 31)) & (1u << (id[u] & 31)));
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        bl[u] = __ballot_sync(FULL, fresh[u]);
        total += __popc(bl[u]);
    }
    int at = 0;
    if (lane == 0 && total) at = atomicAdd(cnt + w0, total);
    at = __shfl_sync(FULL, at, 0);
    unsigned long long *out = keys + w0 * cap;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (fresh[u]) out[at + __popc(bl[u] & lt)] = (unsigned)id[u];
        at += __popc(bl[u]);
    }
}

// ---------------------------------------------------------------- scoring

// 16-byte chunks of each of the G rows a lane has in flight when rows are longer than 4 KB: sixteen
// loads, as for shorter rows (E4M3, d = 10^4: 1.87 ms with two chunks, 1.70 ms with four; fewer rows at
// once read the query from shared memory more often: G = 2 2.5 ms).
constexpr int LONG_UNR = 4;
constexpr unsigned EARLY_GRID = 2048;  // CTAs of a scoring launch of few queries

// Block `part` of B rows of query slot w0's list: ids in, keys (distance, id) out, in place.
template <int PREC, int NC, int G>
__global__ void __launch_bounds__(256, 2) k_list_score(ForestView F, const float *__restrict__ Q, long long q0,
                                                       const int *__restrict__ order, int parts, int B, int cap,
                                                       const int *__restrict__ cnt, unsigned long long *keys) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const long long w0 = blockIdx.x / (unsigned)parts;
    const int lo = (int)(blockIdx.x - (unsigned)w0 * (unsigned)parts) * B;
    float *qs = reinterpret_cast<float *>(smem_raw);
    int *ids = reinterpret_cast<int *>(qs + ldq_of(F.d));
    // few queries: the query row comes in while the admission ends
    const bool early = !order && gridDim.x <= EARLY_GRID;
    if (early) load_query(Q + (q0 + w0) * F.d, F.d, qs);
    pdl_wait();
    pdl_next();
    const int nb = min(B, cnt[w0] - lo);
    if (nb <= 0) return;
    const long long qi = order ? (long long)order[q0 + w0] : q0 + w0;
    unsigned long long *kq = keys + w0 * cap + lo;
    for (int j = threadIdx.x; j < nb; j += blockDim.x) ids[j] = (int)(unsigned)kq[j];
    if (!early) load_query(Q + qi * F.d, F.d, qs);
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int j0 = w * G; j0 < nb; j0 += nw * G) {
        int rid[G];
        float dd[G];
#pragma unroll
        for (int g = 0; g < G; ++g) rid[g] = ids[min(j0 + g, nb - 1)];
        warp_dist_g<PREC, NC, G, LONG_UNR>(F, qs, rid, dd);
        unsigned long long key = KEY_NONE;
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (lane == g) key = make_key(dd[g], rid[g]);
        if (lane < G && j0 + lane < nb) kq[j0 + lane] = key;
    }
}

// ---------------------------------------------------------------- selection and rerank

struct SelectShared {
    unsigned hist[256];
    unsigned long long pref, bound;
    int sid[KEEP_MAX];
    int nheld, hs;
};

// The `keep` smallest (or all, if fewer) of the C distinct keys kq[0..C), ascending in a[] (shared
// memory, SEL_BUF entries, not overlapping kq); returns their number.  The keys are dealt to GROUPS
// groups; the keep-th smallest group minimum bounds the keep-th key from above (each of the keep
// groups holds a key at or below it), and few other keys lie below it (about keep in all when the
// keys' order is unrelated to their size): those are gathered and sorted.  A list in an order that
// leaves more than SEL_BUF below the bound goes through the radix select.  Up to NT KPT keys are read
// once, into registers.
template <int NT, int KPT>
__device__ int select_keys(const unsigned long long *kq, int C, int keep, unsigned long long *a, SelectShared &S) {
    const int tid = threadIdx.x, lane = tid & 31;
    const unsigned lt = (1u << lane) - 1u;
    const bool held = C <= NT * KPT;
    unsigned long long v[KPT];
    if (held) {
#pragma unroll
        for (int u = 0; u < KPT; ++u) v[u] = tid + u * NT < C ? kq[tid + u * NT] : KEY_NONE;
    }
    unsigned long long bound = KEY_NONE;
    if (tid == 0) S.nheld = 0;
    if (C > GROUPS) {
        unsigned long long mn = KEY_NONE;
        if (held) {
#pragma unroll
            for (int u = 0; u < KPT; ++u) mn = v[u] < mn ? v[u] : mn;
        } else {
#pragma unroll 8
            for (int i = tid; i < C; i += NT) {
                const unsigned long long x = kq[i];
                mn = x < mn ? x : mn;
            }
        }
        if (NT > GROUPS) {
            if (tid >= GROUPS) a[tid] = mn;
            __syncthreads();
            if (tid < GROUPS) {
#pragma unroll
                for (int o = GROUPS; o < NT; o += GROUPS) mn = a[tid + o] < mn ? a[tid + o] : mn;
            }
        }
        if (tid < GROUPS) a[tid] = mn;
        __syncthreads();
        if (tid < GROUPS) {
            int rank = 0;
#pragma unroll 8
            for (int j = 0; j < GROUPS; ++j) rank += a[j] < mn;
            if (rank == keep - 1) S.bound = mn;
        }
    }
    __syncthreads();
    if (C > GROUPS) bound = S.bound;
    auto put = [&](unsigned long long x) {
        const bool in = x != KEY_NONE && x <= bound;
        const unsigned bl = __ballot_sync(FULL, in);
        if (bl) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&S.nheld, __popc(bl));
            at = __shfl_sync(FULL, at, 0) + __popc(bl & lt);
            if (in && at < SEL_BUF) a[at] = x;
        }
    };
    auto gather = [&]() {
        if (held) {
#pragma unroll
            for (int u = 0; u < KPT; ++u) put(v[u]);
        } else {
            for (int b0 = 0; b0 < C; b0 += 4 * NT) {
                unsigned long long x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = b0 + u * NT + tid < C ? kq[b0 + u * NT + tid] : KEY_NONE;
#pragma unroll
                for (int u = 0; u < 4; ++u) put(x[u]);
            }
        }
    };
    gather();
    __syncthreads();
    if (S.nheld > SEL_BUF) {  // (uniform)
        bound = gfdev::block_select(kq, C, keep - 1, S.hist, &S.pref, &S.hs);
        if (tid == 0) S.nheld = 0;
        __syncthreads();
        gather();
        __syncthreads();
    }
    const int n = S.nheld;
    sort_distinct(a, n);
    return min(keep, n);
}

// One CTA per query: the keep best of its list, a screen's shortlist rescored in float32, the k nearest.
template <int NCF, int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 3 : 1) k_list_select(ForestView F, const float *__restrict__ Q, long long q0, int k, int keep,
                                                      int rerank, const int *__restrict__ order, int cap,
                                                      const int *__restrict__ cnt, const unsigned long long *__restrict__ keys,
                                                      long long *ids, float *dists, int *ncand_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long *a = reinterpret_cast<unsigned long long *>(smem_raw);  // [SEL_BUF]
    float *qs = reinterpret_cast<float *>(a + SEL_BUF);                        // [ldq], rerank only
    __shared__ SelectShared S;
    const long long w0 = blockIdx.x;
    if (rerank && !order) load_query(Q + (q0 + w0) * F.d, F.d, qs);
    pdl_wait();
    pdl_next();
    const long long qi = order ? (long long)order[q0 + w0] : q0 + w0;
    const int C = cnt[w0];
    if (rerank && order) load_query(Q + qi * F.d, F.d, qs);
    const int kn = select_keys<NT, NT == 256 ? 8 : 24>(keys + w0 * cap, C, keep, a, S);
    if (rerank) {
        for (int j = threadIdx.x; j < kn; j += NT) S.sid[j] = (int)(unsigned)(a[j] & 0xffffffffu);
        __syncthreads();
        rescore_f32<NCF>(F, qs, S.sid, kn, a);
        sort_distinct(a, kn);
    }
    write_topk(a, kn, k, ids + qi * k, dists + qi * k);
    if (threadIdx.x == 0 && ncand_out) ncand_out[qi] = C;
}

// The whole search of a query of at most SEL_BUF candidates in one launch, one CTA a query, for calls
// too small for the launches of the staged steps to pay.  Every warp descends its trees and admits
// their leaves' ids at once; the rows are scored G at a time a warp and selected as above.
template <int PREC, int NC, int NCF, int G>
__global__ void __launch_bounds__(256) k_list_one(ForestView F, const float *__restrict__ Q, int k, int keep, int words,
                                                  long long *ids, float *dists, int *ncand_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long *a = reinterpret_cast<unsigned long long *>(smem_raw);  // [SEL_BUF]
    unsigned long long *kq = a + SEL_BUF;                                      // [SEL_BUF]
    float *qs = reinterpret_cast<float *>(kq + SEL_BUF);                       // [ldq]
    int *table = reinterpret_cast<int *>(qs + ldq_of(F.d));                    // [words]
    __shared__ SelectShared S;
    __shared__ int count;
    const long long qi = blockIdx.x;
    const float *q = Q + qi * F.d;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int i = threadIdx.x; i < words / 4; i += 256) reinterpret_cast<int4 *>(table)[i] = make_int4(-1, -1, -1, -1);
    if (threadIdx.x == 0) count = 0;
    load_query(q, F.d, qs);
    __syncthreads();
    for (int t = w; t < F.T; t += 8) {
        int leaf[1];
        warp_descend<1>(F, t, q, leaf);
        const long long b = leaf[0], lo = (b * F.n) >> F.L;
        const int c = (int)((((b + 1) * F.n) >> F.L) - lo);
        const int32_t *src = F.perm + (size_t)t * F.n + lo;
        for (int i0 = 0; i0 < c; i0 += 128) {
            int id[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) id[u] = i0 + lane + 32 * u < c ? __ldg(src + i0 + lane + 32 * u) : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool fresh = id[u] >= 0 && seen_first<false>(table, words, id[u]);
                __syncwarp();
                const unsigned bl = __ballot_sync(FULL, fresh);
                int at = 0;
                if (lane == 0 && bl) at = atomicAdd(&count, __popc(bl));
                at = __shfl_sync(FULL, at, 0);
                if (fresh) kq[at + __popc(bl & lt)] = (unsigned)id[u];
            }
        }
    }
    __syncthreads();
    const int C = count;
    for (int j0 = w * G; j0 < C; j0 += 8 * G) {
        int rid[G];
        float dd[G];
#pragma unroll
        for (int g = 0; g < G; ++g) rid[g] = (int)(unsigned)kq[min(j0 + g, C - 1)];
        __syncwarp();
        warp_dist_g<PREC, NC, G>(F, qs, rid, dd);
        unsigned long long key = KEY_NONE;
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (lane == g) key = make_key(dd[g], rid[g]);
        if (lane < G && j0 + lane < C) kq[j0 + lane] = key;
    }
    __syncthreads();
    const int kn = select_keys<256, SEL_BUF / 256>(kq, C, keep, a, S);
    if (PREC != P_F32) {
        for (int j = threadIdx.x; j < kn; j += 256) S.sid[j] = (int)(unsigned)(a[j] & 0xffffffffu);
        __syncthreads();
        rescore_f32<NCF>(F, qs, S.sid, kn, a);
        sort_distinct(a, kn);
    }
    write_topk(a, kn, k, ids + qi * k, dists + qi * k);
    if (threadIdx.x == 0 && ncand_out) ncand_out[qi] = C;
}

// The batch in the order of the leaves it reaches in tree 0 (their first ORDER_BITS levels): one CTA,
// a counting sort over the leaves in shared memory.  Queries of one leaf come in no particular order.
constexpr int ORDER_BITS = 14;

__global__ void __launch_bounds__(1024) k_list_order(Leaves V, int L, long long m, int *order) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *bin = reinterpret_cast<int *>(smem_raw);  // [2^min(L, ORDER_BITS)]
    __shared__ int wsum[32];
    const int drop = max(0, L - ORDER_BITS), nb = 1 << (L - drop);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    auto leaf0 = [&](long long i) {
        const unsigned b = V.plist ? V.plist[i * V.S] & ((1u << L) - 1u) : (unsigned)V.leaf[i * V.S];
        return (int)(b >> drop);
    };
    for (int i = tid; i < nb; i += 1024) bin[i] = 0;
    __syncthreads();
    for (long long i = tid; i < m; i += 1024) atomicAdd(bin + leaf0(i), 1);
    __syncthreads();
    // exclusive scan: thread t owns the `per` bins from t per on
    const int per = (nb + 1023) / 1024, beg = min(nb, tid * per), end = min(nb, beg + per);
    int s = 0;
    for (int i = beg; i < end; ++i) s += bin[i];
    int inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
        int x = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        wsum[lane] = x;
    }
    __syncthreads();
    int run = inc - s + (w > 0 ? wsum[w - 1] : 0);
    for (int i = beg; i < end; ++i) {
        const int c = bin[i];
        bin[i] = run;
        run += c;
    }
    __syncthreads();
    for (long long i = tid; i < m; i += 1024) order[atomicAdd(bin + leaf0(i), 1)] = (int)i;
}

int nc_of(int chunks) { return chunks <= 32 ? 1 : chunks <= 64 ? 2 : chunks <= 128 ? 4 : chunks <= 256 ? 8 : 0; }

template <int PREC>
int chunks_of(const gf_forest *F) {
    return PREC == P_F32 ? F->ldx / 4 : PREC == P_BF16 ? F->ldb / 8 : F->ld8 / 16;
}

struct ListPlan {
    long long wave;     // queries per pass over the three steps
    int S, cap;         // leaves per query, list capacity
    int words;          // the shared-memory set's words (0: bitmaps in device memory)
    bool bits_in_smem;  // a bitmap, else a hash set
    long long nwords;   // words of a bitmap in device memory
    size_t leaf, pn, order, cnt, bits, keys, total;
};

// Device scratch: the leaves of the whole batch and its order, then one wave's counters, bitmaps
// and lists.  A wave is as many queries as fit WAVE_BYTES (at least one).
constexpr size_t WAVE_BYTES = (size_t)256 << 20;

ListPlan list_plan(const gf_forest *F, int64_t m, int leaf_budget) {
    auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
    ListPlan P;
    P.S = leaf_budget > 0 ? leaf_budget : F->T;
    P.cap = (int)std::min<long long>(F->n, (long long)P.S * F->max_leaf);  // distinct ids
    const long long tot = (long long)P.S * F->max_leaf;
    P.words = 0;
    P.bits_in_smem = false;
    if (2 * tot <= HASH_MAX) {
        P.words = 256;
        while (P.words < 2 * tot) P.words <<= 1;
    } else if (F->n <= MAP_MAX) {
        P.words = (int)((F->n + 127) / 128 * 4);
        P.bits_in_smem = true;
    }
    P.nwords = P.words ? 0 : (F->n + 31) / 32;
    const size_t per = (size_t)P.nwords * 4 + (size_t)P.cap * 8 + 4;
    P.wave = (long long)std::max<size_t>(1, std::min<size_t>((size_t)m, WAVE_BYTES / per));
    size_t o = 0;
    P.leaf = o; o = al(o + (size_t)m * P.S * 4);
    P.pn = o; o = al(o + (leaf_budget > 0 ? (size_t)m * 4 : 0));
    P.order = o; o = al(o + (m >= ORDER_MIN ? (size_t)m * 4 : 0));
    P.cnt = o; o = al(o + (size_t)P.wave * 4);
    P.bits = o; o = al(o + (size_t)P.wave * P.nwords * 4);  // right after the counters: zeroed with them
    P.keys = o; o = al(o + (size_t)P.wave * P.cap * 8);
    P.total = o;
    return P;
}

size_t select_smem(const gf_forest *F, bool rerank) { return (size_t)SEL_BUF * 8 + (rerank ? (size_t)ldq_of(F->d) * 4 : 0); }

// A launch that may begin while the kernel before it in the stream ends (its threads call pdl_wait).
template <typename... KP, typename... Args>
cudaError_t launch_after(void (*kern)(KP...), long long grid, int block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, static_cast<KP>(args)...);
}

template <bool BITS, bool SHORT, int NT, bool DESC>
cudaError_t launch_admit_d(const gf_forest *F, const float *Q, const Leaves &V, long long q0, long long nq, const int *order,
                         const ListPlan &P, unsigned long long *keys, int *cnt, cudaStream_t st) {
    auto kern = k_list_admit<BITS, SHORT, NT, DESC>;
    const size_t smem = (size_t)P.words * 4;
    const cudaError_t e = gf_smem_limit((const void *)kern, smem);
    if (e != cudaSuccess) return e;
    if (DESC) {  // the call's first launch
        kern<<<(unsigned)nq, NT, smem, st>>>(view_of(F), Q, V, q0, order, P.words, P.cap, keys, cnt);
        return cudaGetLastError();
    }
    return launch_after(kern, nq, NT, smem, st, view_of(F), Q, V, q0, order, P.words, P.cap, keys, cnt);
}

template <bool BITS, int NT>
cudaError_t launch_admit(const gf_forest *F, const float *Q, const Leaves &V, long long q0, long long nq, const int *order,
                         const ListPlan &P, bool desc, unsigned long long *keys, int *cnt, cudaStream_t st) {
    if (F->max_leaf <= 64)
        return desc ? launch_admit_d<BITS, true, NT, true>(F, Q, V, q0, nq, order, P, keys, cnt, st)
                    : launch_admit_d<BITS, true, NT, false>(F, Q, V, q0, nq, order, P, keys, cnt, st);
    return desc ? launch_admit_d<BITS, false, NT, true>(F, Q, V, q0, nq, order, P, keys, cnt, st)
                : launch_admit_d<BITS, false, NT, false>(F, Q, V, q0, nq, order, P, keys, cnt, st);
}

template <int PREC, int NC, int G>
cudaError_t launch_score(const gf_forest *F, const float *Q, long long q0, long long nq, const int *order,
                         const ListPlan &P, const int *cnt, unsigned long long *keys, cudaStream_t st) {
    // rows per CTA: blocks of 256, shorter while the batch would not fill four CTAs an SM
    int B = 256;
    while (B > 8 * G && nq * ((P.cap + B - 1) / B) < 4ll * F->num_sms) B >>= 1;
    const int parts = (P.cap + B - 1) / B;
    const size_t smem = (size_t)ldq_of(F->d) * 4 + (size_t)B * 4;
    auto kern = k_list_score<PREC, NC, G>;
    const cudaError_t e = gf_smem_limit((const void *)kern, smem);
    if (e != cudaSuccess) return e;
    return launch_after(kern, nq * parts, 256, smem, st, view_of(F), Q, q0, order, parts, B, P.cap, cnt, keys);
}

template <int PREC>
cudaError_t score_prec(const gf_forest *F, const float *Q, long long q0, long long nq, const int *order,
                       const ListPlan &P, const int *cnt, unsigned long long *keys, cudaStream_t st) {
    switch (nc_of(chunks_of<PREC>(F))) {
        case 1: return launch_score<PREC, 1, 8>(F, Q, q0, nq, order, P, cnt, keys, st);
        case 2: return launch_score<PREC, 2, 4>(F, Q, q0, nq, order, P, cnt, keys, st);
        case 4: return launch_score<PREC, 4, 4>(F, Q, q0, nq, order, P, cnt, keys, st);
        case 8: return launch_score<PREC, 8, 2>(F, Q, q0, nq, order, P, cnt, keys, st);
    }
    return launch_score<PREC, 0, 4>(F, Q, q0, nq, order, P, cnt, keys, st);
}

template <int NCF, int NT>
cudaError_t launch_select(const gf_forest *F, const float *Q, long long q0, long long nq, int k, int keep, bool rerank,
                          const int *order, const ListPlan &P, const int *cnt, const unsigned long long *keys,
                          int64_t *ids, float *dists, int *ncand_out, cudaStream_t st) {
    const size_t smem = select_smem(F, rerank);
    auto kern = k_list_select<NCF, NT>;
    const cudaError_t e = gf_smem_limit((const void *)kern, smem);
    if (e != cudaSuccess) return e;
    return launch_after(kern, nq, NT, smem, st, view_of(F), Q, q0, k, keep, rerank, order, P.cap, cnt, keys, (long long *)ids,
                        dists, ncand_out);
}

int one_words(const gf_forest *F) {
    int words = 256;
    while (words < 2ll * F->T * F->max_leaf) words <<= 1;
    return words;
}

size_t one_smem(const gf_forest *F) { return (size_t)SEL_BUF * 16 + (size_t)ldq_of(F->d) * 4 + (size_t)one_words(F) * 4; }

template <int PREC, int NC, int NCF>
cudaError_t launch_one(const gf_forest *F, const float *Q, int64_t m, int k, int keep, int64_t *ids, float *dists,
                       int *ncand_out, cudaStream_t st) {
    auto kern = k_list_one<PREC, NC, NCF, NC == 1 ? 8 : NC == 2 ? 4 : 2>;
    const size_t smem = one_smem(F);
    const cudaError_t e = gf_smem_limit((const void *)kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)m, 256, smem, st>>>(view_of(F), Q, k, keep, one_words(F), (long long *)ids, dists, ncand_out);
    return cudaGetLastError();
}

template <int PREC>
cudaError_t one_prec(const gf_forest *F, const float *Q, int64_t m, int k, int keep, int64_t *ids, float *dists,
                     int *ncand_out, cudaStream_t st) {
    const int nc = nc_of(chunks_of<PREC>(F)), ncf = nc_of(F->ldx / 4);
#define GF_ONE(A, B) \
    if (nc == A && ncf == B) return launch_one<PREC, A, B>(F, Q, m, k, keep, ids, dists, ncand_out, st);
    if constexpr (PREC == P_F32) {
        GF_ONE(1, 1) GF_ONE(2, 2) GF_ONE(4, 4) GF_ONE(8, 8)
    } else {
        GF_ONE(1, 1) GF_ONE(1, 2) GF_ONE(1, 4) GF_ONE(2, 4) GF_ONE(2, 8) GF_ONE(4, 8)
    }
#undef GF_ONE
    return cudaErrorInvalidValue;
}

int row_bytes(const gf_forest *F, int32_t precision) {
    return 16 * (precision == GF_FP32 ? chunks_of<P_F32>(F) : precision == GF_BF16_RERANK ? chunks_of<P_BF16>(F) : chunks_of<P_FP8>(F));
}

// One launch for the whole call: few candidates a query, rows of at most 4 KB, no reflections, little
// to score in all, and either little for one CTA (its rows come at some 50 GB/s) or about a CTA an SM.
// Microseconds a call, one launch / the staged steps: 640 candidates of 1 KB, m = 10: 23 / 32, 304:
// 29 / 46, 1000: 68 / 95; 640 of 3840 bytes, m = 10: 56 / 32, 100: 56 / 54, 304: 70 / 97, 1000: 257 / 254;
// 160 of 512 bytes, m = 100: 20 / 33, 1000: 25 / 50 (of which the host's part was about 19; now 13).
bool one_launch(const gf_forest *F, int64_t m, int32_t precision, const QueryExtra &x) {
    if (x.leaf_budget > 0 || F->U || F->cand_cap > SEL_BUF || nc_of(F->ldx / 4) == 0 || m * F->cand_cap > ONE_MAX) return false;
    return (int64_t)F->cand_cap * row_bytes(F, precision) <= ONE_BYTES || m >= F->num_sms;
}

// Whether a call that the sort kernel can answer is better left to it: few candidates a query, so that
// neither the staged steps' launches nor the single launch's eight warps a query pay.  Fitted to 1,400
// searches of 200 to 500,000 points, T = 1 to 64, at most 4096 candidates, 1 to 30,000 queries, every
// precision: the staged steps or the single launch were the slower ones in 148 (down to 0.56 of the
// sort kernel's speed), nearly all of them here; 14 remain (down to 0.81).  Microseconds, this path /
// sort kernel: single launch, leaves of 2, T = 62, m = 1151: 48 / 27; 1, T = 1, m = 2155: 44 / 31; staged,
// 6 candidates of 5.4 KB, m = 11: 22 / 14; 82 of 6 KB (k = 128), m = 551: 50 / 30; 34 of 20 bytes, m = 10,704:
// 150 / 114.
bool few_candidates(const gf_forest *F, int64_t m, int keep, int32_t precision, bool one) {
    const int leaf = F->max_leaf, cap = F->cand_cap, row = row_bytes(F, precision);
    if (one)
        return (row <= 1024 && ((leaf <= 8 && F->T >= 12 && m * F->T >= 4096) || (leaf <= 3 && F->T >= 32))) ||
               (row <= 512 && cap <= 8 && m >= 1024);
    const bool few = m * cap <= 4096 || row >= 4096;
    return (leaf <= 3 && (few || row <= 1024)) || ((cap <= 96 || cap <= keep) && few) || (cap <= 128 && row <= 512);
}

}  // namespace

bool gf_list_usable(const gf_forest *F, int64_t m, int32_t k, int32_t precision, int32_t R, const QueryExtra &x) {
    const int keep = precision == GF_FP32 ? k : R;
    if (keep > KEEP_MAX || x.workspace) return false;
    const int S = x.leaf_budget > 0 ? x.leaf_budget : F->T;
    if ((long long)S * F->max_leaf > (1 << 24) || (long long)m * S > INT_MAX / 2) return false;
    const size_t lim = 227 * 1024;
    return (size_t)ldq_of(F->d) * 4 + 256 * 4 <= lim && select_smem(F, true) + 4096 <= lim;
}

namespace {

// Whether work on st goes into a graph.
bool captured(cudaStream_t st) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &status) != cudaSuccess) {  // the legacy stream beside another's capture: the launches report it
        cudaGetLastError();
        return false;
    }
    return status != cudaStreamCaptureStatusNone;
}

}  // namespace

int gf_launch_list(const gf_forest *F, const float *Q, int64_t m, int32_t k, int32_t precision, int32_t R, bool sorts,
                   cudaStream_t st, int64_t *ids, float *dists, const QueryExtra &x, bool *ran) {
    *ran = false;
    const bool prio = x.leaf_budget > 0, rerank = precision != GF_FP32;
    const int keep = rerank ? R : k;
    const bool one = one_launch(F, m, precision, x);
    if (sorts && few_candidates(F, m, keep, precision, one)) return GF_OK;
    if (one) {
        *ran = true;
        cudaError_t e = gf_record(x, 0, st);
        if (e == cudaSuccess)
            e = precision == GF_FP32 ? one_prec<P_F32>(F, Q, m, k, keep, ids, dists, x.ncand_out, st)
                : precision == GF_BF16_RERANK ? one_prec<P_BF16>(F, Q, m, k, keep, ids, dists, x.ncand_out, st)
                                              : one_prec<P_FP8>(F, Q, m, k, keep, ids, dists, x.ncand_out, st);
        if (e == cudaSuccess) e = gf_record(x, 1, st);
        return e == cudaSuccess ? GF_OK : gf_cuda_fail(e, "k_list_one launch");
    }
    // In a graph the scratch would be an allocation node, and such a graph has one instance at a time and
    // cannot be a node of another: a call that the sort kernel can answer stays with it, which needs none.
    if (sorts && captured(st)) return GF_OK;
    const ListPlan P = list_plan(F, m, x.leaf_budget);
    char *ws = nullptr;
    if (gf_scratch_alloc((void **)&ws, P.total, st) != cudaSuccess) {
        cudaGetLastError();
        return GF_OK;  // not run: the caller takes a path that needs less scratch
    }
    *ran = true;
    int *leaf = (int *)(ws + P.leaf), *pn = (int *)(ws + P.pn), *cnt = (int *)(ws + P.cnt);
    unsigned *bits = (unsigned *)(ws + P.bits);
    unsigned long long *keys = (unsigned long long *)(ws + P.keys);
    auto fail = [&](cudaError_t e, const char *what) {
        gf_scratch_free(ws, st);
        return gf_cuda_fail(e, what);
    };
    cudaError_t e = cudaSuccess;
    int r = GF_OK;
    const long long pairs = (long long)m * F->T;
    // small batches: the admission's warps descend the trees
    const bool desc = !prio && !F->U && P.words && m < ORDER_MIN && pairs <= 16384;
    if (desc) {
    } else if (prio) r = gf_launch_prio_leaves(F, Q, m, P.S, (unsigned *)leaf, pn, st);
    else if (pairs <= 16384 && !F->U) {
        k_list_descend<<<(unsigned)((pairs + 3) / 4), 128, 0, st>>>(view_of(F), Q, pairs, leaf);
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(e, "k_list_descend launch");
    } else r = gf_descend(F, Q, m, leaf, st);
    if (r) {
        gf_scratch_free(ws, st);
        return r;
    }
    Leaves V;
    V.leaf = leaf;
    V.plist = prio ? (const unsigned *)leaf : nullptr;
    V.pn = pn;
    V.S = P.S;
    int *order = nullptr;
    if (m >= ORDER_MIN && x.order != GF_ORDER_GIVEN) {
        order = (int *)(ws + P.order);
        const size_t os = (size_t)4 << std::min(F->L, ORDER_BITS);
        if ((e = gf_smem_limit((const void *)k_list_order, os)) != cudaSuccess) return fail(e, "k_list_order's shared memory");
        k_list_order<<<1, 1024, os, st>>>(V, F->L, m, order);
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(e, "k_list_order launch");
    }
    const int segs = (F->max_leaf + SEG - 1) / SEG;
    const int ncf = nc_of(F->ldx / 4);
    if ((e = gf_record(x, 0, st)) != cudaSuccess) return fail(e, "cudaEventRecord");
    for (long long q0 = 0; q0 < m; q0 += P.wave) {
        const long long nq = std::min<long long>(P.wave, m - q0);
        if (P.words) {
            // few queries: a whole SM's threads for each
            e = P.bits_in_smem ? launch_admit<true, 1024>(F, Q, V, q0, nq, order, P, desc, keys, cnt, st)
                : nq <= F->num_sms ? launch_admit<false, 1024>(F, Q, V, q0, nq, order, P, desc, keys, cnt, st)
                                   : launch_admit<false, 256>(F, Q, V, q0, nq, order, P, desc, keys, cnt, st);
            if (e != cudaSuccess) return fail(e, "k_list_admit launch");
        } else {
            // the counters and the bitmaps lie side by side
            if ((e = cudaMemsetAsync(cnt, 0, P.bits - P.cnt + (size_t)nq * P.nwords * 4, st)) != cudaSuccess)
                return fail(e, "bitmap memset");
            const long long warps = nq * P.S * segs;
            k_list_admit_bits<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(view_of(F), V, q0, nq, order, segs, P.nwords, bits,
                                                                          P.cap, keys, cnt);
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(e, "candidate admission launch");
        e = precision == GF_FP32 ? score_prec<P_F32>(F, Q, q0, nq, order, P, cnt, keys, st)
            : precision == GF_BF16_RERANK ? score_prec<P_BF16>(F, Q, q0, nq, order, P, cnt, keys, st)
                                          : score_prec<P_FP8>(F, Q, q0, nq, order, P, cnt, keys, st);
        if (e != cudaSuccess) return fail(e, "k_list_score launch");
        if (q0 + P.wave >= m && (e = gf_record(x, 1, st)) != cudaSuccess) return fail(e, "cudaEventRecord");
        // few queries with long lists: more threads a query
        const bool wide = nq <= F->num_sms && P.cap > 4096;
#define GF_SEL(N)                                                                                                       \
    (wide ? launch_select<N, 512>(F, Q, q0, nq, k, keep, rerank, order, P, cnt, keys, ids, dists, x.ncand_out, st)      \
          : launch_select<N, 256>(F, Q, q0, nq, k, keep, rerank, order, P, cnt, keys, ids, dists, x.ncand_out, st))
        e = ncf == 1 ? GF_SEL(1) : ncf == 2 ? GF_SEL(2) : ncf == 4 ? GF_SEL(4) : ncf == 8 ? GF_SEL(8) : GF_SEL(0);
#undef GF_SEL
        if (e != cudaSuccess) return fail(e, "k_list_select launch");
    }
    gf_scratch_free(ws, st);
    return GF_OK;
}
