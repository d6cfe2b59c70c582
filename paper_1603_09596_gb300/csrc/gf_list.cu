// gf_list.cu -- the staged per-query path: the search of gf_query.cu (Alg. 2; Eq. 1; Sec. 2.3;
// Sec. 3 "Distance computation") cut into launches, so that the work of a query is not bound to one
// CTA:
//   1. the leaves of every (query, tree): gf_descend, or one warp per pair (k_list_descend), or the
//      priority search's list;
//   2. admit: the points of a query's leaves are written to its candidate list once each (the "seen"
//      array of Sec. 2.3): through a hash set in shared memory, one CTA a query, or through a bitmap
//      over the point ids in device memory, a warp per 128 positions of a leaf;
//   3. score (k_list_score): CTAs take blocks of rows of the lists, a warp G rows at a time;
//   4. select (k_list_select): one CTA a query finds the `keep` smallest keys (distance, id), rescores
//      a screen's shortlist in float32 and writes the k nearest.
// A row's distance is warp_dist_g's, the same arithmetic in the same order as in the other per-query
// kernels, and a key holds (distance, id), so the answers are theirs bit for bit.
//
// Why: a query that is one CTA's alone reads its rows at that CTA's rate, and its descent,
// de-duplication and sorts stand between the reads.  Here step 3 is a flat pass over all rows of the
// batch that the whole chip shares.  Microseconds a call on one GB300, the one-CTA kernels -> this:
//   1 query, 10^6 x 960, T = 32, p = 1024, bf16 (10.9k rows)        1004 -> 41   (streaming)
//   199 queries, 5 10^5 x 960, T = 32, p = 512, bf16 (5.6k rows)     774 -> 357  (streaming)
//   27 queries, 5 10^4 x 512, T = 16, p = 256, float32               164 -> 40   (sort)
//   10^4 queries, 10^6 x 960, T = 32, p = 64, bf16 (1.24k rows)     8822 -> 3216 (sort)
//   5003 queries, 7 10^5 x 101, T = 32, p = 64, float32              902 -> 462  (sort)
// The scoring step is bound by the row loads: 9.8 TB/s of rows at 10^4 queries (most from L2, whose
// register loads peak at 10.6 TB/s), 7.2 TB/s at 199 queries (HBM).
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
constexpr int SEG = 128;           // positions of a leaf a warp admits at once (four a lane)
constexpr int ORDER_MIN = 512;     // batches from here on are walked in the order of tree 0's leaves

// The leaves of the batch: leaf[q][T] (one per tree) or the priority search's lists.
struct Leaves {
    const int *leaf;
    const unsigned *plist;
    const int *pn;
    int S;  // leaves per query
};

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

// One warp per (query, tree): the warp loads the five-level subtree below the current node at once
// (lane i: node i in breadth-first order, with the query's coordinate) and walks it through shuffles,
// so a path of L nodes costs ceil(L / 5) rounds of dependent loads instead of L.  For batches of a
// few thousand pairs, where the chip has warps to spare and the latency of the chain is what counts.
__global__ void __launch_bounds__(128) k_list_descend(ForestView F, const float *__restrict__ Q, long long pairs,
                                                      int *leaf) {
    const int lane = threadIdx.x & 31;
    const long long g = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g >= pairs) return;
    const long long qi = g / F.T;
    const int t = (int)(g - qi * F.T);
    const float *q = Q + qi * F.d;
    const int2 *nodes = F.nodes + (size_t)t * F.nnodes;
    const int lv = 31 - __clz(lane + 1);  // lane's level in the subtree (lanes 0..30)
    int j = 0;
    while (j < F.nnodes) {
        const long long node = (((long long)j + 1) << lv) - 1 + (lane + 1 - (1 << lv));
        bool left = false;
        if (lane < 31 && node < F.nnodes) {
            const int2 nd = __ldg(nodes + node);
            left = __ldg(q + nd.x) < __int_as_float(nd.y);
        }
        const unsigned lefts = __ballot_sync(FULL, left);
        int bi = 0;
        for (int l = 0; l < 5 && j < F.nnodes; ++l) {
            const int right = (lefts >> bi) & 1u ? 1 : 2;
            j = 2 * j + right;
            bi = 2 * bi + right;
        }
    }
    if (lane == 0) leaf[g] = j - F.nnodes;
}

// ---------------------------------------------------------------- admission

// One CTA per query: every id of its leaves goes into a hash set in shared memory (open addressing,
// linear probing; the table has at least twice as many slots as ids, so a probe ends) and, when it
// was not there, to the query's list.
__global__ void __launch_bounds__(256) k_list_admit_hash(ForestView F, Leaves V, long long q0, const int *__restrict__ order,
                                                         int slots, int cap, unsigned long long *keys, int *cnt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *table = reinterpret_cast<int *>(smem_raw);
    __shared__ int count;
    const long long w0 = blockIdx.x;
    const long long qi = order ? (long long)order[q0 + w0] : q0 + w0;
    for (int i = threadIdx.x; i < slots / 4; i += blockDim.x) reinterpret_cast<int4 *>(table)[i] = make_int4(-1, -1, -1, -1);
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int shift = __clz(slots) + 1;  // a multiplicative hash's top log2(slots) bits
    unsigned long long *out = keys + w0 * cap;
    auto admit = [&](int id) {
        bool fresh = false;
        if (id >= 0) {
            unsigned h = ((unsigned)id * 2654435769u) >> shift;
            for (;;) {
                const int old = atomicCAS(table + h, -1, id);
                if (old == -1) { fresh = true; break; }
                if (old == id) break;
                h = (h + 1) & (unsigned)(slots - 1);
            }
        }
        __syncwarp();
        const unsigned bl = __ballot_sync(FULL, fresh);
        int at = 0;
        if (lane == 0 && bl) at = atomicAdd(&count, __popc(bl));
        at = __shfl_sync(FULL, at, 0);
        if (fresh) out[at + __popc(bl & lt)] = (unsigned)id;
    };
    // two leaves of a warp in flight
    for (int s = w; s < V.S; s += 2 * nw) {
        long long b0, b1 = 0;
        const int c0 = leaf_of(F, V, qi, s, b0);
        const int c1 = s + nw < V.S ? leaf_of(F, V, qi, s + nw, b1) : 0;
        for (int i = lane; i - lane < max(c0, c1); i += 64) {
            int id[4];
            id[0] = i < c0 ? __ldg(F.perm + b0 + i) : -1;
            id[1] = i < c1 ? __ldg(F.perm + b1 + i) : -1;
            id[2] = i + 32 < c0 ? __ldg(F.perm + b0 + i + 32) : -1;
            id[3] = i + 32 < c1 ? __ldg(F.perm + b1 + i + 32) : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) admit(id[u]);
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

// Block `part` of B rows of query slot w0's list: ids in, keys (distance, id) out, in place.
template <int PREC, int NC, int G>
__global__ void __launch_bounds__(256, 2) k_list_score(ForestView F, const float *__restrict__ Q, long long q0,
                                                       const int *__restrict__ order, int parts, int B, int cap,
                                                       const int *__restrict__ cnt, unsigned long long *keys) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const long long w0 = blockIdx.x / (unsigned)parts;
    const int lo = (int)(blockIdx.x - (unsigned)w0 * (unsigned)parts) * B;
    const int nb = min(B, cnt[w0] - lo);
    if (nb <= 0) return;
    float *qs = reinterpret_cast<float *>(smem_raw);
    int *ids = reinterpret_cast<int *>(qs + ldq_of(F.d));
    const long long qi = order ? (long long)order[q0 + w0] : q0 + w0;
    unsigned long long *kq = keys + w0 * cap + lo;
    for (int j = threadIdx.x; j < nb; j += blockDim.x) ids[j] = (int)(unsigned)kq[j];
    load_query(Q + qi * F.d, F.d, qs);
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int j0 = w * G; j0 < nb; j0 += nw * G) {
        int rid[G];
        float dd[G];
#pragma unroll
        for (int g = 0; g < G; ++g) rid[g] = ids[min(j0 + g, nb - 1)];
        warp_dist_g<PREC, NC, G>(F, qs, rid, dd);
        unsigned long long key = KEY_NONE;
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (lane == g) key = make_key(dd[g], rid[g]);
        if (lane < G && j0 + lane < nb) kq[j0 + lane] = key;
    }
}

// ---------------------------------------------------------------- selection and rerank

// The `keep` smallest of a query's C keys.  The keys are dealt to GROUPS groups; the keep-th
// smallest group minimum bounds the keep-th key from above (each of the keep groups holds a key at
// or below it), and few other keys lie below it (about keep of them in all when the keys' order is
// unrelated to their size): those are gathered and sorted.  A list in an order that leaves more than
// SEL_BUF below the bound goes through the radix select.
template <int NCF, int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 3 : 1) k_list_select(ForestView F, const float *__restrict__ Q, long long q0, int k, int keep,
                                                      int rerank, const int *__restrict__ order, int cap,
                                                      const int *__restrict__ cnt, const unsigned long long *__restrict__ keys,
                                                      long long *ids, float *dists, int *ncand_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long *a = reinterpret_cast<unsigned long long *>(smem_raw);  // [SEL_BUF]
    float *qs = reinterpret_cast<float *>(a + SEL_BUF);                        // [ldq], rerank only
    __shared__ int sid[KEEP_MAX];
    __shared__ unsigned hist[256];
    __shared__ unsigned long long pref;
    __shared__ int nheld, hs;
    const long long w0 = blockIdx.x;
    const long long qi = order ? (long long)order[q0 + w0] : q0 + w0;
    const int C = cnt[w0];
    const unsigned long long *kq = keys + w0 * cap;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const unsigned lt = (1u << lane) - 1u;
    if (rerank) load_query(Q + qi * F.d, F.d, qs);
    unsigned long long bound = KEY_NONE;
    if (C > GROUPS) {
        unsigned long long mn = KEY_NONE;
#pragma unroll 4
        for (int i = tid; i < C; i += nt) {
            const unsigned long long v = kq[i];
            mn = v < mn ? v : mn;
        }
        a[tid] = mn;
        __syncthreads();
        if (tid < GROUPS) {
            for (int o = tid + GROUPS; o < nt; o += GROUPS) mn = a[o] < mn ? a[o] : mn;
        }
        __syncthreads();
        if (tid < GROUPS) a[tid] = mn;
        block_sort<unsigned long long>(a, GROUPS);
        bound = a[keep - 1];
        __syncthreads();
    }
    if (tid == 0) nheld = 0;
    __syncthreads();
    auto gather = [&]() {
        for (int b0 = 0; b0 < C; b0 += 4 * nt) {
            unsigned long long v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = b0 + u * nt + tid;
                v[u] = i < C ? kq[i] : KEY_NONE;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool in = v[u] != KEY_NONE && v[u] <= bound;
                const unsigned bl = __ballot_sync(FULL, in);
                if (bl) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&nheld, __popc(bl));
                    at = __shfl_sync(FULL, at, 0) + __popc(bl & lt);
                    if (in && at < SEL_BUF) a[at] = v[u];
                }
            }
        }
    };
    gather();
    __syncthreads();
    if (nheld > SEL_BUF) {  // (uniform: nheld is shared)
        bound = gfdev::block_select(kq, C, keep - 1, hist, &pref, &hs);
        if (tid == 0) nheld = 0;
        __syncthreads();
        gather();
        __syncthreads();
    }
    const int n = nheld;
    sort_keys(a, n);
    const int kn = min(keep, n);
    if (rerank) {
        for (int j = tid; j < kn; j += nt) sid[j] = (int)(unsigned)(a[j] & 0xffffffffu);
        __syncthreads();
        rescore_f32<NCF>(F, qs, sid, kn, a);
        sort_keys(a, kn);
    }
    write_topk(a, kn, k, ids + qi * k, dists + qi * k);
    if (tid == 0 && ncand_out) ncand_out[qi] = C;
}

// order keys (tree-0 leaf, query) of the batch
__global__ void k_list_order_keys(Leaves V, int L, long long m, unsigned long long *okeys) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const unsigned b = V.plist ? V.plist[i * V.S] & ((1u << L) - 1u) : (unsigned)V.leaf[i * V.S];
    okeys[i] = ((unsigned long long)b << 32) | (unsigned long long)(i & 0xffffffffll);
}

int nc_of(int chunks) { return chunks <= 32 ? 1 : chunks <= 64 ? 2 : chunks <= 128 ? 4 : chunks <= 256 ? 8 : 0; }

template <int PREC>
int chunks_of(const gf_forest *F) {
    return PREC == P_F32 ? F->ldx / 4 : PREC == P_BF16 ? F->ldb / 8 : F->ld8 / 16;
}

struct ListPlan {
    long long wave;     // queries per pass over the three steps
    int S, cap, slots;  // leaves per query, list capacity, hash slots (0: bitmaps)
    long long nwords;
    size_t leaf, pn, okeys, order, cnt, bits, keys, total;
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
    P.slots = 0;
    if (2 * tot <= HASH_MAX) {
        P.slots = 256;
        while (P.slots < 2 * tot) P.slots <<= 1;
    }
    P.nwords = P.slots ? 0 : (F->n + 31) / 32;
    const size_t per = (size_t)P.nwords * 4 + (size_t)P.cap * 8 + 4;
    P.wave = (long long)std::max<size_t>(1, std::min<size_t>((size_t)m, WAVE_BYTES / per));
    size_t o = 0;
    P.leaf = o; o = al(o + (size_t)m * P.S * 4);
    P.pn = o; o = al(o + (leaf_budget > 0 ? (size_t)m * 4 : 0));
    P.okeys = o; o = al(o + (m >= ORDER_MIN ? (size_t)m * 8 : 0));
    P.order = o; o = al(o + (m >= ORDER_MIN ? (size_t)m * 4 : 0));
    P.cnt = o; o = al(o + (size_t)P.wave * 4);
    P.bits = o; o = al(o + (size_t)P.wave * P.nwords * 4);  // right after the counters: zeroed with them
    P.keys = o; o = al(o + (size_t)P.wave * P.cap * 8);
    P.total = o;
    return P;
}

size_t select_smem(const gf_forest *F, bool rerank) { return (size_t)SEL_BUF * 8 + (rerank ? (size_t)ldq_of(F->d) * 4 : 0); }

template <int PREC, int NC, int G>
cudaError_t launch_score(const gf_forest *F, const float *Q, long long q0, long long nq, const int *order,
                         const ListPlan &P, const int *cnt, unsigned long long *keys, cudaStream_t st) {
    // rows per CTA: blocks of 256, shorter while the batch would not fill four CTAs an SM
    int B = 256;
    while (B > 8 * G && nq * ((P.cap + B - 1) / B) < 4ll * F->num_sms) B >>= 1;
    const int parts = (P.cap + B - 1) / B;
    const size_t smem = (size_t)ldq_of(F->d) * 4 + (size_t)B * 4;
    auto kern = k_list_score<PREC, NC, G>;
    if (smem > 40 * 1024) {  // (beside a few KB of static shared memory)
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kern<<<(unsigned)(nq * parts), 256, smem, st>>>(view_of(F), Q, q0, order, parts, B, P.cap, cnt, keys);
    return cudaGetLastError();
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
    if (smem > 40 * 1024) {  // (beside a few KB of static shared memory)
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kern<<<(unsigned)nq, NT, smem, st>>>(view_of(F), Q, q0, k, keep, rerank, order, P.cap, cnt, keys,
                                              (long long *)ids, dists, ncand_out);
    return cudaGetLastError();
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

int gf_launch_list(const gf_forest *F, const float *Q, int64_t m, int32_t k, int32_t precision, int32_t R,
                   cudaStream_t st, int64_t *ids, float *dists, const QueryExtra &x, bool *ran) {
    *ran = false;
    const bool prio = x.leaf_budget > 0, rerank = precision != GF_FP32;
    const int keep = rerank ? R : k;
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
    if (prio) r = gf_launch_prio_leaves(F, Q, m, P.S, (unsigned *)leaf, pn, st);
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
        unsigned long long *okeys = (unsigned long long *)(ws + P.okeys);
        order = (int *)(ws + P.order);
        k_list_order_keys<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(V, F->L, m, okeys);
        if ((e = gf_sort_order(m, okeys, order, st)) != cudaSuccess) return fail(e, "query order");
    }
    const int segs = (F->max_leaf + SEG - 1) / SEG;
    const int ncf = nc_of(F->ldx / 4);
    if ((e = gf_record(x, 0, st)) != cudaSuccess) return fail(e, "cudaEventRecord");
    for (long long q0 = 0; q0 < m; q0 += P.wave) {
        const long long nq = std::min<long long>(P.wave, m - q0);
        if (P.slots) {
            const size_t hs = (size_t)P.slots * 4;
            if (hs > 40 * 1024 && (e = cudaFuncSetAttribute(k_list_admit_hash, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                            (int)hs)) != cudaSuccess)
                return fail(e, "cudaFuncSetAttribute(k_list_admit_hash)");
            k_list_admit_hash<<<(unsigned)nq, 256, hs, st>>>(view_of(F), V, q0, order, P.slots, P.cap, keys, cnt);
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
