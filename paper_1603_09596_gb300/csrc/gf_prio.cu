// gf_prio.cu -- the leaves a query checks under Alg. 2's shared priority queue (Sec. 2.3).
//
// For each query, in the order of Alg. 2:
//   * every tree is descended from its root (Eq. 1); each node passed pushes the child not taken
//     with key |q_s - v|; the leaf reached is checked (reading: these first T leaves count toward
//     the budget, so a budget of T leaves is exactly the one-leaf-per-tree search);
//   * then, while fewer than `budget` leaves were checked, the entry of smallest
//     (key, tree, node) is taken from the queue and descended the same way to one more leaf.
// The keys are computed in float64 (the difference of two floats is exact there), so the order,
// including ties, is exactly the CPU oracle's.  A key is non-negative, so its IEEE bits order as the
// value does: the queue compares the bits as 64-bit integers (GB300's float64 compare rate is a
// small fraction of its integer rate).
//
// One warp per query.  The queue is two sorted arrays in shared memory: a large one A and a small
// one B (at most 64 entries).  A pop takes the smaller of their heads.  The entries a descent pushes
// (at most L <= 30, one a lane) are merged into B by the warp; once B holds more than 32 it is merged
// into A in place (from the top down), so the large array moves once every few pops instead of at every
// one.  The first phase (one entry per tree and level) merges into A directly.  Entries ranked beyond
// the number of pops still to come can never be taken and are dropped, so A never holds more than
// `budget` - T entries past its start.  The order of the pops is that of a single sorted queue: every
// pop takes the smallest (key, tree, node) held.  The output is the list of leaves in the order
// checked, encoded (tree << L) | leaf.
//
// A pop is a chain of dependent steps (head, subtree loads, walk, merge), so what counts is the length
// of that chain and the warps an SM holds beside each other.  Merges exchange entries by shuffles and
// ballots, and an entry's new place comes from counting, not from binary searches through shared
// memory (six dependent loads an entry); an entry is a key of 8 bytes and a (tree, node) of 4.
// 10^4 queries, L = 14, T = 32, 512 leaves: 5.75 ms with searches and 16-byte entries (16 warps an SM),
// 2.71 ms now (32).
#include "gf_internal.cuh"
#include "gf_trace.cuh"

#include <algorithm>

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int PRIO_WARPS = 4;   // at most this many warps (queries) per CTA
constexpr int PQ_BCAP = 64;     // entries of the small queue array

// bits of the float64 key |q_s - v| (>= 0): they order as the value does
__device__ __forceinline__ unsigned long long pq_key(float qs, float v) {
    return (unsigned long long)__double_as_longlong(fabs((double)qs - (double)v));
}

// A queue entry: the key, and the place (tree << (L + 1)) | node that breaks ties by (tree, node).
// Place: 32 bits where T 2^(L+1) <= 2^32, else 64.
template <typename Place>
struct PQE {
    unsigned long long key;
    Place at;
};

template <typename Place>
__device__ __forceinline__ bool pq_less(const PQE<Place> &a, const PQE<Place> &b) {
    return a.key < b.key || (a.key == b.key && a.at < b.at);
}

template <typename Place>
__device__ __forceinline__ PQE<Place> pq_inf() {
    PQE<Place> e;
    e.key = ~0ull;
    e.at = ~(Place)0;
    return e;
}

// A queue array in shared memory, keys and places apart.
template <typename Place>
struct PQArray {
    unsigned long long *key;
    Place *at;
    __device__ __forceinline__ PQE<Place> get(int i) const {
        PQE<Place> e;
        e.key = key[i];
        e.at = at[i];
        return e;
    }
    __device__ __forceinline__ void set(int i, const PQE<Place> &e) const {
        key[i] = e.key;
        at[i] = e.at;
    }
    __device__ __forceinline__ PQArray from(int i) const {
        PQArray a;
        a.key = key + i;
        a.at = at + i;
        return a;
    }
};

template <typename Place>
__device__ __forceinline__ PQE<Place> pq_shfl(const PQE<Place> &e, int src) {
    PQE<Place> r;
    r.key = __shfl_sync(FULL, e.key, src);
    r.at = __shfl_sync(FULL, e.at, src);
    return r;
}

// Merge the nb entries held one a lane (in any order) into the sorted array b[head .. head + cnt), cnt + nb
// <= PQ_BCAP, and leave the first min(cnt + nb, keep) of the merged order at b[0 ..); returns their number.
// Every entry's place is the number of entries below it, counted as the new ones go round the warp.
template <typename Place>
__device__ int pq_insert(const PQArray<Place> &b, int head, int cnt, const PQE<Place> &mine, int nb, int keep) {
    const int lane = threadIdx.x & 31;
    const bool in0 = lane < cnt, in1 = lane + 32 < cnt;
    const PQE<Place> b0 = in0 ? b.get(head + lane) : pq_inf<Place>(), b1 = in1 ? b.get(head + lane + 32) : pq_inf<Place>();
    int up0 = 0, up1 = 0, pos = keep;
    for (int i = 0; i < nb; ++i) {
        const PQE<Place> e = pq_shfl(mine, i);
        const bool l0 = pq_less(b0, e), l1 = pq_less(b1, e), lm = lane < nb && pq_less(mine, e);
        up0 += !l0;
        up1 += !l1;
        const int below = __popc(__ballot_sync(FULL, in0 && l0)) + __popc(__ballot_sync(FULL, in1 && l1)) +
                          __popc(__ballot_sync(FULL, lm));
        if (lane == i) pos = below;
    }
    __syncwarp();  // every lane has read its entries
    if (in0 && lane + up0 < keep) b.set(lane + up0, b0);
    if (in1 && lane + 32 + up1 < keep) b.set(lane + 32 + up1, b1);
    if (lane < nb && pos < keep) b.set(pos, mine);
    __syncwarp();
    return min(cnt + nb, keep);
}

// Merge the sorted array s[0..ns) (ns <= PQ_BCAP, not overlapping a) into the sorted array a[0..na) in
// place, keeping the first min(na + ns, keep) entries of the merged order in a[]; returns their
// number.  a[] must have room for them.  Entry i of s goes p_i entries of a further on (a binary search a
// lane); an entry j of a moves up by the number of p_i <= j, so a is moved from the top down to the
// smallest p_i, 32 entries at a time, each group read before it is written.  Warp-wide.
template <typename Place>
__device__ int pq_merge_into(const PQArray<Place> &a, int na, const PQArray<Place> &s, int ns, int keep) {
    const int lane = threadIdx.x & 31;
    int p[2];
    PQE<Place> e[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h;
        e[h] = i < ns ? s.get(i) : pq_inf<Place>();
        int lo = 0, hi = i < ns ? na : 0;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (pq_less(a.get(mid), e[h])) lo = mid + 1;
            else hi = mid;
        }
        p[h] = i < ns ? lo : 0x7fffffff;
    }
    const int first = __shfl_sync(FULL, p[0], 0);
    for (int top = na; top > first; top -= 32) {
        const int low = top - 32, j = low + lane;
        PQE<Place> x = pq_inf<Place>();
        if (j >= 0) x = a.get(j);
        int up = __popc(__ballot_sync(FULL, p[0] < low)) + __popc(__ballot_sync(FULL, p[1] < low));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            unsigned here = __ballot_sync(FULL, p[h] >= low && p[h] < top);
            while (here) {
                const int src = __ffs(here) - 1;
                here &= here - 1;
                up += __shfl_sync(FULL, p[h], src) <= j;
            }
        }
        __syncwarp();
        if (j >= 0 && up > 0 && j + up < keep) a.set(j + up, x);
        __syncwarp();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h;
        if (i < ns && i + p[h] < keep) a.set(i + p[h], e[h]);
    }
    __syncwarp();
    return min(na + ns, keep);
}

__device__ __forceinline__ unsigned leaf_code(int tree, int leaf, int L) {
    return ((unsigned)tree << L) | (unsigned)leaf;
}

// entries of the large array: what the pops after the first T leaves can take
__host__ __device__ inline int prio_cap(int budget, int T) { return budget > T ? budget - T : 1; }

// per-warp shared memory: the two arrays' keys, then their places, then one reflection weight per tree
__host__ __device__ inline size_t prio_warp_bytes(int budget, int T, size_t place) {
    const size_t n = prio_cap(budget, T) + PQ_BCAP;
    return (n * 8 + n * place + (size_t)T * 4 + 15) / 16 * 16;
}

template <typename Place>
__global__ void __launch_bounds__(PRIO_WARPS * 32) k_prio_leaves(ForestView F, const float *__restrict__ Q,
                                                                long long m, int budget, unsigned *leaves, int *nleaves) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int cap = prio_cap(budget, F.T);
    PQArray<Place> qa, qb;
    qa.key = reinterpret_cast<unsigned long long *>(smem_raw + (size_t)w * prio_warp_bytes(budget, F.T, sizeof(Place)));
    qb.key = qa.key + cap;
    qa.at = reinterpret_cast<Place *>(qb.key + PQ_BCAP);
    qb.at = qa.at + cap;
    float *w2s = reinterpret_cast<float *>(qb.at + PQ_BCAP);
    const int nn = (1 << F.L) - 1;
    const int nwq = blockDim.x >> 5;
    for (long long qi = (long long)blockIdx.x * nwq + w; qi < m; qi += (long long)gridDim.x * nwq) {
        const float *q = Q + qi * F.d;
        unsigned *out = leaves + qi * budget;
        int acnt = 0, ahead = 0, bcnt = 0, bhead = 0, checked = 0;  // A holds [ahead, acnt), B [bhead, bcnt)
        // ---- first descent of every tree, 32 trees at a time, one level per merge
        for (int t0 = 0; t0 < F.T; t0 += 32) {
            const int t = t0 + lane;
            const bool act = t < F.T;
            float w2 = 0.f;
            if (act && F.U) {  // the query's reflection for this tree (Sec. 2.3)
                w2 = reflect_w2(F.U + (size_t)t * F.d, q, F.d);
                w2s[t] = w2;
            }
            int j = 0;
            for (int l = 0; l < F.L; ++l) {
                PQE<Place> e = pq_inf<Place>();
                if (act) {
                    const int2 nd = __ldg(F.nodes + (size_t)t * F.nnodes + j);
                    const float qx = __ldg(q + nd.x);
                    const float qs = F.U ? reflect_coord(qx, w2, __ldg(F.U + (size_t)t * F.d + nd.x)) : qx;
                    const float v = __int_as_float(nd.y);
                    const bool left = qs < v;
                    e.key = pq_key(qs, v);
                    e.at = ((Place)t << (F.L + 1)) | (Place)(left ? 2 * j + 2 : 2 * j + 1);  // the child not taken
                    j = left ? 2 * j + 1 : 2 * j + 2;
                }
                const int nb = min(32, F.T - t0);
                pq_insert(qb, 0, 0, e, nb, PQ_BCAP);
                acnt = pq_merge_into(qa, acnt, qb, nb, max(0, budget - F.T));
            }
            if (act && t < budget) out[t] = leaf_code(t, j - nn, F.L);
        }
        checked = min(F.T, budget);
        // ---- pops in queue order
        while (checked < budget && (ahead < acnt || bhead < bcnt)) {
            // the smaller head of A and B
            const PQE<Place> ta = ahead < acnt ? qa.get(ahead) : pq_inf<Place>(), tb = bhead < bcnt ? qb.get(bhead) : pq_inf<Place>();
            const bool fromb = pq_less(tb, ta);
            const Place top = fromb ? tb.at : ta.at;
            if (fromb) ++bhead;
            else ++ahead;
            // descend from the popped node, lane i keeping the i-th sibling passed.  The warp loads the
            // five-level subtree below the current node at once (lane i: node i in breadth-first
            // order, with its query coordinate), then walks it through shuffles: five levels cost
            // one round of loads instead of five dependent ones.  Same path, same pushes.
            const int tr = (int)(top >> (F.L + 1));
            const int2 *tnodes = F.nodes + (size_t)tr * F.nnodes;
            const float *u = F.U ? F.U + (size_t)tr * F.d : nullptr;
            const float w2 = u ? w2s[tr] : 0.f;
            const int lv = 31 - __clz(lane + 1);  // lane's level in the subtree (lanes 0..30)
            int j = (int)(top & (((Place)2 << F.L) - 1)), nb = 0;
            PQE<Place> mine = pq_inf<Place>();
            while (j < nn) {
                const long long node = (((long long)j + 1) << lv) - 1 + (lane + 1 - (1 << lv));
                float qs_l = 0.f, v_l = 0.f;
                if (lane < 31 && node < nn) {
                    const int2 nd = __ldg(tnodes + node);
                    const float qx = __ldg(q + nd.x);
                    qs_l = u ? reflect_coord(qx, w2, __ldg(u + nd.x)) : qx;
                    v_l = __int_as_float(nd.y);
                }
                const unsigned lefts = __ballot_sync(FULL, qs_l < v_l);
                const unsigned long long key_l = pq_key(qs_l, v_l);  // of every node, before the walk picks
                int bi = 0;  // breadth-first index of the current node in the loaded subtree
                for (int l = 0; l < 5 && j < nn; ++l) {
                    const unsigned long long key = __shfl_sync(FULL, key_l, bi);
                    const bool left = (lefts >> bi) & 1u;
                    if (lane == nb) {
                        mine.key = key;
                        mine.at = ((Place)tr << (F.L + 1)) | (Place)(left ? 2 * j + 2 : 2 * j + 1);
                    }
                    ++nb;
                    j = left ? 2 * j + 1 : 2 * j + 2;
                    bi = left ? 2 * bi + 1 : 2 * bi + 2;
                }
            }
            if (lane == 0) out[checked] = leaf_code(tr, j - nn, F.L);
            ++checked;
            // the pushes go to B (its popped prefix dropped); keep only what later pops can take
            const int keep = max(0, budget - checked);
            bcnt = pq_insert(qb, bhead, bcnt - bhead, mine, nb, min(PQ_BCAP, keep));
            bhead = 0;
            if (bcnt > PQ_BCAP - 32) {  // the next pushes might not fit: B into A
                acnt = ahead + pq_merge_into(qa.from(ahead), acnt - ahead, qb, bcnt, keep);
                bcnt = 0;
            }
        }
        if (lane == 0) nleaves[qi] = checked;
        __syncwarp();
    }
}

template <typename Place>
int launch_prio(const gf_forest *F, const float *Q, int64_t m, int budget, unsigned *leaves, int *nleaves, cudaStream_t st) {
    int dev = 0, lim = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t per_warp = prio_warp_bytes(budget, F->T, sizeof(Place));
    const int warps = (int)std::min<size_t>(PRIO_WARPS, (size_t)lim / per_warp);
    if (warps < 1) return gf_fail(GF_EUNSUPPORTED, "leaf budget %d needs %zu B of shared memory", budget, per_warp);
    const size_t smem = per_warp * warps;
    GF_CUDA_TRY(gf_smem_limit((const void *)k_prio_leaves<Place>, smem));
    const long long blocks = std::min<long long>((m + warps - 1) / warps, (long long)F->num_sms * 256);
    k_prio_leaves<Place><<<(unsigned)blocks, warps * 32, smem, st>>>(view_of(F), Q, m, budget, leaves, nleaves);
    GF_CUDA_TRY(cudaGetLastError());
    return GF_OK;
}

}  // namespace

int gf_launch_prio_leaves(const gf_forest *F, const float *Q, int64_t m, int budget, unsigned *leaves,
                          int *nleaves, cudaStream_t st) {
    return ((unsigned long long)F->T << (F->L + 1)) <= (1ull << 32)
               ? launch_prio<uint32_t>(F, Q, m, budget, leaves, nleaves, st)
               : launch_prio<unsigned long long>(F, Q, m, budget, leaves, nleaves, st);
}

extern "C" int gf_prio_leaves(const gf_forest *F, const float *Q, int64_t m, int32_t checks, double eps,
                              uint32_t *leaves, int32_t *nleaves, int32_t stride, void *stream) {
    GfRange range("gf_prio_leaves");
    if (!F) return gf_fail(GF_EINVAL, "gf_prio_leaves: null forest");
    if (m < 0 || checks < 0 || !(eps >= 0.0)) return gf_fail(GF_EINVAL, "gf_prio_leaves: bad arguments");
    if (m == 0) return GF_OK;
    if (!Q || !leaves || !nleaves) return gf_fail(GF_EINVAL, "gf_prio_leaves: null pointer");
    if (((unsigned long long)F->T << F->L) > 0xffffffffull)
        return gf_fail(GF_EUNSUPPORTED, "priority search needs T * 2^L <= 2^32");
    const int lb = leaf_budget_of(F, checks, eps);
    const int budget = lb > 0 ? lb : F->T;
    if (budget > 4096) return gf_fail(GF_EUNSUPPORTED, "leaf budget %d above 4096", budget);
    if (stride != budget) return gf_fail(GF_EINVAL, "stride %d, the leaf budget is %d", stride, budget);
    return gf_launch_prio_leaves(F, Q, m, budget, leaves, nleaves, (cudaStream_t)stream);
}
