// gf_forest.cu -- forest lifecycle (import, export, free), screening copies and the query entry
// points of the C ABI.
#include "gf_internal.cuh"

#include "gf_squares.cuh"
#include "gf_trace.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <unordered_map>
#include <vector>

// ---------------------------------------------------------------- errors

static thread_local std::string g_last_error;

int gf_fail(int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_last_error = buf;
    return code;
}

int gf_cuda_fail(cudaError_t e, const char *what) {
    const int code = (e == cudaErrorMemoryAllocation) ? GF_ENOMEM : GF_ECUDA;
    return gf_fail(code, "%s: %s", what, cudaGetErrorString(e));
}

// gf_debug_fail_alloc: the number of library allocations that still succeed before one fails
// (-1: none fails)
static std::atomic<int> g_alloc_countdown{-1};

extern "C" int gf_debug_fail_alloc(int32_t after) {
    g_alloc_countdown.store(after < 0 ? -1 : after);
    return GF_OK;
}

// Whether this allocation is the one that gf_debug_fail_alloc asks to fail.
static bool alloc_refused() {
    for (int c = g_alloc_countdown.load(); c >= 0;)
        if (g_alloc_countdown.compare_exchange_weak(c, c - 1)) return c == 0;
    return false;
}

bool gf_dmalloc_if(void **p, size_t bytes) {
    *p = nullptr;
    if (!alloc_refused() && cudaMalloc(p, bytes) == cudaSuccess) return true;
    cudaGetLastError();
    *p = nullptr;
    return false;
}

int gf_dmalloc(void **p, size_t bytes) {
    *p = nullptr;
    if (bytes == 0) return GF_OK;
    if (alloc_refused()) return gf_fail(GF_ENOMEM, "cudaMalloc(%zu bytes): refused (gf_debug_fail_alloc)", bytes);
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();  // clear the sticky-free allocation error
        return gf_fail(GF_ENOMEM, "cudaMalloc(%zu bytes): %s", bytes, cudaGetErrorString(e));
    }
    return GF_OK;
}

extern "C" const char *gf_last_error(void) { return g_last_error.c_str(); }
extern "C" int32_t gf_version(void) { return 100; }

extern "C" void gf_rand_params_default(gf_rand_params *rp) {
    if (!rp) return;
    rp->t = 5;
    rp->shuffle = 1;
    rp->var_scope = GF_VAR_NODE;
    rp->householder = 0;
}

extern "C" void gf_query_opts_default(gf_query_opts *o) {
    if (!o) return;
    std::memset(o, 0, sizeof *o);
    o->precision = GF_FP32;
}

// ---------------------------------------------------------------- shared memory limits

cudaError_t gf_smem_limit(const void *kern, size_t smem) {
    static std::mutex mu;
    static std::unordered_map<const void *, size_t> fixed;  // kernel -> its static shared memory
    if (smem <= 32 * 1024) return cudaSuccess;  // within the default 48 KB beside any kernel's static share
    int dev = 0, all = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&all, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    size_t own = 0;
    {
        std::lock_guard<std::mutex> g(mu);
        auto it = fixed.find(kern);
        if (it == fixed.end()) {
            cudaFuncAttributes fa;
            if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
            it = fixed.emplace(kern, fa.sharedSizeBytes).first;
        }
        own = it->second;
    }
    if (own + smem > (size_t)all) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, all - (int)own);
}

// ---------------------------------------------------------------- per-call scratch

namespace {

constexpr int MAX_DEVICES = 64;
constexpr uint64_t SCRATCH_KEEP = 1ull << 30;  // bytes a pool keeps across synchronizations
std::mutex g_pool_mu;
cudaMemPool_t g_pool[MAX_DEVICES] = {};
int g_live_forests = 0;  // under g_pool_mu

cudaError_t scratch_pool(cudaMemPool_t *pool) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> g(g_pool_mu);
    if (!g_pool[dev]) {
        cudaMemPoolProps props;
        std::memset(&props, 0, sizeof props);
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        if ((e = cudaMemPoolCreate(&p, &props)) != cudaSuccess) return e;
        uint64_t keep = SCRATCH_KEEP;
        if ((e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
            cudaMemPoolDestroy(p);
            return e;
        }
        g_pool[dev] = p;
    }
    *pool = g_pool[dev];
    return cudaSuccess;
}

}  // namespace

cudaError_t gf_scratch_alloc(void **p, size_t bytes, cudaStream_t st) {
    cudaMemPool_t pool = nullptr;
    const cudaError_t e = scratch_pool(&pool);
    return e == cudaSuccess ? cudaMallocFromPoolAsync(p, bytes, pool, st) : e;
}

void gf_scratch_free(void *p, cudaStream_t st) { cudaFreeAsync(p, st); }

// ---------------------------------------------------------------- forest storage

// Destroy everything the forest owns (tolerates partially built forests).
static void forest_release(gf_forest *F) {
    if (!F) return;
    if (F->owns_x) cudaFree(F->x);
    cudaFree(F->nodes);
    cudaFree(F->perm);
    cudaFree(F->xb);
    cudaFree(F->xbn);
    cudaFree(F->x8);
    cudaFree(F->scale8);
    cudaFree(F->x8n);
    cudaFree(F->U);
    if (F->live) {
        std::lock_guard<std::mutex> g(g_pool_mu);
        if (--g_live_forests == 0)
            for (cudaMemPool_t p : g_pool)
                if (p) cudaMemPoolTrimTo(p, 0);
    }
    delete F;
}

// Shape fields and the storage of x / nodes / perm.  borrow: keep X itself.  X may be a device or
// a host pointer when it is copied (the copies infer the direction from the address).
int gf_forest_alloc(gf_forest **out, const float *X, int64_t n, int32_t d, int32_t T,
                    int32_t leaf_size, bool borrow, cudaStream_t st) {
    *out = nullptr;
    if (!X) return gf_fail(GF_EINVAL, "X is null");
    if (n < 1 || n > 0x7fffffffLL) return gf_fail(GF_EINVAL, "n=%lld outside [1, 2^31)", (long long)n);
    if (d < 1 || d > 65535) return gf_fail(GF_EINVAL, "d=%d outside [1, 65535]", d);
    if (T < 1 || T > 4096) return gf_fail(GF_EINVAL, "T=%d outside [1, 4096]", T);
    if (leaf_size < 1) return gf_fail(GF_EINVAL, "leaf_size=%d < 1", leaf_size);
    gf_forest *F = new gf_forest();
    F->n = n; F->d = d; F->T = T; F->leaf_size = leaf_size;
    F->L = depth_of(n, leaf_size);
    if (F->L > 30) {
        const int32_t L = F->L;
        delete F;
        return gf_fail(GF_EINVAL, "tree depth %d too large", L);
    }
    F->max_leaf = (int32_t)((n + ((int64_t)1 << F->L) - 1) >> F->L);
    const int64_t cap = (int64_t)T * F->max_leaf;
    if (cap > (1 << 24)) { delete F; return gf_fail(GF_EINVAL, "T * leaf size = %lld too large", (long long)cap); }
    F->cand_cap = (int32_t)cap;
    F->ldx = round_up(d, 4);
    F->ldb = round_up(d, 8);
    F->ld8 = round_up(d, 16);
    cudaGetDevice(&F->device);
    cudaDeviceGetAttribute(&F->num_sms, cudaDevAttrMultiProcessorCount, F->device);
    const size_t nn = ((size_t)1 << F->L) - 1;
    int r;
    if (borrow) {
        if (d % 4 != 0 || ((uintptr_t)X & 15) != 0) {
            delete F;
            return gf_fail(GF_EINVAL, "borrowed X needs d %% 4 == 0 and 16-byte alignment");
        }
        F->x = const_cast<float *>(X);
        F->owns_x = false;
    } else {
        if ((r = gf_dmalloc((void **)&F->x, (size_t)n * F->ldx * 4))) { forest_release(F); return r; }
        F->owns_x = true;
        if (F->ldx != d) {
            cudaError_t e = cudaMemsetAsync(F->x, 0, (size_t)n * F->ldx * 4, st);
            if (e == cudaSuccess)
                e = cudaMemcpy2DAsync(F->x, (size_t)F->ldx * 4, X, (size_t)d * 4, (size_t)d * 4, (size_t)n,
                                      cudaMemcpyDefault, st);
            if (e != cudaSuccess) { forest_release(F); return gf_cuda_fail(e, "copy X"); }
        } else {
            cudaError_t e = cudaMemcpyAsync(F->x, X, (size_t)n * d * 4, cudaMemcpyDefault, st);
            if (e != cudaSuccess) { forest_release(F); return gf_cuda_fail(e, "copy X"); }
        }
    }
    if ((r = gf_dmalloc((void **)&F->nodes, (size_t)T * nn * sizeof(int2)))) { forest_release(F); return r; }
    if ((r = gf_dmalloc((void **)&F->perm, (size_t)T * n * 4))) { forest_release(F); return r; }
    F->device_bytes = (borrow ? 0 : (int64_t)n * F->ldx * 4) + (int64_t)(T * nn * sizeof(int2)) + (int64_t)T * n * 4;
    cudaMemPool_t pool;  // made here, so that a query under stream capture does not
    if (scratch_pool(&pool) != cudaSuccess) cudaGetLastError();
    {
        std::lock_guard<std::mutex> g(g_pool_mu);
        F->live = true;
        ++g_live_forests;
    }
    *out = F;
    return GF_OK;
}

void gf_forest_destroy(gf_forest *F) { forest_release(F); }

// Count non-finite entries of X (rows of d floats).
__global__ void k_count_nonfinite(const float *__restrict__ X, long long total, unsigned long long *bad) {
    unsigned long long c = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x)
        c += !isfinite(X[i]);
    c = __reduce_add_sync(0xffffffffu, (unsigned)c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(bad, c);
}

int gf_check_finite(const float *X, int64_t count, cudaStream_t st) {
    unsigned long long *bad = nullptr;
    int r = gf_dmalloc((void **)&bad, sizeof *bad);
    if (r) return r;
    unsigned long long h = 0;
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof *bad, st);
    if (e == cudaSuccess) {
        k_count_nonfinite<<<1216, 256, 0, st>>>(X, count, bad);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, bad, sizeof h, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(bad);
    if (e != cudaSuccess) return gf_cuda_fail(e, "finite check");
    if (h) return gf_fail(GF_EINVAL, "X holds %llu NaN/Inf values", h);
    return GF_OK;
}

// ---------------------------------------------------------------- import / export

// Validate a host tree structure and copy it into F (nodes, perm), then check X for NaN/Inf.
// On error F is left for the caller to release.
int gf_forest_fill_structure(gf_forest *F, const int32_t *split_dim_host, const float *split_val_host,
                             const int32_t *perm_host) {
    const int64_t n = F->n;
    const int32_t d = F->d, T = F->T;
    const size_t nn = ((size_t)1 << F->L) - 1;
    std::vector<int2> nodes((size_t)T * nn);
    for (size_t i = 0; i < nodes.size(); ++i) {
        if (split_dim_host[i] < 0 || split_dim_host[i] >= d)
            return gf_fail(GF_EINVAL, "split_dim[%zu] = %d outside [0, %d)", i, split_dim_host[i], d);
        int32_t bits;
        std::memcpy(&bits, &split_val_host[i], 4);
        nodes[i] = make_int2(split_dim_host[i], bits);
    }
    std::vector<unsigned char> seen((size_t)n);
    for (int32_t t = 0; t < T; ++t) {
        std::fill(seen.begin(), seen.end(), 0);
        for (int64_t i = 0; i < n; ++i) {
            const int32_t v = perm_host[(size_t)t * n + i];
            if (v < 0 || v >= n || seen[v])
                return gf_fail(GF_EINVAL, "perm row %d is not a permutation of 0..n-1", t);
            seen[v] = 1;
        }
    }
    cudaError_t e = cudaMemcpy(F->nodes, nodes.data(), nodes.size() * sizeof(int2), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(F->perm, perm_host, (size_t)T * n * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return gf_cuda_fail(e, "import copy");
    return gf_check_finite(F->x, (int64_t)n * F->ldx, 0);
}

extern "C" int gf_forest_import(const float *X, int64_t n, int32_t d, int32_t T, int32_t leaf_size,
                                const int32_t *split_dim_host, const float *split_val_host,
                                const int32_t *perm_host, gf_forest **out) {
    GfRange range("gf_forest_import");
    if (!out) return gf_fail(GF_EINVAL, "out is null");
    *out = nullptr;
    if (!split_dim_host || !split_val_host || !perm_host) return gf_fail(GF_EINVAL, "null host array");
    gf_forest *F = nullptr;
    int r = gf_forest_alloc(&F, X, n, d, T, leaf_size, false, 0);
    if (r) return r;
    if ((r = gf_forest_fill_structure(F, split_dim_host, split_val_host, perm_host))) {
        forest_release(F);
        return r;
    }
    *out = F;
    return GF_OK;
}

extern "C" int gf_forest_export(const gf_forest *F, int32_t *split_dim_host, float *split_val_host,
                                int32_t *perm_host) {
    if (!F) return gf_fail(GF_EINVAL, "null forest");
    const size_t nn = ((size_t)1 << F->L) - 1;
    std::vector<int2> nodes((size_t)F->T * nn);
    if (!nodes.empty()) GF_CUDA_TRY(cudaMemcpy(nodes.data(), F->nodes, nodes.size() * sizeof(int2), cudaMemcpyDeviceToHost));
    for (size_t i = 0; i < nodes.size(); ++i) {
        if (split_dim_host) split_dim_host[i] = nodes[i].x;
        if (split_val_host) std::memcpy(&split_val_host[i], &nodes[i].y, 4);
    }
    if (perm_host) GF_CUDA_TRY(cudaMemcpy(perm_host, F->perm, (size_t)F->T * F->n * 4, cudaMemcpyDeviceToHost));
    return GF_OK;
}

extern "C" int gf_forest_get_info(const gf_forest *F, gf_forest_info *info) {
    if (!F || !info) return gf_fail(GF_EINVAL, "null argument");
    info->n = F->n; info->d = F->d; info->T = F->T; info->leaf_size = F->leaf_size; info->L = F->L;
    info->max_leaf = F->max_leaf; info->cand_cap = F->cand_cap;
    info->screens = (F->xb ? (1 << GF_BF16_RERANK) : 0) | (F->x8 ? (1 << GF_FP8_RERANK) : 0);
    info->device_bytes = F->device_bytes;
    return GF_OK;
}

// Copy the per-tree Householder vectors (host [T][d]) into the forest.
int gf_forest_set_U(gf_forest *F, const float *U_host) {
    const size_t bytes = (size_t)F->T * F->d * 4;
    if (!F->U) {
        int r = gf_dmalloc((void **)&F->U, bytes);
        if (r) return r;
        F->device_bytes += (int64_t)bytes;
    }
    GF_CUDA_TRY(cudaMemcpy(F->U, U_host, bytes, cudaMemcpyHostToDevice));
    return GF_OK;
}

extern "C" int gf_forest_set_reflections(gf_forest *F, const float *U_host) {
    if (!F || !U_host) return gf_fail(GF_EINVAL, "null argument");
    for (size_t i = 0; i < (size_t)F->T * F->d; ++i)
        if (!std::isfinite(U_host[i])) return gf_fail(GF_EINVAL, "U holds NaN/Inf");
    return gf_forest_set_U(F, U_host);
}

extern "C" int gf_forest_free(gf_forest *F) {
    if (!F) return GF_OK;
    cudaDeviceSynchronize();
    forest_release(F);
    return GF_OK;
}

extern "C" int gf_forest_set_tuning(gf_forest *F, int32_t precision, int32_t warps_per_cta,
                                    int32_t ctas_per_sm, int32_t rerank_R, int32_t rows_in_flight) {
    if (!F || precision < 0 || precision > 2) return gf_fail(GF_EINVAL, "bad forest or precision");
    if (warps_per_cta < 1 || warps_per_cta > 32 || ctas_per_sm < 0 || ctas_per_sm > GF_MAX_CTAS_PER_SM ||
        rerank_R < 0 || rerank_R > GF_MAX_SHORTLIST ||
        (rows_in_flight != 0 && rows_in_flight != 2 && rows_in_flight != 4))
        return gf_fail(GF_EINVAL, "bad tuning values");
    F->tune_warps[precision] = warps_per_cta;
    F->tune_ctas[precision] = ctas_per_sm;
    if (rerank_R > 0) F->tune_R[precision] = rerank_R;
    if (rows_in_flight > 0) F->tune_G[precision] = rows_in_flight;
    return GF_OK;
}

// ---------------------------------------------------------------- screening copies

// Four values of a row from column j on, zeros past d (rows are 16-byte aligned, ldx a multiple of four).
__device__ __forceinline__ float4 row4(const float *r, int j, int d, int ldx) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j < ldx) v = __ldg(reinterpret_cast<const float4 *>(r + j));
    if (j + 1 > d) v.x = 0.f;
    if (j + 2 > d) v.y = 0.f;
    if (j + 3 > d) v.z = 0.f;
    if (j + 4 > d) v.w = 0.f;
    return v;
}

// xb[i][j] = bf16_rne(x[i][j]) for j < d, 0 in the padding; xbn[i] = sum_j xb[i][j]^2, rounded once.  A warp
// per row, eight values a lane at a time, up to eight 16-byte loads in flight: bound by the row's
// bytes in and out (500,000 x 960: 3.09 ms as two passes of scalar loads).
__global__ void __launch_bounds__(256) k_to_bf16(const float *__restrict__ x, int ldx, long long n, int d, int ldb,
                                                 __nv_bfloat16 *xb, float *xbn) {
    const int lane = threadIdx.x & 31;
    for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n;
         i += ((long long)gridDim.x * blockDim.x) >> 5) {
        const float *r = x + i * ldx;
        SquareSum sum;
        for (int j0 = 0; j0 < ldb; j0 += 1024) {
            float4 v[4][2];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + 256 * u + 8 * lane;
                v[u][0] = row4(r, j, d, ldx);
                v[u][1] = row4(r, j + 4, d, ldx);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + 256 * u + 8 * lane;
                __nv_bfloat162 b[4] = {__floats2bfloat162_rn(v[u][0].x, v[u][0].y), __floats2bfloat162_rn(v[u][0].z, v[u][0].w),
                                       __floats2bfloat162_rn(v[u][1].x, v[u][1].y), __floats2bfloat162_rn(v[u][1].z, v[u][1].w)};
                if (j < ldb) *reinterpret_cast<uint4 *>(xb + i * ldb + j) = *reinterpret_cast<const uint4 *>(b);
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const float2 f = __bfloat1622float2(b[h]);
                    sum.add(f.x);
                    sum.add(f.y);
                }
            }
            sum.flush();
        }
        double total = sum.warp_total();
        if (!(total > 1e-20 && total < 1e37)) {  // squares outside float32's range could count: every value in float64 (uniform)
            total = 0.0;
            for (int j = lane; j < d; j += 32) {
                const double v = (double)__bfloat162float(__float2bfloat16_rn(__ldg(r + j)));
                total += v * v;
            }
            for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
        }
        if (lane == 0) xbn[i] = (float)total;
    }
}

// a = max |x|, scale = a / 448, codes = e4m3_rne_satfinite(x * (448 / a)), x8n[i] = sum_j (scale_i
// x8[i][j])^2, rounded once.  A warp per row, sixteen values a lane at a time; the row is read again
// for its codes, from the caches.
__global__ void __launch_bounds__(256) k_to_fp8(const float *__restrict__ x, int ldx, long long n, int d, int ld8, uint8_t *x8,
                                                float *scale, float *x8n) {
    const int lane = threadIdx.x & 31;
    for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n;
         i += ((long long)gridDim.x * blockDim.x) >> 5) {
        const float *r = x + i * ldx;
        float a = 0.f;
#pragma unroll 8
        for (int j = 4 * lane; j < d; j += 128) {
            const float4 v = row4(r, j, d, ldx);
            a = fmaxf(fmaxf(a, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
        const float inv = a > 0.f ? 448.0f / a : 0.f;
        const float s = a > 0.f ? a / 448.0f : 1.0f;
        if (lane == 0) scale[i] = s;
        SquareSum sum;
#pragma unroll 2
        for (int j = 16 * lane; j < ld8; j += 512) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = row4(r, j + 4 * u, d, ldx);
            unsigned w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                // (zeros past d: 0 * inv is NaN where 448 / a overflows)
                const int c = j + 4 * u;
                const float f[4] = {c < d ? v[u].x * inv : 0.f, c + 1 < d ? v[u].y * inv : 0.f,
                                    c + 2 < d ? v[u].z * inv : 0.f, c + 3 < d ? v[u].w * inv : 0.f};
                w[u] = 0;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const __nv_fp8_storage_t code = __nv_cvt_float_to_fp8(f[h], __NV_SATFINITE, __NV_E4M3);
                    w[u] |= (unsigned)code << (8 * h);
                    const __half_raw hr = __nv_cvt_fp8_to_halfraw(code, __NV_E4M3);
                    sum.add(__half2float(*reinterpret_cast<const __half *>(&hr)));
                }
            }
            *reinterpret_cast<uint4 *>(x8 + i * ld8 + j) = make_uint4(w[0], w[1], w[2], w[3]);
            sum.flush();
        }
        const double total = sum.warp_total(), sc = (double)s;
        if (lane == 0) x8n[i] = (float)(total * sc * sc);
    }
}

extern "C" int gf_forest_add_screen(gf_forest *F, int32_t precision, void *stream) {
    GfRange range("gf_forest_add_screen");
    if (!F) return gf_fail(GF_EINVAL, "null forest");
    cudaStream_t st = (cudaStream_t)stream;
    int r;
    if (precision == GF_BF16_RERANK) {
        if (F->xb) return GF_OK;
        if ((r = gf_dmalloc((void **)&F->xb, (size_t)F->n * F->ldb * 2))) return r;
        if ((r = gf_dmalloc((void **)&F->xbn, (size_t)F->n * 4))) { cudaFree(F->xb); F->xb = nullptr; return r; }
        k_to_bf16<<<F->num_sms * 8, 256, 0, st>>>(F->x, F->ldx, F->n, F->d, F->ldb, F->xb, F->xbn);
        F->device_bytes += (int64_t)F->n * F->ldb * 2 + F->n * 4;
    } else if (precision == GF_FP8_RERANK) {
        if (F->x8) return GF_OK;
        if ((r = gf_dmalloc((void **)&F->x8, (size_t)F->n * F->ld8))) return r;
        if ((r = gf_dmalloc((void **)&F->scale8, (size_t)F->n * 4))) { cudaFree(F->x8); F->x8 = nullptr; return r; }
        if ((r = gf_dmalloc((void **)&F->x8n, (size_t)F->n * 4))) {
            cudaFree(F->x8);
            cudaFree(F->scale8);
            F->x8 = nullptr;
            F->scale8 = nullptr;
            return r;
        }
        k_to_fp8<<<F->num_sms * 8, 256, 0, st>>>(F->x, F->ldx, F->n, F->d, F->ld8, F->x8, F->scale8, F->x8n);
        F->device_bytes += (int64_t)F->n * F->ld8 + F->n * 8;
    } else {
        return gf_fail(GF_EINVAL, "precision %d has no screening copy", precision);
    }
    GF_CUDA_TRY(cudaGetLastError());
    GF_CUDA_TRY(cudaStreamSynchronize(st));
    return GF_OK;
}

// ---------------------------------------------------------------- queries

extern "C" int gf_query_ex(const gf_forest *F, const float *Q, int64_t m, int32_t k,
                           const gf_query_opts *o, int64_t *ids, float *dists) {
    GfRange range("gf_query");
    if (!F) return gf_fail(GF_EINVAL, "null forest");
    if (m < 0) return gf_fail(GF_EINVAL, "m < 0");
    if (k < 1) return gf_fail(GF_EINVAL, "k=%d < 1", k);
    if (m == 0) return GF_OK;
    if (!Q || !ids || !dists) return gf_fail(GF_EINVAL, "null pointer");
    gf_query_opts def;
    gf_query_opts_default(&def);
    if (!o) o = &def;
    const int p = o->precision;
    if (p < 0 || p > 2) return gf_fail(GF_EINVAL, "unknown precision %d", p);
    if (p == GF_BF16_RERANK && !F->xb) return gf_fail(GF_EINVAL, "forest has no bf16 copy (gf_forest_add_screen)");
    if (p == GF_FP8_RERANK && !F->x8) return gf_fail(GF_EINVAL, "forest has no fp8 copy (gf_forest_add_screen)");
    const int R = o->rerank_R > 0 ? o->rerank_R : F->tune_R[p];
    if (p != GF_FP32 && k > R) return gf_fail(GF_EINVAL, "k=%d exceeds the shortlist R=%d", k, R);
    const int warps = o->warps_per_cta > 0 ? o->warps_per_cta : F->tune_warps[p];
    if (warps > 32) return gf_fail(GF_EINVAL, "warps_per_cta=%d > 32", warps);
    const int cps = o->ctas_per_sm > 0 ? o->ctas_per_sm : F->tune_ctas[p];
    if (o->algo < GF_ALGO_AUTO || o->algo > GF_ALGO_LEAF) return gf_fail(GF_EINVAL, "unknown algo %d", o->algo);
    QueryExtra x;
    x.algo = o->algo;
    x.workspace = o->workspace;
    x.workspace_bytes = o->workspace_bytes;
    x.ncand_out = o->ncand_out;
    x.rows_in_flight = o->rows_in_flight > 0 ? o->rows_in_flight : F->tune_G[p];
    if (o->order < GF_ORDER_AUTO || o->order > GF_ORDER_LOCALITY) return gf_fail(GF_EINVAL, "unknown order %d", o->order);
    x.order = o->order;
    if (o->checks < 0 || !(o->eps >= 0.0)) return gf_fail(GF_EINVAL, "checks < 0 or eps < 0");
    x.leaf_budget = leaf_budget_of(F, o->checks, o->eps);
    x.events = (cudaEvent_t *)o->events;
    x.shaped = o->warps_per_cta > 0 || o->ctas_per_sm > 0 || o->rows_in_flight > 0;
    if (x.leaf_budget > 0) {
        if (((unsigned long long)F->T << F->L) > 0xffffffffull)
            return gf_fail(GF_EUNSUPPORTED, "priority search needs T * 2^L <= 2^32");
        if (x.leaf_budget > 4096) return gf_fail(GF_EUNSUPPORTED, "leaf budget %d above 4096", x.leaf_budget);
    }
    return gf_launch_query(F, Q, m, k, p, R, warps, cps, (cudaStream_t)o->stream, ids, dists, x);
}

extern "C" int gf_query_workspace_size(const gf_forest *F, int64_t m, const gf_query_opts *o, int64_t *bytes) {
    if (!F || !bytes) return gf_fail(GF_EINVAL, "null argument");
    gf_query_opts def;
    gf_query_opts_default(&def);
    if (!o) o = &def;
    const int p = o->precision;
    if (p < 0 || p > 2) return gf_fail(GF_EINVAL, "unknown precision %d", p);
    // the streaming kernel runs at most 8 warps per CTA; fewer threads per CTA only raise the
    // occupancy-derived grid, so the clamp keeps the size an upper bound
    const int warps = std::min(8, o->warps_per_cta > 0 ? o->warps_per_cta : F->tune_warps[p]);
    const int cps = o->ctas_per_sm > 0 ? o->ctas_per_sm : F->tune_ctas[p];
    const int R = o->rerank_R > 0 ? o->rerank_R : F->tune_R[p];
    long long grid = 0;
    int r = gf_stream_grid(F, m, warps, cps, p, 1, R, &grid);
    if (r) return r;
    // A launch's own grid can be below this one (a larger k or R lowers the occupancy), and AUTO
    // reorders every batch longer than the launch's grid: count the order arrays for any m > 1.
    const bool ordered = o->order == GF_ORDER_LOCALITY || (o->order == GF_ORDER_AUTO && m > 1);
    if ((r = gf_stream_workspace_bytes(F, m, grid, ordered, leaf_budget_of(F, o->checks, o->eps), bytes))) return r;
    if (o->algo == GF_ALGO_LEAF || o->algo == GF_ALGO_AUTO) {
        // the leaf-major path's scratch; AUTO gets the larger of the two
        QueryExtra x;
        x.leaf_budget = leaf_budget_of(F, o->checks, o->eps);
        x.ncand_out = o->ncand_out;
        const bool leaf_ok = gf_leaf_unsupported(F, m, 1, p, R, x) == nullptr;
        const int64_t lb = gf_leaf_workspace_bytes(F, m, p, R, o->order, x.leaf_budget);
        if (o->algo == GF_ALGO_LEAF) *bytes = lb;
        else if (leaf_ok && gf_leaf_preferred(F, m, 1, p, R, x)) *bytes = std::max(*bytes, lb);
    }
    return GF_OK;
}

extern "C" int gf_query(const gf_forest *F, const float *Q, int64_t m, int32_t k, int64_t *ids,
                        float *dists) {
    return gf_query_ex(F, Q, m, k, nullptr, ids, dists);
}
