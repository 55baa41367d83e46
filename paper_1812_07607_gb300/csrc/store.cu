// store.cu -- the device-resident patch store and its derivation pass (K1).
//
// A store keeps a patch collection resident on the GPU (the in-memory form of
// "materialize", Sec. 3.2 / Sec. 4.1 of the paper): int64 ids, the FP32
// feature rows (the ground truth), a zero-padded 16-bit copy (FP16 with one
// scale, or BF16) for the tensor cores, and per-row / per-32-row-chunk
// statistics from which the join kernels derive sound error bounds.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>

#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "internal.h"

namespace dl {

// ------------------------------------------------------------------ errors
static thread_local std::string t_err;

void set_error(const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    t_err = buf;
}

void clear_error() { t_err.clear(); }

const char *last_error() { return t_err.c_str(); }

int cuda_fail(cudaError_t e, const char *what)
{
    set_error("CUDA error %d (%s) in %s", (int)e, cudaGetErrorString(e), what);
    return DL_ECUDA;
}

std::atomic<int64_t> g_launches{0};

// ------------------------------------------------------------------ pools
static std::mutex g_pool_mu;
static bool g_pool_ready[64];

int dev_alloc(void **p, size_t bytes, cudaStream_t st)
{
    int dev = 0;
    DL_CUDA_TRY(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64) {
        std::lock_guard<std::mutex> lk(g_pool_mu);
        if (!g_pool_ready[dev]) {
            // Keep freed blocks in the pool so repeated calls do not return memory
            // to the driver (a per-process pool attribute).
            cudaMemPool_t pool;
            if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
                uint64_t thr = UINT64_MAX;
                cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
            }
            g_pool_ready[dev] = true;
        }
    }
    if (bytes == 0) bytes = 256;
    cudaError_t e = cudaMallocAsync(p, bytes, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("device allocation of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
        *p = nullptr;
        return DL_ENOMEM;
    }
    return DL_OK;
}

void dev_free(void *p, cudaStream_t st)
{
    if (p) cudaFreeAsync(p, st);
}

int device_sm_count()
{
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

// ------------------------------------------------------------------ K1
// Format of a store's 16-bit copy, from the largest feature magnitude of the store and the smallest
// of its non-zero rows' largest: FP16 with one power-of-two scale s (x = s x16, the largest magnitude
// just below 2^15 s) when every row is within 2^18 of the largest, so that a row's rounding stays at
// FP16's 2^-12 of its large features and below 2^-21 of its largest for the small ones; BF16
// otherwise. FP16 rounds eight times finer than BF16 at the same tensor-core rate, which leaves
// about a fifth of the undecided pairs at d = 128 (the accumulation term of the bound stays).
__host__ __device__ inline int half_format(unsigned max_bits, unsigned min_bits, float *scale)
{
    *scale = 1.0f;
    if (max_bits == 0u) return kHalfF16;                        // every feature is 0
    const int e = (int)(max_bits >> 23) - 126, el = (int)(min_bits >> 23) - 126;   // max = m 2^e, m in [1/2, 1)
    if (e < -47 || e > 41 || e - el > 18) return kHalfBF16;   // below 2^-47 two scales' product leaves the normal range
    const unsigned sb = (unsigned)(e - 15 + 127) << 23;         // 2^(e - 15)
    memcpy(scale, &sb, 4);
    return kHalfF16;
}

// Significant bits an FP16 copy keeps (FP16 has 11, BF16 8): 9 for 256 < d <= 512. Those joins are
// bound by the tensor cores under the power cap, where fewer toggling bits mean higher clocks:
// 131,072^2 unit-norm rows, d = 512, back to back, 11 bits 11.87 ms, 10 bits 11.71, 9 bits 11.52, BF16
// 11.53, with 0.51, 0.75, 1.24 and 2.29 M undecided pairs. Narrower joins are bound by their epilogue
// (d = 128: 3.33 ms at any width), wider ones by the recheck's longer rows. A small call at such a d is not
// at the cap and settles more pairs than with 11 bits, but one copy serves every call on a store; it still
// has about half of BF16's undecided pairs.
static int f16_bits(int dp) { return dp > 256 && dp <= 512 ? 9 : 11; }

struct BuildParams {
    const float *src;          // features at the source's row order
    const int64_t *src_ids;
    const int32_t *perm;       // store row i <- source row perm[i] (NULL: row i)
    int64_t n, n_pad;
    int d, dp;
    const unsigned *mm;        // the store's magnitudes (k_sort_keys)
    float *x32;                // outputs below; x32, ids, orig, nq64 and beta may be NULL together
    int64_t *ids;
    int32_t *orig;
    double *nq64;
    float *beta;
    uint16_t *xh;
    float4 *rowb, *cstat;
    float g2, p3_abs;
    int force_bf16;
    int bits;                  // significant bits of the FP16 codes
    int vec;                   // features start on 8 bytes and d is even: load pairs
    int *err;
};

// Chunk statistics of the error bound (see k1_build) from a chunk's rows, one a lane; a padding row
// has zero bounds and beta = +inf.
__device__ __forceinline__ void chunk_stat(float rq, float nqt, float nx, float berr, float bt, float g2, float p3_abs,
                                           float4 *out)
{
    float bmin = bt, bmax = bt < __int_as_float(0x7f800000) ? fabsf(bt) : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        rq = fmaxf(rq, __shfl_xor_sync(0xffffffffu, rq, o));
        nqt = fmaxf(nqt, __shfl_xor_sync(0xffffffffu, nqt, o));
        nx = fmaxf(nx, __shfl_xor_sync(0xffffffffu, nx, o));
        berr = fmaxf(berr, __shfl_xor_sync(0xffffffffu, berr, o));
        bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
        bmin = fminf(bmin, __shfl_xor_sync(0xffffffffu, bmin, o));
    }
    if ((threadIdx.x & 31) == 0) {
        const float p2 = __fmaf_ru(g2, nqt, rq);
        const float p3 = __fadd_ru(__fmaf_ru(5.9604644775390625e-08f, bmax, berr), p3_abs);
        *out = make_float4(nx, p2, p3, bmin);
    }
}

// One CTA per chunk of 32 store rows, four rows a warp, everything a store derives in one pass over
// the source: the gathered FP32 row x, its id and caller row, and
//   nq64  = sum x_k^2 in FP64 (products exact, rounding only in the sum),
//   the 16-bit copy x~ (FP16 times the store's scale, or BF16; zero padded to dp),
//   upper bounds of ||x - x~|| and ||x~|| (FP32 sums of squares rounded up at every step,
//   square roots rounded up), and of ||x|| (from the FP64 sum, inflated by the sum and sqrt
//   rounding),
//   beta = RN32(nq64 / 2) and an upper bound of |beta - ||x||^2 / 2|,
// rows with a non-finite value or |x_k| > 2^40 flagged; then the chunk's column-side maxima of the
// error-bound terms,
//   P1 = max ||x||,   P2 = max ||x - x~|| + (gamma_tc + 1.01 u) max ||x~||,
//   P3 = max |beta err| + u max beta + absolute slack,
//   and the chunk's smallest beta (for the epilogue's whole-chunk reject test),
// so that for a query row q and any column x in the chunk the error of the epilogue value
// h = fl(A~ s - beta) is at most  rq * P1 + ||q~|| * P2 + P3. Padding rows get beta = +inf (they
// never match).
//
// What bounds it: HBM (4 d in, 4 d + 2 dp out a row); a warp keeps four rows' loads in flight. The
// FP64 tail runs on one warp, a row a lane (a warp-wide FP64 instruction costs the same at one
// lane). 100,003 x 128 rows: 47 us; the gather, a 32-rows-a-warp norm pass and the chunk pass took
// 27 + 129 + 4 us, and 54 us where a batch's 9,500 query rows left most of the chip idle.
__global__ void __launch_bounds__(256) k1_build(const BuildParams p)
{
    __shared__ double sm_s1[32];
    __shared__ float sm_s2[32], sm_s3[32];
    __shared__ int sm_bad[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row0 = (int64_t)blockIdx.x * 32 + warp * 4;
    float scale = 1.0f;
    const bool f16 = !p.force_bf16 && half_format(p.mm[2], ~p.mm[3], &scale) == kHalfF16;
    const float inv = 1.0f / scale;   // exact: a power of two
    const float *xr[4];
    double s1[4] = {0.0, 0.0, 0.0, 0.0};
    float s2[4] = {0.f, 0.f, 0.f, 0.f}, s3[4] = {0.f, 0.f, 0.f, 0.f};   // rounded up at every step
    bool bad[4] = {false, false, false, false};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t row = row0 + r;
        const int64_t j = row < p.n ? (p.perm ? (int64_t)p.perm[row] : row) : 0;
        xr[r] = p.src + j * p.d;
        if (p.ids && row < p.n && lane == 0) {
            p.ids[row] = p.src_ids[j];
            p.orig[row] = (int32_t)j;
        }
    }
    for (int k = 2 * lane; k < p.dp; k += 64) {   // two neighbouring features a lane
        float v[4][2];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int h = 0; h < 2; ++h) v[r][h] = 0.0f;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (row0 + r >= p.n) continue;
            if (p.vec) {
                if (k < p.d) *reinterpret_cast<float2 *>(v[r]) = __ldg(reinterpret_cast<const float2 *>(xr[r] + k));
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (k + h < p.d) v[r][h] = __ldg(xr[r] + k + h);
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int64_t row = row0 + r;
            if (row >= p.n) continue;
            uint16_t c[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float x = v[r][h];
                if (!(fabsf(x) <= 1099511627776.0f)) bad[r] = true;   // also catches NaN
                float fx;
                if (f16) {
                    // x / s is exact; its magnitude is rounded to p.bits bits (half up), then to FP16's grid
                    const int sh = 24 - p.bits;
                    const unsigned u = ((__float_as_uint(x * inv) + (1u << (sh - 1))) >> sh) << sh;
                    const __half q = __float2half_rn(__uint_as_float(u));
                    c[h] = __half_as_ushort(q);
                    fx = __half2float(q) * scale;
                } else {
                    const __nv_bfloat16 q = __float2bfloat16_rn(x);
                    c[h] = __bfloat16_as_ushort(q);
                    fx = __bfloat162float(q);
                }
                const float e = x - fx;   // exact: x~ shares x's leading bits, or is 0
                s1[r] = __fma_rn((double)x, (double)x, s1[r]);
                s2[r] = __fmaf_ru(e, e, s2[r]);
                s3[r] = __fmaf_ru(fx, fx, s3[r]);
                if (p.x32 && (p.d & 1) && k + h < p.d) p.x32[row * p.d + k + h] = x;
            }
            if (p.x32 && !(p.d & 1) && k < p.d)   // store rows of an even length start on 8 bytes
                *reinterpret_cast<float2 *>(p.x32 + row * p.d + k) = make_float2(v[r][0], v[r][1]);
            *reinterpret_cast<uint32_t *>(p.xh + row * p.dp + k) = (uint32_t)c[0] | ((uint32_t)c[1] << 16);
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s1[r] = __dadd_rn(s1[r], __shfl_xor_sync(0xffffffffu, s1[r], o));
            s2[r] = __fadd_ru(s2[r], __shfl_xor_sync(0xffffffffu, s2[r], o));
            s3[r] = __fadd_ru(s3[r], __shfl_xor_sync(0xffffffffu, s3[r], o));
        }
        const bool any = __any_sync(0xffffffffu, bad[r]);
        if (lane == 0) {
            sm_s1[warp * 4 + r] = s1[r];
            sm_s2[warp * 4 + r] = s2[r];
            sm_s3[warp * 4 + r] = s3[r];
            sm_bad[warp * 4 + r] = any;
        }
    }
    __syncthreads();
    if (warp) return;
    const int64_t row = (int64_t)blockIdx.x * 32 + lane;
    float rq = 0.f, nqt = 0.f, nx = 0.f, berr = 0.f, bt = __int_as_float(0x7f800000);   // a padding row
    if (row < p.n) {
        const double q1 = sm_s1[lane];
        if (sm_bad[lane]) atomicOr(p.err, 1);
        // Any-order FP64 sum of dp non-negative exact terms: relative error <= (dp-1) 2^-53.
        const double fac = 1.0 + (double)(p.dp + 4) * 2.220446049250313e-16;
        const double grow = 1.0 + 8.881784197001252e-16;   // 1 + 2^-50 covers the sqrt / product roundings
        rq = __fsqrt_ru(sm_s2[lane]);
        nqt = __fsqrt_ru(sm_s3[lane]);
        nx = __double2float_ru(sqrt(q1 * fac) * grow);
        const double h = 0.5 * q1;
        bt = __double2float_rn(h);
        berr = __double2float_ru((fabs((double)bt - h) + h * (double)(p.dp + 2) * 2.220446049250313e-16) * grow);
        if (p.nq64) p.nq64[row] = q1;
        p.rowb[row] = make_float4(rq, nqt, nx, berr);
    }
    if (p.beta) p.beta[row] = bt;
    chunk_stat(rq, nqt, nx, berr, bt, p.g2, p.p3_abs, p.cstat + blockIdx.x);
}

// The inner-product join's column term (0, +inf on padding rows) and its chunk statistics, one warp
// per chunk.
__global__ void __launch_bounds__(256) k1_ip_stats(const float4 *__restrict__ rowb, int64_t n, int64_t n_pad, float g2,
                                                   float p3_abs, float *__restrict__ beta_ip, float4 *__restrict__ cstat)
{
    const int64_t chunk = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (chunk * 32 >= n_pad) return;
    const int64_t row = chunk * 32 + (threadIdx.x & 31);
    const float4 rb = row < n ? rowb[row] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float bt = row < n ? 0.f : __int_as_float(0x7f800000);
    beta_ip[row] = bt;
    chunk_stat(rb.x, rb.y, rb.z, rb.w, bt, g2, p3_abs, cstat + chunk);
}

// ------------------------------------------------------------------ norm ordering
// A store keeps its rows ordered by squared norm (a bucket sort into 65,536
// equal-width buckets between the smallest and largest norm; order inside a
// bucket is arbitrary). Neighbouring rows then have nearly equal ||x||^2/2, so
// the join epilogue can bound a whole 32-column chunk with the chunk's
// smallest beta. The caller's row index of every store row is kept (orig).
constexpr int kSortBuckets = 65536;
static size_t align256(size_t x);

// Squared norms of the rows (row i: source row gather[i] when given) and the store's magnitudes, kept
// by atomicMax on zeroed words: mm[0] = ~(smallest squared norm's bits), mm[1] = the largest's,
// mm[2] = the largest |x_k|'s bits, mm[3] = ~(the smallest non-zero row's largest |x_k|'s).
__global__ void __launch_bounds__(256) k_sort_keys(const float *__restrict__ x, const int32_t *__restrict__ gather,
                                                   int64_t n, int d, float *__restrict__ keys, unsigned *__restrict__ mm)
{
    __shared__ unsigned sm[8][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row0 = ((int64_t)blockIdx.x * 8 + warp) * 4;   // four rows a warp
    float s[4] = {0.f, 0.f, 0.f, 0.f}, m[4] = {0.f, 0.f, 0.f, 0.f};
    const float *xr[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t row = row0 + r;
        xr[r] = x + (row < n ? (gather ? (int64_t)gather[row] : row) : 0) * d;
    }
    for (int k = lane; k < d; k += 32) {
        float v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = row0 + r < n ? __ldg(xr[r] + k) : 0.f;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            s[r] = fmaf(v[r], v[r], s[r]);
            m[r] = fmaxf(m[r], fabsf(v[r]));
        }
    }
    unsigned w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
            m[r] = fmaxf(m[r], __shfl_xor_sync(0xffffffffu, m[r], o));
        }
        if (!(s[r] <= 3.0e38f)) s[r] = 3.0e38f;   // non-finite rows are rejected later; keep the key ordered
        if (row0 + r < n) {
            if (lane == 0) keys[row0 + r] = s[r];
            const unsigned sb = __float_as_uint(s[r]), mb = __float_as_uint(m[r]);   // non-negative floats order like their bits
            w[0] = max(w[0], ~sb);
            w[1] = max(w[1], sb);
            w[2] = max(w[2], mb);
            if (mb) w[3] = max(w[3], ~mb);
        }
    }
    if (lane < 4) sm[warp][lane] = lane == 0 ? w[0] : lane == 1 ? w[1] : lane == 2 ? w[2] : w[3];
    __syncthreads();
    if (threadIdx.x < 4) {   // one atomic of each kind per block of 32 rows
        unsigned v = 0u;
        for (int i = 0; i < 8; ++i) v = max(v, sm[i][threadIdx.x]);
        if (v) atomicMax(mm + threadIdx.x, v);
    }
}

__device__ __forceinline__ int sort_bucket(float k, const unsigned *mm)
{
    const float lo = __uint_as_float(~mm[0]), hi = __uint_as_float(mm[1]);
    if (!(hi > lo)) return 0;
    const float f = (k - lo) / (hi - lo) * (float)kSortBuckets;
    int b = (int)f;
    return b < 0 ? 0 : (b >= kSortBuckets ? kSortBuckets - 1 : b);
}

__global__ void __launch_bounds__(256) k_sort_hist(const float *__restrict__ keys, int64_t n,
                                                   const unsigned *__restrict__ minmax, unsigned *__restrict__ hist)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) atomicAdd(hist + sort_bucket(keys[i], minmax), 1u);
}

// Exclusive prefix sum of the 65,536 bucket counts, one block of 1024 threads, 64 counts each, read
// 16 bytes at a time with every load of a pass in flight (70 us when a loop of single loads did it).
__global__ void __launch_bounds__(1024) k_sort_scan(unsigned *__restrict__ hist)
{
    __shared__ unsigned part[32];
    constexpr int kQuads = kSortBuckets / 1024 / 4;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    uint4 *h4 = reinterpret_cast<uint4 *>(hist) + t * kQuads;
    unsigned loc = 0;
#pragma unroll
    for (int i = 0; i < kQuads; ++i) {
        const uint4 v = h4[i];
        loc += v.x + v.y + v.z + v.w;
    }
    unsigned run = loc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, run, o);
        if (lane >= o) run += y;
    }
    if (lane == 31) part[w] = run;
    __syncthreads();
    unsigned before = lane < w ? part[lane] : 0u;
    before = __reduce_add_sync(0xffffffffu, before);
    run += before - loc;
#pragma unroll
    for (int i = 0; i < kQuads; ++i) {
        const uint4 c = h4[i];
        const uint4 o = make_uint4(run, run + c.x, run + c.x + c.y, run + c.x + c.y + c.z);
        run = o.w + c.w;
        h4[i] = o;
    }
}

__global__ void __launch_bounds__(256) k_sort_scatter(const float *__restrict__ keys, int64_t n,
                                                      const unsigned *__restrict__ minmax, unsigned *__restrict__ offs,
                                                      int32_t *__restrict__ perm)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) perm[atomicAdd(offs + sort_bucket(keys[i], minmax), 1u)] = (int32_t)i;
}

// ------------------------------------------------------------------ FP8 copy
// Every 32-row chunk shares one power-of-two scale s: the largest over its rows of the
// power of two s_row with max|x| / s_row <= 448 (the largest finite e4m3). Codes are
// RN_e4m3(x / s) (x / s is exact, and max|x| / s <= 448 still holds in every row). One
// scale per chunk lets the epilogue bound a whole chunk from its raw accumulators:
// h_j = fl(A_j s_q s - beta_j) <= fl_ru(max_j A_j * s_q s - beta_min).

// One warp per row: the row's own scale s_row.
__global__ void __launch_bounds__(256) k1_fp8_row_scale(const float *__restrict__ x32, int64_t n, int d,
                                                        float *__restrict__ sc8)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 8 + warp;
    if (row >= n) return;
    const float *xr = x32 + row * d;
    float mx = 0.f;
    for (int k = lane; k < d; k += 32) mx = fmaxf(mx, fabsf(__ldg(xr + k)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float sc = 1.0f;
    if (mx > 0.f) {
        int e;
        const float m = frexpf(mx / 448.0f, &e);   // mx/448 = m 2^e, m in [0.5, 1)
        int c = (m == 0.5f) ? e - 1 : e;           // ceil(log2(mx / 448))
        if (c < -126) c = -126;
        sc = ldexpf(1.0f, c);
        while (mx / sc > 448.0f) sc *= 2.0f;
    }
    if (lane == 0) sc8[row] = sc;
}

// One warp per 32-row chunk: the chunk scale (the largest row scale), written to the chunk
// table and to every row of the chunk (1 on padding rows).
__global__ void __launch_bounds__(256) k1_fp8_chunk_scale(int64_t n, int64_t n_pad, float *__restrict__ sc8,
                                                          float *__restrict__ scc8)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t chunk = (int64_t)blockIdx.x * 8 + warp;
    if (chunk * 32 >= n_pad) return;
    const int64_t row = chunk * 32 + lane;
    float sc = row < n ? sc8[row] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sc = fmaxf(sc, __shfl_xor_sync(0xffffffffu, sc, o));
    if (sc == 0.f) sc = 1.0f;
    sc8[row] = row < n ? sc : 1.0f;
    if (lane == 0) scc8[chunk] = sc;
}

// One warp per row: codes with the row's (chunk) scale, and upper bounds of
// ||x - s*dec(codes)|| and ||s*dec(codes)|| (FP32 sums of squares rounded up at every step,
// square roots rounded up).
__global__ void __launch_bounds__(256) k1_fp8(const float *__restrict__ x32, int64_t n, int d, int dp8,
                                              const float *__restrict__ sc8, uint8_t *__restrict__ x8,
                                              float2 *__restrict__ rowb8)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 8 + warp;
    if (row >= n) return;
    const float *xr = x32 + row * d;
    const float sc = sc8[row];
    uint8_t *br = x8 + row * dp8;
    float s2 = 0.f, s3 = 0.f;
    for (int k = lane; k < dp8; k += 32) {
        const float v = (k < d) ? __ldg(xr + k) : 0.0f;
        const __nv_fp8_storage_t q = __nv_cvt_float_to_fp8(v / sc, __NV_SATFINITE, __NV_E4M3);
        br[k] = (uint8_t)q;
        const float dec = __half2float(__half(__nv_cvt_fp8_to_halfraw(q, __NV_E4M3))) * sc;   // exact
        const float e = v - dec;   // exact: |e| is below half an e4m3 step of v / s, times s
        s2 = __fmaf_ru(e, e, s2);
        s3 = __fmaf_ru(dec, dec, s3);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s2 = __fadd_ru(s2, __shfl_xor_sync(0xffffffffu, s2, o));
        s3 = __fadd_ru(s3, __shfl_xor_sync(0xffffffffu, s3, o));
    }
    if (lane == 0) rowb8[row] = make_float2(__fsqrt_ru(s2), __fsqrt_ru(s3));
}

// Per 32-row chunk: {max ||x||, max r8 + (gamma_tc8 + 1.01u) max ||x~8||, P3 (as BF16), beta_min}.
__global__ void __launch_bounds__(256) k1_fp8_stats(const float2 *__restrict__ rowb8, const float4 *__restrict__ cstat,
                                                    int64_t n, int64_t n_pad, float g2, float4 *__restrict__ cstat8)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t chunk = (int64_t)blockIdx.x * 8 + warp;
    if (chunk * 32 >= n_pad) return;
    const int64_t row = chunk * 32 + lane;
    float rq = 0.f, nqt = 0.f;
    if (row < n) {
        const float2 rb = rowb8[row];
        rq = rb.x;
        nqt = rb.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        rq = fmaxf(rq, __shfl_xor_sync(0xffffffffu, rq, o));
        nqt = fmaxf(nqt, __shfl_xor_sync(0xffffffffu, nqt, o));
    }
    if (lane == 0) {
        const float4 c = cstat[chunk];
        cstat8[chunk] = make_float4(c.x, __fmaf_ru(g2, nqt, rq), c.z, c.w);
    }
}

int ensure_fp8(Store *s, cudaStream_t st)
{
    std::lock_guard<std::mutex> lk(s->mu);
    if (s->fp8_block) return DL_OK;
    const int dp8 = (s->d + 127) / 128 * 128;
    const size_t b_x = align256((size_t)s->n * dp8), b_sc = align256(sizeof(float) * s->n_pad),
                 b_rb = align256(sizeof(float2) * std::max<int64_t>(s->n, 1)),
                 b_cs = align256(sizeof(float4) * (s->n_pad / 32)), b_scc = align256(sizeof(float) * (s->n_pad / 32));
    void *blk = nullptr;
    int rc = dev_alloc(&blk, b_x + b_sc + b_rb + b_cs + b_scc, st);
    if (rc) return rc;
    char *p = (char *)blk;
    uint8_t *x8 = (uint8_t *)p;
    float *sc8 = (float *)(p + b_x);
    float2 *rowb8 = (float2 *)(p + b_x + b_sc);
    float4 *cstat8 = (float4 *)(p + b_x + b_sc + b_rb);
    float *scc8 = (float *)(p + b_x + b_sc + b_rb + b_cs);
    const unsigned chunk_blocks = (unsigned)((s->n_pad / 32 + 7) / 8);
    if (s->n > 0) {
        k1_fp8_row_scale<<<(unsigned)((s->n + 7) / 8), 256, 0, st>>>(s->x32, s->n, s->d, sc8);
        count_launch();
    }
    k1_fp8_chunk_scale<<<chunk_blocks, 256, 0, st>>>(s->n, s->n_pad, sc8, scc8);
    count_launch();
    if (s->n > 0) {
        k1_fp8<<<(unsigned)((s->n + 7) / 8), 256, 0, st>>>(s->x32, s->n, s->d, dp8, sc8, x8, rowb8);
        count_launch();
    }
    const float g2 = f32_ru(gamma_tc8(dp8) + 1.01 * kU32);
    k1_fp8_stats<<<chunk_blocks, 256, 0, st>>>(rowb8, s->h.cstat, s->n, s->n_pad, g2, cstat8);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        dev_free(blk, st);
        return cuda_fail(e, "FP8 store copy");
    }
    s->dp8 = dp8;
    s->x8 = x8;
    s->sc8 = sc8;
    s->scc8 = scc8;
    s->rowb8 = rowb8;
    s->cstat8 = cstat8;
    s->fp8_block = blk;
    return DL_OK;
}

// BF16 copy of a store whose 16-bit copy is FP16 (for joins that ask for BF16, and with stores that
// hold BF16), built once, on first use.
static int ensure_bf16(Store *s, cudaStream_t st)
{
    std::lock_guard<std::mutex> lk(s->mu);
    if (s->h.fmt == kHalfBF16 || s->alt_block) return DL_OK;
    const size_t b_x = align256(sizeof(uint16_t) * s->n * s->dp), b_rb = align256(sizeof(float4) * s->n),
                 b_cs = align256(sizeof(float4) * (s->n_pad / 32));
    void *blk = nullptr;
    int rc = dev_alloc(&blk, b_x + b_rb + b_cs + 256, st);
    if (rc) return rc;
    char *q = (char *)blk;
    BuildParams p{};
    p.src = s->x32;
    p.n = s->n;
    p.n_pad = s->n_pad;
    p.d = s->d;
    p.dp = s->dp;
    p.xh = (uint16_t *)q;
    p.rowb = (float4 *)(q + b_x);
    p.cstat = (float4 *)(q + b_x + b_rb);
    p.err = (int *)(q + b_x + b_rb + b_cs);   // the features were checked when the store was made
    p.g2 = f32_ru(gamma_tc(s->dp) + 1.01 * kU32);
    p.p3_abs = f32_ru(abs_slack_tc(s->dp));
    p.force_bf16 = 1;
    p.bits = f16_bits(s->dp);
    p.vec = (s->d & 1) == 0;
    k1_build<<<(unsigned)(s->n_pad / 32), 256, 0, st>>>(p);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        dev_free(blk, st);
        return cuda_fail(e, "BF16 store copy");
    }
    s->alt.fmt = kHalfBF16;
    s->alt.x = p.xh;
    s->alt.rowb = p.rowb;
    s->alt.cstat = p.cstat;
    s->alt_block = blk;
    return DL_OK;
}

int get_half(Store *s, int fmt, cudaStream_t st, Half **out)
{
    *out = nullptr;
    if (s->h.fmt == fmt) {
        *out = &s->h;
        return DL_OK;
    }
    if (fmt != kHalfBF16) {
        set_error("the store's features span too wide a range for an FP16 copy");
        return DL_EUNSUPPORTED;
    }
    const int rc = ensure_bf16(s, st);
    if (!rc) *out = &s->alt;
    return rc;
}

// Row i of a store of n: i p mod n, with p near the golden section of n and without a common divisor, so
// that neighbours part evenly.
__global__ void __launch_bounds__(256) k_part_rows(int64_t n, int64_t p, int32_t *__restrict__ row)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) row[i] = (int32_t)((unsigned long long)i * (unsigned long long)p % (unsigned long long)n);
}
__global__ void __launch_bounds__(256) k_compose_rows(int64_t n, const int32_t *__restrict__ of, int32_t *__restrict__ perm)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) perm[i] = of[perm[i]];
}

// What bounds it: the rows' reads, twice. 131,072 x 128: 0.27 ms more on the store's first top-k, 1.5 ms
// for 1,000,000 x 128, the pool's first growth included.
int get_search(Store *s, int fmt, cudaStream_t st, Store::SearchCopy **out)
{
    *out = nullptr;
    if (fmt == kHalfF16 && s->h.fmt != kHalfF16) {
        set_error("the store's features span too wide a range for an FP16 copy");
        return DL_EUNSUPPORTED;
    }
    std::lock_guard<std::mutex> lk(s->mu);
    Store::SearchCopy &c = s->search[fmt];
    if (c.blk) {
        *out = &c;
        return DL_OK;
    }
    const int64_t n = s->n;
    const size_t b_x = align256(sizeof(uint16_t) * n * s->dp), b_rb = align256(sizeof(float4) * n),
                 b_cs = align256(sizeof(float4) * (s->n_pad / 32)), b_b = align256(sizeof(float) * s->n_pad),
                 b_row = align256(sizeof(int32_t) * n), b_keys = align256(sizeof(float) * n);
    void *blk = nullptr, *tmp = nullptr;
    int rc = dev_alloc(&blk, b_x + b_rb + b_cs + b_b + b_row, st);
    if (rc) return rc;
    rc = dev_alloc(&tmp, b_keys + b_row + sizeof(unsigned) * kSortBuckets + 256, st);
    if (rc) {
        dev_free(blk, st);
        return rc;
    }
    char *q = (char *)blk;
    c.row = (int32_t *)(q + b_x + b_rb + b_cs + b_b);
    float *keys = (float *)tmp;
    int32_t *part = (int32_t *)((char *)tmp + b_keys);
    unsigned *hist = (unsigned *)((char *)tmp + b_keys + b_row), *mm = hist + kSortBuckets;
    int64_t p = std::max<int64_t>(1, (int64_t)(0.6180339887498949 * (double)n));
    auto common = [](int64_t a, int64_t b) {
        while (b) {
            const int64_t r = a % b;
            a = b;
            b = r;
        }
        return a;
    };
    while (common(n, p) != 1) ++p;
    const unsigned gt = (unsigned)((n + 255) / 256);
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(unsigned) * kSortBuckets + 256, st);
    if (e == cudaSuccess) {
        k_part_rows<<<gt, 256, 0, st>>>(n, p, part);
        k_sort_keys<<<(unsigned)((n + 31) / 32), 256, 0, st>>>(s->x32, part, n, s->d, keys, mm);
        k_sort_hist<<<gt, 256, 0, st>>>(keys, n, mm, hist);
        k_sort_scan<<<1, 1024, 0, st>>>(hist);
        k_sort_scatter<<<gt, 256, 0, st>>>(keys, n, mm, hist, c.row);
        k_compose_rows<<<gt, 256, 0, st>>>(n, part, c.row);
        BuildParams b{};
        b.src = s->x32;
        b.perm = c.row;
        b.n = n;
        b.n_pad = s->n_pad;
        b.d = s->d;
        b.dp = s->dp;
        b.mm = mm;
        b.beta = (float *)(q + b_x + b_rb + b_cs);
        b.xh = (uint16_t *)q;
        b.rowb = (float4 *)(q + b_x);
        b.cstat = (float4 *)(q + b_x + b_rb);
        b.g2 = f32_ru(gamma_tc(s->dp) + 1.01 * kU32);
        b.p3_abs = f32_ru(abs_slack_tc(s->dp));
        b.force_bf16 = fmt == kHalfBF16;
        b.bits = f16_bits(s->dp);
        b.vec = (s->d & 1) == 0;
        b.err = (int *)(mm + 8);   // the features were checked when the store was made
        k1_build<<<(unsigned)(s->n_pad / 32), 256, 0, st>>>(b);
        count_launch(7);
        e = cudaGetLastError();
        c.beta = b.beta;
        c.h.x = b.xh;
        c.h.rowb = b.rowb;
        c.h.cstat = b.cstat;
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    dev_free(tmp, st);
    if (e != cudaSuccess) {
        dev_free(blk, st);
        return cuda_fail(e, "search copy");
    }
    c.h.fmt = fmt;
    c.h.scale = fmt == kHalfF16 ? s->h.scale : 1.0f;
    c.blk = blk;
    *out = &c;
    return DL_OK;
}

// The inner-product join's column term is 0: h = q.x. Its chunk stats are those of the 16-bit copy, so
// P1 and P2 (the encoding and accumulation terms of the bound) are the copy's own and P3 keeps the
// L2 beta error (a conservative extra); padding rows get +inf, so they never match.
int get_ip(Store *s, const Half *h, cudaStream_t st, const Store::IpColumns **out)
{
    std::lock_guard<std::mutex> lk(s->mu);
    Store::IpColumns &c = s->ip[h->fmt];
    *out = &c;
    if (c.blk) return DL_OK;
    const size_t b_b = align256(sizeof(float) * s->n_pad), b_cs = align256(sizeof(float4) * (s->n_pad / 32));
    void *blk = nullptr;
    const int rc = dev_alloc(&blk, b_b + b_cs, st);
    if (rc) return rc;
    float *beta_ip = (float *)blk;
    float4 *cstat_ip = (float4 *)((char *)blk + b_b);
    k1_ip_stats<<<(unsigned)((s->n_pad / 32 + 7) / 8), 256, 0, st>>>(h->rowb, s->n, s->n_pad,
                                                                     f32_ru(gamma_tc(s->dp) + 1.01 * kU32),
                                                                     f32_ru(abs_slack_tc(s->dp)), beta_ip, cstat_ip);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        dev_free(blk, st);
        return cuda_fail(e, "inner-product column arrays");
    }
    c.beta = beta_ip;
    c.cstat = cstat_ip;
    c.blk = blk;
    return DL_OK;
}

// ------------------------------------------------------------------ tensor maps
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void *p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

int get_tmap(Store *s, Half *h, int box_rows, const CUtensorMap **out)
{
    std::lock_guard<std::mutex> lk(s->mu);
    for (auto &t : h->tmaps)
        if (t.valid && t.box_rows == box_rows) {
            *out = &t.map;
            return DL_OK;
        }
    TmapCache *slot = nullptr;
    for (auto &t : h->tmaps)
        if (!t.valid) {
            slot = &t;
            break;
        }
    if (!slot) slot = &h->tmaps[0];
    auto fn = encode_fn();
    if (!fn) {
        set_error("cuTensorMapEncodeTiled is not available from the driver");
        return DL_ECUDA;
    }
    cuuint64_t gdim[2] = {(cuuint64_t)s->dp, (cuuint64_t)(s->n > 0 ? s->n : 1)};
    cuuint64_t gstride[1] = {(cuuint64_t)s->dp * sizeof(uint16_t)};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t estride[2] = {1, 1};
    CUresult r = fn(&slot->map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, (void *)h->x, gdim, gstride, box, estride,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed (%d) for dp=%d rows=%lld box=%d", (int)r, s->dp,
                  (long long)s->n, box_rows);
        return DL_ECUDA;
    }
    slot->valid = true;
    slot->box_rows = box_rows;
    *out = &slot->map;
    return DL_OK;
}

int get_tmap8(Store *s, int box_rows, const CUtensorMap **out)
{
    std::lock_guard<std::mutex> lk(s->mu);
    for (auto &t : s->tmaps8)
        if (t.valid && t.box_rows == box_rows) {
            *out = &t.map;
            return DL_OK;
        }
    TmapCache *slot = nullptr;
    for (auto &t : s->tmaps8)
        if (!t.valid) {
            slot = &t;
            break;
        }
    if (!slot) slot = &s->tmaps8[0];
    auto fn = encode_fn();
    if (!fn || !s->x8) {
        set_error("FP8 tensor map: driver entry point or FP8 copy missing");
        return DL_ECUDA;
    }
    cuuint64_t gdim[2] = {(cuuint64_t)s->dp8, (cuuint64_t)(s->n > 0 ? s->n : 1)};
    cuuint64_t gstride[1] = {(cuuint64_t)s->dp8};
    cuuint32_t box[2] = {128, (cuuint32_t)box_rows};
    cuuint32_t estride[2] = {1, 1};
    CUresult r = fn(&slot->map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, (void *)s->x8, gdim, gstride, box, estride,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled (FP8) failed (%d)", (int)r);
        return DL_ECUDA;
    }
    slot->valid = true;
    slot->box_rows = box_rows;
    *out = &slot->map;
    return DL_OK;
}

static size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace dl

namespace dl {

// Create a store. With gather == NULL the rows are put in squared-norm order;
// otherwise store row i is caller row gather[i] (device array of n indices).
int store_create_impl(dl_store **out, const int64_t *ids, const float *feats, int64_t n, int32_t d, int32_t where,
                      void *cuda_stream, const int32_t *gather)
{
    clear_error();
    if (!out) {
        set_error("dl_store_create: out is NULL");
        return DL_EINVAL;
    }
    *out = nullptr;
    if (n < 0 || n >= (int64_t(1) << 31)) {
        set_error("dl_store_create: n=%lld out of range [0, 2^31)", (long long)n);
        return DL_EINVAL;
    }
    if (d < 1 || d > 1024) {
        set_error("dl_store_create: d=%d out of range [1, 1024]", d);
        return DL_EINVAL;
    }
    if (n > 0 && (!ids || !feats)) {
        set_error("dl_store_create: ids/feats is NULL");
        return DL_EINVAL;
    }
    if (where != DL_MEM_HOST && where != DL_MEM_DEVICE) {
        set_error("dl_store_create: bad memory kind %d", where);
        return DL_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    dl_store *s = new dl_store();
    s->n = n;
    s->d = d;
    s->dp = (d + 63) / 64 * 64;
    s->n_pad = (n + 255) / 256 * 256;
    if (s->n_pad == 0) s->n_pad = 256;
    DL_CUDA_TRY(cudaGetDevice(&s->device));

    const size_t b_ids = align256(sizeof(int64_t) * n), b_orig = align256(sizeof(int32_t) * n),
                 b_x32 = align256(sizeof(float) * n * d), b_xh = align256(sizeof(uint16_t) * n * s->dp),
                 b_nq = align256(sizeof(double) * n), b_beta = align256(sizeof(float) * s->n_pad),
                 b_rowb = align256(sizeof(float4) * n), b_cst = align256(sizeof(float4) * (s->n_pad / 32)),
                 b_err = 256;
    const size_t total = b_ids + b_orig + b_x32 + b_xh + b_nq + b_beta + b_rowb + b_cst + b_err;
    void *base = nullptr;
    int rc = dev_alloc(&base, total, st);
    if (rc != DL_OK) {
        delete s;
        return rc;
    }
    char *p = (char *)base;
    s->ids = (int64_t *)p;
    p += b_ids;
    s->orig = (int32_t *)p;
    p += b_orig;
    s->x32 = (float *)p;
    p += b_x32;
    s->h.x = (uint16_t *)p;
    p += b_xh;
    s->nq64 = (double *)p;
    p += b_nq;
    s->beta = (float *)p;
    p += b_beta;
    s->h.rowb = (float4 *)p;
    p += b_rowb;
    s->h.cstat = (float4 *)p;
    p += b_cst;
    int *d_err = (int *)p;

    // scratch for the norm ordering (and for host inputs, the uploaded rows)
    const bool host = (where == DL_MEM_HOST);
    const size_t t_x = host ? align256(sizeof(float) * n * d) : 0, t_ids = host ? align256(sizeof(int64_t) * n) : 0,
                 t_keys = align256(sizeof(float) * n), t_perm = align256(sizeof(int32_t) * n),
                 t_hist = sizeof(unsigned) * kSortBuckets;
    void *tmp = nullptr;
    if (n > 0) {
        rc = dev_alloc(&tmp, t_x + t_ids + t_keys + t_perm + t_hist, st);
        if (rc != DL_OK) {
            dev_free(base, st);
            delete s;
            return rc;
        }
    }
    auto fail = [&](int code) {
        dev_free(base, st);
        dev_free(tmp, st);
        cudaStreamSynchronize(st);
        delete s;
        return code;
    };
    cudaError_t e = cudaMemsetAsync(d_err, 0, b_err, st);
    if (e != cudaSuccess) return fail(cuda_fail(e, "dl_store_create memset"));
    unsigned *mm = (unsigned *)d_err + 4;   // the store's magnitudes, beside the error word
    BuildParams bp{};
    bp.src = feats;
    bp.src_ids = ids;
    bp.perm = gather;
    if (n > 0) {
        char *q = (char *)tmp;
        if (host) {
            float *hx = (float *)q;
            int64_t *hid = (int64_t *)(q + t_x);
            e = cudaMemcpyAsync(hx, feats, sizeof(float) * n * d, cudaMemcpyHostToDevice, st);
            if (e == cudaSuccess) e = cudaMemcpyAsync(hid, ids, sizeof(int64_t) * n, cudaMemcpyHostToDevice, st);
            if (e != cudaSuccess) return fail(cuda_fail(e, "dl_store_create upload"));
            bp.src = hx;
            bp.src_ids = hid;
        }
        q += t_x + t_ids;
        float *keys = (float *)q;
        int32_t *perm = (int32_t *)(q + t_keys);
        unsigned *hist = (unsigned *)(q + t_keys + t_perm);
        const unsigned gt = (unsigned)((n + 255) / 256);
        k_sort_keys<<<(unsigned)((n + 31) / 32), 256, 0, st>>>(bp.src, gather, n, d, keys, mm);
        count_launch();
        if (!gather) {
            e = cudaMemsetAsync(hist, 0, t_hist, st);
            if (e != cudaSuccess) return fail(cuda_fail(e, "dl_store_create memset"));
            k_sort_hist<<<gt, 256, 0, st>>>(keys, n, mm, hist);
            k_sort_scan<<<1, 1024, 0, st>>>(hist);
            k_sort_scatter<<<gt, 256, 0, st>>>(keys, n, mm, hist, perm);
            count_launch(3);
            bp.perm = perm;
        }
    }
    bp.n = n;
    bp.n_pad = s->n_pad;
    bp.d = d;
    bp.dp = s->dp;
    bp.mm = mm;
    bp.x32 = s->x32;
    bp.ids = s->ids;
    bp.orig = s->orig;
    bp.nq64 = s->nq64;
    bp.beta = s->beta;
    bp.xh = s->h.x;
    bp.rowb = s->h.rowb;
    bp.cstat = s->h.cstat;
    bp.g2 = f32_ru(gamma_tc(s->dp) + 1.01 * kU32);
    bp.p3_abs = f32_ru(abs_slack_tc(s->dp));
    bp.vec = (d & 1) == 0 && (reinterpret_cast<uintptr_t>(bp.src) & 7) == 0;
    bp.bits = f16_bits(s->dp);
    bp.err = d_err;
    k1_build<<<(unsigned)(s->n_pad / 32), 256, 0, st>>>(bp);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(cuda_fail(e, "store kernels launch"));
    unsigned h_back[8] = {0u};   // the error word, then (from word 4) the magnitudes
    e = cudaMemcpyAsync(h_back, d_err, sizeof h_back, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(cuda_fail(e, "dl_store_create sync"));
    if (h_back[0]) {
        set_error("dl_store_create: a feature is non-finite or exceeds 2^40 in magnitude");
        return fail(DL_EINVAL);
    }
    std::memcpy(&s->nq_max, &h_back[5], sizeof s->nq_max);
    std::memcpy(&s->x_max, &h_back[6], sizeof s->x_max);
    s->h.fmt = half_format(h_back[6], ~h_back[7], &s->h.scale);
    dev_free(tmp, st);
    *out = s;
    return DL_OK;
}

// ------------------------------------------------------------------ cosine metric
// One warp per store row: the unit-normalized row, written at the caller's row index.
//   n = fl32(sqrt(sum_k x_k^2)), the sum in FP64 with k ascending and each addition
//   rounded to nearest (the products of two floats are exact in FP64); x^_k = fl32(x_k / n).
// A row whose norm is zero has no direction: it is flagged and left zero.
__global__ void __launch_bounds__(256) k_normalize_rows(const float *__restrict__ x32, const int64_t *__restrict__ ids,
                                                        const int32_t *__restrict__ orig, int64_t n, int d,
                                                        float *__restrict__ out, int64_t *__restrict__ out_ids,
                                                        int *__restrict__ err)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 8 + warp;
    if (row >= n) return;
    const float *xr = x32 + row * d;
    double s = 0.0;
    for (int k0 = 0; k0 < d; k0 += 32) {
        const int k = k0 + lane;
        double sq = 0.0;
        if (k < d) {
            const double v = (double)__ldg(xr + k);
            sq = __dmul_rn(v, v);
        }
        const int lim = min(32, d - k0);
        for (int l = 0; l < lim; ++l) s = __dadd_rn(s, __shfl_sync(0xffffffffu, sq, l));
    }
    const float nr = __double2float_rn(__dsqrt_rn(s));
    const int64_t dst = orig[row];
    float *o = out + dst * d;
    if (!(nr > 0.0f)) {
        for (int k = lane; k < d; k += 32) o[k] = 0.0f;
        if (lane == 0) atomicOr(err, 1);
    } else {
        for (int k = lane; k < d; k += 32) o[k] = __fdiv_rn(__ldg(xr + k), nr);
    }
    if (lane == 0) out_ids[dst] = ids[row];
}

// ------------------------------------------------------------------ chi-square domain
__global__ void __launch_bounds__(256) k_any_negative(const float *__restrict__ x, int64_t n, int *flag)
{
    bool neg = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        neg |= __ldg(x + i) < 0.f;
    if (__any_sync(0xffffffffu, neg) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

int store_nonneg(Store *s, cudaStream_t st, bool *ok)
{
    {
        std::lock_guard<std::mutex> lk(s->mu);
        if (s->nonneg) {
            *ok = s->nonneg == 1;
            return DL_OK;
        }
    }
    const int64_t n = s->n * (int64_t)s->d;
    int h = 0;
    if (n > 0) {
        void *tmp = nullptr;
        int rc = dev_alloc(&tmp, 16, st);
        if (rc) return rc;
        int *flag = (int *)tmp;
        cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int), st);
        if (e == cudaSuccess) {
            const int grid = (int)std::min<int64_t>((n + 255) / 256, (int64_t)device_sm_count() * 8);
            k_any_negative<<<grid, 256, 0, st>>>(s->x32, n, flag);
            count_launch();
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        dev_free(tmp, st);
        if (e != cudaSuccess) return cuda_fail(e, "store_nonneg");
    }
    std::lock_guard<std::mutex> lk(s->mu);
    s->nonneg = h ? 2 : 1;
    *ok = !h;
    return DL_OK;
}

}  // namespace dl

using namespace dl;

extern "C" {

int dl_store_create(dl_store **out, const int64_t *ids, const float *feats, int64_t n, int32_t d, int32_t where,
                    void *cuda_stream)
{
    dl::NvtxScope nvtx_scope("dl_store_create");
    return store_create_impl(out, ids, feats, n, d, where, cuda_stream, nullptr);
}

int dl_store_normalize(const dl_store *in, dl_store **out, void *cuda_stream)
{
    dl::NvtxScope nvtx_scope("dl_store_normalize");
    clear_error();
    if (!in || !out) {
        set_error("dl_store_normalize: NULL argument");
        return DL_EINVAL;
    }
    *out = nullptr;
    int dev = -1;
    DL_CUDA_TRY(cudaGetDevice(&dev));
    if (dev != in->device) {
        set_error("dl_store_normalize: store lives on device %d but device %d is current", in->device, dev);
        return DL_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int64_t n = in->n;
    const int d = in->d;
    void *tmp = nullptr;
    const size_t b_x = align256(sizeof(float) * (size_t)std::max<int64_t>(n, 1) * d);
    const size_t b_ids = align256(sizeof(int64_t) * (size_t)std::max<int64_t>(n, 1));
    int rc = dev_alloc(&tmp, b_x + b_ids + 256, st);
    if (rc) return rc;
    float *xn = (float *)tmp;
    int64_t *idn = (int64_t *)((char *)tmp + b_x);
    int *d_err = (int *)((char *)tmp + b_x + b_ids);
    cudaError_t e = cudaMemsetAsync(d_err, 0, sizeof(int), st);
    if (e == cudaSuccess && n > 0) {
        k_normalize_rows<<<(unsigned)((n + 7) / 8), 256, 0, st>>>(in->x32, in->ids, in->orig, n, d, xn, idn, d_err);
        count_launch();
        e = cudaGetLastError();
    }
    int h_err = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        dev_free(tmp, st);
        return cuda_fail(e, "dl_store_normalize");
    }
    if (h_err) {
        dev_free(tmp, st);
        set_error("dl_store_normalize: a row has a zero norm (no direction for the cosine metric)");
        return DL_EINVAL;
    }
    dl_store *s = nullptr;
    rc = store_create_impl(&s, idn, xn, n, d, DL_MEM_DEVICE, cuda_stream, nullptr);
    cudaStreamSynchronize(st);
    dev_free(tmp, st);
    if (rc) return rc;
    s->unit = true;
    *out = s;
    return DL_OK;
}

int dl_store_destroy(dl_store *s)
{
    if (!s) return DL_OK;
    int prev = 0;
    cudaGetDevice(&prev);
    if (prev != s->device) cudaSetDevice(s->device);
    dev_free(s->ids, 0);   // ids is the base of the store's single allocation
    if (s->fp8_block) dev_free(s->fp8_block, 0);
    if (s->alt_block) dev_free(s->alt_block, 0);
    for (auto &c : s->ip)
        if (c.blk) dev_free(c.blk, 0);
    if (s->clabel) dev_free(s->clabel, 0);
    for (auto &c : s->search)
        if (c.blk) dev_free(c.blk, 0);
    for (auto &b : s->balls)
        if (b.blk) dev_free(b.blk, 0);
    if (prev != s->device) cudaSetDevice(prev);
    delete s;
    return DL_OK;
}

int dl_store_shape(const dl_store *s, int64_t *n, int32_t *d)
{
    if (!s) {
        set_error("dl_store_shape: NULL store");
        return DL_EINVAL;
    }
    if (n) *n = s->n;
    if (d) *d = s->d;
    return DL_OK;
}

const char *dl_last_error(void) { return dl::last_error(); }

const char *dl_version(void) { return "dl-simjoin 0.1 (sm_103a)"; }

int64_t dl_kernel_launches(void) { return dl::g_launches.load(); }

}  // extern "C"
