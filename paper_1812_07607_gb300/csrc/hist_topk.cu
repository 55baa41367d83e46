// hist_topk.cu -- the top-k join under the histogram distances (L1, chi-square): for every query
// row, the k store rows with the smallest canonical distance, ordered by (distance, store row)
// (Sec. 6.2 q1 -- the closest images to a query image -- with the colour-histogram distances of
// Sec. 4.1). These distances are not contractions, so they run on the CUDA cores.
//
// Query rows are taken in chunks that bound the scratch memory. For each chunk:
//   k_hist_dist (many query rows) or k_hist_dist_few (a few)
//                   the FP32 distance D32 of every (query, store) pair of the chunk (against a few
//                   store rows: k_hist_select itself);
//   k_hist_select   one CTA per query row at a time: with |D32 - D| <= g32 D + a32 (the SIMT
//                   join's bound, which holds for any summation order of the non-negative terms),
//                   1. a bound T on the row's k-th smallest D32: the k-th smallest of the minima
//                      of 2,048 groups of its columns;
//                   2. the columns whose lower bound reaches T's upper bound (widened by the
//                      canonical sum's slack), then the exact k-th smallest D32 among them and
//                      the columns that reach its upper bound;
//                   3. their canonical FP64 distances (k ascending, every operation rounded to
//                      nearest: t = q_k - x_k, then s += |t| (L1), or u = q_k + x_k and, where
//                      u > 0, s += t*t / u);
//                   4. the exact rank by (canonical distance, caller's store row); rank < k is
//                      written.
#include <algorithm>

#include "cta.cuh"
#include "exact.cuh"
#include "kernels.h"
#include "simt_tile.cuh"

namespace dl {

namespace {

constexpr int kHtCap = 8192;     // candidates a row can rank (more: DL_EOVERFLOW, many exact ties)
constexpr int kHtShared = 1024;  // candidates kept in shared memory (more: the CTA's global scratch)
constexpr int kHtGroups = 8;     // column groups of each of the 256 threads
constexpr int kHtTermK = 32;     // canonical terms of a candidate staged at a time
// Up to this many features, and with more than 32 candidates, a thread forms and adds its candidate's terms
// alone: staged, 32 - d of 32 threads would wait. Chi-square, 3,000 rows against 147, k = 100, whole
// calls, a thread alone against staged: d = 3 253 / 431 us, 8 293 / 438, 16 366 / 441; d = 32 no gain.
constexpr int kHtChain = 16;
// Up to this many store rows a row's CTA forms its distances itself: a launch less, and no tile padded
// to 128 columns. Whole calls, one kernel against two: L1, d = 64, k = 100, 300 rows against 11, 115 and
// 500: 52 / 70, 90 / 107 and 115 / 105 us; chi-square 53 / 93, 127 / 157 and 141 / 158; 3,000 rows, d = 11,
// k = 3, L1, against 32, 115 and 200: 94 / 98, 114 / 100 and 126 / 104. Where query rows leave SMs idle the
// line lies higher: 40 rows, d = 64, k = 100, against 200 and 500: L1 81 / 95 and 104 / 106, chi-square
// 101 / 132 and 120 / 144; d = 11, k = 3, L1, 57 / 58 and 68 / 55.
constexpr int own_rows(int rows) { return rows <= 256 ? 200 : 128; }
// Up to this many query rows the distances come from k_hist_dist_few: a warp's lanes share one
// pair's features (16-byte slices, a shuffle tree per pair), so no work goes into padding a query
// tile to 128 rows. Whole calls against 65,536 x 128, few against tile: L1 112 / 175 us at 1 row,
// 180 / 180 at 16, 219 / 183 at 24; chi-square 109 / 320, 297 / 318 at 32, 397 / 320 at 48.
constexpr int few_rows(int metric) { return metric == 1 ? 16 : 32; }

struct HistTk {
    const float *Q, *S;
    int d, nS, k;
    int64_t row0;             // first query row of this chunk
    int rows;                 // its query rows
    float *dist;              // [rows][ld] FP32 distances
    int64_t ld;
    uint32_t *scr_c;          // [CTAs of k_hist_select][kHtCap]
    float *scr_v;             // [CTAs][kHtCap]
    double *scr_d;            // [CTAs][kHtCap]
    const int32_t *q_orig, *s_orig;
    const int64_t *s_ids;
    int64_t *out_ids;
    double *out_d;
    float g32, a32, slack;
    float up;                 // chi-square: the features' scale, and that of `dist`
    int *err;
    unsigned long long *n_fp64;
};

// The distances of a chunk's rows by the SIMT pair tile: bounded by the FP32 pipe as the join is.
// With k_hist_select behind it, 1,000 rows against 65,536 x 128 take 1.76 ms under chi-square,
// top 10 (44.4 ms with one CTA reading every store row for each query row).
template <int M, bool VEC>
__global__ void __launch_bounds__(256, 2) k_hist_dist(const HistTk f)
{
    __shared__ __align__(16) SimtSmem sm;
    const int r0 = blockIdx.y * kSimtTile, c0 = blockIdx.x * kSimtTile;
    float acc[8][8];
    simt_tile<M, VEC>(f.Q + (size_t)f.row0 * f.d, f.S, f.rows, f.nS, f.d, r0, c0, f.up, sm, acc);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = r0 + simt_sub(ty, i);
        if (r >= f.rows) continue;
        float *o = f.dist + (size_t)r * f.ld;   // rows padded to 128 columns: whole quads are in bounds
        *reinterpret_cast<float4 *>(o + c0 + tx * 4) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        *reinterpret_cast<float4 *>(o + c0 + 64 + tx * 4) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
    }
}

// The FP32 distance of one pair by a warp.
template <int M, bool VEC>
__device__ __forceinline__ float warp_hist_dist(const float *q, const float *x, int d, float up)
{
    const int lane = threadIdx.x & 31;
    float s = 0.f;
    if constexpr (VEC) {
        for (int k = lane * 4; k < d; k += 128) {
            const float4 a = __ldg(reinterpret_cast<const float4 *>(q + k));
            const float4 b = __ldg(reinterpret_cast<const float4 *>(x + k));
            dist_terms<M>(a.x, a.y, b.x, b.y, up, s);
            dist_terms<M>(a.z, a.w, b.z, b.w, up, s);
        }
    } else {
        for (int k = lane * 2; k < d; k += 64) {
            const bool two = k + 1 < d;   // an absent second feature is 0 in both rows: a zero term
            dist_terms<M>(__ldg(q + k), two ? __ldg(q + k + 1) : 0.f, __ldg(x + k), two ? __ldg(x + k + 1) : 0.f, up, s);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// The same for a few rows: a warp takes store rows in turn and every query row against each.
template <int M, bool VEC>
__global__ void __launch_bounds__(256) k_hist_dist_few(const HistTk f)
{
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)((gridDim.x * blockDim.x) >> 5);
    const float *Q = f.Q + (size_t)f.row0 * f.d;
    for (int j = w; j < f.nS; j += nw) {
        const float *x = f.S + (size_t)j * f.d;
        for (int r = 0; r < f.rows; ++r) {
            const float s = warp_hist_dist<M, VEC>(Q + (size_t)r * f.d, x, f.d, f.up);
            if ((threadIdx.x & 31) == 0) f.dist[(size_t)r * f.ld + j] = s;
        }
    }
}

template <int M>
__device__ __forceinline__ double canon_term(float q, float x)
{
    const double a = widen(q), b = widen(x);
    const double t = __dsub_rn(a, b);
    if constexpr (M == 1) {
        return fabs(t);
    } else {
        const double u = __dadd_rn(a, b);
        return u > 0.0 ? __ddiv_rn(__dmul_rn(t, t), u) : 0.0;   // adding 0.0 leaves a sum as it is
    }
}

// Bits of the k-th smallest of non-negative floats (which order like their bits): the largest value
// with fewer than k below it, found bit by bit. count(x) = how many of this thread's values have
// bits below x. At least k values: theirs; fewer: all ones below the sign, above every float.
template <class F>
__device__ __forceinline__ unsigned cta_kth_bits(int k, unsigned *s_cnt, int &turn, F count)
{
    unsigned res = 0u;
    for (int bit = 30; bit >= 0; --bit) {
        const unsigned t = res | (1u << bit);
        if (cta_count(count(t), s_cnt, turn++) < (unsigned)k) res = t;
    }
    return res;
}

// One query row at a time. What bounds it: reading the row's distances twice (the minima, then the
// columns under the bound), from L2 or HBM; what follows touches about k columns. OWN: the row's
// distances are formed here first (stores of up to own_rows; VEC as in the distance kernels).
template <int M, bool VEC, bool OWN>
__global__ void __launch_bounds__(256) k_hist_select(const HistTk f)
{
    __shared__ uint32_t sh_c[kHtShared];
    __shared__ float sh_v[kHtShared];
    __shared__ double sh_d[kHtShared];
    __shared__ double sh_t[32][kHtTermK + 1];
    __shared__ unsigned s_cnt[2];
    __shared__ int s_m;
    const int tid = threadIdx.x;
    if (tid < 2) s_cnt[tid] = 0u;
    __syncthreads();
    int turn = 0;
    for (int row = blockIdx.x; row < f.rows; row += gridDim.x) {
        float *D = f.dist + (size_t)row * f.ld;
        const float *q = f.Q + (size_t)(f.row0 + row) * f.d;
        if constexpr (OWN) {
            for (int j = tid >> 5; j < f.nS; j += 8) {
                const float s = warp_hist_dist<M, VEC>(q, f.S + (size_t)j * f.d, f.d, f.up);
                if ((tid & 31) == 0) D[j] = s;
            }
            __syncthreads();
        }
        auto upper = [&](float v) { return __fmul_ru(__fadd_ru(__fmul_ru(v, 1.0f + f.g32), f.a32), 1.0f + f.slack); };
        auto lower = [&](float v) { return __fsub_rd(__fmul_rd(v, 1.0f - f.g32), f.a32); };
        // 1. the k-th smallest group minimum
        float mn[kHtGroups];
#pragma unroll
        for (int g = 0; g < kHtGroups; ++g) mn[g] = __int_as_float(0x7f800000);
        for (int j0 = tid * 4; j0 < f.nS; j0 += 2048) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = j0 + h * 1024;
                if (j < f.nS) {
                    const float4 v = *reinterpret_cast<const float4 *>(D + j);
                    mn[4 * h] = fminf(mn[4 * h], v.x);
                    if (j + 1 < f.nS) mn[4 * h + 1] = fminf(mn[4 * h + 1], v.y);
                    if (j + 2 < f.nS) mn[4 * h + 2] = fminf(mn[4 * h + 2], v.z);
                    if (j + 3 < f.nS) mn[4 * h + 3] = fminf(mn[4 * h + 3], v.w);
                }
            }
        }
        unsigned kb = 0x7f800000u;
        if (f.nS > f.k) {
            kb = cta_kth_bits(f.k, s_cnt, turn, [&](unsigned t) {
                unsigned c = 0;
#pragma unroll
                for (int g = 0; g < kHtGroups; ++g) c += __float_as_uint(mn[g]) < t ? 1u : 0u;
                return c;
            });
        }
        // 2. the columns under the bound: into shared memory, or past it into the CTA's scratch
        uint32_t *cl = sh_c;
        float *cv = sh_v;
        double *cd = sh_d;
        int m = 0;
        for (int attempt = 0;; ++attempt) {
            const float lim = kb < 0x7f800000u ? upper(__uint_as_float(kb)) : __int_as_float(0x7f800000);
            const int cap = cl == sh_c ? kHtShared : kHtCap;
            if (tid == 0) s_m = 0;
            __syncthreads();
            for (int j = tid * 4; j < f.nS; j += 1024) {
                const float4 v4 = *reinterpret_cast<const float4 *>(D + j);
                const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (j + e < f.nS && lower(v[e]) <= lim) {
                        const int pos = atomicAdd(&s_m, 1);
                        if (pos < cap) {
                            cl[pos] = (uint32_t)(j + e);
                            cv[pos] = v[e];
                        }
                    }
            }
            __syncthreads();
            m = s_m;
            __syncthreads();
            if (m <= cap || attempt == 2) break;
            if (cl == sh_c) {   // more than shared memory holds: the CTA's scratch
                cl = f.scr_c + (size_t)blockIdx.x * kHtCap;
                cv = f.scr_v + (size_t)blockIdx.x * kHtCap;
                cd = f.scr_d + (size_t)blockIdx.x * kHtCap;
            }
            if (m > kHtCap)     // and more than that holds: the row's exact k-th smallest distance
                kb = cta_kth_bits(f.k, s_cnt, turn, [&](unsigned t) {
                    unsigned c = 0;
                    for (int j = tid; j < f.nS; j += 256) c += __float_as_uint(D[j]) < t ? 1u : 0u;
                    return c;
                });
        }
        if (m > kHtCap) {
            if (tid == 0) atomicExch(f.err, 1);
            continue;
        }
        // the k-th smallest of the row is among them: those above its own upper bound go
        if (m > f.k) {
            kb = cta_kth_bits(f.k, s_cnt, turn, [&](unsigned t) {
                unsigned c = 0;
                for (int a = tid; a < m; a += 256) c += __float_as_uint(cv[a]) < t ? 1u : 0u;
                return c;
            });
            const float lim = upper(__uint_as_float(kb));
            int kept = 0;
            for (int a0 = 0; a0 < m; a0 += 256) {   // compacted in place, a block of 256 at a time
                const int a = a0 + tid;
                const bool keep = a < m && lower(cv[a]) <= lim;
                const uint32_t c = a < m ? cl[a] : 0u;
                if (tid == 0) s_m = kept;
                __syncthreads();
                if (keep) cl[atomicAdd(&s_m, 1)] = c;   // at or below this block's own entries, all read
                __syncthreads();
                kept = s_m;
                __syncthreads();
            }
            m = kept;
        }
        // 3. canonical distances, 32 candidates at a time: every thread forms terms, one per candidate
        // adds them in order (few features: see kHtChain)
        if (tid == 0 && m) atomicAdd(f.n_fp64, (unsigned long long)m);
        const bool chain = f.d <= kHtChain && m > 32;   // a thread a candidate
        if (chain) {
            for (int a = tid; a < m; a += 256) {
                const float *x = f.S + (size_t)cl[a] * f.d;
                double s = 0.0;
                for (int k = 0; k < f.d; ++k) s = __dadd_rn(s, canon_term<M>(__ldg(q + k), __ldg(x + k)));
                cd[a] = s;
                cv[a] = __int_as_float(f.s_orig[cl[a]]);
            }
        }
        for (int a0 = chain ? m : 0; a0 < m; a0 += 32) {
            const int na = min(32, m - a0);
            double s = 0.0;
            for (int k0 = 0; k0 < f.d; k0 += kHtTermK) {
                const int nk = min(kHtTermK, f.d - k0);
                for (int e = tid; e < na * kHtTermK; e += 256) {
                    const int a = e / kHtTermK, k = e % kHtTermK;
                    if (k < nk) sh_t[a][k] = canon_term<M>(__ldg(q + k0 + k), __ldg(f.S + (size_t)cl[a0 + a] * f.d + k0 + k));
                }
                __syncthreads();
                if (tid < na)
                    for (int k = 0; k < nk; ++k) s = __dadd_rn(s, sh_t[tid][k]);
                __syncthreads();
            }
            if (tid < na) {
                cd[a0 + tid] = s;
                cv[a0 + tid] = __int_as_float(f.s_orig[cl[a0 + tid]]);   // the FP32 distances are done with
            }
        }
        __syncthreads();
        // 4. exact rank by (canonical distance, caller's store row)
        const int64_t base = (int64_t)f.q_orig[f.row0 + row] * f.k;
        for (int a = tid; a < m; a += 256) {
            const double da = cd[a];
            const int32_t oa = __float_as_int(cv[a]);
            int rank = 0;
#pragma unroll 4
            for (int bb = 0; bb < m; ++bb) {   // every load unconditional: ties by the thousand wait for none
                const double db = cd[bb];
                const int32_t ob = __float_as_int(cv[bb]);
                rank += (db < da) | ((db == da) & (ob < oa));
            }
            if (rank < f.k) {
                f.out_ids[base + rank] = f.s_ids[cl[a]];
                f.out_d[base + rank] = da;
            }
        }
        for (int t = m + tid; t < f.k; t += 256) {
            f.out_ids[base + t] = -1;
            f.out_d[base + t] = -1.0;
        }
        __syncthreads();   // the lists are this row's until here
    }
}

template <int M, bool VEC>
int launch_hist_chunk(const HistTk &f, int grid_sel, cudaStream_t st)   // kernels launched
{
    const bool own = f.nS <= own_rows(f.rows);
    if (own) {
        k_hist_select<M, VEC, true><<<(unsigned)grid_sel, 256, 0, st>>>(f);
    } else {
        if (f.rows <= few_rows(M))
            k_hist_dist_few<M, VEC><<<(unsigned)std::min((f.nS + 7) / 8, device_sm_count() * 8), 256, 0, st>>>(f);
        else
            k_hist_dist<M, VEC><<<dim3((unsigned)((f.nS + kSimtTile - 1) / kSimtTile), (unsigned)((f.rows + kSimtTile - 1) / kSimtTile)),
                                  256, 0, st>>>(f);
        count_launch();
        k_hist_select<M, false, false><<<(unsigned)grid_sel, 256, 0, st>>>(f);
    }
    count_launch();
    return own ? 1 : 2;
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

int hist_topk(const dl_store *Q, const dl_store *S, int metric, int k, int64_t *out_ids, double *out_d,
              cudaStream_t st, dl_join_stats *stats)
{
    const int d = Q->d;
    const int64_t nQ = Q->n, nS = S->n;
    if (nQ == 0) return DL_OK;
    // the SIMT join's bounds (|D32 - D| <= g32 D + a32) and the canonical sum's relative error g64
    const double g32 = metric == 1 ? (d + 4) * 1.1920928955078125e-07 : chi2_g32(d);
    const double a32 = metric == 1 ? d * 7.52316384526264e-37 : chi2_abs32(d);   // L1: d 2^-120
    const double g64 = (metric == 1 ? d + 4 : d + 8) * 1.1102230246251565e-16;
    HistTk f{};
    f.Q = Q->x32;
    f.S = S->x32;
    f.d = d;
    f.nS = (int)nS;
    f.k = k;
    f.q_orig = Q->orig;
    f.s_orig = S->orig;
    f.s_ids = S->ids;
    f.out_ids = out_ids;
    f.out_d = out_d;
    f.g32 = f32_ru(g32);
    f.a32 = f32_ru(a32);
    f.up = chi2_scale(std::max(Q->x_max, S->x_max));
    f.slack = f32_ru(4.0 * g64 + 1e-12);   // (1 + g64) / (1 - g64) and this product's roundings
    // rows per chunk: about 256 MB of distances (rows padded to whole 128-column tiles)
    f.ld = (nS + kSimtTile - 1) / kSimtTile * kSimtTile;
    const int64_t per_row = std::max<int64_t>(f.ld * 4, 256);
    int64_t rows = std::max<int64_t>(1, std::min<int64_t>(nQ, std::min<int64_t>((256LL << 20) / per_row, 65535LL * kSimtTile)));
    int sel = 1;   // CTAs of k_hist_select
    void *blk = nullptr;
    size_t b_v = 0, b_c = 0, b_d = 0;
    int rc = DL_OK;
    for (;; rows = (rows + 1) / 2) {   // fewer where memory is short
        sel = (int)std::min<int64_t>(rows, (int64_t)device_sm_count() * 4);
        b_v = al256((size_t)rows * f.ld * 4);
        b_c = al256((size_t)sel * kHtCap * 4);
        b_d = al256((size_t)sel * kHtCap * 8);
        rc = dev_alloc(&blk, b_v + 2 * b_c + b_d + 256, st);
        if (rc != DL_ENOMEM || rows == 1) break;
        clear_error();
    }
    if (rc) return rc;
    f.dist = (float *)blk;
    f.scr_c = (uint32_t *)((char *)blk + b_v);
    f.scr_v = (float *)((char *)blk + b_v + b_c);
    f.scr_d = (double *)((char *)blk + b_v + 2 * b_c);
    int *err = (int *)((char *)blk + b_v + 2 * b_c + b_d);
    unsigned long long *nf = (unsigned long long *)(err + 2);
    f.err = err;
    f.n_fp64 = nf;
    int launches = 0;
    cudaError_t e = cudaMemsetAsync(err, 0, 16, st);
    for (int64_t r0 = 0; r0 < nQ && e == cudaSuccess; r0 += rows) {
        f.row0 = r0;
        f.rows = (int)std::min<int64_t>(rows, nQ - r0);
        const bool vec = (d & 3) == 0;   // store rows start on 16 bytes
        const int gs = std::min(f.rows, sel);
        if (metric == 1)
            launches += vec ? launch_hist_chunk<1, true>(f, gs, st) : launch_hist_chunk<1, false>(f, gs, st);
        else
            launches += vec ? launch_hist_chunk<2, true>(f, gs, st) : launch_hist_chunk<2, false>(f, gs, st);
        e = cudaGetLastError();
    }
    int herr = 0;
    unsigned long long hf = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof herr, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hf, nf, sizeof hf, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    dev_free(blk, st);
    if (e != cudaSuccess) return cuda_fail(e, "histogram top-k");
    if (herr) {
        set_error("dl_topk_join: more than %d columns tie within the bound of a row's k-th distance", kHtCap);
        return DL_EOVERFLOW;
    }
    if (stats) {
        stats->pairs_evaluated = nQ * nS;
        stats->fp64_pairs = (int64_t)hf;
        stats->precision = DL_PREC_FP32;
        stats->kernels_launched = launches;
    }
    return DL_OK;
}

}  // namespace dl
