// topk.cu -- the top-k join (K4 + K7): for every query row, the k store rows
// with the smallest canonical distance, ordered by (distance, store row).
//
// The paper's reverse-image-search query (Sec. 6.2, q1: the closest image to a
// query image) is the k = 1 case. With h = q.x - ||x||^2/2 (D = ||q||^2 - 2h), on the caller's
// stream, for query rows in chunks that bound the workspace:
//   k_rowpar_topk      per query row: the bound terms and the canonical slack;
//   tc_join_kernel<.., kModeMaxima>   over every f-th tile of the store: each group of 16 or 64
//                      columns' best lower bound of h;
//   k_topk_theta       per row the k-th largest of them: at least k columns have h at or above it;
//   tc_join_kernel<.., kModeEps>      over the whole store, with that as the row's threshold: the
//                      epsilon-join's epilogue lists every column whose upper bound reaches it;
//   k_topk_dist        the candidates' FP32 distances, into a list per row;
//   k_topk_keep        per row: the k-th smallest upper bound of the listed distances and the columns
//                      that can still be in the top k;
//   k_topk_canon       their canonical FP64 distances;
//   k_topk_out         per row: an exact rank by (D64, caller's store row index).
// About k f columns of a row are listed: f balances the first pass against them (topk_stride). (While k
// stays well below the 1,024 maxima that k_topk_theta keeps apart: 256 rows against 262,144 x 128 take
// 0.98 ms at k = 700, and 24 at k = 1,024, with some 8,000 columns a row, more passes and a seventh of the
// rows scanned; the heaps below took 83 and 87.) A row with more than its list holds (near-duplicates side by side in the store) gets a tighter threshold
// from the distances it did list and the rows like it another pass (k_topk_refine); one that
// overflows again takes
//   k_topk_fallback    an exact scan of the whole store for that row (FP32 bound + radix select +
//                      FP64 + rank).
// The candidates of all rows share one list, which grows to what is left of kTkWorkspace (and holds at
// least as much as the rows' lists do together). Where the 16-bit bound exceeds the spread of the
// distances rows may list every column, and it overflows all the same: then fewer rows are taken at a
// time, down to 128 (a million candidates each). Past that some row holds more than its own list: those
// are tightened kTkRedos times, or go to the exact scan, and the others' candidates are listed again.
// (Bounded by the rows' lists alone, ordinary overflows took that way, with thresholds from the columns
// listed first: 512 rows, k = 10, against 1,000,000 x 128 in tight clusters 1.7 -> 520 ms.)
// Store rows are in norm order; outputs are written at the caller's row order. Thresholds from maxima of
// neighbouring columns of every f-th tile need near rows to be spread over the store. A store in cluster
// order puts them side by side: the passes over it run on a copy of its 16-bit rows in norm order
// (get_search), kept with the store. 2,048 queries, k = 100, against 131,072 x 128 of 1,024 views an
// object: 45.6 ms on the rows as they lie, nearly every list overflowing and 919 rows scanned; 0.45 ms so.
//
// Heaps of lower bounds kept by the epilogue's lanes in global memory did this in one pass over the
// store; every insert sifted through dependent loads while the other lanes of its warp waited.
// 4,096 queries against 1,000,003 x 256, k = 100: 18.6 ms then, 2.94 now; one query, k = 1: 0.53 ms, 0.195 (its 16
// column splits left 136 SMs idle).
// What bounds it now, of the 2.94 ms: the two tensor-core passes 0.30 + 1.17 ms, the candidates' rows 0.30,
// the canonical sums 0.49; of the 0.195 ms: the store's 512 MB of FP16 rows, 76 us.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "checked.cuh"
#include "cta.cuh"
#include "exact.cuh"
#include "kernels.h"

namespace dl {

constexpr int kTkGroups = 1024;      // group maxima k_topk_theta keeps apart (more are folded)
constexpr int kTkTermC = 64;         // candidates whose canonical terms are staged together
constexpr int kTkTerms = kTkTermC * 33;   // staged terms, padding included
constexpr int kTkRefines = 2;        // passes with tightened thresholds before the exact scan
constexpr int kTkScan = 1 << 30;     // list count of a row that is left to the exact scan
constexpr int kTkRedos = 2;          // passes with tightened thresholds while the shared list overflows
constexpr int kTkScanPasses = 4;     // then passes that name rows for the scan while it does (then: all)
constexpr int64_t kTkWorkspace = 1LL << 30;   // bytes of lists and candidates of a chunk of query rows
constexpr int kTkFallbackCap = 8192; // candidates a fallback block can rank

// Per query row: {canonical slack of h, unused, ||q - q~|| up, ||q~|| up}; padding rows get zeros.
__global__ void __launch_bounds__(256) k_rowpar_topk(const double *__restrict__ nq64, const float4 *__restrict__ rowb,
                                                     int64_t n, int64_t n_tot, double g64, double nq_max_s,
                                                     float4 *__restrict__ rowpar)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_tot) return;
    if (i >= n) {
        rowpar[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    // |h_canonical - h| <= |D64 - D| / 2 <= g64 * (||q||^2 + ||x||^2); doubled for margin
    const double delta = 2.0 * g64 * (nq64[i] + nq_max_s) * 1.0001 + 1e-30;
    const float4 rb = rowb[i];
    rowpar[i] = make_float4(__double2float_ru(delta), 0.f, rb.x, rb.y);
}

// Threshold of each row's listing pass from its group maxima: with T the k-th largest of them, a
// column of the top k has h + E + slack >= T, so the row lists the columns whose h~ reaches
// (T - slack) - E (-inf with fewer than k groups). Padding rows (+inf) list nothing. One warp per row,
// 32 values a lane (groups folded by maximum past 1,024: disjoint groups stay disjoint), no barriers;
// T is found bit by bit from the values' common prefix on and cut off after kTkBits bits, downwards. That
// resolves T to 2^-14 of its octave where the maxima share one, and to 2^-5 of it where they have both
// signs (the sign and the exponent take nine of the bits), which lets more columns in. A row's groups are
// loaded all at once: what bounds a few rows is that latency (one row of 976 groups: 4 us, 18 with a load
// at a time), what bounds many the counting steps (4,096 rows of 1,953 groups, k = 100: 54 us; 66 with a
// load at a time, 105 with a CTA a row and all 32 bits besides). It also empties the rows' lists.
constexpr int kTkBits = 14;

__global__ void __launch_bounds__(256) k_topk_theta(const float4 *__restrict__ rowpar, const float *__restrict__ gmax, int n_groups,
                                                    int64_t row0, int64_t nQ, int64_t rows_tot, int k, const int *__restrict__ row_k,
                                                    float4 *__restrict__ thr, int *__restrict__ cnt)
{
    const int lane = threadIdx.x & 31;
    const int64_t lr = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int64_t i = row0 + lr;
    if (i >= rows_tot) return;
    if (lane == 0 && i < nQ) cnt[lr] = 0;   // the row's list, empty
    const float inf = __int_as_float(0x7f800000);
    if (i >= nQ) {
        if (lane == 0) thr[i] = make_float4(inf, inf, 0.f, 0.f);
        return;
    }
    const float4 rp = rowpar[i];
    const unsigned kk = (unsigned)(row_k ? row_k[i] : k);
    float th = -inf;
    if (n_groups >= (int)kk) {
        unsigned v[kTkGroups / 32];
        const float *g = gmax + (size_t)lr * n_groups;
        unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll
        for (int s = 0; s < kTkGroups / 32; ++s)   // every load in flight
            v[s] = __float_as_uint(s * 32 + lane < n_groups ? __ldg(g + s * 32 + lane) : -inf);
        for (int j0 = kTkGroups; j0 < n_groups; j0 += kTkGroups)
#pragma unroll
            for (int s = 0; s < kTkGroups / 32; ++s)
                if (j0 + s * 32 + lane < n_groups) v[s] = __float_as_uint(fmaxf(__uint_as_float(v[s]), __ldg(g + j0 + s * 32 + lane)));
#pragma unroll
        for (int s = 0; s < kTkGroups / 32; ++s) {
            const float m = __uint_as_float(v[s]);
            v[s] = float_order_code(m);
            hi = max(hi, v[s]);
            if (m > -inf) lo = min(lo, v[s]);
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (kk == 1u) {
            th = float_from_order_code(hi);   // -inf when every group is padding
        } else if (lo <= hi) {
            // the largest code that at least kk values reach: its bits above the highest one in which
            // lo and hi differ are theirs (if kk values are finite at all)
            const int top = lo == hi ? -1 : 31 - __clz((int)(lo ^ hi));
            unsigned code = top < 31 ? hi & ~((2u << max(top, 0)) - 1u) : 0u;
            if (top < 0) code = hi;
            for (int bit = top; bit >= 0 && bit > top - kTkBits; --bit) {
                const unsigned t = code | (1u << bit);
                unsigned c = 0;
#pragma unroll
                for (int s = 0; s < kTkGroups / 32; ++s) c += v[s] >= t ? 1u : 0u;
                if (__reduce_add_sync(0xffffffffu, c) >= kk) code = t;
            }
            unsigned c = 0;   // with fewer than kk finite groups not even the prefix is reached
#pragma unroll
            for (int s = 0; s < kTkGroups / 32; ++s) c += v[s] >= code ? 1u : 0u;
            if (__reduce_add_sync(0xffffffffu, c) >= kk && code > float_order_code(-inf)) th = float_from_order_code(code);
        }
    }
    if (lane == 0) thr[i] = make_float4(inf, __fsub_rd(th, rp.x), rp.z, rp.w);
}

struct TopkRows {
    const float *Q, *S;
    int d, nS, k;
    int64_t row0, rows;    // this chunk's query rows
    int cap;               // list capacity of a row
    int *cnt;              // [rows] columns that reached the row's threshold (may exceed cap)
    uint32_t *col;         // [rows][cap]
    float *d32;            // [rows][cap] FP32 distances
    double *d64;           // [rows][cap] canonical distances of the kept columns
    uint32_t *kept;        // the kept columns' places in those lists, row by row
    unsigned long long *n_kept;
    const int32_t *s_row;  // store row of each column of the passes (NULL: the same)
    const int32_t *q_orig, *s_orig;
    const int64_t *s_ids;
    int64_t *out_ids;
    double *out_d2;
    const int *row_k;      // per query row k (NULL: k for every row)
    const int64_t *row_off;// per query row first output slot (NULL: caller row * k)
    float g32, abs32;      // FP32 distance bound: |D32 - D| <= g32 * D + abs32
    float slack;           // canonical slack factor for the keep test (relative)
};

// The listed candidates' FP32 distances (8-lane groups, 16-byte slices, four candidates a warp at a
// time), each into its row's list. What bounds it: the rows' reads, 8 d bytes a candidate and past the
// L2 for a store of its size. The grid is what is resident and windows are short until every warp has
// many: 1.6 M candidates, d = 256, 299 us (413 with 32-wide windows over a grid of one and a third
// times what is resident).
__global__ void __launch_bounds__(256) k_topk_dist(const TopkRows f, const uint2 *__restrict__ cand,
                                                   const unsigned long long *__restrict__ cand_cnt, unsigned long long cand_cap)
{
    const unsigned lane = threadIdx.x & 31;
    const unsigned long long n = min(*cand_cnt, cand_cap);
    const unsigned long long w0 = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned long long nw = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    // few candidates: four a warp, one round trip each; more: eight, until each warp has 256
    const unsigned win = n <= nw * 4 ? 4u : n < nw * 256 ? 8u : 32u;
    const bool in = lane < win;
    uint2 nxt = in && w0 * win + lane < n ? cand[w0 * win + lane] : make_uint2(0u, 0u);
    for (unsigned long long base = w0 * win; base < n; base += nw * win) {
        const unsigned long long i = base + lane;
        bool valid = in && i < n;
        const uint2 e = nxt;
        nxt = in && i + nw * win < n ? cand[i + nw * win] : make_uint2(0u, 0u);   // the next window, loaded early
        const int64_t lr = (int64_t)e.x - f.row0;
        uint32_t c = e.y & ~kBandFlag;
        if (valid && !DL_CHECK(lr >= 0 && lr < f.rows && c < (unsigned)f.nS, 10, i)) valid = false;
        if (valid && f.s_row) c = (uint32_t)__ldg(f.s_row + c);
        const unsigned vm = __ballot_sync(0xffffffffu, valid);
        const float s = warp_pairs_sq32(vm, f.Q + (valid ? (size_t)e.x * f.d : 0), f.S + (valid ? (size_t)c * f.d : 0), f.d);
        if (valid) {   // a place in the row's list: one atomic per run of lanes with the same row
            const unsigned peers = __match_any_sync(vm, e.x);
            const int leader = __ffs(peers) - 1;
            int at = 0;
            if ((int)lane == leader) at = atomicAdd(f.cnt + lr, __popc(peers));
            at = __shfl_sync(peers, at, leader) + __popc(peers & ((1u << lane) - 1u));
            if (at < f.cap) {
                f.col[(size_t)lr * f.cap + at] = c;
                f.d32[(size_t)lr * f.cap + at] = s;
            }
        }
    }
}

__device__ __forceinline__ float upper32(const TopkRows &f, float s)
{
    return __fmul_ru(__fadd_ru(__fmul_ru(s, 1.0f + f.g32), f.abs32), 1.0f + f.slack);
}
__device__ __forceinline__ float lower32(const TopkRows &f, float s)
{
    return __fsub_rd(__fmul_rd(s, 1.0f - f.g32), f.abs32);
}

// Thresholds of another listing pass: an overflowed row's from the k-th smallest of the distances it
// did list (at least k columns lie within its upper bound u, so a column with D > u (1 + slack) is not
// in the top k: h < RD((||q||^2_dn - e2 (1 + 2 g64)) / 2) - E proves that, as in k_rowpar), or none and
// the exact scan (`scan`; 2: every row); every other row lists nothing, its list stands -- or, when the
// shared list was too short (`redo`), what its threshold admits once more. One CTA per row of the chunk.
__global__ void __launch_bounds__(256) k_topk_refine(const TopkRows f, const double *__restrict__ nq64, int dp, double g64,
                                                     int64_t rows_pad, int redo, int scan, const float4 *__restrict__ rowpar,
                                                     float4 *__restrict__ thr)
{
    __shared__ unsigned s_cnt[2];
    const int64_t lr = blockIdx.x;
    const int64_t i = f.row0 + lr;
    const float inf = __int_as_float(0x7f800000);
    const float4 none = make_float4(inf, inf, 0.f, 0.f);
    const int m = lr >= f.rows || scan == 2 ? kTkScan : f.cnt[lr];
    if (m <= f.cap && redo) {
        if (threadIdx.x == 0) f.cnt[lr] = 0;
        return;
    }
    if (m <= f.cap || m >= kTkScan || scan) {
        if (threadIdx.x == 0) {
            if (lr < rows_pad) thr[i] = none;
            if (lr < f.rows && m > f.cap) f.cnt[lr] = kTkScan;
        }
        return;
    }
    if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0u;
    __syncthreads();
    const int kk = f.row_k ? f.row_k[i] : f.k;   // at most k, and a list holds more than k
    const float *v = f.d32 + (size_t)lr * f.cap;
    unsigned kb = 0u;
    int turn = 0;
    for (int bit = 30; bit >= 0; --bit) {   // bits of the k-th smallest (non-negative floats order like them)
        const unsigned t = kb | (1u << bit);
        unsigned c = 0;
        for (int a = threadIdx.x; a < f.cap; a += 256) c += __float_as_uint(v[a]) < t ? 1u : 0u;
        if (cta_count(c, s_cnt, turn++) < (unsigned)kk) kb = t;
    }
    if (threadIdx.x == 0) {
        const double e2 = (double)upper32(f, __uint_as_float(kb));
        const double nq_dn = __dmul_rd(nq64[i], 1.0 - (double)(dp + 2) * 2.220446049250313e-16);
        const double rej = __dsub_rd(nq_dn, __dmul_ru(e2, 1.0 + 2.0 * g64)) * 0.5;
        const float4 rp = rowpar[i];
        // never below the pass before: its candidates fitted the shared list, so will these
        thr[i] = make_float4(inf, fmaxf(thr[i].y, __fsub_rd(__double2float_rd(rej), rp.x)), rp.z, rp.w);
        f.cnt[lr] = 0;
    }
}

__global__ void __launch_bounds__(256) k_topk_name(int *__restrict__ rows, int row0, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) rows[i] = row0 + i;
}

// One warp per query row: the columns of its list that can still be in the top k, moved to the list's
// front (their count becomes the row's) and named in the chunk's kept list. A row whose list
// overflowed is named in over_rows instead (n_over: how many, and above bit 32 those not yet left to the
// exact scan).
__global__ void __launch_bounds__(256) k_topk_keep(const TopkRows f, int *__restrict__ over_rows, unsigned long long *__restrict__ n_over)
{
    constexpr int kReg = 8;   // distances a lane keeps in registers
    const int lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t lr = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; lr < f.rows; lr += nw) {
        const int m0 = f.cnt[lr];
        if (m0 > f.cap) {
            if (lane == 0) over_rows[(unsigned)atomicAdd(n_over, m0 < kTkScan ? 1ULL | 1ULL << 32 : 1ULL)] = (int)(f.row0 + lr);
            continue;
        }
        const unsigned kk = (unsigned)(f.row_k ? f.row_k[f.row0 + lr] : f.k);
        float *d32 = f.d32 + (size_t)lr * f.cap;
        uint32_t *col = f.col + (size_t)lr * f.cap;
        float lim = __int_as_float(0x7f800000);
        if (m0 > (int)kk) {   // the k-th smallest distance's upper bound: at least k columns lie within it
            unsigned v[kReg], lo = 0x7fffffffu, hi = 0u;
#pragma unroll
            for (int s = 0; s < kReg; ++s) {
                v[s] = s * 32 + lane < m0 ? __float_as_uint(d32[s * 32 + lane]) : 0x7fffffffu;
                lo = min(lo, v[s]);
                if (v[s] != 0x7fffffffu) hi = max(hi, v[s]);
            }
            for (int a = kReg * 32 + lane; a < m0; a += 32) {
                const unsigned w = __float_as_uint(d32[a]);
                lo = min(lo, w);
                hi = max(hi, w);
            }
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            unsigned kb = lo;   // the k-th smallest's bits: its prefix is lo's and hi's common one
            if (kk > 1u && lo != hi) {
                const int top = 31 - __clz((int)(lo ^ hi));
                kb = hi & ~((2u << top) - 1u);
                for (int bit = top; bit >= 0; --bit) {
                    const unsigned t = kb | (1u << bit);
                    unsigned c = 0;
#pragma unroll
                    for (int s = 0; s < kReg; ++s) c += v[s] < t ? 1u : 0u;
                    for (int a = kReg * 32 + lane; a < m0; a += 32) c += __float_as_uint(d32[a]) < t ? 1u : 0u;
                    if (__reduce_add_sync(0xffffffffu, c) < kk) kb = t;
                }
            }
            lim = upper32(f, __uint_as_float(kb));
        }
        int m = 0;
        for (int b = 0; b < m0; b += 32) {   // moved down in place: a window is read before it is written
            const int a = b + lane;
            const float w = a < m0 ? d32[a] : 0.f;
            const uint32_t c = a < m0 ? col[a] : 0u;
            const bool keep = a < m0 && lower32(f, w) <= lim;
            const unsigned km = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                d32[m + __popc(km & lt)] = w;
                col[m + __popc(km & lt)] = c;
            }
            __syncwarp();
            m += __popc(km);
        }
        unsigned long long at = 0;
        if (lane == 0) {
            f.cnt[lr] = m;
            if (m) at = atomicAdd(f.n_kept, (unsigned long long)m);
        }
        at = __shfl_sync(0xffffffffu, at, 0);
        for (int a = lane; a < m; a += 32) f.kept[at + a] = (uint32_t)((size_t)lr * f.cap + a);
    }
}

// The kept columns' canonical distances, up to 64 columns of any rows at a time: every thread forms
// terms, a run of each column's, then a thread per column adds its own in ascending k. What bounds it:
// the FP64 pipe, costed per warp instruction (16 cycles of an SM): two operations a term with every
// lane busy, the subtraction and the conversions done by the integer units (abs_diff64). The whole call
// of 4,096 queries, k = 100, d = 256: 3.12 -> 2.94 ms against three operations; with the squares in
// integers too (128-bit products, some 150 instructions) 3.13.
__global__ void __launch_bounds__(128) k_topk_canon(const TopkRows f)
{
    __shared__ double sh_t[kTkTerms];
    __shared__ const float *sh_q[kTkTermC], *sh_x[kTkTermC];
    const int tid = threadIdx.x;
    const unsigned long long n = *f.n_kept;
    for (unsigned long long b0 = (unsigned long long)blockIdx.x * kTkTermC; b0 < n; b0 += (unsigned long long)gridDim.x * kTkTermC) {
        const int na = (int)min((unsigned long long)kTkTermC, n - b0);
        uint32_t slot = 0;
        if (tid < na) {
            slot = f.kept[b0 + tid];
            const uint32_t c = f.col[slot];
            sh_q[tid] = f.Q + (size_t)(f.row0 + slot / f.cap) * f.d;
            sh_x[tid] = f.S + (size_t)(DL_CHECK(c < (unsigned)f.nS, 11, c) ? c : 0u) * f.d;
        }
        const int run = na > 32 ? 32 : na > 16 ? 64 : na > 8 ? 128 : 256;   // terms of a column staged at a time
        const int sh = 31 - __clz(run), ld = run + 1;   // na * ld <= kTkTerms
        double s = 0.0;
        __syncthreads();
        for (int k0 = 0; k0 < f.d; k0 += run) {
            const int nk = min(run, f.d - k0);
#pragma unroll 4
            for (int e = tid; e < na << sh; e += 128) {
                const int a = e >> sh, k = e & (run - 1);
                if (k < nk) {
                    const double t = abs_diff64(__ldg(sh_q[a] + k0 + k), __ldg(sh_x[a] + k0 + k));
                    sh_t[a * ld + k] = __dmul_rn(t, t);
                }
            }
            __syncthreads();
            if (tid < na)
                for (int k = 0; k < nk; ++k) s = __dadd_rn(s, sh_t[tid * ld + k]);
            __syncthreads();
        }
        if (tid < na) f.d64[slot] = s;
    }
}

// One warp per query row: the exact rank of its kept columns by (canonical distance, caller's store
// row) and its outputs.
__global__ void __launch_bounds__(256) k_topk_out(const TopkRows f)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t lr = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; lr < f.rows; lr += nw) {
        const int m = f.cnt[lr];
        if (m > f.cap) continue;   // overflowed: solved elsewhere
        const int64_t i = f.row0 + lr;
        const int kk = f.row_k ? f.row_k[i] : f.k;
        const double *d64 = f.d64 + (size_t)lr * f.cap;
        const uint32_t *col = f.col + (size_t)lr * f.cap;
        const int64_t base = f.row_off ? f.row_off[i] : (int64_t)f.q_orig[i] * f.k;
        for (int a0 = 0; a0 < m; a0 += 32) {
            const int a = a0 + lane;
            const uint32_t ca = a < m ? col[a] : 0u;
            const double da = a < m ? d64[a] : 0.0;
            const int32_t oa = a < m ? f.s_orig[ca] : 0;
            int rank = 0;
            for (int b0 = 0; b0 < m; b0 += 32) {   // 32 others at a time, passed around the warp
                const int bb = b0 + lane;
                const uint32_t cb = bb < m ? col[bb] : 0u;
                const double db = bb < m ? d64[bb] : 0.0;
                const int32_t ob = bb < m ? f.s_orig[cb] : 0;
                const int nb = min(32, m - b0);
                for (int j = 0; j < nb; ++j) {
                    const double dj = __shfl_sync(0xffffffffu, db, j);
                    const int32_t oj = __shfl_sync(0xffffffffu, ob, j);
                    // canonical distances are non-negative: they order like their bits
                    rank += __double_as_longlong(dj) < __double_as_longlong(da) || (__double_as_longlong(dj) == __double_as_longlong(da) && oj < oa);
                }
            }
            if (a < m && rank < kk) {
                f.out_ids[base + rank] = f.s_ids[ca];
                f.out_d2[base + rank] = da;
            }
        }
        for (int t = m + lane; t < kk; t += 32) {
            f.out_ids[base + t] = -1;
            f.out_d2[base + t] = -1.0;
        }
    }
}

__device__ __forceinline__ double canon_d64(const float *__restrict__ q, const float *__restrict__ x, int d)
{
    double s = 0.0;
    for (int k = 0; k < d; ++k) {
        const double t = __dsub_rn((double)__ldg(q + k), (double)__ldg(x + k));
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

struct TopkFb {
    const float *Q, *S;
    int d, nS, k;
    const int *rows;        // flagged query rows (store order)
    int n_rows;
    float *scr_u, *scr_l;   // [n_rows][nS]
    uint32_t *scr_c;        // [n_rows][kTkFallbackCap]
    double *scr_d;          // [n_rows][kTkFallbackCap]
    const int32_t *q_orig, *s_orig;
    const int64_t *s_ids;
    int64_t *out_ids;
    double *out_d2;
    const int *row_k;
    const int64_t *row_off;
    float g32, abs32, slack;
    int *err;               // set to 1 when a row has more near-ties than the fallback can rank
    unsigned long long *n_fp64;
};

// One block per flagged row: exact scan of the whole store.
__global__ void __launch_bounds__(256) k_topk_fallback(const TopkFb f)
{
    __shared__ unsigned hist[256];
    __shared__ unsigned s_prefix, s_rank;
    __shared__ int s_m;
    const int b = blockIdx.x;
    if (b >= f.n_rows) return;
    const int i = f.rows[b];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    float *u = f.scr_u + (size_t)b * f.nS;
    float *l = f.scr_l + (size_t)b * f.nS;
    uint32_t *cl = f.scr_c + (size_t)b * kTkFallbackCap;
    double *cd = f.scr_d + (size_t)b * kTkFallbackCap;
    const float *q = f.Q + (size_t)i * f.d;
    // 1. FP32 distance bounds to every store row
    for (int j = warp; j < f.nS; j += nw) {
        const float *x = f.S + (size_t)j * f.d;
        float s = 0.f;
        for (int k = lane; k < f.d; k += 32) {
            const float t = __ldg(q + k) - __ldg(x + k);
            s = fmaf(t, t, s);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            u[j] = __fadd_ru(__fmul_ru(s, 1.0f + f.g32), f.abs32);
            l[j] = __fsub_rd(__fmul_rd(s, 1.0f - f.g32), f.abs32);
        }
    }
    __syncthreads();
    // 2. k-th smallest upper bound by radix select on the (non-negative) float bits
    const int kk = f.row_k ? f.row_k[i] : f.k;
    float kth = __int_as_float(0x7f800000);
    if (f.nS > kk) {
        if (tid == 0) {
            s_prefix = 0u;
            s_rank = (unsigned)(kk - 1);
        }
        for (int shift = 24; shift >= 0; shift -= 8) {
            for (int t = tid; t < 256; t += blockDim.x) hist[t] = 0u;
            __syncthreads();
            const unsigned pre = s_prefix;
            const unsigned mask_hi = (shift == 24) ? 0u : (0xffffffffu << (shift + 8));
            for (int j = tid; j < f.nS; j += blockDim.x) {
                const unsigned v = __float_as_uint(u[j]);
                if ((v & mask_hi) == (pre & mask_hi)) atomicAdd(&hist[(v >> shift) & 255u], 1u);
            }
            __syncthreads();
            if (tid == 0) {
                unsigned r = s_rank, acc = 0u;
                int dg = 0;
                for (; dg < 256; ++dg) {
                    if (acc + hist[dg] > r) break;
                    acc += hist[dg];
                }
                s_rank = r - acc;
                s_prefix = pre | ((unsigned)dg << shift);
            }
            __syncthreads();
        }
        kth = __uint_as_float(s_prefix);
    }
    kth = __fmul_ru(kth, 1.0f + f.slack);
    // 3. every row whose lower bound is within the k-th upper bound
    if (tid == 0) s_m = 0;
    __syncthreads();
    for (int j = tid; j < f.nS; j += blockDim.x) {
        if (l[j] <= kth) {
            const int pos = atomicAdd(&s_m, 1);
            if (pos < kTkFallbackCap) cl[pos] = (uint32_t)j;
        }
    }
    __syncthreads();
    const int m = s_m;
    if (m > kTkFallbackCap) {
        if (tid == 0) atomicExch(f.err, 1);
        return;
    }
    // 4. canonical distances, 5. exact rank by (D64, caller's store row)
    for (int a = tid; a < m; a += blockDim.x) cd[a] = canon_d64(q, f.S + (size_t)cl[a] * f.d, f.d);
    if (tid == 0) atomicAdd(f.n_fp64, (unsigned long long)m);
    __syncthreads();
    const int64_t base = f.row_off ? f.row_off[i] : (int64_t)f.q_orig[i] * f.k;
    int64_t *oid = f.out_ids + base;
    double *od = f.out_d2 + base;
    for (int a = tid; a < m; a += blockDim.x) {
        const double da = cd[a];
        const int32_t oa = f.s_orig[cl[a]];
        int rank = 0;
        for (int bb = 0; bb < m; ++bb) {
            const double db = cd[bb];
            rank += (db < da) || (db == da && f.s_orig[cl[bb]] < oa);
        }
        if (rank < kk) {
            oid[rank] = f.s_ids[cl[a]];
            od[rank] = da;
        }
    }
    for (int t = m + tid; t < kk; t += blockDim.x) {
        oid[t] = -1;
        od[t] = -1.0;
    }
}

// ------------------------------------------------------------------ host side
static size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

// Every how many-th tile the first pass takes. That pass costs 2 d nS / f operations a row, and about
// k f columns of a row are listed at some 0.2 ns each (a slow-path visit and an 8 d byte recheck):
// the sum is least at f = sqrt(d nS / (1.6e5 k)). At most 16 (a row's list grows with f), and above 1
// only as far as 8 k groups of 16 columns stay.
static int topk_stride(int64_t nS, int dp, int k)
{
    const double f = std::sqrt((double)nS * dp / (1.6e5 * k));
    return (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)std::min(f, 16.0), nS / (128LL * k)));
}

struct TopkShape {
    int stride;         // tiles of the first pass
    int cap;            // list capacity of a row
    int gran;           // columns of a group
    int n_groups;       // groups of a row (0: every column fits the list, no first pass)
    int64_t per_cand;   // candidates of a row provided for at first (never more than cap)
    int64_t bytes() const { return 4LL * n_groups + 20LL * cap + 4 + 8LL * cap; }   // of a row, its list's candidates included
};

static TopkShape topk_shape(int64_t nS, int dp, int k, int BN)
{
    TopkShape s;
    s.stride = topk_stride(nS, dp, k);
    // the k-th best of every f-th tile is about the k f-th of the store, with a spread of f sqrt(k)
    // (at k = 1 geometric: a row in 10^11 has more than 24 f columns above it)
    s.cap = (2 * k * s.stride + 16 * s.stride + 128 + 31) / 32 * 32;
    const int64_t nt_sub = ((nS + BN - 1) / BN + s.stride - 1) / s.stride;
    s.gran = nt_sub * BN / 64 >= 8LL * k ? 64 : 16;
    const bool all = nS <= s.cap;
    s.n_groups = all ? 0 : (int)(nt_sub * BN / s.gran);
    s.per_cand = all ? nS : std::min<int64_t>(nS, (int64_t)k * s.stride * 3 / 2 + 16LL * s.stride + 64);
    return s;
}

// Query rows whose lists and candidates stay within kTkWorkspace (whole 128-row tiles, at least one).
static int64_t topk_chunk_rows(int64_t rows, int64_t per_row)
{
    return std::min<int64_t>(rows, std::max<int64_t>(1, kTkWorkspace / (per_row * 128)) * 128);
}

int64_t topk_scratch_bytes(int64_t nQ, int64_t nS, int dp, int k)
{
    const int64_t per_row = topk_shape(nS, dp, k, 256).bytes();
    return std::min(nQ, topk_chunk_rows((nQ + 127) / 128 * 128, per_row)) * per_row + 65536 * 8;
}

// Top-k of every row of Q against S into out_ids / out_d2. k is the largest k of
// any row; row_k (device, optional) gives each row's own k and
// row_off (device, optional) each row's first output slot (default: caller row * k).
int topk_core(const dl_store *Q, const dl_store *S, int k, const int *row_k, const int64_t *row_off,
              int64_t *out_ids, double *out_d2, const dl_join_opts &o, cudaStream_t st, dl_join_stats *stats)
{
    const int64_t nQ = Q->n, nS = S->n;
    const int d = Q->d;
    if (o.tile_n != 0 && o.tile_n != 128 && o.tile_n != 256) {
        set_error("top-k: tile_n must be 0, 128 or 256");
        return DL_EINVAL;
    }
    const bool use_tc = (o.precision != DL_PREC_FP32) && Q->dp <= 512;
    // the 16-bit copies' format: FP16 where both stores hold it, unless BF16 was asked for
    const bool f16 = Q->h.fmt == kHalfF16 && S->h.fmt == kHalfF16;
    if (o.precision == DL_PREC_FP16 && !(f16 && use_tc)) {
        set_error("top-k: FP16 needs features within FP16's range in both stores and d <= 512");
        return DL_EUNSUPPORTED;
    }
    const int fmt = f16 && o.precision != DL_PREC_BF16 ? kHalfF16 : kHalfBF16;
    bool tune_trial = false;
    if ((o.epilogue_warps != 0 && o.epilogue_warps != 8 && o.epilogue_warps != 16) ||
        (o.epilogue_warps == 16 && o.tile_n == 128)) {
        set_error("top-k: epilogue_warps must be 0, 8 or 16 (16: tile_n 0 or 256)");
        return DL_EINVAL;
    }
    int code = (o.tile_n ? o.tile_n : 256) | (o.epilogue_warps == 16 ? kTuneWide : 0);
    const int tune_kind = fmt == kHalfF16 ? kTuneTopk16 : kTuneTopk;
    const int prec = !use_tc ? DL_PREC_FP32 : fmt == kHalfF16 ? DL_PREC_FP16 : DL_PREC_BF16;
    if (nQ == 0) {   // no rows: nothing to run, time or tune
        if (stats) {
            stats->precision = prec;
            stats->tile_n = use_tc ? tune_bn(code) : 0;
            stats->epilogue_warps = !use_tc ? 0 : tune_wide(code) ? 16 : 8;
        }
        return DL_OK;
    }
    if (use_tc && o.tile_n == 0 && o.epilogue_warps == 0) code = tune_pick(Q->dp, tune_kind, nQ, nS, &tune_trial);
    const int BN = tune_bn(code);
    const bool wide = use_tc && tune_wide(code);   // 16 epilogue warps
    const int sms = device_sm_count();
    const int64_t mt = (nQ + 127) / 128, rows = mt * 128;
    const int64_t nt = (nS + BN - 1) / BN;

    // the two passes' shape, and the query rows of a chunk
    const TopkShape sh = topk_shape(nS, Q->dp, k, BN);
    const int f = sh.stride, cap = sh.cap, gran = sh.gran, n_groups = sh.n_groups;
    const int64_t nt_sub = (nt + f - 1) / f, per_cand = sh.per_cand;
    const bool all = n_groups == 0;   // every column fits a row's list: no first pass
    int64_t chunk_rows = topk_chunk_rows(rows, sh.bytes());

    const size_t b_rowpar = al256((size_t)rows * sizeof(float4)), b_frows = al256((size_t)nQ * sizeof(int));
    const bool timing = o.timing || tune_trial;
    void *ws = nullptr, *cws = nullptr;
    int rc = dev_alloc(&ws, 2 * b_rowpar + b_frows + 256, st);
    if (rc) return rc;
    float4 *rowpar = (float4 *)ws, *thr = (float4 *)((char *)ws + b_rowpar);
    int *frows = (int *)((char *)ws + 2 * b_rowpar);
    // [0] rows named in frows (k_topk_keep) [1] fp64 evals [2] more near-ties than the fallback ranks [3] wait expired
    // [4] candidates of a pass [5] columns kept by it
    unsigned long long *misc = (unsigned long long *)((char *)ws + 2 * b_rowpar + b_frows);
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    if (timing)
        for (auto &e : ev) cudaEventCreate(&e);
    auto done = [&](int code) {
        for (auto &e : ev)
            if (e) cudaEventDestroy(e);
        dev_free(cws, st);
        dev_free(ws, st);
        if (code) cudaStreamSynchronize(st);
        return code;
    };
    unsigned long long *h = nullptr;
    rc = pinned_counters(&h);
    if (rc) return done(rc);
    std::memset(h, 0, 48);
    cudaError_t e = cudaMemsetAsync(misc, 0, 256, st);
    if (e != cudaSuccess) return done(cuda_fail(e, "top-k memset"));
    if (timing) cudaEventRecord(ev[0], st);
    int launches = 0;
    auto launched = [&](const char *what) {
        count_launch();
        ++launches;
        const cudaError_t le = cudaGetLastError();
        return le == cudaSuccess ? DL_OK : cuda_fail(le, what);
    };
    auto reset = [&]() {   // a pass's counters
        cudaError_t re = cudaMemsetAsync(misc, 0, 8, st);
        if (re == cudaSuccess) re = cudaMemsetAsync(misc + 4, 0, 16, st);
        return re == cudaSuccess ? DL_OK : cuda_fail(re, "top-k memset");
    };
    auto read_misc = [&]() {
        cudaError_t re = cudaMemcpyAsync(h, misc, 48, cudaMemcpyDeviceToHost, st);
        if (re == cudaSuccess) re = cudaStreamSynchronize(st);
        return re == cudaSuccess ? DL_OK : cuda_fail(re, "top-k");
    };
    const double g64 = gamma64(d), g32 = gamma32(d);
    TopkRows t{};
    t.Q = Q->x32;
    t.S = S->x32;
    t.d = d;
    t.nS = (int)nS;
    t.k = k;
    t.cap = cap;
    t.q_orig = Q->orig;
    t.s_orig = S->orig;
    t.s_ids = S->ids;
    t.out_ids = out_ids;
    t.out_d2 = out_d2;
    t.row_k = row_k;
    t.row_off = row_off;
    t.g32 = f32_ru(g32 * 1.0000001);
    t.abs32 = f32_ru((double)(d + 8) * 1.401298464324817e-45 * 4.0);
    t.slack = f32_ru(4.0 * g64 + 1e-12);
    t.n_kept = misc + 5;
    int64_t flagged = 0;   // rows named in frows for the exact scan
    int64_t fp64 = 0;      // canonical distances of the other rows
    if (nS == 0 || use_tc) {
        Half *hQ = nullptr, *hS = nullptr;
        const float *beta = S->beta;
        const CUtensorMap *tmA = nullptr, *tmB = nullptr;
        if (nS > 0) {
            rc = get_half(const_cast<dl_store *>(Q), fmt, st, &hQ);
            if (!rc && S->clabel && !all) {   // a store in cluster order: its copy in norm order, memory permitting
                Store::SearchCopy *sc = nullptr;
                rc = get_search(const_cast<dl_store *>(S), fmt, st, &sc);
                if (!rc) {
                    hS = &sc->h;
                    beta = sc->beta;
                    t.s_row = sc->row;
                } else if (rc == DL_ENOMEM) {
                    rc = DL_OK;
                    clear_error();
                }
            }
            if (!rc && !hS) rc = get_half(const_cast<dl_store *>(S), fmt, st, &hS);
            if (!rc) rc = get_tmap(const_cast<dl_store *>(Q), hQ, 128, &tmA);
            if (!rc) rc = get_tmap(const_cast<dl_store *>(S), hS, BN, &tmB);
            if (!rc) {
                k_rowpar_topk<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(Q->nq64, hQ->rowb, nQ, rows, g64,
                                                                              (double)S->nq_max * 1.0001, rowpar);
                rc = launched("k_rowpar_topk launch");
            }
        }
        int64_t cand_cap = 0, cand_max = 0;
        size_t b_g = 0, b_l = 0, b_n = 0, b_d = 0;
        auto size_chunk = [&]() {
            cand_max = chunk_rows * cap + 65536;
            cand_cap = std::min<int64_t>(std::min<int64_t>(chunk_rows, nQ) * per_cand + 65536, cand_max);
            cand_max = std::max<int64_t>(cand_max, (kTkWorkspace - chunk_rows * (sh.bytes() - 8LL * cap)) / 8);
            b_g = al256((size_t)chunk_rows * n_groups * 4);
            b_l = al256((size_t)chunk_rows * cap * 4);
            b_n = al256((size_t)chunk_rows * 4);
            b_d = al256((size_t)chunk_rows * cap * 8);
        };
        size_chunk();
        for (int64_t row0 = 0; row0 < nQ && !rc;) {
            int64_t cr = 0;
            int refined = 0, redos = 0;
            unsigned long long listed = 0, open = 0;   // of the last complete pass: candidates, rows past their lists
            bool redo = false;   // the pass before overflowed the shared list
            for (int pass = 0; !rc; ++pass) {   // listing passes over this chunk
                while (!cws) {
                    rc = dev_alloc(&cws, b_g + 3 * b_l + b_n + b_d + (size_t)cand_cap * 8, st);
                    if (rc != DL_ENOMEM) break;
                    // memory is short: a list that is no larger than it must be, then fewer rows at a time
                    if (cand_cap > chunk_rows * cap + 65536) {
                        cand_cap = cand_max = chunk_rows * cap + 65536;
                    } else if (chunk_rows > 128) {
                        chunk_rows = std::max<int64_t>(128, chunk_rows / 256 * 128);
                        size_chunk();
                    } else {
                        break;
                    }
                    clear_error();
                }
                if (rc) break;
                cr = std::min(chunk_rows, nQ - row0);
                const int64_t cr_pad = (cr + 127) / 128 * 128;
                float *gmax = (float *)cws;
                t.col = (uint32_t *)((char *)cws + b_g);
                t.d32 = (float *)((char *)cws + b_g + b_l);
                t.kept = (uint32_t *)((char *)cws + b_g + 2 * b_l);
                t.cnt = (int *)((char *)cws + b_g + 3 * b_l);
                t.d64 = (double *)((char *)cws + b_g + 3 * b_l + b_n);
                uint2 *cand = (uint2 *)((char *)cws + b_g + 3 * b_l + b_n + b_d);
                t.row0 = row0;
                t.rows = cr;
                TcLaunch L;
                std::memset(&L.p, 0, sizeof L.p);
                if (nS > 0) {
                    L.tmA = tmA;
                    L.tmB = tmB;
                    L.BN = BN;
                    L.wide = wide;
                    L.p.nR = (int)nQ;
                    L.p.nS = (int)nS;
                    L.p.kc = Q->dp / 64;
                    L.p.fmt = fmt == kHalfBF16;
                    L.p.scale = hQ->scale * hS->scale;
                    tc_plan(BN, Q->dp / 64, &L.p.stages, &L.p.a_slots, false, false, wide);
                    L.p.beta = beta;
                    L.p.cstat = hS->cstat;
                    L.p.err = (int *)(misc + 3);
                    L.p.m0 = (int)(row0 / 128);
                }
                if (pass == 0) {   // thresholds from the first pass's group maxima
                    if (nS > 0 && !all) {
                        L.p.rowpar = rowpar;
                        L.p.tile_stride = f;
                        L.p.gmax = gmax;
                        L.p.n_groups = n_groups;
                        L.p.gran = gran;
                        L.p.row0 = (int)row0;
                        tc_grid_units(&L, cr_pad / 128, nt_sub, sms);
                        rc = launch_tc_join(L, st, kModeMaxima);
                        ++launches;
                        L.p.tile_stride = 1;
                    }
                    if (!rc && nS > 0) {
                        k_topk_theta<<<(unsigned)(cr_pad / 8), 256, 0, st>>>(rowpar, gmax, n_groups, row0, nQ, row0 + cr_pad, k, row_k, thr, t.cnt);
                        rc = launched("k_topk_theta launch");
                    } else if (!rc) {   // an empty store: empty lists
                        e = cudaMemsetAsync(t.cnt, 0, b_n, st);
                        if (e != cudaSuccess) rc = cuda_fail(e, "top-k memset");
                    }
                } else {   // tighter thresholds for the rows whose list overflowed, then the exact scan
                    redo ? ++redos : ++refined;
                    const int scan = !redo || redos <= kTkRedos ? 0 : redos <= kTkRedos + kTkScanPasses ? 1 : 2;
                    k_topk_refine<<<(unsigned)cr_pad, 256, 0, st>>>(t, Q->nq64, Q->dp, g64, cr_pad, redo, scan, rowpar, thr);
                    rc = launched("k_topk_refine launch");
                    if (!rc) rc = reset();
                }
                if (!rc && nS > 0) {
                    L.p.rowpar = thr;
                    L.p.cand = cand;
                    L.p.cand_cnt = misc + 4;
                    L.p.cand_cap = (unsigned long long)cand_cap;
                    tc_plan(BN, Q->dp / 64, &L.p.stages, &L.p.a_slots, false, false, wide, true);
                    tc_grid_units(&L, cr_pad / 128, nt, sms);
                    rc = launch_tc_join(L, st);
                    ++launches;
                    if (!rc) {
                        const int64_t grid = std::min<int64_t>((cand_cap + 255) / 256, (int64_t)sms * 6);   // 6 resident a SM
                        k_topk_dist<<<(unsigned)grid, 256, 0, st>>>(t, cand, misc + 4, (unsigned long long)cand_cap);
                        rc = launched("k_topk_dist launch");
                    }
                }
                if (!rc) {
                    const unsigned gw = (unsigned)std::min<int64_t>((cr + 7) / 8, (int64_t)sms * 32);   // a warp a row
                    k_topk_keep<<<gw, 256, 0, st>>>(t, frows + flagged, misc);
                    rc = launched("k_topk_keep launch");
                    if (!rc && nS > 0) {
                        k_topk_canon<<<(unsigned)std::min<int64_t>((cr * cap + kTkTermC - 1) / kTkTermC, (int64_t)sms * 12), 128, 0, st>>>(t);
                        rc = launched("k_topk_canon launch");
                    }
                    if (!rc) {
                        k_topk_out<<<gw, 256, 0, st>>>(t);
                        rc = launched("k_topk_out launch");
                    }
                }
                if (timing && row0 + cr >= nQ && pass == 0) cudaEventRecord(ev[1], st);
                if (!rc) rc = read_misc();
                if (rc) break;
                if (h[3]) {
                    set_error("top-k: a bounded device wait expired");
                    return done(DL_ETIMEOUT);
                }
                redo = h[4] > (unsigned long long)cand_cap;   // lists short of candidates: what came of them is written again
                // nearly every column of nearly every row: no lists, the chunk's rows all take the scan
                if (redo && 4 * n_groups >= 5 * k && 8 * h[4] > 7ULL * (unsigned long long)cr * (unsigned long long)nS) {
                    k_topk_name<<<(unsigned)((cr + 255) / 256), 256, 0, st>>>(frows + flagged, (int)row0, (int)cr);
                    rc = launched("k_topk_name launch");
                    flagged += cr;
                    break;
                }
                if (redo && (cand_cap < cand_max || chunk_rows > 128)) {   // again, with the list's exact size or fewer rows
                    const int64_t want = (int64_t)(h[4] + h[4] / 8) + 1024;
                    if (cand_cap < cand_max) {
                        cand_cap = std::min(want, cand_max);
                    } else {
                        chunk_rows = std::max<int64_t>(128, (int64_t)((double)cr * (double)cand_max / (double)want) / 128 * 128);
                        size_chunk();
                        cand_cap = cand_max;
                    }
                    dev_free(cws, st);
                    cws = nullptr;
                    pass = -1;
                    refined = redos = 0;
                    listed = open = 0;
                    rc = reset();
                    continue;
                }
                // rows that no threshold helps, the bound being as wide as the distances lie apart: three
                // quarters of all columns past one from enough groups, or a tighter one that left nearly
                // every row and candidate. 3,000 rows against 3,737 x 76 with an offset, k = 100: 4.2 ms with
                // every row tightened twice and scanned in the end, 2.9 so, 2.2 without lists at all (3.0 with the heaps).
                const bool stuck = refined > 0 ? 10 * (h[0] >> 32) > 9 * open && 4 * h[4] > 3 * listed
                                               : 4 * n_groups >= 5 * k && 4 * h[4] > 3ULL * (unsigned long long)cr * (unsigned long long)nS;
                if (!redo && ((h[0] >> 32) == 0 || refined == kTkRefines || stuck)) {
                    flagged += (int64_t)(h[0] & 0xffffffffULL);
                    fp64 += (int64_t)h[5];
                    break;
                }
                if (!redo) {
                    listed = h[4];
                    open = h[0] >> 32;
                }
            }
            row0 += cr;
            if (!rc && row0 < nQ) rc = reset();   // this chunk's named rows stay; its counters start over
        }
    } else {   // no tensor-core pass for this shape: every row takes the exact scan
        std::vector<int> every((size_t)nQ);
        for (int64_t i = 0; i < nQ; ++i) every[(size_t)i] = (int)i;
        e = cudaMemcpyAsync(frows, every.data(), (size_t)nQ * sizeof(int), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = cuda_fail(e, "top-k rows");
        flagged = nQ;
        if (timing) cudaEventRecord(ev[1], st);
    }
    // exact scan of the named rows
    if (!rc && flagged > 0) {
        const int64_t per_row = (int64_t)nS * 8 + (int64_t)kTkFallbackCap * 12;
        const int64_t batch = std::max<int64_t>(1, std::min<int64_t>(flagged, (256LL << 20) / per_row));
        void *fb = nullptr;
        rc = dev_alloc(&fb, al256(batch * (size_t)nS * 8) + al256(batch * (size_t)kTkFallbackCap * 12), st);
        if (!rc) {
            TopkFb g;
            g.Q = Q->x32;
            g.S = S->x32;
            g.d = d;
            g.nS = (int)nS;
            g.k = k;
            g.scr_u = (float *)fb;
            g.scr_l = g.scr_u + batch * nS;
            g.scr_c = (uint32_t *)((char *)fb + al256(batch * (size_t)nS * 8));
            g.scr_d = (double *)(g.scr_c + batch * kTkFallbackCap);
            g.q_orig = Q->orig;
            g.s_orig = S->orig;
            g.s_ids = S->ids;
            g.out_ids = out_ids;
            g.out_d2 = out_d2;
            g.row_k = row_k;
            g.row_off = row_off;
            g.g32 = t.g32;
            g.abs32 = t.abs32;
            g.slack = t.slack;
            g.err = (int *)(misc + 2);
            g.n_fp64 = misc + 1;
            for (int64_t b0 = 0; b0 < flagged && !rc; b0 += batch) {
                g.rows = frows + b0;
                g.n_rows = (int)std::min<int64_t>(batch, flagged - b0);
                k_topk_fallback<<<g.n_rows, 256, 0, st>>>(g);
                count_launch();
                ++launches;
                e = cudaGetLastError();
                if (e != cudaSuccess) rc = cuda_fail(e, "k_topk_fallback launch");
            }
            dev_free(fb, st);
        }
    }
    if (timing) cudaEventRecord(ev[2], st);
    if (!rc && flagged > 0) rc = read_misc();   // otherwise the last listing pass read them
    if (!rc && h[2]) {
        set_error("top-k: more than %d store rows tie within rounding at the k-th distance of a query",
                  kTkFallbackCap);
        rc = DL_EUNSUPPORTED;
    }
    if (rc) return done(rc);
    if (stats) {
        dl_join_stats &s = *stats;
        s.pairs_evaluated = nQ * nS;
        s.pairs_out = 0;
        s.band_pairs = flagged;   // rows re-solved by the exact scan
        s.fp64_pairs = fp64 + (int64_t)h[1];
        s.precision = prec;
        s.tile_n = use_tc ? BN : 0;
        s.epilogue_warps = use_tc ? (wide ? 16 : 8) : 0;
        s.kernels_launched = launches;
        if (timing) {
            cudaEventElapsedTime(&s.ms_main, ev[0], ev[1]);
            cudaEventElapsedTime(&s.ms_recheck, ev[1], ev[2]);
            cudaEventElapsedTime(&s.ms_total, ev[0], ev[2]);
        }
    }
    if (tune_trial && flagged == 0) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev[0], ev[1]);
        tune_record(Q->dp, tune_kind, nQ, nS, code, ms, (double)nQ * (double)nS);
    }
    return done(DL_OK);
}

}  // namespace dl

using namespace dl;

extern "C" int dl_topk_join(const dl_store *Q, const dl_store *S, int32_t metric, int32_t k, const dl_join_opts *opts,
                            dl_result **out)
{
    dl::NvtxScope nvtx_scope("dl_topk_join");
    clear_error();
    if (!out) {
        set_error("dl_topk_join: out is NULL");
        return DL_EINVAL;
    }
    *out = nullptr;
    if (!Q || !S) {
        set_error("dl_topk_join: NULL store");
        return DL_EINVAL;
    }
    const bool hist = metric == DL_METRIC_L1 || metric == DL_METRIC_CHI2;
    if (metric == DL_METRIC_COSINE) {   // the most similar rows are the nearest normalized rows
        if (!Q->unit || !S->unit) {
            set_error("dl_topk_join: the cosine metric needs stores made by dl_store_normalize");
            return DL_EINVAL;
        }
    } else if (metric != DL_METRIC_L2 && !hist) {
        set_error("dl_topk_join: unsupported metric %d", metric);
        return DL_EINVAL;
    }
    if (k < 1 || k > 1024) {
        set_error("dl_topk_join: k=%d out of range [1, 1024]", k);
        return DL_EINVAL;
    }
    if (Q->d != S->d) {
        set_error("dl_topk_join: dimension mismatch %d vs %d", Q->d, S->d);
        return DL_EINVAL;
    }
    int dev = -1;
    DL_CUDA_TRY(cudaGetDevice(&dev));
    if (dev != Q->device || dev != S->device) {
        set_error("dl_topk_join: stores live on another device");
        return DL_EINVAL;
    }
    dl_join_opts o;
    if (opts)
        o = *opts;
    else
        dl_join_opts_default(&o);
    if (o.precision != DL_PREC_AUTO && o.precision != DL_PREC_BF16 && o.precision != DL_PREC_FP16 &&
        o.precision != DL_PREC_FP32) {
        set_error("dl_topk_join: precision %d not available for top-k", o.precision);
        return DL_EUNSUPPORTED;
    }
    cudaStream_t st = (cudaStream_t)o.cuda_stream;
    if (hist && (o.precision == DL_PREC_BF16 || o.precision == DL_PREC_FP16)) {
        set_error("dl_topk_join: the L1 and chi-square distances run in DL_PREC_FP32 (not on tensor cores)");
        return DL_EUNSUPPORTED;
    }
    int rc = DL_OK;
    if (metric == DL_METRIC_CHI2) {
        bool ok = false;
        rc = store_nonneg(const_cast<dl_store *>(Q), st, &ok);
        if (!rc && ok) rc = store_nonneg(const_cast<dl_store *>(S), st, &ok);
        if (rc) return rc;
        if (!ok) {
            set_error("dl_topk_join: the chi-square distance needs non-negative features");
            return DL_EINVAL;
        }
    }
    const int64_t nQ = Q->n;
    void *resb = nullptr;
    rc = dev_alloc(&resb, std::max<size_t>(16, (size_t)nQ * k * 16), st);
    if (rc) return rc;
    int64_t *out_ids = (int64_t *)resb;
    double *out_d2 = (double *)(out_ids + (size_t)nQ * k);
    dl_join_stats stats{};
    if (hist)
        rc = hist_topk(Q, S, metric == DL_METRIC_L1 ? 1 : 2, k, out_ids, out_d2, st, &stats);
    else
        rc = topk_core(Q, S, k, nullptr, nullptr, out_ids, out_d2, o, st, &stats);
    if (rc) {
        dev_free(resb, st);
        return rc;
    }
    stats.pairs_out = nQ * std::min<int64_t>(k, S->n);
    dl_result *res = new dl_result();
    res->kind = 1;
    res->device = dev;
    res->stream = st;
    res->k = k;
    res->nq = nQ;
    res->d_ids = out_ids;
    res->d_d2 = out_d2;
    res->stats = stats;
    *out = res;
    return DL_OK;
}

DL_CHECK_READER(topk)
