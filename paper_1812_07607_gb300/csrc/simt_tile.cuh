// simt_tile.cuh -- the CUDA-core pair tile shared by the FP32 SIMT join (join_simt.cu) and the
// histogram top-k (hist_topk.cu): the FP32 distances of a 128-row x 128-column tile of pairs,
// 8 x 8 pairs in each of 256 threads.
//
// What bounds it: the FP32 pipe (an addition and an FMA a term for squared L2, two additions for
// L1, five operations and half a reciprocal for chi-square), so the loop has to keep it fed: two
// CTAs of 8 warps per SM (128 registers a thread); the next 16-wide K slice is loaded to registers
// while the current one is computed from shared memory, and stored to the other of two buffers
// after it, one barrier a slice. A thread stages 32 contiguous bytes of one row of each operand (a
// whole sector) and writes them transposed, [k][row], so a warp's lanes write neighbouring words.
// Additions and FMAs run as packed pairs (two columns an instruction), half the issue slots. The
// K loop is not unrolled: its body is 200 to 500 instructions already, and unrolled eight times it
// left the instruction cache (L1: 29 ms). Measured, 65,536 x 128 self-join (2.1 G pairs): 18.2 ms
// under L1, 46.7 under chi-square, 16.9 under squared L2; with single instead of packed operations
// 20.8, 55.8 and 20.9; with, besides, one 32-wide buffer and a reciprocal a term 22.0, 70.6, 22.1.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace dl {

constexpr int kSimtTile = 128;
constexpr int kSimtK = 16;

struct SimtSmem {
    float a[2][kSimtK][kSimtTile + 4];
    float b[2][kSimtK][kSimtTile + 4];
};

// Chi-square terms clamp their denominators from below (an empty bin in both rows is 0 / 0): a
// term with a + b below it is itself at most a + b, so the clamp costs at most 2^-50 a term.
constexpr float kChi2Floor = 8.8817841970012523e-16f;   // 2^-50

// Chi-square distances scale with the features, the clamp does not: the features enter the tile times a
// power of two that brings the two stores' largest just below 2^40 (the domain's end, so nothing grows
// past it), and distances are compared at that scale. The clamp then lies 2^90 below the largest feature. Without
// it rows that sum to 1e-12, or rows of any sum that differ by 1e-6 of it, lay within the clamp's error
// of each other. The rows' features are scaled when they are staged, the columns' within the FMAs that
// form a difference and a sum: chi-square top-10 of 1,000 rows against 65,536 x 128 1,752 us without any
// scaling, 1,747 so, 1,764 with both scaled when staged.
inline float chi2_scale(float x_max)
{
    int e = 0;
    std::frexp(x_max, &e);   // x_max < 2^e
    const int s = x_max > 0.f ? std::min(std::max(40 - e, 0), 126) : 0;
    return std::ldexp(1.f, s);
}

// FP32 error of a chi-square distance of scaled features: |D32 - D| <= chi2_g32(d) D + chi2_abs32(d).
//   Relative: a pair of terms, (t1^2 u2 + t2^2 u1) / (u1 u2), has at most 11 roundings of 2^-24 on
//   any path (rcp.approx counted as two) and d / 2 accumulations follow: below (d + 16) 2^-23.
//   Absolute, per pair of terms: the clamp (2 x 2^-50) and what underflows below the normal range
//   (2^-150 / (u1 u2) <= 2^-50 for each product, u >= 2^-50): below 2^-47, so d 2^-48 in all.
inline double chi2_g32(int d) { return (d + 16) * 1.1920928955078125e-07; }
inline double chi2_abs32(int d) { return d * 3.552713678800501e-15; }

// Packed pairs of floats (add / mul / fma.f32x2): each half rounds as the scalar operation does.
__device__ __forceinline__ uint64_t pack2(float x, float y)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Adds the terms k and k + 1 of metric M for a pair (a, b) of feature values to acc:
//   M = 0: squared L2; M = 1: L1; M = 2: chi-square on non-negative features, times `up`. One reciprocal
//   serves two chi-square terms: the MUFU unit (16 lanes an SM) would otherwise bound the loop. Packed:
//   the two features' scaling, sum and difference take three instructions.
template <int M>
__device__ __forceinline__ void dist_terms(float a0, float a1, float b0, float b1, float up, float &acc)
{
    if constexpr (M == 2) {
        const uint64_t b = pack2(b0, b1), as = mul2(pack2(a0, a1), pack2(up, up));
        const uint64_t t = fma2(b, pack2(-up, -up), as);
        float u0, u1, s0, s1, r;
        unpack2(fma2(b, pack2(up, up), as), u0, u1);
        u0 = fmaxf(u0, kChi2Floor);
        u1 = fmaxf(u1, kChi2Floor);
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(u0 * u1));
        unpack2(mul2(t, t), s0, s1);
        acc = fmaf(fmaf(s1, u0, s0 * u1), r, acc);
    } else {
        const float t0 = a0 - b0, t1 = a1 - b1;
        if constexpr (M == 0) {
            acc = fmaf(t0, t0, acc);
            acc = fmaf(t1, t1, acc);
        } else {
            acc += fabsf(t0);
            acc += fabsf(t1);
        }
    }
}

// dist_terms for two neighbouring columns at once: the row's features twice in a0 / a1, the
// columns' in b0 / b1, the same operations and roundings (b (-1) + a rounds once, as a - b).
// Chi-square: the rows' features come scaled, the columns' are scaled here, within those two FMAs.
template <int M>
__device__ __forceinline__ void dist_terms2(uint64_t a0, uint64_t a1, uint64_t b0, uint64_t b1, float up, float &c0, float &c1)
{
    const uint64_t m1 = M == 2 ? pack2(-up, -up) : pack2(-1.f, -1.f);
    const uint64_t t0 = fma2(b0, m1, a0), t1 = fma2(b1, m1, a1);
    if constexpr (M == 0) {
        uint64_t c = pack2(c0, c1);
        c = fma2(t0, t0, c);
        c = fma2(t1, t1, c);
        unpack2(c, c0, c1);
    } else if constexpr (M == 1) {
        float x, y;
        unpack2(t0, x, y);
        c0 += fabsf(x);
        c1 += fabsf(y);
        unpack2(t1, x, y);
        c0 += fabsf(x);
        c1 += fabsf(y);
    } else {
        float x, y, z, w, p, q, rp, rq;
        unpack2(fma2(b0, pack2(up, up), a0), x, y);
        unpack2(fma2(b1, pack2(up, up), a1), z, w);
        const uint64_t u0 = pack2(fmaxf(x, kChi2Floor), fmaxf(y, kChi2Floor)), u1 = pack2(fmaxf(z, kChi2Floor), fmaxf(w, kChi2Floor));
        unpack2(mul2(u0, u1), p, q);
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rp) : "f"(p));
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rq) : "f"(q));
        const uint64_t n = fma2(mul2(t1, t1), u0, mul2(mul2(t0, t0), u1));
        unpack2(fma2(n, pack2(rp, rq), pack2(c0, c1)), c0, c1);
    }
}

// Eight consecutive features of a row from column k on (0 past the row's end and for rows past
// the operand). VEC: d is a multiple of 4, so rows start on 16 bytes and a quad is in or out.
template <bool VEC>
__device__ __forceinline__ void load_slice8(const float *__restrict__ x, bool row_ok, int k, int d, float (&v)[8])
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int kk = k + 4 * h;
        if constexpr (VEC) {
            const float4 q = row_ok && kk < d ? __ldg(reinterpret_cast<const float4 *>(x + kk)) : make_float4(0.f, 0.f, 0.f, 0.f);
            v[4 * h] = q.x;
            v[4 * h + 1] = q.y;
            v[4 * h + 2] = q.z;
            v[4 * h + 3] = q.w;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[4 * h + e] = row_ok && kk + e < d ? __ldg(x + kk + e) : 0.f;
        }
    }
}

// acc[i][j] = distance of rows r0 + simt_sub(ty, i) of R and c0 + simt_sub(tx, j) of S, with
// tx = tid & 15 and ty = tid >> 4; chi-square: times `up`. Every thread of the CTA (256) calls it.
__device__ __forceinline__ int simt_sub(int t, int i) { return (i < 4) ? t * 4 + i : 64 + t * 4 + i - 4; }

template <int M, bool VEC>
__device__ __forceinline__ void simt_tile(const float *__restrict__ R, const float *__restrict__ S, int nR, int nS, int d,
                                          int r0, int c0, float up, SimtSmem &sm, float (&acc)[8][8])
{
    auto staged = [&](float x) { return M == 2 ? x * up : x; };
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int row = tid & 127, kh = (tid >> 7) * 8;   // this thread stages features kh .. kh + 7 of a slice
    const bool a_ok = r0 + row < nR, b_ok = c0 + row < nS;
    const float *ra = R + (size_t)(a_ok ? r0 + row : 0) * d;
    const float *rb = S + (size_t)(b_ok ? c0 + row : 0) * d;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
    float va[8], vb[8];
    load_slice8<VEC>(ra, a_ok, kh, d, va);
    load_slice8<VEC>(rb, b_ok, kh, d, vb);
    int buf = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        sm.a[0][kh + e][row] = staged(va[e]);
        sm.b[0][kh + e][row] = vb[e];
    }
    __syncthreads();
    for (int k0 = 0; k0 < d; k0 += kSimtK) {
        const bool more = k0 + kSimtK < d;
        if (more) {
            load_slice8<VEC>(ra, a_ok, k0 + kSimtK + kh, d, va);
            load_slice8<VEC>(rb, b_ok, k0 + kSimtK + kh, d, vb);
        }
#pragma unroll 1
        for (int k = 0; k < kSimtK; k += 2) {
            float a[2][8], b[2][8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                *reinterpret_cast<float4 *>(&a[h][0]) = *reinterpret_cast<const float4 *>(&sm.a[buf][k + h][ty * 4]);
                *reinterpret_cast<float4 *>(&a[h][4]) = *reinterpret_cast<const float4 *>(&sm.a[buf][k + h][64 + ty * 4]);
                *reinterpret_cast<float4 *>(&b[h][0]) = *reinterpret_cast<const float4 *>(&sm.b[buf][k + h][tx * 4]);
                *reinterpret_cast<float4 *>(&b[h][4]) = *reinterpret_cast<const float4 *>(&sm.b[buf][k + h][64 + tx * 4]);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; j += 2)
                    dist_terms2<M>(pack2(a[0][i], a[0][i]), pack2(a[1][i], a[1][i]), pack2(b[0][j], b[0][j + 1]), pack2(b[1][j], b[1][j + 1]),
                                   up, acc[i][j], acc[i][j + 1]);
        }
        if (more) {
            buf ^= 1;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                sm.a[buf][kh + e][row] = staged(va[e]);
                sm.b[buf][kh + e][row] = vb[e];
            }
            __syncthreads();
        }
    }
}

}  // namespace dl
