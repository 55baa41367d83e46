// join_simt.cu -- K8: the FP32 SIMT join (plain baseline and exact-path front end).
//
// The nested-loop join of Sec. 5 evaluated directly as D32 = sum_k fl(q_k - x_k)^2
// with an FMA chain per pair, register-tiled 8x8 pairs per thread over a
// 128 x 128 pair tile staged through shared memory in 16-wide K slices (simt_tile.cuh).
// The same tiling evaluates the histogram distances (L1, chi-square), which are not
// contractions and so stay on the CUDA cores; their thresholds carry their own
// FP32 bounds and their band pairs go to k_hist_recheck.
//
//   plain (DL_PREC_FP32_PLAIN): accept iff D32 <= fl32(eps)^2 -- the usual FP32
//     GPU join, the throughput baseline; not exact near the threshold.
//   exact (DL_PREC_FP32): accept iff D32 <= t_acc, reject iff D32 > t_rej, where
//     the thresholds carry the FP32 error bound |D32 - D| <= (d+8) 2^-24 D plus
//     the canonical-FP64 slack; undecided pairs go to the recheck (K6).
#include "kernels.h"
#include "simt_tile.cuh"

namespace dl {

__device__ __forceinline__ long long tri_start(int m, int T) { return (long long)m * T - (long long)m * (m - 1) / 2; }

template <int M, bool VEC>
__global__ void __launch_bounds__(256, 2) k8_simt_join(const SimtParams p)
{
    __shared__ __align__(16) SimtSmem sm;
    int tm, tn;
    if (p.upper) {
        const int T = p.tiles_m;
        const long long l = blockIdx.x;
        const double tt = 2.0 * T + 1.0;
        int m = (int)floor((tt - sqrt(tt * tt - 8.0 * (double)l)) * 0.5);
        if (m < 0) m = 0;
        if (m > T - 1) m = T - 1;
        while (m > 0 && tri_start(m, T) > l) --m;
        while (m + 1 < T && tri_start(m + 1, T) <= l) ++m;
        tm = m;
        tn = m + (int)(l - tri_start(m, T));
    } else {
        tm = blockIdx.y;
        tn = blockIdx.x;
    }
    const int r0 = tm * kSimtTile, c0 = tn * kSimtTile;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;

    float acc[8][8];
    simt_tile<M, VEC>(p.R, p.S, p.nR, p.nS, p.d, r0, c0, p.up, sm, acc);

    // classify: the common case is "no candidate anywhere in this thread's 64 pairs"
    bool any = false;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) any |= (p.exact ? (acc[i][j] <= p.t_rej) : (acc[i][j] <= p.t_acc));
    if (!__any_sync(0xffffffffu, any)) return;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = r0 + simt_sub(ty, i);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = c0 + simt_sub(tx, j);
            const bool valid = (r < p.nR) && (c < p.nS) && (!p.upper || c > r);
            const float v = acc[i][j];
            const bool a = valid && (v <= p.t_acc);
            const bool b = valid && p.exact && !a && (v <= p.t_rej);
            warp_emit(p.out, a, b, r, c);
        }
    }
}



template <int M>
static void launch_k8(const SimtParams &p, dim3 grid, cudaStream_t st)
{
    if ((p.d & 3) == 0)
        k8_simt_join<M, true><<<grid, 256, 0, st>>>(p);
    else
        k8_simt_join<M, false><<<grid, 256, 0, st>>>(p);
}

int launch_simt_join(SimtParams p, cudaStream_t st)
{
    const int tm = (p.nR + kSimtTile - 1) / kSimtTile;
    const int tn = (p.nS + kSimtTile - 1) / kSimtTile;
    p.tiles_m = tm;
    if (tm == 0 || tn == 0) return DL_OK;
    dim3 grid;
    if (p.upper) {
        const long long blocks = (long long)tm * (tm + 1) / 2;
        if (blocks > 2147483647LL) {
            set_error("self-join too large for the SIMT path");
            return DL_EUNSUPPORTED;
        }
        grid = dim3((unsigned)blocks);
    } else {
        if (tm > 65535) {
            set_error("R too large for the SIMT path grid");
            return DL_EUNSUPPORTED;
        }
        grid = dim3((unsigned)tn, (unsigned)tm);
    }
    if (p.metric == 1)
        launch_k8<1>(p, grid, st);
    else if (p.metric == 2)
        launch_k8<2>(p, grid, st);
    else
        launch_k8<0>(p, grid, st);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "k8_simt_join launch");
    return DL_OK;
}

}  // namespace dl
