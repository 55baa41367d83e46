// join_tc.cu -- K2 + K3 + K5: the tensor-core epsilon-join kernel.
//
// The nested-loop join of Sec. 5 evaluates every pair (q, x). With
//   D(q, x) = ||q||^2 + ||x||^2 - 2 q.x
// the only pair-wise term is the dot product, a dense contraction. This kernel
// computes A = Q~ X~^T on the tcgen05 tensor cores (FP16, BF16 or FP8 e4m3 in, FP32
// accumulate in TMEM) and classifies every pair in a fused epilogue against per-row
// thresholds that carry a proven error bound, so that each pair is either a proven
// match, a proven non-match, or an undecided "band" pair that the recheck settles
// exactly. With h = q.x - ||x||^2/2 the epilogue works on h~ = fl(A s - beta)
// (s = 1 for BF16, the power of two s_R s_S of the two stores for FP16, and for FP8 the power of two
// s_q s_chunk of the row and the 32-column chunk).
//
// Per CTA (persistent, one per SM, 320 threads -- 576 with the wide epilogue -- warp-specialised):
//   warp 0      TMA producer: the 128-row R tile (all K chunks of 128 bytes: 64 16-bit
//               or 128 FP8 columns) is loaded once per unit into one of one or two A
//               slots; S tiles stream through a ring of stages, one K chunk of BN
//               rows per stage (128-byte swizzle). Each tile's column data (beta, chunk stats,
//               FP8 chunk scales) goes by bulk copies into a ring of eight tiles.
//   warp 1      MMA issuer: 4 x tcgen05.mma (K = 32 bytes each) per stage into one of
//               the 512 / BN TMEM accumulators (128 lanes x BN FP32 columns each: two
//               of 256 or four of 128 columns), then tcgen05.commit to free the stage
//               and to publish the accumulator.
//   the rest    epilogue: two warps per TMEM lane quadrant, each owning half of the
//               tile's columns (the wide epilogue: two such groups of eight warps, taking
//               alternate tiles). Per 32-column chunk: tcgen05.ld, then a three-input max
//               tree over the raw accumulators and one compare
//               of fl_ru(max A * s - beta_min of the chunk) against the row's reject
//               threshold (about half an issue slot per pair; store rows are in norm
//               order so a chunk's betas are nearly equal). Rows that this bound cannot reject are
//               put aside in shared memory (a few per tile) and classified pair by pair after the
//               accumulator has been released, or, when there are many, on the spot (slow_many):
//               proven matches and band pairs go to a per-warp shared-memory buffer as (r, c)
//               candidates, flushed to the global candidate list with one atomic per
//               flush. k_finalize turns the candidates into id pairs.
//
// What bounds it at small d: a tile's MMAs (128 clocks each, 8 at d = 128) against everything that
// keeps them waiting or takes shared-memory cycles from their operand reads -- the S tiles' own
// arrival, polling warps, the issuing thread's instructions between two MMAs (its queue is short).
// 262,144-row self-join, d = 128 (34.4 G pairs, 1.05 M tiles): 6.25 ms with per-warp cp.async column
// staging, hits classified before the release and 64-bit barrier arithmetic in every wait; 6.24 with
// bulk copies, rows put aside and alternating groups; 5.8 to 5.96 with the issuing loop reduced to
// additions; 5.44 to 5.67 with waits that suspend (1,560 clocks a tile; TMA and MMAs alone with an
// epilogue that only reduces take 1,270). A second issuing thread for alternate tiles gained nothing
// (5.97) and lost with 16 epilogue warps (6.4). At d = 512 and above the join runs at the power cap.
// A unit is (R tile m, S tiles [nb, ne)); units are handed out round-robin, in the
// S-range-major order their builders produce.
#include <algorithm>
#include <atomic>

#include <cuda.h>

#include "kernels.h"
#include "checked.cuh"
#include "ptx.cuh"

namespace dl {

__device__ __forceinline__ bool mbar_wait_plain(uint32_t bar, uint32_t parity)
{
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > kWaitBudgetClocks) return false;
    return true;
}

// The S tile after n in a unit of R tile m ending at `end`: n + 1, or with a tile mask the
// next tile whose bit is set (end when there is none). Every role steps through a unit with
// it, so all of them see the same tile sequence.
template <bool MASK>
__device__ __forceinline__ int tile_after(const TcParams &p, int m, int n, int end)
{
    ++n;
    if constexpr (MASK) {
        const uint32_t *row = p.tile_mask + (size_t)m * p.mask_ntw;
        while (n < end) {
            const uint32_t w = __ldg(row + (n >> 5)) >> (n & 31);
            if (w) return min(n + __ffs((int)w) - 1, end);
            n = (n | 31) + 1;
        }
        return end;
    }
    return n;
}

// Unit u: from the list, or one of the grid units. (Out of line: the tile loops are read through it
// only between units, and its divisions would sit in their instruction stream.)
__device__ __noinline__ int4 unit_of(const int4 *units, int m0, int mt, int len, int nt, int u)
{
    if (units) return units[u];
    const int nb = u / mt * len;
    return make_int4(m0 + u % mt, nb, min(nb + len, nt), 0);
}
__device__ __forceinline__ int4 unit_at(const TcParams &p, int u)
{
    return unit_of(p.units, p.m0, p.mt, p.unit_len, p.unit_nt, u);
}

// Walks this CTA's (unit, S tile) sequence.
template <bool MASK>
struct TileIter {
    int u, n;
    int4 un;
    bool valid;
    int stride;
    int nu;   // unit count
    __device__ __forceinline__ void start(const TcParams &p, int first, int step, int n_units)
    {
        u = first;
        stride = step;
        nu = n_units;
        valid = u < nu;
        if (valid) {
            un = unit_at(p, u);
            n = un.y;
        }
    }
    __device__ __forceinline__ void next(const TcParams &p)
    {
        if (!valid) return;
        n = tile_after<MASK>(p, un.x, n, un.z);
        if (n == un.z) {
            u += stride;
            valid = u < nu;
            if (valid) {
                un = unit_at(p, u);
                n = un.y;
            }
        }
    }
};

// Epilogue warps: 8, each owning half of every tile's columns, or -- the wide epilogue on 256-column
// tiles -- 16 in two groups of 8 that take alternate tiles, so that a warp has two tiles' time for one.
__host__ __device__ constexpr int tc_epi_warps(bool wide) { return wide ? 16 : 8; }
__host__ __device__ constexpr int tc_threads(bool wide) { return 64 + 32 * tc_epi_warps(wide); }
__host__ __device__ constexpr int tc_stage_cap(bool wide) { return wide ? 64 : 128; }   // candidates a warp buffers
constexpr int kTileWarps = 8;    // epilogue warps that share a tile
constexpr int kColRing = 8;      // tiles whose column data (beta, chunk stats, FP8 scales) is kept
constexpr int kDefer = 4;        // rows of hit chunks a warp puts aside until it has released the accumulator
constexpr int kDeferPitch = 36;  // floats of one (32 used; 16-byte aligned, shifted by 4 banks)
// Column data of a tile: BN betas, BN / 32 chunk stats, BN / 32 FP8 chunk scales.
__host__ __device__ constexpr int tc_col_bytes(int BN, bool fp8) { return BN * 4 + BN / 32 * 16 + (fp8 ? BN / 32 * 4 : 0); }

// Copy a warp's buffered candidates to the global list (one atomic per flush).
__device__ __forceinline__ void flush_stage(const TcParams &p, uint2 *stg, uint32_t &scnt)
{
    const unsigned lane = threadIdx.x & 31;
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0 && scnt) base = atomicAdd(p.cand_cnt, (unsigned long long)scnt);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (uint32_t i = lane; i < scnt; i += 32) {
        const unsigned long long idx = base + i;
        if (idx < p.cand_cap) p.cand[idx] = stg[i];
    }
    __syncwarp();
    scnt = 0;
}

// One 32-column chunk with many rows that its bound could not reject, for pairs (r, c0 + j) with
// h = fl(A s - beta_j) (s an exact power of two, so one rounding). A pair with
// h >= tau_rej of its row -- a proven match
// (h >= tau_acc) or a band pair -- becomes a candidate. Warp-collective; `hit` marks the
// lanes (rows) whose chunk bound failed, the others have no candidate in this chunk. Every lane
// classifies its own row's 32 columns into a bit mask, a warp prefix sum of the mask counts places
// each lane's candidates.
template <int CAP>
__device__ __forceinline__ uint32_t slow_many(const TcParams &p, const uint32_t (&v)[32], const float *bt, float sc,
                                              float tau_acc, float tau_rej, bool hit, int r, int c0, uint2 *stg,
                                              uint32_t scnt)
{
    const unsigned lane = threadIdx.x & 31;
    uint32_t cm = 0, am = 0;
    if (hit) {
        const float4 *bt4 = reinterpret_cast<const float4 *>(bt);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 b4 = bt4[q];
            const float bq[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int j = 4 * q + i;
                const float h = __fmaf_rn(__uint_as_float(v[j]), sc, -bq[i]);
                cm |= (h >= tau_rej ? 1u : 0u) << j;
                am |= (h >= tau_acc ? 1u : 0u) << j;
            }
        }
        const int rem = p.nS - c0;   // columns past the store
        if (rem < 32) cm &= rem <= 0 ? 0u : ((1u << rem) - 1u);
        if (p.upper) {   // upper mode: only pairs with c > r
            const int k = r - c0;
            if (k >= 31)
                cm = 0u;
            else if (k >= 0)
                cm &= ~((2u << k) - 1u);
        }
    }
    const uint32_t nl = __popc(cm);
    uint32_t incl = nl;
#pragma unroll
    for (int sft = 1; sft < 32; sft <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, sft);
        if ((int)lane >= sft) incl += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (total == 0) return scnt;
    uint2 *dst;
    unsigned long long lim;
    if (total <= (uint32_t)CAP) {
        if (scnt + total > (uint32_t)CAP) flush_stage(p, stg, scnt);
        dst = stg + scnt;
        lim = ~0ULL;
        scnt += total;
    } else {   // more than a buffer: reserve the space in the global list directly
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(p.cand_cnt, (unsigned long long)total);
        base = __shfl_sync(0xffffffffu, base, 0);
        dst = p.cand + base;
        lim = base < p.cand_cap ? p.cand_cap - base : 0ULL;
    }
    unsigned long long k = incl - nl;
    while (cm) {
        const int j = __ffs(cm) - 1;
        cm &= cm - 1u;
        // staged (lim = ~0) entries must stay inside the warp's buffer
        if (k < lim && DL_CHECK(lim != ~0ULL || k < (unsigned long long)CAP, 1, k))
            dst[k] = make_uint2((uint32_t)r, (uint32_t)(c0 + j) | (((am >> j) & 1u) ? 0u : kBandFlag));
        ++k;
    }
    return scnt;
}

// Maximum of v with three-input max.f32 (17 instructions, depth 4).
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ float max_tree32(const uint32_t (&v)[32])
{
    float m[11];
#pragma unroll
    for (int i = 0; i < 10; ++i)
        m[i] = fmax3(__uint_as_float(v[3 * i]), __uint_as_float(v[3 * i + 1]), __uint_as_float(v[3 * i + 2]));
    m[10] = fmaxf(__uint_as_float(v[30]), __uint_as_float(v[31]));
    const float a = fmax3(m[0], m[1], m[2]), b = fmax3(m[3], m[4], m[5]), c = fmax3(m[6], m[7], m[8]);
    const float e = fmaxf(m[9], m[10]);
    return fmaxf(fmax3(a, b, c), e);
}

// CG2: a CTA pair (cluster of two) computes 256-row tiles with tcgen05 cta_group::2. Each
// CTA loads its own 128 rows of A and its own half (BN/2 rows) of every S tile into its own
// shared memory, signalling its own barriers; the peer CTA's otherwise idle MMA warp forwards
// each of its completions to the leader (rank 0), whose single thread issues M = 256 MMAs that
// read both CTAs' operands and write each CTA's 128 rows into that CTA's TMEM; commits are
// multicast to both CTAs. Each CTA's epilogue handles its own rows; the peer releases an
// accumulator with a remote arrive on the leader's barrier. Half the B bytes per stage means
// twice the stages in the same shared memory beside a resident R tile.
template <int BN, int MODE, bool FP8, bool CG2, bool WIDE, bool MASK, bool STREAM>
__global__ void __launch_bounds__(tc_threads(WIDE), 1)
    tc_join_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const TcParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int kc = p.kc, stages = p.stages, a_slots = p.a_slots;
    constexpr uint32_t kStageBytes = (CG2 ? BN / 2 : BN) * 128;   // this CTA's rows of an S tile x 128 B
    // STREAM: no resident R tile; each stage also carries the R tile's matching 128-byte K chunk
    // (128 rows, 16 KB), so a large d keeps four stages instead of two beside a resident tile
    constexpr bool MAXIMA = MODE == kModeMaxima;
    static_assert(!STREAM || (!CG2 && !MAXIMA && !MASK), "streamed R chunks serve the one-SM epsilon-join");
    constexpr uint32_t kStageStride = STREAM ? kStageBytes + 16384 : kStageBytes;
    constexpr int kChunkCols = FP8 ? 128 : 64;   // columns per 128-byte K chunk
    constexpr int kAcc = 512 / BN;              // TMEM accumulators: 2 of 256 or 4 of 128 columns
    constexpr uint32_t kTmemCols = 512;
    static_assert(!WIDE || BN == 256, "the wide epilogue serves 256-column tiles");
    constexpr int kEpi = tc_epi_warps(WIDE);   // epilogue warps
    constexpr int HC = BN / 2;               // columns of a tile each epilogue warp owns
    constexpr int kSubW = HC / 32;           // 32-column chunks per warp per tile
    constexpr int kCap = tc_stage_cap(WIDE);
    constexpr uint32_t kColBytes = tc_col_bytes(BN, FP8);
    const uint32_t a_bytes = (uint32_t)kc * 16384;
    uint8_t *sA = smem;                                    // a_slots x kc x [128 rows x 128 B]
    uint8_t *sB = smem + (STREAM ? 0 : a_slots * a_bytes);   // stages x [BN rows x 128 B (+ R chunk)]
    uint8_t *s_col = sB + stages * kStageStride;                               // kColRing x a tile's column data
    float *s_def = reinterpret_cast<float *>(s_col + kColRing * kColBytes);    // kEpi x kDefer rows put aside
    uint2 *s_stage = reinterpret_cast<uint2 *>(s_def + kEpi * kDefer * kDeferPitch);   // kEpi x kCap candidates
    uint64_t *bars = reinterpret_cast<uint64_t *>(s_stage + kEpi * kCap);
    // barriers, by shared-memory address, 8 bytes each
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t full = bar0, empty = bar0 + 8 * 8;                  // [8] each: S stages
    const uint32_t a_full = bar0 + 16 * 8, a_empty = bar0 + 18 * 8;    // [2] each: R tile slots
    const uint32_t acc_full = bar0 + 20 * 8, acc_empty = bar0 + 24 * 8;   // [kAcc <= 4] each: accumulators
    const uint32_t done = bar0 + 28 * 8;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 29);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 30);
    const uint32_t pfull = bar0 + 32 * 8;      // CG2 leader: [8] the peer's half of the stage landed
    const uint32_t pa_full = bar0 + 40 * 8;    // CG2 leader: [2] the peer's rows of the R tile landed
    const uint32_t col_full = bar0 + 42 * 8;   // [kColRing] a tile's column data landed
    const uint32_t col_empty = col_full + kColRing * 8;   // [kColRing] its epilogue warps are done with it
    const uint32_t sA32 = smem_u32(sA), sB32 = smem_u32(sB);
    const bool expired = p.wait_budget < kExpireAtOnce;   // a test's budget: every role gives up at once
    const int tile_step = MAXIMA ? p.tile_stride : 1;   // S tile n of a unit is the store's tile n * tile_step
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t crank = CG2 ? cluster_ctarank() : 0u;   // this CTA's rank in its pair
    const bool leader = crank == 0u;
    const int ufirst = CG2 ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;   // units are per CTA pair with CG2
    const int ustride = CG2 ? (int)(gridDim.x >> 1) : (int)gridDim.x;
    const int n_units = MASK ? *p.n_units_dev : p.n_units;   // MASK: units built on the device
    constexpr int kRowTiles = CG2 ? 2 : 1;    // 128-row tiles per unit row tile
    // Raise the abort flag of this CTA (and of the peer, so that it stops waiting too).
    auto raise_abort = [&]() {
        *abort_flag = 1;
        if constexpr (CG2) st_shared_remote_u32(mapa_shared(smem_u32(const_cast<int *>(abort_flag)), crank ^ 1u), 1u);
        atomicExch(p.err, 1);
    };

    if (threadIdx.x < 64) {   // one barrier a thread (words 29 .. 31 are the TMEM address and the abort flag)
        const int w = (int)threadIdx.x;
        uint32_t count = 1;
        if (w >= 24 && w < 28) count = CG2 ? 2 * kTileWarps : kTileWarps;       // acc_empty; CG2 (leader): both CTAs' warps
        if (w >= 42 + kColRing && w < 42 + 2 * kColRing) count = kTileWarps;    // col_empty
        if (w < 29 || w >= 32) mbar_init(bars + w, count);
        if (w == 30) *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc<CG2>(tmem_slot, kTmemCols);
        tmem_relinquish<CG2>();
    }
    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (CG2) cluster_sync_all();   // both CTAs' barriers initialised and TMEM allocated
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t stage = 0, phase = 0;
            bool ok = !expired;
            uint32_t t = 0, col_tiles = 0;      // tiles so far, tiles whose column data was asked for
            uint32_t a_units = 0, s_loads = 0;  // R tiles and stages asked for
            int i = 0;   // unit count of this CTA
            for (int u = ufirst; u < n_units && ok; u += ustride, ++i) {
                const int4 un = unit_at(p, u);
                if constexpr (!STREAM) {
                    const int slot = i % a_slots;
                    const uint32_t use = (uint32_t)(i / a_slots);
                    if (!mbar_wait(a_empty + slot * 8, (use & 1) ^ 1, abort_flag, p.wait_budget)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(a_full + slot * 8, a_bytes);
                    for (int c = 0; c < kc; ++c)   // a K chunk is 128 bytes: 64 16-bit or 128 FP8 columns
                        tma_load_2d(sA32 + slot * a_bytes + c * 16384, &tmA, a_full + slot * 8, c * kChunkCols,
                                    (un.x * kRowTiles + (int)crank) * 128);
                    ++a_units;
                }
                for (int n = un.y; n < un.z && ok; n = tile_after<MASK>(p, un.x, n, un.z), ++t) {
                    // the tile's column data: whole 256-column tiles of beta [n_pad] and chunk stats
                    // [n_pad / 32], so every copy is in bounds and a multiple of 16 bytes
                    const uint32_t cs = t % kColRing, cbar = col_full + cs * 8;
                    if (!mbar_wait(col_empty + cs * 8, ((t / kColRing) & 1) ^ 1, abort_flag, p.wait_budget)) {
                        ok = false;
                        break;
                    }
                    const int c0 = n * tile_step * BN;
                    if (DL_CHECK(c0 + BN <= (p.nS + 255) / 256 * 256, 4, c0)) {
                        const uint32_t cd = smem_u32(s_col) + cs * kColBytes;
                        mbar_arrive_expect_tx(cbar, kColBytes);
                        bulk_load(cd, p.beta + c0, BN * 4, cbar);
                        bulk_load(cd + BN * 4, p.cstat + (c0 >> 5), BN / 32 * 16, cbar);
                        if constexpr (FP8) bulk_load(cd + BN * 4 + BN / 32 * 16, p.sc_s + (c0 >> 5), BN / 32 * 4, cbar);
                    } else {
                        mbar_arrive(cbar);
                    }
                    col_tiles = t + 1;
                    for (int c = 0; c < kc; ++c) {
                        if (!mbar_wait(empty + stage * 8, phase ^ 1, abort_flag, p.wait_budget)) {
                            ok = false;
                            break;
                        }
                        const uint32_t dst = sB32 + stage * kStageStride, bar = full + stage * 8;
                        mbar_arrive_expect_tx(bar, kStageStride);
                        tma_load_2d(dst, &tmB, bar, c * kChunkCols, c0 + (CG2 ? (int)crank * (BN / 2) : 0));
                        if constexpr (STREAM)   // the R tile's chunk c beside it
                            tma_load_2d(dst + kStageBytes, &tmA, bar, c * kChunkCols, un.x * 128);
                        ++s_loads;
                        if (++stage == (uint32_t)stages) {
                            stage = 0;
                            phase ^= 1;
                        }
                    }
                }
            }
            if (!ok) raise_abort();
            // Every copy this thread started lands before the CTA exits (after an abort nobody else
            // may have waited for them; otherwise they all have landed).
            // The last use of each barrier is among its ring's last loads.
            auto land = [&](uint32_t bars_at, uint32_t ring, uint32_t n) {
                for (uint32_t q = n > ring ? n - ring : 0u; q < n; ++q) mbar_wait_plain(bars_at + q % ring * 8, (q / ring) & 1);
            };
            land(full, (uint32_t)stages, s_loads);
            land(a_full, STREAM ? 1u : (uint32_t)a_slots, a_units);
            land(col_full, kColRing, col_tiles);
        }
    } else if (warp == 1 && CG2 && !leader) {
        // ------------------------------------------------------------ peer: completion forwarder
        // The leader's MMAs read this CTA's shared memory too: forward each completion of this
        // CTA's own R-tile and stage barriers, in the producer's order, to the leader.
        if (lane == 0) {
            const uint32_t r_pfull = mapa_shared(pfull, 0u), r_pa_full = mapa_shared(pa_full, 0u);
            uint32_t stage = 0, phase = 0;
            bool ok = !expired;
            int i = 0;
            for (int u = ufirst; u < n_units && ok; u += ustride, ++i) {
                const int4 un = unit_at(p, u);
                const int slot = i % a_slots;
                const uint32_t use = (uint32_t)(i / a_slots);
                if (!mbar_wait(a_full + slot * 8, use & 1, abort_flag, p.wait_budget)) {
                    ok = false;
                    break;
                }
                mbar_arrive_remote(r_pa_full + (uint32_t)slot * 8u);
                for (int n = un.y; n < un.z && ok; n = tile_after<MASK>(p, un.x, n, un.z)) {
                    for (int c = 0; c < kc; ++c) {
                        if (!mbar_wait(full + stage * 8, phase, abort_flag, p.wait_budget)) {
                            ok = false;
                            break;
                        }
                        mbar_arrive_remote(r_pfull + stage * 8u);
                        if (++stage == (uint32_t)stages) {
                            stage = 0;
                            phase ^= 1;
                        }
                    }
                }
            }
            if (!ok) raise_abort();
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t idesc = FP8 ? idesc_e4m3_f32(CG2 ? 256 : 128, BN)
                                       : idesc_f16_f32(CG2 ? 256 : 128, BN) | (p.fmt ? kIdescBF16 : 0u);
            // The tensor core takes MMAs from a short queue, so whatever this thread does between two of
            // them and the queue does not cover is time without an MMA: addresses and descriptors are
            // formed once and advanced by additions, and the waits' long form is out of line.
            uint32_t stage = 0, phase = 0, t = 0;
            bool ok = !expired, any_mma = false;
            const uint32_t a_lo0 = smem_desc_lo(sA32), b_lo0 = smem_desc_lo(sB32);
            uint32_t b_lo = b_lo0;    // of the current stage
            int i = 0;
            for (int u = ufirst; u < n_units && ok; u += ustride, ++i) {
                const int4 un = unit_at(p, u);
                const int slot = STREAM ? 0 : i % a_slots;
                uint32_t a_lo = a_lo0;
                if constexpr (!STREAM) {   // the unit's resident R tile
                    const uint32_t use = (uint32_t)(i / a_slots);
                    if (!mbar_wait(a_full + slot * 8, use & 1, abort_flag, p.wait_budget)) {
                        ok = false;
                        break;
                    }
                    if constexpr (CG2) {   // the peer's rows of the R tile
                        if (!mbar_wait<true>(pa_full + slot * 8, use & 1, abort_flag, p.wait_budget)) {
                            ok = false;
                            break;
                        }
                    }
                    tc_fence_after();
                    a_lo = a_lo0 + (uint32_t)slot * (a_bytes >> 4);
                }
                for (int n = un.y; n < un.z; n = tile_after<MASK>(p, un.x, n, un.z), ++t) {
                    const uint32_t b = t % kAcc;
                    if (!mbar_wait<CG2>(acc_empty + b * 8, ((t / kAcc) & 1) ^ 1, abort_flag, p.wait_budget)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + b * BN;
                    uint32_t ac_lo = a_lo;
                    int c = 0;
#pragma unroll 1
                    for (; c < kc; ++c) {
                        if (!mbar_wait(full + stage * 8, phase, abort_flag, p.wait_budget)) break;
                        if constexpr (CG2)   // the peer's half of this stage
                            if (!mbar_wait<true>(pfull + stage * 8, phase, abort_flag, p.wait_budget)) break;
                        tc_fence_after();
                        if constexpr (STREAM) ac_lo = b_lo + (kStageBytes >> 4);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {   // 4 x 32 bytes of K per 128-byte chunk
                            const uint64_t ad = smem_desc(ac_lo + 2 * k), bd = smem_desc(b_lo + 2 * k);
                            if constexpr (CG2 && FP8)
                                mma_f8_cg2(d_tmem, ad, bd, idesc, (c | k) != 0);
                            else if constexpr (CG2)
                                mma_f16_cg2(d_tmem, ad, bd, idesc, (c | k) != 0);
                            else if constexpr (FP8)
                                mma_f8(d_tmem, ad, bd, idesc, (c | k) != 0);
                            else
                                mma_f16(d_tmem, ad, bd, idesc, (c | k) != 0);
                        }
                        if constexpr (CG2)
                            mma_commit_cg2_mc(empty + stage * 8, 3);   // both CTAs may refill their halves
                        else
                            mma_commit(empty + stage * 8);
                        if constexpr (!STREAM) ac_lo += 16384 >> 4;
                        b_lo += kStageStride >> 4;
                        if (++stage == (uint32_t)stages) {
                            stage = 0;
                            phase ^= 1;
                            b_lo = b_lo0;
                        }
                    }
                    if (c < kc) {
                        ok = false;
                        any_mma |= c > 0;
                        break;
                    }
                    if constexpr (CG2)
                        mma_commit_cg2_mc(acc_full + b * 8, 3);   // both CTAs' rows are in their TMEM
                    else
                        mma_commit(acc_full + b * 8);
                }
                if (ok && !STREAM) {
                    if constexpr (CG2)
                        mma_commit_cg2_mc(a_empty + slot * 8, 3);
                    else
                        mma_commit(a_empty + slot * 8);
                }
            }
            if (!ok) raise_abort();
            // No MMA may still be running when TMEM is released. (A CTA that issued none -- one
            // that got no unit, or whose first wait ran out -- has nothing to wait for.)
            if (CG2 || any_mma || t > 0) {
                if constexpr (CG2)
                    mma_commit_cg2(done);
                else
                    mma_commit(done);
                mbar_wait_plain(done, 0);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int e = warp - 2;            // 0 .. kEpi-1
        const int quad = warp & 3;         // TMEM lanes this warp may access: 32*quad .. +31
        const int half = (e >> 2) & 1;     // which half of the tile's columns this warp owns
        const int group = e >> 3;          // WIDE: tiles t = group, group + 2, ... are this warp's
        constexpr int kGroups = kEpi / kTileWarps;
        const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
        const unsigned lt = lanemask_lt();
        float *my_def = s_def + e * (kDefer * kDeferPitch);
        uint2 *my_stg = s_stage + e * kCap;
        uint32_t scnt = 0;
        TileIter<MASK> cur;
        cur.start(p, ufirst, ustride, n_units);
        if (group) cur.next(p);
        uint32_t t = group;
        bool ok = !expired;
        int last_u = -1;
        float4 rp = make_float4(0.f, 0.f, 0.f, 0.f);
        float sq = 1.0f;          // FP8: this row's scale
        while (ok && cur.valid) {
            const int r = (cur.un.x * kRowTiles + (int)crank) * 128 + quad * 32 + lane;
            if (cur.u != last_u) {
                last_u = cur.u;
                // per-row parameters cover whole R tiles (256-row tiles for SM pairs)
                if (DL_CHECK(r < (p.nR + kRowTiles * 128 - 1) / (kRowTiles * 128) * (kRowTiles * 128), 3, r))
                    rp = p.rowpar[r];
                if constexpr (FP8) sq = (r < p.nR) ? p.sc_r[r] : 1.0f;
            }
            const uint32_t b = t % kAcc, cs_slot = t % kColRing;
            if (!mbar_wait(col_full + cs_slot * 8, (t / kColRing) & 1, abort_flag, p.wait_budget) ||
                !mbar_wait(acc_full + b * 8, (t / kAcc) & 1, abort_flag, p.wait_budget)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t tbase = tmem_base + lane_base + b * BN + half * HC;
            const uint8_t *cd = s_col + cs_slot * kColBytes;
            const float *beta = reinterpret_cast<const float *>(cd) + half * HC;
            const float4 *cst = reinterpret_cast<const float4 *>(cd + BN * 4) + half * kSubW;
            const float *sxs = reinterpret_cast<const float *>(cd + BN * 4 + BN / 32 * 16) + half * kSubW;   // FP8 only
            const int colw = cur.n * tile_step * BN + half * HC;   // first column this warp owns in the tile
            int nd = 0;           // rows put aside, and which: byte i = lane | chunk << 5 of row i
            uint32_t dmeta = 0;
            float4 gm;            // kModeMaxima: the current 64 columns' group bounds

            // FP8: h = fl(A s_q s_chunk - beta), one rounding (the scale product is an exact power of two)
            auto scale_of = [&](int ci) { return FP8 ? sq * sxs[ci] : p.scale; };
            auto bound_of = [&](int ci) {
                const float4 cs = cst[ci];
                return __fmaf_ru(rp.z, cs.x, __fmaf_ru(rp.w, cs.y, cs.z));
            };
            // kModeMaxima: a lower bound of the best h of columns 16 i .. 16 i + 15 of chunk ci
            auto best16 = [&](const uint32_t (&v)[32], int ci, int i) {
                const float4 *b4 = reinterpret_cast<const float4 *>(beta + ci * 32 + 16 * i);
                float m = __int_as_float(0xff800000);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 bq = b4[q];
                    const int j = 16 * i + 4 * q;
                    m = fmax3(m, __fmaf_rn(__uint_as_float(v[j]), p.scale, -bq.x), __fmaf_rn(__uint_as_float(v[j + 1]), p.scale, -bq.y));
                    m = fmax3(m, __fmaf_rn(__uint_as_float(v[j + 2]), p.scale, -bq.z), __fmaf_rn(__uint_as_float(v[j + 3]), p.scale, -bq.w));
                }
                return __fsub_rd(m, __fadd_ru(bound_of(ci), rp.x));
            };
            // One 32-column chunk ci of this warp's HC columns
            auto chunk = [&](const uint32_t (&v)[32], int ci) {
                if constexpr (MODE == kModeDump) {   // diagnostics: every pair's h and bound, at caller row order
                    const float sc = scale_of(ci), eh = bound_of(ci);
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int c = colw + ci * 32 + j;
                        if (r < p.nR && c < p.nS) {
                            const size_t oi = (size_t)p.orig_r[r] * p.nS + p.orig_s[c];
                            p.dump_h[oi] = __fmaf_rn(__uint_as_float(v[j]), sc, -beta[ci * 32 + j]);
                            p.dump_e[oi] = eh;
                        }
                    }
                } else if constexpr (MAXIMA) {
                    if (ci & 1) {
                        gm.z = best16(v, ci, 0);
                        gm.w = best16(v, ci, 1);
                        if (r < p.nR) {   // group bounds of 64 columns
                            float *o = p.gmax + (size_t)(r - p.row0) * p.n_groups;
                            const int g64 = cur.n * (BN / 64) + half * (HC / 64) + (ci >> 1);
                            if (p.gran == 64)
                                o[g64] = fmaxf(fmaxf(gm.x, gm.y), fmaxf(gm.z, gm.w));
                            else
                                *reinterpret_cast<float4 *>(o + 4 * g64) = gm;   // n_groups is a multiple of 4 here
                        }
                    } else {
                        gm.x = best16(v, ci, 0);
                        gm.y = best16(v, ci, 1);
                    }
                } else {
                    // Whole-chunk reject: with beta_j >= beta_min(chunk) and one scale s > 0 per chunk,
                    // every h_j = fl(A_j s - beta_j) is <= fl_ru(max_j A_j * s - beta_min); rows are in
                    // norm order, so beta_min is tight.
                    const float sc = scale_of(ci), eh = bound_of(ci);
                    const bool hit = __fmaf_ru(max_tree32(v), sc, -cst[ci].w) >= __fsub_rd(rp.y, eh);
                    unsigned hm = __ballot_sync(0xffffffffu, hit);
                    if (hm) {
                        const int nh = __popc(hm);
                        if (nd + nh <= kDefer) {   // put the rows' values aside: classified after the release
                            if (hit) {
                                float4 *x4 = reinterpret_cast<float4 *>(my_def + (nd + __popc(hm & lt)) * kDeferPitch);
#pragma unroll
                                for (int i = 0; i < 8; ++i)
                                    x4[i] = make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]),
                                                        __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3]));
                            }
                            for (; hm; hm &= hm - 1u, ++nd) dmeta |= (uint32_t)(__ffs((int)hm) - 1 + (ci << 5)) << (8 * nd);
                        } else {
                            scnt = slow_many<kCap>(p, v, beta + ci * 32, sc, __fadd_ru(rp.x, eh), __fsub_rd(rp.y, eh), hit, r,
                                                   colw + ci * 32, my_stg, scnt);
                        }
                    }
                }
            };
            auto release_acc = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {   // TMEM buffer free; the rest is in registers
                    if constexpr (CG2) {
                        if (leader)
                            mbar_arrive(acc_empty + b * 8);
                        else
                            mbar_arrive_remote(mapa_shared(acc_empty + b * 8, 0u));
                    } else {
                        mbar_arrive(acc_empty + b * 8);
                    }
                }
            };
            // 32 columns at a time: with 8 warps the next load is in flight while one is processed, with
            // 16 (96 registers a thread) the other three warps of the SM sub-partition hide it
            if constexpr (WIDE) {
                uint32_t v[32];
#pragma unroll
                for (int ci = 0; ci < kSubW; ++ci) {
                    tmem_ld_32x32b_x32(tbase + 32 * ci, v);
                    tmem_ld_wait_regs(v);
                    if (ci == kSubW - 1) release_acc();
                    chunk(v, ci);
                }
            } else {
                uint32_t va[32], vb[32];
                tmem_ld_32x32b_x32(tbase, va);
                tmem_ld_wait_regs(va);
                tmem_ld_32x32b_x32(tbase + 32, vb);
                chunk(va, 0);
                tmem_ld_wait_regs(vb);
                if constexpr (kSubW == 4) {
                    tmem_ld_32x32b_x32(tbase + 64, va);
                    chunk(vb, 1);
                    tmem_ld_wait_regs(va);
                    tmem_ld_32x32b_x32(tbase + 96, vb);
                    chunk(va, 2);
                    tmem_ld_wait_regs(vb);
                }
                release_acc();
                chunk(vb, kSubW - 1);
            }
            if (MODE == kModeEps && nd) {
                // the rows put aside, one at a time: lane j classifies column j, the candidates' buffer
                // positions come from a ballot prefix
                __syncwarp();
                for (int i = 0; i < nd; ++i, dmeta >>= 8) {
                    const int k = (int)(dmeta & 31u), ci = (int)((dmeta >> 5) & 7u);
                    const float eh = bound_of(ci);
                    const float ta = __shfl_sync(0xffffffffu, __fadd_ru(rp.x, eh), k);
                    const float tr = __shfl_sync(0xffffffffu, __fsub_rd(rp.y, eh), k);
                    const float sc = FP8 ? __shfl_sync(0xffffffffu, scale_of(ci), k) : p.scale;
                    const int rk = r - lane + k, c = colw + ci * 32 + lane;
                    const float h = __fmaf_rn(my_def[i * kDeferPitch + lane], sc, -beta[ci * 32 + lane]);
                    const bool cand = c < p.nS && h >= tr && (!p.upper || c > rk);   // upper mode: pairs with c > r only
                    const unsigned cm = __ballot_sync(0xffffffffu, cand);
                    if (cm) {
                        if (scnt + __popc(cm) > (uint32_t)kCap) flush_stage(p, my_stg, scnt);
                        if (cand && DL_CHECK(scnt + __popc(cm & lt) < (uint32_t)kCap, 2, scnt + __popc(cm & lt)))
                            my_stg[scnt + __popc(cm & lt)] = make_uint2((uint32_t)rk, (uint32_t)c | (h >= ta ? 0u : kBandFlag));
                        scnt += __popc(cm);
                    }
                }
            }
            __syncwarp();   // every lane is done with the column data and the rows put aside
            if (lane == 0) mbar_arrive(col_empty + cs_slot * 8);
#pragma unroll
            for (int g = 0; g < kGroups; ++g) cur.next(p);
            t += kGroups;
        }
        if constexpr (MODE == kModeEps) flush_stage(p, my_stg, scnt);
        if (!ok) raise_abort();
    }

    __syncthreads();
    // CG2: neither CTA of the pair releases its TMEM or exits while the other may still use
    // it -- the leader's MMAs write the peer's TMEM and read its shared memory, and the peer
    // arrives on the leader's barriers. Every path of every thread reaches this point.
    if constexpr (CG2) cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc<CG2>(tmem_base, kTmemCols);
    }
}

static size_t tc_extra_bytes(int BN, bool fp8, bool wide)
{
    // the column ring; per epilogue warp the rows put aside and the candidate buffer; 64 barrier and
    // flag words
    const size_t epi = (size_t)tc_epi_warps(wide);
    return (size_t)kColRing * tc_col_bytes(BN, fp8) + epi * (kDefer * kDeferPitch * 4 + tc_stage_cap(wide) * 8) + 64 * 8;
}

// One S stage per CTA: a 128-byte K chunk of the CTA's rows of an S tile (all BN rows, or
// BN/2 for a CTA pair).
static size_t tc_stage_bytes(int BN, bool cg2) { return (size_t)(cg2 ? BN / 2 : BN) * 128; }

// a_slots == 0: streamed R chunks, 16 KB more per stage and no resident tile
static size_t tc_smem_bytes(int BN, int kc, int stages, int a_slots, bool fp8, bool cg2, bool wide)
{
    return 1024 + (size_t)a_slots * kc * 16384 + (size_t)stages * (tc_stage_bytes(BN, cg2) + (a_slots ? 0 : 16384)) +
           tc_extra_bytes(BN, fp8, wide);
}

// Shared-memory plan: two A slots when that still leaves at least three S stages, else one;
// with `stream` (the one-SM epsilon-join), a plan that would be left with fewer than three
// stages beside one resident R tile streams the R tile's chunks with the S chunks instead
// (a_slots = 0).
void tc_plan(int BN, int kc, int *stages, int *a_slots, bool fp8, bool cg2, bool wide, bool stream)
{
    const long cap = 232448;
    for (int slots = 2; slots >= 1; --slots) {
        const long avail = cap - 1024 - (long)tc_extra_bytes(BN, fp8, wide) - (long)slots * kc * 16384;
        long s = avail / (long)tc_stage_bytes(BN, cg2);
        if (s > 8) s = 8;
        if (s >= 3 || slots == 1) {
            *stages = (int)s;
            *a_slots = slots;
            if (s >= 3 || !stream || cg2) return;
            break;
        }
    }
    long s = (cap - 1024 - (long)tc_extra_bytes(BN, fp8, wide)) / (long)(tc_stage_bytes(BN, cg2) + 16384);
    if (s > 8) s = 8;
    *stages = (int)s;
    *a_slots = 0;
}

static std::atomic<long long> g_wait_budget{0};

long long tc_wait_budget()
{
    const long long b = g_wait_budget.load(std::memory_order_relaxed);
    return b > 0 ? b : kWaitBudgetClocks;
}

template <int BN, int MODE, bool FP8, bool CG2, bool WIDE = false, bool MASK = false, bool STREAM = false>
static int launch_one(const TcLaunch &L, size_t smem, cudaStream_t st, int *grid_out)
{
    auto kern = tc_join_kernel<BN, MODE, FP8, CG2, WIDE, MASK, STREAM>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(tc_join_kernel)");
    TcParams p = L.p;
    p.wait_budget = tc_wait_budget();
    if constexpr (CG2) {
        cudaLaunchConfig_t cfg = {};
        cfg.blockDim = dim3(tc_threads(WIDE));
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        // persistent pairs: no more than can be resident at once (GPCs may leave an SM unpaired)
        cfg.gridDim = dim3(2);
        int pairs = 0;
        e = cudaOccupancyMaxActiveClusters(&pairs, kern, &cfg);
        if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveClusters(tc_join_kernel)");
        if (pairs < 1) {
            set_error("tensor-core join: no CTA pair fits on this device");
            return DL_EUNSUPPORTED;
        }
        const int want = std::max(1, L.grid / 2);
        cfg.gridDim = dim3((unsigned)(2 * std::min(want, pairs)));
        e = cudaLaunchKernelEx(&cfg, kern, *L.tmA, *L.tmB, p);
        if (e != cudaSuccess) return cuda_fail(e, "tc_join_kernel (CTA pairs) launch");
        if (grid_out) *grid_out = (int)cfg.gridDim.x;
    } else {
        kern<<<L.grid, tc_threads(WIDE), smem, st>>>(*L.tmA, *L.tmB, p);
        if (grid_out) *grid_out = L.grid;
    }
    return DL_OK;
}

void tc_grid_units(TcLaunch *L, int64_t mt, int64_t nt, int sms)
{
    // the range length whose last wave wastes least: units are handed out round-robin, one CTA an SM,
    // and each loads its R tile (counted as half an S tile); ties go to the longer range
    int64_t best = 1;
    double best_cost = 1e300;
    for (int64_t len = std::min<int64_t>(nt, 64); len >= 1; --len) {
        const int64_t units = mt * ((nt + len - 1) / len);
        const double cost = (double)((units + sms - 1) / sms) * ((double)len + 0.5);
        if (cost < best_cost) {
            best_cost = cost;
            best = len;
        }
    }
    const int64_t units = mt * ((nt + best - 1) / best);
    L->p.units = nullptr;
    L->p.mt = (int)mt;
    L->p.unit_nt = (int)nt;
    L->p.unit_len = (int)best;
    L->p.n_units = (int)units;
    L->grid = (int)std::min<int64_t>(units, sms);
}

int launch_tc_join(const TcLaunch &L, cudaStream_t st, int mode, bool fp8, int *grid_out)
{
    const bool topk = mode == kModeMaxima;
    const bool dump = mode == kModeDump;
    if (topk && fp8) {
        set_error("top-k group maxima run on the 16-bit path only");
        return DL_EUNSUPPORTED;
    }
    if ((L.cg2 && (topk || L.BN != 256 || L.wide)) || (L.wide && L.BN != 256)) {
        set_error("tensor-core join: CTA pairs serve the 256-column epsilon-join, the wide epilogue 256-column tiles");
        return DL_EUNSUPPORTED;
    }
    const size_t smem = tc_smem_bytes(L.BN, L.p.kc, L.p.stages, L.p.a_slots, fp8, L.cg2, L.wide);
    if (L.p.stages < 2 || smem > 232448) {
        set_error("tensor-core join: no shared-memory plan for d=%d, tile %d", L.p.kc * 64, L.BN);
        return DL_EUNSUPPORTED;
    }
    int rc;
    if (dump) {   // diagnostics: one configuration
        if (L.cg2 || L.wide || L.BN != 256 || L.p.tile_mask) {
            set_error("tensor-core join: scores are dumped from the one-SM 256-column tiles");
            return DL_EUNSUPPORTED;
        }
        if (L.p.a_slots == 0)
            rc = fp8 ? launch_one<256, kModeDump, true, false, false, false, true>(L, smem, st, grid_out)
                     : launch_one<256, kModeDump, false, false, false, false, true>(L, smem, st, grid_out);
        else
            rc = fp8 ? launch_one<256, kModeDump, true, false>(L, smem, st, grid_out)
                     : launch_one<256, kModeDump, false, false>(L, smem, st, grid_out);
    } else if (L.p.a_slots == 0) {   // streamed R chunks (tc_plan with stream): the one-SM epsilon-join
        if (topk || L.cg2 || L.p.tile_mask) {
            set_error("tensor-core join: streamed R chunks serve the dense one-SM epsilon-join");
            return DL_EUNSUPPORTED;
        }
        if (L.wide)
            rc = fp8 ? launch_one<256, kModeEps, true, false, true, false, true>(L, smem, st, grid_out)
                     : launch_one<256, kModeEps, false, false, true, false, true>(L, smem, st, grid_out);
        else if (L.BN == 256)
            rc = fp8 ? launch_one<256, kModeEps, true, false, false, false, true>(L, smem, st, grid_out)
                     : launch_one<256, kModeEps, false, false, false, false, true>(L, smem, st, grid_out);
        else if (L.BN == 128)
            rc = fp8 ? launch_one<128, kModeEps, true, false, false, false, true>(L, smem, st, grid_out)
                     : launch_one<128, kModeEps, false, false, false, false, true>(L, smem, st, grid_out);
        else {
            set_error("tensor-core tile width %d not supported (128 or 256)", L.BN);
            return DL_EINVAL;
        }
    } else if (L.p.tile_mask) {   // the pruned join: units and their count built on the device
        if (topk || L.cg2 || !L.p.n_units_dev) {
            set_error("tensor-core join: a tile mask serves the one-SM epsilon-join with device-built units");
            return DL_EUNSUPPORTED;
        }
        if (L.wide)
            rc = fp8 ? launch_one<256, kModeEps, true, false, true, true>(L, smem, st, grid_out)
                     : launch_one<256, kModeEps, false, false, true, true>(L, smem, st, grid_out);
        else if (L.BN == 256)
            rc = fp8 ? launch_one<256, kModeEps, true, false, false, true>(L, smem, st, grid_out)
                     : launch_one<256, kModeEps, false, false, false, true>(L, smem, st, grid_out);
        else if (L.BN == 128)
            rc = fp8 ? launch_one<128, kModeEps, true, false, false, true>(L, smem, st, grid_out)
                     : launch_one<128, kModeEps, false, false, false, true>(L, smem, st, grid_out);
        else {
            set_error("tensor-core tile width %d not supported (128 or 256)", L.BN);
            return DL_EINVAL;
        }
    } else if (L.cg2)
        rc = fp8 ? launch_one<256, kModeEps, true, true>(L, smem, st, grid_out) : launch_one<256, kModeEps, false, true>(L, smem, st, grid_out);
    else if (L.wide)
        rc = topk ? launch_one<256, kModeMaxima, false, false, true>(L, smem, st, grid_out)
                  : (fp8 ? launch_one<256, kModeEps, true, false, true>(L, smem, st, grid_out)
                         : launch_one<256, kModeEps, false, false, true>(L, smem, st, grid_out));
    else if (L.BN == 256)
        rc = topk ? launch_one<256, kModeMaxima, false, false>(L, smem, st, grid_out)
                  : (fp8 ? launch_one<256, kModeEps, true, false>(L, smem, st, grid_out)
                         : launch_one<256, kModeEps, false, false>(L, smem, st, grid_out));
    else if (L.BN == 128)
        rc = topk ? launch_one<128, kModeMaxima, false, false>(L, smem, st, grid_out)
                  : (fp8 ? launch_one<128, kModeEps, true, false>(L, smem, st, grid_out)
                         : launch_one<128, kModeEps, false, false>(L, smem, st, grid_out));
    else {
        set_error("tensor-core tile width %d not supported (128 or 256)", L.BN);
        return DL_EINVAL;
    }
    if (rc) return rc;
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "tc_join_kernel launch");
    return DL_OK;
}

}  // namespace dl

// Diagnostics: shorten the abortable pipeline waits of every tensor-core kernel
// launched from now on (0 restores the default), so tests can make a healthy
// join's wait run out and exercise the abort path.
extern "C" int dl_debug_set_wait_budget(int64_t clocks)
{
    dl::clear_error();
    if (clocks < 0) {
        dl::set_error("dl_debug_set_wait_budget: clocks must be >= 0 (got %lld)", (long long)clocks);
        return DL_EINVAL;
    }
    dl::g_wait_budget.store(clocks, std::memory_order_relaxed);
    return DL_OK;
}

DL_CHECK_READER(join_tc)
