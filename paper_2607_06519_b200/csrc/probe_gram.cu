// Routing probe on second moments (bf16 storage, head_dim 128): the error term of Eq. 2 for the keys that every probe
// query sees.
//
// With the operand R (shared: R = Z1 of K; residual: R with the kept entries zeroed) and the probe rows Q,
//     sum over rows r, keys j of (Q_r . R_j)^2  =  sum_{a,b} (R^T R)[a][b] * (Q^T Q)[a][b],
// so once all rows see a range of keys their error needs the 128 x 128 second moments of the range instead of a product
// with every row: 2 * 128 * 128 flops per key and candidate whatever the number of rows (512 rows of a pair at group
// size 4 and 64 probe queries: a quarter of the product's), and Z1 is read once for both candidates, the second formed
// in shared memory from the bit map of the kept entries.  The keys from the first probe position on, which some rows do
// not see, stay with probe_tc_kernel.
//
//   * One persistent CTA per SM; CTA c takes an even share of the flat list of (operand, 128-token tile) pairs; a segment
//     is its run of tiles of one operand (Z1 of a unit, or one layer's deviation of a block of four).
//   * warp 0: TMA ring (tile: two 64-channel boxes, 128-byte swizzle; the tile's 2 KiB of the bit map);
//     warps 6-13: write the tile with its kept entries zeroed next to it; warp 1: both products, tokens on K, so the
//     operands are MN-major views of the row-major tiles, A and B the same tile (8 + 8 tcgen05.mma, M = N = 128, K = 16);
//     warps 2-5: epilogue.
//   * Q^T Q of the segment's rows comes first, through the same ring and accumulators, 32 rows at a time: the epilogue adds them up
//     in a third 128-column region of tensor memory.
//   * The sums are drained every two tiles, one candidate's while the other's products run: <R^T R, Q^T Q> in float32 over 32
//     columns of a row, added up in float64.
//   * Precision.  The tensor core rounds its accumulators towards zero, so what counts is the number of steps that one takes: 16 for
//     R^T R (the products: eight and a square) and two for Q^T Q (all rows in one accumulator: 1.3e-6 off float64 at 512 rows, 5.5e-6
//     at 2 048; 128 rows: 6e-7).
//     The sum cancels where queries and coefficients are nearly orthogonal, which the products, sums of squares, do not.  So the
//     traces are kept too: tr(R^T R) tr(Q^T Q) is the sum of |Q_r|^2 |R_j|^2, and a unit whose error is a small part of it (or not
//     finite) is done again by products (probe_tc.cu).
// A tile takes 1.6 us (32 layers of 32k tokens: 428 us a probe call).  The products read 128 KiB of operands per tile from shared
// memory, the masking 64 KiB, the copy 32 KiB: 0.9 us at 128 bytes per cycle; HBM's share is 0.7 us; the rest is the hand-over of
// the accumulators at every drain.
#include <algorithm>

#include "fdkv_internal.h"
#include "umma.cuh"

namespace fdkv {

namespace {

constexpr int kGT = 128;                  // tokens per tile
constexpr int kGStages = 3;
constexpr int kGHalf = kGT * 128;         // one 64-channel half of a tile: 16 KiB
constexpr int kGTile = 2 * kGHalf;
constexpr int kGStage = 2 * kGTile;       // the tile and its copy without the kept entries
constexpr int kGBits = kGT * 16;          // the tile's part of the bit map
constexpr int kGHdr = 1024;
constexpr int kGSmem = kGHdr + kGStages * (kGStage + kGBits);  // 199 KiB
constexpr int kGMaskWarps = 8;
constexpr int kGThreads = (6 + kGMaskWarps) * 32;
constexpr int kGroup = 2;                 // tiles per drain
constexpr int kQSteps = 2;                // steps of 16 probe rows per drain
constexpr int kGColF = 0, kGColD = 128, kGColA = 256;  // tensor memory: R^T R of both candidates, Q^T Q
constexpr uint32_t kGIdesc = umma_idesc(128, 128, true);
// (accumulator barriers: the shared candidate's at +0, the residual's at +8)
constexpr int gFull = 0, gMasked = 32, gEmpty = 64, gAccFull = 96, gAccEmpty = 112, gSlot = 128, gAbort = 132, gRed = 144;

struct GramPlan {
    int n_ops;    // operands per unit: 1, or 4 for a block of four layers
    int nt;       // tiles per operand
    int ncta;
    int maxseg;   // part slots per operand
    int rows;     // probe rows per operand
    int qtiles;   // 128-row tiles of them
};

// the CTA whose share holds tile g of the flat list of n tiles (CTA c starts at c * n / ncta, rounded down)
__device__ __forceinline__ int gram_cta_of(int64_t g, int64_t n, int ncta) { return (int)(((g + 1) * ncta - 1) / n); }

__global__ void __launch_bounds__(kGThreads, 1)
probe_gram_kernel(const __grid_constant__ CUtensorMap tmap, ProbeArgs a, GramPlan pl) {
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sm0 = s_u32(smem);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + gAbort);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (sm0 & 1023u) {
        if (threadIdx.x == 0) atomicMax(a.status, (int32_t)kFlagCountMismatch);
        return;
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < kGStages; ++s) {
            mb_init(sm0 + gFull + 8 * s, 1);
            mb_init(sm0 + gMasked + 8 * s, kGMaskWarps);
            mb_init(sm0 + gEmpty + 8 * s, 1);
        }
        for (int c = 0; c < 2; ++c) { mb_init(sm0 + gAccFull + 8 * c, 1); mb_init(sm0 + gAccEmpty + 8 * c, 4); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm0 + gSlot), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + gSlot);
    const uint32_t stage0 = sm0 + kGHdr, bits0 = stage0 + kGStages * kGStage;
    const int64_t n_tiles = (int64_t)a.unit_count * pl.n_ops * pl.nt;
    const int64_t g_begin = (int64_t)blockIdx.x * n_tiles / pl.ncta, g_end = (int64_t)(blockIdx.x + 1) * n_tiles / pl.ncta;

    // every role walks the same sequence: per segment its Q tiles, then its token tiles; item `it` uses stage it % kGStages
    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            for (int64_t g = g_begin; g < g_end;) {
                const int op = (int)(g / pl.nt), t0 = (int)(g % pl.nt);
                const int n = (int)min((int64_t)pl.nt - t0, g_end - g);
                const int unit = a.unit_begin + op / pl.n_ops, layer = op % pl.n_ops;
                const int64_t row0 = ((int64_t)unit * pl.n_ops + layer) * a.Tmax;
                const uint8_t* bits = reinterpret_cast<const uint8_t*>(a.keep + (int64_t)unit * a.keep_stride);
                for (int i = -pl.qtiles; i < n; ++i, ++it) {
                    const int s = it % kGStages;
                    const uint32_t full = sm0 + gFull + 8 * s;
                    mb_wait(sm0 + gEmpty + 8 * s, ((uint32_t)(it / kGStages) & 1u) ^ 1u, abort_flag, a.status);
                    if (*abort_flag) break;
                    if (i < 0) { mb_arrive(full); continue; }
                    const uint32_t dst = stage0 + s * kGStage;
                    const int t = t0 + i;
                    mb_expect_tx(full, kGTile + kGBits);
                    tma_2d(dst, &tmap, 0, (int)(row0 + (int64_t)t * kGT), full);
                    tma_2d(dst + kGHalf, &tmap, 64, (int)(row0 + (int64_t)t * kGT), full);
                    bulk_load(bits0 + s * kGBits, bits + (int64_t)t * kGBits, kGBits, full);
                }
                if (*abort_flag) break;
                g += n;
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int it = 0;
            uint32_t gen0 = 0, gen1 = 0;  // drains of either accumulator
            for (int64_t g = g_begin; g < g_end;) {
                const int t0 = (int)(g % pl.nt), n = (int)min((int64_t)pl.nt - t0, g_end - g);
                for (int i = -pl.qtiles; i < n; ++i, ++it) {
                    const int s = it % kGStages;
                    const uint32_t par = (uint32_t)(it / kGStages) & 1u;
                    mb_wait(sm0 + gFull + 8 * s, par, abort_flag, a.status);
                    mb_wait(sm0 + gMasked + 8 * s, par, abort_flag, a.status);
                    if (*abort_flag) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t df = smem_desc_sw128(stage0 + s * kGStage, kGHalf, 1024);
                    const uint64_t dd = smem_desc_sw128(stage0 + s * kGStage + kGTile, kGHalf, 1024);
                    auto open = [&](int c) {
                        mb_wait(sm0 + gAccEmpty + 8 * c, ((c ? gen1 : gen0) & 1u) ^ 1u, abort_flag, a.status);
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    };
                    auto close = [&](int c) {
                        umma_commit(sm0 + gAccFull + 8 * c);
                        if (c) ++gen1; else ++gen0;
                    };
                    if (i < 0) {  // probe rows: kQSteps steps per drain, the accumulators in turn
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const int c = k / kQSteps & 1;
                            if (k % kQSteps == 0) open(c);
                            umma_ss<kGIdesc>(tmem + (c ? kGColD : kGColF), dd + k * (2048 >> 4), dd + k * (2048 >> 4), k % kQSteps > 0);
                            if (k % kQSteps == kQSteps - 1) close(c);
                        }
                    } else {
                        // one candidate's accumulator is drained while the other's products run
                        const bool opens = i % kGroup == 0, closes = i % kGroup == kGroup - 1 || i == n - 1;
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            if (opens) open(c);
                            const uint64_t desc = c ? dd : df;
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                umma_ss<kGIdesc>(tmem + (c ? kGColD : kGColF), desc + k * (2048 >> 4), desc + k * (2048 >> 4), k > 0 || !opens);
                            if (closes) close(c);
                        }
                    }
                    umma_commit(sm0 + gEmpty + 8 * s);
                }
                if (*abort_flag) break;
                g += n;
            }
        }
    } else if (warp < 6) {
        // ---- epilogue: thread = row of the 128 x 128 moments (tensor memory lane) ----
        const int lq = warp & 3;
        const uint32_t tq = tmem + ((uint32_t)(lq * 32) << 16);
        uint32_t gen0 = 0, gen1 = 0;  // drains of either accumulator
        // this row's diagonal element, if it is in these columns' block b (picked by the bits of the lane)
        auto diagonal = [&](int b, const uint32_t (&r)[32]) {
            if (b != lq) return 0.f;
            uint32_t x[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) x[j] = lane & 16 ? r[j + 16] : r[j];
#pragma unroll
            for (int w = 8; w; w >>= 1)
#pragma unroll
                for (int j = 0; j < w; ++j) x[j] = lane & w ? x[j + w] : x[j];
            return __uint_as_float(x[0]);
        };
        auto await = [&](int c) {
            mb_wait(sm0 + gAccFull + 8 * c, (c ? gen1 : gen0) & 1u, abort_flag, a.status);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        };
        auto drained = [&](int c) {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mb_arrive(sm0 + gAccEmpty + 8 * c);
            if (c) ++gen1; else ++gen0;
        };
        for (int64_t g = g_begin; g < g_end;) {
            const int op = (int)(g / pl.nt), t0 = (int)(g % pl.nt), n = (int)min((int64_t)pl.nt - t0, g_end - g);
            double sum0 = 0.0, sum1 = 0.0;
            float tr0 = 0.f, tr1 = 0.f, tr_q = 0.f;  // (only a measure: a few digits will do)
            const int qdrains = pl.qtiles * (8 / kQSteps);
#pragma unroll 1
            for (int q = 0; q < qdrains; ++q) {
                const int c = q & 1;
                await(c);
                if (!*abort_flag) {
#pragma unroll 1
                    for (int b = 0; b < 4; ++b) {
                        uint32_t rr[32], ra[32];
                        tmem_ld32(tq + (c ? kGColD : kGColF) + b * 32, rr);
                        tmem_ld32(tq + kGColA + b * 32, ra);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int j = 0; j < 32; ++j) rr[j] = q > 0 ? __float_as_uint(__uint_as_float(rr[j]) + __uint_as_float(ra[j])) : rr[j];
                        tmem_st32(tq + kGColA + b * 32, rr);
                        if (q == qdrains - 1) tr_q += diagonal(b, rr);
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                }
                drained(c);
            }
            for (int i0 = 0; i0 < n; i0 += kGroup) {
#pragma unroll 1
                for (int c = 0; c < 2; ++c) {
                    await(c);
                    if (!*abort_flag) {
                        double e = 0.0;
                        float dg = 0.f;
#pragma unroll 2
                        for (int b = 0; b < 4; ++b) {  // (unrolled it takes more registers than a thread has)
                            uint32_t rr[32], ra[32];
                            tmem_ld32(tq + (c ? kGColD : kGColF) + b * 32, rr);
                            tmem_ld32(tq + kGColA + b * 32, ra);
                            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                            float f0 = 0.f, f1 = 0.f;
#pragma unroll
                            for (int j = 0; j < 32; j += 2) {
                                f0 = fmaf(__uint_as_float(rr[j]), __uint_as_float(ra[j]), f0);
                                f1 = fmaf(__uint_as_float(rr[j + 1]), __uint_as_float(ra[j + 1]), f1);
                            }
                            e += (double)f0 + (double)f1;
                            dg += diagonal(b, rr);
                        }
                        (c ? sum1 : sum0) += e;
                        (c ? tr1 : tr0) += dg;
                    }
                    drained(c);
                }
            }
            // the four warps' five sums: both candidates' errors and traces, the queries' trace
            double v[5] = {sum0, sum1, (double)tr0, (double)tr1, (double)tr_q};
            double* const red = reinterpret_cast<double*>(smem + gRed);
#pragma unroll
            for (int k = 0; k < 5; ++k) {
#pragma unroll
                for (int o = 16; o; o >>= 1) v[k] += __shfl_xor_sync(0xFFFFFFFFu, v[k], o);
                if (lane == 0) red[4 * k + lq] = v[k];
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (warp == 2) {
                // part slots of the operand: one per CTA that holds some of its tiles, in order; the last of them clears the rest
                const int c0 = gram_cta_of((int64_t)op * pl.nt, n_tiles, pl.ncta);
                const int unit = a.unit_begin + op / pl.n_ops;
                const int first = (op % pl.n_ops) * pl.maxseg, slot = (int)blockIdx.x - c0;
                double* const p = a.part + ((int64_t)unit * a.nptiles_max + first) * 2;
                double* const m = a.scale + ((int64_t)unit * kMaxGramSlots + first) * 2;
                auto all = [&](int k) { return (red[4 * k] + red[4 * k + 1]) + (red[4 * k + 2] + red[4 * k + 3]); };
                if (lane < 2) {
                    p[slot * 2 + lane] = all(lane);
                    m[slot * 2 + lane] = all(2 + lane) * all(4);
                }
                if (t0 + n == pl.nt)
                    for (int i = (slot + 1) * 2 + lane; i < pl.maxseg * 2; i += 32) p[i] = m[i] = 0.0;
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (*abort_flag) break;
            g += n;
        }
    } else {
        // ---- the ring's second half: probe rows, or the tile with its kept entries zeroed ----
        const int tm = threadIdx.x - 6 * 32;
        int it = 0;
        for (int64_t g = g_begin; g < g_end;) {
            const int op = (int)(g / pl.nt), t0 = (int)(g % pl.nt), n = (int)min((int64_t)pl.nt - t0, g_end - g);
            const int unit = a.unit_begin + op / pl.n_ops, h = unit % a.Hkv, blk = unit / a.Hkv;
            for (int i = -pl.qtiles; i < n; ++i, ++it) {
                const int s = it % kGStages;
                uint8_t* const full = smem + kGHdr + s * kGStage;
                uint8_t* const drop = full + kGTile;
                mb_wait(sm0 + gFull + 8 * s, (uint32_t)(it / kGStages) & 1u, abort_flag, a.status);
                if (*abort_flag) break;
                if (i < 0) {
                    // row r of the operand's probe rows: ((layer *) G + g) * W + qi -> Q[layer][qi][h * G + g][:]; zeros behind the last
                    const int rb = (i + pl.qtiles) * 128, rows_layer = a.G * a.W;
#pragma unroll
                    for (int q = 0; q < 2048 / (kGMaskWarps * 32); ++q) {
                        const int v = q * (kGMaskWarps * 32) + tm, rl = v >> 4, chunk = v & 15, r = rb + rl;
                        uint4 x = make_uint4(0u, 0u, 0u, 0u);
                        if (r < pl.rows) {
                            const int layer = pl.n_ops == 4 ? op & 3 : r / rows_layer, rr = pl.n_ops == 4 ? r : r % rows_layer;
                            const __nv_bfloat16* src = reinterpret_cast<const __nv_bfloat16*>(a.q_layers_dev[a.B * blk + layer]);
                            x = *reinterpret_cast<const uint4*>(src + ((int64_t)(rr % a.W) * a.Hq + h * a.G + rr / a.W) * 128 + chunk * 8);
                        }
                        *reinterpret_cast<uint4*>(drop + (chunk >> 3) * kGHalf + rl * 128 + (((chunk & 7) ^ (rl & 7)) << 4)) = x;
                    }
                } else {
                    const uint8_t* const bits = smem + kGHdr + kGStages * kGStage + s * kGBits;
#pragma unroll
                    for (int q = 0; q < 2048 / (kGMaskWarps * 32); ++q) {
                        const int v = q * (kGMaskWarps * 32) + tm;  // 16-byte vectors in shared-memory order
                        const int row = (v >> 3) & 127, half = v >> 10, chunk = (v & 7) ^ (row & 7);
                        const uint4 x = *reinterpret_cast<const uint4*>(full + v * 16);
                        *reinterpret_cast<uint4*>(drop + v * 16) = drop_kept(x, bits[row * 16 + half * 8 + chunk]);
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic stores, read by the tensor core
                __syncwarp();
                if (lane == 0) mb_arrive(sm0 + gMasked + 8 * s);
            }
            if (*abort_flag) break;
            g += n;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);  // let copies and MMAs in flight finish before the memory goes away
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

}  // namespace

// Keys [0, t_full), a multiple of 128, which every probe row sees; *nparts part slots of every unit are written.
cudaError_t launch_probe_gram(const ProbeArgs& a, int t_full, cudaStream_t st, int* nparts) {
    static PerDevice once;
    int sm_count = 0;
    cudaError_t e = once.ensure([&]() { return cudaFuncSetAttribute(probe_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGSmem); }, &sm_count);
    if (e != cudaSuccess) return e;
    GramPlan pl;
    pl.n_ops = a.B == 4 ? 4 : 1;
    pl.nt = t_full / kGT;
    pl.rows = (a.B == 4 ? 1 : a.B) * a.G * a.W;
    pl.qtiles = (pl.rows + 127) / 128;
    const int64_t n = (int64_t)a.unit_count * pl.n_ops * pl.nt;
    pl.ncta = (int)std::min<int64_t>(std::min(sm_count, kMaxGramCtas), n);
    pl.maxseg = (int)((int64_t)pl.nt * pl.ncta / n) + 2;  // CTAs that can share an operand's tiles
    *nparts = pl.n_ops * pl.maxseg;
    probe_gram_kernel<<<pl.ncta, kGThreads, kGSmem, st>>>(*reinterpret_cast<const CUtensorMap*>(a.tmap_z1_128), a, pl);
    count_launch(1);
    return cudaGetLastError();
}

}  // namespace fdkv
