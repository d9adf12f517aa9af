// Routing probe on the 5th-generation tensor cores (bf16 storage, head_dim 128): the error term of Eq. 2.
//
// For a unit and a candidate (shared: R = Z1 of K; residual: R = Z1 of K with the kept entries zeroed) the probe
// needs sum_{rows, keys j <= pos(row)} (Q_row . R_j)^2 over the 2*G*W probe rows (2 layers x G group heads x W
// probe queries).  That is a dense [rows x 128] x [128 x T] contraction whose result is squared, masked causally
// and summed without ever leaving the SM:
//   * work item = (unit, layer of the pair, block of 128 probe rows, candidate, range of 256-token key tiles);
//     one CTA per item, 6 warps: warp 0 = TMA producer, warp 1 = MMA issuer (and TMEM owner), warps 2-5 = epilogue;
//   * A (the item's 128 Q rows) is written once into shared memory by the epilogue threads, in the
//     128-byte-swizzled K-major layout a TMA copy would give it; B tiles (256 tokens x 128 channels, same layout)
//     stream through a TMA ring of three stages (one in short items);
//   * per key tile 8 tcgen05.mma (M = 128, N = 256, K = 16, kind::f16, both operands from shared memory,
//     bf16 x bf16 -> f32) fill one of two alternating 128 x 256 f32 accumulators: all 512 columns of tensor memory.
//     (In short items there is one.)
//     The hand-over of an accumulator (commit -> epilogue -> release -> next MMA) is a round trip of about a
//     microsecond; with a single set it was paid on every tile and cost as much as the arithmetic, which is why A
//     lives in shared memory: the columns it took in tensor memory buy the second set.  (Two M tiles against
//     128-token key tiles, the same bytes per flop, measured 4 % slower.);
//   * epilogue: tcgen05.ld (32 lanes x 32 columns per instruction), square, mask keys after the row's probe
//     position, accumulate; the set is released as soon as its last columns are in registers; one float64 sum per
//     item, summed across items in a fixed order by the finalize kernel.
// Every mbarrier wait is bounded; on expiry the CTA flags the device status word, stops waiting and still frees
// its tensor memory before it retires.
#include <algorithm>
#include <cmath>

#include "fdkv_internal.h"
#include "umma.cuh"

namespace fdkv {

namespace {

constexpr int kBN = kProbeBoxRows;             // key tokens per tile (N of the MMA)
constexpr int kMT = 256 / kBN;                 // M tiles (128 Q rows each) per work item: 2 at N = 128, 1 at N = 256
static_assert(kMT == 1, "one M tile per item");
constexpr int kBHalf = kBN * 128;              // one 64-channel half of a B tile: 32 KiB
constexpr int kBStageBytes = 2 * kBHalf;       // 64 KiB
constexpr int kHdr = 1024;
constexpr int kAHalf = 128 * 128;              // one 64-channel half of an A tile (128 Q rows): 16 KiB
constexpr int kABytes = kMT * 2 * kAHalf;      // the item's M tiles
constexpr int probe_smem(int stages) { return kHdr + kABytes + stages * kBStageBytes; }  // 225 KiB with three, 97 with one
constexpr int kPThreads = 6 * 32;
// Tensor memory (512 columns): alternating sets of kMT 128 x kBN f32 accumulators (one per M tile).
constexpr int kAccSet = kMT * kBN;
static_assert(2 * kAccSet <= 512, "tensor memory budget");
// header: full[8] @0, empty[8] @64, tfull[2] @128, tempty[2] @144, tmem slot @160, abort @164, reduce @192 (4 doubles)
constexpr uint32_t kIdesc = umma_idesc(128, kBN, false);
constexpr int oFull = 0, oEmpty = 64, oTFull = 128, oTEmpty = 144, oSlot = 160, oAbort = 164, oRed = 192;


struct TcPlan {
    int items_per_unit;  // B layers x mblocks x 2 candidates x nsplits
    int mblocks, nsplits, ntiles, tiles_per_split;
    int pos_min, pos_max;
    int tile_first;   // first 256-key tile (the keys before it are probe_gram_kernel's)
    int slot0;        // first part slot
    // Units whose second moments are not exact enough: the keys before tile_first again, by the blocks behind the first sure_items
    int sure_items, redo_per_unit, redo_nsplits, redo_tiles_per_split, redo_slot0;
};

// kBStages, kAccSets: three and two for items of many tiles; one and one for items of a tile or two, whose time is the chain from
// the loads to the sum: two such blocks share an SM where there are that many.  Us a probe of 32 layers, one block against two per
// SM: 300 tokens (one or two tiles) 87 and 64, 1k (four) 110 and 89, 2k (eight) 143 and 128, 8k by products alone (nine or more) 338
// and 363; 128 items of seven tiles 37 and 42.
constexpr int kShortItem = 8;
template <int kBStages, int kAccSets>
__global__ void __launch_bounds__(kPThreads, kBStages == 1 ? 2 : 1)
probe_tc_kernel(const __grid_constant__ CUtensorMap tmap_z1, const __grid_constant__ CUtensorMap tmap_drop, ProbeArgs a, TcPlan pl) {
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int kTmemCols = kAccSets * kAccSet;
    const uint32_t sm0 = s_u32(smem);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + oAbort);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (sm0 & 1023u) {
        if (threadIdx.x == 0) atomicMax(a.status, (int32_t)kFlagCountMismatch);
        return;
    }
    const bool again = (int)blockIdx.x >= pl.sure_items;
    if (again) {  // (almost always there is nothing to do again)
        int any = 0;
        for (int u = threadIdx.x; u < a.unit_count; u += kPThreads) any |= a.redo[a.unit_begin + u];
        if (!__syncthreads_or(any)) return;
    }
    const int rows_layer = a.G * a.W;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kBStages; ++s) { mb_init(sm0 + oFull + 8 * s, 1); mb_init(sm0 + oEmpty + 8 * s, 1); }
        for (int s = 0; s < 2; ++s) { mb_init(sm0 + oTFull + 8 * s, 1); mb_init(sm0 + oTEmpty + 8 * s, 4); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {  // tensor memory
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm0 + oSlot), "r"((uint32_t)kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(smem + oSlot);
    const int per_unit = again ? pl.redo_per_unit : pl.items_per_unit, nsplits = again ? pl.redo_nsplits : pl.nsplits;
    const int per_split = again ? pl.redo_tiles_per_split : pl.tiles_per_split;
    int done = 0;  // tiles of the items before: the stages and accumulators go on in turn
    for (int item = again ? (int)blockIdx.x - pl.sure_items : (int)blockIdx.x; item < a.unit_count * per_unit; item += (int)gridDim.x - pl.sure_items) {
    // ---- decode the work item ----
    int it = item;
    const int unit = a.unit_begin + it / per_unit;
    if (again && !a.redo[unit]) continue;
    it %= per_unit;
    const int split = it % nsplits; it /= nsplits;
    const int cand = it & 1; it >>= 1;
    const int mblock = it % pl.mblocks; it /= pl.mblocks;
    const int layer = it;  // layer inside the depth block: 0 .. B-1
    const int h = unit % a.Hkv, pair = unit / a.Hkv;
    const int tile0 = (again ? 0 : pl.tile_first) + split * per_split;
    const int tile1 = min(again ? pl.tile_first : pl.ntiles, tile0 + per_split);
    const int ntile = max(0, tile1 - tile0);
    // ---- A operand: row r = mblock*256 + mt*128 + rl of this layer's probe block, r = g*W + qi -> Q[layer][qi][h*G+g][:],
    //      row rl of M tile mt: 16 chunks of 16 bytes, chunk c of a 64-channel half stored at chunk c ^ (rl & 7) ----
    if (warp >= 2) {
        const int rl = (warp & 3) * 32 + lane;
        const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(a.q_layers_dev[a.B * pair + layer]);
#pragma unroll 1
        for (int mt = 0; mt < kMT; ++mt) {
            const int r = mblock * (128 * kMT) + mt * 128 + rl;
            uint8_t* const arow = smem + kHdr + mt * 2 * kAHalf + rl * 128;
            const uint4* src = reinterpret_cast<const uint4*>(q + ((int64_t)(r % a.W) * a.Hq + h * a.G + r / a.W) * 128);
#pragma unroll
            for (int i = 0; i < 16; ++i)  // (padding rows are zero: they contribute nothing)
                *reinterpret_cast<uint4*>(arow + (i >> 3) * kAHalf + (((i & 7) ^ (rl & 7)) << 4)) = r < rows_layer ? src[i] : make_uint4(0u, 0u, 0u, 0u);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic stores, read by the tensor core
    }
    __syncthreads();
    const uint32_t b0 = sm0 + kHdr + kABytes;

    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            const CUtensorMap* map = cand ? &tmap_drop : &tmap_z1;
            // rows of this unit's K coefficients (a block of four stages one operand per layer)
            const int64_t row0 = a.B == 4 ? ((int64_t)unit * 4 + layer) * a.Tmax : (int64_t)unit * a.Tmax;
            for (int i = 0; i < ntile; ++i) {
                const int s = (done + i) % kBStages;
                const uint32_t ph = (uint32_t)((done + i) / kBStages) & 1u;
                mb_wait(sm0 + oEmpty + 8 * s, ph ^ 1u, abort_flag, a.status);
                if (*abort_flag) break;
                const uint32_t full = sm0 + oFull + 8 * s, dst = b0 + s * kBStageBytes;
                const int y = (int)(row0 + (int64_t)(tile0 + i) * kBN);
                mb_expect_tx(full, kBStageBytes);
                tma_2d(dst, map, 0, y, full);
                tma_2d(dst + kBHalf, map, 64, y, full);
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        if (lane == 0) {
            for (int i = 0; i < ntile; ++i) {
                const int s = (done + i) % kBStages, as = (done + i) % kAccSets;
                mb_wait(sm0 + oTEmpty + 8 * as, ((uint32_t)((done + i) / kAccSets) & 1u) ^ 1u, abort_flag, a.status);
                mb_wait(sm0 + oFull + 8 * s, (uint32_t)((done + i) / kBStages) & 1u, abort_flag, a.status);
                if (*abort_flag) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // one descriptor per stage and for A; the k steps and the two M tiles only add compile-time constants
                const uint64_t db_stage = smem_desc(b0 + s * kBStageBytes);
                const uint64_t da_all = smem_desc(sm0 + kHdr);
                const uint32_t d0 = tmem_base + (uint32_t)(as * kAccSet);
#pragma unroll
                for (int k = 0; k < 8; ++k) {  // 8 steps of 16 channels: 32 bytes inside the swizzle atom of either operand
#pragma unroll
                    for (int mt = 0; mt < kMT; ++mt) {  // the M tiles alternate: consecutive MMAs never wait for each other's accumulator
                        const uint64_t db = db_stage + (uint64_t)(((k >> 2) * kBHalf + (k & 3) * 32) >> 4);
                        const uint64_t da = da_all + (uint64_t)((mt * 2 * kAHalf + (k >> 2) * kAHalf + (k & 3) * 32) >> 4);
                        umma_ss<kIdesc>(d0 + mt * kBN, da, db, k > 0);
                    }
                }
                umma_commit(sm0 + oEmpty + 8 * s);    // the B stage is free once these MMAs have read it
                umma_commit(sm0 + oTFull + 8 * as);   // the accumulators are complete
            }
        }
    } else {
        // ================= epilogue: warps 2..5 own TMEM lanes 32*(warp%4) .. +31 =================
        const int lq = warp & 3;
        const int rl = lq * 32 + lane;  // row within a 128-row M tile == TMEM lane
        int pos_row[kMT];
#pragma unroll
        for (int mt = 0; mt < kMT; ++mt) {
            const int r = mblock * (128 * kMT) + mt * 128 + rl;
            pos_row[mt] = r < rows_layer ? a.pos[r % a.W] : -1;  // padding rows never count
        }
        double total = 0.0;
        for (int i = 0; i < ntile; ++i) {
            const int as = (done + i) % kAccSets;
            const int t0 = (tile0 + i) * kBN;
            mb_wait(sm0 + oTFull + 8 * as, (uint32_t)((done + i) / kAccSets) & 1u, abort_flag, a.status);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            float acc = 0.f;
            if (!*abort_flag) {
                const bool all_visible = t0 + kBN - 1 <= pl.pos_min;  // every key of the tile precedes every probe position
#pragma unroll
                for (int round = 0; round < kAccSet / 64; ++round) {  // 64 accumulator columns of this lane per round, two loads in flight
                    const int mt = round / (kBN / 64), c0 = (round % (kBN / 64)) * 64;
                    uint32_t r0[32], r1[32];
                    const uint32_t ta = tmem_base + ((uint32_t)(lq * 32) << 16) + (uint32_t)(as * kAccSet + mt * kBN + c0);
                    const int tc = t0 + c0;
                    tmem_ld32(ta, r0);
                    tmem_ld32(ta + 32, r1);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (round == kAccSet / 64 - 1) {  // the set's last columns are in registers: hand it back before the arithmetic
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mb_arrive(sm0 + oTEmpty + 8 * as);
                    }
                    if (all_visible && pos_row[mt] >= 0) {
                        float acc1 = 0.f;
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const float u = __uint_as_float(r0[j]), v = __uint_as_float(r1[j]);
                            acc = fmaf(u, u, acc);
                            acc1 = fmaf(v, v, acc1);
                        }
                        acc += acc1;
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const float u = __uint_as_float(r0[j]), v = __uint_as_float(r1[j]);
                            if (tc + j <= pos_row[mt]) acc = fmaf(u, u, acc);
                            if (tc + 32 + j <= pos_row[mt]) acc = fmaf(v, v, acc);
                        }
                    }
                }
            } else {
                __syncwarp();
                if (lane == 0) mb_arrive(sm0 + oTEmpty + 8 * as);
            }
            total += (double)acc;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) total += __shfl_xor_sync(0xFFFFFFFFu, total, o);
        if (lane == 0) reinterpret_cast<double*>(smem + oRed)[lq] = total;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (threadIdx.x == 0) {
        const double* red = reinterpret_cast<const double*>(smem + oRed);
        // part slot of this item inside its unit: (layer, mblock, split); candidate selects the column
        const int slot = (again ? pl.redo_slot0 : pl.slot0) + (layer * pl.mblocks + mblock) * nsplits + split;
        a.part[((int64_t)unit * a.nptiles_max + slot) * 2 + cand] = red[0] + red[1] + red[2] + red[3];
    }
    if (!again || *abort_flag) break;
    done += ntile;
    }
    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);  // let copies and MMAs in flight finish before the memory goes away
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)kTmemCols) : "memory");
    }
}

// A second-moment sum has to be at least this part of the sum of |Q_r|^2 |R_j|^2: a quarter of what independent directions give
// (1 / head_dim).  It is off by up to 3e-7 of that much, so an error that passes is off by about 1e-6.
constexpr double kMomentShare = 1.0 / (4.0 * 128.0);

// Rows [t0, t1) of every operand with the kept entries zeroed: the residual candidate's operand.  grid (blocks, units, operands
// per unit), one 16-byte vector per thread and step.  With second moments (gram part slots) it says which units are done again by
// products, and forms all of their rows.
__global__ void __launch_bounds__(256) drop_rows_kernel(ProbeArgs a, int n_ops, int t0, int t1, int gram) {
    const int unit = a.unit_begin + blockIdx.y;
    if (gram > 0) {
        __shared__ int s_redo;
        if (threadIdx.x < 32) {
            const double* p = a.part + (int64_t)unit * a.nptiles_max * 2;
            const double* m = a.scale + (int64_t)unit * kMaxGramSlots * 2;
            double v[4] = {0.0, 0.0, 0.0, 0.0};
            for (int i = threadIdx.x; i < gram; i += 32) {
                v[0] += p[2 * i]; v[1] += p[2 * i + 1];
                v[2] += m[2 * i]; v[3] += m[2 * i + 1];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int o = 16; o; o >>= 1) v[k] += __shfl_xor_sync(0xFFFFFFFFu, v[k], o);
            // (written so that what is not a number counts as not exact enough)
            const bool fine = v[0] >= kMomentShare * v[2] && v[1] >= kMomentShare * v[3] && isfinite(v[0]) && isfinite(v[1]);
            if (threadIdx.x == 0) {
                s_redo = !fine;
                if (blockIdx.x == 0 && blockIdx.z == 0) a.redo[unit] = !fine;
            }
        }
        __syncthreads();
        if (s_redo) t0 = 0;
    }
    const int64_t op = ((int64_t)unit * n_ops + blockIdx.z) * a.unit_stride;
    const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(a.z1) + op);
    uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.z1drop) + op);
    const uint8_t* bits = reinterpret_cast<const uint8_t*>(a.keep + (int64_t)unit * a.keep_stride);
    for (int64_t v = (int64_t)t0 * 16 + (int64_t)blockIdx.x * 256 + threadIdx.x; v < (int64_t)t1 * 16; v += (int64_t)gridDim.x * 256) {
        dst[v] = drop_kept(src[v], bits[v]);
    }
}

}  // namespace

// How `base` items of `tiles` 256-key tiles are cut: so that the grid fills the machine several times over, but ranges of eight tiles
// or more.
struct Cut {
    int nsplits, per_split;
};
static Cut cut_tiles(int base, int tiles, int sms) {
    if (tiles <= 0) return {0, 0};
    const int n = std::max(1, std::min((4 * sms + base - 1) / base, (tiles + 7) / 8)), per = (tiles + n - 1) / n;
    return {(tiles + per - 1) / per, per};
}
static bool short_items(int items, int per_split, int sms) { return per_split <= kShortItem && items > sms; }

// Whether second moments of the first `tiles` 256-key tiles take less time than their products; both estimated in us, from what the
// parts took.  Products: turns of the device (3.5 us and 0.85 a tile; two blocks per SM 1.5), or the keys' bytes, and the
// residual candidate's copy of the keys.  Moments: a thread block forms every operand's Q^T Q in each segment that it works on (4 us
// per 128 rows, 6 where the queries of all units crowd L2) before its own tiles (1.6, both candidates).  Us a probe call, products of
// all keys against moments:
//   pairs, 512 rows an operand:    2 operands 8k keys 40 and 53; 16 operands 4k 47 and 73, 8k 73 and 77, 16k 130 and 87;
//                                  128 operands 1k 88 and 105, 2k 132 and 123, 32k 1 214 and 428
//   pairs, 2 048 rows an operand:  16 operands 8k 161 and 172, 16k 267 and 191; 128 operands 2k 323 and 366, 3k 419 and 382
//   pairs, 8 rows an operand:      2 operands 8k 44 and 38; 16 operands 3k 43 and 48, 8k 56 and 52
//   blocks of four, 256 rows:      32 operands 4k 51 and 61, 8k 89 and 73; 1 024 rows 8k 184 and 131
static bool moments_pay(const ProbeArgs& a, int tiles, int sms) {
    if (tiles <= 0) return false;
    const int mblocks = (a.G * a.W + 127) / 128, base = a.unit_count * a.B * mblocks * 2;
    const double ops = (double)a.unit_count * (a.B == 4 ? 4 : 1);
    const Cut cut = cut_tiles(base, tiles, sms);
    const bool shorts = short_items(base * cut.nsplits, cut.per_split, sms);
    const double turns = std::ceil((double)base * cut.nsplits / (shorts ? 2 * sms : sms));
    const double tile_bytes = kBN * 256.0, rate = 6e6;  // (bytes per us)
    const double products = std::max(turns * (3.5 + cut.per_split * (shorts ? 1.5 : 0.85)), (double)a.unit_count * a.B * 2 * tiles * tile_bytes / rate) +
                            ops * tiles * 2 * tile_bytes / rate;
    const double qtiles = ((a.B == 4 ? 1 : a.B) * a.G * a.W + 127) / 128, per_op = 2.0 * tiles, all = ops * per_op;
    const double per_block = std::ceil(all / std::min<double>(std::min(sms, kMaxGramCtas), all));
    const double segments = per_block <= 1 ? 1 : 1 + std::ceil((per_block - 1) / per_op);
    const double q_bytes = (double)a.unit_count * a.B * a.G * a.W * 256.0;
    const double moments = 4.0 + segments * qtiles * (q_bytes > 32e6 ? 6.0 : 4.0) + per_block * 1.6;
    return 1.1 * moments < products;
}

cudaError_t launch_probe_tc(const ProbeArgs& a, int dtype, cudaStream_t st, bool* handled, ProbeParts* parts) {
    *handled = false;
    if (dtype != FDKV_BF16 || a.d != 128 || !a.tmap_z1 || !a.tmap_drop) return cudaSuccess;
    static PerDevice once;
    int sm_count = 0;
    cudaError_t e0 = once.ensure([&]() {
        const cudaError_t e = cudaFuncSetAttribute(probe_tc_kernel<3, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, probe_smem(3));
        return e != cudaSuccess ? e : cudaFuncSetAttribute(probe_tc_kernel<1, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, probe_smem(1));
    }, &sm_count);
    if (e0 != cudaSuccess) return e0;
    TcPlan pl;
    pl.pos_min = a.pos_host[0];
    pl.pos_max = a.pos_host[a.W - 1];
    pl.ntiles = pl.pos_max / kBN + 1;  // keys after the last probe position never count
    // keys that every probe query sees: second moments (one read of Z1 and 2 x 2 x 128 x 128 flops per key, against a second
    // copy of Z1 and 2 x 2 x rows x 128 flops here; 32 layers of 32k tokens, 512 rows per pair: 1 190 -> 428 us with this
    // kernel's share of the last keys)
    pl.tile_first = (pl.pos_min + 1) / kBN;
    if (a.moments == 0 ? !moments_pay(a, pl.tile_first, sm_count) : a.moments == 2) pl.tile_first = 0;
    pl.slot0 = 0;
    if (pl.tile_first > 0) {
        cudaError_t e = launch_probe_gram(a, pl.tile_first * kBN, st, &pl.slot0);
        if (e != cudaSuccess) return e;
    }
    const int ntiles = pl.ntiles - pl.tile_first;
    pl.mblocks = (a.G * a.W + 128 * kMT - 1) / (128 * kMT);
    const Cut cut = cut_tiles(a.unit_count * a.B * pl.mblocks * 2, ntiles, sm_count);
    const int nsplits = cut.nsplits;
    pl.tiles_per_split = cut.per_split;
    pl.nsplits = nsplits;
    pl.items_per_unit = a.B * pl.mblocks * 2 * nsplits;
    pl.sure_items = a.unit_count * pl.items_per_unit;
    // units to do again: ranges of eight tiles as above, by as many blocks as run at one time
    const bool shorts = short_items(pl.sure_items, pl.tiles_per_split, sm_count);
    const int redo_blocks = pl.tile_first > 0 ? (shorts ? 2 : 1) * sm_count : 0;
    pl.redo_nsplits = (pl.tile_first + 7) / 8;
    pl.redo_tiles_per_split = 8;
    pl.redo_per_unit = a.B * pl.mblocks * 2 * pl.redo_nsplits;
    pl.redo_slot0 = pl.slot0 + a.B * pl.mblocks * nsplits;
    const int slots = pl.redo_slot0 + a.B * pl.mblocks * pl.redo_nsplits;
    if (slots > a.nptiles_max) return cudaErrorInvalidValue;  // cannot happen: the part array is sized for all of them
    if (pl.sure_items + redo_blocks > 0) {
        const int t0 = pl.tile_first * kBN, t1 = std::min(a.T, pl.ntiles * kBN), n_ops = a.B == 4 ? 4 : 1;
        const int blocks = (int)std::min<int64_t>(64, ((int64_t)std::max(t1 - t0, 1) * 16 + 255) / 256);
        drop_rows_kernel<<<dim3(blocks, a.unit_count, n_ops), 256, 0, st>>>(a, n_ops, t0, t1, pl.slot0);
        const CUtensorMap &mz = *reinterpret_cast<const CUtensorMap*>(a.tmap_z1), &md = *reinterpret_cast<const CUtensorMap*>(a.tmap_drop);
        if (shorts) probe_tc_kernel<1, 1><<<pl.sure_items + redo_blocks, kPThreads, probe_smem(1), st>>>(mz, md, a, pl);
        else probe_tc_kernel<3, 2><<<pl.sure_items + redo_blocks, kPThreads, probe_smem(3), st>>>(mz, md, a, pl);
        count_launch(2);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    count_kernel(FDKV_KERNEL_PROBE_TC);
    *parts = {pl.slot0, pl.redo_slot0, slots};
    *handled = true;
    return cudaSuccess;
}

}  // namespace fdkv
