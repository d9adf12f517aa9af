// Token-granular sparse residual (the paper's rule, Method between Eq. 2 and Eq. 3).  The tensor-core kernels below
// serve bf16 storage with head_dim 128; other storage types and head dimensions take token_score_tile_kernel, a plain
// float32 product, and the same selection.
//
//   s_t = max over (layer of the depth block, group query head, probe query q with pos[q] >= t) | Q_l . (K_l[t,:] - Khat_l^shared[t,:]) |
//       = | Q_l . (+-c Z1K[t,:]) | for a pair, | Q_l . dev_l[t,:] | for a block of four (dev_l = layer l's deviation from the block mean);
//   keep the k_tok tokens with the largest s_t (ties: lowest t); they keep all 128 high-frequency values of K and of V
//   (of every layer of a block of four).
//
// 1. token_score_kernel (tcgen05): the transposed probe product D[token][probe row] = Z1K . Q^T, so that a thread
//    of the epilogue owns one token (TMEM lane) and takes the maximum over its row's columns in registers.  A = 128
//    tokens of Z1K per tile (TMA ring, shared memory), B = the item's Q rows (64, 128 or 256 of them; shared memory, the next
//    item's in a second buffer), M = 128, N = 64, 128 or 256, K = 16, two accumulator sets of N TMEM columns.  Items of the two layers / row blocks of a
//    unit merge with atomicMax on the (non-negative) float bit patterns, which is order-independent.
//    The same registers give Eq. 2's errors: the token's sum of D^2 over the rows that see it, one float per item.  Shared
//    drops every token's high-frequency row, residual every unselected one's, so both errors are sums of these numbers
//    and the probe needs no second product (it was two more passes over T x rows x 128, and a copy of Z1K with the
//    selected rows zeroed to run one of them on: 8 191 tokens, 8 blocks of four: the probe 627 -> 250 us).
// 2. token_select_kernel: per unit an MSB-first radix select (12, 12 and 7 bits) of the k_tok-th largest score and an
//    index-ordered compaction: ascending token list, per-16-token-slice counts, and the two error sums in float64.
// (The commit step forms the selected rows from the caller's K and V: token_gather_kernel in compress.cu.)
#include <algorithm>
#include <cstdlib>

#include "fdkv_internal.h"
#include "umma.cuh"

namespace fdkv {

namespace {

constexpr int kTM = 128;                    // tokens per tile (M of the MMA)
constexpr int kTN = 256;                    // probe rows per item (N of the MMA) at most
constexpr int kTStages = 3;
constexpr int kTAHalf = kTM * 128;          // one 64-channel half of a token tile: 16 KiB
constexpr int kTAStage = 2 * kTAHalf;       // 32 KiB
constexpr int kTHdr = 2048;                 // barriers, TMEM slot, abort flag, the epilogue's exchange
constexpr int kTThreads = 20 * 32;          // copies, MMAs, probe rows, one idle, sixteen of the epilogue
constexpr int tFull = 0, tEmpty = 32, tTFull = 64, tTEmpty = 80, tSlot = 96, tAbort = 100, tBFull = 112, tBEmpty = 128, tExch = 256;
constexpr int score_smem(int nt) { return kTHdr + 2 * nt * 256 + kTStages * kTAStage; }
static_assert(score_smem(kTN) <= 227 * 1024, "shared memory budget");

// The product of all items' tiles: item = (unit, layer, block of NT probe rows), ntiles tiles each; block b of the grid takes the
// tiles [total b / blocks, total (b + 1) / blocks) of them.
struct ScorePlan {
    int mblocks, ntiles, total, pos_min;
};

// NT: probe rows per item (64, 128 or 256: the smallest that holds a layer's rows, so that few probe rows do not pay for 256).
// One persistent block per SM.  Warp 0 streams the token tiles, warp 2 the probe rows of the next item into the other of two
// buffers, one thread of warp 1 issues the MMAs, sixteen warps take the results: four per quarter of the TMEM lanes, a fourth of the columns
// each (64 rows: two, a half).  Bound by the hand-overs between copies, MMAs (1 024 cycles a tile of 128 x 256 x 128) and epilogue: 8 191 tokens, 8
// blocks of four, 8 heads, 256 rows a layer: four epilogue warps, and a block per item and third of its tiles, each with its own probe
// rows, the last of six waves a fifth full, 214 us; eight warps 165; sixteen 159 (117 without an epilogue).
// Tiles that some query does not see take a comparison per column, with the query that the column is for and the token's first one (probe call of
// 8 191 tokens, 8 layers in blocks of four, 64 positions all over the prompt: 135 us; with a division and a load per column 363; the last 64
// positions 98).
template <int NT>
__global__ void __launch_bounds__(kTThreads, 1)
token_score_kernel(const __grid_constant__ CUtensorMap tmap, TokenArgs a, ScorePlan pl) {
    constexpr uint32_t kIdesc = umma_idesc(kTM, NT, false);
    constexpr int kBHalf = NT * 128, kBBytes = 2 * kBHalf;  // one 64-channel half of the probe rows, both
    constexpr uint32_t kCols = 2 * NT;                      // TMEM columns: two accumulators
    constexpr int kParts = NT >= 128 ? 4 : 2;               // epilogue warps that share a lane's columns
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sm0 = s_u32(smem);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + tAbort);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (sm0 & 1023u) {
        if (threadIdx.x == 0) atomicMax(a.status, (int32_t)kFlagCountMismatch);
        return;
    }
    const int g_begin = (int)((int64_t)pl.total * blockIdx.x / gridDim.x), g_end = (int)((int64_t)pl.total * (blockIdx.x + 1) / gridDim.x);
    const int rows_layer = a.G * a.W;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kTStages; ++s) { mb_init(sm0 + tFull + 8 * s, 1); mb_init(sm0 + tEmpty + 8 * s, 1); }
        for (int s = 0; s < 2; ++s) {
            mb_init(sm0 + tTFull + 8 * s, 1); mb_init(sm0 + tTEmpty + 8 * s, 4 * kParts);
            mb_init(sm0 + tBFull + 8 * s, 1); mb_init(sm0 + tBEmpty + 8 * s, 1);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm0 + tSlot), "r"(kCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(smem + tSlot);
    const uint32_t b_base = sm0 + kTHdr, a_base = b_base + 2 * kBBytes;
    // every role walks the block's items: f(its number here, unit, layer, row block, first tile, tiles, number of the first tile here)
    auto items = [&](auto&& f) {
        for (int g = g_begin, seg = 0; g < g_end; ++seg) {
            const int item = g / pl.ntiles, t0 = g - item * pl.ntiles, n = min(pl.ntiles - t0, g_end - g);
            const int mblock = item % pl.mblocks, ul = item / pl.mblocks;
            f(seg, a.unit_begin + ul / a.B, ul % a.B, mblock, t0, n, g - g_begin);
            g += n;
        }
    };

    if (warp == 0) {
        if (lane == 0)
            items([&](int, int unit, int layer, int, int t0, int n, int i0) {
                // K high-frequency rows of the unit (a block of four stages one operand per layer)
                const int64_t row0 = a.B == 4 ? ((int64_t)unit * 4 + layer) * a.Tmax : (int64_t)unit * a.Tmax;
                for (int i = i0; i < i0 + n; ++i) {
                    const int s = i % kTStages;
                    mb_wait(sm0 + tEmpty + 8 * s, ((uint32_t)(i / kTStages) & 1u) ^ 1u, abort_flag, a.status);
                    if (*abort_flag) break;
                    const uint32_t full = sm0 + tFull + 8 * s, dst = a_base + s * kTAStage;
                    const int y = (int)(row0 + (int64_t)(t0 + i - i0) * kTM);
                    mb_expect_tx(full, kTAStage);
                    tma_2d(dst, &tmap, 0, y, full);
                    tma_2d(dst + kTAHalf, &tmap, 64, y, full);
                }
            });
    } else if (warp == 1) {
        if (lane == 0)
            items([&](int seg, int, int, int, int, int n, int i0) {
                const int bs = seg & 1;
                const uint64_t db0 = smem_desc(b_base + bs * kBBytes);
                mb_wait(sm0 + tBFull + 8 * bs, ((uint32_t)seg >> 1) & 1u, abort_flag, a.status);
                for (int i = i0; i < i0 + n; ++i) {
                    const int s = i % kTStages, as = i & 1;
                    mb_wait(sm0 + tTEmpty + 8 * as, (((uint32_t)i >> 1) & 1u) ^ 1u, abort_flag, a.status);
                    mb_wait(sm0 + tFull + 8 * s, (uint32_t)(i / kTStages) & 1u, abort_flag, a.status);
                    if (*abort_flag) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t da0 = smem_desc(a_base + s * kTAStage);
                    const uint32_t d_tmem = tmem_base + (uint32_t)(as * NT);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const uint64_t da = da0 + (uint64_t)(((k >> 2) * kTAHalf + (k & 3) * 32) >> 4);
                        const uint64_t db = db0 + (uint64_t)(((k >> 2) * kBHalf + (k & 3) * 32) >> 4);
                        umma_ss<kIdesc>(d_tmem, da, db, k > 0);
                    }
                    umma_commit(sm0 + tEmpty + 8 * s);
                    umma_commit(sm0 + tTFull + 8 * as);
                }
                if (!*abort_flag) umma_commit(sm0 + tBEmpty + 8 * bs);
            });
    } else if (warp == 2) {
        // probe rows r = mblock * NT + i of the layer, r = g*W + qi -> Q[layer][qi][h*G+g][:]; padding rows zero
        items([&](int seg, int unit, int layer, int mblock, int, int, int) {
            const int bs = seg & 1, h = unit % a.Hkv, pair = unit / a.Hkv;
            mb_wait(sm0 + tBEmpty + 8 * bs, (((uint32_t)seg >> 1) & 1u) ^ 1u, abort_flag, a.status);
            const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(a.q_layers_dev[a.B * pair + layer]);
            const int chunk = lane & 15;
#pragma unroll 4
            for (int i = lane >> 4; i < NT; i += 2) {
                const int r = mblock * NT + i;
                const uint32_t dst = b_base + bs * kBBytes + (chunk >> 3) * kBHalf + i * 128 + (((chunk & 7) ^ (i & 7)) << 4);
                if (r < rows_layer) {
                    const int g = r / a.W;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(q + ((int64_t)(r - g * a.W) * a.Hq + h * a.G + g) * 128 + chunk * 8)
                                 : "memory");
                } else {
                    asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(dst), "r"(0u) : "memory");
                }
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mb_arrive(sm0 + tBFull + 8 * bs);
        });
    } else if (warp >= 4 && warp < 4 + 4 * kParts) {
        // ---- epilogue: lane = token (TMEM lane); maximum of |D| and sum of D^2 over the probe rows that see the token ----
        const int lq = warp & 3, part = (warp - 4) >> 2;
        constexpr int kPart = NT / kParts;  // columns of a warp: 32 or 64
        float* const exch = reinterpret_cast<float*>(smem + tExch) + lq * 32 + lane;  // [kParts - 1][128] sums
        const float c32 = a.B == 4 ? 1.f : __uint_as_float(0x3F3504F3u);  // a pair's rows are Z1: K - Khat^shared = +-c Z1
        items([&](int, int unit, int layer, int mblock, int t0, int n, int i0) {
            float* const err = a.err + ((int64_t)unit * a.nslots + layer * pl.mblocks + mblock) * a.Tmax;
            uint32_t* const score = a.score + (int64_t)unit * a.Tmax;
            const int row0 = mblock * NT + part * kPart;  // probe row of the warp's first column
            for (int i = i0; i < i0 + n; ++i) {
                const int as = i & 1, tile_t0 = (t0 + i - i0) * kTM;
                const int t = tile_t0 + lq * 32 + lane;
                // First query that sees the token: the positions ascend, so it is the number of those before it.  All of them are looked at,
                // four a lane: those before the warp's 32 tokens are counted, those among them set a bit.
                int q_seen = 0;
                if (tile_t0 + kTM - 1 > pl.pos_min) {
                    uint32_t inside = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int rel = 32 * k + lane < a.W ? a.pos[32 * k + lane] - (t - lane) : 32;
                        q_seen += __popc(__ballot_sync(0xFFFFFFFFu, rel < 0));
                        if (rel >= 0 && rel < 32) inside |= 1u << rel;
                    }
                    q_seen += __popc(__reduce_or_sync(0xFFFFFFFFu, inside) & ((1u << lane) - 1u));
                }
                mb_wait(sm0 + tTFull + 8 * as, ((uint32_t)i >> 1) & 1u, abort_flag, a.status);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                float m0 = 0.f, m1 = 0.f, e0 = 0.f, e1 = 0.f;
                if (!*abort_flag) {
                    uint32_t r[kPart / 32][32];
                    const uint32_t ta = tmem_base + ((uint32_t)(lq * 32) << 16) + (uint32_t)(as * NT + part * kPart);
#pragma unroll
                    for (int p = 0; p < kPart / 32; ++p) tmem_ld32(ta + 32 * p, r[p]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    // read: the next product may take the accumulator
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mb_arrive(sm0 + tTEmpty + 8 * as);
                    if (tile_t0 + kTM - 1 <= pl.pos_min) {  // every row sees every token
#pragma unroll
                        for (int p = 0; p < kPart / 32; ++p)
#pragma unroll
                            for (int j = 0; j < 32; j += 4) {
                                const float u = __uint_as_float(r[p][j]), v = __uint_as_float(r[p][j + 1]);
                                const float w = __uint_as_float(r[p][j + 2]), x = __uint_as_float(r[p][j + 3]);
                                m0 = fmaxf(m0, fmaxf(fabsf(u), fabsf(v)));
                                m1 = fmaxf(m1, fmaxf(fabsf(w), fabsf(x)));
                                e0 = fmaf(u, u, e0);
                                e1 = fmaf(v, v, e1);
                                e0 = fmaf(w, w, e0);
                                e1 = fmaf(x, x, e1);
                            }
                    } else {
                        int q = row0 % a.W;  // (the columns go through the queries, head after head)
#pragma unroll
                        for (int p = 0; p < kPart / 32; ++p)
#pragma unroll
                            for (int j = 0; j < 32; ++j) {
                                const float u = __uint_as_float(r[p][j]);
                                if (q >= q_seen && row0 + 32 * p + j < rows_layer) {
                                    if (j & 2) m1 = fmaxf(m1, fabsf(u)); else m0 = fmaxf(m0, fabsf(u));
                                    if (j & 1) e1 = fmaf(u, u, e1); else e0 = fmaf(u, u, e0);
                                }
                                q = q + 1 == a.W ? 0 : q + 1;
                            }
                    }
                    const float m = fmaxf(m0, m1);
                    if (t < a.T && m > 0.f) atomicMax(score + t, __float_as_uint(m * c32));
                }
                // The parts' sums in their order: written behind the barrier that says that part 0 has read those of the tile before (not of
                // the first), read behind the one that says that all are there.
                const float e = e0 + e1;
                if (part > 0) {
                    if (i > 0) asm volatile("bar.sync %0, %1;" ::"r"(5 + lq), "n"(32 * kParts) : "memory");
                    exch[128 * (part - 1)] = e;
                }
                asm volatile("bar.sync %0, %1;" ::"r"(1 + lq), "n"(32 * kParts) : "memory");
                if (part == 0) {
                    float sum = e;
#pragma unroll
                    for (int p = 0; p < kParts - 1; ++p) sum += exch[128 * p];
                    if (t < a.T && !*abort_flag) err[t] = sum;
                    if (g_begin + i + 1 < g_end) asm volatile("bar.arrive %0, %1;" ::"r"(5 + lq), "n"(32 * kParts) : "memory");
                }
            }
        });
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kCols) : "memory");
}

constexpr int kSelThreads = 1024, kSelBins = 4096;

// exclusive sum over the block of a value per thread, and the total; s_warp: 32 words
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* s_warp, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += x;
    }
    __syncthreads();  // s_warp may still be read from the previous call
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t w = s_warp[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, w, o);
        if (lane >= o) w += x;
    }
    *total = __shfl_sync(0xFFFFFFFFu, w, 31);
    const uint32_t before = __shfl_sync(0xFFFFFFFFu, w, (warp + 31) & 31);
    return (warp ? before : 0u) + incl - v;
}

// One CTA per unit: threshold of the k-th largest score (32-bit patterns of non-negative floats order like the
// floats; three digits of 12, 12 and 7 bits: the first has 16 bins per octave, on which a warp's atomics seldom collide), then
// the ascending list of kept tokens (score above the threshold, or equal and among the first `need` such tokens), the number of kept
// tokens before every 16-token slice, and the unit's two error sums: all tokens' (shared) and the unselected ones' (residual),
// float64 over the score kernel's per-token sums in a fixed order.  Bound by the chain of its steps: with digits of 8 bits, found by
// one thread, and a scan of flags and one of ranks for every 1 024 tokens, 8 191 tokens took 46 us, now 15.
__global__ void __launch_bounds__(kSelThreads) token_select_kernel(TokenArgs a) {
    __shared__ __align__(16) uint32_t s_hist[kSelBins];
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_digit, s_above;
    const int unit = a.unit_begin + blockIdx.x, tid = threadIdx.x;
    const uint32_t* key = a.score + (int64_t)unit * a.Tmax;
    const float* err = a.err + (int64_t)unit * a.nslots * a.Tmax;
    int32_t* list = a.list + (int64_t)unit * a.ktok_cap;
    int32_t* off = a.off + (int64_t)unit * (a.ntiles_max + 1);
    const int T = a.T;
    const int nslice = (T + kResTile - 1) / kResTile;
    uint32_t tau = 0xFFFFFFFFu, need = 0;
    if (a.k_tok > 0) {
        uint32_t prefix = 0, left = (uint32_t)a.k_tok;
#pragma unroll 1
        for (int pass = 0; pass < 3; ++pass) {
            const int shift = pass == 0 ? 19 : pass == 1 ? 7 : 0, bits = pass == 2 ? 7 : 12;
            *reinterpret_cast<uint4*>(&s_hist[4 * tid]) = make_uint4(0u, 0u, 0u, 0u);
            __syncthreads();
#pragma unroll 4
            for (int t = tid; t < T; t += kSelThreads) {
                const uint32_t k = key[t];
                if (pass == 0 || (k >> (shift + bits)) == prefix) atomicAdd(&s_hist[(k >> shift) & ((1u << bits) - 1u)], 1u);
            }
            __syncthreads();
            // the bin, from the top, in which the running count reaches `left`: four bins per thread, the largest first
            const uint4 v = *reinterpret_cast<const uint4*>(&s_hist[kSelBins - 4 - 4 * tid]);
            const uint32_t c[4] = {v.w, v.z, v.y, v.x};
            uint32_t total, before = block_excl_scan(c[0] + c[1] + c[2] + c[3], s_warp, &total);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (before < left && left <= before + c[i]) { s_digit = (uint32_t)(kSelBins - 1 - 4 * tid - i); s_above = before; }
                before += c[i];
            }
            __syncthreads();
            prefix = prefix << bits | s_digit;
            left -= s_above;
        }
        tau = prefix;
        need = left;
    }
    // ordered compaction: eight consecutive tokens per thread and round, counts of those above in the high half, equal in the low
    uint32_t base_gt = 0, base_eq = 0;
    double sum_all = 0.0, sum_dropped = 0.0;
    const int seen = min(T, a.pos_last + 1);  // later tokens are seen by no probe query: no error, nothing was written
    for (int t0 = 0; t0 < T; t0 += 8 * kSelThreads) {
        const int t8 = t0 + 8 * tid;
        uint32_t gt = 0, eq = 0;
        if (a.k_tok > 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t k = t8 + i < T ? key[t8 + i] : 0u;
                gt |= (uint32_t)(t8 + i < T && k > tau) << i;
                eq |= (uint32_t)(t8 + i < T && k == tau) << i;
            }
        }
        uint32_t total;
        const uint32_t before = block_excl_scan((uint32_t)__popc(gt) << 16 | (uint32_t)__popc(eq), s_warp, &total);
        const uint32_t eq_before = base_eq + (before & 0xFFFFu);
        uint32_t at = base_gt + (before >> 16) + min(eq_before, need);
        const int ties = (int)min((uint32_t)__popc(eq), need - min(eq_before, need));  // of the thread's, the first
        uint32_t kept = gt, rest = eq;
        for (int i = 0; i < ties; ++i) {
            kept |= rest & (0u - rest);
            rest &= rest - 1;
        }
        if (t8 < T && (t8 & (kResTile - 1)) == 0) off[t8 / kResTile] = (int32_t)at;
        for (uint32_t b = kept; b; b &= b - 1) list[at++] = t8 + __ffs((int)b) - 1;
        double e[8] = {};
        for (int j = 0; j < a.nslots; ++j)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (t8 + i < seen) e[i] += (double)err[(int64_t)j * a.Tmax + t8 + i];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            sum_all += e[i];
            if (!(kept >> i & 1u)) sum_dropped += e[i];
        }
        base_gt += total >> 16;
        base_eq += total & 0xFFFFu;
    }
    __shared__ double s_err[2][32];
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        sum_all += __shfl_xor_sync(0xFFFFFFFFu, sum_all, o);
        sum_dropped += __shfl_xor_sync(0xFFFFFFFFu, sum_dropped, o);
    }
    if ((tid & 31) == 0) { s_err[0][tid >> 5] = sum_all; s_err[1][tid >> 5] = sum_dropped; }
    __syncthreads();
    if (tid < 2) {
        double e = 0.0;
        for (int w = 0; w < 32; ++w) e += s_err[tid][w];
        a.part[(int64_t)unit * a.nptiles_max * 2 + tid] = e;
    }
    if (tid == 0) {
        const uint32_t kept = base_gt + min(base_eq, need);
        off[nslice] = (int32_t)kept;
        if ((int64_t)kept != a.k_tok) atomicMax(a.status, (int32_t)kFlagCountMismatch);
    }
}

// ---- storage types and head dimensions without the tensor-core kernel: the same score as a float32 product ----
template <typename T>
__device__ __forceinline__ float to_f32(T x);
template <>
__device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

constexpr int kSTile = 64;   // tokens per thread block
constexpr int kSRows = 16;   // probe rows staged per round
// grid (64-token tiles, units), 256 threads: thread (token j, row group rg) takes the maximum of |q_r . z[t]| and the sum of
// its square over the rows r of its group whose probe position sees token t; the groups' maxima merge by atomicMax on
// the bit patterns of the non-negative floats, their sums through shared memory.
template <typename T>
__global__ void __launch_bounds__(256) token_score_tile_kernel(TokenArgs a, int d) {
    extern __shared__ float ssm[];
    const int ld = d + 1;
    float* zs = ssm;                 // [64][d + 1]
    float* qs = zs + kSTile * ld;    // [16][d]
    const int unit = a.unit_begin + blockIdx.y;
    const int t0 = blockIdx.x * kSTile;
    const int nt = min(kSTile, a.T - t0);
    const int h = unit % a.Hkv, pair = unit / a.Hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j = (warp & 1) * 32 + lane, rg = warp >> 1;
    const int n_ops = a.B == 4 ? 4 : 1;
    const int M = (a.B == 4 ? 1 : 2) * a.G * a.W;  // probe rows per operand
    float best = 0.f, esum = 0.f;
    for (int op = 0; op < n_ops; ++op) {
        const T* z1 = reinterpret_cast<const T*>(a.z1) + ((int64_t)unit * n_ops + op) * a.unit_stride + (int64_t)t0 * d;
        for (int i = threadIdx.x; i < kSTile * d; i += blockDim.x) {
            const int t = i / d, c = i % d;
            zs[t * ld + c] = t < nt ? to_f32<T>(z1[i]) : 0.f;
        }
        __syncthreads();
        for (int rb = 0; rb < M; rb += kSRows) {
            for (int i = threadIdx.x; i < kSRows * d; i += blockDim.x) {
                const int r = rb + i / d, c = i % d;
                float v = 0.f;
                if (r < M) {
                    const int layer = a.B == 4 ? op : r / (a.G * a.W), g = (r / a.W) % a.G, qi = r % a.W;
                    const T* q = reinterpret_cast<const T*>(a.q_layers_dev[a.B * pair + layer]);
                    v = to_f32<T>(q[((int64_t)qi * a.Hq + h * a.G + g) * d + c]);
                }
                qs[i] = v;
            }
            __syncthreads();
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            const float* zr = zs + j * ld;
            const float* qr = qs + rg * 4 * d;
            for (int c = 0; c < d; ++c) {
                const float zv = zr[c];
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i] = fmaf(qr[i * d + c], zv, acc[i]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = rb + rg * 4 + i;
                if (r < M && j < nt && t0 + j <= a.pos[r % a.W]) {
                    best = fmaxf(best, fabsf(acc[i]));
                    esum = fmaf(acc[i], acc[i], esum);
                }
            }
            __syncthreads();
        }
    }
    float* const s_e = qs;  // [4][64]: the row groups' sums (every product is done: the loop ends on a barrier)
    s_e[rg * kSTile + j] = esum;
    __syncthreads();
    if (rg == 0 && j < nt) a.err[(int64_t)unit * a.nslots * a.Tmax + t0 + j] = (s_e[j] + s_e[kSTile + j]) + (s_e[2 * kSTile + j] + s_e[3 * kSTile + j]);
    // the score carries the factor of Eq. 1's inverse (c for a pair; a block of four's deviations are in layer space already)
    if (j < nt) atomicMax(a.score + (int64_t)unit * a.Tmax + t0 + j, __float_as_uint(best * (a.B == 4 ? 1.f : __uint_as_float(0x3F3504F3u))));
}

}  // namespace

cudaError_t launch_token_select(const TokenArgs& a, int dtype, int d, bool tensor_core, cudaStream_t st) {
    if (a.unit_count <= 0) return cudaSuccess;
    static PerDevice once;
    int sm_count = 0;
    const size_t tile_smem = (size_t)(kSTile * (d + 1) + kSRows * d) * sizeof(float);
    cudaError_t e0 = once.ensure([&]() {
        cudaError_t e1 = cudaFuncSetAttribute(token_score_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, score_smem(64));
        if (e1 == cudaSuccess) e1 = cudaFuncSetAttribute(token_score_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, score_smem(128));
        if (e1 == cudaSuccess) e1 = cudaFuncSetAttribute(token_score_kernel<kTN>, cudaFuncAttributeMaxDynamicSharedMemorySize, score_smem(kTN));
        if (e1 == cudaSuccess) e1 = cudaFuncSetAttribute(token_score_tile_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
        if (e1 == cudaSuccess) e1 = cudaFuncSetAttribute(token_score_tile_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
        return e1;
    }, &sm_count);
    if (e0 != cudaSuccess) return e0;
    cudaError_t e = cudaMemsetAsync(a.score + (int64_t)a.unit_begin * a.Tmax, 0, (size_t)a.unit_count * a.Tmax * 4, st);
    if (e != cudaSuccess) return e;
    if (!tensor_core) {
        // tokens after the last probe position are seen by nobody: score 0
        const int ntiles = std::min(a.T - 1, a.pos_host[a.W - 1]) / kSTile + 1;
        if (dtype == FDKV_BF16)
            token_score_tile_kernel<__nv_bfloat16><<<dim3(ntiles, a.unit_count), 256, tile_smem, st>>>(a, d);
        else
            token_score_tile_kernel<float><<<dim3(ntiles, a.unit_count), 256, tile_smem, st>>>(a, d);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        token_select_kernel<<<a.unit_count, kSelThreads, 0, st>>>(a);
        count_launch(2);
        count_kernel(FDKV_KERNEL_PROBE_PORTABLE);
        return cudaGetLastError();
    }
    ScorePlan pl;
    pl.pos_min = a.pos_host[0];
    pl.ntiles = a.pos_host[a.W - 1] / kTM + 1;  // tokens after the last probe position are seen by nobody: score 0
    pl.mblocks = (a.G * a.W + kTN - 1) / kTN;   // (a.nslots = B x mblocks)
    const int64_t total = (int64_t)a.unit_count * a.B * pl.mblocks * pl.ntiles;
    if (total > 0x7FFFFFFF) return cudaErrorInvalidValue;  // cannot happen: units x tokens are in memory
    pl.total = (int)total;
    auto score = [&](auto* kernel, int smem) {  // (blocks of fewer than four tiles would wait for their probe rows most of the time)
        kernel<<<(int)std::min<int64_t>(sm_count, (total + 3) / 4), kTThreads, smem, st>>>(*reinterpret_cast<const CUtensorMap*>(a.tmap_z1_128), a, pl);
    };
    if (a.G * a.W <= 64) score(token_score_kernel<64>, score_smem(64));
    else if (a.G * a.W <= 128) score(token_score_kernel<128>, score_smem(128));
    else score(token_score_kernel<kTN>, score_smem(kTN));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    token_select_kernel<<<a.unit_count, kSelThreads, 0, st>>>(a);
    count_launch(2);
    count_kernel(FDKV_KERNEL_TOKEN_SCORE);
    count_kernel(FDKV_KERNEL_PROBE_TC);  // (it is the probe's product too)
    return cudaGetLastError();
}

}  // namespace fdkv
