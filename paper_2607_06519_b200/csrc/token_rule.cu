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
//    tokens of Z1K per tile (TMA ring, shared memory), B = the item's 256 Q rows (shared memory, resident),
//    M = 128, N = 256, K = 16, two accumulator sets of 256 TMEM columns.  Items of the two layers / row blocks of a
//    unit merge with atomicMax on the (non-negative) float bit patterns, which is order-independent.
//    The same registers give Eq. 2's errors: the token's sum of D^2 over the rows that see it, one float per item.  Shared
//    drops every token's high-frequency row, residual every unselected one's, so both errors are sums of these numbers
//    and the probe needs no second product (it was two more passes over T x rows x 128, and a copy of Z1K with the
//    selected rows zeroed to run one of them on: 8 191 tokens, 8 blocks of four: the probe 627 -> 250 us).
// 2. token_select_kernel: per unit an MSB-first radix select (4 x 8 bits) of the k_tok-th largest score and an
//    index-ordered compaction: ascending token list, per-16-token-slice counts, and the two error sums in float64.
// (The commit step forms the selected rows from the caller's K and V: token_gather_kernel in compress.cu.)
#include <algorithm>
#include <cstdlib>

#include "fdkv_internal.h"
#include "umma.cuh"

namespace fdkv {

namespace {

constexpr int kTM = 128;                    // tokens per tile (M of the MMA)
constexpr int kTN = 256;                    // probe rows per item (N of the MMA)
constexpr int kTStages = 4;
constexpr int kTAHalf = kTM * 128;          // one 64-channel half of a token tile: 16 KiB
constexpr int kTAStage = 2 * kTAHalf;       // 32 KiB
constexpr int kTBHalf = kTN * 128;          // one 64-channel half of the Q block: 32 KiB
constexpr int kTBBytes = 2 * kTBHalf;       // 64 KiB
constexpr int kTHdr = 2048;                 // barriers, TMEM slot, abort flag, probe position of every column
constexpr int kTSmem = kTHdr + kTBBytes + kTStages * kTAStage;  // 194 KiB
constexpr int kTThreads = 6 * 32;
constexpr uint32_t kTIdesc = umma_idesc(kTM, kTN, false);
constexpr int tFull = 0, tEmpty = 32, tTFull = 64, tTEmpty = 80, tSlot = 96, tAbort = 100, tPosCol = 1024;  // pos_col: 256 ints


struct ScorePlan {
    int items_per_unit, mblocks, nsplits, ntiles, tiles_per_split, pos_min;
};

__global__ void __launch_bounds__(kTThreads, 1)
token_score_kernel(const __grid_constant__ CUtensorMap tmap, TokenArgs a, ScorePlan pl) {
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sm0 = s_u32(smem);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + tAbort);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (sm0 & 1023u) {
        if (threadIdx.x == 0) atomicMax(a.status, (int32_t)kFlagCountMismatch);
        return;
    }
    int it = blockIdx.x;
    const int unit = a.unit_begin + it / pl.items_per_unit;
    it %= pl.items_per_unit;
    const int split = it % pl.nsplits; it /= pl.nsplits;
    const int mblock = it % pl.mblocks; it /= pl.mblocks;
    const int layer = it;
    const int h = unit % a.Hkv, pair = unit / a.Hkv;
    const int tile0 = split * pl.tiles_per_split;
    const int ntile = max(0, min(pl.ntiles, tile0 + pl.tiles_per_split) - tile0);
    const int rows_layer = a.G * a.W;
    int* const pos_col = reinterpret_cast<int*>(smem + tPosCol);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kTStages; ++s) { mb_init(sm0 + tFull + 8 * s, 1); mb_init(sm0 + tEmpty + 8 * s, 1); }
        for (int s = 0; s < 2; ++s) { mb_init(sm0 + tTFull + 8 * s, 1); mb_init(sm0 + tTEmpty + 8 * s, 4); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // ---- B: probe rows r = mblock*256 + i of this layer, r = g*W + qi -> Q[layer][qi][h*G+g][:]; padding rows zero ----
    {
        const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(a.q_layers_dev[a.B * pair + layer]);
        for (int v = threadIdx.x; v < kTN * 16; v += kTThreads) {
            const int i = v >> 4, chunk = v & 15;
            const int r = mblock * kTN + i;
            uint4 val = make_uint4(0u, 0u, 0u, 0u);
            if (r < rows_layer)
                val = *reinterpret_cast<const uint4*>(q + ((int64_t)(r % a.W) * a.Hq + h * a.G + r / a.W) * 128 + chunk * 8);
            *reinterpret_cast<uint4*>(smem + kTHdr + (chunk >> 3) * kTBHalf + i * 128 + (((chunk & 7) ^ (i & 7)) << 4)) = val;
        }
        for (int i = threadIdx.x; i < kTN; i += kTThreads) {
            const int r = mblock * kTN + i;
            pos_col[i] = r < rows_layer ? a.pos[r % a.W] : -1;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm0 + tSlot), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(smem + tSlot);
    const uint32_t b_base = sm0 + kTHdr, a_base = b_base + kTBBytes;

    if (warp == 0) {
        if (lane == 0) {
            // K high-frequency rows of the unit (a block of four stages one operand per layer)
            const int64_t row0 = a.B == 4 ? ((int64_t)unit * 4 + layer) * a.Tmax : (int64_t)unit * a.Tmax;
            for (int i = 0; i < ntile; ++i) {
                const int s = i % kTStages;
                mb_wait(sm0 + tEmpty + 8 * s, ((uint32_t)(i / kTStages) & 1u) ^ 1u, abort_flag, a.status);
                if (*abort_flag) break;
                const uint32_t full = sm0 + tFull + 8 * s, dst = a_base + s * kTAStage;
                const int y = (int)(row0 + (int64_t)(tile0 + i) * kTM);
                mb_expect_tx(full, kTAStage);
                tma_2d(dst, &tmap, 0, y, full);
                tma_2d(dst + kTAHalf, &tmap, 64, y, full);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint64_t db0 = smem_desc(b_base);
            for (int i = 0; i < ntile; ++i) {
                const int s = i % kTStages, as = i & 1;
                mb_wait(sm0 + tTEmpty + 8 * as, (((uint32_t)i >> 1) & 1u) ^ 1u, abort_flag, a.status);
                mb_wait(sm0 + tFull + 8 * s, (uint32_t)(i / kTStages) & 1u, abort_flag, a.status);
                if (*abort_flag) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t da0 = smem_desc(a_base + s * kTAStage);
                const uint32_t d_tmem = tmem_base + (uint32_t)(as * kTN);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint64_t da = da0 + (uint64_t)(((k >> 2) * kTAHalf + (k & 3) * 32) >> 4);
                    const uint64_t db = db0 + (uint64_t)(((k >> 2) * kTBHalf + (k & 3) * 32) >> 4);
                    umma_ss<kTIdesc>(d_tmem, da, db, k > 0);
                }
                umma_commit(sm0 + tEmpty + 8 * s);
                umma_commit(sm0 + tTFull + 8 * as);
            }
        }
    } else {
        // ---- epilogue: thread = token (TMEM lane); maximum of |D| and sum of D^2 over the probe rows that see the token ----
        const int lq = warp & 3;
        float* const err = a.err + ((int64_t)unit * a.nslots + layer * pl.mblocks + mblock) * a.Tmax;
        const float c32 = a.B == 4 ? 1.f : __uint_as_float(0x3F3504F3u);  // a pair's rows are Z1: K - Khat^shared = +-c Z1
        uint32_t* score = a.score + (int64_t)unit * a.Tmax;
        for (int i = 0; i < ntile; ++i) {
            const int as = i & 1;
            const int t = (tile0 + i) * kTM + lq * 32 + lane;
            mb_wait(sm0 + tTFull + 8 * as, ((uint32_t)i >> 1) & 1u, abort_flag, a.status);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            float m = 0.f, e0 = 0.f, e1 = 0.f;
            if (!*abort_flag) {
                const bool all_visible = (tile0 + i) * kTM + kTM - 1 <= pl.pos_min;
#pragma unroll
                for (int cp = 0; cp < 4; ++cp) {
                    uint32_t r0[32], r1[32];
                    const uint32_t ta = tmem_base + ((uint32_t)(lq * 32) << 16) + (uint32_t)(as * kTN + cp * 64);
                    tmem_ld32(ta, r0);
                    tmem_ld32(ta + 32, r1);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (all_visible) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const float u = __uint_as_float(r0[j]), v = __uint_as_float(r1[j]);
                            m = fmaxf(m, fmaxf(fabsf(u), fabsf(v)));
                            e0 = fmaf(u, u, e0);
                            e1 = fmaf(v, v, e1);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const float u = __uint_as_float(r0[j]), v = __uint_as_float(r1[j]);
                            if (pos_col[cp * 64 + j] >= t) { m = fmaxf(m, fabsf(u)); e0 = fmaf(u, u, e0); }
                            if (pos_col[cp * 64 + 32 + j] >= t) { m = fmaxf(m, fabsf(v)); e1 = fmaf(v, v, e1); }
                        }
                    }
                }
            }
            if (t < a.T && !*abort_flag) {
                if (m > 0.f) atomicMax(score + t, __float_as_uint(m * c32));
                err[t] = e0 + e1;
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mb_arrive(sm0 + tTEmpty + 8 * as);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

// ---- block-wide helpers for the select kernel (1024 threads) ----
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
    if (warp == 0) {
        uint32_t w = s_warp[lane];
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, wi, o);
            if (lane >= o) wi += x;
        }
        s_warp[lane] = wi - w;
        if (lane == 31) s_warp[32] = wi;
    }
    __syncthreads();
    *total = s_warp[32];
    return s_warp[warp] + incl - v;
}

// One CTA per unit: threshold of the k-th largest score (32-bit patterns of non-negative floats order like the
// floats), then the ascending list of kept tokens (score above the threshold, or equal and among the first `need`
// such tokens), the number of kept tokens before every 16-token slice, and the unit's two error sums: all tokens'
// (shared) and the unselected ones' (residual), float64 over the score kernel's per-token sums in a fixed order.
__global__ void __launch_bounds__(1024) token_select_kernel(TokenArgs a) {
    __shared__ uint32_t s_hist[256];
    __shared__ uint32_t s_warp[33];
    __shared__ uint32_t s_prefix, s_krem;
    const int unit = a.unit_begin + blockIdx.x;
    const uint32_t* key = a.score + (int64_t)unit * a.Tmax;
    const float* err = a.err + (int64_t)unit * a.nslots * a.Tmax;
    int32_t* list = a.list + (int64_t)unit * a.ktok_cap;
    int32_t* off = a.off + (int64_t)unit * (a.ntiles_max + 1);
    const int T = a.T;
    const int nslice = (T + kResTile - 1) / kResTile;
    uint32_t tau = 0xFFFFFFFFu, need = 0;
    if (a.k_tok > 0) {
        if (threadIdx.x == 0) { s_prefix = 0; s_krem = (uint32_t)a.k_tok; }
        for (int pass = 0; pass < 4; ++pass) {
            const int shift = 24 - 8 * pass;
            if (threadIdx.x < 256) s_hist[threadIdx.x] = 0;
            __syncthreads();
            const uint32_t prefix = s_prefix;
            for (int t = threadIdx.x; t < T; t += blockDim.x) {
                const uint32_t k = key[t];
                if (pass == 0 || (k >> (shift + 8)) == prefix) atomicAdd(&s_hist[(k >> shift) & 0xFFu], 1u);
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                uint32_t above = 0, krem = s_krem;
                int b = 255;
                for (; b > 0; --b) {
                    if (above + s_hist[b] >= krem) break;
                    above += s_hist[b];
                }
                s_prefix = (prefix << 8) | (uint32_t)b;
                s_krem = krem - above;
            }
            __syncthreads();
        }
        tau = s_prefix;
        need = s_krem;
    }
    // ordered compaction, 1024 tokens per round
    uint32_t base_keep = 0, base_eq = 0;
    double sum_all = 0.0, sum_dropped = 0.0;
    const int seen = min(T, a.pos_last + 1);  // later tokens are seen by no probe query: no error, nothing was written
    for (int t0 = 0; t0 < T; t0 += 1024) {
        const int t = t0 + threadIdx.x;
        const uint32_t k = t < T ? key[t] : 0u;
        const uint32_t gt = t < T && a.k_tok > 0 && k > tau, eq = t < T && a.k_tok > 0 && k == tau;
        uint32_t tot_eq, tot_keep;
        const uint32_t rank_eq = base_eq + block_excl_scan(eq, s_warp, &tot_eq);
        const uint32_t keep = gt || (eq && rank_eq < need);
        const uint32_t posk = base_keep + block_excl_scan(keep, s_warp, &tot_keep);
        if (t < seen) {
            double e = 0.0;
            for (int j = 0; j < a.nslots; ++j) e += (double)err[(int64_t)j * a.Tmax + t];
            sum_all += e;
            if (!keep) sum_dropped += e;
        }
        if (t < T) {
            if (keep) list[posk] = t;
            if ((t & (kResTile - 1)) == 0) off[t / kResTile] = (int32_t)posk;
        }
        base_eq += tot_eq;
        base_keep += tot_keep;
    }
    __shared__ double s_err[2][32];
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        sum_all += __shfl_xor_sync(0xFFFFFFFFu, sum_all, o);
        sum_dropped += __shfl_xor_sync(0xFFFFFFFFu, sum_dropped, o);
    }
    if ((threadIdx.x & 31) == 0) { s_err[0][threadIdx.x >> 5] = sum_all; s_err[1][threadIdx.x >> 5] = sum_dropped; }
    __syncthreads();
    if (threadIdx.x < 2) {
        double e = 0.0;
        for (int w = 0; w < 32; ++w) e += s_err[threadIdx.x][w];
        a.part[(int64_t)unit * a.nptiles_max * 2 + threadIdx.x] = e;
    }
    if (threadIdx.x == 0) {
        off[nslice] = (int32_t)base_keep;
        if ((int64_t)base_keep != a.k_tok) atomicMax(a.status, (int32_t)kFlagCountMismatch);
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
        cudaError_t e1 = cudaFuncSetAttribute(token_score_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTSmem);
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
        token_select_kernel<<<a.unit_count, 1024, 0, st>>>(a);
        count_launch(2);
        count_kernel(FDKV_KERNEL_PROBE_PORTABLE);
        return cudaGetLastError();
    }
    ScorePlan pl;
    pl.pos_min = a.pos_host[0];
    pl.ntiles = a.pos_host[a.W - 1] / kTM + 1;  // tokens after the last probe position are seen by nobody: score 0
    pl.mblocks = (a.G * a.W + kTN - 1) / kTN;  // (a.nslots = B x mblocks)
    const int base_items = a.unit_count * a.B * pl.mblocks;
    int nsplits = std::max(1, std::min((4 * sm_count + base_items - 1) / base_items, (pl.ntiles + 7) / 8));
    pl.tiles_per_split = (pl.ntiles + nsplits - 1) / nsplits;
    pl.nsplits = (pl.ntiles + pl.tiles_per_split - 1) / pl.tiles_per_split;
    pl.items_per_unit = a.B * pl.mblocks * pl.nsplits;
    token_score_kernel<<<a.unit_count * pl.items_per_unit, kTThreads, kTSmem, st>>>(*reinterpret_cast<const CUtensorMap*>(a.tmap_z1_128), a, pl);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    token_select_kernel<<<a.unit_count, 1024, 0, st>>>(a);
    count_launch(2);
    count_kernel(FDKV_KERNEL_TOKEN_SCORE);
    count_kernel(FDKV_KERNEL_PROBE_TC);  // (it is the probe's product too)
    return cudaGetLastError();
}

}  // namespace fdkv
