// Prefill compression with the entry rule (Eq. 1 and Eq. 3): depth split, threshold and index-ordered compaction of the
// sparse residual, for pairs and for blocks of four layers, in one read of K and V.
//
// What is stored per position (float32, never contracted; rs = rounding to the storage type):
//   pair:           z0 = rs((x0 + x1) c), z1 = rs((x0 - x1) c); key = magnitude of z1
//   block of four:  s = (x0 + x1) + (x2 + x3), z0 = rs(s / 2), dev_l = rs(x_l - z0 / 2) (F_4's first row is 1/2 four
//                   times, so z0 / 2 is the block mean and the other three coefficients contribute x_l - mean);
//                   key = e = (dev_0^2 + dev_1^2) + (dev_2^2 + dev_3^2), the squared error dropping the position costs
// and the k positions of largest key (31-bit patterns of non-negative floats; ties to the lowest flat index) are listed in
// ascending order with their values.
//
//   1. sample_kernel     one block per unit-tensor reads up to 64 Ki positions (whole rows, spread over the tokens with a
//                        fixed jitter; all of them where there are no more) and sets a bound that about 1.2 k positions reach;
//   2. split_kernel      reads every row once, writes Z0 (and, of K, the high-frequency rows the probe reads) and appends the
//                        positions that reach the bound, in order, to the chunk's candidate list;
//   3. threshold_kernel  one block per unit-tensor (a cluster of them for few and long ones): the k-th largest key among the
//                        candidates (a radix select in shared memory), then the keys above and equal to it before every chunk;
//   4. compact_kernel    one warp per chunk: candidates -> the lists, the offsets of the 16-token tiles and, of K, a bit
//                        map of the kept positions.
// (Few short unit-tensors take small_kernel instead of all of these.)
// The bound is only a guess: where fewer than k positions reach it, step 3 says so and steps 2 and 3 run again for that
// unit-tensor with bound 0 (a chunk's list holds all of its positions), so the result never depends on the sample.  Where most
// positions are kept, or where Z0 overwrites the rows, every position is a candidate from the start.
// Bound by HBM: K and V are read once and about k / N x 1.2 of them written again; a pass that writes all high-frequency
// values and reads them back to select (what this replaces) moved 5 instead of 3.6 times a tensor's bytes, and its
// histogram of every key took 128 KiB of shared memory, one block per SM.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "fdkv_internal.h"

namespace fdkv {

namespace {

constexpr int kSplitThreads = 256;
constexpr int kSampleThreads = 512, kSampleBins = 4096;
constexpr int64_t kSampleElems = 65536;
constexpr int kThrThreads = 1024, kThrBins = 4096;
constexpr uint32_t kNoKey = 0xFFFFFFFFu;  // a bound or threshold above every key
// Of the positions are kept: from there on every position is taken for a candidate (4 layers of 32k tokens, all kept, 2 940 -> 872 us).
constexpr double kAllShare = 0.6;

// two float32 operations at a time, each rounded to nearest
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(uint32_t lo, uint32_t hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ f32x2 bf2(uint32_t w) { return pack2(w << 16, w & 0xFFFF0000u); }  // two bf16 values, widened
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) { f32x2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) { f32x2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {  // a + (-1) b, rounded once: the difference
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(pack2(0xBF800000u, 0xBF800000u)), "l"(a));
    return r;
}
__device__ __forceinline__ uint32_t to_bf2(f32x2 a) {  // both halves to nearest-even bf16
    uint32_t lo, hi, r;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(a));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(__uint_as_float(hi)), "f"(__uint_as_float(lo)));
    return r;
}

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }

// the key of a position from its stored high-frequency value(s)
template <int B>
__device__ __forceinline__ uint32_t key_of(const float* v) {
    if constexpr (B == 2) return __float_as_uint(v[0]) & 0x7FFFFFFFu;
    else
        return __float_as_uint(__fadd_rn(__fadd_rn(__fmul_rn(v[0], v[0]), __fmul_rn(v[1], v[1])),
                                         __fadd_rn(__fmul_rn(v[2], v[2]), __fmul_rn(v[3], v[3])))) & 0x7FFFFFFFu;
}

// bits of four words' eight 16-bit halves whose sums g carry into bit 15 / 31, in order
__device__ __forceinline__ uint32_t pair_mask8(uint32_t g0, uint32_t g1, uint32_t g2, uint32_t g3) {
    uint32_t t = (g0 >> 15) & 0x00010001u;  // word j -> bits 2j and 16 + 2j
    t |= (g1 >> 13) & 0x00040004u;
    t |= (g2 >> 11) & 0x00100010u;
    t |= (g3 >> 9) & 0x00400040u;
    return (t | (t >> 15)) & 0xFFu;
}

// Eight consecutive positions as 16-byte vectors, Q of them per row.  split: x[layer] -> shared coefficients z0 and
// high-frequency values hf[1 or 4]; keys: f(position, key) for each; reach: bit i = position i's key is at least lo.
template <typename T, int B>
struct Eight {
    static constexpr int Q = (int)sizeof(T) / 2, NB = B == 4 ? 4 : 1;
    __device__ static void split(const uint4 (&x)[B][Q], uint4 (&z0)[Q], uint4 (&hf)[NB][Q]) {
        if constexpr (sizeof(T) == 2) {
            const f32x2 c = pack2(0x3F3504F3u, 0x3F3504F3u), half1 = pack2(0x3F000000u, 0x3F000000u);  // the float32 nearest 1/sqrt 2; 1/2
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                f32x2 v[B];
#pragma unroll
                for (int l = 0; l < B; ++l) v[l] = bf2(word(x[l][0], w));
                if constexpr (B == 2) {
                    word(z0[0], w) = to_bf2(mul2(add2(v[0], v[1]), c));
                    word(hf[0][0], w) = to_bf2(mul2(sub2(v[0], v[1]), c));
                } else {
                    const uint32_t z = to_bf2(mul2(half1, add2(add2(v[0], v[1]), add2(v[2], v[3]))));
                    word(z0[0], w) = z;
                    const f32x2 half = mul2(half1, bf2(z));  // exact
#pragma unroll
                    for (int l = 0; l < 4; ++l) word(hf[l][0], w) = to_bf2(sub2(v[l], half));
                }
            }
        } else {
            const float c32 = __uint_as_float(0x3F3504F3u);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float f[B];
#pragma unroll
                for (int l = 0; l < B; ++l) f[l] = __uint_as_float(word(x[l][i >> 2], i & 3));
                if constexpr (B == 2) {
                    word(z0[i >> 2], i & 3) = __float_as_uint(__fmul_rn(__fadd_rn(f[0], f[1]), c32));
                    word(hf[0][i >> 2], i & 3) = __float_as_uint(__fmul_rn(__fsub_rn(f[0], f[1]), c32));
                } else {
                    const float z = __fmul_rn(0.5f, __fadd_rn(__fadd_rn(f[0], f[1]), __fadd_rn(f[2], f[3])));
                    const float half = __fmul_rn(0.5f, z);  // exact
                    word(z0[i >> 2], i & 3) = __float_as_uint(z);
#pragma unroll
                    for (int l = 0; l < 4; ++l) word(hf[l][i >> 2], i & 3) = __float_as_uint(__fsub_rn(f[l], half));
                }
            }
        }
    }
    template <typename F>
    __device__ static void keys(const uint4 (&hf)[NB][Q], F&& f) {
        if constexpr (sizeof(T) == 2) {
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                if constexpr (B == 2) {
                    const uint32_t h = word(hf[0][0], w);
                    f(2 * w, (h << 16) & 0x7FFF0000u);
                    f(2 * w + 1, h & 0x7FFF0000u);
                } else {
                    f32x2 v[4];
#pragma unroll
                    for (int l = 0; l < 4; ++l) { v[l] = bf2(word(hf[l][0], w)); v[l] = mul2(v[l], v[l]); }
                    const f32x2 e = add2(add2(v[0], v[1]), add2(v[2], v[3]));
                    f(2 * w, (uint32_t)e & 0x7FFFFFFFu);
                    f(2 * w + 1, (uint32_t)(e >> 32) & 0x7FFFFFFFu);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float h[NB];
#pragma unroll
                for (int l = 0; l < NB; ++l) h[l] = __uint_as_float(word(hf[l][i >> 2], i & 3));
                f(i, key_of<B>(h));
            }
        }
    }
    __device__ static uint32_t reach(const uint4 (&hf)[NB][Q], uint32_t lo) {
        if (lo == kNoKey) return 0u;
        if constexpr (sizeof(T) == 2 && B == 2) {
            // bit 15 (31) of a + (0x8000 - lo16) * 0x10001 says that the low (high) half reaches lo16: no carry crosses
            const uint32_t add = (0x8000u - (lo >> 16)) * 0x00010001u;
            const uint4& h = hf[0][0];
            return pair_mask8((h.x & 0x7FFF7FFFu) + add, (h.y & 0x7FFF7FFFu) + add, (h.z & 0x7FFF7FFFu) + add, (h.w & 0x7FFF7FFFu) + add);
        } else {
            uint32_t k8[8], m = 0;
            keys(hf, [&](int i, uint32_t key) { k8[i] = key - lo; });  // (both below 2^31: bit 31 says that the key is smaller)
#pragma unroll
            for (int i = 7; i >= 0; --i) m = __funnelshift_l(k8[i], m, 1);
            return ~m & 0xFFu;
        }
    }

private:
    __device__ static uint32_t& word(uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
    __device__ static uint32_t word(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
};

// programmatic dependent launch: the next kernel of the chain may start its prologue now; nothing is read before the kernels
// ahead are complete
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The bin, from the top, at which the running count of BINS shared-memory bins first reaches `target`: every thread of the
// block gets (bin, count in larger bins); false if the total is smaller.  A thread owns BINS / THREADS consecutive bins.
template <int THREADS, int BINS>
__device__ __forceinline__ bool find_bin(const uint32_t* bins, uint32_t target, uint32_t& bin, uint32_t& above) {
    __shared__ uint32_t s_tot[THREADS / 32], s_bin, s_above;
    constexpr int PER = BINS / THREADS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int hi = BINS - PER * tid;
    uint32_t c[PER], mine = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) { c[i] = bins[hi - 1 - i]; mine += c[i]; }
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_tot[warp] = incl;
    __syncthreads();
    uint32_t before = incl - mine, total = 0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
        if (w < warp) before += s_tot[w];
        total += s_tot[w];
    }
    if (before < target && target <= before + mine) {
        bool found = false;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            if (!found && before + c[i] >= target) { s_bin = (uint32_t)(hi - 1 - i); s_above = before; found = true; }
            before += c[i];
        }
    }
    __syncthreads();
    bin = s_bin;
    above = s_above;
    __syncthreads();  // (the scratch words may be reused)
    return target <= total;
}

// ---- 1: the bound -------------------------------------------------------------------------------------
// grid (heads x tensors, blocks of the launch)
template <typename T, int B>
__global__ void __launch_bounds__(kSampleThreads) sample_kernel(CompressArgs a, int n_rows, uint32_t target, uint32_t among) {
    __shared__ uint32_t s_hist[kSampleBins];
    constexpr int NB = B == 4 ? 4 : 1, Q = Eight<T, B>::Q;
    const int tid = threadIdx.x;
    const int ut = a.ut_base + blockIdx.y * gridDim.x + blockIdx.x;
    const int h = blockIdx.x / a.tensors, is_v = blockIdx.x % a.tensors;
    for (int i = tid; i < kSampleBins; i += kSampleThreads) s_hist[i] = 0;
    chain_wait();
    __syncthreads();
    const T* x[B];
#pragma unroll
    for (int l = 0; l < B; ++l) x[l] = reinterpret_cast<const T*>(is_v ? a.v[B * blockIdx.y + l] : a.k[B * blockIdx.y + l]) + (int64_t)h * a.stride_h;
    const int vshift = a.d == 128 ? 4 : 3, nvec = n_rows << vshift;
    // groups of eight whose rows are requested together (float32 blocks of four: four of them spill, and the kernel took 32 or 50 us, whichever code
    // stood beside it; 4 layers, 16 heads, 4 096 tokens: 223 -> 213 us in all)
    constexpr int U = B * Q > 4 ? 2 : 4;
    for (int v0 = tid; v0 < nvec; v0 += U * kSampleThreads) {
        uint4 f[U][B][Q];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int v = v0 + q * kSampleThreads;
            if (v >= nvec) break;
            const int r = v >> vshift, cv = (v & ((1 << vshift) - 1)) * 8;
            int t = r;
            if (n_rows < a.T) {  // row r of the sample: somewhere in the r-th of n_rows equal parts of the tokens
                const uint32_t jitter = (uint32_t)r * 2654435761u >> 16;  // (a multiplicative hash, 16 bits)
                t = (int)((((uint64_t)(uint32_t)r << 16 | jitter) * (uint64_t)a.T) / ((uint64_t)n_rows << 16));
            }
#pragma unroll
            for (int l = 0; l < B; ++l)
#pragma unroll
                for (int k = 0; k < Q; ++k) f[q][l][k] = reinterpret_cast<const uint4*>(x[l] + (int64_t)t * a.stride_t + cv)[k];
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            if (v0 + q * kSampleThreads >= nvec) break;
            uint4 z0[Q], hf[NB][Q];
            Eight<T, B>::split(f[q], z0, hf);
            Eight<T, B>::keys(hf, [&](int, uint32_t key) { atomicAdd(&s_hist[key >> 19], 1u); });
        }
    }
    __syncthreads();
    uint32_t bin, above;
    const bool enough = find_bin<kSampleThreads, kSampleBins>(s_hist, target, bin, above);
    if (tid == 0) {
        a.sel[ut].redo = 0;
        a.sel[ut].lo = a.n_keep == 0 ? kNoKey : enough ? bin << 19 : 0u;
        // is the k-th among the 63 bf16 keys from the bound up: seven bins and seven eighths of one?
        for (uint32_t i = 1; i < 7 && bin + i < (uint32_t)kSampleBins; ++i) above -= s_hist[bin + i];
        a.sel[ut].tau = enough && 8 * above < 8 * among + (bin + 7 < (uint32_t)kSampleBins ? 7 * s_hist[bin + 7] : 0u);
    }
}

// ---- 2: one read of K and V ---------------------------------------------------------------------------
// Persistent blocks over (chunk, head x tensor) items; heads and tensors vary fastest, so the blocks that run at one time read
// neighbouring rows.  A warp owns NV * 256 consecutive positions of a chunk, a lane eight of them per step.  The rows of the
// next item are copied to shared memory (cp.async, 16 bytes per lane and layer, every lane its own) while one is worked on; the
// high-frequency values take the place of the rows they came from.  A byte per eight positions goes to a bit map; then
// the positions of every lane's NV * 8 go behind those of the lanes and warps before it, and the lists leave in runs.  One
// block barrier per item (the warps' counts).  The issue slots are nearly as busy as HBM here (60 % and 69 %), hence the packed arithmetic, the
// bit tricks and the running item coordinates (with scalar arithmetic, a binary search per list entry and divisions per item:
// 1 550 us for 32 layers of 32k tokens).
// ALL: every position is a candidate, the values go to the list in their order and no positions are written (see kAllShare).
template <typename T, int B, bool ALL>
__global__ void __launch_bounds__(kSplitThreads, 3) split_kernel(CompressArgs a, int items, int redo) {
    constexpr int NB = B == 4 ? 4 : 1, Q = Eight<T, B>::Q;
    constexpr int CE = compress_chunk(B, (int)sizeof(T)), NV = CE / kSplitThreads / 8;
    constexpr int BITS = NV * 8;         // bits of the map per lane = words per warp
    constexpr int ROW = CE * (int)sizeof(T);  // bytes of a layer's part of a stage
    constexpr int STAGE = B * ROW;       // 32 KiB
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_map[8][BITS], s_cnt[2][8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int uts = a.Hkv * a.tensors;
    chain_wait();
    if (redo) {  // (almost always there is nothing to do again)
        const int n_ut = items / a.chunks;
        int any = 0;
        for (int i = tid; i < n_ut; i += kSplitThreads) any |= (int)a.sel[a.ut_base + i].redo;
        if (!__syncthreads_or(any)) return;
    }
    const int64_t n_e = (int64_t)a.T * a.d;
    const int dshift = a.d == 128 ? 7 : 6;
    // an item's coordinates: head x tensor, chunk, block of the launch; a step is gridDim.x items
    struct Item { int u, chunk, blk; };
    const int step_u = gridDim.x % uts, step_r = gridDim.x / uts;
    auto norm = [&](Item& m) {
        while (m.chunk >= a.chunks) { m.chunk -= a.chunks; ++m.blk; }
    };
    auto advance = [&](Item& m) {
        m.u += step_u;
        m.chunk += step_r;
        if (m.u >= uts) { m.u -= uts; ++m.chunk; }
        norm(m);
    };
    const int p0 = warp * (NV * 256) + lane * 8;  // position of the lane's first eight; step q adds 256 q
    const int64_t q_step = (int64_t)(256 >> dshift) * a.stride_t;
    const uint32_t dst0 = (uint32_t)__cvta_generic_to_shared(smem) + p0 * (int)sizeof(T);
    auto request = [&](const Item& m, int stage) {
        const int h = m.u / a.tensors, is_v = m.u - h * a.tensors;
        const int64_t e = (int64_t)m.chunk * CE + p0;
        const int64_t off = (e >> dshift) * a.stride_t + (int64_t)h * a.stride_h + ((int)e & (a.d - 1));
#pragma unroll
        for (int l = 0; l < B; ++l) {
            const T* src = reinterpret_cast<const T*>(is_v ? a.v[B * m.blk + l] : a.k[B * m.blk + l]) + off;
#pragma unroll
            for (int q = 0; q < NV; ++q, src += q_step)
                if (e + 256 * q < n_e)
#pragma unroll
                    for (int k = 0; k < Q; ++k)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst0 + stage * STAGE + l * ROW + 256 * q * (int)sizeof(T) + 16 * k),
                                     "l"(reinterpret_cast<const uint4*>(src) + k)
                                     : "memory");
        }
    };
    Item now = {(int)(blockIdx.x % uts), (int)(blockIdx.x / uts), 0}, ahead;
    norm(now);
    ahead = now;
    int left = (items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x, to_request = left;  // items of this block
    auto request_next = [&](int stage) {
        if (to_request > 0) {
            request(ahead, stage);
            advance(ahead);
            --to_request;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    request_next(0);
    request_next(1);
    // The warps' counts alternate between two sets with the items that are worked on, not with the stages: the barrier of the next such
    // item is what separates a set's reads from its next writes, and in a second run other items lie between.
    int cs = 0;
    for (int it = 0; left > 0; --left, it ^= 1, advance(now)) {
        const int ut = a.ut_base + now.blk * uts + now.u;
        const int64_t e0 = (int64_t)now.chunk * CE;
        const uint32_t lo = ALL ? 0u : a.sel[ut].lo;
        uint8_t* const st = smem + it * STAGE;
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        if (ALL || !redo || a.sel[ut].redo) {  // (block-uniform)
            const int h = now.u / a.tensors;
            const bool is_k = now.u == h * a.tensors;
            T* const val = reinterpret_cast<T*>(a.cand_val) + (int64_t)ut * NB * a.cand_stride + e0;
            T* const z0 = reinterpret_cast<T*>(a.z0) + (int64_t)ut * a.z0_stride + e0 + p0;
            T* const z1 = a.z1 && is_k ? reinterpret_cast<T*>(a.z1) + (int64_t)(now.blk * a.Hkv + h + a.ut_base / a.tensors) * NB * a.unit_stride + e0 + p0 : nullptr;
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                uint32_t m8 = 0;
                if (e0 + p0 + 256 * q < n_e) {
                    uint4 x[B][Q], z[Q], hf[NB][Q];
#pragma unroll
                    for (int l = 0; l < B; ++l)
#pragma unroll
                        for (int k = 0; k < Q; ++k) x[l][k] = reinterpret_cast<const uint4*>(st + l * ROW + (p0 + 256 * q) * sizeof(T))[k];
                    Eight<T, B>::split(x, z, hf);
                    if constexpr (!ALL) m8 = Eight<T, B>::reach(hf, lo);
#pragma unroll
                    for (int k = 0; k < Q; ++k) {
                        if (!redo) reinterpret_cast<uint4*>(z0 + 256 * q)[k] = z[k];
#pragma unroll
                        for (int l = 0; l < NB; ++l) {
                            if (z1 && !redo) reinterpret_cast<uint4*>(z1 + (int64_t)l * a.unit_stride + 256 * q)[k] = hf[l][k];
                            if constexpr (ALL) reinterpret_cast<uint4*>(val + (int64_t)l * a.cand_stride + p0 + 256 * q)[k] = hf[l][k];
                            else reinterpret_cast<uint4*>(st + l * ROW + (p0 + 256 * q) * sizeof(T))[k] = hf[l][k];
                        }
                    }
                }
                if constexpr (!ALL) reinterpret_cast<uint8_t*>(s_map[warp])[32 * q + lane] = (uint8_t)m8;
            }
            __syncwarp();
            if constexpr (ALL) {
                if (tid == 0) a.cand_n[(int64_t)ut * a.chunks_max + now.chunk] = (int32_t)min((int64_t)CE, n_e - e0);
                request_next(it);
                continue;
            }
            // the lane's BITS consecutive positions of the warp's part
            uint32_t bits = BITS == 32   ? s_map[warp][lane]
                            : BITS == 16 ? (uint32_t)reinterpret_cast<const uint16_t*>(s_map[warp])[lane]
                                         : (uint32_t)reinterpret_cast<const uint8_t*>(s_map[warp])[lane];
            const uint32_t mine = __popc(bits);
            uint32_t incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) s_cnt[cs][warp] = incl;
            __syncthreads();
            uint32_t at = incl - mine, n = 0;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                const uint32_t y = s_cnt[cs][w];
                if (w < warp) at += y;
                n += y;
            }
            cs ^= 1;
            if (tid == 0) a.cand_n[(int64_t)ut * a.chunks_max + now.chunk] = (int32_t)n;
            uint16_t* const pos = a.cand_pos + (int64_t)ut * a.cand_stride + e0;
            const uint32_t first = warp * (NV * 256) + lane * BITS;
            // positions into shared memory, then both lists in runs (two-byte stores at every lane's own place took most of the time
            // where many positions are candidates: keep 1/2, 32k tokens, 1 080 of 1 740 us)
            uint16_t* const s_pos = B == 2 ? reinterpret_cast<uint16_t*>(st + ROW + warp * (NV * 256) * sizeof(T))  // (a layer's rows that are done with)
                                           : reinterpret_cast<uint16_t*>(smem + 2 * STAGE) + warp * (NV * 256);
            for (uint32_t i = incl - mine; bits; bits &= bits - 1, ++i) s_pos[i] = (uint16_t)(first + __ffs((int)bits) - 1);
            const uint32_t n_w = __shfl_sync(0xFFFFFFFFu, incl, 31);
            at -= incl - mine;  // the warp's first
            __syncwarp();
            for (uint32_t i = lane; i < n_w; i += 32) {
                const uint32_t p = s_pos[i];
                pos[at + i] = (uint16_t)p;
#pragma unroll
                for (int l = 0; l < NB; ++l) val[(int64_t)l * a.cand_stride + at + i] = reinterpret_cast<const T*>(st + l * ROW)[p];
            }
            __syncwarp();  // (the warp's part of the stage is read)
        }
        request_next(it);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// ---- 3: the threshold ---------------------------------------------------------------------------------
// f(key) for every candidate of chunk c; eight candidates per lane and load, STEPS of them requested together
template <typename T, int B, typename F>
__device__ __forceinline__ void each_candidate(const CompressArgs& a, int ut, int c, int n, F&& f) {
    constexpr int NB = B == 4 ? 4 : 1, Q = Eight<T, B>::Q;
    constexpr int CE = compress_chunk(B, (int)sizeof(T));
    constexpr int STEPS = NB * Q == 1 ? 3 : NB * Q == 2 ? 2 : 1;
    const int lane = threadIdx.x & 31;
    const T* const val = reinterpret_cast<const T*>(a.cand_val) + (int64_t)ut * NB * a.cand_stride + (int64_t)c * CE;
    for (int i0 = lane * 8; i0 < n; i0 += 256 * STEPS) {
        uint4 v[STEPS][NB][Q];
#pragma unroll
        for (int s = 0; s < STEPS; ++s)
            if (i0 + 256 * s < n)
#pragma unroll
                for (int l = 0; l < NB; ++l)
#pragma unroll
                    for (int k = 0; k < Q; ++k) v[s][l][k] = reinterpret_cast<const uint4*>(val + (int64_t)l * a.cand_stride + i0 + 256 * s)[k];
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
            const int m = n - i0 - 256 * s;  // candidates from this vector on
            if (m >= 8) Eight<T, B>::keys(v[s], [&](int, uint32_t key) { f(key); });
            else if (m > 0) Eight<T, B>::keys(v[s], [&](int j, uint32_t key) { if (j < m) f(key); });
        }
    }
}

__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the sum over the cluster of two consecutive 32-bit words at a shared-memory address, eight loads in flight together
template <int MOST = 8>  // blocks of a cluster at most
__device__ __forceinline__ uint2 cluster_sum2(uint32_t addr, int blocks) {
    uint2 sum = make_uint2(0, 0);
#pragma unroll
    for (int r0 = 0; r0 < MOST; r0 += 8) {
        if (r0 > 0 && r0 >= blocks) break;
        uint2 v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            uint32_t at;
            asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(addr), "r"(r0 + r < blocks ? r0 + r : 0));
            asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(v[r].x), "=r"(v[r].y) : "r"(at));
        }
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if (r0 + r < blocks) { sum.x += v[r].x; sum.y += v[r].y; }
    }
    return sum;
}

// counts of chunks [c_begin, c_end) (written by this block, a barrier ago) -> counts before each, the two given ones included
__device__ __forceinline__ void scan_chunks(int2* base, int c_begin, int c_end, uint32_t run_gt, uint32_t run_eq, uint32_t (&s_sum)[2][32]) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int c0 = c_begin; c0 < c_end; c0 += kThrThreads) {
        const int c = c0 + tid;
        const int2 m = c < c_end ? __ldcg(base + c) : make_int2(0, 0);  // (counted by atomics, which pass by the L1)
        uint32_t ig = (uint32_t)m.x, ie = (uint32_t)m.y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t yg = __shfl_up_sync(0xFFFFFFFFu, ig, o), ye = __shfl_up_sync(0xFFFFFFFFu, ie, o);
            if (lane >= o) { ig += yg; ie += ye; }
        }
        __syncthreads();
        if (lane == 31) { s_sum[0][warp] = ig; s_sum[1][warp] = ie; }
        __syncthreads();
        uint32_t tg = 0, te = 0, bg = run_gt, be = run_eq;
#pragma unroll
        for (int w = 0; w < 32; ++w) {
            if (w < warp) { bg += s_sum[0][w]; be += s_sum[1][w]; }
            tg += s_sum[0][w];
            te += s_sum[1][w];
        }
        if (c < c_end) base[c] = make_int2((int)(bg + ig) - m.x, (int)(be + ie) - m.y);
        run_gt += tg;
        run_eq += te;
    }
}

// One block per unit-tensor (grid ut_count).  First digit: the key's top 15 bits, in a window of 4 095 bins from the bound up
// (32 octaves; the last bin counts what is larger, and in the unheard-of case that the k-th key is there the window moves
// up): with 128 bins per octave the atomics hardly collide, and 16 KiB leave room for two blocks on an SM.  32-bit keys:
// two more digits of 12 and 4 bits among the few keys that share the first, which the second pass gathers while it counts the larger
// ones of every chunk (a pass per digit and one for the counts: 12 289 tokens, 128 tensors of blocks of four: 112 -> 76 us), where the first
// one's histogram says that they fit.
// bf16 magnitudes: where the k-th is within half an octave of the bound, a chunk's counts of the 63 keys from the bound up, kept in shared memory,
// give both the threshold and the counts before every chunk in one pass (a second one for the counts: 256 tensors of 32k tokens, behind the split:
// 149 -> 88 us).  The sample says whether it is: with keep 1/3 and more of log-normal channel scales it is not, and a pass for nothing made 128
// tensors of 8 192 tokens at keep 1/2 673 us instead of 622.
// Where these don't hold the digits are counted one after the other.
constexpr int kThrMini = 512;  // chunks whose counts are kept: 64 KiB, 32k x 128 positions.  (Longer tensors take the passes; more chunks were not measured.)
template <typename T, int B>
__global__ void __launch_bounds__(kThrThreads) threshold_kernel(CompressArgs a, int ut_begin, int redo) {
    __shared__ __align__(16) uint32_t s_hist[kThrBins];
    __shared__ uint32_t s_sum[2][32], s_found[2], s_near;
    extern __shared__ __align__(16) uint32_t s_dyn[];  // bf16 pairs: [chunks][32] two counts a word; else [kThrBins] keys that share the first digit
    constexpr bool F32KEY = !(sizeof(T) == 2 && B == 2);  // a bf16 magnitude is 15 bits
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ut = ut_begin + blockIdx.x, chunks = a.chunks;
    SelState* const sel = a.sel + ut;
    chain_wait();
    if (redo && !sel->redo) return;
    const int32_t* const cn = a.cand_n + (int64_t)ut * a.chunks_max;
    auto all_candidates = [&](auto&& f) {
        int n = warp < chunks ? cn[warp] : 0;
        for (int c = warp; c < chunks; c += 32) {
            const int n_next = c + 32 < chunks ? cn[c + 32] : 0;
            each_candidate<T, B>(a, ut, c, n, f);
            n = n_next;
        }
    };
    uint32_t tau = kNoKey, need = 0;
    if (a.n_keep > 0) {
        // are there k candidates?
        uint32_t mine = 0;
        for (int c = tid; c < chunks; c += kThrThreads) mine += (uint32_t)cn[c];
#pragma unroll
        for (int o = 16; o; o >>= 1) mine += __shfl_xor_sync(0xFFFFFFFFu, mine, o);
        if (lane == 0) s_sum[0][warp] = mine;
        __syncthreads();
        uint32_t total = 0;
#pragma unroll
        for (int w = 0; w < 32; ++w) total += s_sum[0][w];
        if ((int64_t)total < a.n_keep) {
            if (tid == 0) { sel->redo = 1; sel->lo = 0; }
            return;
        }
        if constexpr (!F32KEY)
            if (chunks <= kThrMini && !redo && sel->tau) {
                uint32_t* const mini = s_hist + 64 * warp;
                uint32_t* const total_of = s_hist + 64 * 32;
                const uint32_t lo16 = sel->lo >> 16;
                *reinterpret_cast<uint2*>(mini + 2 * lane) = make_uint2(0u, 0u);
                if (tid < 64) total_of[tid] = 0;
                __syncthreads();
                uint2 sum = make_uint2(0u, 0u);
                int n = warp < chunks ? cn[warp] : 0;
                for (int c = warp; c < chunks; c += 32) {
                    const int n_next = c + 32 < chunks ? cn[c + 32] : 0;
                    each_candidate<T, B>(a, ut, c, n, [&](uint32_t key) {
                        const uint32_t k = (key >> 16) - lo16;
                        if (k < 63u) atomicAdd(&mini[k], 1u);
                    });
                    __syncwarp();
                    uint2 v = *reinterpret_cast<const uint2*>(mini + 2 * lane);
                    const uint32_t inside = __reduce_add_sync(0xFFFFFFFFu, v.x + v.y);
                    if (lane == 31) v.y = (uint32_t)n - inside;  // the larger ones
                    s_dyn[32 * c + lane] = v.x | v.y << 16;      // (a chunk has at most 2^13 positions)
                    sum.x += v.x;
                    sum.y += v.y;
                    *reinterpret_cast<uint2*>(mini + 2 * lane) = make_uint2(0u, 0u);
                    __syncwarp();
                    n = n_next;
                }
                atomicAdd(&total_of[2 * lane], sum.x);
                atomicAdd(&total_of[2 * lane + 1], sum.y);
                __syncthreads();
                if (warp == 0) {  // a lane's two bins, the largest first
                    const uint32_t c0 = total_of[63 - 2 * lane], c1 = total_of[62 - 2 * lane], k = (uint32_t)a.n_keep;
                    uint32_t before = c0 + c1;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, before, o);
                        if (lane >= o) before += y;
                    }
                    before -= c0 + c1;
                    if (before < k && k <= before + c0) { s_found[0] = 63 - 2 * lane; s_found[1] = before; }
                    if (before + c0 < k && k <= before + c0 + c1) { s_found[0] = 62 - 2 * lane; s_found[1] = before + c0; }
                }
                __syncthreads();
                const int bin = (int)s_found[0];
                if (bin < 63) {
                    if (tid == 0) { sel->tau = (lo16 + bin) << 16; sel->need = (uint32_t)a.n_keep - s_found[1]; }
                    int2* const base = a.chunk_base + (int64_t)ut * a.chunks_max;
                    for (int c = tid; c < chunks; c += kThrThreads) {
                        uint32_t gt = 0, eq = 0;
                        for (int i = 0; i < 32; ++i) {
                            const int j = (i + c) & 31;  // (the threads of a warp in different banks)
                            const uint32_t w = s_dyn[32 * c + j], x = w & 0xFFFFu, y = w >> 16;
                            gt += (2 * j > bin ? x : 0u) + (2 * j + 1 > bin ? y : 0u);
                            eq += (2 * j == bin ? x : 0u) + (2 * j + 1 == bin ? y : 0u);
                        }
                        base[c] = make_int2((int)gt, (int)eq);
                    }
                    __syncthreads();
                    scan_chunks(base, 0, chunks, 0, 0, s_sum);
                    return;
                }
                __syncthreads();
            }
        uint32_t k_rem = (uint32_t)a.n_keep, prefix, above, in_bin;
        for (uint32_t from = sel->lo >> 16;; from += kThrBins - 1) {
            for (int i = tid; i < kThrBins; i += kThrThreads) s_hist[i] = 0;
            __syncthreads();
            all_candidates([&](uint32_t key) {
                const uint32_t k16 = key >> 16;
                if (k16 >= from) atomicAdd(&s_hist[min(k16 - from, (uint32_t)kThrBins - 1)], 1u);
            });
            __syncthreads();
            uint32_t bin;
            find_bin<kThrThreads, kThrBins>(s_hist, k_rem, bin, above);
            prefix = from + bin;
            in_bin = s_hist[bin];
            __syncthreads();
            if (bin < kThrBins - 1 || from + kThrBins - 1 >= 32767) break;
        }
        k_rem -= above;
        if constexpr (F32KEY) {
            const uint32_t top = prefix;
            if (chunks <= 0x10000 && in_bin <= (uint32_t)kThrBins) {
                // ---- larger keys of every chunk, and those that share the first digit: chunk and low half ----
                int2* const base = a.chunk_base + (int64_t)ut * a.chunks_max;
                if (tid == 0) s_near = 0;
                __syncthreads();
                int n = warp < chunks ? cn[warp] : 0;
                for (int c = warp; c < chunks; c += 32) {
                    const int n_next = c + 32 < chunks ? cn[c + 32] : 0;
                    uint32_t gt = 0;
                    each_candidate<T, B>(a, ut, c, n, [&](uint32_t key) {
                        gt += key >> 16 > top ? 1u : 0u;
                        if (key >> 16 == top) {
                            const uint32_t i = atomicAdd(&s_near, 1u);
                            if (i < (uint32_t)kThrBins) s_dyn[i] = (uint32_t)c << 16 | (key & 0xFFFFu);
                        }
                    });
                    gt = __reduce_add_sync(0xFFFFFFFFu, gt);
                    if (lane == 0) base[c] = make_int2((int)gt, 0);
                    n = n_next;
                }
                __syncthreads();
                const uint32_t near = s_near;
                // (it fits, as in_bin says; without the two tests the compiler's code is slower: one float32 pair of 8 192 tokens 63.8 -> 67.4 us)
                if (near <= (uint32_t)kThrBins) {
                    uint32_t low = 0;
#pragma unroll 1
                    for (int pass = 0; pass < 2; ++pass) {
                        const int shift = pass == 0 ? 4 : 0, bits = pass == 0 ? 12 : 4;
                        for (int i = tid; i < kThrBins; i += kThrThreads) s_hist[i] = 0;
                        __syncthreads();
                        for (uint32_t i = tid; i < near; i += kThrThreads) {
                            const uint32_t key = s_dyn[i] & 0xFFFFu;
                            if (pass == 0 || key >> 4 == low) atomicAdd(&s_hist[(key >> shift) & ((1u << bits) - 1u)], 1u);
                        }
                        __syncthreads();
                        uint32_t bin;
                        find_bin<kThrThreads, kThrBins>(s_hist, k_rem, bin, above);
                        low = low << bits | bin;
                        k_rem -= above;
                    }
                    if (tid == 0) { sel->tau = top << 16 | low; sel->need = k_rem; }
                    for (uint32_t i = tid; i < near; i += kThrThreads) {
                        const uint32_t c = s_dyn[i] >> 16, key = s_dyn[i] & 0xFFFFu;
                        if (key > low) atomicAdd(&base[c].x, 1);
                        else if (key == low) atomicAdd(&base[c].y, 1);
                    }
                    __syncthreads();
                    scan_chunks(base, 0, chunks, 0, 0, s_sum);
                    return;
                }
                __syncthreads();
            }
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                const int shift = pass == 0 ? 4 : 0, bits = pass == 0 ? 12 : 4;
                for (int i = tid; i < kThrBins; i += kThrThreads) s_hist[i] = 0;
                __syncthreads();
                const uint32_t want = pass == 0 ? top : prefix;
                all_candidates([&](uint32_t key) {
                    if ((key >> (shift + bits)) == want) atomicAdd(&s_hist[(key >> shift) & ((1u << bits) - 1u)], 1u);
                });
                __syncthreads();
                uint32_t bin;
                find_bin<kThrThreads, kThrBins>(s_hist, k_rem, bin, above);
                prefix = (want << bits) | bin;
                k_rem -= above;
            }
        }
        tau = F32KEY ? prefix : prefix << 16;
        need = k_rem;
    }
    if (tid == 0) { sel->tau = tau; sel->need = need; }
    // ---- keys above and equal to the threshold before every chunk ----
    int2* const base = a.chunk_base + (int64_t)ut * a.chunks_max;
    {
        int n = warp < chunks ? cn[warp] : 0;
        for (int c = warp; c < chunks; c += 32) {
            const int n_next = c + 32 < chunks ? cn[c + 32] : 0;
            uint32_t both = 0;  // above in the low half, equal in the high half (a lane meets at most 2^13 candidates of a chunk)
            if (a.n_keep > 0) each_candidate<T, B>(a, ut, c, n, [&](uint32_t key) { both += key > tau ? 1u : key == tau ? 0x10000u : 0u; });
            // (sums of 32 lanes stay below 2^16: a chunk has at most 2^13 positions)
#pragma unroll
            for (int o = 16; o; o >>= 1) both += __shfl_xor_sync(0xFFFFFFFFu, both, o);
            if (lane == 0) base[c] = make_int2((int)(both & 0xFFFFu), (int)(both >> 16));
            n = n_next;
        }
    }
    __syncthreads();
    scan_chunks(base, 0, chunks, 0, 0, s_sum);
}

// The same by a cluster of `blocks` blocks per unit-tensor, a range of its chunks each: few unit-tensors of many candidates leave most of
// the device to others otherwise (64 of 32k x 128 positions at keep 1/8: 119 us by a block each), and where every position is a candidate.
// Where all entries are kept there is nothing to look for.
template <typename T, int B>
__global__ void __launch_bounds__(kThrThreads) threshold_cluster_kernel(CompressArgs a, int ut_begin, int redo, int blocks) {
    __shared__ __align__(16) uint32_t s_hist[kThrBins], s_all[kThrBins];
    __shared__ uint32_t s_sum[2][32];
    __shared__ __align__(8) uint32_t s_range[2];
    constexpr bool F32KEY = !(sizeof(T) == 2 && B == 2);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = blockIdx.x % blocks, ut = ut_begin + blockIdx.x / blocks, chunks = a.chunks;
    const int c_begin = (int)((int64_t)chunks * rank / blocks), c_end = (int)((int64_t)chunks * (rank + 1) / blocks);
    SelState* const sel = a.sel + ut;
    chain_wait();
    if (redo && !sel->redo) return;  // (the same for the whole cluster, as every branch below)
    const int32_t* const cn = a.cand_n + (int64_t)ut * a.chunks_max;
    // the threads' sums of two counts over the cluster's first `ranks` blocks
    auto cluster_total = [&](uint32_t x, uint32_t y, int ranks) {
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
            y += __shfl_xor_sync(0xFFFFFFFFu, y, o);
        }
        __syncthreads();
        if (lane == 0) { s_sum[0][warp] = x; s_sum[1][warp] = y; }
        __syncthreads();
        if (tid == 0) {
            x = y = 0;
            for (int w = 0; w < kThrThreads / 32; ++w) { x += s_sum[0][w]; y += s_sum[1][w]; }
            s_range[0] = x;
            s_range[1] = y;
        }
        cluster_sync();
        const uint2 t = cluster_sum2((uint32_t)__cvta_generic_to_shared(s_range), ranks);
        cluster_sync();  // (before s_range is written again)
        return t;
    };
    auto each = [&](auto&& f) {
        int n = c_begin + warp < c_end ? cn[c_begin + warp] : 0;
        for (int c = c_begin + warp; c < c_end; c += kThrThreads / 32) {
            const int n_next = c + 32 < c_end ? cn[c + 32] : 0;
            f(c, n);
            n = n_next;
        }
    };
    // counts of f's bins over the cluster, the one where their running sum from the top reaches `target` and the count above it
    auto bin_of = [&](auto&& f, uint32_t target, uint32_t& bin, uint32_t& above) {
        for (int i = tid; i < kThrBins; i += kThrThreads) s_hist[i] = 0;
        __syncthreads();
        each([&](int c, int n) { each_candidate<T, B>(a, ut, c, n, f); });
        cluster_sync();
        for (int i = 2 * tid; i < kThrBins; i += 2 * kThrThreads)
            *reinterpret_cast<uint2*>(&s_all[i]) = cluster_sum2((uint32_t)__cvta_generic_to_shared(&s_hist[i]), blocks);
        cluster_sync();  // (before anybody's counts start again)
        return find_bin<kThrThreads, kThrBins>(s_all, target, bin, above);
    };
    uint32_t tau = a.n_keep > 0 ? 0u : kNoKey, need = (uint32_t)a.n_keep;  // (all of them: above 0 or equal to it)
    if (a.n_keep > 0 && a.n_keep < (int64_t)a.T * a.d) {
        uint32_t mine = 0;
        each([&](int, int n) { mine += lane == 0 ? (uint32_t)n : 0u; });
        const uint2 total = cluster_total(mine, 0, blocks);
        if ((int64_t)total.x < a.n_keep) {
            if (tid == 0 && rank == 0) { sel->redo = 1; sel->lo = 0; }
            return;
        }
        uint32_t k_rem = (uint32_t)a.n_keep, prefix, above, bin;
        for (uint32_t from = sel->lo >> 16;;) {
            const bool found = bin_of([&](uint32_t key) {
                const uint32_t k16 = key >> 16;
                if (k16 >= from) atomicAdd(&s_hist[min(k16 - from, (uint32_t)kThrBins - 1)], 1u);
            }, k_rem, bin, above);
            if (!found) {  // (every position is a candidate and the sample misled: from the smallest key on)
                from = 0;
                continue;
            }
            prefix = from + bin;
            if (bin < kThrBins - 1 || from + kThrBins - 1 >= 32767) break;
            from += kThrBins - 1;
        }
        k_rem -= above;
        if constexpr (F32KEY) {
            const uint32_t top = prefix;
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                const int shift = pass == 0 ? 4 : 0, bits = pass == 0 ? 12 : 4;
                const uint32_t want = pass == 0 ? top : prefix;
                bin_of([&](uint32_t key) {
                    if ((key >> (shift + bits)) == want) atomicAdd(&s_hist[(key >> shift) & ((1u << bits) - 1u)], 1u);
                }, k_rem, bin, above);
                prefix = (want << bits) | bin;
                k_rem -= above;
            }
        }
        tau = F32KEY ? prefix : prefix << 16;
        need = k_rem;
    }
    if (tid == 0 && rank == 0) { sel->tau = tau; sel->need = need; }
    // ---- keys above and equal to the threshold before every chunk ----
    int2* const base = a.chunk_base + (int64_t)ut * a.chunks_max;
    uint32_t range_gt = 0, range_eq = 0;
    each([&](int c, int n) {
        uint32_t both = 0;  // (see threshold_kernel)
        each_candidate<T, B>(a, ut, c, n, [&](uint32_t key) { both += key > tau ? 1u : key == tau ? 0x10000u : 0u; });
#pragma unroll
        for (int o = 16; o; o >>= 1) both += __shfl_xor_sync(0xFFFFFFFFu, both, o);
        if (lane == 0) {
            base[c] = make_int2((int)(both & 0xFFFFu), (int)(both >> 16));
            range_gt += both & 0xFFFFu;
            range_eq += both >> 16;
        }
    });
    const uint2 before = cluster_total(range_gt, range_eq, rank);  // of the blocks before this one
    scan_chunks(base, c_begin, c_end, before.x, before.y, s_sum);
}

// ---- 4: the lists -------------------------------------------------------------------------------------
// Packed entry of the bf16 / head_dim 128 decode kernel: low half = value bits, high half = (byte offset / 2) of the position
// inside a 16-token x 128-channel tile of two 64-channel halves with 128-byte rows whose 16-byte chunks are XOR-swizzled
// with the row.  p: position in a chunk (a whole number of tiles).
__device__ __forceinline__ uint32_t packed_place(uint32_t p) {
    const uint32_t half = (p >> 6) & 1u, row = (p >> 7) & 15u, chunk = ((p >> 3) ^ (p >> 7)) & 7u;
    return (half << 10 | row << 6 | chunk << 3 | (p & 7u)) << 16;
}

// grid (groups of eight chunks, unit-tensors), a chunk per warp: no block barriers.  A round takes 256 candidates, eight per lane (of float32
// blocks of four 128, four per lane): one warp scan of their counts, then positions and values of those that stay go through shared memory, so that the lists leave in runs.
// Bound by instructions: issue slots 80 % busy, HBM 24 % (counters on 4 layers of 32k tokens).  32 layers of 32k tokens (0.32 GB of candidates read,
// 0.67 GB of lists written) 300 -> 266 us, 8 blocks of four of 12 289 147 -> 130, against 32 candidates a round with two votes each.  (One chunk
// per block with a block scan per round took 767.)  Four candidates per lane where eight are 32 registers of values and as many of the next ones':
// with eight, float32 blocks of four had 119 registers and two blocks on an SM, 8 layers of 65 536 tokens 2 389 us in all, now 2 338.
template <typename T, int B, bool ALL>
__global__ void __launch_bounds__(256) compact_kernel(CompressArgs a, int ut_begin) {
    constexpr int NB = B == 4 ? 4 : 1, CE = compress_chunk(B, (int)sizeof(T)), WORDS = CE / 32;
    constexpr int PER = NB * sizeof(T) > 8 ? 4 : 8, Q = PER * (int)sizeof(T) / 16;  // candidates per lane and round; 16-byte vectors of theirs per layer
    constexpr uint32_t FULL = (1u << PER) - 1u;
    constexpr bool TWO = sizeof(T) == 2 && B == 2;
    __shared__ uint32_t s_map[8][WORDS];
    __shared__ __align__(16) uint16_t s_pos[8][32 * PER];
    __shared__ __align__(16) T s_val[8][NB][32 * PER];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ut = ut_begin + blockIdx.y, c = blockIdx.x * 8 + warp;
    chain_wait();
    if (c >= a.chunks) return;
    const bool map_k = a.keep && !(ut % a.tensors);  // K: a bit map of the kept positions
    uint32_t* const map = s_map[warp];
    if (map_k)
        for (int w = lane; w < WORDS; w += 32) map[w] = 0;
    const uint32_t tau = a.sel[ut].tau, need = a.sel[ut].need;
    const int n = a.cand_n[(int64_t)ut * a.chunks_max + c];
    const int2 b0 = a.chunk_base[(int64_t)ut * a.chunks_max + c];
    const int64_t e0 = (int64_t)c * CE, n_e = (int64_t)a.T * a.d;
    const uint2* const pos = reinterpret_cast<const uint2*>(a.cand_pos + (int64_t)ut * a.cand_stride + e0);
    const T* const val = reinterpret_cast<const T*>(a.cand_val) + (int64_t)ut * NB * a.cand_stride + e0;
    uint32_t run_gt = (uint32_t)b0.x, run_eq = (uint32_t)b0.y;
    int32_t* const idx = a.idx + (int64_t)ut * a.kcap;
    T* const out = reinterpret_cast<T*>(a.val) + (int64_t)ut * NB * a.kcap;
    uint32_t* const packed = sizeof(T) == 2 && a.packed ? a.packed + (int64_t)ut * NB * a.kcap : nullptr;
    const int tile_shift = a.d == 128 ? 11 : 10;  // positions of a 16-token tile
    int32_t* const off = a.tile_off + (int64_t)ut * (a.ntiles_max + 1) + (int)(e0 >> tile_shift);
    int tile = -1;  // of the entry before
    __syncwarp();
    uint2 p_next[PER / 4] = {};
    uint4 v_next[NB][Q];
    auto load = [&](int i) {
        if (i >= n) return;
        if constexpr (!ALL) {
            if constexpr (PER == 8) {
                const uint4 x = reinterpret_cast<const uint4*>(pos)[i >> 3];
                p_next[0] = make_uint2(x.x, x.y);
                p_next[PER / 4 - 1] = make_uint2(x.z, x.w);
            } else {
                p_next[0] = pos[i >> 2];
            }
        }
#pragma unroll
        for (int l = 0; l < NB; ++l)
#pragma unroll
            for (int k = 0; k < Q; ++k) v_next[l][k] = reinterpret_cast<const uint4*>(val + (int64_t)l * a.cand_stride + i)[k];
    };
    load(PER * lane);
    for (int base = 0; base < n; base += 32 * PER) {
        const int i = base + PER * lane;
        uint32_t pw[PER / 2];
#pragma unroll
        for (int k = 0; k < PER / 4; ++k) { pw[2 * k] = p_next[k].x; pw[2 * k + 1] = p_next[k].y; }
        uint4 v8[NB][Q];
#pragma unroll
        for (int l = 0; l < NB; ++l)
#pragma unroll
            for (int k = 0; k < Q; ++k) v8[l][k] = v_next[l][k];
        load(i + 32 * PER);
        const uint32_t valid = i >= n || tau == kNoKey ? 0u : n - i >= PER ? FULL : (1u << (n - i)) - 1u;
        uint32_t gt = 0, eq = 0;
        if constexpr (TWO) {
            gt = Eight<T, B>::reach(v8, tau + 0x10000u);
            eq = Eight<T, B>::reach(v8, tau) & ~gt;
        } else if constexpr (PER == 4) {
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                float h[NB];
#pragma unroll
                for (int l = 0; l < NB; ++l) h[l] = to_f32(reinterpret_cast<const T*>(&v8[l][0])[k]);
                const uint32_t key = key_of<B>(h);
                gt |= (uint32_t)(key > tau) << k;
                eq |= (uint32_t)(key == tau) << k;
            }
        } else {
            Eight<T, B>::keys(v8, [&](int k, uint32_t key) {
                gt |= (uint32_t)(key > tau) << k;
                eq |= (uint32_t)(key == tau) << k;
            });
        }
        gt &= valid;
        eq &= valid;
        const uint32_t cnt = (uint32_t)__popc(gt) << 16 | (uint32_t)__popc(eq);
        uint32_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31), before = incl - cnt;
        // ties in index order while fewer than `need` precede them
        const uint32_t eq_before = run_eq + (before & 0xFFFFu);
        const uint32_t first = run_gt + min(run_eq, need);  // list position of the round's first entry
        uint32_t kept = gt, ties = min((uint32_t)__popc(eq), need - min(eq_before, need));
        if (ties == (uint32_t)__popc(eq)) kept |= eq;
        else
            for (uint32_t rest = eq; ties; --ties, rest &= rest - 1) kept |= rest & (0u - rest);
        uint32_t at = run_gt + (before >> 16) + min(eq_before, need) - first;
        run_gt += total >> 16;
        run_eq += total & 0xFFFFu;
        const uint32_t n_out = run_gt + min(run_eq, need) - first;
        if (ALL && map_k && kept) atomicOr(&map[i >> 5], kept << (i & 31));  // (the lane's positions follow one another)
        if (ALL && kept == FULL && at % PER == 0) {
#pragma unroll
            for (int k = 0; k < PER; k += 2) reinterpret_cast<uint32_t*>(s_pos[warp])[(at + k) / 2] = (uint32_t)(i + k) | (uint32_t)(i + k + 1) << 16;
#pragma unroll
            for (int l = 0; l < NB; ++l)
#pragma unroll
                for (int k = 0; k < Q; ++k) reinterpret_cast<uint4*>(s_val[warp][l])[at * Q / PER + k] = v8[l][k];
        } else {
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                if (!(kept >> k & 1u)) continue;
                s_pos[warp][at] = ALL ? (uint16_t)(i + k) : (uint16_t)(pw[k >> 1] >> (16 * (k & 1)));
#pragma unroll
                for (int l = 0; l < NB; ++l) s_val[warp][l][at] = reinterpret_cast<const T*>(&v8[l][0])[k];
                ++at;
            }
        }
        __syncwarp();
        for (uint32_t j = lane; j < n_out; j += 32) {
            const uint32_t p = s_pos[warp][j];
            const int t = (int)(p >> tile_shift), t_before = j ? (int)(s_pos[warp][j - 1] >> tile_shift) : tile;
            for (int x = t_before + 1; x <= t; ++x) off[x] = (int32_t)(first + j);
            if (!ALL && map_k) atomicOr(&map[p >> 5], 1u << (p & 31));
            idx[first + j] = (int)e0 + (int)p;
            const uint32_t place = sizeof(T) == 2 ? packed_place(p) : 0u;
#pragma unroll
            for (int l = 0; l < NB; ++l) {
                const T raw = s_val[warp][l][j];
                out[(int64_t)l * a.kcap + first + j] = raw;
                // (a block of four scales its rows by 1/2 at decode time and its deviations by 1: twice the deviation is stored)
                if constexpr (sizeof(T) == 2)
                    if (packed) packed[(int64_t)l * a.kcap + first + j] = (__float_as_uint(B == 4 ? 2.f * to_f32(raw) : to_f32(raw)) >> 16) | place;
            }
        }
        if (n_out) tile = (int)(s_pos[warp][n_out - 1] >> tile_shift);
        __syncwarp();
    }
    // K: whole chunks (the map is padded like the candidate lists)
    if (map_k) {
        uint32_t* const keep = a.keep + (int64_t)(ut / a.tensors) * a.keep_stride + e0 / 32;
        for (int w = lane; w < WORDS; w += 32) keep[w] = map[w];
    }
    // tiles behind the last entry
    const int tiles = (int)((min((int64_t)CE, n_e - e0) + (1 << tile_shift) - 1) >> tile_shift);
    const uint32_t end = run_gt + min(run_eq, need);
    for (int x = tile + 1 + lane; x < tiles; x += 32) off[x] = (int32_t)end;
    if (lane == 0 && c == a.chunks - 1) {
        off[tiles] = (int32_t)end;
        if ((int64_t)end != a.n_keep) atomicMax(a.status, (int32_t)kFlagCountMismatch);
    }
}

// ---- all of it for a short unit-tensor ------------------------------------------------------------------
// One cluster per unit-tensor, a range of whole 16-token tiles per block, at most W x kSmallElems positions and fewer than 2^16: the
// high-frequency values stay in shared memory.  Every block adds up the cluster's histograms of the key's top 15 bits, a window of 32 octaves, from
// their shared memories; for bf16 pairs that is the threshold and says how many of the kept positions the blocks before have.  Wider
// keys: those that share the threshold's top half are gathered and looked through by every block, or counted in two more digits (10 and 6
// bits) where they are many.  A thread writes the entries of its W x 32 consecutive positions.  Bound by the chain of its steps (loads,
// cluster barriers with reads across the cluster between, block scans), not by bytes: one bf16 pair of 509 x 128 12.0 us with three exchanges, 9.4 with one (24.5 by the four kernels); 1000 x 128
// 32.8 -> 12.9 and eight of 900 x 128 47.9 -> 26.6 against the four kernels, with three exchanges.
// Taken while the clusters need two turns at most (two blocks fit an SM up to 88 KiB of values each): 32 tensors
// of blocks of four, 1000 x 128, two turns, 66 us against 64; 256 pairs of 1024 x 128, seven turns, 195 against 133.
// W: words of 32 positions per thread.  (Keys of few different values meet in the histogram's bins: two tensors of 1000 x 128, bf16 all equal 32.9 us,
// five values 16.5; float32 36.2 and 25.9; adding a thread's eight equal ones at once made the float32 32.5, and normal bf16 11.3 -> 11.8.)
constexpr int kSmallNear = 1024;  // keys that are gathered at most
// Of them are compared each with all others; digits among more.  (All compared, up to 1 024: 4096 x 128 float32 at keep 1/2 109.9 us, now 48.7;
// 1000 x 128 at keep 1/4, some 160 keys, 23.3 and 19.9.)
constexpr int kSmallRank = 128;
constexpr int kSmallThreads = 512, kSmallElems = 32 * kSmallThreads, kSmallSmem = 128 * 1024;

template <typename T, int B, int W>
__global__ void __launch_bounds__(kSmallThreads, W > 2 ? 1 : 2) small_kernel(CompressArgs a, int blocks, int range) {
    constexpr int NB = B == 4 ? 4 : 1, Q = Eight<T, B>::Q;
    constexpr bool TWO = sizeof(T) == 2 && B == 2;  // (the key's lower 16 bits are zero)
    constexpr int CH = 4 * Q;                       // 16-byte chunks of 32 positions
    constexpr int MOST = W == 1 ? 8 : 16;           // blocks of a cluster
    extern __shared__ __align__(16) uint8_t smem[];  // [NB][range] values, the chunks of a word of 32 positions swizzled
    // Histogram of the key's top 15 bits in a window (two counts of 16 bits a word), its sums over the cluster.  When the threshold's top half is
    // known the sums are done with: their place holds this block's keys with that top half, and then the cluster's, or the digits'
    // histograms.  (With arrays of their own blocks of four at 513 to 640 tokens had one block on an SM instead of two: 4 layers of 640
    // tokens, 16 heads 49.0 us against 29.8, 8 heads 33.8 against 25.5.)
    __shared__ __align__(16) uint32_t s_h1[2048], s_all[4096];
    uint16_t* const s_near = reinterpret_cast<uint16_t*>(s_all + 3072);  // [kSmallNear]
    static_assert(sizeof(s_h1) + sizeof(s_all) + 1024 + 88 * 1024 + 1024 <= 228 * 1024 / 2, "two blocks fit an SM with 88 KiB of values each");
    __shared__ uint32_t s_count, s_warp[kSmallThreads / 32], s_before[2][kSmallThreads / 32], s_n, s_off[17], s_low[2], s_below;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = blockIdx.x % blocks, item = blockIdx.x / blocks, uts = a.Hkv * a.tensors;
    const int ut = a.ut_base + item, blk = item / uts, u = item % uts, h = u / a.tensors, is_v = u % a.tensors;
    const int n_e = a.T * a.d, e0 = rank * range, n = max(0, min(range, n_e - e0));
    const int dshift = a.d == 128 ? 7 : 6;
    const int plane = range * (int)sizeof(T);
    const bool every = a.n_keep == n_e;  // all of them are kept: above zero or equal to it
    for (int i = tid; i < 2048; i += kSmallThreads) s_h1[i] = 0;
    if (tid == 0) s_n = 0;
    // a key's bin: 4 094 values of its top 15 bits above `from`, 32 octaves, the last bin for what is larger, the first for all others: zero (rows
    // that are the same in both layers, or padding) and what is below the window.  At first 2^-24 to 2^8, of energies 2^-16 to 2^16.
    uint32_t from = (127u - (B == 4 ? 16u : 24u)) << 7;
    auto count_key = [&](uint32_t key) {
        const uint32_t bin = min(max(key >> 16, from) - from, 4095u);
        atomicAdd(&s_h1[bin >> 1], 1u << (16 * (bin & 1)));  // (a block has fewer than 2^16 positions)
    };
    auto chunk_at = [&](int word, int j) { return (word * CH + (j ^ (Q == 1 ? (word >> 1) & 3 : word & 7))) * 16; };
    chain_wait();
    __syncthreads();
    const T* x[B];
#pragma unroll
    for (int l = 0; l < B; ++l) x[l] = reinterpret_cast<const T*>(is_v ? a.v[B * blk + l] : a.k[B * blk + l]) + (int64_t)h * a.stride_h;
    T* const z0 = reinterpret_cast<T*>(a.z0) + (int64_t)ut * a.z0_stride + e0;
    T* const z1 = a.z1 && !is_v ? reinterpret_cast<T*>(a.z1) + (int64_t)(ut / a.tensors) * NB * a.unit_stride + e0 : nullptr;
    constexpr int U = B == 4 ? 1 : 2;  // groups of eight whose rows are requested together
    for (int v0 = tid; v0 < n / 8; v0 += U * kSmallThreads) {
        uint4 f[U][B][Q];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int p = (v0 + q * kSmallThreads) * 8;
            if (p >= n) break;
            const int64_t off = (int64_t)((e0 + p) >> dshift) * a.stride_t + ((e0 + p) & (a.d - 1));
#pragma unroll
            for (int l = 0; l < B; ++l)
#pragma unroll
                for (int k = 0; k < Q; ++k) f[q][l][k] = reinterpret_cast<const uint4*>(x[l] + off)[k];
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int p = (v0 + q * kSmallThreads) * 8;
            if (p >= n) break;
            uint4 z[Q], hf[NB][Q];
            Eight<T, B>::split(f[q], z, hf);
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                reinterpret_cast<uint4*>(z0 + p)[k] = z[k];
#pragma unroll
                for (int l = 0; l < NB; ++l) {
                    if (z1) reinterpret_cast<uint4*>(z1 + (int64_t)l * a.unit_stride + p)[k] = hf[l][k];
                    *reinterpret_cast<uint4*>(smem + l * plane + chunk_at(p >> 5, ((p >> 3) & 3) * Q + k)) = hf[l][k];
                }
            }
            if (!every) Eight<T, B>::keys(hf, [&](int, uint32_t key) { count_key(key); });
        }
    }
    // f(w, i, key) for position i of the thread's word w, whose 32 positions are all there or none of them
    const int word0 = W * tid;
    auto each = [&](auto&& f) {
#pragma unroll
        for (int w = 0; w < W; ++w) {
            if (32 * (word0 + w) >= n) return;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                uint4 hf[NB][Q];
#pragma unroll
                for (int l = 0; l < NB; ++l)
#pragma unroll
                    for (int k = 0; k < Q; ++k) hf[l][k] = *reinterpret_cast<const uint4*>(smem + l * plane + chunk_at(word0 + w, g * Q + k));
                Eight<T, B>::keys(hf, [&](int i, uint32_t key) { f(w, 8 * g + i, key); });
            }
        }
    };
    // ---- the n_keep-th largest key of the cluster ----
    uint32_t tau = every ? 0u : kNoKey, need = every ? (uint32_t)n_e : 0u;
    uint32_t gt_before = every && tid == 0 ? (uint32_t)e0 : 0u, eq_before = 0;  // this thread's part of the counts of the blocks before this one
    bool counted = true;                                                        // (the same for the whole cluster)
    cluster_sync();
    if (a.n_keep > 0 && !every) {  // (the same for every block)
        // The blocks' histograms give the threshold's top half and, of the blocks before this one, how many keys are above it and equal to it:
        // for bf16 magnitudes one exchange in all.
        uint32_t bin, above, of_before[8];
        for (;;) {
            const uint32_t at = (uint32_t)__cvta_generic_to_shared(s_h1) + 16 * tid;  // four words, eight bins
            uint32_t all[8] = {};
#pragma unroll
            for (int i = 0; i < 8; ++i) of_before[i] = 0;
#pragma unroll
            for (int r0 = 0; r0 < MOST; r0 += 8) {
                if (r0 > 0 && r0 >= blocks) break;
                uint4 v[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    uint32_t remote;
                    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(at), "r"(r0 + r < blocks ? r0 + r : 0));
                    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[r].x), "=r"(v[r].y), "=r"(v[r].z), "=r"(v[r].w) : "r"(remote));
                }
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    if (r0 + r >= blocks) continue;
                    const uint32_t x[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t n_i = i & 1 ? x[i >> 1] >> 16 : x[i >> 1] & 0xFFFFu;
                        all[i] += n_i;
                        if (r0 + r < rank) of_before[i] += n_i;
                    }
                }
            }
            *reinterpret_cast<uint4*>(&s_all[8 * tid]) = make_uint4(all[0], all[1], all[2], all[3]);
            *reinterpret_cast<uint4*>(&s_all[8 * tid + 4]) = make_uint4(all[4], all[5], all[6], all[7]);
            __syncthreads();
            find_bin<kSmallThreads, 4096>(s_all, (uint32_t)a.n_keep, bin, above);
            if ((bin > 0 || from == 0) && (bin < 4095 || from + 4095 >= 32767)) break;
            if (bin == 0) {
                // the k-th is zero unless a key lies between zero and the window: a look at the keys instead of another window
                bool below = false;
                each([&](int, int, uint32_t key) { below |= key != 0 && key >> 16 <= from; });
                const int any = __syncthreads_or(below);
                if (tid == 0) s_below = any;
                cluster_sync();
                uint32_t at, v;
                asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(&s_below)), "r"(lane < blocks ? lane : 0));
                asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
                from = 0;
                if (!__any_sync(0xFFFFFFFFu, v != 0)) break;
            } else {
                from += 4094;
            }
            // another window (the same for the whole cluster): from the smallest key on, or above
            cluster_sync();
            for (int i = tid; i < 2048; i += kSmallThreads) s_h1[i] = 0;
            __syncthreads();
            each([&](int, int, uint32_t key) { count_key(key); });
            cluster_sync();
        }
        tau = (from + bin) << 16;
        need = (uint32_t)a.n_keep - above;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (8 * tid + i > (int)bin) gt_before += of_before[i];
            if (8 * tid + i == (int)bin) eq_before += of_before[i];
        }
        if constexpr (!TWO) {
            // The few keys with that top half (a 128th of an octave) are gathered, and every block looks through all of them: one more exchange
            // instead of two digits and the counts.  float32 pairs, us: 509 x 128 15.7 -> 13.8, 2048 x 128 31.5 -> 26.5.  Where many share it
            // (equal keys) the digits are counted by the cluster at once.
            const uint32_t top = from + bin, m = s_all[bin];
            uint32_t left = need;
            eq_before = 0;
            counted = m <= (uint32_t)kSmallNear;  // (the cluster's count: the same for all of its blocks)
            __syncthreads();                      // (the sums are read)
            if (counted) {
                each([&](int, int, uint32_t key) {
                    if (key >> 16 == top) s_near[atomicAdd(&s_n, 1u)] = (uint16_t)key;
                });
                cluster_sync();
                uint32_t mine_n = 0;
                {
                    uint32_t at;
                    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(&s_n)), "r"(lane < blocks ? lane : 0));
                    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(mine_n) : "r"(at) : "memory");
                    if (lane >= blocks) mine_n = 0;
                }
                uint32_t off_n = mine_n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, off_n, o);
                    if (lane >= o) off_n += y;
                }
                if (warp == 0 && lane < 17) s_off[lane] = off_n - mine_n;  // ([blocks, 16]: all of them)
                __syncthreads();
                for (uint32_t i = tid; i < m; i += kSmallThreads) {
                    int r = 0;
#pragma unroll
                    for (int k = 1; k < MOST; ++k) r += k < blocks && s_off[k] <= i;
                    uint32_t at;
                    uint16_t low;
                    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(s_near) + 2 * (i - s_off[r])), "r"(r));
                    asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(low) : "r"(at) : "memory");
                    s_all[i] = (uint32_t)low | (uint32_t)r << 16;
                }
                __syncthreads();
                uint32_t low = 0;
                if (m <= (uint32_t)kSmallRank) {  // each against all others
                    for (uint32_t i = tid; i < m; i += kSmallThreads) {
                        const uint32_t one = s_all[i] & 0xFFFFu;
                        uint32_t g = 0, e = 0;
#pragma unroll 2
                        for (uint32_t k = 0; k < m; k += 4) {
                            const uint4 v = *reinterpret_cast<const uint4*>(&s_all[k]);
                            const uint32_t other[4] = {v.x & 0xFFFFu, v.y & 0xFFFFu, v.z & 0xFFFFu, v.w & 0xFFFFu};
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                g += k + q < m && other[q] > one;
                                e += k + q < m && other[q] == one;
                            }
                        }
                        if (g < left && left <= g + e) { s_low[0] = one; s_low[1] = g; }
                    }
                    __syncthreads();
                    low = s_low[0];
                    left -= s_low[1];
                } else {  // digits of 10 and 6 bits among them
#pragma unroll 1
                    for (int shift = 6; shift >= 0; shift -= 6) {
                        for (int i = tid; i < 1024; i += kSmallThreads) s_all[2048 + i] = 0;
                        __syncthreads();
                        for (uint32_t i = tid; i < m; i += kSmallThreads) {
                            const uint32_t one = s_all[i] & 0xFFFFu;
                            if (shift || one >> 6 == low) atomicAdd(&s_all[2048 + (shift ? one >> 6 : one & 63u)], 1u);
                        }
                        __syncthreads();
                        find_bin<kSmallThreads, 1024>(s_all + 2048, left, bin, above);
                        low = low << 6 | bin;
                        left -= above;
                    }
                }
                tau = top << 16 | low;
                need = left;
                for (uint32_t i = tid; i < m; i += kSmallThreads) {
                    const uint32_t one = s_all[i] & 0xFFFFu;
                    if ((int)(s_all[i] >> 16) < rank) {
                        gt_before += one > low;
                        eq_before += one == low;
                    }
                }
            } else {  // digits of 10 and 6 bits
                tau = top;
                for (int i = tid; i < 2048; i += kSmallThreads) s_all[i] = 0;
                __syncthreads();
                auto level = [&](uint32_t* hist, int shift, int bits) {
                    each([&](int, int, uint32_t key) { if (key >> (shift + bits) == tau) atomicAdd(&hist[key >> shift & ((1u << bits) - 1u)], 1u); });
                    cluster_sync();
                    *reinterpret_cast<uint2*>(&s_all[2048 + 2 * tid]) = cluster_sum2<MOST>((uint32_t)__cvta_generic_to_shared(hist) + 8 * tid, blocks);
                    __syncthreads();
                    find_bin<kSmallThreads, 1024>(s_all + 2048, left, bin, above);
                    left -= above;
                    tau = tau << bits | bin;
                };
                level(s_all, 6, 10);
                level(s_all + 1024, 0, 6);
                need = left;  // of the positions whose key is tau, the lowest
            }
        }
    }
    // ---- entries: those above in the blocks, warps and threads before, then those equal (counts in halves: a block has fewer than 2^16) ----
    uint32_t gt[W] = {}, eq[W] = {}, cnt = 0;
    each([&](int w, int i, uint32_t key) {
        gt[w] |= (uint32_t)(key > tau) << i;
        eq[w] |= (uint32_t)(key == tau) << i;
    });
#pragma unroll
    for (int w = 0; w < W; ++w) cnt += (uint32_t)__popc(gt[w]) << 16 | (uint32_t)__popc(eq[w]);
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    gt_before = __reduce_add_sync(0xFFFFFFFFu, gt_before);
    eq_before = __reduce_add_sync(0xFFFFFFFFu, eq_before);
    if (lane == 0) { s_before[0][warp] = gt_before; s_before[1][warp] = eq_before; }
    __syncthreads();
    uint32_t before = incl - cnt, total = 0;
#pragma unroll
    for (int w = 0; w < kSmallThreads / 32; ++w) {
        if (w < warp) before += s_warp[w];
        total += s_warp[w];
    }
    uint32_t run_gt = before >> 16, run_eq = before & 0xFFFFu;
    if (counted) {
#pragma unroll
        for (int w = 0; w < kSmallThreads / 32; ++w) { run_gt += s_before[0][w]; run_eq += s_before[1][w]; }
    } else {
        if (tid == 0) s_count = total;
        cluster_sync();
        uint32_t at, v;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(&s_count)), "r"(lane < rank ? lane : rank));
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
        if (lane >= rank) v = 0;
        run_gt += __reduce_add_sync(0xFFFFFFFFu, v >> 16);
        run_eq += __reduce_add_sync(0xFFFFFFFFu, v & 0xFFFFu);
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // (nothing is read from another block after this)
    int32_t* const idx = a.idx + (int64_t)ut * a.kcap;
    T* const out = reinterpret_cast<T*>(a.val) + (int64_t)ut * NB * a.kcap;
    uint32_t* const packed = sizeof(T) == 2 && a.packed ? a.packed + (int64_t)ut * NB * a.kcap : nullptr;
    const int tile_words = kResTile * a.d / 32;
    int32_t* const off = a.tile_off + (int64_t)ut * (a.ntiles_max + 1);
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const int word = word0 + w;
        if (32 * word >= n) break;
        uint32_t at = run_gt + min(run_eq, need);
        if (word % tile_words == 0) off[(e0 / 32 + word) / tile_words] = (int32_t)at;
        // the ties that are kept: while fewer than `need` precede them
        const int ties = (int)min((uint32_t)__popc(eq[w]), need - min(run_eq, need));
        uint32_t kept = gt[w], rest = eq[w];
        for (int i = 0; i < ties; ++i) {
            kept |= rest & (0u - rest);
            rest &= rest - 1;
        }
        run_gt += (uint32_t)__popc(gt[w]);
        run_eq += (uint32_t)__popc(eq[w]);
        if (a.keep && !is_v) a.keep[(int64_t)(ut / a.tensors) * a.keep_stride + e0 / 32 + word] = kept;
        for (uint32_t bits = kept; bits; bits &= bits - 1, ++at) {
            const int i = __ffs((int)bits) - 1, p = 32 * word + i;
            idx[at] = e0 + p;
            const uint32_t place = sizeof(T) == 2 ? packed_place((uint32_t)p) : 0u;
            constexpr int PER = 16 / (int)sizeof(T);
            const int from = chunk_at(word, i / PER) + (i % PER) * (int)sizeof(T);
#pragma unroll
            for (int l = 0; l < NB; ++l) {
                const T raw = *reinterpret_cast<const T*>(smem + l * plane + from);
                out[(int64_t)l * a.kcap + at] = raw;
                // (a block of four scales its rows by 1/2 at decode time and its deviations by 1: twice the deviation is stored)
                if constexpr (sizeof(T) == 2)
                    if (packed) packed[(int64_t)l * a.kcap + at] = (__float_as_uint(B == 4 ? 2.f * to_f32(raw) : to_f32(raw)) >> 16) | place;
            }
        }
        if (e0 + 32 * (word + 1) == n_e) {  // the last positions of all
            off[(n_e / 32 + tile_words - 1) / tile_words] = (int32_t)at;
            if ((int64_t)at != a.n_keep) atomicMax(a.status, (int32_t)kFlagCountMismatch);
        }
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename... A>
cudaError_t launch_chain(int cluster, void (*kernel)(A...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster ? 2 : 1;
    count_launch(1);
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Words of 32 positions per thread of a cluster of sixteen at most: with four bytes a position or more two words fill the shared memory.
template <typename T, int B>
constexpr int most_words() { return sizeof(T) == 2 && B == 2 ? 4 : 2; }
typedef void (*SmallKernel)(CompressArgs, int, int);
template <typename T, int B>
SmallKernel small_of(int words) {
    if constexpr (most_words<T, B>() == 4)
        if (words == 4) return small_kernel<T, B, 4>;
    return words == 2 ? small_kernel<T, B, 2> : small_kernel<T, B, 1>;
}

template <typename T, int B>
cudaError_t compress(CompressArgs& a, const void* const* k_layers, const void* const* v_layers, int block_begin, int block_end, cudaStream_t st) {
    static PerDevice once;
    constexpr int kMostWords = most_words<T, B>();
    static std::atomic<int> long_clusters[PerDevice::kMaxDevices][2][kSmallSmem / 4096 + 1];  // [two or four words][4 KiB of shared memory]; 0: not known
    int sms = 0;
    constexpr int CE = compress_chunk(B, (int)sizeof(T));
    const size_t smem = 2 * (size_t)B * CE * sizeof(T) + (B == 4 ? CE * sizeof(uint16_t) : 0);  // (a block of four: room for positions)
    cudaError_t e = once.ensure([&]() {
        cudaError_t e1 = cudaFuncSetAttribute(split_kernel<T, B, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e1 == cudaSuccess) e1 = cudaFuncSetAttribute(threshold_kernel<T, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, kThrMini * 128);
        if (e1 == cudaSuccess) e1 = cudaFuncSetAttribute(split_kernel<T, B, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        for (int w = 1; w <= kMostWords && e1 == cudaSuccess; w *= 2) {
            e1 = cudaFuncSetAttribute(small_of<T, B>(w), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmem);
            if (e1 == cudaSuccess && w > 1) e1 = cudaFuncSetAttribute(small_of<T, B>(w), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        }
        return e1;
    }, &sms);
    if (e != cudaSuccess) return e;
    const int64_t n = (int64_t)a.T * a.d;
    a.chunks = (int)((n + CE - 1) / CE);
    // few short unit-tensors: a cluster each, of as many blocks as have a tile, two blocks per SM
    const int tile_e = kResTile * a.d;
    const int64_t tiles = (n + tile_e - 1) / tile_e;
    const int uts = a.Hkv * a.tensors, n_ut = uts * (block_end - block_begin);
    // (blocks of four with nearly all entries: a thread writes too many of its own; 1000 x 128 293 and 108 us, 300 x 128 68 and 87)
    const bool few = B == 2 || (double)a.n_keep <= kAllShare * (double)n || n <= 40 * 1024;
    int cluster = 8, words = 1;
    while (cluster > tiles) cluster /= 2;
    int64_t range = 0;
    size_t small_smem = 0;
    auto fits = [&]() {
        range = (tiles + cluster - 1) / cluster * tile_e;
        small_smem = (size_t)range * (B == 4 ? 4 : 1) * sizeof(T);
        return range <= (int64_t)words * kSmallElems && range < 65536 && small_smem <= (size_t)kSmallSmem;  // (counts of 16 bits)
    };
    bool small = few && fits() && (int64_t)cluster * n_ut <= 2 * sms;
    // Longer ones take clusters of sixteen blocks, two or four words of positions per thread, while all of the clusters run at one
    // time (us, one tensor, keep 1/16, against the four kernels: bf16 192k positions 33.7 -> 16.1, 512k 39.9 -> 21.1; float32 256k 44.7 -> 31.5, 512k
    // 55.9 -> 36.6).  Where everything is kept a thread's entries are many and there is nothing to select: up to 384 Ki positions in all (one
    // bf16 tensor of 384k 54.6 us, four kernels 66.6, 512k 84.6 and 66.8; float32 39.6 and 53.1, 66.0 and 63.1; eight bf16 tensors of 256k 103.9 and 91.5).
    if (few && !small && (int64_t)16 * n_ut <= 2 * sms && tiles >= 16 && (a.n_keep < n || n * n_ut <= 384 * 1024)) {
        cluster = 16;
        for (words = 2; words < kMostWords && !fits();) words *= 2;
        if (fits()) {
            const int wi = words / 4, bucket = (int)((small_smem + 4095) / 4096);
            int dev = 0, at_once = 0;
            if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
            if ((at_once = long_clusters[dev][wi][bucket].load(std::memory_order_relaxed)) == 0) {  // (asked once per amount of shared memory)
                cudaLaunchConfig_t q = {};
                q.gridDim = dim3(16);
                q.blockDim = dim3(kSmallThreads);
                q.dynamicSmemBytes = (size_t)bucket * 4096;
                cudaLaunchAttribute attr[1];
                attr[0].id = cudaLaunchAttributeClusterDimension;
                attr[0].val.clusterDim.x = 16; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
                q.attrs = attr;
                q.numAttrs = 1;
                if ((e = cudaOccupancyMaxActiveClusters(&at_once, small_of<T, B>(words), &q)) != cudaSuccess) return e;
                long_clusters[dev][wi][bucket].store(at_once > 0 ? at_once : -1, std::memory_order_relaxed);
            }
            small = n_ut <= at_once;
        }
    }
    if (small) {
        // A few clusters take an SM per block: they are put two on an SM otherwise while others are idle (eight tensors, 600 tokens: blocks of four 20.3
        // -> 18.1 us, bf16 pairs 12.2 -> 11.0).  Sixteen clusters of eight do not fit that way.
        if (cluster == 8 && n_ut <= 8) small_smem = std::max<size_t>(small_smem, 92 * 1024);
        const SmallKernel kernel = small_of<T, B>(words);
        for (int b0 = block_begin; b0 < block_end; b0 += kSplitLayers / B) {
            const int nb = std::min(block_end - b0, kSplitLayers / B);
            for (int l = 0; l < nb * B; ++l) {
                a.k[l] = k_layers[B * b0 + l];
                a.v[l] = v_layers[B * b0 + l];
            }
            a.ut_base = b0 * uts;
            if ((e = launch_chain(cluster, kernel, dim3(cluster * uts * nb), kSmallThreads, small_smem, st, a, cluster, (int)range)) != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    const int ut_begin = block_begin * uts, ut_count = (block_end - block_begin) * uts;
    const int n_rows = (int)std::min<int64_t>(a.T, std::max<int64_t>(1, kSampleElems / a.d));
    const bool exact = n_rows == a.T;
    const double expect = (double)a.n_keep * n_rows / a.T;
    const bool all = a.in_place || (double)a.n_keep > kAllShare * (double)n;
    // about 1.2 k candidates (and four standard deviations of a small sample on top); a sample of everything is exact
    const uint32_t target = exact ? (uint32_t)a.n_keep : (uint32_t)std::ceil(1.2 * expect + 4.0 * std::sqrt(expect) + 16.0);
    const uint32_t among = (uint32_t)std::ceil(std::max(0.0, expect - 2.0 * std::sqrt(expect)));  // of the sample, at least, of the k largest
    // blocks per unit-tensor for the threshold: one per SM, where each has a chunk per warp or the candidates are all.  (Two per SM leave
    // clusters waiting: 32 tensors of 32k x 128, eight blocks each 316 us, four 277; keep 1/2 724 and 653.)
    // The joins cost about 5 us a digit: 64 lists of 98k entries 147 -> 136 us, of 65k 263 -> 278, one of 33k float32 entries 57 -> 67.
    constexpr int kDigits = sizeof(T) == 2 && B == 2 ? 1 : 3;
    int blocks = all || a.n_keep >= 96 * 1024 * (kDigits + 1) / 2 ? 8 : 1;
    while (blocks > 1 && ((int64_t)blocks * ut_count > sms || a.chunks < (all ? 4 : 32) * blocks)) blocks /= 2;
    const size_t thr_smem = kDigits == 1 ? (a.chunks <= kThrMini ? (size_t)a.chunks * 128 : 0) : (size_t)kThrBins * 4;
    // (items are counted in 32 bits)
    const int per_launch = (int)std::max<int64_t>(1, std::min<int64_t>(kSplitLayers / B, 0x7FFFFFFF / ((int64_t)a.chunks * uts) / 4));
    for (int redo = 0; redo < (all || exact || a.n_keep == 0 ? 1 : 2); ++redo) {
        for (int b0 = block_begin; b0 < block_end; b0 += per_launch) {
            const int nb = std::min(block_end - b0, per_launch);
            for (int l = 0; l < nb * B; ++l) {
                a.k[l] = k_layers[B * b0 + l];
                a.v[l] = v_layers[B * b0 + l];
            }
            a.ut_base = b0 * uts;
            if (!redo && (e = launch_chain(0, sample_kernel<T, B>, dim3(uts, nb), kSampleThreads, 0, st, a, n_rows, target, among)) != cudaSuccess) return e;
            const int items = a.chunks * uts * nb;
            if ((e = launch_chain(0, all ? split_kernel<T, B, true> : split_kernel<T, B, false>, dim3(std::min(items, 3 * sms)), kSplitThreads, smem, st, a, items,
                                  redo)) != cudaSuccess)
                return e;
        }
        e = all || blocks > 1 ? launch_chain(blocks, threshold_cluster_kernel<T, B>, dim3(ut_count * blocks), kThrThreads, 0, st, a, ut_begin, redo, blocks)
                              : launch_chain(0, threshold_kernel<T, B>, dim3(ut_count), kThrThreads, thr_smem, st, a, ut_begin, redo);
        if (e != cudaSuccess) return e;
    }
    constexpr int kMostRows = 65535;  // of a grid
    for (int u0 = 0; u0 < ut_count; u0 += kMostRows) {
        const dim3 grid((a.chunks + 7) / 8, std::min(ut_count - u0, kMostRows));
        if ((e = launch_chain(0, all ? compact_kernel<T, B, true> : compact_kernel<T, B, false>, grid, 256, 0, st, a, ut_begin + u0)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_compress(CompressArgs& a, int B, int dtype, const void* const* k_layers, const void* const* v_layers, int block_begin, int block_end,
                            cudaStream_t st) {
    if (a.T <= 0 || block_end <= block_begin) return cudaSuccess;
    if (dtype == FDKV_BF16)
        return B == 4 ? compress<__nv_bfloat16, 4>(a, k_layers, v_layers, block_begin, block_end, st)
                      : compress<__nv_bfloat16, 2>(a, k_layers, v_layers, block_begin, block_end, st);
    return B == 4 ? compress<float, 4>(a, k_layers, v_layers, block_begin, block_end, st)
                  : compress<float, 2>(a, k_layers, v_layers, block_begin, block_end, st);
}

}  // namespace fdkv
