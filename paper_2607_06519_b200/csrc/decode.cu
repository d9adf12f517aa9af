// Decode attention over the compressed cache (the fused reconstruct-and-attend step after Eq. 3):
// split-K partial attention with per-mode reconstruction (which also appends the generated token), split-K combine.
// This file holds the portable kernel (float32 or bf16 storage, head_dim 64/128, any group size up to 8);
// the bulk-copy / tensor-core kernel for bf16, head_dim 128 lives in decode_fast.cu.
#include <algorithm>
#include <type_traits>

#include "fdkv_internal.h"

namespace fdkv {

namespace {

template <typename T>
__device__ __forceinline__ float ldf(const T* p);
template <>
__device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <>
__device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// eight consecutive channels of a row
__device__ __forceinline__ void load8(const float* p, float (&f)[8]) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&f)[8]) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        f[2 * i] = __uint_as_float(w[i] << 16);
        f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
}

template <typename ACC>
__device__ __forceinline__ ACC dot8(const float (&x)[8], const float (&y)[8]) {
    ACC a = (ACC)x[0] * (ACC)y[0], b = (ACC)x[4] * (ACC)y[4];
#pragma unroll
    for (int i = 1; i < 4; ++i) {
        a = fma((ACC)x[i], (ACC)y[i], a);
        b = fma((ACC)x[i + 4], (ACC)y[i + 4], b);
    }
    return a + b;
}

constexpr int kWarps = 8;
constexpr int kParts = 4;  // floats before a part's accumulators: max, sum, 2 pad

// grid (splits, Hkv, batch); eight warps, each on whole 16-token tiles (the granularity of the residual lists).  D / 8 lanes
// share a token, eight channels each, so a warp works on 256 / D tokens at a time; every such lane group keeps a softmax
// state of its own (maximum, sum, D accumulators) over the tokens it meets, and the groups are joined once at the end:
// a score costs log2(D / 8) shuffles per head and the weighted sum of V none.  A residual tile is scattered into a zeroed
// float32 tile in shared memory and read beside the rows.  Bound by latency at the sizes this path serves:
// a tile's K and V rows are requested together, and the split gives every warp few tiles.
// A layer of 4 099 tokens, two KV heads of two query heads, float32 / 64 channels: 36.9 -> 9.5 us against one lane group per
// warp with a five-step reduction per token and head, 32-token tiles and shared-memory atomics for the residual, in a few
// blocks, and an append kernel of its own; bf16 with 8 query heads per KV head at 6 000 tokens 70.7 -> 11.1.
template <typename T, int D, int G>
__global__ void __launch_bounds__(kWarps * 32, G <= 2 && sizeof(T) == 2 ? 2 : 1) decode_generic_kernel(DecodeArgs a, int splits) {
    // float32 storage: logits of a few tens, whose rounding the exponential magnifies to more than the outputs' own; float64
    // products cost nothing here (less than 1 % of the time)
    using ACC = typename std::conditional<sizeof(T) == 4, double, float>::type;
    constexpr int LPT = D / 8;         // lanes per token
    constexpr int TPI = 32 / LPT;      // tokens per step
    constexpr int STEPS = kResTile / TPI;
    constexpr int PF = D == 128 ? (G == 8 ? 2 : 4) : STEPS;  // steps whose rows are requested together
    extern __shared__ __align__(16) float smem[];  // [kWarps][16][D] residual tiles; at the end the warps' accumulators [kWarps][G][D]
    __shared__ float s_m[kWarps][G], s_l[kWarps][G];
    const int split = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = lane / LPT, c0 = (lane % LPT) * 8;
    float* const tilez = smem + warp * (kResTile * D);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const UnitDesc u = a.desc[((int64_t)b * a.L + a.layer) * a.Hkv + h];  // (static since commit)
    const bool coef = u.mode != FDKV_MODE_EXACT;
    const bool resid = u.mode == FDKV_MODE_RESIDUAL;
    const int ntiles = (u.T + kResTile - 1) / kResTile;
    const int per = (ntiles + splits - 1) / splits;
    const int j0 = min(ntiles, split * per), j1 = min(ntiles, j0 + per);
    asm volatile("griddepcontrol.wait;" ::: "memory");  // q, the tails and the parts belong to the kernels ahead
    const T* const qg = reinterpret_cast<const T*>(a.q) + ((int64_t)b * a.Hq + h * G) * D + c0;
    float q[G][8], acc[G][8], m[G], l[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        load8(qg + g * D, q[g]);
        m[g] = -INFINITY;
        l[g] = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[g][i] = 0.f;
    }
    const float inv_sqrt_d = rsqrtf((float)D);

    // adds the residual of this tile (K or V side) to the zeroed shared-memory tile
    auto scatter = [&](int jt, const int32_t* idx, const void* vals, const int32_t* off) {
        const int e0 = off[jt], e1 = off[jt + 1];
#pragma unroll
        for (int i = 0; i < kResTile * D / 4; i += 32) *reinterpret_cast<float4*>(tilez + (i + lane) * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();
        const T* const val = reinterpret_cast<const T*>(vals);
        if (u.res_kind == 1) {  // whole rows of selected tokens
            for (int e = e0; e < e1; ++e) {
                const int tt = idx[e] - jt * kResTile;
                for (int c = lane; c < D; c += 32) tilez[tt * D + c] = ldf<T>(val + (int64_t)e * D + c);
            }
        } else {
            const int base = jt * kResTile * D;
            for (int e = e0 + lane; e < e1; e += 32) tilez[idx[e] - base] = ldf<T>(val + e);
        }
        __syncwarp();
    };
    // one tile: rows [0, nrows) of kb / vb (rows behind the last are read as the last and masked)
    auto tile = [&](const T* kb, const T* vb, int nrows, float kscale, float vscale, bool with_res, int jt) {
        float p[G][STEPS], kf[PF][8], vf[PF][8];
#pragma unroll
        for (int s0 = 0; s0 < STEPS; s0 += PF) {
#pragma unroll
            for (int s = 0; s < PF; ++s) {
                const int t = min((s0 + s) * TPI + grp, nrows - 1);
                load8(kb + (int64_t)t * D + c0, kf[s]);
                if (s0 == 0) load8(vb + (int64_t)t * D + c0, vf[s]);
            }
            if (with_res && s0 == 0) scatter(jt, u.k_idx, u.k_val, u.k_off);
#pragma unroll
            for (int s = 0; s < PF; ++s) {
                const int t = (s0 + s) * TPI + grp;
                // the residual's product is its own sum: adding it to the row first would round every coefficient once more
                float z[8];
                if (with_res) load8(tilez + t * D + c0, z);
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    ACC d = dot8<ACC>(q[g], kf[s]);
                    if (with_res) d = fma((ACC)u.sign, dot8<ACC>(q[g], z), d);
#pragma unroll
                    for (int o = LPT / 2; o; o >>= 1) d += __shfl_xor_sync(0xFFFFFFFFu, d, o);
                    p[g][s0 + s] = t < nrows ? (float)d * kscale : -INFINITY;
                }
            }
        }
        if (with_res) {
            __syncwarp();
            scatter(jt, u.v_idx ? u.v_idx : u.k_idx, u.v_val, u.v_off ? u.v_off : u.k_off);
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            float mx = m[g];
#pragma unroll
            for (int s = 0; s < STEPS; ++s) mx = fmaxf(mx, p[g][s]);
            if (mx > m[g]) {
                const float alpha = __expf(m[g] - mx);
                l[g] *= alpha;
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[g][i] *= alpha;
                m[g] = mx;
            }
#pragma unroll
            for (int s = 0; s < STEPS; ++s) {
                p[g][s] = p[g][s] == -INFINITY ? 0.f : __expf(p[g][s] - mx);
                l[g] += p[g][s];
                p[g][s] *= vscale;
            }
        }
#pragma unroll
        for (int s0 = 0; s0 < STEPS; s0 += PF) {
            if (s0 > 0)
#pragma unroll
                for (int s = 0; s < PF; ++s) load8(vb + (int64_t)min((s0 + s) * TPI + grp, nrows - 1) * D + c0, vf[s]);
#pragma unroll
            for (int s = 0; s < PF; ++s) {
                if (with_res) {
                    float z[8];
                    load8(tilez + ((s0 + s) * TPI + grp) * D + c0, z);
#pragma unroll
                    for (int i = 0; i < 8; ++i) vf[s][i] = fmaf(u.sign, z[i], vf[s][i]);
                }
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int i = 0; i < 8; ++i) acc[g][i] = fmaf(p[g][s0 + s], vf[s][i], acc[g][i]);
            }
        }
        if (with_res) __syncwarp();
    };

    // ---- prefill rows of this split ----
    {
        const T* kr = reinterpret_cast<const T*>(u.k_rows);
        const T* vr = reinterpret_cast<const T*>(u.v_rows);
        const float kscale = coef ? u.scale * inv_sqrt_d : inv_sqrt_d, vscale = coef ? u.scale : 1.f;
        for (int jt = j0 + warp; jt < j1; jt += kWarps) {
            const int t0 = jt * kResTile;
            tile(kr + (int64_t)t0 * D, vr + (int64_t)t0 * D, min(kResTile, u.T - t0), kscale, vscale, resid, jt);
        }
    }
    // ---- uncompressed tail rows (last split only) ----
    if (split == splits - 1) {
        int n = min(a.tail_len[a.layer * a.max_batch + b], a.max_tail);
        const int64_t o = (((int64_t)a.layer * a.max_batch + b) * a.Hkv + h) * a.tail_rows * D;
        T* tk = reinterpret_cast<T*>(a.tail_k) + o;
        T* tv = reinterpret_cast<T*>(a.tail_v) + o;
        if (a.k_new) {  // this call's row joins the tail here (the length is advanced by the combine kernel)
            if (n < a.max_tail) {
                for (int c = threadIdx.x; c < D; c += kWarps * 32) {
                    const int64_t src = ((int64_t)b * a.Hkv + h) * D + c;
                    tk[(int64_t)n * D + c] = reinterpret_cast<const T*>(a.k_new)[src];
                    tv[(int64_t)n * D + c] = reinterpret_cast<const T*>(a.v_new)[src];
                }
                ++n;
            } else if (threadIdx.x == 0) {
                atomicMax(a.status, (int32_t)kFlagTailFull);
            }
            __syncthreads();
        }
        for (int t0 = warp * kResTile; t0 < n; t0 += kWarps * kResTile)
            tile(tk + (int64_t)t0 * D, tv + (int64_t)t0 * D, min(kResTile, n - t0), inv_sqrt_d, 1.f, false, 0);
    }

    // ---- join the lane groups, then the warps, and write the split's part ----
#pragma unroll
    for (int g = 0; g < G; ++g) {
        float M = m[g];
#pragma unroll
        for (int o = LPT; o < 32; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, o));
        const float f = m[g] == -INFINITY ? 0.f : __expf(m[g] - M);
        l[g] *= f;
#pragma unroll
        for (int o = LPT; o < 32; o <<= 1) l[g] += __shfl_xor_sync(0xFFFFFFFFu, l[g], o);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            acc[g][i] *= f;
#pragma unroll
            for (int o = LPT; o < 32; o <<= 1) acc[g][i] += __shfl_xor_sync(0xFFFFFFFFu, acc[g][i], o);
        }
        m[g] = M;
    }
    __syncthreads();  // (the residual tiles are read)
    float* const s_acc = smem + warp * G * D;
    if (grp == 0)
#pragma unroll
        for (int g = 0; g < G; ++g) {
            *reinterpret_cast<float4*>(s_acc + g * D + c0) = make_float4(acc[g][0], acc[g][1], acc[g][2], acc[g][3]);
            *reinterpret_cast<float4*>(s_acc + g * D + c0 + 4) = make_float4(acc[g][4], acc[g][5], acc[g][6], acc[g][7]);
            if (lane == 0) { s_m[warp][g] = m[g]; s_l[warp][g] = l[g]; }
        }
    __syncthreads();
    for (int i = threadIdx.x; i < G * D; i += kWarps * 32) {
        const int g = i / D, ch = i % D;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) M = fmaxf(M, s_m[w][g]);
        float L = 0.f, A = 0.f;
        if (M != -INFINITY)
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const float f = s_m[w][g] == -INFINITY ? 0.f : __expf(s_m[w][g] - M);
                L = fmaf(s_l[w][g], f, L);
                A = fmaf(smem[(w * G + g) * D + ch], f, A);
            }
        float* part = a.partials + (((int64_t)b * a.Hq + h * G + g) * kMaxSplits + split) * (D + kParts);
        if (ch == 0) { part[0] = M; part[1] = L; }
        part[kParts + ch] = A;
    }
}

// out = sum_s e^{m_s - M} acc_s / sum_s e^{m_s - M} l_s.  grid (D / 32, Hq, batch), eight warps: lane = channel, the warps take
// every eighth part, so that a head's parts are read in a few rounds of loads.  Also advances the tail lengths of a call
// that appended.
template <int D>
__global__ void __launch_bounds__(256) combine_kernel(DecodeArgs a, int splits) {
    __shared__ float s_m[8], s_l[8], s_a[8][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.y, b = blockIdx.z, ch = blockIdx.x * 32 + lane;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const float* p = a.partials + ((int64_t)b * a.Hq + i) * kMaxSplits * (D + kParts);
    float M = -INFINITY, L = 0.f, A = 0.f;
    for (int s0 = warp; s0 < splits; s0 += 32) {
        float ms[4], ls[4], as[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool on = s0 + 8 * k < splits;
            const float* ps = p + (int64_t)(on ? s0 + 8 * k : s0) * (D + kParts);
            ms[k] = on ? __ldcg(ps) : -INFINITY;
            ls[k] = on ? __ldcg(ps + 1) : 0.f;
            as[k] = on ? __ldcg(ps + kParts + ch) : 0.f;
        }
        const float Mn = fmaxf(fmaxf(M, fmaxf(ms[0], ms[1])), fmaxf(ms[2], ms[3]));
        if (Mn == -INFINITY) continue;
        const float f = M == -INFINITY ? 0.f : __expf(M - Mn);
        L *= f;
        A *= f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float w = ms[k] == -INFINITY ? 0.f : __expf(ms[k] - Mn);
            L = fmaf(ls[k], w, L);
            A = fmaf(as[k], w, A);
        }
        M = Mn;
    }
    if (lane == 0) { s_m[warp] = M; s_l[warp] = L; }
    s_a[warp][lane] = A;
    __syncthreads();
    if (warp == 0) {
        M = -INFINITY;
#pragma unroll
        for (int w = 0; w < 8; ++w) M = fmaxf(M, s_m[w]);
        L = A = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const float f = s_m[w] == -INFINITY ? 0.f : __expf(s_m[w] - M);
            L = fmaf(s_l[w], f, L);
            A = fmaf(s_a[w][lane], f, A);
        }
        const float r = L > 0.f ? A / L : 0.f;
        const int64_t o = ((int64_t)b * a.Hq + i) * D + ch;
        if (a.out_dtype == FDKV_BF16)
            reinterpret_cast<__nv_bfloat16*>(a.out)[o] = __float2bfloat16_rn(r);
        else
            reinterpret_cast<float*>(a.out)[o] = r;
        if (a.k_new && i == 0 && blockIdx.x == 0 && lane == 0) {
            int32_t* len = a.tail_len + a.layer * a.max_batch + b;
            if (*len < a.max_tail) ++*len;
        }
    }
}

template <typename T, int D, int G>
cudaError_t launch_generic_g(const DecodeArgs& a, int splits, cudaLaunchConfig_t& cfg) {
    static PerDevice once;
    cfg.dynamicSmemBytes = (size_t)kWarps * std::max(kResTile, G) * D * sizeof(float);
    cudaError_t e = once.ensure([&]() { return cudaFuncSetAttribute(decode_generic_kernel<T, D, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes); });
    return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, decode_generic_kernel<T, D, G>, a, splits);
}

template <typename T, int D>
cudaError_t launch_generic(const DecodeArgs& a, int splits, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(splits, a.Hkv, a.batch);
    cfg.blockDim = dim3(kWarps * 32);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    switch (a.G) {
        case 1: e = launch_generic_g<T, D, 1>(a, splits, cfg); break;
        case 2: e = launch_generic_g<T, D, 2>(a, splits, cfg); break;
        case 4: e = launch_generic_g<T, D, 4>(a, splits, cfg); break;
        case 8: e = launch_generic_g<T, D, 8>(a, splits, cfg); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3(D / 32, a.Hq, a.batch);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = 0;
    return cudaLaunchKernelEx(&cfg, combine_kernel<D>, a, splits);
}

}  // namespace

__global__ void set_tail_len_kernel(int32_t* tail_len, int L, int max_batch, int seq, int n) {
    for (int l = threadIdx.x; l < L; l += blockDim.x) tail_len[l * max_batch + seq] = n;
}
cudaError_t launch_set_tail_len(int32_t* tail_len, int L, int max_batch, int seq, int n, cudaStream_t st) {
    set_tail_len_kernel<<<1, 128, 0, st>>>(tail_len, L, max_batch, seq, n);
    count_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_decode_fast(const DecodeArgs& a, cudaStream_t st, bool* handled);

cudaError_t launch_decode(const DecodeArgs& a, int dtype, cudaStream_t st) {
    cudaError_t e;
    bool handled = false;
    if ((e = launch_decode_fast(a, st, &handled)) != cudaSuccess) return e;  // (appends k_new / v_new itself)
    if (handled) return cudaSuccess;
    if (a.packed_lists) return cudaErrorNotSupported;  // packed residual lists are only read by the kernel above

    // one tile per warp while the blocks are resident at one time (two on an SM for bf16 up to two heads per group), then longer ranges
    static PerDevice once;
    int sms = 0;
    if ((e = once.ensure([]() { return cudaSuccess; }, &sms)) != cudaSuccess) return e;
    const int ntiles = (a.Tmax_batch + kResTile - 1) / kResTile, units = a.Hkv * a.batch;
    const int splits = std::max(1, std::min(std::min(((a.G <= 2 && dtype == FDKV_BF16 ? 2 : 1) * sms + units - 1) / units, kMaxSplits), (ntiles + kWarps - 1) / kWarps));
    if (dtype == FDKV_BF16)
        e = a.d == 128 ? launch_generic<__nv_bfloat16, 128>(a, splits, st) : launch_generic<__nv_bfloat16, 64>(a, splits, st);
    else
        e = a.d == 128 ? launch_generic<float, 128>(a, splits, st) : launch_generic<float, 64>(a, splits, st);
    if (e != cudaSuccess) return e;
    count_launch(2);
    count_kernel(FDKV_KERNEL_DECODE_PORTABLE);
    return cudaGetLastError();
}

}  // namespace fdkv
