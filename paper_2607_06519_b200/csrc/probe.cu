// Routing probe (Eq. 2 and the argmin of Eq. 3): logit-error of the shared and residual candidates over the
// probe window, then the mode rule.  This file holds the portable float32-FMA kernel (any dtype / head_dim);
// the tcgen05 tensor-core kernel for bf16 lives in probe_tc.cu.
#include "fdkv_internal.h"

namespace fdkv {

namespace {

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
    const uint2 w = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xFFFF0000u));
}

constexpr int kRowsBlk = 32, kProbeThreads = 512, kProbePad = 4;
constexpr size_t probe_tile_smem(int d) { return (size_t)(2 * kProbeTile * (d + kProbePad) + 2 * kRowsBlk * d) * sizeof(float); }

// grid (probe tiles, units).  Each CTA: 64 tokens of one unit, all 2*G*W probe rows, both candidates; a thread has one token and
// four of 32 rows, whose values the next turn's loads replace in the other half of the buffer.  Four channels per shared-memory
// load: 6 loads for 32 multiply-adds (with one channel per load, 16 rows and the loads between two barriers: 4k tokens of four
// layers, two heads, head_dim 64, 58 -> 19 us).
template <typename T>
__global__ void __launch_bounds__(kProbeThreads) probe_tile_kernel(ProbeArgs a) {
    extern __shared__ __align__(16) float smem[];
    const int d = a.d, ld = d + kProbePad, d4 = d / 4, s4 = d == 128 ? 5 : 4;
    float* full = smem;                      // [64][d+4]  Z1 of K: what the shared candidate drops
    float* drop = full + kProbeTile * ld;    // [64][d+4]  Z1 of K minus the kept entries: what residual drops
    float* qs = drop + kProbeTile * ld;      // [2][32][d]
    __shared__ double s_red[2][kProbeThreads / 32];

    const int unit = a.unit_begin + blockIdx.y;
    const int t0 = blockIdx.x * kProbeTile;
    const int nt = min(kProbeTile, a.T - t0);
    const int h = unit % a.Hkv, pair = unit / a.Hkv;
    const int ut = unit * 2;  // K
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j = (warp & 1) * 32 + lane;  // token within the tile
    const int rg = warp >> 1;              // 8 groups of 4 rows
    // A pair has one high-frequency operand (Z1) that both layers' queries see; a block of four layers has one
    // operand per layer (its deviation from the block mean), seen by that layer's queries only.
    const int n_ops = a.B == 4 ? 4 : 1;
    const int M = (a.B == 4 ? 1 : 2) * a.G * a.W;  // probe rows per operand
    float sum_f = 0.f, sum_d = 0.f;
    for (int op = 0; op < n_ops; ++op) {
        // 32 probe rows from rb on: row r = (layer*G + g)*W + qi  ->  Q[layer][qi][h*G + g][:], this thread's 16-byte vectors
        constexpr int QV = kRowsBlk * 32 / kProbeThreads;  // (head_dim 64 has half of them)
        float4 qv[QV];
        auto load_q = [&](int rb) {
#pragma unroll
            for (int q = 0; q < QV; ++q) {
                const int i = threadIdx.x + q * kProbeThreads, r = rb + (i >> s4), c = (i & (d4 - 1)) * 4;
                qv[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i < kRowsBlk * d4 && r < M) {
                    const int layer = a.B == 4 ? op : r / (a.G * a.W), g = (r / a.W) % a.G, qi = r % a.W;
                    qv[q] = ld4(reinterpret_cast<const T*>(a.q_layers_dev[a.B * pair + layer]) + ((int64_t)qi * a.Hq + h * a.G + g) * d + c);
                }
            }
        };
        auto store_q = [&](int half) {
#pragma unroll
            for (int q = 0; q < QV; ++q) {
                const int i = threadIdx.x + q * kProbeThreads;
                if (i < kRowsBlk * d4) *reinterpret_cast<float4*>(qs + half * kRowsBlk * d + 4 * i) = qv[q];
            }
        };
        load_q(0);
        const T* z1 = reinterpret_cast<const T*>(a.z1) + ((int64_t)unit * n_ops + op) * a.unit_stride + (int64_t)t0 * d;
        for (int i = threadIdx.x; i < kProbeTile * d4; i += kProbeThreads) {
            const int t = i >> s4, c = (i & (d4 - 1)) * 4;
            const float4 v = t < nt ? ld4(z1 + 4 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
            *reinterpret_cast<float4*>(full + t * ld + c) = v;
            *reinterpret_cast<float4*>(drop + t * ld + c) = v;
        }
        store_q(0);
        __syncthreads();
        const int32_t* off = a.tile_off + (int64_t)ut * (a.ntiles_max + 1);
        const int ntiles = (a.T + kResTile - 1) / kResTile;
        const int j0 = t0 / kResTile, j1 = min(ntiles, (t0 + kProbeTile) / kResTile);
        const int32_t* idx = a.idx + (int64_t)ut * a.kcap;
        for (int e = off[j0] + threadIdx.x; e < off[j1]; e += kProbeThreads) {
            const int f = idx[e] - t0 * d;
            drop[(f >> (s4 + 2)) * ld + (f & (d - 1))] = 0.f;
        }
        __syncthreads();
        for (int rb = 0, half = 0; rb < M; rb += kRowsBlk, half ^= 1) {
            const bool more = rb + kRowsBlk < M;
            if (more) load_q(rb + kRowsBlk);
            float af[4] = {0.f, 0.f, 0.f, 0.f}, ad[4] = {0.f, 0.f, 0.f, 0.f};
            const float* zf = full + j * ld;
            const float* zd = drop + j * ld;
            const float* qr = qs + half * kRowsBlk * d + rg * 4 * d;
#pragma unroll 4
            for (int c = 0; c < d; c += 4) {
                const float4 vf = ld4(zf + c), vd = ld4(zd + c);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 w = ld4(qr + i * d + c);
                    af[i] = fmaf(w.x, vf.x, af[i]); af[i] = fmaf(w.y, vf.y, af[i]); af[i] = fmaf(w.z, vf.z, af[i]); af[i] = fmaf(w.w, vf.w, af[i]);
                    ad[i] = fmaf(w.x, vd.x, ad[i]); ad[i] = fmaf(w.y, vd.y, ad[i]); ad[i] = fmaf(w.z, vd.z, ad[i]); ad[i] = fmaf(w.w, vd.w, ad[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = rb + rg * 4 + i;
                if (r < M && j < nt && t0 + j <= a.pos[r % a.W]) {  // causal: keys at or before the probe position
                    sum_f = fmaf(af[i], af[i], sum_f);
                    sum_d = fmaf(ad[i], ad[i], sum_d);
                }
            }
            if (more) store_q(half ^ 1);  // (read two turns ago, behind the last barrier)
            __syncthreads();
        }
    }
    double df = sum_f, dd = sum_d;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        df += __shfl_xor_sync(0xFFFFFFFFu, df, o);
        dd += __shfl_xor_sync(0xFFFFFFFFu, dd, o);
    }
    if (lane == 0) { s_red[0][warp] = df; s_red[1][warp] = dd; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double tf = 0, td = 0;
        for (int w = 0; w < kProbeThreads / 32; ++w) { tf += s_red[0][w]; td += s_red[1][w]; }
        double* p = a.part + ((int64_t)unit * a.nptiles_max + blockIdx.x) * 2;
        p[0] = tf;
        p[1] = td;
    }
}

}  // namespace

// Sums the per-tile partials in a fixed order, applies the (c/sqrt d)^2 / (2 G W) factor and the mode rule.
__global__ void __launch_bounds__(256) probe_finalize_kernel(ProbeArgs a, ProbeParts parts) {
    __shared__ double s0[256], s1[256];
    const int unit = a.unit_begin + blockIdx.x;
    const double* p = a.part + (int64_t)unit * a.nptiles_max * 2;
    double x0 = 0, x1 = 0;
    const bool redo = parts.all > parts.sure && a.redo[unit];
    const int first = redo ? parts.gram : 0, last = redo ? parts.all : parts.sure;
    for (int i = first + threadIdx.x; i < last; i += blockDim.x) { x0 += p[2 * i]; x1 += p[2 * i + 1]; }
    s0[threadIdx.x] = x0;
    s1[threadIdx.x] = x1;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (threadIdx.x < o) { s0[threadIdx.x] += s0[threadIdx.x + o]; s1[threadIdx.x] += s1[threadIdx.x + o]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        // (c / sqrt d)^2 over 2 G W rows for a pair's Z1; (1 / sqrt d)^2 over 4 G W rows for a block's deviations
        const double norm = a.B == 4 ? 1.0 / (double)a.d / (double)(4 * a.G * a.W) : 0.5 / (double)a.d / (double)(2 * a.G * a.W);
        const double e_sh = s0[0] * norm, e_rs = s1[0] * norm;
        a.scores[2 * unit] = e_sh;
        a.scores[2 * unit + 1] = e_rs;
        const double L0 = e_sh + a.lambda * a.omega[0];
        const double L1 = e_rs + a.lambda * a.omega[1];
        const double L2 = a.lambda * a.omega[2];
        int m = 0;
        double best = L0;
        if (L1 < best) { best = L1; m = 1; }
        if (L2 < best) { best = L2; m = 2; }
        a.modes[unit] = m;
        if (a.modes_out) a.modes_out[blockIdx.x] = m;
        if (a.scores_out) {
            a.scores_out[2 * blockIdx.x] = (float)e_sh;
            a.scores_out[2 * blockIdx.x + 1] = (float)e_rs;
        }
    }
}

// The positions and pointers travel in the launch parameters: a captured call carries them, and nothing is copied from pageable
// memory.
struct ProbeInputs {
    int32_t pos[kMaxW];
    const void* q[kSplitLayers];
};
__global__ void __launch_bounds__(kMaxW) probe_inputs_kernel(ProbeInputs in, int32_t* pos, int W, const void** q, int n) {
    const int i = threadIdx.x;
    if (i < W) pos[i] = in.pos[i];
    if (i < n) q[i] = in.q[i];
}
static_assert(kSplitLayers <= kMaxW, "a thread per pointer");

cudaError_t launch_probe_inputs(int32_t* pos_dev, const int32_t* pos, int W, const void** q_dev, const void* const* q_layers, int layer_begin, int layer_end,
                                cudaStream_t st) {
    ProbeInputs in = {};
    for (int i = 0; i < W; ++i) in.pos[i] = pos[i];
    for (int l = layer_begin; l < layer_end; l += kSplitLayers) {
        const int n = layer_end - l < kSplitLayers ? layer_end - l : kSplitLayers;
        for (int i = 0; i < n; ++i) in.q[i] = q_layers[l + i];
        probe_inputs_kernel<<<1, kMaxW, 0, st>>>(in, pos_dev, W, q_dev + l, n);
        count_launch(1);
    }
    return cudaGetLastError();
}

cudaError_t launch_probe_tc(const ProbeArgs& a, int dtype, cudaStream_t st, bool* handled, ProbeParts* parts);

cudaError_t launch_probe(const ProbeArgs& a, int dtype, cudaStream_t st) {
    if (a.unit_count <= 0) return cudaSuccess;
    const int nparts = a.sums_ready ? 1 : (a.T + kProbeTile - 1) / kProbeTile;
    ProbeParts parts = {0, nparts, nparts};
    bool handled = a.sums_ready;
    cudaError_t e = cudaSuccess;
    if (!handled && (e = launch_probe_tc(a, dtype, st, &handled, &parts)) != cudaSuccess) return e;
    if (!handled) {
        const size_t smem = probe_tile_smem(a.d);
        static PerDevice once;
        e = once.ensure([&]() {
            cudaError_t e2 = cudaFuncSetAttribute(probe_tile_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)probe_tile_smem(128));
            if (e2 != cudaSuccess) return e2;
            return cudaFuncSetAttribute(probe_tile_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)probe_tile_smem(128));
        });
        if (e != cudaSuccess) return e;
        dim3 grid(nparts, a.unit_count);
        if (dtype == FDKV_BF16)
            probe_tile_kernel<__nv_bfloat16><<<grid, kProbeThreads, smem, st>>>(a);
        else
            probe_tile_kernel<float><<<grid, kProbeThreads, smem, st>>>(a);
        count_launch(1);
        count_kernel(FDKV_KERNEL_PROBE_PORTABLE);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    probe_finalize_kernel<<<a.unit_count, 256, 0, st>>>(a, parts);
    count_launch(1);
    return cudaGetLastError();
}

}  // namespace fdkv
