// Prefill kernels beside the selection (select.cu): the depth split of the token rule (Eq. 1), the rows it keeps, the copies
// of the commit step, and the entry point that compresses one tensor pair without a context.
#include <algorithm>
#include <mutex>

#include "fdkv_internal.h"

namespace fdkv {

namespace {

// ----- storage traits -------------------------------------------------------------------------------
template <typename T>
struct Store;
template <>
struct Store<float> {
    static constexpr int VEC = 4;
    using vec_t = float4;
    __device__ static void unpack(const vec_t& v, float* f) { f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w; }
    __device__ static vec_t pack(const float* f) { return make_float4(f[0], f[1], f[2], f[3]); }
};
template <>
struct Store<__nv_bfloat16> {
    static constexpr int VEC = 8;
    using vec_t = uint4;
    __device__ static void unpack(const vec_t& v, float* f) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[2 * i] = __uint_as_float(w[i] << 16);
            f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
    // f holds float32 values; round each to nearest-even bf16
    __device__ static vec_t pack(const float* f) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(f[2 * i]));
            uint32_t hi = __bfloat16_as_ushort(__float2bfloat16_rn(f[2 * i + 1]));
            w[i] = lo | (hi << 16);
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};

// value as stored, widened back to float32 (exact)
template <typename T>
__device__ __forceinline__ float stored(float x);
template <>
__device__ __forceinline__ float stored<float>(float x) { return x; }
template <>
__device__ __forceinline__ float stored<__nv_bfloat16>(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// ----- the split without a selection (token rule: the probe selects) ---------------------------------
// Shared coefficients of K and V and the high-frequency rows of K (Z1 of a pair, or the four layers' deviations: what the
// probe scores), in the arithmetic of select.cu.  V's high-frequency rows are only wanted for
// the few tokens that are kept, so the commit step forms those from the caller's rows instead of staging all of them.
// Bound by HBM: no histogram, so no shared memory, full occupancy and one launch over all blocks (it shared the histogram
// kernel before, one launch per block of four: 8 191 tokens, 8 blocks of four: 963 us); two vectors of every
// layer in flight per thread.
template <typename T, int B>
__global__ void __launch_bounds__(256) split_rows_kernel(SplitRowsArgs a) {
    using S = Store<T>;
    constexpr int VEC = S::VEC;
    constexpr int NV = 2;
    const int h = blockIdx.y >> 1, is_v = blockIdx.y & 1, blk = blockIdx.z;
    const int64_t ut = a.ut_base + (int64_t)blk * a.Hkv * 2 + blockIdx.y;
    T* const z0 = reinterpret_cast<T*>(a.z0) + ut * a.z0_stride;
    T* const hf = reinterpret_cast<T*>(a.hf) + (ut >> 1) * (B == 4 ? 4 : 1) * a.unit_stride;
    const float c32 = __uint_as_float(0x3F3504F3u);
    const int vpr = a.d / VEC;
    const int nvec = a.T * vpr;
    typename S::vec_t r[NV][B];
    int64_t off_out[NV];
    bool live[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) {
        const int v = (blockIdx.x * NV + u) * 256 + (int)threadIdx.x;
        live[u] = v < nvec;
        const int t = v / vpr, cv = (v - t * vpr) * VEC;
        const int64_t off_in = (int64_t)t * a.stride_t + (int64_t)h * a.stride_h + cv;
        off_out[u] = (int64_t)v * VEC;
        if (live[u])
#pragma unroll
            for (int l = 0; l < B; ++l)
                r[u][l] = *reinterpret_cast<const typename S::vec_t*>(reinterpret_cast<const T*>(is_v ? a.v[B * blk + l] : a.k[B * blk + l]) + off_in);
    }
#pragma unroll
    for (int u = 0; u < NV; ++u) {
        if (!live[u]) continue;
        float f[B][VEC], z[VEC];
#pragma unroll
        for (int l = 0; l < B; ++l) S::unpack(r[u][l], f[l]);
        if constexpr (B == 2) {
            float f1[VEC];
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                z[i] = __fmul_rn(__fadd_rn(f[0][i], f[1][i]), c32);
                f1[i] = __fmul_rn(__fsub_rn(f[0][i], f[1][i]), c32);
            }
            if (!is_v) *reinterpret_cast<typename S::vec_t*>(hf + off_out[u]) = S::pack(f1);
        } else {
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                z[i] = stored<T>(__fmul_rn(0.5f, __fadd_rn(__fadd_rn(f[0][i], f[1][i]), __fadd_rn(f[2][i], f[3][i]))));
                const float half = __fmul_rn(0.5f, z[i]);  // exact
#pragma unroll
                for (int l = 0; l < B; ++l) f[l][i] = __fsub_rn(f[l][i], half);
            }
            if (!is_v)
#pragma unroll
                for (int l = 0; l < B; ++l) *reinterpret_cast<typename S::vec_t*>(hf + (int64_t)l * a.unit_stride + off_out[u]) = S::pack(f[l]);
        }
        *reinterpret_cast<typename S::vec_t*>(z0 + off_out[u]) = S::pack(z);
    }
}

// Token rule, commit: the high-frequency rows of the selected tokens, densely packed, formed from the caller's rows of the
// block's layers (one job per unit-tensor, one thread per 16-byte vector: reads B rows, writes one row per stored
// tensor).  `twice` doubles the stored rows (bf16 rows of the tensor-core decode kernel; exact): a block of four scales its
// rows by 1/2 at decode time and its deviations by 1.
template <typename T, int B>
__global__ void __launch_bounds__(256) token_gather_kernel(const TokenGatherJob* jobs, int d) {
    using S = Store<T>;
    constexpr int VEC = S::VEC;
    const TokenGatherJob& jb = jobs[blockIdx.y];
    const int vpr = d / VEC;
    const int64_t v = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int64_t j = v / vpr;
    if (j >= jb.k_tok) return;
    const int cv = (int)(v - j * vpr) * VEC;
    const int64_t off_in = (int64_t)jb.list[j] * jb.stride_t + cv;
    float f[B][VEC];
#pragma unroll
    for (int l = 0; l < B; ++l) S::unpack(*reinterpret_cast<const typename S::vec_t*>(reinterpret_cast<const T*>(jb.x[l]) + off_in), f[l]);
    if constexpr (B == 2) {
        const float c32 = __uint_as_float(0x3F3504F3u);
#pragma unroll
        for (int i = 0; i < VEC; ++i) f[0][i] = __fmul_rn(__fsub_rn(f[0][i], f[1][i]), c32);
        *reinterpret_cast<typename S::vec_t*>(reinterpret_cast<T*>(jb.dst[0]) + v * VEC) = S::pack(f[0]);
    } else {
        const float k = jb.twice ? 2.f : 1.f;
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            const float z = stored<T>(__fmul_rn(0.5f, __fadd_rn(__fadd_rn(f[0][i], f[1][i]), __fadd_rn(f[2][i], f[3][i]))));
            const float half = __fmul_rn(0.5f, z);  // exact
#pragma unroll
            for (int l = 0; l < B; ++l) f[l][i] = stored<T>(__fsub_rn(f[l][i], half)) * k;
        }
#pragma unroll
        for (int l = 0; l < B; ++l) *reinterpret_cast<typename S::vec_t*>(reinterpret_cast<T*>(jb.dst[l]) + v * VEC) = S::pack(f[l]);
    }
}

}  // namespace

cudaError_t launch_split_rows(const SplitRowsArgs& a, int B, int dtype, cudaStream_t st) {
    if (a.T <= 0 || a.n_blocks <= 0) return cudaSuccess;
    const int per_block = 2 * 256 * (dtype == FDKV_BF16 ? 8 : 4);  // elements one thread block covers
    dim3 grid((unsigned)(((int64_t)a.T * a.d + per_block - 1) / per_block), a.Hkv * 2, a.n_blocks);
    if (dtype == FDKV_BF16) {
        if (B == 4) split_rows_kernel<__nv_bfloat16, 4><<<grid, 256, 0, st>>>(a);
        else split_rows_kernel<__nv_bfloat16, 2><<<grid, 256, 0, st>>>(a);
    } else {
        if (B == 4) split_rows_kernel<float, 4><<<grid, 256, 0, st>>>(a);
        else split_rows_kernel<float, 2><<<grid, 256, 0, st>>>(a);
    }
    count_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_token_gather_jobs(const TokenGatherJob* jobs_dev, int njobs, int64_t k_tok, int d, int B, int dtype, cudaStream_t st) {
    if (njobs <= 0 || k_tok <= 0) return cudaSuccess;
    const int64_t nvec = k_tok * (d / (dtype == FDKV_BF16 ? 8 : 4));
    for (int j0 = 0; j0 < njobs; j0 += 65535) {
        const dim3 grid((unsigned)((nvec + 255) / 256), std::min(njobs - j0, 65535));
        if (dtype == FDKV_BF16) {
            if (B == 4) token_gather_kernel<__nv_bfloat16, 4><<<grid, 256, 0, st>>>(jobs_dev + j0, d);
            else token_gather_kernel<__nv_bfloat16, 2><<<grid, 256, 0, st>>>(jobs_dev + j0, d);
        } else {
            if (B == 4) token_gather_kernel<float, 4><<<grid, 256, 0, st>>>(jobs_dev + j0, d);
            else token_gather_kernel<float, 2><<<grid, 256, 0, st>>>(jobs_dev + j0, d);
        }
        count_launch(1);
    }
    return cudaGetLastError();
}

// grid (chunks of 32 KiB of the largest job, jobs): the device-to-device copies of a commit or a fold (row streams, strided
// source rows of exact units, residual lists, offset tables, tail rows) and the zero fills as one launch per class of job
// size, so that few blocks find nothing to do, instead of several hundred copy and fill calls of about 1.2 us each on the
// host and on the device (a fold of 16 tokens over 32 layers, about 770 of them: 2.3 ms)
constexpr int kCopyChunk = 32 * 1024;
__global__ void __launch_bounds__(256) copy_jobs_kernel(const CopyJob* jobs) {
    const CopyJob jb = jobs[blockIdx.y];
    const int64_t c0 = (int64_t)blockIdx.x * kCopyChunk;
    if (c0 >= jb.bytes) return;
    const int64_t c1 = min(jb.bytes, c0 + kCopyChunk);
    if (!jb.src) {
        for (int64_t o = c0 + threadIdx.x * 4; o < c1; o += 256 * 4) *reinterpret_cast<uint32_t*>(jb.dst + o) = 0u;
        return;
    }
    if (jb.add) {  // 32-bit list positions or offsets
        for (int64_t o = c0 + threadIdx.x * 4; o < c1; o += 256 * 4)
            *reinterpret_cast<int32_t*>(jb.dst + o) = *reinterpret_cast<const int32_t*>(jb.src + o) + jb.add;
        return;
    }
    if (((uintptr_t)jb.src | (uintptr_t)jb.dst | (uintptr_t)jb.bytes) & 3) {  // 2-byte values of a list behind an odd number of others
        for (int64_t o = c0 + threadIdx.x * 2; o < c1; o += 256 * 2)
            *reinterpret_cast<uint16_t*>(jb.dst + o) = *reinterpret_cast<const uint16_t*>(jb.src + o);
        return;
    }
    const bool plain = jb.src_pitch == jb.row_bytes;
    auto src_of = [&](int64_t o) {
        if (plain) return o;
        const int64_t r = o / jb.row_bytes;
        return r * jb.src_pitch + (o - r * jb.row_bytes);
    };
    // 16-byte vectors when both sides allow it (offset tables of later unit-tensors start on 4-byte boundaries only)
    const bool vec_ok = (((uintptr_t)jb.src | (uintptr_t)jb.dst) & 15) == 0;
    const int64_t v1 = vec_ok ? (c1 & ~(int64_t)15) : c0;
#pragma unroll 4
    for (int64_t o = c0 + threadIdx.x * 16; o < v1; o += 256 * 16)
        *reinterpret_cast<uint4*>(jb.dst + o) = *reinterpret_cast<const uint4*>(jb.src + src_of(o));
    for (int64_t o = v1 + threadIdx.x * 4; o < c1; o += 256 * 4)
        *reinterpret_cast<uint32_t*>(jb.dst + o) = *reinterpret_cast<const uint32_t*>(jb.src + src_of(o));
}
cudaError_t launch_copy_jobs(const CopyJob* jobs_dev, int njobs, int64_t bytes_max, cudaStream_t st) {
    for (int j0 = 0; j0 < njobs && bytes_max > 0; j0 += 65535) {
        copy_jobs_kernel<<<dim3((unsigned)((bytes_max + kCopyChunk - 1) / kCopyChunk), std::min(njobs - j0, 65535)), 256, 0, st>>>(jobs_dev + j0);
        count_launch(1);
    }
    return cudaGetLastError();
}

}  // namespace fdkv

// ---------------------------------------------------------------------------------------------------------------
// Allocation-free compression of one [T][d] tensor pair (declared in fdkv.h as fdkv_compress_unit_noalloc).
// Same kernels as fdkv_compress_prefill; the scratch they need (the candidate lists, the select state and the tile
// offsets) lives in the file-scope device array below instead of a caller-provided workspace.  Every GPU that loads this library holds the array until the process exits.
// ---------------------------------------------------------------------------------------------------------------
namespace fdkv {
namespace {

constexpr int64_t kNoAllocMaxElems = FDKV_NOALLOC_MAX_ELEMS;                    // T * head_dim
constexpr int64_t kNoAllocMaxTiles = kNoAllocMaxElems / 64 / fdkv::kResTile;    // head_dim >= 64
constexpr int64_t kNoAllocChunks = kNoAllocMaxElems / fdkv::compress_chunk(2, 4);  // (the smallest chunk a pair has)
constexpr size_t kNaPos = 0;
constexpr size_t kNaVal = kNaPos + (size_t)kNoAllocMaxElems * 2;                // float32 worst case
constexpr size_t kNaCount = kNaVal + (size_t)kNoAllocMaxElems * 4;
constexpr size_t kNaBase = kNaCount + (size_t)kNoAllocChunks * 4;
constexpr size_t kNaSel = kNaBase + (size_t)kNoAllocChunks * 8;
constexpr size_t kNaStatus = kNaSel + 256;
constexpr size_t kNaOff = kNaStatus + 256;
constexpr size_t kNaBytes = (kNaOff + (size_t)(kNoAllocMaxTiles + 1) * 4 + 255) / 256 * 256;
static_assert(kNoAllocMaxElems % fdkv::kMaxCompressChunk == 0 && kNaSel % 256 == 0, "whole chunks, aligned parts");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

// In host code the array's name is only a handle: the device address comes from cudaGetSymbolAddress, once per
// device, with that device current.
constexpr int kMaxDevices = 64;
void* g_noalloc_ptr[kMaxDevices] = {};
std::mutex g_noalloc_mutex;

cudaError_t noalloc_scratch(char** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = p;
    }
    *out = static_cast<char*>(g_noalloc_ptr[dev]);
    return cudaSuccess;
}

}  // namespace
}  // namespace fdkv

extern "C" fdkv_status fdkv_compress_unit_noalloc(const void* x0, const void* x1, int64_t stride_t, int32_t T,
                                                  int32_t head_dim, int32_t dtype, int32_t keep_num, int32_t keep_den,
                                                  void* z0_out, int32_t* idx_out, void* val_out, int32_t* count_host,
                                                  void* stream) {
    using namespace fdkv;
    if (!x0 || !x1 || !z0_out || T < 1) return FDKV_ERR_INVALID_ARG;
    if (head_dim != 64 && head_dim != 128) return FDKV_ERR_UNSUPPORTED;
    if (dtype != FDKV_F32 && dtype != FDKV_BF16) return FDKV_ERR_UNSUPPORTED;
    if (keep_den <= 0 || keep_num < 0 || keep_num > keep_den) return FDKV_ERR_INVALID_ARG;
    if (stride_t < head_dim || (stride_t % 8)) return FDKV_ERR_INVALID_ARG;
    if ((int64_t)T * head_dim > kNoAllocMaxElems) return FDKV_ERR_TOO_LARGE;  // the static scratch cannot hold it
    const int64_t k = (int64_t)T * head_dim * keep_num / keep_den;
    if (k > 0 && (!idx_out || !val_out)) return FDKV_ERR_INVALID_ARG;
    for (const void* p : {x0, x1, (const void*)z0_out, (const void*)idx_out, (const void*)val_out})
        if (reinterpret_cast<uintptr_t>(p) % 16) return FDKV_ERR_INVALID_ARG;
    if (count_host) *count_host = (int32_t)k;

    char* sc = nullptr;
    cudaError_t e = noalloc_scratch(&sc);
    if (e != cudaSuccess) return record_cuda_error(e);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // (the array keeps the previous call's contents: the kernels write what they read; the status word is nobody's here)
    CompressArgs a;
    a.stride_t = stride_t; a.stride_h = 0;
    a.T = T; a.d = head_dim; a.Hkv = 1; a.tensors = 1;
    a.unit_stride = 0; a.z0_stride = 0;
    a.z0 = z0_out; a.z1 = nullptr;
    a.sel = reinterpret_cast<SelState*>(sc + kNaSel);
    a.cand_pos = reinterpret_cast<uint16_t*>(sc + kNaPos);
    a.cand_val = sc + kNaVal;
    a.cand_n = reinterpret_cast<int32_t*>(sc + kNaCount);
    a.chunk_base = reinterpret_cast<int2*>(sc + kNaBase);
    a.cand_stride = kNoAllocMaxElems; a.chunks_max = (int)kNoAllocChunks;
    a.n_keep = k; a.kcap = 0;
    // (a layer's rows that z0 overwrites must not be read a second time)
    const size_t esize = dtype == FDKV_BF16 ? 2 : 4;
    const uintptr_t z0_at = reinterpret_cast<uintptr_t>(z0_out), z0_end = z0_at + (size_t)T * head_dim * esize;
    a.in_place = false;
    for (const void* x : {x0, x1}) {
        const uintptr_t at = reinterpret_cast<uintptr_t>(x), end = at + ((size_t)(T - 1) * stride_t + head_dim) * esize;
        a.in_place = a.in_place || (z0_at < end && at < z0_end);
    }
    a.ntiles_max = (int)kNoAllocMaxTiles;
    a.tile_off = reinterpret_cast<int32_t*>(sc + kNaOff);
    a.idx = idx_out; a.val = val_out; a.packed = nullptr;
    a.keep = nullptr; a.keep_stride = 0;
    a.status = reinterpret_cast<int32_t*>(sc + kNaStatus);
    const void* const layers[2] = {x0, x1};
    if ((e = launch_compress(a, 2, dtype, layers, layers, 0, 1, st)) != cudaSuccess) return record_cuda_error(e);
    return FDKV_OK;
}
