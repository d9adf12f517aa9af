// Test hooks (include/fdkv_testing.h): reach the library's failure handling without a fault, a trap or a hang.
#include <cstring>

#include "../../include/fdkv_testing.h"
#include "fdkv_internal.h"
#include "mbar_wait.cuh"

namespace fdkv {
namespace {

// Thread 0 waits on a barrier nobody arrives at; the bounded wait gives up after `cap` polls and reports through the
// abort flag and the status word, as in the product kernels.  The other threads wait for it at the block barrier.
__global__ void __launch_bounds__(32) wait_expiry_kernel(int32_t* status, uint32_t cap, int32_t* polls_seen) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t abort_flag;
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(&bar);
    if (threadIdx.x == 0) {
        abort_flag = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(1u));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        mbar_wait_bounded(b, 0u, &abort_flag, status, cap);
        // a second wait of the same block returns at once: the abort flag is up
        mbar_wait_bounded(b, 0u, &abort_flag, status, cap);
        if (polls_seen) *polls_seen = (int32_t)abort_flag;
    }
    __syncthreads();
}

}  // namespace
}  // namespace fdkv

extern "C" {

fdkv_status fdkv_test_wait_expiry(fdkv_ctx* c, int32_t poll_cap, void* stream) {
    if (!c || poll_cap < 1 || poll_cap > 65536) return FDKV_ERR_INVALID_ARG;
    int32_t* status = reinterpret_cast<int32_t*>(c->work + c->ws.status);
    fdkv::wait_expiry_kernel<<<1, 32, 0, reinterpret_cast<cudaStream_t>(stream)>>>(status, (uint32_t)poll_cap, status + 1);
    fdkv::count_launch(1);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? FDKV_OK : fdkv::record_cuda_error(e);
}

fdkv_status fdkv_test_clear_device_status(fdkv_ctx* c, void* stream) {
    if (!c) return FDKV_ERR_INVALID_ARG;
    const cudaError_t e = cudaMemsetAsync(c->work + c->ws.status, 0, 256, reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? FDKV_OK : fdkv::record_cuda_error(e);
}

fdkv_status fdkv_test_probe_moments(fdkv_ctx* c, int32_t form) {
    if (!c || form < 0 || form > 2) return FDKV_ERR_INVALID_ARG;
    c->probe_moments = form;
    return FDKV_OK;
}

fdkv_status fdkv_test_plan_clusters(int32_t batch, int32_t n_kv_heads, int32_t group, const int32_t* T, const int32_t* modes, const int32_t* tails,
                                    int32_t keep_num, int32_t keep_den, int32_t row_format, int32_t n_ctas, const int32_t* max_clusters,
                                    uint32_t* start_out, int32_t* n_ctas_out, int32_t* cluster_out) {
    if (!T || !modes || !tails || !max_clusters || !start_out || !n_ctas_out || !cluster_out || batch < 1 || n_kv_heads < 1 || n_ctas < 1 ||
        n_ctas > fdkv::kMaxSplits || (int64_t)batch * n_kv_heads > fdkv::kFastMaxUnits || keep_den < 1)
        return FDKV_ERR_INVALID_ARG;
    fdkv::DecodeArgs a;
    std::memset(&a, 0, sizeof(a));
    a.batch = batch; a.Hkv = n_kv_heads; a.G = group; a.d = 128;
    a.host_T = T; a.host_modes = modes; a.host_tail = tails; a.max_tail = 1 << 20;
    a.keep_num = keep_num; a.keep_den = keep_den; a.rows_f8 = row_format != 0;
    std::vector<int32_t> parts((size_t)batch * n_kv_heads);
    const cudaError_t e = fdkv::plan_decode_host(a, n_ctas, reinterpret_cast<const int*>(max_clusters), start_out, n_ctas_out, parts.data(), cluster_out);
    return e == cudaSuccess ? FDKV_OK : FDKV_ERR_INVALID_ARG;
}

int32_t fdkv_test_per_device_visits(const int32_t* devs, int32_t n) {
    if (!devs || n < 0) return -1;
    return fdkv::per_device_first_visits(reinterpret_cast<const int*>(devs), n);
}

}  // extern "C"
