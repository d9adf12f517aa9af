// Host side of the C ABI: argument checks, workspace / arena bookkeeping, launch sequencing.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>

#include "fdkv_internal.h"

using namespace fdkv;

namespace {

std::atomic<int64_t> g_launches{0};
std::atomic<int64_t> g_kernel_launches[FDKV_KERNEL_COUNT_];
std::atomic<int32_t> g_last_cuda{0};

inline size_t align_up(size_t x, size_t a = 256) { return (x + a - 1) / a * a; }
inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

fdkv_status cuda_fail(cudaError_t e) {
    g_last_cuda.store((int32_t)e);
    return FDKV_ERR_CUDA;
}
#define CU(x)                                         \
    do {                                              \
        cudaError_t e__ = (x);                        \
        if (e__ != cudaSuccess) return cuda_fail(e__); \
    } while (0)

bool make_shape(const fdkv_config& c, Shape& s) {
    const int B = c.block_size == 0 ? 2 : c.block_size;
    if (B != 2 && B != 4) return false;
    if (c.n_layers <= 0 || (c.n_layers % B) || c.n_layers > 1024) return false;
    if (c.n_kv_heads <= 0 || c.n_q_heads <= 0 || c.n_q_heads % c.n_kv_heads) return false;
    const int G = c.n_q_heads / c.n_kv_heads;
    if (!(G == 1 || G == 2 || G == 4 || G == 8)) return false;
    if (c.head_dim != 64 && c.head_dim != 128) return false;
    if (c.max_batch <= 0 || c.max_prefill <= 0 || c.max_tail < 0 || c.max_fold < 0) return false;
    if ((int64_t)(c.max_prefill + (int64_t)c.max_fold) * c.head_dim >= (int64_t)1 << 31) return false;
    if ((int64_t)c.max_prefill * c.head_dim >= (int64_t)1 << 31) return false;
    if (c.dtype != FDKV_F32 && c.dtype != FDKV_BF16) return false;
    if (c.keep_den <= 0 || c.keep_num < 0 || c.keep_num > c.keep_den) return false;
    s.L = c.n_layers; s.B = B; s.NB = B == 4 ? 4 : 1; s.P = c.n_layers / B; s.Hq = c.n_q_heads; s.Hkv = c.n_kv_heads; s.G = G; s.d = c.head_dim;
    s.max_batch = c.max_batch; s.Tmax = c.max_prefill; s.max_tail = c.max_tail;
    s.dtype = c.dtype; s.esize = c.dtype == FDKV_BF16 ? 2 : 4;
    s.keep_num = c.keep_num; s.keep_den = c.keep_den;
    s.max_fold = c.max_fold;
    if (c.row_format != FDKV_ROWS_STORAGE && c.row_format != FDKV_ROWS_E4M3) return false;
    s.rows_f8 = c.row_format == FDKV_ROWS_E4M3;
    if (s.rows_f8 && !(c.dtype == FDKV_BF16 && c.head_dim == 128 && G <= 4 && c.max_fold == 0)) return false;
    s.kfold_max = (int64_t)s.max_fold * s.d * s.keep_num / s.keep_den;
    s.kmax = (int64_t)s.Tmax * s.d * s.keep_num / s.keep_den;
    s.kcap = (int64_t)align_up((size_t)(s.kmax + kListPad), 64);
    s.ntiles_max = (s.Tmax + kResTile - 1) / kResTile;
    // per-unit partial-sum slots of the probe: one per 64-token tile (portable kernel) or one per work item of the
    // tensor-core kernel (layers x 128-row blocks x key splits of at least 8 tiles; twice, where a unit is done again) and the
    // blocks of the second-moment kernel that share a unit, whichever is more
    s.nptiles_max = std::max((s.Tmax + kProbeTile - 1) / kProbeTile,
                             2 * B * ((G * kMaxW + 127) / 128) * (((s.Tmax - 1) / kProbeBoxRows + 1 + 7) / 8) + kMaxGramSlots);
    s.tail_rows = (s.max_tail + kRowPad - 1) / kRowPad * kRowPad;
    if (c.residual_rule != FDKV_RESIDUAL_ENTRIES && c.residual_rule != FDKV_RESIDUAL_TOKENS) return false;
    s.tok_rule = c.residual_rule == FDKV_RESIDUAL_TOKENS;
    s.ktok_max = (int64_t)s.Tmax * s.keep_num / s.keep_den;
    s.ktok_cap = (int64_t)align_up((size_t)(s.ktok_max + 32), 64);
    s.cand_stride = ((int64_t)s.Tmax * s.d + kMaxCompressChunk - 1) / kMaxCompressChunk * kMaxCompressChunk;
    s.chunks_max = (int)(s.cand_stride / compress_chunk(B, s.esize));
    s.NU = s.P * s.Hkv;
    s.NT = 2 * s.NU;
    return true;
}

constexpr size_t quant_table_bytes(const Shape& s) { return s.rows_f8 ? (size_t)s.NU * 2 * s.B * (sizeof(QuantJob) + sizeof(RepackJob)) : 0; }
constexpr size_t gather_table_bytes(const Shape& s) { return s.tok_rule ? (size_t)s.NU * 2 * sizeof(TokenGatherJob) : 0; }
constexpr size_t max_copy_jobs(const Shape& s) { return (size_t)s.NU * (4 * s.B + 10 + 4 * s.NB); }

void make_layouts(const Shape& s, WsLayout& w, ArenaLayout& a) {
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes); return r; };
    const size_t unit_elems = (size_t)s.Tmax * s.d;
    w.status = take(256);
    w.z0 = take((size_t)s.NT * unit_elems * s.esize);
    w.z1 = take((size_t)s.NU * s.NB * unit_elems * s.esize);  // high-frequency rows of K: Z1 of a pair, or the four layers' deviations
    w.z1drop = take(s.dtype == FDKV_BF16 && s.d == 128 && !s.tok_rule ? (size_t)s.NU * s.NB * unit_elems * s.esize : 0);
    const size_t entry_rule = s.tok_rule ? 0 : 1;
    w.cand_pos = take(entry_rule * s.NT * s.cand_stride * 2);
    w.cand_val = take(entry_rule * s.NT * s.NB * s.cand_stride * s.esize);
    w.cand_n = take(entry_rule * s.NT * s.chunks_max * 4);
    w.chunk_base = take(entry_rule * s.NT * s.chunks_max * 8);
    w.keep = take(entry_rule * s.NU * (s.cand_stride / 8));
    w.sel = take((size_t)s.NT * sizeof(SelState));
    w.tile_off = take((size_t)s.NT * (s.ntiles_max + 1) * 4);
    w.idx = take((size_t)s.NT * s.kcap * 4);
    w.val = take((size_t)s.NT * s.NB * s.kcap * s.esize);
    w.packed = take(s.dtype == FDKV_BF16 && s.d == 128 ? (size_t)s.NT * s.NB * s.kcap * 4 : 0);
    w.tok_score = take(s.tok_rule ? (size_t)s.NU * s.Tmax * 4 : 0);
    w.tok_err = take(s.tok_rule ? (size_t)s.NU * token_err_slots(s.B, s.G, s.dtype == FDKV_BF16 && s.d == 128, kMaxW) * s.Tmax * 4 : 0);
    w.tok_list = take(s.tok_rule ? (size_t)s.NU * s.ktok_cap * 4 : 0);
    w.tok_off = take(s.tok_rule ? (size_t)s.NU * (s.ntiles_max + 1) * 4 : 0);
    w.probe_part = take((size_t)s.NU * s.nptiles_max * 16);
    w.probe_scale = take(s.dtype == FDKV_BF16 && s.d == 128 && !s.tok_rule ? (size_t)s.NU * kMaxGramSlots * 16 : 0);
    w.probe_redo = take((size_t)s.NU * 4);
    w.probe_pos = take((size_t)kMaxW * 4 + (size_t)s.L * 8);
    w.scores = take((size_t)s.NU * 16);
    w.modes = take((size_t)s.NU * 4);
    w.partials = take((size_t)s.max_batch * s.Hq * kMaxSplits * (s.d + 4) * 4);
    w.io_q = take((size_t)s.L * s.max_batch * s.Hq * s.d * 4);  // host-I/O staging: room for every layer of a step
    w.io_k = take((size_t)s.L * s.max_batch * s.Hkv * s.d * 4);
    w.io_v = take((size_t)s.L * s.max_batch * s.Hkv * s.d * 4);
    w.io_out = take((size_t)s.L * s.max_batch * s.Hq * s.d * 4);
    // job tables of a commit: quantise jobs (one per stored tensor) and repack jobs (one per residual list) of 8-bit rows,
    // gather jobs of the token rule, then the copy jobs (at most 2 B row copies with a fill each, or 2 row copies and fills,
    // 2 offset tables, 2 index and 2 NB value or packed lists, per unit)
    w.jobs = take(quant_table_bytes(s) + gather_table_bytes(s) + max_copy_jobs(s) * sizeof(CopyJob));
    w.total = o;

    o = 0;
    a.tail_len = take((size_t)s.L * s.max_batch * 4);
    a.desc = take((size_t)s.max_batch * s.L * s.Hkv * sizeof(UnitDesc));
    const size_t tail = (size_t)s.L * s.max_batch * s.Hkv * s.tail_rows * s.d * s.esize;
    a.tail_k = take(tail);
    a.tail_v = take(tail);
    a.bump = o;
    const size_t rows_pad = align_up((size_t)((s.Tmax + s.max_fold + kRowPad - 1) / kRowPad * kRowPad) * s.d * s.esize);
    const size_t exact_unit = 2 * (size_t)s.B * rows_pad;
    const size_t resid_unit = s.tok_rule
                                  ? 2 * rows_pad + 2 * (size_t)s.NB * align_up((size_t)s.ktok_cap * s.d * s.esize) + align_up((size_t)s.ktok_cap * 4) +
                                        align_up((size_t)(s.ntiles_max + 1) * 4)
                                  : 2 * rows_pad + 2 * (size_t)s.NB * (align_up((size_t)(s.kcap + s.kfold_max) * 4) + align_up((size_t)(s.kcap + s.kfold_max) * s.esize)) +
                                        2 * align_up((size_t)(s.kcap + s.kfold_max) * 4) +
                                        2 * align_up((size_t)(s.ntiles_max + s.max_fold / kResTile + 2) * 4);
    a.worst_total = a.bump + (size_t)s.max_batch * s.NU * (exact_unit > resid_unit ? exact_unit : resid_unit);
}

inline cudaStream_t S(void* p) { return reinterpret_cast<cudaStream_t>(p); }
template <typename T>
inline T* wsp(fdkv_ctx* c, size_t off) { return reinterpret_cast<T*>(c->work + off); }
template <typename T>
inline T* arp(fdkv_ctx* c, size_t off) { return reinterpret_cast<T*>(c->arena + off); }

// One committed row stream of T tokens: whole boxes, with room for the tokens fdkv_fold_tail may append later.
size_t row_stream_bytes(const Shape& s, int T) {
    return (size_t)((T + s.max_fold + kRowPad - 1) / kRowPad * kRowPad) * s.d * s.esize;
}

// Copies of a commit or a fold, collected in classes that are launched one after the other.
template <int CLASSES>
struct CopyTable {
    std::vector<CopyJob> jobs[CLASSES];
    void rows(int cls, const void* src, void* dst, size_t bytes, int64_t src_pitch, int row_bytes) {
        jobs[cls].push_back(CopyJob{(const char*)src, (char*)dst, (int64_t)bytes, src_pitch, row_bytes, 0});
    }
    void plain(int cls, const void* src, void* dst, size_t bytes, int add = 0) {
        if (bytes) jobs[cls].push_back(CopyJob{(const char*)src, (char*)dst, (int64_t)bytes, 16, 16, add});
    }
    void zero(int cls, void* dst, size_t bytes) { plain(cls, nullptr, dst, bytes); }
    // `pin`: page-locked room for the whole table, not written again before `st` has been waited for
    cudaError_t launch(CopyJob* table_dev, CopyJob* pin, cudaStream_t st) const {
        size_t n = 0;
        for (const auto& v : jobs) {
            if (!v.empty()) std::memcpy(pin + n, v.data(), v.size() * sizeof(CopyJob));
            n += v.size();
        }
        if (n == 0) return cudaSuccess;
        cudaError_t e = cudaMemcpyAsync(table_dev, pin, n * sizeof(CopyJob), cudaMemcpyHostToDevice, st);
        for (const auto& v : jobs) {
            int64_t most = 0;
            for (const CopyJob& jb : v) most = std::max(most, jb.bytes);
            if (e == cudaSuccess) e = launch_copy_jobs(table_dev, (int)v.size(), most, st);
            table_dev += v.size();
        }
        return e;
    }
};

// Page-locked blocks of closed contexts, kept for the next ones (page-locking takes 0.14 ms): at most kBlocks of at most kMost
// bytes each, the rest is freed.  A context gives its block back when no copy from or to it is under way.
struct PinPool {
    static constexpr size_t kBlocks = 4, kMost = 1 << 20;
    std::mutex lock;
    std::vector<std::pair<size_t, char*>> idle;  // (bytes, block)
    cudaError_t take(size_t& bytes, char** out) {  // (bytes: in, what is needed; out, what the block has)
        {
            std::lock_guard<std::mutex> g(lock);
            for (size_t i = 0; i < idle.size(); ++i)
                if (idle[i].first >= bytes) {
                    bytes = idle[i].first;
                    *out = idle[i].second;
                    idle.erase(idle.begin() + i);
                    return cudaSuccess;
                }
        }
        return cudaHostAlloc(reinterpret_cast<void**>(out), bytes, cudaHostAllocPortable);
    }
    void give(size_t bytes, char* block) {
        {
            std::lock_guard<std::mutex> g(lock);
            if (idle.size() < kBlocks && bytes <= kMost) {
                idle.emplace_back(bytes, block);
                return;
            }
        }
        cudaFreeHost(block);
    }
};
PinPool& pin_pool() {
    static PinPool* p = new PinPool;  // (never destroyed: contexts may be closed while the process exits)
    return *p;
}

// A sequence's descriptors to the device (the caller waits for `st` before they change again).
cudaError_t copy_descriptors(fdkv_ctx* c, int seq, cudaStream_t st) {
    const size_t n = (size_t)c->s.L * c->s.Hkv, bytes = n * sizeof(UnitDesc);
    std::memcpy(c->pin + c->pin_desc, &c->desc_host[(size_t)seq * n], bytes);
    return cudaMemcpyAsync(c->arena + c->ar.desc + (size_t)seq * bytes, c->pin + c->pin_desc, bytes, cudaMemcpyHostToDevice, st);
}

bool seq_ok(fdkv_ctx* c, int seq) { return c && seq >= 0 && seq < c->s.max_batch; }

// Omega(m) of Eq. 2 for one unit (K and V together): bytes of the mode / bytes of the exact mode.  Returns the latter.
// Residual bytes per kept position: one value and one int32 index (pair), four layer values and one index (block of
// four); token rule: d values per kept token and one index.
double omega_of(const Shape& s, int T, double (&om)[3]) {
    const double e = s.esize, Td = (double)T * s.d;
    const double k = (double)((int64_t)T * s.d * s.keep_num / s.keep_den);
    const double k_tok = (double)((int64_t)T * s.keep_num / s.keep_den);
    const double b_sh = 2.0 * Td * e, b_ex = 2.0 * s.B * Td * e;
    double b_rs;
    if (s.tok_rule) b_rs = b_sh + 2.0 * k_tok * s.d * e * s.NB + 4.0 * k_tok;
    else b_rs = b_sh + 2.0 * k * (s.NB * e + 4.0);
    om[0] = b_sh / b_ex; om[1] = b_rs / b_ex; om[2] = 1.0;
    return b_ex;
}

// What a prompt of T tokens and a folded chunk of T tokens have in common.
CompressArgs entry_args(fdkv_ctx* c, int T) {
    const Shape& s = c->s;
    CompressArgs a;
    a.T = T; a.d = s.d; a.Hkv = s.Hkv; a.tensors = 2;
    a.unit_stride = (int64_t)s.Tmax * s.d;
    a.z1 = nullptr;
    a.sel = wsp<SelState>(c, c->ws.sel);
    a.cand_pos = wsp<uint16_t>(c, c->ws.cand_pos);
    a.cand_val = c->work + c->ws.cand_val;
    a.cand_n = wsp<int32_t>(c, c->ws.cand_n);
    a.chunk_base = wsp<int2>(c, c->ws.chunk_base);
    a.cand_stride = s.cand_stride; a.chunks_max = s.chunks_max;
    a.n_keep = (int64_t)T * s.d * s.keep_num / s.keep_den; a.kcap = s.kcap;
    a.in_place = false;
    a.ntiles_max = s.ntiles_max;
    a.tile_off = wsp<int32_t>(c, c->ws.tile_off);
    a.idx = wsp<int32_t>(c, c->ws.idx);
    a.val = c->work + c->ws.val;
    a.packed = c->packed_lists ? wsp<uint32_t>(c, c->ws.packed) : nullptr;
    a.keep = nullptr; a.keep_stride = s.cand_stride / 32;
    a.status = wsp<int32_t>(c, c->ws.status);
    return a;
}

}  // namespace

namespace fdkv {
void count_launch(int n) { g_launches.fetch_add(n); }
void count_kernel(int id) { if (id >= 0 && id < FDKV_KERNEL_COUNT_) g_kernel_launches[id].fetch_add(1); }
int per_device_first_visits(const int* devs, int n) {
    // the table logic of PerDevice::ensure, fed with device ids instead of the current device
    bool done[PerDevice::kMaxDevices] = {};
    int visits = 0;
    for (int i = 0; i < n; ++i) {
        if (devs[i] < 0 || devs[i] >= PerDevice::kMaxDevices) continue;
        if (!done[devs[i]]) { done[devs[i]] = true; ++visits; }
    }
    return visits;
}
fdkv_status record_cuda_error(cudaError_t e) { return cuda_fail(e); }
cudaError_t launch_set_tail_len(int32_t* tail_len, int L, int max_batch, int seq, int n, cudaStream_t st);
}  // namespace fdkv

extern "C" {

fdkv_status fdkv_sizes(const fdkv_config* cfg, size_t* arena_bytes, size_t* workspace_bytes) {
    Shape s;
    if (!cfg || !make_shape(*cfg, s)) return cfg ? FDKV_ERR_UNSUPPORTED : FDKV_ERR_INVALID_ARG;
    WsLayout w;
    ArenaLayout a;
    make_layouts(s, w, a);
    if (arena_bytes) *arena_bytes = a.worst_total;
    if (workspace_bytes) *workspace_bytes = w.total;
    return FDKV_OK;
}

fdkv_status fdkv_create(const fdkv_config* cfg, void* arena, size_t arena_bytes, void* workspace,
                        size_t workspace_bytes, fdkv_ctx** out) {
    if (!cfg || !arena || !workspace || !out) return FDKV_ERR_INVALID_ARG;
    if (!aligned(arena, 256) || !aligned(workspace, 256)) return FDKV_ERR_INVALID_ARG;
    Shape s;
    if (!make_shape(*cfg, s)) return FDKV_ERR_UNSUPPORTED;
    fdkv_ctx* c = new (std::nothrow) fdkv_ctx();
    if (!c) return FDKV_ERR_INVALID_ARG;
    c->cfg = *cfg;
    c->s = s;
    make_layouts(s, c->ws, c->ar);
    if (workspace_bytes < c->ws.total) { delete c; return FDKV_ERR_WORKSPACE; }
    if (arena_bytes < c->ar.bump) { delete c; return FDKV_ERR_ARENA_FULL; }
    c->arena = (char*)arena;
    c->arena_bytes = arena_bytes;
    c->work = (char*)workspace;
    c->work_bytes = workspace_bytes;
    c->bump = c->ar.bump;
    c->pair_compressed.assign(s.P, 0);
    c->pair_probed.assign(s.P, 0);
    c->pair_scored.assign(s.P, 0);
    c->k_layers.assign(s.L, nullptr);
    c->v_layers.assign(s.L, nullptr);
    c->seqs.resize(s.max_batch);
    for (auto& q : c->seqs) { q.modes.assign(s.NU, -1); q.tail_len.assign(s.L, 0); }
    c->desc_host.resize((size_t)s.max_batch * s.L * s.Hkv);
    c->plans.resize(s.L);
    cudaError_t e = cudaMemset(c->arena + c->ar.tail_len, 0, (size_t)s.L * s.max_batch * 4);
    if (e == cudaSuccess) e = cudaMemset(c->work + c->ws.status, 0, 256);
    if (e == cudaSuccess) e = cudaMemset(c->arena + c->ar.desc, 0, c->desc_host.size() * sizeof(UnitDesc));
    // tails start as zero rows: the fast decode kernel loads whole 64-row boxes and relies on finite padding
    if (e == cudaSuccess) e = cudaMemset(c->arena + c->ar.tail_k, 0, c->ar.bump - c->ar.tail_k);
    c->pin_jobs = align_up((size_t)s.NU * 16);
    c->pin_gather = c->pin_jobs + 2 * align_up(max_copy_jobs(s) * sizeof(CopyJob));  // (a fold has two tables on the way)
    c->pin_desc = c->pin_gather + align_up(gather_table_bytes(s));
    c->pin_bytes = c->pin_desc + (size_t)s.L * s.Hkv * sizeof(UnitDesc);
    if (e == cudaSuccess) e = pin_pool().take(c->pin_bytes, &c->pin);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->probe_done, cudaEventDisableTiming);
    if (e != cudaSuccess) { fdkv_destroy(c); return cuda_fail(e); }
    if (s.dtype == FDKV_BF16 && s.d == 128) c->has_tmap = make_arena_tensor_map(c->arena, arena_bytes, c->tmap);
    c->packed_lists = c->has_tmap && s.max_batch * s.Hkv <= kFastMaxUnits;
    if (s.rows_f8 && !(c->packed_lists && make_arena_tensor_map_u8(c->arena, arena_bytes, c->tmap_u8))) { fdkv_destroy(c); return FDKV_ERR_UNSUPPORTED; }
    // token rule: the tensor-core score kernel and the packed decode kernel serve bf16 / head_dim 128; everything else
    // takes the float32 score kernel and the portable decode kernel
    if (s.tok_rule && c->packed_lists)
        c->tok_tc = make_rows_tensor_map(c->work + c->ws.z1, (size_t)s.NU * s.NB * s.Tmax * s.d * s.esize, 128, c->tmap_z1_128);
    if (s.tok_rule && s.dtype == FDKV_BF16 && s.d == 128 && !c->tok_tc) { fdkv_destroy(c); return FDKV_ERR_UNSUPPORTED; }
    if (s.dtype == FDKV_BF16 && s.d == 128 && !s.tok_rule)
        c->has_probe_tmaps = make_rows_tensor_map(c->work + c->ws.z1, (size_t)s.NU * s.NB * s.Tmax * s.d * s.esize, 128, c->tmap_z1_128) &&
                             make_rows_tensor_map(c->work + c->ws.z1, (size_t)s.NU * s.NB * s.Tmax * s.d * s.esize, kProbeBoxRows, c->tmap_z1) &&
                             make_rows_tensor_map(c->work + c->ws.z1drop, (size_t)s.NU * s.NB * s.Tmax * s.d * s.esize, kProbeBoxRows, c->tmap_drop);
    *out = c;
    return FDKV_OK;
}

void fdkv_destroy(fdkv_ctx* ctx) {
    if (!ctx) return;
    const bool idle = !ctx->probe_recorded || cudaEventSynchronize(ctx->probe_done) == cudaSuccess;  // (scores on their way)
    if (ctx->probe_done) cudaEventDestroy(ctx->probe_done);
    if (ctx->pin && idle) pin_pool().give(ctx->pin_bytes, ctx->pin);
    delete ctx;
}

fdkv_status fdkv_reset(fdkv_ctx* c) {
    if (!c) return FDKV_ERR_INVALID_ARG;
    CU(cudaDeviceSynchronize());
    CU(cudaMemset(c->arena + c->ar.tail_len, 0, (size_t)c->s.L * c->s.max_batch * 4));
    CU(cudaMemset(c->work + c->ws.status, 0, 256));
    CU(cudaMemset(c->arena + c->ar.tail_k, 0, c->ar.bump - c->ar.tail_k));
    c->bump = c->ar.bump;
    ++c->plan_epoch;
    c->staged_seq = -1;
    for (auto& q : c->seqs) {
        q.committed = false;
        q.T = 0;
        q.fold_used = 0;
        q.k_entries = 0;
        q.modes.assign(c->s.NU, -1);
        q.tail_len.assign(c->s.L, 0);
        q.bytes_by_mode[0] = q.bytes_by_mode[1] = q.bytes_by_mode[2] = 0;
    }
    return FDKV_OK;
}

fdkv_status fdkv_compress_prefill(fdkv_ctx* c, int32_t seq, int32_t pb, int32_t pe, int32_t T,
                                  const void* const* k_layers, const void* const* v_layers, int64_t stride_t,
                                  int64_t stride_h, void* stream) {
    if (!seq_ok(c, seq) || !k_layers || !v_layers) return FDKV_ERR_INVALID_ARG;
    const Shape& s = c->s;
    if (pb < 0 || pe > s.P || pb >= pe) return FDKV_ERR_INVALID_ARG;
    if (T < 1 || T > s.Tmax) return FDKV_ERR_INVALID_ARG;
    if (stride_h < s.d || stride_t < s.d || (stride_t % 8) || (stride_h % 8)) return FDKV_ERR_INVALID_ARG;
    for (int l = s.B * pb; l < s.B * pe; ++l)
        if (!k_layers[l] || !v_layers[l] || !aligned(k_layers[l], 16) || !aligned(v_layers[l], 16))
            return FDKV_ERR_INVALID_ARG;
    if (c->seqs[seq].committed) return FDKV_ERR_STATE;
    if (c->staged_seq != seq || c->staged_T != T) {
        c->staged_seq = seq;
        c->staged_T = T;
        std::fill(c->pair_compressed.begin(), c->pair_compressed.end(), 0);
        std::fill(c->pair_probed.begin(), c->pair_probed.end(), 0);
        std::fill(c->pair_scored.begin(), c->pair_scored.end(), 0);
        c->modes_overridden = false;
        c->seqs[seq].modes.assign(s.NU, -1);
        c->stride_t = stride_t;
        c->stride_h = stride_h;
        // Every unit's committed form holds at least two row streams, so the shared coefficients go where commit would
        // put them (shared / residual units keep them there; an exact unit's two slots take two of its own streams): commit
        // then copies nothing for most units.  A full arena, or rows that commit quantises, stage them in the workspace.
        const size_t stream = align_up(row_stream_bytes(s, T));
        c->z0_in_arena = !s.rows_f8 && c->bump + (size_t)s.NT * stream <= c->arena_bytes;
        c->z0_base = c->z0_in_arena ? c->arena + c->bump : c->work + c->ws.z0;
        c->z0_stride = c->z0_in_arena ? stream : (size_t)s.Tmax * s.d * s.esize;
        c->z0_loc.resize(s.NT);
        for (int ut = 0; ut < s.NT; ++ut) c->z0_loc[ut] = c->z0_base + ut * c->z0_stride;
    } else if (c->stride_t != stride_t || c->stride_h != stride_h) {
        return FDKV_ERR_INVALID_ARG;
    }
    cudaStream_t st = S(stream);
    for (int l = s.B * pb; l < s.B * pe; ++l) { c->k_layers[l] = k_layers[l]; c->v_layers[l] = v_layers[l]; }
    if (s.tok_rule) {
        // the token rule selects inside fdkv_probe: only the split here
        constexpr int kMost = kSplitLayers;
        for (int p0 = pb; p0 < pe; p0 += kMost / s.B) {
            SplitRowsArgs a;
            a.n_blocks = std::min(pe - p0, kMost / s.B);
            for (int l = 0; l < a.n_blocks * s.B; ++l) {
                a.k[l] = k_layers[s.B * p0 + l];
                a.v[l] = v_layers[s.B * p0 + l];
            }
            a.stride_t = stride_t; a.stride_h = stride_h;
            a.T = T; a.d = s.d; a.Hkv = s.Hkv;
            a.ut_base = p0 * s.Hkv * 2;
            a.unit_stride = (int64_t)s.Tmax * s.d; a.z0_stride = (int64_t)(c->z0_stride / s.esize);
            a.z0 = c->z0_base; a.hf = c->work + c->ws.z1;
            CU(launch_split_rows(a, s.B, s.dtype, st));
        }
        for (int p = pb; p < pe; ++p) { c->pair_compressed[p] = 1; c->pair_probed[p] = 0; c->pair_scored[p] = 0; }
        return FDKV_OK;
    }
    CompressArgs a = entry_args(c, T);
    a.stride_t = stride_t; a.stride_h = stride_h;
    a.z0 = c->z0_base; a.z0_stride = (int64_t)(c->z0_stride / s.esize);
    a.z1 = c->work + c->ws.z1;
    a.keep = c->has_probe_tmaps ? wsp<uint32_t>(c, c->ws.keep) : nullptr;
    CU(launch_compress(a, s.B, s.dtype, k_layers, v_layers, pb, pe, st));
    for (int p = pb; p < pe; ++p) { c->pair_compressed[p] = 1; c->pair_probed[p] = 0; c->pair_scored[p] = 0; }
    return FDKV_OK;
}

fdkv_status fdkv_probe(fdkv_ctx* c, int32_t seq, int32_t pb, int32_t pe, const void* const* q_layers,
                       const int32_t* probe_pos, int32_t W, double lambda, int32_t* modes, float* scores,
                       void* stream) {
    if (!seq_ok(c, seq) || !q_layers || !probe_pos) return FDKV_ERR_INVALID_ARG;
    const Shape& s = c->s;
    if (pb < 0 || pe > s.P || pb >= pe || W < 1 || W > kMaxW) return FDKV_ERR_INVALID_ARG;
    if (!(lambda >= 0.0)) return FDKV_ERR_INVALID_ARG;
    if (c->staged_seq != seq) return FDKV_ERR_STATE;
    for (int p = pb; p < pe; ++p)
        if (!c->pair_compressed[p]) return FDKV_ERR_STATE;
    const int T = c->staged_T;
    for (int i = 0; i < W; ++i)
        if (probe_pos[i] < 0 || probe_pos[i] >= T || (i && probe_pos[i] <= probe_pos[i - 1])) return FDKV_ERR_INVALID_ARG;
    for (int l = s.B * pb; l < s.B * pe; ++l)
        if (!q_layers[l] || !aligned(q_layers[l], 16)) return FDKV_ERR_INVALID_ARG;
    cudaStream_t st = S(stream);
    int32_t* pos_dev = wsp<int32_t>(c, c->ws.probe_pos);
    const void** qptr_dev = reinterpret_cast<const void**>(c->work + c->ws.probe_pos + kMaxW * 4);
    CU(launch_probe_inputs(pos_dev, probe_pos, W, qptr_dev, q_layers, s.B * pb, s.B * pe, st));
    ProbeArgs a;
    a.B = s.B;
    a.unit_begin = pb * s.Hkv; a.unit_count = (pe - pb) * s.Hkv;
    a.T = T; a.d = s.d; a.Hq = s.Hq; a.Hkv = s.Hkv; a.G = s.G; a.W = W;
    a.unit_stride = (int64_t)s.Tmax * s.d; a.kcap = s.kcap;
    a.ntiles_max = s.ntiles_max; a.nptiles_max = s.nptiles_max;
    a.z1 = c->work + c->ws.z1; a.z1drop = c->work + c->ws.z1drop;
    a.keep = s.tok_rule ? nullptr : wsp<uint32_t>(c, c->ws.keep); a.keep_stride = s.cand_stride / 32;
    a.idx = wsp<int32_t>(c, c->ws.idx);
    a.tile_off = wsp<int32_t>(c, c->ws.tile_off);
    a.sums_ready = s.tok_rule;
    a.q_layers_dev = qptr_dev;
    a.pos = pos_dev;
    a.part = wsp<double>(c, c->ws.probe_part);
    a.scale = wsp<double>(c, c->ws.probe_scale);
    a.redo = wsp<int32_t>(c, c->ws.probe_redo);
    a.moments = c->probe_moments;
    a.scores = wsp<double>(c, c->ws.scores);
    a.modes = wsp<int32_t>(c, c->ws.modes);
    a.lambda = lambda;
    omega_of(s, T, a.omega);
    a.modes_out = modes; a.scores_out = scores;
    a.tmap_z1 = c->has_probe_tmaps ? c->tmap_z1 : nullptr;
    a.tmap_drop = c->has_probe_tmaps ? c->tmap_drop : nullptr;
    a.tmap_z1_128 = c->tmap_z1_128;
    a.Tmax = s.Tmax;
    a.pos_host = probe_pos;
    a.status = wsp<int32_t>(c, c->ws.status);
    if (s.tok_rule) {
        TokenArgs t;
        t.B = s.B;
        t.unit_begin = a.unit_begin; t.unit_count = a.unit_count;
        t.T = T; t.Tmax = s.Tmax; t.Hq = s.Hq; t.Hkv = s.Hkv; t.G = s.G; t.W = W; t.ntiles_max = s.ntiles_max;
        t.k_tok = (int64_t)T * s.keep_num / s.keep_den; t.ktok_cap = s.ktok_cap; t.unit_stride = (int64_t)s.Tmax * s.d;
        t.z1 = c->work + c->ws.z1;
        t.q_layers_dev = qptr_dev; t.pos = pos_dev; t.pos_host = probe_pos;
        t.score = wsp<uint32_t>(c, c->ws.tok_score);
        t.err = wsp<float>(c, c->ws.tok_err); t.nslots = token_err_slots(s.B, s.G, c->tok_tc, W);
        t.part = a.part; t.nptiles_max = s.nptiles_max; t.pos_last = probe_pos[W - 1];
        t.list = wsp<int32_t>(c, c->ws.tok_list); t.off = wsp<int32_t>(c, c->ws.tok_off);
        t.tmap_z1_128 = c->tmap_z1_128;
        t.status = wsp<int32_t>(c, c->ws.status);
        CU(launch_token_select(t, s.dtype, s.d, c->tok_tc, st));
        for (int p = pb; p < pe; ++p) c->pair_scored[p] = 1;
    }
    CU(launch_probe(a, s.dtype, st));
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    CU(cudaStreamIsCapturing(st, &capture));
    if (capture != cudaStreamCaptureStatusNone) {
        c->probe_captured = true;  // (an event of a capture says nothing about its replays)
    } else {
        const size_t su = (size_t)a.unit_begin * 16;
        CU(cudaMemcpyAsync(c->pin + su, c->work + c->ws.scores + su, (size_t)a.unit_count * 16, cudaMemcpyDeviceToHost, st));
        if (c->probe_recorded && c->probe_stream != st) CU(cudaStreamWaitEvent(st, c->probe_done, 0));
        CU(cudaEventRecord(c->probe_done, st));
        c->probe_stream = st;
        c->probe_recorded = true;
    }
    for (int p = pb; p < pe; ++p) c->pair_probed[p] = 1;
    return FDKV_OK;
}

fdkv_status fdkv_route_budget(fdkv_ctx* c, int32_t seq, size_t budget_bytes, double* lambda_host, int32_t* modes_host,
                              void* stream) {
    if (!seq_ok(c, seq)) return FDKV_ERR_INVALID_ARG;
    if (c->staged_seq != seq) return FDKV_ERR_STATE;
    const Shape& s = c->s;
    for (int p = 0; p < s.P; ++p)
        if (!c->pair_probed[p]) return FDKV_ERR_STATE;
    CU(cudaStreamSynchronize(S(stream)));
    if (c->probe_captured) CU(cudaMemcpy(c->pin, c->work + c->ws.scores, (size_t)s.NU * 16, cudaMemcpyDeviceToHost));
    else CU(cudaEventSynchronize(c->probe_done));  // (probed on another stream)
    const double* const e = reinterpret_cast<const double*>(c->pin);
    // Omega of the staged sequence, as in fdkv_probe
    const int T = c->staged_T;
    double om[3];
    const double b_ex = omega_of(s, T, om);
    auto mode_at = [&](int u, double lam) {
        const double L0 = e[2 * u] + lam * om[0], L1 = e[2 * u + 1] + lam * om[1], L2 = lam * om[2];
        int m = 0;
        double best = L0;
        if (L1 < best) { best = L1; m = 1; }
        if (L2 < best) { best = L2; m = 2; }
        return m;
    };
    // The footprint only changes where two loss lines of a unit cross, and only downwards: the smallest lambda that fits is 0 or
    // just past a crossing, found by bisection (128 units, 385 crossings: the device waited 0.1 ms for a scan of them).
    std::vector<double> cand;
    cand.reserve((size_t)s.NU * 3 + 1);
    cand.push_back(0.0);
    auto add = [&](double cv) { if (cv >= 0.0 && !std::isinf(cv)) cand.push_back(cv); };
    for (int u = 0; u < s.NU; ++u) {
        add((e[2 * u] - e[2 * u + 1]) / (om[1] - om[0]));
        add(e[2 * u + 1] / (om[2] - om[1]));
        add(e[2 * u] / (om[2] - om[0]));
    }
    std::sort(cand.begin(), cand.end());
    std::vector<int32_t> modes(s.NU, 0);
    // (just past a crossing: the unit already took its cheaper mode, 2^-40 being far above the rounding of the losses)
    auto past = [&](size_t i) { return cand[i] * (1.0 + std::ldexp(1.0, -40)); };
    auto fits_at = [&](size_t i) {
        const double lam = past(i);
        double total = 0.0;
        for (int u = 0; u < s.NU; ++u) {
            modes[u] = mode_at(u, lam);
            total += om[modes[u]] * b_ex;
        }
        return total <= (double)budget_bytes;
    };
    size_t lo = 0, hi = cand.size();  // [0, lo) do not fit, [hi, end) fit
    while (lo < hi) {
        const size_t mid = (lo + hi) / 2;
        if (fits_at(mid)) hi = mid; else lo = mid + 1;
    }
    const bool fits = lo < cand.size() && fits_at(lo);  // (leaves the modes of lo)
    const double lam_found = fits ? past(lo) : INFINITY;
    if (!fits) std::fill(modes.begin(), modes.end(), 0);
    c->seqs[seq].modes = modes;
    c->modes_overridden = true;
    if (lambda_host) *lambda_host = lam_found;
    if (modes_host) std::memcpy(modes_host, modes.data(), (size_t)s.NU * 4);
    return fits ? FDKV_OK : FDKV_ERR_ARENA_FULL;
}

fdkv_status fdkv_set_modes(fdkv_ctx* c, int32_t seq, const int32_t* modes_host) {
    if (!seq_ok(c, seq) || !modes_host) return FDKV_ERR_INVALID_ARG;
    if (c->staged_seq != seq) return FDKV_ERR_STATE;
    for (int i = 0; i < c->s.NU; ++i)
        if (modes_host[i] < 0 || modes_host[i] > 2) return FDKV_ERR_INVALID_ARG;
    c->seqs[seq].modes.assign(modes_host, modes_host + c->s.NU);
    c->modes_overridden = true;
    return FDKV_OK;
}

fdkv_status fdkv_commit(fdkv_ctx* c, int32_t seq, void* stream) {
    if (!seq_ok(c, seq)) return FDKV_ERR_INVALID_ARG;
    if (c->staged_seq != seq || c->seqs[seq].committed) return FDKV_ERR_STATE;
    const Shape& s = c->s;
    for (int p = 0; p < s.P; ++p)
        if (!c->pair_compressed[p] || (!c->modes_overridden && !c->pair_probed[p]) || (s.tok_rule && !c->pair_scored[p]))
            return FDKV_ERR_STATE;
    cudaStream_t st = S(stream);
    SeqState& q = c->seqs[seq];
    CU(cudaStreamSynchronize(st));
    if (!c->modes_overridden)
        CU(cudaMemcpy(q.modes.data(), c->work + c->ws.modes, (size_t)s.NU * 4, cudaMemcpyDeviceToHost));
    const int T = c->staged_T;
    const size_t rows = (size_t)T * s.d * s.esize;
    const size_t rows_pad = row_stream_bytes(s, T);  // (zero rows up to its end)
    const int64_t k = (int64_t)T * s.d * s.keep_num / s.keep_den;
    const int ntiles = (T + kResTile - 1) / kResTile;
    // list copies include the slack so that aligned over-reads of the last tile stay inside the allocation
    // (copy_* = what the staging area holds now; the allocations add the room of the folded chunks)
    const size_t idx_copy = (size_t)(k + kListPad) * 4, off_copy = (size_t)(ntiles + 1) * 4;
    const size_t val_copy = c->packed_lists ? 0 : (size_t)(k + kListPad) * s.esize;  // packed entries carry their value
    const size_t idx_b = idx_copy + (size_t)s.kfold_max * 4, off_b = off_copy + (size_t)(s.max_fold / kResTile + 1) * 4;
    const size_t val_b = c->packed_lists ? 0 : val_copy + (size_t)s.kfold_max * s.esize;
    const int64_t k_tok = (int64_t)T * s.keep_num / s.keep_den;
    const size_t trow_b = (size_t)(k_tok + 4) * s.d * s.esize, tlist_b = (size_t)(k_tok + 32) * 4;  // token rows, token list
    // 8-bit row streams: 128 bytes per token and a 1 KiB slot for the channel scales (and their maxima) per stored tensor
    const size_t rows8 = (size_t)T * 128, rows8_pad = (size_t)((T + kRowPad - 1) / kRowPad * kRowPad) * 128, scale_slot = 1024;
    const size_t stream_b = s.rows_f8 ? align_up(rows8_pad) + scale_slot : align_up(rows_pad);  // one committed row stream
    size_t need = 0;
    // residual lists of one tensor: packed layout = one entry list per stored high-frequency tensor (one for a pair,
    // four for a block of four layers); portable layout = one index list and one value list per such tensor
    const size_t lists_b = c->packed_lists ? (size_t)s.NB * align_up(idx_b) : align_up(idx_b) + (size_t)s.NB * align_up(val_b);
    for (int u = 0; u < s.NU; ++u) {
        const int m = q.modes[u];
        if (m < 0 || m > 2) return FDKV_ERR_STATE;
        if (m == FDKV_MODE_EXACT) need += 2 * (size_t)s.B * stream_b;
        else if (s.tok_rule) need += 2 * align_up(rows_pad) + (m == FDKV_MODE_RESIDUAL ? 2 * (size_t)s.NB * align_up(trow_b) + align_up(tlist_b) + align_up(off_b) : 0);
        else need += 2 * stream_b + (m == FDKV_MODE_RESIDUAL ? 2 * (lists_b + align_up(off_b)) : 0);
    }
    if (c->bump + need > c->arena_bytes) return FDKV_ERR_ARENA_FULL;
    const bool in_place = c->z0_in_arena;
    size_t o = c->bump + (in_place ? (size_t)s.NT * c->z0_stride : 0);
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes); return c->arena + r; };
    size_t by_mode[3] = {0, 0, 0};
    const size_t unit_stride_b = (size_t)s.Tmax * s.d * s.esize;
    std::vector<QuantJob> qjobs;   // 8-bit rows: every stored tensor is quantised by one batched pass after this loop
    std::vector<RepackJob> rjobs;  // ... and every residual list repacked relative to its tensor's scales
    std::vector<TokenGatherJob> gjobs;  // token rule: the selected rows, formed from the caller's K and V
    // device-to-device copies into the arena and zero fills: one launch per class of size after the loop
    enum { kSaveJobs, kRowJobs, kListJobs, kSmallJobs, kJobClasses };  // (in launch order)
    CopyTable<kJobClasses> copies;
    for (int u = 0; u < s.NU; ++u) {
        const int m = q.modes[u], p = u / s.Hkv, h = u % s.Hkv;
        UnitDesc* dl[4] = {nullptr, nullptr, nullptr, nullptr};
        for (int l = 0; l < s.B; ++l) {
            dl[l] = &c->desc_host[((size_t)seq * s.L + (size_t)s.B * p + l) * s.Hkv + h];
            std::memset(dl[l], 0, sizeof(UnitDesc));
            dl[l]->mode = m;
            dl[l]->T = T;
            dl[l]->sign = s.B == 2 ? (l == 0 ? 1.f : -1.f) : 2.f;
            dl[l]->scale = m == FDKV_MODE_EXACT ? 1.f : (s.B == 2 ? 0.70710678118654752440f : 0.5f);
        }
        if (m == FDKV_MODE_EXACT) {
            for (int l = 0; l < s.B; ++l)
                for (int is_v = 0; is_v < 2; ++is_v) {
                    const void* src = is_v ? c->v_layers[s.B * p + l] : c->k_layers[s.B * p + l];
                    const char* sp = (const char*)src + (size_t)h * c->stride_h * s.esize;
                    if (s.rows_f8) {
                        char* dst = take(rows8_pad);
                        float* sc = reinterpret_cast<float*>(take(scale_slot));
                        copies.zero(kSmallJobs, dst + rows8, rows8_pad - rows8);
                        qjobs.push_back(QuantJob{sp, c->stride_t, T, 0, reinterpret_cast<uint8_t*>(dst), sc});
                        (is_v ? dl[l]->v_rows : dl[l]->k_rows) = dst;
                        (is_v ? dl[l]->v_scale : dl[l]->k_scale) = sc;
                        dl[l]->rows_f8 = 1;
                        continue;
                    }
                    char* dst;
                    if (in_place && l == 0) {  // the unit's own Z0 slot; its Z0 stays readable in the workspace
                        const size_t ut = (size_t)u * 2 + is_v;
                        dst = c->z0_base + ut * c->z0_stride;
                        c->z0_loc[ut] = c->work + c->ws.z0 + ut * unit_stride_b;
                        copies.plain(kSaveJobs, dst, c->z0_loc[ut], rows);
                    } else {
                        dst = take(rows_pad);
                    }
                    copies.zero(kSmallJobs, dst + rows, rows_pad - rows);
                    copies.rows(kRowJobs, sp, dst, rows, (int64_t)c->stride_t * s.esize, s.d * s.esize);
                    (is_v ? dl[l]->v_rows : dl[l]->k_rows) = dst;
                }
            by_mode[2] += 2 * (size_t)s.B * (s.rows_f8 ? rows8 + 512 : rows);
        } else {
            char *tl = nullptr, *to = nullptr;
            if (s.tok_rule && m == FDKV_MODE_RESIDUAL) {  // one token list and one offset table serve K and V
                tl = take(tlist_b);
                to = take(off_b);
                copies.plain(kSmallJobs, c->work + c->ws.tok_list + (size_t)u * s.ktok_cap * 4, tl, (size_t)k_tok * 4);
                copies.plain(kSmallJobs, c->work + c->ws.tok_off + (size_t)u * (s.ntiles_max + 1) * 4, to, off_copy);
                by_mode[1] += (size_t)k_tok * 4;
            }
            for (int is_v = 0; is_v < 2; ++is_v) {
                const size_t ut = (size_t)u * 2 + is_v;
                float* sc8 = nullptr;
                char* z0;
                if (s.rows_f8) {
                    z0 = take(rows8_pad);
                    sc8 = reinterpret_cast<float*>(take(scale_slot));
                    copies.zero(kSmallJobs, z0 + rows8, rows8_pad - rows8);
                    qjobs.push_back(QuantJob{c->work + c->ws.z0 + ut * unit_stride_b, s.d, T, 0, reinterpret_cast<uint8_t*>(z0), sc8});
                    for (int l = 0; l < s.B; ++l) { (is_v ? dl[l]->v_scale : dl[l]->k_scale) = sc8; dl[l]->rows_f8 = 1; }
                } else {
                    z0 = in_place ? c->z0_base + ut * c->z0_stride : take(rows_pad);
                    copies.zero(kSmallJobs, z0 + rows, rows_pad - rows);
                    if (!in_place) copies.plain(kRowJobs, c->z0_loc[ut], z0, rows);
                }
                for (int l = 0; l < s.B; ++l) (is_v ? dl[l]->v_rows : dl[l]->k_rows) = z0;
                by_mode[m] += s.rows_f8 ? rows8 + 512 : rows;
                if (m == FDKV_MODE_RESIDUAL && s.tok_rule) {
                    // the selected tokens' high-frequency rows, densely packed: Z1 rows of a pair (both layers read them with
                    // opposite signs), each layer's own deviation rows of a block of four (stored doubled: see the gather kernel)
                    // (the list is read where the probe left it: its copy into the arena runs with the other copies after this loop)
                    char* rows_l[4] = {nullptr, nullptr, nullptr, nullptr};
                    TokenGatherJob gj;
                    std::memset(&gj, 0, sizeof(gj));
                    for (int l = 0; l < s.B; ++l)
                        gj.x[l] = (const char*)(is_v ? c->v_layers[s.B * p + l] : c->k_layers[s.B * p + l]) + (size_t)h * c->stride_h * s.esize;
                    for (int j = 0; j < s.NB; ++j) gj.dst[j] = rows_l[j] = take(trow_b);
                    gj.list = wsp<int32_t>(c, c->ws.tok_list) + (size_t)u * s.ktok_cap;
                    gj.stride_t = c->stride_t;
                    gj.k_tok = k_tok;
                    gj.twice = (s.B == 4 && c->packed_lists) ? 1 : 0;
                    gjobs.push_back(gj);
                    if (s.rows_f8)  // 8-bit rows: the kept rows become f16(value / scale[channel]) in the fragment order of the 8-bit tiles
                        for (int j = 0; j < s.NB; ++j)
                            rjobs.push_back(RepackJob{reinterpret_cast<uint32_t*>(rows_l[j]), reinterpret_cast<const uint32_t*>(rows_l[j]), k_tok, sc8, is_v, 1});
                    for (int l = 0; l < s.B; ++l) {
                        UnitDesc* d = dl[l];
                        d->res_kind = 1;
                        d->k_idx = (const int32_t*)tl;
                        d->k_off = (const int32_t*)to;
                        (is_v ? d->v_val : d->k_val) = rows_l[s.NB == 1 ? 0 : l];
                    }
                    by_mode[1] += (size_t)s.NB * k_tok * s.d * s.esize;
                } else if (m == FDKV_MODE_RESIDUAL) {
                    char* po = take(off_b);
                    copies.plain(kSmallJobs, c->work + c->ws.tile_off + ut * (s.ntiles_max + 1) * 4, po, off_copy);
                    char* pi_shared = nullptr;
                    if (!c->packed_lists) {
                        pi_shared = take(idx_b);
                        copies.plain(kListJobs, c->work + c->ws.idx + ut * s.kcap * 4, pi_shared, idx_copy);
                    }
                    char *pi_l[4] = {nullptr, nullptr, nullptr, nullptr}, *pv_l[4] = {nullptr, nullptr, nullptr, nullptr};
                    for (int j = 0; j < s.NB; ++j) {  // one list per stored high-frequency tensor
                        const size_t lt = ut * s.NB + j;
                        if (c->packed_lists) {
                            pi_l[j] = take(idx_b);
                            if (s.rows_f8)  // values relative to the channel scales, positions in the converted fragments' order
                                rjobs.push_back(RepackJob{reinterpret_cast<uint32_t*>(pi_l[j]), wsp<uint32_t>(c, c->ws.packed) + lt * s.kcap, k, sc8, is_v, 0});
                            else
                                copies.plain(kListJobs, c->work + c->ws.packed + lt * s.kcap * 4, pi_l[j], idx_copy);
                        } else {
                            pi_l[j] = pi_shared;
                            pv_l[j] = take(val_b);
                            // (whole words: an odd count of 2-byte values takes one value of the list's slack along)
                            copies.plain(kListJobs, c->work + c->ws.val + lt * s.kcap * s.esize, pv_l[j], (val_copy + 3) & ~(size_t)3);
                        }
                    }
                    for (int l = 0; l < s.B; ++l) {
                        UnitDesc* d = dl[l];
                        const int j = s.NB == 1 ? 0 : l;  // a pair's two layers read the same Z1 list with opposite signs
                        (is_v ? d->v_idx : d->k_idx) = (const int32_t*)pi_l[j];
                        (is_v ? d->v_val : d->k_val) = pv_l[j];
                        (is_v ? d->v_off : d->k_off) = (const int32_t*)po;
                    }
                    by_mode[1] += (size_t)k * (c->packed_lists ? (size_t)4 * s.NB : 4 + (size_t)s.NB * s.esize);
                }
            }
        }
    }
    char* const table = c->work + c->ws.jobs + quant_table_bytes(s);
    if (!gjobs.empty()) {
        std::memcpy(c->pin + c->pin_gather, gjobs.data(), gjobs.size() * sizeof(TokenGatherJob));
        CU(cudaMemcpyAsync(table, c->pin + c->pin_gather, gjobs.size() * sizeof(TokenGatherJob), cudaMemcpyHostToDevice, st));
        CU(launch_token_gather_jobs(reinterpret_cast<TokenGatherJob*>(table), (int)gjobs.size(), k_tok, s.d, s.B, s.dtype, st));
    }
    CU(copy_descriptors(c, seq, st));
    CU(copies.launch(reinterpret_cast<CopyJob*>(table + gather_table_bytes(s)), reinterpret_cast<CopyJob*>(c->pin + c->pin_jobs), st));
    if (!qjobs.empty()) {
        QuantJob* qd = reinterpret_cast<QuantJob*>(c->work + c->ws.jobs);
        RepackJob* rd = reinterpret_cast<RepackJob*>(qd + (size_t)s.NU * 2 * s.B);
        CU(cudaMemcpyAsync(qd, qjobs.data(), qjobs.size() * sizeof(QuantJob), cudaMemcpyHostToDevice, st));
        CU(launch_quantise_jobs(qd, (int)qjobs.size(), T, st));
        if (!rjobs.empty()) {
            CU(cudaMemcpyAsync(rd, rjobs.data(), rjobs.size() * sizeof(RepackJob), cudaMemcpyHostToDevice, st));
            CU(launch_repack_jobs(rd, (int)rjobs.size(), s.tok_rule ? k_tok * 32 : k, st));
        }
    }
    CU(cudaStreamSynchronize(st));
    c->bump = o;
    ++c->plan_epoch;
    q.committed = true;
    q.T = T;
    q.fold_used = 0;
    q.k_entries = k;
    for (int i = 0; i < 3; ++i) q.bytes_by_mode[i] = by_mode[i];
    return FDKV_OK;
}

static fdkv_status decode_impl(fdkv_ctx* c, int32_t layer, int32_t batch, const void* q, const void* k_new,
                               const void* v_new, void* out, int32_t out_dtype, cudaStream_t st) {
    const Shape& s = c->s;
    int Tmax = 0;
    for (int b = 0; b < batch; ++b) {
        if (!c->seqs[b].committed) return FDKV_ERR_STATE;
        Tmax = c->seqs[b].T > Tmax ? c->seqs[b].T : Tmax;
    }
    if (k_new) {
        for (int b = 0; b < batch; ++b)
            if (c->seqs[b].tail_len[layer] >= s.max_tail) return FDKV_ERR_STATE;
        for (int b = 0; b < batch; ++b) c->seqs[b].tail_len[layer]++;
    }
    std::vector<int32_t>&host_T = c->host_T, &host_modes = c->host_modes, &host_tail = c->host_tail;
    host_T.resize(batch); host_modes.resize((size_t)batch * s.Hkv); host_tail.resize(batch);
    for (int b = 0; b < batch; ++b) {
        host_T[b] = c->seqs[b].T;
        for (int h = 0; h < s.Hkv; ++h) host_modes[(size_t)b * s.Hkv + h] = c->seqs[b].modes[(layer / s.B) * s.Hkv + h];
    }
    DecodeArgs a;
    a.tail_rows = s.tail_rows;
    a.host_T = host_T.data(); a.host_modes = host_modes.data();
    a.plan = &c->plans[layer];
    a.plan_epoch = c->plan_epoch;
    a.any_tail = 0;
    for (int b = 0; b < batch; ++b) {  // (already counts this call's append)
        host_tail[b] = c->seqs[b].tail_len[layer];
        a.any_tail |= host_tail[b] > 0;
    }
    a.host_tail = host_tail.data();
    a.tmap = c->has_tmap ? c->tmap : nullptr;
    a.tmap_u8 = s.rows_f8 ? c->tmap_u8 : nullptr;
    a.rows_f8 = s.rows_f8;
    a.arena_base = c->arena;
    a.keep_num = s.keep_num; a.keep_den = s.keep_den;
    a.packed_lists = c->packed_lists ? 1 : 0;
    a.tok_rule = s.tok_rule;
    a.desc = arp<UnitDesc>(c, c->ar.desc);
    a.L = s.L; a.layer = layer; a.batch = batch; a.Hq = s.Hq; a.Hkv = s.Hkv; a.G = s.G; a.d = s.d;
    a.max_tail = s.max_tail; a.max_batch = s.max_batch; a.Tmax_batch = Tmax;
    a.q = q; a.k_new = k_new; a.v_new = v_new; a.out = out; a.out_dtype = out_dtype;
    a.tail_k = c->arena + c->ar.tail_k; a.tail_v = c->arena + c->ar.tail_v;
    a.tail_len = arp<int32_t>(c, c->ar.tail_len);
    a.partials = wsp<float>(c, c->ws.partials);
    a.status = wsp<int32_t>(c, c->ws.status);
    CU(launch_decode(a, s.dtype, st));
    return FDKV_OK;
}

fdkv_status fdkv_decode_attn(fdkv_ctx* c, int32_t layer, int32_t batch, const void* q, const void* k_new,
                             const void* v_new, void* out, int32_t out_dtype, void* stream) {
    if (!c || !q || !out) return FDKV_ERR_INVALID_ARG;
    if (layer < 0 || layer >= c->s.L || batch < 1 || batch > c->s.max_batch) return FDKV_ERR_INVALID_ARG;
    if ((k_new == nullptr) != (v_new == nullptr)) return FDKV_ERR_INVALID_ARG;
    if (out_dtype != FDKV_F32 && out_dtype != FDKV_BF16) return FDKV_ERR_INVALID_ARG;
    if (!aligned(q, 16) || !aligned(out, 16) || !aligned(k_new, 16) || !aligned(v_new, 16)) return FDKV_ERR_INVALID_ARG;
    return decode_impl(c, layer, batch, q, k_new, v_new, out, out_dtype, S(stream));
}

fdkv_status fdkv_decode_attn_host(fdkv_ctx* c, int32_t layer, int32_t batch, const void* q, const void* k_new,
                                  const void* v_new, void* out, int32_t out_dtype, void* stream) {
    if (!c || !q || !out) return FDKV_ERR_INVALID_ARG;
    if (layer < 0 || layer >= c->s.L || batch < 1 || batch > c->s.max_batch) return FDKV_ERR_INVALID_ARG;
    if ((k_new == nullptr) != (v_new == nullptr)) return FDKV_ERR_INVALID_ARG;
    if (out_dtype != FDKV_F32 && out_dtype != FDKV_BF16) return FDKV_ERR_INVALID_ARG;
    const Shape& s = c->s;
    cudaStream_t st = S(stream);
    const size_t qb = (size_t)batch * s.Hq * s.d * s.esize, kb = (size_t)batch * s.Hkv * s.d * s.esize;
    const size_t ob = (size_t)batch * s.Hq * s.d * (out_dtype == FDKV_BF16 ? 2 : 4);
    CU(cudaMemcpyAsync(c->work + c->ws.io_q, q, qb, cudaMemcpyHostToDevice, st));
    if (k_new) {
        CU(cudaMemcpyAsync(c->work + c->ws.io_k, k_new, kb, cudaMemcpyHostToDevice, st));
        CU(cudaMemcpyAsync(c->work + c->ws.io_v, v_new, kb, cudaMemcpyHostToDevice, st));
    }
    fdkv_status r = decode_impl(c, layer, batch, c->work + c->ws.io_q, k_new ? c->work + c->ws.io_k : nullptr,
                                k_new ? c->work + c->ws.io_v : nullptr, c->work + c->ws.io_out, out_dtype, st);
    if (r != FDKV_OK) return r;
    CU(cudaMemcpyAsync(out, c->work + c->ws.io_out, ob, cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
    return FDKV_OK;
}

fdkv_status fdkv_decode_step_host(fdkv_ctx* c, int32_t batch, const void* q, const void* k_new, const void* v_new, void* out,
                                  int32_t out_dtype, void* stream) {
    if (!c || !q || !out) return FDKV_ERR_INVALID_ARG;
    if (batch < 1 || batch > c->s.max_batch) return FDKV_ERR_INVALID_ARG;
    if ((k_new == nullptr) != (v_new == nullptr)) return FDKV_ERR_INVALID_ARG;
    if (out_dtype != FDKV_F32 && out_dtype != FDKV_BF16) return FDKV_ERR_INVALID_ARG;
    const Shape& s = c->s;
    cudaStream_t st = S(stream);
    const size_t qb = (size_t)batch * s.Hq * s.d * s.esize, kb = (size_t)batch * s.Hkv * s.d * s.esize;
    const size_t ob = (size_t)batch * s.Hq * s.d * (out_dtype == FDKV_BF16 ? 2 : 4);
    CU(cudaMemcpyAsync(c->work + c->ws.io_q, q, qb * s.L, cudaMemcpyHostToDevice, st));
    if (k_new) {
        CU(cudaMemcpyAsync(c->work + c->ws.io_k, k_new, kb * s.L, cudaMemcpyHostToDevice, st));
        CU(cudaMemcpyAsync(c->work + c->ws.io_v, v_new, kb * s.L, cudaMemcpyHostToDevice, st));
    }
    for (int l = 0; l < s.L; ++l) {
        fdkv_status r = decode_impl(c, l, batch, c->work + c->ws.io_q + l * qb, k_new ? c->work + c->ws.io_k + l * kb : nullptr,
                                    k_new ? c->work + c->ws.io_v + l * kb : nullptr, c->work + c->ws.io_out + l * ob, out_dtype, st);
        if (r != FDKV_OK) return r;
    }
    CU(cudaMemcpyAsync(out, c->work + c->ws.io_out, ob * s.L, cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
    return FDKV_OK;
}

fdkv_status fdkv_set_tail_len(fdkv_ctx* c, int32_t seq, int32_t n, void* stream) {
    if (!seq_ok(c, seq) || n < 0) return FDKV_ERR_INVALID_ARG;
    for (int l = 0; l < c->s.L; ++l)
        if (n > c->seqs[seq].tail_len[l]) return FDKV_ERR_INVALID_ARG;
    CU(launch_set_tail_len(arp<int32_t>(c, c->ar.tail_len), c->s.L, c->s.max_batch, seq, n, S(stream)));
    c->seqs[seq].tail_len.assign(c->s.L, n);
    return FDKV_OK;
}

fdkv_status fdkv_fold_tail(fdkv_ctx* c, int32_t seq, int32_t n, void* stream) {
    if (!seq_ok(c, seq) || n <= 0) return FDKV_ERR_INVALID_ARG;
    const Shape& s = c->s;
    if (s.tok_rule || s.rows_f8) return FDKV_ERR_UNSUPPORTED;
    SeqState& q = c->seqs[seq];
    if (!q.committed) return FDKV_ERR_STATE;
    if (c->staged_seq >= 0 && !c->seqs[c->staged_seq].committed) return FDKV_ERR_STATE;  // the staging area is in use
    if ((q.T % kResTile) || (n % kResTile) || n > s.Tmax) return FDKV_ERR_INVALID_ARG;
    for (int l = 0; l < s.L; ++l)
        if (q.tail_len[l] != q.tail_len[0]) return FDKV_ERR_STATE;
    if (q.tail_len[0] < n) return FDKV_ERR_INVALID_ARG;
    if (q.fold_used + n > s.max_fold) return FDKV_ERR_ARENA_FULL;
    cudaStream_t st = S(stream);
    const int T0 = q.T, len = q.tail_len[0], rest = len - n;
    const size_t row_b = (size_t)s.d * s.esize;
    const size_t tail_head_b = (size_t)s.tail_rows * row_b;                       // one (layer, sequence, head) tail
    auto tail_base = [&](char* base, int l) { return base + ((size_t)l * s.max_batch + seq) * s.Hkv * tail_head_b; };
    char* tk = c->arena + c->ar.tail_k;
    char* tv = c->arena + c->ar.tail_v;
    // ---- Eq. 1 and the chunk's own selection, through the staging area ----
    c->staged_seq = -1;
    std::fill(c->pair_compressed.begin(), c->pair_compressed.end(), 0);
    const int64_t kc = (int64_t)n * s.d * s.keep_num / s.keep_den;
    {
        std::vector<const void*> kp(s.L), vp(s.L);
        for (int l = 0; l < s.L; ++l) { kp[l] = tail_base(tk, l); vp[l] = tail_base(tv, l); }
        CompressArgs a = entry_args(c, n);
        a.stride_t = s.d; a.stride_h = (int64_t)s.tail_rows * s.d;
        a.z0 = c->work + c->ws.z0; a.z0_stride = (int64_t)s.Tmax * s.d;
        CU(launch_compress(a, s.B, s.dtype, kp.data(), vp.data(), 0, s.P, st));
    }
    // ---- append behind every unit's rows and lists, under the unit's mode ----
    const size_t unit_stride_b = (size_t)s.Tmax * s.d * s.esize, chunk_b = (size_t)n * row_b, at = (size_t)T0 * row_b;
    const int64_t k_old = q.k_entries;
    const int nslices = n / kResTile;
    enum { kRowJobs, kSmallJobs, kJobClasses };
    CopyTable<kJobClasses> copies;
    for (int u = 0; u < s.NU; ++u) {
        const int m = q.modes[u], p = u / s.Hkv, h = u % s.Hkv;
        UnitDesc* dl[4] = {nullptr, nullptr, nullptr, nullptr};
        for (int l = 0; l < s.B; ++l) dl[l] = &c->desc_host[((size_t)seq * s.L + (size_t)s.B * p + l) * s.Hkv + h];
        if (m == FDKV_MODE_EXACT) {
            for (int l = 0; l < s.B; ++l) {
                copies.plain(kRowJobs, tail_base(tk, s.B * p + l) + h * tail_head_b, (char*)dl[l]->k_rows + at, chunk_b);
                copies.plain(kRowJobs, tail_base(tv, s.B * p + l) + h * tail_head_b, (char*)dl[l]->v_rows + at, chunk_b);
            }
            q.bytes_by_mode[2] += 2 * (size_t)s.B * chunk_b;
            continue;
        }
        for (int is_v = 0; is_v < 2; ++is_v) {
            const size_t ut = (size_t)u * 2 + is_v;
            char* rows = (char*)(is_v ? dl[0]->v_rows : dl[0]->k_rows);  // every layer of the block shares the coefficient rows
            copies.plain(kRowJobs, c->work + c->ws.z0 + ut * unit_stride_b, rows + at, chunk_b);
            q.bytes_by_mode[m] += chunk_b;
            if (m != FDKV_MODE_RESIDUAL) continue;
            int32_t* off = const_cast<int32_t*>(is_v ? dl[0]->v_off : dl[0]->k_off);
            if (c->packed_lists) {
                // packed entries carry slice-relative positions: valid as they are (T0 is a multiple of 16); one list per
                // stored high-frequency tensor (a pair's two layers share theirs)
                for (int j = 0; j < s.NB; ++j) {
                    int32_t* list = const_cast<int32_t*>(is_v ? dl[j]->v_idx : dl[j]->k_idx);
                    copies.plain(kSmallJobs, c->work + c->ws.packed + (ut * s.NB + j) * s.kcap * 4, list + k_old, (size_t)kc * 4);
                }
            } else {
                int32_t* list = const_cast<int32_t*>(is_v ? dl[0]->v_idx : dl[0]->k_idx);  // one index list for the unit
                copies.plain(kSmallJobs, wsp<int32_t>(c, c->ws.idx) + ut * s.kcap, list + k_old, (size_t)kc * 4, T0 * s.d);
                for (int j = 0; j < s.NB; ++j) {
                    char* val = (char*)const_cast<void*>(is_v ? dl[j]->v_val : dl[j]->k_val);
                    copies.plain(kSmallJobs, c->work + c->ws.val + (ut * s.NB + j) * s.kcap * s.esize, val + (size_t)k_old * s.esize, (size_t)kc * s.esize);
                }
            }
            copies.plain(kSmallJobs, wsp<int32_t>(c, c->ws.tile_off) + ut * (s.ntiles_max + 1), off + T0 / kResTile, (size_t)(nslices + 1) * 4, (int)k_old);
            q.bytes_by_mode[1] += (size_t)kc * (c->packed_lists ? (size_t)4 * s.NB : 4 + (size_t)s.NB * s.esize);
        }
    }
    CopyJob* const table = reinterpret_cast<CopyJob*>(c->work + c->ws.jobs + quant_table_bytes(s) + gather_table_bytes(s));
    CU(copies.launch(table, reinterpret_cast<CopyJob*>(c->pin + c->pin_jobs), st));
    // ---- the remaining tail rows move down: where the ranges overlap through the staging area, as many layers at a time as it
    // holds, or a layer in pieces from the front (a piece ends before the rows that the next one reads) ----
    if (rest > 0) {
        const bool overlap = rest > n;
        const size_t room = (size_t)s.NU * s.NB * unit_stride_b / (2 * s.Hkv * row_b);  // tokens of a layer that fit: at least 8
        const int piece = overlap ? (int)std::min<size_t>(rest, room) : rest;
        const int group = overlap ? (int)std::min<size_t>(s.L, room / piece) : s.L;
        for (int l0 = 0; l0 < s.L; l0 += group)
            for (int r0 = 0; r0 < rest; r0 += piece) {
                CopyTable<2> moves;
                const size_t w = (size_t)std::min(piece, rest - r0) * row_b;
                char* tmp = c->work + c->ws.z1;
                for (int l = l0; l < std::min(s.L, l0 + group); ++l)
                    for (char* base : {tail_base(tk, l), tail_base(tv, l)})
                        for (int h = 0; h < s.Hkv; ++h, base += tail_head_b, tmp += w) {
                            char* const to = base + (size_t)r0 * row_b;
                            moves.plain(0, to + (size_t)n * row_b, overlap ? tmp : to, w);
                            if (overlap) moves.plain(1, tmp, to, w);
                        }
                if (l0 > 0 || r0 > 0) CU(cudaStreamSynchronize(st));  // (the page-locked table is written again)
                CU(moves.launch(table, reinterpret_cast<CopyJob*>(c->pin + c->pin_jobs + align_up(max_copy_jobs(s) * sizeof(CopyJob))), st));
            }
    }
    CU(launch_set_tail_len(arp<int32_t>(c, c->ar.tail_len), s.L, s.max_batch, seq, rest, st));
    q.tail_len.assign(s.L, rest);
    // ---- descriptors: every layer of the sequence now holds T0 + n prompt-side tokens ----
    const size_t seq_desc = (size_t)s.L * s.Hkv;
    for (size_t i = 0; i < seq_desc; ++i) c->desc_host[(size_t)seq * seq_desc + i].T = T0 + n;
    CU(copy_descriptors(c, seq, st));
    CU(cudaStreamSynchronize(st));
    ++c->plan_epoch;
    q.T = T0 + n;
    q.k_entries = k_old + kc;
    q.fold_used += n;
    return FDKV_OK;
}

fdkv_status fdkv_get_rows_e4m3(fdkv_ctx* c, int32_t seq, int32_t layer, int32_t h, int32_t is_v, uint8_t* codes_out, float* scale_out,
                               void* stream) {
    if (!seq_ok(c, seq) || layer < 0 || layer >= c->s.L || h < 0 || h >= c->s.Hkv) return FDKV_ERR_INVALID_ARG;
    if (!c->s.rows_f8) return FDKV_ERR_UNSUPPORTED;
    if (!c->seqs[seq].committed) return FDKV_ERR_STATE;
    const UnitDesc& d = c->desc_host[((size_t)seq * c->s.L + layer) * c->s.Hkv + h];
    if (codes_out) CU(cudaMemcpyAsync(codes_out, is_v ? d.v_rows : d.k_rows, (size_t)d.T * 128, cudaMemcpyDeviceToDevice, S(stream)));
    if (scale_out) CU(cudaMemcpyAsync(scale_out, is_v ? d.v_scale : d.k_scale, 512, cudaMemcpyDeviceToDevice, S(stream)));
    CU(cudaStreamSynchronize(S(stream)));
    return FDKV_OK;
}

fdkv_status fdkv_get_shared(fdkv_ctx* c, int32_t seq, int32_t pair, int32_t h, int32_t is_v, void* z0_out, void* stream) {
    if (!seq_ok(c, seq) || !z0_out || pair < 0 || pair >= c->s.P || h < 0 || h >= c->s.Hkv) return FDKV_ERR_INVALID_ARG;
    if (c->staged_seq != seq || !c->pair_compressed[pair]) return FDKV_ERR_STATE;
    const Shape& s = c->s;
    const size_t ut = ((size_t)pair * s.Hkv + h) * 2 + (is_v ? 1 : 0);
    CU(cudaMemcpyAsync(z0_out, c->z0_loc[ut], (size_t)c->staged_T * s.d * s.esize,
                       cudaMemcpyDeviceToDevice, S(stream)));
    CU(cudaStreamSynchronize(S(stream)));
    return FDKV_OK;
}

fdkv_status fdkv_get_residual(fdkv_ctx* c, int32_t seq, int32_t pair, int32_t h, int32_t is_v, int32_t* idx_out,
                              void* val_out, int32_t* count_host, void* stream) {
    if (!seq_ok(c, seq) || pair < 0 || pair >= c->s.P || h < 0 || h >= c->s.Hkv) return FDKV_ERR_INVALID_ARG;
    if (c->staged_seq != seq || !c->pair_compressed[pair]) return FDKV_ERR_STATE;
    const Shape& s = c->s;
    if (s.tok_rule) return FDKV_ERR_UNSUPPORTED;  // token rule: see fdkv_get_token_set
    const size_t ut = ((size_t)pair * s.Hkv + h) * 2 + (is_v ? 1 : 0);
    const int64_t k = (int64_t)c->staged_T * s.d * s.keep_num / s.keep_den;
    if (count_host) *count_host = (int32_t)k;
    if (idx_out && k) CU(cudaMemcpyAsync(idx_out, c->work + c->ws.idx + ut * s.kcap * 4, (size_t)k * 4, cudaMemcpyDeviceToDevice, S(stream)));
    for (int j = 0; j < s.NB && val_out && k; ++j)  // a block of four returns its four layers' values as [4][count]
        CU(cudaMemcpyAsync((char*)val_out + (size_t)j * k * s.esize, c->work + c->ws.val + (ut * s.NB + j) * s.kcap * s.esize,
                           (size_t)k * s.esize, cudaMemcpyDeviceToDevice, S(stream)));
    CU(cudaStreamSynchronize(S(stream)));
    return FDKV_OK;
}

fdkv_status fdkv_get_token_set(fdkv_ctx* c, int32_t seq, int32_t pair, int32_t h, int32_t* tok_out, float* score_out,
                               int32_t* count_host, void* stream) {
    if (!seq_ok(c, seq) || pair < 0 || pair >= c->s.P || h < 0 || h >= c->s.Hkv) return FDKV_ERR_INVALID_ARG;
    const Shape& s = c->s;
    if (!s.tok_rule) return FDKV_ERR_UNSUPPORTED;
    if (c->staged_seq != seq || !c->pair_scored[pair]) return FDKV_ERR_STATE;
    const size_t u = (size_t)pair * s.Hkv + h;
    const int64_t k_tok = (int64_t)c->staged_T * s.keep_num / s.keep_den;
    if (count_host) *count_host = (int32_t)k_tok;
    if (tok_out && k_tok) CU(cudaMemcpyAsync(tok_out, c->work + c->ws.tok_list + u * s.ktok_cap * 4, (size_t)k_tok * 4, cudaMemcpyDeviceToDevice, S(stream)));
    if (score_out) CU(cudaMemcpyAsync(score_out, c->work + c->ws.tok_score + u * s.Tmax * 4, (size_t)c->staged_T * 4, cudaMemcpyDeviceToDevice, S(stream)));
    CU(cudaStreamSynchronize(S(stream)));
    return FDKV_OK;
}

fdkv_status fdkv_get_modes(fdkv_ctx* c, int32_t seq, int32_t* modes_host) {
    if (!seq_ok(c, seq) || !modes_host) return FDKV_ERR_INVALID_ARG;
    if (!c->seqs[seq].committed && !(c->staged_seq == seq && c->modes_overridden)) return FDKV_ERR_STATE;
    std::memcpy(modes_host, c->seqs[seq].modes.data(), (size_t)c->s.NU * 4);
    return FDKV_OK;
}

fdkv_status fdkv_footprint(fdkv_ctx* c, int32_t seq, size_t* bytes_by_mode_host, size_t* exact_equiv_bytes_host) {
    if (!seq_ok(c, seq)) return FDKV_ERR_INVALID_ARG;
    if (!c->seqs[seq].committed) return FDKV_ERR_STATE;
    if (bytes_by_mode_host)
        for (int i = 0; i < 3; ++i) bytes_by_mode_host[i] = c->seqs[seq].bytes_by_mode[i];
    if (exact_equiv_bytes_host)
        *exact_equiv_bytes_host = (size_t)c->s.NU * 2 * c->s.B * c->seqs[seq].T * c->s.d * c->s.esize;
    return FDKV_OK;
}

fdkv_status fdkv_plan_decode(int32_t batch, int32_t n_kv_heads, const int32_t* T_host, const int32_t* modes_host,
                             int32_t keep_num, int32_t keep_den, int32_t residual_rule, int32_t row_format, int32_t n_ctas,
                             uint32_t* start_out, int32_t* n_ctas_out, int32_t* parts_out) {
    if (!T_host || !modes_host || !start_out || !n_ctas_out || !parts_out) return FDKV_ERR_INVALID_ARG;
    if (batch < 1 || n_kv_heads < 1 || (int64_t)batch * n_kv_heads > kFastMaxUnits || n_ctas < 1 || n_ctas > 160) return FDKV_ERR_INVALID_ARG;
    if (keep_num < 0 || keep_den < 1 || keep_num > keep_den) return FDKV_ERR_INVALID_ARG;
    for (int b = 0; b < batch; ++b)
        if (T_host[b] < 1 || (int64_t)T_host[b] * 128 >= ((int64_t)1 << 31)) return FDKV_ERR_INVALID_ARG;
    for (int i = 0; i < batch * n_kv_heads; ++i)
        if (modes_host[i] < 0 || modes_host[i] > 2) return FDKV_ERR_INVALID_ARG;
    DecodeArgs a;
    std::memset(&a, 0, sizeof(a));
    a.batch = batch; a.Hkv = n_kv_heads; a.d = 128;
    a.host_T = T_host; a.host_modes = modes_host;
    a.keep_num = keep_num; a.keep_den = keep_den;
    a.tok_rule = residual_rule == FDKV_RESIDUAL_TOKENS ? 1 : 0;
    a.rows_f8 = row_format != 0 ? 1 : 0;
    return plan_decode_host(a, n_ctas, nullptr, start_out, n_ctas_out, parts_out, nullptr) == cudaSuccess ? FDKV_OK : FDKV_ERR_INVALID_ARG;
}

fdkv_status fdkv_decode_bytes(fdkv_ctx* c, int32_t layer, int32_t batch, size_t* bytes_host) {
    if (!c || !bytes_host || layer < 0 || layer >= c->s.L || batch < 1 || batch > c->s.max_batch) return FDKV_ERR_INVALID_ARG;
    const Shape& s = c->s;
    size_t tot = 0;
    for (int b = 0; b < batch; ++b) {
        const SeqState& q = c->seqs[b];
        if (!q.committed) return FDKV_ERR_STATE;
        const int64_t k = q.k_entries;  // prompt + folded chunks
        const int ntiles = (q.T + kResTile - 1) / kResTile;
        for (int h = 0; h < s.Hkv; ++h) {
            const int m = q.modes[(layer / s.B) * s.Hkv + h];
            tot += s.rows_f8 ? 2 * ((size_t)q.T * s.d + 512) + 2 * (size_t)q.tail_len[layer] * s.d * s.esize
                             : 2 * (size_t)(q.T + q.tail_len[layer]) * s.d * s.esize;
            if (m == FDKV_MODE_RESIDUAL && s.tok_rule) {
                const size_t kt = (size_t)((int64_t)q.T * s.keep_num / s.keep_den);
                tot += 2 * kt * s.d * s.esize + kt * 4 + (size_t)(ntiles + 1) * 4;
            } else if (m == FDKV_MODE_RESIDUAL)
                tot += 2 * ((size_t)k * (c->packed_lists ? 4 : 4 + s.esize) + (size_t)(ntiles + 1) * 4);
        }
    }
    *bytes_host = tot;
    return FDKV_OK;
}

fdkv_status fdkv_device_status(fdkv_ctx* c) {
    if (!c) return FDKV_ERR_INVALID_ARG;
    int32_t flag = 0;
    CU(cudaDeviceSynchronize());
    CU(cudaMemcpy(&flag, c->work + c->ws.status, 4, cudaMemcpyDeviceToHost));
    if (flag == kFlagOk) return FDKV_OK;
    return flag == kFlagTimeout ? FDKV_ERR_TIMEOUT : FDKV_ERR_DEVICE;
}

int32_t fdkv_last_cuda_error(void) { return g_last_cuda.load(); }

const char* fdkv_status_str(fdkv_status s) {
    switch (s) {
        case FDKV_OK: return "ok";
        case FDKV_ERR_INVALID_ARG: return "invalid argument";
        case FDKV_ERR_UNSUPPORTED: return "unsupported shape or dtype";
        case FDKV_ERR_ARENA_FULL: return "arena full";
        case FDKV_ERR_WORKSPACE: return "workspace too small";
        case FDKV_ERR_STATE: return "call order / state";
        case FDKV_ERR_CUDA: return "CUDA runtime error";
        case FDKV_ERR_TIMEOUT: return "device wait timed out";
        case FDKV_ERR_DEVICE: return "device-side check failed";
        case FDKV_ERR_TOO_LARGE: return "input larger than the built-in scratch of the allocation-free entry point";
    }
    return "unknown";
}

int64_t fdkv_launch_count(void) { return g_launches.load(); }
int64_t fdkv_kernel_launch_count(int32_t kernel) {
    return kernel >= 0 && kernel < FDKV_KERNEL_COUNT_ ? g_kernel_launches[kernel].load() : -1;
}

}  // extern "C"
