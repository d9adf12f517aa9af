// Internal declarations shared by the translation units of libfdkv (not part of the public ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <mutex>
#include <vector>

#include "../../include/fdkv.h"

namespace fdkv {

constexpr int kResTile = 16;         // tokens per residual-offset tile: off[j] = first list entry of tokens >= 16 j
constexpr int kMaxSplits = 160;      // split-K partial slots per (sequence, query head)
constexpr int kMaxW = 128;           // probe queries
constexpr int kListPad = 32;         // slack entries after each residual list (aligned over-reads stay in bounds)
constexpr int kMaxGroup = 8;
constexpr int kProbeBoxRows = 256;   // key tokens per tile of the tensor-core probe (rows of its TMA boxes)
constexpr int kFastMaxUnits = 1024;   // (sequences x KV heads) one launch of the bf16 / head_dim 128 decode kernel plans for
constexpr int kProbeTile = 64;       // tokens per probe CTA (generic kernel)
constexpr int kRowPad = 128;         // packed row blocks and tails are padded (zero rows) to this many tokens

enum DeviceFlag : int32_t { kFlagOk = 0, kFlagTimeout = 1, kFlagCountMismatch = 2, kFlagTailFull = 3 };

// What decode reads for one (sequence, layer, KV head).
struct UnitDesc {
    const void* k_rows;  // [T][d]: Z0 of K (shared / residual) or the layer's original K rows (exact)
    const void* v_rows;
    // residual mode only.  Portable layout: ascending flat indices t*d + ch and the stored values.  Packed layout
    // (bf16, head_dim 128): k_idx holds one 32-bit word per entry, value bits in the low half and the entry's
    // position inside its 16-token slice (a ready-made shared-memory offset / 2) in the high half; k_val is null.
    const int32_t* k_idx;
    const void* k_val;
    const int32_t* k_off;  // [ceil(T/16) + 1] first entry of each 16-token tile
    const int32_t* v_idx;
    const void* v_val;
    const int32_t* v_off;
    int32_t mode;
    int32_t T;
    float sign;  // multiplier of the residual values relative to the rows: +1 / -1 for the two layers of a pair,
                 // 2 for a layer of a four-layer block (rows scaled by 1/2, deviations by 1)
    int32_t res_kind;  // residual layout: 0 packed entries (k_idx / v_idx), 1 token rows (k_idx = token list, k_val / v_val = rows, k_off = per-slice counts)
    float scale;       // what the stored rows are multiplied by: 1/sqrt 2 (pair coefficients), 1/2 (block of four), 1 (exact)
    int32_t rows_f8;   // 1: k_rows / v_rows hold e4m3 codes (128 bytes per token) with per-channel scales below
    const float* k_scale;  // [d] float32, rows_f8 only
    const float* v_scale;
};

// Schedule of one launch of the bf16 / head_dim 128 decode kernel (decode_fast.cu): travels in the launch parameters.
struct FastSched {
    uint32_t start[kMaxSplits + 1];  // unit << 20 | first 16-token slice of CTA c; start[ncta] = units << 20
    uint8_t slot[kMaxSplits];        // split-K part of CTA c's first unit that CTA c writes (its later units start with it: part 0)
    int ncta, units;
    int cluster;   // thread blocks per unit, one cluster each, in one kernel; 0: the ranges are free and a second kernel combines
    float inv_share;  // (clusters) 1 / outputs of a unit that one block joins
    int any_tail;  // some sequence of the batch holds generated tokens in this layer's tail (host mirror)
};
struct PartCount {
    uint8_t n[kFastMaxUnits];  // split-K parts per unit (at most kMaxSplits)
};
// The schedule depends on the committed lengths and modes, the batch and the tails in whole tiles, and costs more host time
// than the rest of a call: every layer keeps its last one (in the context) until one of these changes.
struct FastPlan {
    uint64_t epoch = 0;             // fdkv_ctx::plan_epoch it was made in (0: none yet)
    int batch = 0;
    int sm_count = 0;
    std::vector<int32_t> tail_tiles;  // [batch]
    FastSched sch;
    PartCount pc;
};

struct SelState {
    uint32_t lo;      // bound the candidates reach (31-bit key pattern; bf16 magnitudes are shifted left by 16)
    uint32_t tau;     // threshold key: that of the k-th largest (until it is known: whether the sample puts it near the bound)
    uint32_t need;    // entries with key == tau to keep (lowest flat indices first)
    uint32_t redo;    // fewer than k positions reached the bound: split and threshold run again with bound 0
};

struct Shape {
    int L, P, Hq, Hkv, G, d;
    int max_batch, Tmax, max_tail;
    int dtype, esize;
    int keep_num, keep_den;
    int64_t kmax;      // floor(Tmax*d*num/den)
    int64_t kcap;      // list capacity incl. slack
    int ntiles_max;    // ceil(Tmax/16)
    int nptiles_max;   // ceil(Tmax/kProbeTile)
    int NU, NT;        // units and unit-tensors (K and V) of one sequence
    int tail_rows;     // max_tail rounded up to kRowPad
    int tok_rule;      // 1: token-granular residual chosen by the probe
    int B;             // layers per depth block: 2 or 4
    int max_fold;      // generated tokens that may be folded into the compressed form per sequence
    int rows_f8;       // committed row streams are e4m3 codes with per-channel scales
    int64_t kfold_max; // floor(max_fold*d*num/den): list room reserved for them
    int NB;            // high-frequency tensors per unit-tensor: 1 (Z1 of a pair) or 4 (the layers' deviations)
    int64_t cand_stride;  // Tmax*d rounded up to whole candidate chunks
    int chunks_max;
    int64_t ktok_max, ktok_cap;  // floor(Tmax*num/den) and the list capacity incl. slack
};

struct WsLayout {
    size_t tok_score, tok_err, tok_list, tok_off;
    size_t status, z0, z1, z1drop, cand_pos, cand_val, cand_n, chunk_base, keep, sel, tile_off, idx, val, packed, probe_part, probe_scale, probe_redo,
        probe_pos, scores, modes,
        partials, io_q, io_k, io_v, io_out, jobs, total;  // io_*: host-I/O staging, [L] layers each
};
struct ArenaLayout {
    size_t tail_len, desc, tail_k, tail_v, bump, worst_total;
};

struct SeqState {
    bool committed = false;
    int T = 0;
    std::vector<int32_t> modes;  // [NU], -1 unknown
    size_t bytes_by_mode[3] = {0, 0, 0};
    std::vector<int32_t> tail_len;  // host mirror per layer
    int fold_used = 0;              // tokens folded so far
    int64_t k_entries = 0;          // entries per residual list (prompt + folded chunks)
};

}  // namespace fdkv

struct fdkv_ctx {
    fdkv_config cfg;
    fdkv::Shape s;
    fdkv::WsLayout ws;
    fdkv::ArenaLayout ar;
    char* arena;
    size_t arena_bytes;
    char* work;
    size_t work_bytes;
    size_t bump;  // next free arena offset
    int staged_seq = -1;
    int staged_T = 0;
    std::vector<uint8_t> pair_compressed, pair_probed;
    // Shared coefficients of the staged sequence: [NT] at z0_base, z0_stride bytes apart -- in the arena where commit leaves
    // them when it has room for them (z0_in_arena), else in the workspace; z0_loc is where each can be read now.
    char* z0_base = nullptr;
    size_t z0_stride = 0;
    bool z0_in_arena = false;
    std::vector<char*> z0_loc;
    std::vector<const void*> k_layers, v_layers;
    int64_t stride_t = 0, stride_h = 0;
    bool modes_overridden = false;
    std::vector<fdkv::SeqState> seqs;
    std::vector<fdkv::UnitDesc> desc_host;  // [max_batch][L][Hkv]
    uint64_t plan_epoch = 1;                // advanced whenever a committed length or mode changes
    std::vector<fdkv::FastPlan> plans;      // [L]
    std::vector<int32_t> host_T, host_modes, host_tail;  // what a decode call's launch is planned from (kept: no allocation per call)
    alignas(64) unsigned char tmap[128];    // CUtensorMap of the arena (bf16, head_dim 128 only)
    bool has_tmap = false;
    alignas(64) unsigned char tmap_z1[128], tmap_drop[128];  // probe operands (bf16, head_dim 128 only)
    bool has_probe_tmaps = false;
    alignas(64) unsigned char tmap_z1_128[128];  // staged Z1 with 128-token boxes (token-score and second-moment kernels)
    bool tok_tc = false;                         // token rule served by the tensor-core kernels (bf16, head_dim 128)
    // Page-locked host memory, so that the tables of a commit or a fold go to the device without being staged by the driver, and
    // the probe's scores come back behind the probe's kernels instead of in a copy of their own when the budget is solved.
    char* pin = nullptr;
    size_t pin_bytes = 0, pin_jobs = 0, pin_gather = 0, pin_desc = 0;  // its size and offsets (the scores come first)
    cudaEvent_t probe_done = nullptr;                   // the scores of every probe call so far have landed
    cudaStream_t probe_stream = nullptr;                // where it was recorded last
    bool probe_recorded = false;
    int probe_moments = 0;                              // ProbeArgs::moments (set by tests)
    bool probe_captured = false;                        // a probe call was captured: its replays leave the scores on the device only
    std::vector<uint8_t> pair_scored;            // token rule: the probe has chosen this pair's token sets
    bool packed_lists = false;              // decode runs the bf16 / head_dim 128 kernel on packed residual entries
    alignas(64) unsigned char tmap_u8[128]; // CUtensorMap of the arena as 128-byte rows (8-bit row streams)
};

namespace fdkv {

// ---- launchers implemented in compress.cu / probe.cu / decode.cu; each returns cudaGetLastError() ----
// The split alone (token rule), either block size; layer B * j + l is layer l of the launch's block j.
constexpr int kSplitLayers = 64;  // layers one launch covers
struct SplitRowsArgs {
    const void *k[kSplitLayers], *v[kSplitLayers];
    int n_blocks;
    int64_t stride_t, stride_h;
    int T, d, Hkv;
    int ut_base;          // first unit-tensor of the first block
    int64_t unit_stride;  // elements between staged tensors (Tmax*d)
    int64_t z0_stride;    // elements between the unit-tensors' shared coefficients
    void* z0;             // [NT][z0_stride]
    void* hf;             // [unit][1 or 4][unit_stride]: Z1 of K of a pair, or the layers' deviations of a block of four
};
cudaError_t launch_split_rows(const SplitRowsArgs& a, int B, int dtype, cudaStream_t st);

// ---- entry rule: split, threshold, lists (select.cu) ----
// positions of a candidate chunk: 256 threads take 8 positions of B layers as 128 bytes of each thread's loads
__host__ __device__ constexpr int compress_chunk(int B, int esize) { return 8 / (B * esize / 2) * 256 * 8; }
constexpr int kMaxCompressChunk = 8192;
struct CompressArgs {
    const void *k[kSplitLayers], *v[kSplitLayers];  // set by launch_compress: layer B * j + l is layer l of the launch's block j
    int64_t stride_t, stride_h;
    int T, d, Hkv;
    int tensors;          // 2: K and V of every head (unit-tensor = head*2 + is_v); 1: K only (unit-tensor = head)
    int ut_base;          // set by launch_compress
    int64_t unit_stride;  // elements between staged high-frequency tensors (Tmax*d)
    int64_t z0_stride;    // elements between the unit-tensors' shared coefficients
    void* z0;             // [NT][z0_stride]
    void* z1;             // optional [unit][1 or 4][unit_stride]: high-frequency rows of K (Z1 of a pair, the deviations of a block of four)
    SelState* sel;        // [NT]
    uint16_t* cand_pos;   // [NT][cand_stride] positions inside the chunk, ascending; chunk c's at c * compress_chunk
    void* cand_val;       // [NT][1 or 4][cand_stride] their high-frequency values
    int32_t* cand_n;      // [NT][chunks_max] candidates per chunk
    int2* chunk_base;     // [NT][chunks_max] keys above / equal to the threshold in the chunks before
    int64_t cand_stride;  // Tmax*d rounded up to whole chunks
    int chunks_max;
    int chunks;           // set by launch_compress: chunks of T tokens
    int64_t n_keep, kcap; // entries per list and list capacity
    bool in_place;        // z0 may be written where a layer's rows are
    int ntiles_max;
    int32_t* tile_off;    // [NT][ntiles_max + 1]
    int32_t* idx;         // [NT][kcap]
    void* val;            // [NT][1 or 4][kcap]
    uint32_t* packed;     // optional [NT][1 or 4][kcap] packed entries of the bf16 / head_dim 128 decode kernel
    uint32_t* keep;       // optional [unit][keep_stride] bit map of the kept positions of K
    int64_t keep_stride;  // 32-bit words
    int32_t* status;
};
cudaError_t launch_compress(CompressArgs& a, int B, int dtype, const void* const* k_layers, const void* const* v_layers, int block_begin, int block_end,
                            cudaStream_t st);

struct ProbeArgs {
    int B;  // layers per block: 2 (one Z1 operand, both layers' queries) or 4 (one deviation operand per layer)
    int unit_begin, unit_count;  // units of the pair range (unit = pair*Hkv + h)
    int T, d, Hq, Hkv, G, W;
    int64_t unit_stride, kcap;
    int ntiles_max, nptiles_max;
    const void* z1;        // [unit][1 or 4][unit_stride] high-frequency rows of K
    void* z1drop;          // [unit][1 or 4][unit_stride] room for a copy without the kept entries (tensor-core probe), or null
    const uint32_t* keep;  // [unit][keep_stride] bit map of the kept positions of K
    int64_t keep_stride;
    const int32_t* idx;
    const int32_t* tile_off;
    bool sums_ready;                  // token rule: part slot 0 of every unit holds the error sums already
    const void* const* q_layers_dev;  // device array [L] of pointers
    const int32_t* pos;
    double* part;    // [NU][nptiles_max][2]
    double* scale;   // [NU][kMaxGramSlots][2] what the second moments' sums are to be large against
    int moments;     // second moments where they pay (0), for all keys that every query sees (1: tests), never (2: tests)
    int32_t* redo;   // [NU] the second moments' sums are not exact enough: the unit is done again by products
    double* scores;  // [NU][2]
    int32_t* modes;  // [NU]
    double lambda, omega[3];
    int32_t* modes_out;  // user buffers for the pair range, may be null
    float* scores_out;
    // tensor-core path (bf16, head_dim 128): tensor maps over the staged Z1 and the dropped copy, viewed as
    // [rows][128] bf16 with 128-token x 64-channel boxes; null when unavailable
    const void *tmap_z1, *tmap_drop;
    const void* tmap_z1_128;  // the staged Z1 with 128-token boxes
    int Tmax;
    const int32_t* pos_host;
    int32_t* status;
};
cudaError_t launch_probe(const ProbeArgs& a, int dtype, cudaStream_t st);
// The probe positions and the query pointers of layers [layer_begin, layer_end) to the device, from HOST arrays.
cudaError_t launch_probe_inputs(int32_t* pos_dev, const int32_t* pos, int W, const void** q_dev, const void* const* q_layers, int layer_begin, int layer_end,
                                cudaStream_t st);
constexpr int kMaxGramCtas = 160;  // blocks of the second-moment kernel
constexpr int kMaxGramSlots = kMaxGramCtas + 2 * 4;  // ... and so part slots a unit may need
// Part slots of a unit: [0, gram) second moments, [gram, sure) products, [sure, all) products in the place of the second moments
// for units that are done again.
struct ProbeParts {
    int gram, sure, all;
};
cudaError_t launch_probe_gram(const ProbeArgs& a, int t_full, cudaStream_t st, int* nparts);

struct DecodeArgs {
    const UnitDesc* desc;  // [batch][.. layer ..] : desc + (b*L + layer)*Hkv + h
    int L, layer, batch, Hq, Hkv, G, d, max_tail, max_batch;
    int Tmax_batch;  // largest T among the batch (host side, sizes the grid)
    const void *q, *k_new, *v_new;
    void* out;
    int out_dtype;
    void *tail_k, *tail_v;  // [L][max_batch][Hkv][tail_rows][d], tail_rows = max_tail rounded up to kRowPad
    int tail_rows;
    // host-side views used only to plan the launch (valid during the call)
    const int32_t* host_T;      // [batch]
    const int32_t* host_modes;  // [batch][Hkv] modes of this layer's pair
    const int32_t* host_tail;   // [batch] generated tokens in this layer's tail per sequence (after this call's append), or null
    FastPlan* plan;             // the layer's kept schedule, or null (planning without a context)
    uint64_t plan_epoch;
    int any_tail;               // some sequence of the batch has generated tokens in this layer's tail (after this call's append)
    const void* tmap;           // CUtensorMap over the arena as rows of 256 bytes, or null
    const void* tmap_u8;        // the same arena as rows of 128 bytes (8-bit row streams), or null
    int rows_f8;
    const void* arena_base;
    int keep_num, keep_den;
    int packed_lists;
    int tok_rule;
    int32_t* tail_len;      // [L][max_batch]
    float* partials;        // [batch][Hq][kMaxSplits][d+4]: max, sum, 2 pad, d accumulators
    int32_t* status;
};
cudaError_t launch_decode(const DecodeArgs& a, int dtype, cudaStream_t st);
// Encodes a 2-D tensor map over the arena viewed as [rows][128] bf16 (256-byte rows), 64x64 boxes, 128-byte swizzle.
bool make_arena_tensor_map(void* arena, size_t arena_bytes, void* tmap_out);
// Same view ([rows][128] bf16, 64-channel x box_rows boxes, 128-byte swizzle) over any 256-byte aligned region.
bool make_rows_tensor_map(void* base, size_t bytes, int box_rows, void* tmap_out);
// ---- 8-bit row streams (rows_fp8.cu) ----
// One stored tensor: codes[t][c] = e4m3(src[t*stride_t + c] / scale[c]), scale[c] = max_t |src| / 448 (1 if zero); src bf16,
// d = 128; scale points at a 1 KiB slot whose second half holds the channel maxima while the job runs.
struct QuantJob {
    const void* src;
    int64_t stride_t;
    int32_t T, pad_;
    uint8_t* codes;
    float* scale;
};
// One residual list of a unit whose rows are 8-bit: value -> f16(value / scale[channel]), position permuted inside its
// 16-channel group to the order the kernel's converted fragments use (K and V differ).
// (rows = 1: dst == src are n densely packed 128-channel bf16 rows of the token rule, converted in place.)
struct RepackJob {
    uint32_t* dst;
    const uint32_t* src;
    int64_t n;
    const float* scale;
    int32_t is_v, rows;
};
// One copy of a commit or a fold: dst[0, bytes) = consecutive rows of row_bytes taken every src_pitch bytes from src
// (row_bytes == src_pitch: a plain copy; src null: zeros; add != 0: a plain copy of 32-bit words with `add` added).
// row_bytes and src_pitch multiples of 16, strided sources and destinations 16-byte aligned, bytes a multiple of 4 (of 2
// for plain copies).  All copies of a step run as one launch per size class over a job table.
struct CopyJob {
    const char* src;
    char* dst;
    int64_t bytes;
    int64_t src_pitch;
    int32_t row_bytes, add;
};
// Token rule: the selected tokens' high-frequency rows of one unit-tensor, formed from the caller's rows of the block's layers.
struct TokenGatherJob {
    const void* x[4];   // layer rows of the head (element (t, c) at t*stride_t + c); two for a pair
    void* dst[4];       // one stored tensor for a pair, four for a block of four
    const int32_t* list;
    int64_t stride_t, k_tok;
    int32_t twice, pad_;
};
cudaError_t launch_token_gather_jobs(const TokenGatherJob* jobs_dev, int njobs, int64_t k_tok, int d, int B, int dtype, cudaStream_t st);
cudaError_t plan_decode_host(const DecodeArgs& a, int n_ctas, const int* max_clusters, uint32_t* start_out, int32_t* ncta_out, int32_t* parts_out,
                             int32_t* cluster_out);
cudaError_t launch_copy_jobs(const CopyJob* jobs_dev, int njobs, int64_t bytes_max, cudaStream_t st);
cudaError_t launch_quantise_jobs(const QuantJob* jobs_dev, int njobs, int T_max, cudaStream_t st);
cudaError_t launch_repack_jobs(const RepackJob* jobs_dev, int njobs, int64_t n_max, cudaStream_t st);
bool make_arena_tensor_map_u8(void* arena, size_t arena_bytes, void* tmap_out);


// ---- token-granular residual (token_rule.cu) ----
struct TokenArgs {
    int B;  // layers per depth block: 2 (one Z1 operand, both layers' queries) or 4 (one deviation operand per layer)
    int unit_begin, unit_count;
    int T, Tmax, Hq, Hkv, G, W, ntiles_max;
    int64_t k_tok, ktok_cap, unit_stride;
    const void* z1;                    // [unit][1 or 4][unit_stride] high-frequency rows of K
    const void* const* q_layers_dev;
    const int32_t* pos;
    const int32_t* pos_host;
    uint32_t* score;                   // [unit][Tmax] float bits (non-negative)
    float* err;                        // [unit][nslots][Tmax] sum of squared products per token
    int nslots;                        // items a token's sum is spread over: layers x 256-row blocks, or 1 (float32 kernel)
    double* part;                      // [NU][nptiles_max][2]: slot 0 gets the unit's error sums (shared, residual)
    int nptiles_max;
    int pos_last;                      // the last probe position
    int32_t* list;                     // [unit][ktok_cap]
    int32_t* off;                      // [unit][ntiles_max + 1]
    const void* tmap_z1_128;
    int32_t* status;
};
// TokenArgs::nslots of a context for W probe queries
inline int token_err_slots(int B, int G, bool tensor_core, int W) { return tensor_core ? B * ((G * W + 255) / 256) : 1; }
// tensor_core: bf16 / head_dim 128 contexts (tcgen05 score kernel); otherwise the float32 score kernel
cudaError_t launch_token_select(const TokenArgs& a, int dtype, int d, bool tensor_core, cudaStream_t st);

// Function attributes (the opt-in to large dynamic shared memory) and the SM count belong to a device, not to the
// process: every launcher keeps one of these and runs its set-up the first time it meets the current device.
struct PerDevice {
    static constexpr int kMaxDevices = 64;
    std::mutex mu;
    bool done[kMaxDevices] = {};
    int sms[kMaxDevices] = {};
    // init() -> cudaError_t runs once per device (under the lock); *sm_count (optional) receives the device's SM count.
    template <typename F>
    cudaError_t ensure(F&& init, int* sm_count = nullptr) {
        int dev = -1;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(mu);
        if (!done[dev]) {
            e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = init();
            if (e != cudaSuccess) return e;
            done[dev] = true;
        }
        if (sm_count) *sm_count = sms[dev];
        return cudaSuccess;
    }
};
// The bookkeeping of PerDevice::ensure without a device (host-side test hook): how many of the `n` device ids in `devs`
// would run their set-up, in order, on a fresh table.
int per_device_first_visits(const int* devs, int n);

void count_launch(int n);
void count_kernel(int id);  // id: fdkv_kernel_id
// Remembers a failed CUDA runtime call for fdkv_last_cuda_error() and returns FDKV_ERR_CUDA.
fdkv_status record_cuda_error(cudaError_t e);

}  // namespace fdkv
