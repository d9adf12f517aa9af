// Decode attention over the packed cache for bf16 storage, head_dim 128 (the paragraph after Eq. 3: shared
// coefficients broadcast to both layers of the pair, residual coefficients added only where indexed, the full
// cache never materialised).
//
// One persistent CTA of eight warps per SM.  128-token (8-bit rows: 256-token) K and V boxes of the packed cache stream through a ring of
// shared-memory stages with TMA (128-byte swizzle, mbarrier completion).  The CTA's tile sequence sits in a small
// segment table in shared memory; whichever warp finishes a tile last re-arms its stage with the tile three ahead,
// so no warp is a dedicated producer.  Each warp owns 16 tokens of a stage and a private online-softmax state:
//   S = K q^T        mma.sync m16n8k16, tokens on M (ldmatrix of the swizzled K box), the G query heads on N;
//   P = exp2(S - max) per column; for G <= 4 columns 4-7 repeat the heads and carry the bf16 rounding remainder of
//                    P, so P acts with ~16 bits; movmatrix turns the accumulator layout into the next B operand;
//   O^T += V^T P^T   mma.sync, channels on M (ldmatrix.trans of the V box).
// (Heads on M, as in a prefill kernel, would use 4 of 16 rows and twice the instructions: mma.sync runs at a quarter
// of the tcgen05 rate on this part and was the limiter in that form.)
// Residual units: the warp scatters its slice's kept Z1 entries into a private zeroed 16x128 bf16 scratch tile
// and runs the same two products on it with the layer's sign, so the correction is exact in float32.  (Adding the
// entries into the landed rows in place, rounded to bf16, was faster to write but quadrupled the output error.)
// The list ranges are loaded one tile per lane 32-64 tiles ahead and handed out by shuffle; the lists themselves
// are pulled into L2 three tiles ahead and into registers one tile ahead.
// Work is a flat list of (unit, tile) pairs cut into one contiguous range per CTA (cost-weighted), so a CTA may
// finish one unit and start the next; each (CTA, unit) segment writes one split-K partial and a second small kernel
// (decode_combine_kernel) joins a head's parts.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "fdkv_internal.h"
#include "mbar_wait.cuh"

namespace fdkv {

namespace {

constexpr int kTT = 128;         // tokens per stage
constexpr int kTT8 = 256;        // tokens per stage of 8-bit rows: the same bytes
// Stages: three; two in clusters, whose blocks have few tiles and need room for their peers' parts, and with 8-bit rows, whose
// warps hold two residual tiles.
constexpr int stages_of(bool f8, bool cl) { return f8 || cl ? 2 : 3; }
constexpr int kCW = kTT / 16;    // warps, 16 tokens of a stage each
constexpr int kThreads = kCW * 32;  // 256 threads: two warps per scheduler, so up to 255 registers per thread
constexpr int kHalfBytes = kTT * 128;        // one 64-channel box of 128 tokens
constexpr int kStageBytes = 4 * kHalfBytes;  // K ch 0-63, K ch 64-127, V ch 0-63, V ch 64-127
constexpr int kScratchTile = 4096;           // 16 tokens x 128 channels bf16: the residual of one slice
// per warp (also its O tile at merge): two of them for the two slices of 8-bit rows, and in clusters for K and V
__host__ __device__ constexpr int scratch_of(bool f8, bool cl) { return f8 || cl ? 2 * kScratchTile : kScratchTile; }
constexpr int kHeaderBytes = 2048;
constexpr int kMaxSeg = 24;  // (unit, range) segments one CTA can walk: at most units / CTAs + 2
constexpr int kJointBytes = 8 * 128 * 4 + 2 * 8 * 8 * 4;  // a cluster's parts of this block's outputs: [blocks][share], then maxima and sums [blocks][8]
constexpr int smem_of(bool f8, bool cl) {
    return kHeaderBytes + stages_of(f8, cl) * kStageBytes + kCW * scratch_of(f8, cl) + (cl ? kJointBytes : 0);
}
constexpr int kMaxCtas = kMaxSplits;
constexpr int kMaxUnits = kFastMaxUnits;
constexpr int kMaxCluster = 8;  // thread blocks of a cluster (the largest portable size)
constexpr int kPartStride = 128 + 4;  // floats per split-K part: max, sum, 2 pad, 128 accumulators (16-byte aligned)
static_assert(kTT == kRowPad, "row blocks are padded to whole stages");
static_assert(smem_of(false, false) <= 227 * 1024 && smem_of(true, true) <= 227 * 1024, "shared memory budget");
static_assert(kTT8 * 128 * 2 == kStageBytes, "a stage holds as many bytes in either row format");

// (The host copies a kernel's parameters at every launch: up to kFewSeqs sequences travel in a short list.  6.4 KiB of parameters took
// 0.7 us longer to issue than 1.5 KiB.)
constexpr int kFewSeqs = 64;
template <int NB>
struct TailLens {
    int32_t n[NB];  // generated tokens in this layer's tail per sequence, this call's append included (host mirror)
};
static_assert(kMaxSplits < 256 && kMaxSplits % 32 == 0, "part counts are bytes; the combine holds one part per lane and round");

// header offsets
constexpr int kOffFull = 0, kOffJoint = 64, kOffAbort = 128, kOffM = 256, kOffL = 512, kOffSeg = 1024, kOffSegInfo = 1920,
              kOffCnt = 1936;
// one (unit, tile range) segment of a CTA: arena rows of its K / V boxes and tail, first tile, prefill tiles, first
// index in the CTA's tile sequence, and the sequence / head whose tail it also streams (or -1)
struct Seg {
    int krow, vrow, tkrow, tvrow;
    int tb, rows16, npre;  // first token of the range, its tokens rounded up to 16, its 128-token tiles (the last may be partial)
    int it0, tail_u;       // first tile in the CTA's sequence; the unit whose tail follows the range, or -1
};
static_assert(kMaxSeg * sizeof(Seg) <= 896, "segment table fits its header slot");

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t movmatrix_t(uint32_t a) {  // transpose an 8 x 8 matrix of 16-bit elements held by the warp
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the two e4m3 bytes in the low half of x -> two f16 values (exact).  (An integer form - byte permute, shift, mask, with a
// factor 2^-8 folded into the scales - was measured: 15 % slower alone, 9 % slower when sharing the work half and half.)
__device__ __forceinline__ uint32_t cvt_e4m3x2(uint32_t x) {
    uint32_t d;
    asm("{\n\t.reg .b16 t;\n\tcvt.u16.u32 t, %1;\n\tcvt.rn.f16x2.e4m3x2 %0, t;\n\t}" : "=r"(d) : "r"(x));
    return d;
}
__device__ __forceinline__ uint32_t prmt1(uint32_t a, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %1, %2;" : "=r"(d) : "r"(a), "r"(sel));
    return d;
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t peer_smem(uint32_t addr, int rank) {  // the same shared-memory address in another block of the cluster
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// two floats into a peer's shared memory; its barrier counts the bytes when they have landed
__device__ __forceinline__ void st_peer2(uint32_t addr, float x, float y, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(x), "f"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_shared_u16(uint32_t addr, uint16_t v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(v) : "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void st_shared_zero16(uint32_t addr) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(addr), "r"(0u) : "memory");
}

// byte offset of (row, channel chunk of 8) inside a [rows][64 ch] box with the 128-byte swizzle
__device__ __forceinline__ uint32_t swz(int row, int chunk8) { return (uint32_t)(row * 128 + (((chunk8 & 7) ^ (row & 7)) << 4)); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
}


// F8: the packed rows are e4m3 codes (one 128-byte row per token, per-channel float32 scales): the codes are converted
// to f16 in registers after ldmatrix, both products run as f16 mma with the K scales folded into q and the V scales
// applied to the output; the residual scratch tile then holds f16 values relative to the scales, in the converted
// fragments' channel order (the commit step writes the lists that way).  The generated-token tails stay bf16: when a
// segment reaches them the warp stashes the softmax state of its 8-bit tiles, runs the tails with the plain bf16 code
// on a fresh state and joins the two at the merge.
// (at most 232 registers: two warps of this kernel on a quarter of an SM leave 1 536 of its 16 384, one warp of
// decode_combine_kernel with at most 48)
// CL: every unit's thread blocks form a cluster (its dimension is the unit's number of blocks) and join their states through
// distributed shared memory, so that a call is one kernel: for short contexts, whose cost is the chain of hand-overs.
// NB: room for the tail lengths in the parameters.
// SPLIT: at most four query heads per KV head.
template <bool F8, bool CL, int NB, bool SPLIT>
__global__ void __maxnreg__(232)
decode_fast_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap tmap8, DecodeArgs a, FastSched sch,
                   TailLens<NB> tl) {
    constexpr int kStages = CL || F8 ? 2 : 3, kScratchBytes = scratch_of(F8, CL);
    // Clusters: the entries of K and of V have a tile each, filled before the tile is worked on (of the first one before the dependency
    // wait), so that neither their stores nor the clearing between lie in the chain from q to the outputs (1 024 tokens and a tail 7.3 -> 6.9 us).
    constexpr bool DUAL = CL && !F8;
    constexpr int TT = F8 ? kTT8 : kTT;   // tokens of a packed tile
    constexpr int SW = TT / 16 / kCW;     // 16-token slices of it per warp
    // Residual entries prefetched per lane and list (the rest are loaded when used).  8-bit rows, two slices per warp, us a layer of 32k at
    // keep 1/32, 1/16 and 1/8: eight 21.2, 21.5 and 27.3, twelve 21.6, 21.8 and 25.0.
    constexpr int kPF = F8 ? 12 : 8;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t smem0 = smem_u32(smem_raw);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem_raw + kOffAbort);
    if (smem0 & 1023u) {  // the swizzled boxes need 1024-byte alignment; report instead of computing garbage
        if (threadIdx.x == 0) atomicMax(a.status, (int32_t)kFlagCountMismatch);
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Let the next kernel in the stream start its own prologue as soon as SMs free up (programmatic dependent
    // launch); everything this kernel reads before its own griddepcontrol.wait is static since commit.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(smem0 + kOffFull + 8 * s, 1);
        }
        if constexpr (CL) {  // counts the bytes of every block's part of this block's share: its channels, a maximum and a sum per head
            uint32_t rank, nb;
            asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
            asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nb));
            const uint32_t share = (uint32_t)a.G * 128 / nb, heads = ((rank + 1) * share - 1) / 128 - rank * share / 128 + 1;
            mbar_init(smem0 + kOffJoint, 1);
            mbar_expect_tx(smem0 + kOffJoint, nb * (share * 4 + heads * 8));
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if constexpr (CL) {  // awaited before the first write to a peer
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }

    const int cta = blockIdx.x;
    const uint32_t s0 = sch.start[cta], s1 = sch.start[cta + 1];
    const int u_first = (int)(s0 >> 20), t_first = (int)(s0 & 0xFFFFFu);
    const int u_last = (int)(s1 >> 20), t_last = (int)(s1 & 0xFFFFFu);
    const uint64_t arena = reinterpret_cast<uint64_t>(a.arena_base);
    const uint32_t stage0 = smem0 + kHeaderBytes;
    const bool is_producer = threadIdx.x == 0;
    // The second layer of a pair walks every range backwards: it starts on the Z0 rows the first layer read last,
    // which are the ones most likely still in L2 (both layers of a shared / residual unit stream the same Z0).
    // (Measured: 1.4 % per step; L2 eviction hints on the TMA loads did not add to it.)
    const bool rev = (a.layer & 1) != 0;

    // ================= the CTA's tile sequence: a small segment table in shared memory =================
    // Tile `it` of the CTA (all segments, prefill tiles then tail tiles of each) always lands in stage it % kStages.
    // Whichever warp is the last to finish a tile refills its stage with tile it + kStages at once (a counter per
    // stage, no waiting producer), so copies are issued the moment a stage is free.
    Seg* const segs = reinterpret_cast<Seg*>(smem_raw + kOffSeg);
    int* const seg_info = reinterpret_cast<int*>(smem_raw + kOffSegInfo);  // [0] segments, [1] tiles in total
    int* const stage_cnt = reinterpret_cast<int*>(smem_raw + kOffCnt);
    auto issue_rows = [&](int s, int kr, int vr, bool f8_box) {  // s = the tile's stage (its index in the CTA's sequence mod kStages)
        const uint32_t full = smem0 + kOffFull + 8 * s;
        const uint32_t dst = stage0 + s * kStageBytes;
        if (F8 && f8_box) {  // one 256-token x 128-byte box per tensor
            mbar_expect_tx(full, kStageBytes);
            tma_load_2d(dst, &tmap8, 0, kr, full);
            tma_load_2d(dst + 2 * kHalfBytes, &tmap8, 0, vr, full);
        } else {
            mbar_expect_tx(full, kStageBytes);
            tma_load_2d(dst, &tmap, 0, kr, full);
            tma_load_2d(dst + kHalfBytes, &tmap, 64, kr, full);
            tma_load_2d(dst + 2 * kHalfBytes, &tmap, 0, vr, full);
            tma_load_2d(dst + 3 * kHalfBytes, &tmap, 64, vr, full);
        }
    };
    auto issue_tile = [&](int it) {
        int si = 0;
        while (si + 1 < seg_info[0] && it >= segs[si + 1].it0) ++si;
        const Seg g = segs[si];
        const int j = it - g.it0;
        // ranges start on any 16-token slice and their tiles count from there; the box of the partial tile that ends a
        // range is moved back over rows the CTA has read already (masked when used), so that no copy passes the range's end
        const int tok = max(0, g.tb + min((rev ? g.npre - 1 - j : j) * TT, g.rows16 - TT));
        const int kr = j < g.npre ? g.krow + tok : g.tkrow + (j - g.npre) * kTT;
        const int vr = j < g.npre ? g.vrow + tok : g.tvrow + (j - g.npre) * kTT;
        issue_rows(it % kStages, kr, vr, j < g.npre);
    };
    int prologue_issued = 0;
    if (is_producer) {
        // static part (packed cache, fixed since commit; tail lengths are the host's): may run before the dependency wait
        int n = 0, it0 = 0;
        for (int u = u_first; u <= u_last && u < sch.units; ++u) {
            const int b = u / a.Hkv, h = u % a.Hkv;
            const UnitDesc* ud = a.desc + ((int64_t)b * a.L + a.layer) * a.Hkv + h;
            const int nsl = (ud->T + kResTile - 1) / kResTile;
            const int sb = u == u_first ? t_first : 0;
            const int se = u == u_last ? t_last : nsl;
            if (se <= sb) continue;
            if (n == kMaxSeg) { atomicMax(a.status, (int32_t)kFlagCountMismatch); break; }  // cannot happen: see the launcher
            Seg g;
            g.krow = (int)((reinterpret_cast<uint64_t>(ud->k_rows) - arena) >> (F8 ? 7 : 8));  // rows of 128 or 256 bytes
            g.vrow = (int)((reinterpret_cast<uint64_t>(ud->v_rows) - arena) >> (F8 ? 7 : 8));
            g.tkrow = g.tvrow = 0;
            g.tb = sb * kResTile;
            g.rows16 = (min(se, nsl) - sb) * kResTile;
            g.npre = (g.rows16 + TT - 1) / TT;
            g.it0 = it0;
            g.tail_u = se == nsl ? u : -1;  // this CTA also streams the unit's tail
            it0 += g.npre;
            if (sch.any_tail && g.tail_u >= 0) {
                const int64_t o = (((int64_t)a.layer * a.max_batch + b) * a.Hkv + h) * a.tail_rows;
                g.tkrow = (int)(((reinterpret_cast<uint64_t>(a.tail_k) - arena) >> 8) + o);
                g.tvrow = (int)(((reinterpret_cast<uint64_t>(a.tail_v) - arena) >> 8) + o);
                it0 += (min(tl.n[b], a.max_tail) + kTT - 1) / kTT;
            }
            segs[n++] = g;
        }
        seg_info[0] = n;
        seg_info[1] = it0;
        for (int s = 0; s < kStages; ++s) stage_cnt[s] = 0;
        // fill the stages up to the first tile of a tail, whose rows may still be written by the kernels ahead; all but one of them (not in
        // clusters): with all, the copies of 148 blocks keep the memory busy while the kernels ahead join their parts, whose few loads wait
        // for them (us a call, 32k: all three stages 26.2, two 25.8, one 26.1; 8-bit rows, two stages: 21.3 and 20.7 with one)
        if (n > 0)
            for (; prologue_issued < (CL ? kStages : kStages - 1) && prologue_issued < segs[0].npre; ++prologue_issued)
                issue_tile(prologue_issued);
    }
    // per-warp scratch starts zeroed
    for (int i = threadIdx.x; i < kCW * kScratchBytes / 16; i += kThreads)
        st_shared_zero16(smem0 + kHeaderBytes + kStages * kStageBytes + i * 16);
    __syncthreads();  // barriers initialised, table built (still inside the previous kernel's shadow)
    // Everything that may depend on the kernels launched before this one (q, appended tail rows, partial slots) comes
    // behind this: called by every thread of the block in its first segment, after that segment's static reads.
    bool waited = false;
    auto dependency_wait = [&]() {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        waited = true;
        if (is_producer)
            for (int it = prologue_issued; it < kStages && it < seg_info[1]; ++it) issue_tile(it);
    };

    // ================= compute: every warp takes 16 tokens of every stage =================
    {
        const int gid = lane >> 2, tig = lane & 3;  // mma fragment coordinates: head row, column pair
        const int r0 = warp * 16;
        const uint32_t scratch = smem0 + kHeaderBytes + kStages * kStageBytes + warp * kScratchBytes;
        float* const scratch_f = reinterpret_cast<float*>(smem_raw + kHeaderBytes + kStages * kStageBytes + warp * kScratchBytes);
        float* const sm_m = reinterpret_cast<float*>(smem_raw + kOffM);
        float* const sm_l = reinterpret_cast<float*>(smem_raw + kOffL);
        const float kLog2e = 1.4426950408889634f;
        const float kLazyMax = 8.f;  // (log2 units) the running maximum is only moved when a score passes it by more than this
        const float inv_sqrt_d = 0.08838834764831845f;  // 1/sqrt(128)

        int it = 0;
        for (int u = u_first; u <= u_last && u < sch.units; ++u) {
            const int b = u / a.Hkv, h = u % a.Hkv;
            const UnitDesc ud = a.desc[((int64_t)b * a.L + a.layer) * a.Hkv + h];
            const int T = ud.T;
            const int nres = (T + kResTile - 1) / kResTile;
            const int sb = u == u_first ? t_first : 0;
            const int se = u == u_last ? t_last : nres;
            if (se <= sb) continue;
            // this CTA's tokens of the unit: [tok_b, tok_e), cut on 16-token slices; tiles count from tok_b
            const int tok_b = sb * kResTile, tok_e = min(se * kResTile, T), rows16 = (se - sb) * kResTile;
            int ntail = 0, n_tail_rows = 0;
            if (sch.any_tail && se == nres) {
                n_tail_rows = min(tl.n[b], a.max_tail);
                ntail = (n_tail_rows + kTT - 1) / kTT;
            }
            // The row that this call appends is the last of the tail.  Its copy from the tail is stale: the warp that owns it takes
            // it from the caller, puts it into the landed tile and stores it to the tail for later calls, so that the tail's
            // copy is requested right behind the dependency wait and no store has to become visible to it.
            const bool append = ntail > 0 && a.k_new && warp == ((n_tail_rows - 1) & (kTT - 1)) >> 4;
            const int npre = (rows16 + TT - 1) / TT, nseg = npre + ntail;
            const bool coef = ud.mode != FDKV_MODE_EXACT, resid = ud.mode == FDKV_MODE_RESIDUAL;
            const uint32_t sgn = ud.sign < 0.f ? 0x80008000u : 0u;

            // O^T[channel][column]: eight 16-channel m-tiles; this thread holds columns 2 tig, 2 tig + 1
            float oacc[8][4];
#pragma unroll
            for (int j = 0; j < 8; ++j) oacc[j][0] = oacc[j][1] = oacc[j][2] = oacc[j][3] = 0.f;
            float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};  // per held column; l is this thread's share
            float m_st[2] = {-INFINITY, -INFINITY}, l_st[2] = {0.f, 0.f};     // 8-bit rows: the state stashed before the bf16 tails
            bool stashed = false;
            const int slot = u == u_first ? sch.slot[cta] : 0;

            // ---- residual lists (packed entries): ranges two tiles ahead, entries one tile ahead ----
            const uint32_t* k_ent = reinterpret_cast<const uint32_t*>(ud.k_idx);
            const uint32_t* v_ent = reinterpret_cast<const uint32_t*>(ud.v_idx);
            constexpr int NR = 2 * (SW + 1);
            // {bounds of the warp's slices in the K list, the same in the V list}: this tile, next, the one after
            int cr[NR] = {}, nr[NR] = {}, fr[NR] = {};
            uint32_t pke[kPF], pve[kPF];
            // token-granular residual: one ascending token list (k_idx) with per-slice counts (k_off) for K and V,
            // and the selected tokens' Z1 rows packed densely (k_val / v_val, 256 bytes each)
            const bool tokmode = resid && ud.res_kind == 1;
            const uint4* t_krows = reinterpret_cast<const uint4*>(ud.k_val);
            const uint4* t_vrows = reinterpret_cast<const uint4*>(ud.v_val);
            int ptk[2] = {0, 0}, ptv[2] = {0, 0};
            // List ranges of this warp's slices, one tile per lane: lane l of a batch holds tile rb + l of the segment, loaded
            // 32 to 64 tiles before use and handed out by shuffle.
            int rb = 0, rk[NR] = {}, rk_n[NR] = {};
            auto load_batch = [&](int jb, int (&k)[NR]) {
                const int jj = jb + lane;
#pragma unroll
                for (int i = 0; i < NR; ++i) k[i] = 0;
                if (resid && jj < npre) {
                    // the tile's slices not yet read: [first, se); the box may start before them (see issue_tile)
                    const int first = sb + (rev ? npre - 1 - jj : jj) * (TT / kResTile);
                    const int o = max(0, min(first, se - TT / kResTile)) + SW * warp;
#pragma unroll
                    for (int i = 0; i <= SW; ++i) {
                        const int oi = min(max(o + i, first), se);
                        k[i] = ud.k_off[oi];
                        k[SW + 1 + i] = tokmode ? k[i] : ud.v_off[oi];
                    }
                }
            };
            auto get_ranges = [&](int j, int (&r)[NR]) {  // rb <= j < rb + 64
                const bool nx = j - rb >= 32;
                const int src = (j - rb) & 31;
#pragma unroll
                for (int i = 0; i < NR; ++i) r[i] = __shfl_sync(0xFFFFFFFFu, nx ? rk_n[i] : rk[i], src);
            };
            // pull a tile's list slices (or selected token rows) into L2 a few tiles ahead: lanes 0-15 the K side,
            // lanes 16-31 the V side, one 128-byte line each
            auto l2_prefetch = [&](const int (&r)[NR]) {
                const int hl = lane & 15;
                const void* ptr = nullptr;
                if (tokmode) {
                    const int j = r[0] + (hl >> 1);
                    if (j < r[SW]) ptr = reinterpret_cast<const char*>(lane < 16 ? t_krows : t_vrows) + (int64_t)j * 256 + (hl & 1) * 128;
                } else {
                    const int e0 = lane < 16 ? r[0] : r[SW + 1], e1 = lane < 16 ? r[SW] : r[2 * SW + 1];
                    const int e = (e0 & ~31) + 32 * hl;
                    if (e < e1) ptr = (lane < 16 ? k_ent : v_ent) + e;
                }
                if (ptr) asm volatile("prefetch.global.L2 [%0];" ::"l"(ptr));
            };
            auto prefetch = [&](const uint32_t* ent, int e0, int e1, uint32_t (&pe)[kPF]) {
#pragma unroll
                for (int i = 0; i < kPF; ++i) {
                    if (i == 8 && e0 + 256 >= e1) break;
                    const int e = e0 + lane + 32 * i;
                    if (e < e1) pe[i] = ent[e];
                }
            };
            // scatter one list slice into the scratch tile: each entry carries its own shared-memory offset
            // (with two slices per warp, entries from `mid` on belong to the second)
            auto scatter = [&](const uint32_t* ent, int e0, int mid, int e1, const uint32_t (&pe)[kPF], uint32_t to) {
#pragma unroll
                for (int i = 0; i < kPF; ++i) {
                    if (i == 8 && e0 + 256 >= e1) break;
                    const int e = e0 + lane + 32 * i;
                    if (e < e1) st_shared_u16(to + ((pe[i] >> 16) << 1) + (SW == 2 && e >= mid ? kScratchTile : 0), (uint16_t)(pe[i] & 0xFFFFu));
                }
                for (int eb = e0 + 32 * kPF; eb < e1; eb += 128) {  // dense slices: direct loads, four in flight
                    uint32_t w[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) w[i] = eb + lane + 32 * i < e1 ? ent[eb + lane + 32 * i] : 0u;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int e = eb + lane + 32 * i;
                        if (e < e1) st_shared_u16(to + ((w[i] >> 16) << 1) + (SW == 2 && e >= mid ? kScratchTile : 0), (uint16_t)(w[i] & 0xFFFFu));
                    }
                }
            };
            // token rows: two tokens per round (half a warp each, 16 bytes per lane), two rounds in registers
            auto prefetch_tok = [&](const uint4* rows, int e0, int e1, uint32_t (&pe)[kPF], int (&pt)[2]) {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int j = e0 + 2 * r + (lane >> 4);
                    if (j < e1) {
                        const uint4 v = rows[(int64_t)j * 16 + (lane & 15)];
                        pe[4 * r] = v.x; pe[4 * r + 1] = v.y; pe[4 * r + 2] = v.z; pe[4 * r + 3] = v.w;
                        pt[r] = k_ent[j];  // the token list sits where the packed layout keeps the K entries
                    }
                }
            };
            auto scatter_tok = [&](const uint4* rows, int e0, int mid, int e1, const uint32_t (&pe)[kPF], const int (&pt)[2], uint32_t to) {
                const int chunk = lane & 15;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int j = e0 + 2 * r + (lane >> 4);
                    if (j < e1) {
                        const int row = pt[r] & 15;
                        st_shared_v4(to + (SW == 2 && j >= mid ? kScratchTile : 0) + (chunk >> 3) * 2048 + swz(row, chunk), pe[4 * r], pe[4 * r + 1], pe[4 * r + 2], pe[4 * r + 3]);
                    }
                }
                for (int j = e0 + 4 + (lane >> 4); j < e1; j += 2) {  // more than four selected tokens in the slice
                    const int row = (int)k_ent[j] & 15;
                    const uint4 v = rows[(int64_t)j * 16 + chunk];
                    st_shared_v4(to + (SW == 2 && j >= mid ? kScratchTile : 0) + (chunk >> 3) * 2048 + swz(row, chunk), v.x, v.y, v.z, v.w);
                }
            };
            auto zero_scratch = [&]() {
#pragma unroll
                for (int i = 0; i < kScratchBytes / 16 / 32; ++i) st_shared_zero16(scratch + (lane + 32 * i) * 16);
            };
            if (resid) {
                load_batch(0, rk);
                load_batch(32, rk_n);
                get_ranges(0, cr);
                get_ranges(1, nr);
                get_ranges(2, fr);
                l2_prefetch(nr);
                l2_prefetch(fr);
                if (tokmode) {
                    prefetch_tok(t_krows, cr[0], cr[SW], pke, ptk);
                    prefetch_tok(t_vrows, cr[SW + 1], cr[2 * SW + 1], pve, ptv);
                } else {
                    prefetch(k_ent, cr[0], cr[SW], pke);
                    prefetch(v_ent, cr[SW + 1], cr[2 * SW + 1], pve);
                }
            }
            // (DUAL) both entry tiles of the tile whose ranges are in cr, then the entries of the next on their way
            auto fill_both = [&]() {
                if (tokmode) {
                    scatter_tok(t_krows, cr[0], cr[1], cr[1], pke, ptk, scratch);
                    scatter_tok(t_vrows, cr[2], cr[3], cr[3], pve, ptv, scratch + kScratchTile);
                    prefetch_tok(t_krows, nr[0], nr[1], pke, ptk);
                    prefetch_tok(t_vrows, nr[2], nr[3], pve, ptv);
                } else {
                    scatter(k_ent, cr[0], cr[1], cr[1], pke, scratch);
                    scatter(v_ent, cr[2], cr[3], cr[3], pve, scratch + kScratchTile);
                    prefetch(k_ent, nr[0], nr[1], pke);
                    prefetch(v_ent, nr[2], nr[3], pve);
                }
                __syncwarp();
            };
            if constexpr (DUAL)
                if (resid) fill_both();

            if (!waited) dependency_wait();
            uint4 appended = make_uint4(0u, 0u, 0u, 0u);  // (clusters: requested with q, or the block with the tail is another round trip behind)
            if constexpr (CL)
                if (append) appended = reinterpret_cast<const uint4*>(lane < 16 ? a.k_new : a.v_new)[((int64_t)b * a.Hkv + h) * 16 + (lane & 15)];
            // q fragments: B operand columns = the G query heads of this KV head.  With G <= 4 columns 4-7 repeat
            // them: in the second product those columns carry the bf16 rounding remainder of P, so P acts in ~16 bits.
            // (More heads fill the columns: their remainder is a second B operand with the same V fragments.)
            const bool split = SPLIT && a.G <= 4;  // (a constant cost the 32k workloads 0.5 to 0.9 %)
            const int qcol = split ? (gid & 3) : gid;
            uint32_t qb[8][2];
            auto load_q = [&](bool f8) {
                const __nv_bfloat16* qh = reinterpret_cast<const __nv_bfloat16*>(a.q) + ((int64_t)b * a.Hq + h * a.G + qcol) * 128;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    if (F8 && f8) {
                        // a converted register holds channels 4 tig .. 4 tig + 3 of the 16-channel step: its low pair is the
                        // first k-slot pair, its high pair the second; q carries the K scales, as f16
                        const int c0 = 16 * kk + 4 * tig;
                        float qv[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) qv[i] = qcol < a.G ? __bfloat162float(qh[c0 + i]) * ud.k_scale[c0 + i] : 0.f;
                        qb[kk][0] = pack_f16(qv[0], qv[1]);
                        qb[kk][1] = pack_f16(qv[2], qv[3]);
                    } else {
                        qb[kk][0] = qcol < a.G ? *reinterpret_cast<const uint32_t*>(qh + 16 * kk + 2 * tig) : 0u;
                        qb[kk][1] = qcol < a.G ? *reinterpret_cast<const uint32_t*>(qh + 16 * kk + 8 + 2 * tig) : 0u;
                    }
                }
            };
            if constexpr (F8) {
                load_q(true);
            } else {  // (kept inline for the bf16 kernel: routing it through the lambda cost 0.5 %)
                const __nv_bfloat16* qh = reinterpret_cast<const __nv_bfloat16*>(a.q) + ((int64_t)b * a.Hq + h * a.G + qcol) * 128;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    qb[kk][0] = qcol < a.G ? *reinterpret_cast<const uint32_t*>(qh + 16 * kk + 2 * tig) : 0u;
                    qb[kk][1] = qcol < a.G ? *reinterpret_cast<const uint32_t*>(qh + 16 * kk + 8 + 2 * tig) : 0u;
                }
            }

            // A warp is done reading stage s (tile j of this segment): the last of the eight refills it.  Three tiles ahead
            // is usually still a packed tile of this segment, whose rows follow from registers; only across a segment
            // boundary (or into the tails) the segment table is walked.  The refill sits on the critical path of the ring.
            const int unit_kr = (int)((reinterpret_cast<uint64_t>(ud.k_rows) - arena) >> (F8 ? 7 : 8));
            const int unit_vr = (int)((reinterpret_cast<uint64_t>(ud.v_rows) - arena) >> (F8 ? 7 : 8));
            auto release_here = [&](int s, int j) {
                __syncwarp();  // (also between what a lane has cleared in the scratch and what the others write there next)
                if (CL && it + j + kStages >= seg_info[1]) return;  // (nothing follows in this stage)
                if (lane == 0) {
                    // (atomicInc wraps the counter back to zero at the eighth arrival; tile j + kStages reuses stage s)
                    const unsigned old = atomicInc(reinterpret_cast<unsigned*>(stage_cnt) + s, kCW - 1);
                    if (old == kCW - 1) {
                        const int jn = j + kStages;
                        if (jn < npre) {
                            const int tok = max(0, tok_b + min((rev ? npre - 1 - jn : jn) * TT, rows16 - TT));
                            issue_rows(s, unit_kr + tok, unit_vr + tok, true);
                        } else if (it + jn < seg_info[1]) {
                            issue_tile(it + jn);
                        }
                    }
                }
            };
            // O[head][channel] into the warp's float scratch: column g plus (G <= 4) its remainder column g + 4, held by the
            // lane two over: of two m-tiles such a pair of lanes adds up and stores one each.  Rows gid / gid + 8 of an m-tile are
            // channels gid and gid + 8, or (8-bit tiles) 2 gid and 2 gid + 1, whose code sums are still to be multiplied by the
            // channel's V scale.  Channels are stored xor 8 (column / 2 mod 4): the columns of a store lie in different banks.
            const int ocol = split ? 2 * (tig & 1) : 2 * tig, oswz = (split ? tig & 1 : tig) << 3;
            auto store_o = [&](bool f8_layout, bool accumulate, float f0, float f1) {
                auto put = [&](int jm, const float (&v)[4]) {
                    const int ch_a = f8_layout ? 16 * jm + 2 * gid : 16 * jm + gid, ch_b = f8_layout ? ch_a + 1 : ch_a + 8;
                    const float sa = f8_layout ? ud.v_scale[ch_a] : 1.f, sb = f8_layout ? ud.v_scale[ch_b] : 1.f;
                    float* p0 = scratch_f + ocol * 128;
                    float* p1 = p0 + 128;
                    const int a_ = ch_a ^ oswz, b_ = ch_b ^ oswz;
                    if (accumulate) {
                        p0[a_] += v[0] * sa * f0; p1[a_] += v[1] * sa * f1; p0[b_] += v[2] * sb * f0; p1[b_] += v[3] * sb * f1;
                    } else {
                        p0[a_] = v[0] * sa; p1[a_] = v[1] * sa; p0[b_] = v[2] * sb; p1[b_] = v[3] * sb;
                    }
                };
                if (split) {
#pragma unroll
                    for (int jm = 0; jm < 8; jm += 2) {
                        const bool odd = tig >= 2;
                        float v[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float other = __shfl_xor_sync(0xFFFFFFFFu, odd ? oacc[jm][i] : oacc[jm + 1][i], 2);
                            v[i] = (odd ? oacc[jm + 1][i] : oacc[jm][i]) + other;
                        }
                        put(odd ? jm + 1 : jm, v);
                    }
                } else {
#pragma unroll
                    for (int jm = 0; jm < 8; ++jm) put(jm, oacc[jm]);
                }
            };
            // (the tile bodies are textual includes: as a generic lambda one cost the bf16 kernel 6 %)
            if constexpr (F8) {
                for (int j = 0; j < npre; ++j)
#include "decode_fast_tile8.inc"
            }
            for (int j = F8 ? npre : 0; j < nseg; ++j)
#include "decode_fast_tile.inc"
            it += nseg;

            // ---- merge the eight warps' states into this segment's split-K partial ----
            {
                float lq[2] = {l_run[0], l_run[1]};
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    lq[0] += __shfl_xor_sync(0xFFFFFFFFu, lq[0], o);
                    lq[1] += __shfl_xor_sync(0xFFFFFFFFu, lq[1], o);
                }
                if (F8 && stashed) {
                    // join the stashed state of the 8-bit tiles (already in the scratch) with the tails' state
                    float f_st[2], f_tl[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float M = fmaxf(m_st[e], m_run[e]);
                        f_st[e] = m_st[e] == -INFINITY ? 0.f : ex2(m_st[e] - M);
                        f_tl[e] = m_run[e] == -INFINITY ? 0.f : ex2(m_run[e] - M);
                        lq[e] = l_st[e] * f_st[e] + lq[e] * f_tl[e];
                        m_run[e] = M;
                    }
                    // (the positions this lane wrote at the stash)
#pragma unroll
                    for (int jm = 0; jm < 8; ++jm) {
                        if (split && (jm & 1) != (tig >> 1)) continue;
                        float* p0 = scratch_f + ocol * 128 + ((16 * jm + 2 * gid) ^ oswz);
                        p0[0] *= f_st[0]; p0[1] *= f_st[0]; p0[128] *= f_st[1]; p0[129] *= f_st[1];
                    }
                    __syncwarp();
                    store_o(false, true, f_tl[0], f_tl[1]);
                } else {
                    store_o(F8, false, 1.f, 1.f);
                }
                if (gid == 0) {
#pragma unroll
                    for (int e = 0; e < 2; ++e) { sm_m[warp * 8 + 2 * tig + e] = m_run[e]; sm_l[warp * 8 + 2 * tig + e] = lq[e]; }
                }
                __syncthreads();
                uint32_t rank = 0, nb = 1, share = 1024;
                const uint32_t joint0 = smem0 + kHeaderBytes + kStages * kStageBytes + kCW * kScratchBytes;
                if constexpr (CL) {
                    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
                    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nb));
                    share = (uint32_t)a.G * 128 / nb;  // outputs of the unit that a block joins
                    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // (the peers' barriers are set up)
                }
                for (int i = threadIdx.x; i < a.G * 64; i += kThreads) {  // two channels per thread
                    const int g = i >> 6, ch = 2 * (i & 63);
                    float M = -INFINITY;
#pragma unroll
                    for (int w = 0; w < kCW; ++w) M = fmaxf(M, sm_m[w * 8 + g]);
                    float L = 0.f;
                    float2 A = make_float2(0.f, 0.f);
                    if (M != -INFINITY) {
#pragma unroll
                        for (int w = 0; w < kCW; ++w) {
                            const float f = ex2(sm_m[w * 8 + g] - M);
                            L = fmaf(sm_l[w * 8 + g], f, L);
                            const float2 o = *reinterpret_cast<const float2*>(smem_raw + kHeaderBytes + kStages * kStageBytes + w * kScratchBytes + (g * 128 + (ch ^ ((g >> 1 & 3) << 3))) * 4);
                            A.x = fmaf(o.x, f, A.x);
                            A.y = fmaf(o.y, f, A.y);
                        }
                    }
                    if constexpr (CL) {
                        // to the block that joins these channels, counted by its barrier
                        const uint32_t o = (uint32_t)(g * 128 + ch), to = (uint32_t)(((float)o + 0.5f) * sch.inv_share);
                        const uint32_t joint = peer_smem(joint0, (int)to), bar = peer_smem(smem0 + kOffJoint, (int)to), at = o - to * share;
                        st_peer2(joint + (rank * share + at) * 4, A.x, A.y, bar);
                        if (at == 0 || ch == 0) st_peer2(joint + (1024 + 2 * (rank * 8 + g)) * 4, M, L, bar);  // (a share starts inside a head or covers whole heads)
                    } else {
                        float* part = a.partials + (((int64_t)b * a.Hq + h * a.G + g) * kMaxSplits + slot) * kPartStride;
                        if (ch == 0) { part[0] = M * 0.6931471805599453f; part[1] = L; }  // the combine step works in natural-log units
                        *reinterpret_cast<float2*>(part + 4 + ch) = A;
                    }
                }
                if constexpr (CL) {
                    // All parts of this block's share.  Every block sends its parts whatever happened to its copies, so this wait ends
                    // when the slowest one is through; no block leaves before, so that nobody writes to one that has left.
                    if (!mbar_try_wait(smem0 + kOffJoint, 0)) {
                        uint32_t polls = 0;
                        while (!mbar_try_wait(smem0 + kOffJoint, 0) && ++polls < 4 * kWaitCap) {}
                        if (polls >= 4 * kWaitCap) { *abort_flag = 1; atomicMax(a.status, (int32_t)kFlagTimeout); }
                    }
                    const float* const joint = reinterpret_cast<const float*>(smem_raw + kHeaderBytes + kStages * kStageBytes + kCW * kScratchBytes);
                    for (uint32_t i = threadIdx.x; i < share; i += kThreads) {
                        const uint32_t o = rank * share + i, g = o >> 7;
                        float m[kMaxCluster], M = -INFINITY, L = 0.f, A = 0.f;
#pragma unroll
                        for (int c = 0; c < kMaxCluster; ++c) {
                            m[c] = c < (int)nb ? joint[1024 + 2 * (c * 8 + g)] : -INFINITY;
                            M = fmaxf(M, m[c]);
                        }
#pragma unroll
                        for (int c = 0; c < kMaxCluster; ++c)
                            if (c < (int)nb) {
                                const float f = m[c] == -INFINITY ? 0.f : ex2(m[c] - M);
                                L = fmaf(joint[1024 + 2 * (c * 8 + g) + 1], f, L);
                                A = fmaf(joint[c * share + i], f, A);
                            }
                        const float r = L > 0.f ? A / L : 0.f;
                        const int64_t at = ((int64_t)b * a.Hq + h * a.G) * 128 + o;
                        if (a.out_dtype == FDKV_BF16) reinterpret_cast<__nv_bfloat16*>(a.out)[at] = __float2bfloat16_rn(r);
                        else reinterpret_cast<float*>(a.out)[at] = r;
                    }
                }
                if (u < u_last && u + 1 < sch.units) {  // (another segment may follow: the scratch tiles and sums are read by now)
                    __syncthreads();
                    zero_scratch();
                    __syncthreads();
                }
            }
        }
    }
    // after a timed-out wait: give copies that may still be in flight time to land before the CTA retires
    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
}

// out = sum_s e^{m_s - M} acc_s / sum_s e^{m_s - M} l_s over a query head's split-K parts.  One warp per 32 or 128 channels of a
// head; it rides on programmatic dependent launch between two decode launches.  A block has 32 threads and few registers
// so that it becomes resident beside a decode block (which leaves 2 048 registers and 1 KiB of shared memory of an SM) and
// its start costs nothing.  Latency-bound: the maxima and sums of 32 parts are requested together, then accumulators by 20 (VEC 2) or 4.
// (Before, the last block of a unit combined behind an atomic ticket: a release, an atomic round trip and two rounds of
// loads on the critical path of every layer call, and the SM it ran on started the next call late.)
// VEC 4: a lane has four channels of every part, four parts in flight (many heads, few parts each).  VEC 2: a lane has two channels of
// every other part, so that 20 parts are in flight at once (few heads, whose 18 or 19 parts took two rounds of 16 one after the other:
// eight KV heads, us a call: 2 047 tokens 8.36 -> 8.26, 32k 26.2 -> 26.1, 32k of 8-bit rows 21.3 -> 21.2).
template <int VEC>
__global__ void __maxnreg__(48) decode_combine_kernel(const float* partials, int Hq, int Hkv, int G, PartCount pc, void* out, int out_dtype) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int WAYS = VEC == 2 ? 2 : 1, BATCH = VEC == 2 ? 10 : 4;  // lanes that share a channel; parts a lane has in flight
    const int lane = threadIdx.x, i = blockIdx.y, b = blockIdx.z;
    const int way = WAYS == 2 ? lane >> 4 : 0, ch = (blockIdx.x * (32 / WAYS) + (lane & (32 / WAYS - 1))) * VEC;
    const int n = pc.n[b * Hkv + i / G];
    const float* const pp = partials + ((int64_t)b * Hq + i) * kMaxSplits * kPartStride;
    float M = -INFINITY, L = 0.f, A[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) A[k] = 0.f;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int base = 0; base < n; base += 32) {
        float m = -INFINITY, l = 0.f;
        if (base + lane < n) {
            const float2 ml = __ldcg(reinterpret_cast<const float2*>(pp + (base + lane) * kPartStride));
            m = ml.x;
            l = ml.y;
        }
        float w = 0.f;
        for (int j0 = 0; j0 < 32 && base + j0 < n; j0 += BATCH * WAYS) {
            float v[BATCH][VEC];
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
                const int part = j0 + j * WAYS + way;
#pragma unroll
                for (int k = 0; k < VEC; ++k) v[j][k] = 0.f;
                if (part < 32 && base + part < n) {
                    const float* p = pp + (base + part) * kPartStride + 4 + ch;
                    if constexpr (VEC == 4) {
                        const float4 x = __ldcg(reinterpret_cast<const float4*>(p));
                        v[j][0] = x.x; v[j][1] = x.y; v[j][2] = x.z; v[j][3] = x.w;
                    } else {
                        const float2 x = __ldcg(reinterpret_cast<const float2*>(p));
                        v[j][0] = x.x; v[j][1] = x.y;
                    }
                }
            }
            if (j0 == 0) {
                float mx = m;
#pragma unroll
                for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
                mx = fmaxf(mx, M);
                w = m == -INFINITY ? 0.f : __expf(m - mx);
                const float f = M == -INFINITY ? 0.f : __expf(M - mx);
                float ls = l * w;
#pragma unroll
                for (int o = 16; o; o >>= 1) ls += __shfl_xor_sync(0xFFFFFFFFu, ls, o);
                L = fmaf(L, f, ls);
#pragma unroll
                for (int k = 0; k < VEC; ++k) A[k] *= f;
                M = mx;
            }
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
                const int part = j0 + j * WAYS + way;
                const float wj = __shfl_sync(0xFFFFFFFFu, w, part & 31);  // (a part that is not there has zeros)
#pragma unroll
                for (int k = 0; k < VEC; ++k) A[k] = fmaf(v[j][k], wj, A[k]);
            }
        }
    }
    if constexpr (WAYS == 2) {
#pragma unroll
        for (int k = 0; k < VEC; ++k) A[k] += __shfl_xor_sync(0xFFFFFFFFu, A[k], 16);
        if (way) return;
    }
    const int64_t o = ((int64_t)b * Hq + i) * 128 + ch;
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        const float r = L > 0.f ? A[k] / L : 0.f;
        if (out_dtype == FDKV_BF16) reinterpret_cast<__nv_bfloat16*>(out)[o + k] = __float2bfloat16_rn(r);
        else reinterpret_cast<float*>(out)[o + k] = r;
    }
}

}  // namespace

bool make_rows_tensor_map(void* base, size_t bytes, int box_rows, void* tmap_out) {
    typedef CUresult (*encode_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
        qres != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        return false;
    }
    const cuuint64_t rows = bytes / 256;
    if (rows == 0 || rows > 0x7FFFFFFFull || box_rows < 1 || box_rows > 256) return false;
    const cuuint64_t gdim[2] = {128, rows};
    const cuuint64_t gstride[1] = {256};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};  // 64 channels x box_rows tokens
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = reinterpret_cast<encode_fn>(fn)(reinterpret_cast<CUtensorMap*>(tmap_out), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base,
                                                 gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// The same region viewed as rows of 128 bytes (8-bit row streams): one 128-byte x box_rows box per copy, 128-byte swizzle.
bool make_rows_tensor_map_u8(void* base, size_t bytes, int box_rows, void* tmap_out) {
    typedef CUresult (*encode_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
        qres != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        return false;
    }
    const cuuint64_t rows = bytes / 128;
    if (rows == 0 || rows > 0x7FFFFFFFull || box_rows < 1 || box_rows > 256) return false;
    const cuuint64_t gdim[2] = {128, rows};
    const cuuint64_t gstride[1] = {128};
    const cuuint32_t box[2] = {128, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = reinterpret_cast<encode_fn>(fn)(reinterpret_cast<CUtensorMap*>(tmap_out), CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, base, gdim,
                                                 gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

bool make_arena_tensor_map_u8(void* arena, size_t arena_bytes, void* tmap_out) {
    return make_rows_tensor_map_u8(arena, arena_bytes, kTT8, tmap_out);
}
bool make_arena_tensor_map(void* arena, size_t arena_bytes, void* tmap_out) {
    return make_rows_tensor_map(arena, arena_bytes, kTT, tmap_out);
}

// Host side of a launch: the cost-weighted cut of the batch's (unit, 16-token slice) list into one range per CTA and the
// split-K part count of every unit.  Uses only the host views in `a` (lengths, modes, shape); no device access.
// max_clusters[i]: clusters of 2^i blocks that fit the device at one time (null: plan without clusters).
static cudaError_t plan_decode_schedule(const DecodeArgs& a, int units, int sm_count, const int* max_clusters, FastSched& sch, PartCount& cs) {
    // ---- cost-weighted schedule: whole CTAs per unit when there are enough CTAs, else a flat cut of the (unit, tile) list ----
    std::vector<int64_t> wp(units + 1, 0);
    // ranges are cut on 16-token slices (the granularity of the residual lists), so that the CTAs of a unit differ by
    // at most one slice; each range is streamed as 128-token tiles from its first slice, the last one partial
    std::vector<int> nt(units), ns(units), es(units), wt(units);  // 128-token tiles, 16-token slices, slices + tail, cost per tile
    int64_t total_tiles = 0;
    for (int u = 0; u < units; ++u) {
        const int T = a.host_T[u / a.Hkv];
        nt[u] = (T + kTT - 1) / kTT;
        ns[u] = (T + kResTile - 1) / kResTile;
        if (ns[u] >= (1 << 20)) return cudaErrorInvalidValue;  // cannot happen: T * 128 < 2^31
        total_tiles += nt[u];
    }
    // cost per tile: bytes in units of 512 B (the K and V boxes, plus the lists' share for residual units), residual
    // tiles scaled by the measured ratio of their compute time to a plain tile's (rc)
    // With whole CTAs per unit (latency-bound regime) a residual tile of the entry form costs a fixed part (the scratch
    // tile and the second products) plus a part per list entry: measured 2.0 plain tiles at 1024 entries per tile and
    // tensor (keep 1/16), 1.65 at 512 (keep 1/32); with 8-bit rows (a dearer plain tile) about 1.9 at either
    // density (32k, us a layer with the fixed part at 1.55, 1.65, 1.75, 1.85 and 2.0: keep 1/16 23.2, 22.7, 22.1, 22.0, 22.8, keep 1/32
    // 21.6, 21.5, 21.3, 21.5, 22.6).
    const double res_a = a.rows_f8 ? 1.75 : 1.25;
    const double res_b = a.rows_f8 ? 0.15 : 0.87;
    const int ctas = (int)std::min<int64_t>(std::min(std::min(sm_count, kMaxCtas), kMaxSplits), total_tiles);
    auto weigh = [&](double rc) {
        for (int u = 0; u < units; ++u) {
            const int T = a.host_T[u / a.Hkv];
            const int64_t k = (int64_t)T * 128 * a.keep_num / a.keep_den;
            wt[u] = 2 * kTT * 256 / 512;
            if (a.host_modes[u] == FDKV_MODE_RESIDUAL) {
                const int64_t res_bytes = a.tok_rule ? 2 * ((int64_t)T * a.keep_num / a.keep_den) * 260 : 2 * k * 4;  // rows + index, or packed entries
                if (rc == 0.0) wt[u] = (int)(wt[u] * (res_a + res_b * (double)k / nt[u] / 1024.0));
                else wt[u] = (int)((wt[u] + (res_bytes / nt[u] + 511) / 512) * rc);
                wt[u] = std::max(1, wt[u]);
            }
            // the CTA that ends a unit also streams its tail of generated tokens (whole plain tiles): counted as slices
            // of the unit's kind behind the unit's own, so that this CTA gets correspondingly fewer of those
            const int tail = a.host_tail ? std::min(a.host_tail[u / a.Hkv], a.max_tail) : 0;
            // Measured: it runs behind its siblings at equal shares (cause not found); charging it five eighths of a block's share, at
            // most eight plain tiles, on top is within 0.3 % of the best of a sweep at 2k to 128k and on a batch (against no
            // charge: 32k 26.5 -> 26.2 us a layer, 128k 84.7 -> 83.1, batch of eight 132.8 -> 130.7).
            const int64_t end_extra = std::min<int64_t>(64, 5 * total_tiles / std::max(1, ctas));  // (eighths of a plain tile)
            es[u] = ns[u] + ((tail + kTT - 1) / kTT * (kTT / kResTile) + (int)end_extra) * (2 * kTT * 256 / 512) / std::max(1, wt[u]);
            wp[u + 1] = wp[u] + (int64_t)es[u] * wt[u];  // (in eighths of the tile cost)
        }
    };
    // (measured best: 1.7 when every unit gets whole CTAs, 1.5 in the flat cut of a batch)
    weigh(a.tok_rule ? 1.7 : 0.0);
    const int ncta = ctas;
    sch.ncta = ncta;
    sch.any_tail = a.any_tail;
    sch.units = units;
    sch.cluster = 0;
    // Clusters, as many blocks per unit as fit: one kernel instead of two, where that is worth more than the blocks that are
    // left out.  Measured on a stream, us a call of bf16 rows (clusters with 0.8 KiB more of parameters, which took 0.15, 8-bit rows 0.25): clusters
    // 3.55 + 1.03 for each plain tile of the slowest block (a tail tile counts 1.2),
    // two kernels 5.7 + 1.1 for each of the average block and at least 7.75 (8.4 with tails), the two hand-overs.  Eight KV heads, clusters against
    // two kernels: 1 024 tokens 5.4 and 7.7, 2 047 6.8 and 7.8, 3 000 8.1 and 7.8, 8 191 15.5 and 11.1; with a tail 1 024 6.3 and 8.4, 1 500
    // 7.2 and 8.5, 2 047 8.0 and 8.4, 3 000 9.9 and 8.8; two KV heads 2 047 5.7 and 7.7, with a tail 6.7 and 8.4, 4 096 8.4 and 7.8.
    // 8-bit rows (4.6 + 1.05 against 5.7 + 1.15 and 7.9): 1 024 7.1 and 7.9, 2 047 8.3 and 8.1, 3 000 9.7 and 8.5; their tails make the last block
    // of the other cut later (at least 10.5): 1 024 9.3 and 10.5, 3 000 10.5 and 11.3, 4 096 12.3 and 11.1.
    // Up to five tiles per SM, the other cut also pays for rounding its shares to tiles, about what a block that ends a unit is
    // charged: that counts then (units of bf16, ragged lengths up to the given one, a third to a half residual; clusters and two
    // kernels: 128 of 459 tokens 11.9 and 14.8, 64 of 1181 9.4 and 10.8, 32 of 3267 10.7 and 11.7).  Longer ones don't (128 of 2174 36.1 and
    // 31.7, 64 of 2972 26.1 and 20.4, 144 of 3000 43.0 and 36.3), nor 8-bit rows (48 of 537 10.1 and 8.8, 32 of 2270 13.2 and 11.3, though 128 of
    // 949 20.5 and 22.4).
    if (max_clusters) {
        bool tails = false;
        for (int b = 0; b < a.batch && a.host_tail; ++b) tails = tails || a.host_tail[b] > 0;
        const double gain = tails ? 2.7 : a.rows_f8 ? 1.0 : 2.1, least_other = a.rows_f8 ? 2.1 : 1.9;
        int least = ns[0];
        for (int u = 1; u < units; ++u) least = std::min(least, ns[u]);
        int lg = 3;
        while (lg > 0 && (units > max_clusters[lg] || (1 << lg) > least)) --lg;
        const int C = 1 << lg;
        if (units <= max_clusters[lg] && units * C <= kMaxCtas && a.batch <= kFewSeqs) {
            double worst = 0.0, tile = 2 * kTT * 256 / 512, all = 0.0;  // in plain tiles
            // A block's time is its number of tiles, full or not, and the last block has the tail on top: so the blocks before it
            // take equal shares, or the next smaller or larger whole number of tiles where that leaves the slowest block with less.
            // (1024 tokens on eight blocks, eight slices each instead of up to nine: 7.0 -> 5.7 us a layer.)
            const int tsl = (a.rows_f8 ? kTT8 : kTT) / kResTile;  // slices of a tile
            std::vector<int> per(units);                          // slices of every block but the last
            for (int u = 0; u < units; ++u) {
                const int tail = a.host_tail ? (std::min(a.host_tail[u / a.Hkv], a.max_tail) + kTT - 1) / kTT : 0;
                const int even = (ns[u] + tail * (kTT / kResTile) + C - 1) / C;
                // (Latencies of one block: a residual tile is less far above a plain one than in the throughput of a full device, and a
                // tail tile, whose copy starts after the wait for the kernels ahead, takes a fifth of a tile more, with 8-bit rows half of one.  With a
                // half for all, 2 047 tokens and a tail were cut into blocks of 18 slices, three tiles, to spare the last block: 8.4 us a call against
                // 8.0, of four heads 8.2 and 7.6.  A 256-token tile of 8-bit rows counts as 1.7 plain ones.)
                const double rl = std::sqrt(wt[u] / tile) * (a.rows_f8 ? 1.7 : 1.0), tl = (a.rows_f8 ? 1.5 : 1.2) * tail;
                double best = -1.0;
                for (int p : {even / tsl * tsl, even, (even + tsl - 1) / tsl * tsl}) {
                    p = std::min(p, C > 1 ? (ns[u] - 1) / (C - 1) : 0);
                    if (p < (C > 1)) continue;
                    const int rest = ns[u] - (C - 1) * p;
                    const double t = std::max((p + tsl - 1) / tsl * rl, (rest + tsl - 1) / tsl * rl + tl);
                    if (best < 0.0 || t < best) { best = t; per[u] = p; }
                }
                worst = std::max(worst, best);
                all += (double)ns[u] * wt[u] / (kTT / kResTile) / tile + tail;
                if (!a.rows_f8 && total_tiles <= 5 * ctas) all += (double)(5 * total_tiles / ctas) / 8.0;
            }
            if (worst <= std::max(least_other, all / ctas) + gain) {
                int c = 0;
                for (int u = 0; u < units; ++u)
                    for (int j = 0; j < C; ++j, ++c) {
                        sch.start[c] = ((uint32_t)u << 20) | (uint32_t)(per[u] * j);
                        sch.slot[c] = (uint8_t)j;
                    }
                sch.start[c] = (uint32_t)units << 20;
                sch.ncta = c;
                sch.cluster = C;
                sch.inv_share = (float)C / (float)(128 * a.G);
                for (int u = 0; u < kMaxUnits; ++u) cs.n[u] = u < units ? C : 0;
                return cudaSuccess;
            }
        }
    }
    bool whole = units <= ncta;
    std::vector<int> nc(units, 1);
    if (whole) {
        // Whole CTAs per unit (no CTA pays a second merge): shares proportional to the unit's cost, at least
        // one each, the remainder to the units with the largest cost per CTA; never more CTAs than tiles.
        int given = units;
        for (int u = 0; u < units; ++u) {
            const int extra = std::min<int64_t>((int64_t)nt[u] - 1, (int64_t)((double)(ncta - units) * (double)(wp[u + 1] - wp[u]) / (double)wp[units]));
            nc[u] += std::max(0, extra);
            given += std::max(0, extra);
        }
        while (given < ncta) {
            int best = -1;
            double best_load = 0.0;
            for (int u = 0; u < units; ++u) {
                const double load = (double)(wp[u + 1] - wp[u]) / nc[u];
                if (nc[u] < nt[u] && load > best_load) { best_load = load; best = u; }
            }
            if (best < 0) break;
            ++nc[best];
            ++given;
        }
        if (given != ncta) whole = false;
        // with few CTAs per unit the integer shares are too uneven (2 vs 3 CTAs is +50 %): cut the flat list instead, unless
        // the unevenness is less than what a CTA that straddles two units pays for its second merge
        // (short contexts: a layer call of 2k tokens 9.7 us with the flat cut, 7.0 us without)
        constexpr double kFlatExtra = 4.0;  // (plain tiles)
        double worst = 0.0;
        for (int u = 0; u < units; ++u) worst = std::max(worst, (double)(wp[u + 1] - wp[u]) / nc[u]);
        if (worst > (double)wp[units] / ncta + kFlatExtra * (kTT / kResTile) * (2 * kTT * 256 / 512)) whole = false;
    }
    if (whole) {
        int c = 0;
        for (int u = 0; u < units; ++u)
            for (int j = 0; j < nc[u]; ++j) sch.start[c++] = ((uint32_t)u << 20) | (uint32_t)std::min<int64_t>(ns[u] - 1, (int64_t)es[u] * j / nc[u]);
        sch.start[ncta] = (uint32_t)units << 20;
    } else {
        weigh(1.5);
        int u = 0;
        for (int c = 0; c < ncta; ++c) {
            const int64_t target = wp[units] * c / ncta;
            while (u + 1 < units && wp[u + 1] <= target) ++u;
            const int slice = (int)std::min<int64_t>(ns[u], (target - wp[u]) / wt[u]);
            sch.start[c] = ((uint32_t)u << 20) | (uint32_t)slice;
        }
        sch.start[ncta] = (uint32_t)units << 20;
        // A CTA's segment table holds kMaxSeg units: where the cost cut gives one CTA a longer run of very short units
        // (a batch of one long and many one-token sequences), move whole units to its neighbours: first towards the
        // front, then towards the back.  Ranges stay ordered; a CTA may end up without work.
        auto nseg = [&](uint32_t s0, uint32_t s1) {
            const int ua = (int)(s0 >> 20), ta = (int)(s0 & 0xFFFFFu), ub = (int)(s1 >> 20), tb = (int)(s1 & 0xFFFFFu);
            int n = 0;
            for (int u2 = ua; u2 <= ub && u2 < units; ++u2)
                if ((u2 == ub ? tb : ns[u2]) > (u2 == ua ? ta : 0)) ++n;
            return n;
        };
        for (int c = ncta - 1; c >= 1; --c)
            while (nseg(sch.start[c], sch.start[c + 1]) > kMaxSeg) sch.start[c] = ((sch.start[c] >> 20) + 1) << 20;
        for (int c = 0; c + 1 < ncta; ++c)
            while (nseg(sch.start[c], sch.start[c + 1]) > kMaxSeg)
                sch.start[c + 1] = (sch.start[c + 1] & 0xFFFFFu) ? (sch.start[c + 1] >> 20) << 20 : ((sch.start[c + 1] >> 20) - 1) << 20;
    }
    // parts per unit = CTAs whose range contains at least one of its tiles
    for (int u = 0; u < kMaxUnits; ++u) cs.n[u] = 0;
    for (int c = 0; c < ncta; ++c) {
        sch.slot[c] = (sch.start[c] >> 20) < (uint32_t)units ? cs.n[sch.start[c] >> 20] : 0;
        const int ua = (int)(sch.start[c] >> 20), ta = (int)(sch.start[c] & 0xFFFFFu);
        const int ub = (int)(sch.start[c + 1] >> 20), tb = (int)(sch.start[c + 1] & 0xFFFFFu);
        int nseg_cta = 0;
        for (int u = ua; u <= ub && u < units; ++u) {
            const int b0 = u == ua ? ta : 0, b1 = u == ub ? tb : ns[u];
            if (b1 > b0) ++nseg_cta;
            if (b1 > b0 && cs.n[u] < 255) cs.n[u]++;
        }
        if (nseg_cta > kMaxSeg) return cudaErrorInvalidValue;  // only when units > kMaxSeg * CTAs (see the pass above)
    }
    for (int u = 0; u < units; ++u)
        if (cs.n[u] > kMaxSplits) return cudaErrorInvalidValue;  // cannot happen: ncta <= kMaxSplits
    return cudaSuccess;
}

// The plan alone, for a given number of CTAs (fdkv_plan_decode: host only, no device is touched).  max_clusters: as above.
cudaError_t plan_decode_host(const DecodeArgs& a, int n_ctas, const int* max_clusters, uint32_t* start_out, int32_t* ncta_out, int32_t* parts_out,
                             int32_t* cluster_out) {
    const int units = a.batch * a.Hkv;
    if (units < 1 || units > kMaxUnits || n_ctas < 1) return cudaErrorInvalidValue;
    FastSched sch;
    PartCount cs;
    const cudaError_t e = plan_decode_schedule(a, units, n_ctas, max_clusters, sch, cs);
    if (e != cudaSuccess) return e;
    for (int c = 0; c <= sch.ncta; ++c) start_out[c] = sch.start[c];
    for (int u = 0; u < units; ++u) parts_out[u] = cs.n[u];
    *ncta_out = sch.ncta;
    if (cluster_out) *cluster_out = sch.cluster;
    return cudaSuccess;
}

cudaError_t launch_decode_fast(const DecodeArgs& a, cudaStream_t st, bool* handled) {
    *handled = false;
    const int units = a.batch * a.Hkv;
    if (!a.tmap || !a.packed_lists || a.d != 128 || units > kMaxUnits || units < 1) return cudaSuccess;
    if (a.rows_f8 && !a.tmap_u8) return cudaSuccess;
    static PerDevice once;
    static int max_clusters_of[PerDevice::kMaxDevices][4];  // [device][log2 of the blocks]
    int sm_count = 0, dev = 0;
    cudaError_t e0 = cudaGetDevice(&dev);
    if (e0 == cudaSuccess) e0 = once.ensure([&]() {
        cudaError_t e = cudaSuccess;
        auto opt_in = [&](auto kernel, int smem) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        };
        opt_in(decode_fast_kernel<false, false, kFewSeqs, true>, smem_of(false, false));
        opt_in(decode_fast_kernel<false, false, kFewSeqs, false>, smem_of(false, false));
        opt_in(decode_fast_kernel<true, false, kFewSeqs, true>, smem_of(true, false));
        opt_in(decode_fast_kernel<false, false, kMaxUnits, true>, smem_of(false, false));
        opt_in(decode_fast_kernel<false, false, kMaxUnits, false>, smem_of(false, false));
        opt_in(decode_fast_kernel<true, false, kMaxUnits, true>, smem_of(true, false));
        opt_in(decode_fast_kernel<false, true, kFewSeqs, true>, smem_of(false, true));
        opt_in(decode_fast_kernel<false, true, kFewSeqs, false>, smem_of(false, true));
        opt_in(decode_fast_kernel<true, true, kFewSeqs, true>, smem_of(true, true));
        // the same division of the SM's memory as the decode kernel's, or the two could not share an SM
        if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_combine_kernel<2>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_combine_kernel<4>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        for (int lg = 0; lg < 4 && e == cudaSuccess; ++lg) {
            cudaLaunchConfig_t q = {};
            q.gridDim = dim3(8 << lg);
            q.blockDim = dim3(kThreads);
            q.dynamicSmemBytes = smem_of(true, true);
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = 1u << lg; at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            q.attrs = at;
            q.numAttrs = 1;
            e = cudaOccupancyMaxActiveClusters(&max_clusters_of[dev][lg], decode_fast_kernel<true, true, kFewSeqs, true>, &q);
        }
        return e;
    }, &sm_count);
    if (e0 != cudaSuccess) return e0;
    FastPlan& plan = *a.plan;
    bool current = plan.epoch == a.plan_epoch && plan.batch == a.batch && plan.sm_count == sm_count;
    for (int b = 0; current && b < a.batch; ++b) current = plan.tail_tiles[b] == (a.host_tail[b] + kTT - 1) / kTT;
    if (!current) {
        plan.epoch = 0;
        const cudaError_t pe = plan_decode_schedule(a, units, sm_count, max_clusters_of[dev], plan.sch, plan.pc);
        if (pe != cudaSuccess) return pe;
        plan.epoch = a.plan_epoch; plan.batch = a.batch; plan.sm_count = sm_count;
        plan.tail_tiles.resize(a.batch);
        for (int b = 0; b < a.batch; ++b) plan.tail_tiles[b] = (a.host_tail[b] + kTT - 1) / kTT;
    }
    const FastSched& sch = plan.sch;
    const PartCount& cs = plan.pc;
    const int ncta = sch.ncta;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ncta);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem_of(a.rows_f8, sch.cluster > 0);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = std::max(1, sch.cluster); attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = sch.cluster ? 2 : 1;
    const CUtensorMap& m16 = *reinterpret_cast<const CUtensorMap*>(a.tmap);
    const CUtensorMap& m8 = *reinterpret_cast<const CUtensorMap*>(a.rows_f8 ? a.tmap_u8 : a.tmap);
    auto launch = [&](auto* kernel, auto tl) {
        for (int b = 0; b < a.batch; ++b) tl.n[b] = a.host_tail[b];
        return cudaLaunchKernelEx(&cfg, kernel, m16, m8, a, sch, tl);
    };
    cudaError_t e;
    const bool split = a.G <= 4;  // (8-bit rows take no more)
    if (sch.cluster)
        e = launch(a.rows_f8 ? decode_fast_kernel<true, true, kFewSeqs, true>
                   : split   ? decode_fast_kernel<false, true, kFewSeqs, true>
                             : decode_fast_kernel<false, true, kFewSeqs, false>, TailLens<kFewSeqs>());
    else if (a.batch <= kFewSeqs)
        e = launch(a.rows_f8 ? decode_fast_kernel<true, false, kFewSeqs, true>
                   : split   ? decode_fast_kernel<false, false, kFewSeqs, true>
                             : decode_fast_kernel<false, false, kFewSeqs, false>, TailLens<kFewSeqs>());
    else
        e = launch(a.rows_f8 ? decode_fast_kernel<true, false, kMaxUnits, true>
                   : split   ? decode_fast_kernel<false, false, kMaxUnits, true>
                             : decode_fast_kernel<false, false, kMaxUnits, false>, TailLens<kMaxUnits>());
    if (e != cudaSuccess) return e;
    count_launch(1);
    count_kernel(FDKV_KERNEL_DECODE_FAST);
    *handled = true;
    if (sch.cluster) return cudaSuccess;
    // two ways per channel where a head has many parts (few heads: latency), one where the heads fill the machine
    const bool wide = units * a.G > sm_count;
    cfg.gridDim = dim3(wide ? 1 : 4, a.Hq, a.batch);
    cfg.blockDim = dim3(32);
    cfg.dynamicSmemBytes = 0;
    cfg.numAttrs = 1;
    const float* parts = a.partials;
    e = wide ? cudaLaunchKernelEx(&cfg, decode_combine_kernel<4>, parts, a.Hq, a.Hkv, a.G, cs, a.out, a.out_dtype)
             : cudaLaunchKernelEx(&cfg, decode_combine_kernel<2>, parts, a.Hq, a.Hkv, a.G, cs, a.out, a.out_dtype);
    if (e != cudaSuccess) return e;
    count_launch(1);
    return cudaGetLastError();
}

}  // namespace fdkv
