// Host side of the C ABI declared in include/disco.h: context, argument checks, kernel selection
// and launches.  No PyTorch types; plain pointers and sizes only.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>

#include "disco.h"
#include "stream_tail.cuh"
#include "umma_tail.cuh"
#include "draft_batch.cuh"
#include "draft_few.cuh"
#include "fetch.cuh"
#include "sample.cuh"
#include "umma_gemv_loop.cuh"

using namespace disco;

namespace {

constexpr int kStreamWarps = 16;     // consumer warps of the streaming kernel
constexpr int kMaxHidden = 16384;    // widest hidden dimension the kernels accept
constexpr int kSlotTargetBytes = 6144;

constexpr int kMaxDevices = 64;
// Hidden states that disco_iteration_host has a kernel bring over rather than the copy engine: by then the engine's second copy,
// which runs beside the draft phase, has made up for what its first one and the events around it cost (us per call, 32000 x 768
// and a target of the width given, engine -> kernel: 37 KB 69.0 -> 65.0, 150 KB 107.6 -> 104.4, 230 KB 108.1 -> 106.0, 256 KB 106.6 ->
// 104.0, 420 KB 106.7 -> 109.5, 490 KB 84.4 -> 86.5).
constexpr size_t kFetchBytes = 288 * 1024;

// One-time, per-device configuration of one kernel (its dynamic shared-memory limit).  Every template
// instance of a launcher owns one of these; the lock makes first calls from several host threads, and
// contexts on several devices, safe.
struct KernelSetup {
    std::mutex mu;
    bool done[kMaxDevices] = {};
    size_t dyn_limit[kMaxDevices] = {};
};

// Where an LM-head pass leaves its records (m, Z first) of consecutive vocabulary slabs: what a draw is located with.
struct RecordLayout {
    const float4* recs;
    int step, row, NP, slab;   // record and row strides in float4; records per row, vocabulary rows per record
};

struct StreamPlan {
    int rows_per_cta, grid, rps, stages;
    uint32_t slot_bytes;
    size_t smem;
    bool ok;
};

}  // namespace

struct disco_ctx {
    int device;
    int V, d_draft, d_target, max_batch, max_rows, clf_hidden;
    int sm_count;
    size_t smem_optin;
    int path;
    int pdl;  // launch the streaming kernel with programmatic stream serialization (DISCO_PDL=0 turns it off)
    long long launches;
    cudaStream_t last_stream;  // stream of the most recent enqueue (disco_last_device_status waits for it only)
    unsigned int test_stamp_skew;  // disco_test_hooks
    void* device_mem;  // every device buffer below
    void* host_mem;    // the pinned staging below
    // scratch for cross-block reductions
    int part_rows;  // rows the partial buffers can hold
    int max_grid;
    unsigned long long* keys;
    unsigned int* ticket;
    int* status;
    float* final_stats;            // [part_rows][2] (m, Z) of the rows of a pass
    float* final_stats2;           // the same for the second pass of a feature extraction
    uint8_t* chain_alive;          // [max_batch] draft phase on the device: which sequences still draft
    double* sample_seg_tot;        // verification with sampling: [max_batch][kSampleMaxSegments][2] sums of weights
    int32_t* sample_seg_last;      //   the same shape: last index with positive weight
    unsigned int* sample_tickets;  //   [max_batch]
    void* pack_rows;               // fixed-shape verification with many rows: the rows that count, packed
    int32_t* pack_off;             // [max(max_batch, max_rows) + 1] their offsets; the last entry is the row count
    void* loop_rec;                // persistent draft-phase kernel: stamped 80-byte records, [4][CTA]; written by nothing else
    void* part_rec;                // draft step: 64-byte partial records, [sequence][CTA]
    void* stamped_rec;             // batched draft step: stamped 80-byte records, [sequence][CTA]; written by nothing else
    unsigned int* row_bound;       // batched draft step: two sets of [part_rows][kDbBoundStride] words, see DraftBatchParams
    int part_slots;                // partials per row the buffers can hold
    void* encode_tiled;            // cuTensorMapEncodeTiled, resolved through the runtime
    void* pointer_attributes;      // cuPointerGetAttributes, the same way
    // device staging for the *_host entry points
    void* stage_hidden;
    void* stage_hidden_draft;      // disco_iteration_host: the draft hidden states of all steps
    int32_t* stage_dev;            // disco_iteration_host: pos0 | sl_forced (max_batch each) | draft_ids (max_rows)
    cudaStream_t copy_stream;      // disco_iteration_host: the target hidden states travel beside the draft phase
    cudaEvent_t copy_done;
    // Small inputs and outputs of the *_host entry points live in pinned host memory that the GPU maps:
    // the kernels read and write it in place, so a host call costs one copy (the hidden states), one
    // launch and one synchronisation.  *_h: host address, *_d: the same memory as the device sees it.
    int32_t *stage_int_h, *stage_int_d;    // pos | n_drafted | token | draft_ids | row_off | n_accept | bonus | target_ids
    float *stage_float_h, *stage_float_d;  // conf | feats
    uint8_t *stage_byte_h, *stage_byte_d;  // active | halt
};

namespace {

// With DISCO_DEBUG set in the environment, failed CUDA runtime calls are reported on stderr.
inline bool cuda_ok(cudaError_t e, const char* what) {
    if (e == cudaSuccess) return true;
    static const bool verbose = std::getenv("DISCO_DEBUG") != nullptr;
    if (verbose) std::fprintf(stderr, "[disco] %s: %s\n", what, cudaGetErrorString(e));
    return false;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Raise a kernel's dynamic shared-memory limit once per device: to `bytes`, or (bytes == 0) to all that the
// device allows beside the kernel's static shared memory.  *limit receives the value in force.
template <typename Kern>
bool raise_smem_limit(const disco_ctx* c, KernelSetup& ks, Kern kern, size_t bytes, size_t* limit) {
    if (c->device < 0 || c->device >= kMaxDevices) return false;
    std::lock_guard<std::mutex> lock(ks.mu);
    if (!ks.done[c->device]) {
        size_t want = bytes;
        if (want == 0) {
            cudaFuncAttributes fa;
            if (!cuda_ok(cudaFuncGetAttributes(&fa, kern), "cudaFuncGetAttributes")) return false;
            want = c->smem_optin - fa.sharedSizeBytes;
        }
        if (!cuda_ok(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)want),
                     "cudaFuncSetAttribute"))
            return false;
        ks.dyn_limit[c->device] = want;
        ks.done[c->device] = true;
    }
    if (limit) *limit = ks.dyn_limit[c->device];
    return true;
}

StreamPlan plan_stream(const disco_ctx* c, int V, int d, int RT, int clf_H) {
    StreamPlan pl{};
    const uint32_t row_bytes = (uint32_t)d * 2u;
    int rpc = (V + c->sm_count - 1) / c->sm_count;
    rpc = std::max(1, std::min(rpc, 2048));
    pl.rows_per_cta = rpc;
    pl.grid = (V + rpc - 1) / rpc;
    int rps = std::max(1, kSlotTargetBytes / (int)row_bytes);
    rps = std::min(rps, rpc);
    pl.rps = rps;
    pl.slot_bytes = (uint32_t)rps * row_bytes;
    const size_t fixed = stream_tail_smem_bytes(RT, kStreamWarps, d, 0, 0, clf_H);
    const size_t budget = c->smem_optin > 2048 ? c->smem_optin - 2048 : 0;
    if (budget <= fixed) return pl;
    long long stages = (long long)((budget - fixed) / (pl.slot_bytes + 16));
    stages = std::min<long long>(stages, 2 * kStreamWarps);
    if (stages > kStreamWarps) stages -= stages % kStreamWarps;  // slots are dealt round-robin to the warps
    if (stages < 2) return pl;
    pl.stages = (int)stages;
    pl.smem = stream_tail_smem_bytes(RT, kStreamWarps, d, pl.stages, pl.slot_bytes, clf_H);
    pl.ok = true;
    return pl;
}

template <int RT, bool DRAFT, int KC>
int launch_stream(disco_ctx* c, TailParams& p, const StreamPlan& pl, cudaStream_t st) {
    auto kern = stream_tail_kernel<RT, DRAFT, kStreamWarps, KC>;
    static KernelSetup setup;
    size_t dyn_limit = 0;
    if (!raise_smem_limit(c, setup, kern, 0, &dyn_limit)) return DISCO_ERR_CUDA;
    if (pl.smem > dyn_limit) return DISCO_ERR_UNSUPPORTED_SHAPE;
    // Programmatic dependent launch: the kernel may start while the preceding kernel of the stream is
    // still in its tail; it streams the LM head (never written by this library) and waits with
    // griddepcontrol.wait before it touches anything else.
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)pl.grid);
    cfg.blockDim = dim3((kStreamWarps + 1) * 32);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = c->pdl ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, p);
    c->launches += 1;
    return cuda_ok(e, "stream_tail_kernel launch") ? DISCO_OK : DISCO_ERR_CUDA;
}

template <bool DRAFT>
int run_stream(disco_ctx* c, TailParams& p, int clf_H, cudaStream_t st) {
    const int RT = p.R == 1 ? 1 : (p.R == 2 ? 2 : 4);
    const StreamPlan pl = plan_stream(c, p.V, p.d, RT, clf_H);
    if (!pl.ok) return DISCO_ERR_UNSUPPORTED_SHAPE;
    if (DRAFT && (pl.grid > c->max_grid || p.R > c->part_rows)) return DISCO_ERR_WORKSPACE;
    p.rows_per_cta = pl.rows_per_cta;
    p.rps = pl.rps;
    p.stages = pl.stages;
    p.slot_bytes = pl.slot_bytes;
    switch (RT) {
        case 1:  // one hidden row: the warp can hold its share of h in registers (32 * 8 * KC values)
            if (p.d <= 768) return launch_stream<1, DRAFT, 3>(c, p, pl, st);
            if (p.d <= 1024) return launch_stream<1, DRAFT, 4>(c, p, pl, st);
            return launch_stream<1, DRAFT, 0>(c, p, pl, st);
        case 2: return launch_stream<2, DRAFT, 0>(c, p, pl, st);
        default: return launch_stream<4, DRAFT, 0>(c, p, pl, st);
    }
}


// ------------------------------------------------------------------------------------------------
// tcgen05 path
// ------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// bf16 [rows, d] row-major, boxes of box_rows x 64 elements, 128-byte swizzle, zero fill out of bounds
bool encode_bf16_2d(const disco_ctx* c, CUtensorMap* map, const void* base, int rows, int d, int box_rows) {
    if (!c->encode_tiled) return false;
    const cuuint64_t gdim[2] = {(cuuint64_t)d, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)d * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kUmmaBK, (cuuint32_t)box_rows};
    const cuuint32_t estride[2] = {1, 1};
    const CUresult r = reinterpret_cast<EncodeTiledFn>(c->encode_tiled)(
        map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estride,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}


// Clusters of two CTAs, and programmatic stream serialization where that is on.
int launch_attributes(const disco_ctx* c, bool pair, cudaLaunchAttribute (&attr)[2]) {
    int n = 0;
    if (pair) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = 2;
        attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (c->pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    return n;
}

// Vocabulary on the TMEM lanes (umma_tail.cuh): few rows, and the first rows beyond one tile of 128, where the other form
// multiplies by 256.  In between and beyond it has no fewer multiplications and the dearer epilogue.  (Launches one after
// the other at the power limit, 32000 x 5120, 34 / 64 / 96 / 130 / 160 / 192 rows: 61.4 -> 56.2, 61.6 -> 58.2, 63.1 -> 62.5,
// 79.7 -> 68.9, 81.2 -> 72.6, 82.8 -> 81.1 us; 49152 x 6144, 64 / 96 / 160 / 192 rows: 113 -> 109, 115 -> 121, 158 -> 153,
// 160 -> 171 us.)  A head that takes less than some 10 us does not reach the power limit, and its epilogue is a larger part
// (6 rows, 8000 x 512: 7.1 us, 7.7 with the vocabulary on the lanes).  So a lower limit on the head's size for either band,
// from launches one after the other with the other form -> this one.  Up to 64 rows, 64 MB (d = 2048, 6 / 11 / 30 / 64 rows):
// 32 MB 11.8 / 12.0 / 12.9 / 13.4 -> 12.5 / 13.0 / 15.3 / 13.5 us; 64 MB 16.5 / 16.5 / 16.6 / 17.4 -> 16.6 / 16.8 / 18.4 / 17.2
// (17 to 32 rows catch up at 131 MB: 29.4 -> 28.6); 131 MB 29.3 / 29.3 / 29.4 / 29.9 -> 27.0 / 27.3 / 28.6 / 28.1.
// 129 to 160 rows, 45 MB, where the other form multiplies by 256 (130 / 160 rows): d = 1024, 32 MB 16.2 / 16.2 -> 15.0 / 15.0,
// 45 MB 18.3 / 18.4 -> 18.6 / 18.8, 96 MB 32.8 / 32.8 -> 32.3 / 33.3; d = 2048, 45 MB 20.4 / 20.3 -> 17.9 / 18.6, 131 MB
// 39.9 / 39.2 -> 34.3 / 36.1; d = 5120, 45 MB 29.6 / 29.6 -> 27.4 / 29.6, 320 MB 83.2 / 80.8 -> 67.1 / 71.3.  (It pays below
// 45 MB as well where the contraction is long.)  Forced path 2 takes no account of the size.
bool verify_on_lanes(const disco_ctx* c, int R, int d) {
    const size_t head_bytes = (size_t)c->V * d * 2;
    const bool few = R <= 64 && (head_bytes >= (size_t)64 << 20 || c->path == 2);
    const bool beyond = R > 128 && R <= 160 && (head_bytes >= (size_t)45 << 20 || c->path == 2);
    return few || beyond;
}

// Verification by pairs of CTAs (VerifyTiling::in_pairs).  A count in device memory: only where it is likely to be large, since the
// tiling that the kernel derives then may be one that pays or one that does not (whole iterations of 256 / 180 sequences with
// look-aheads up to 16 / 12, single CTAs -> pairs, us under continuous load: 32000 x 5120, 769 / 1350 / 1408 / 1676 / 2432 rows 384 / 547 /
// 547 / 542 / 832 -> 372 / 506 / 498 / 571 / 828; 49152 x 6144, 662 / 906 / 899 / 930 / 1421 -> 601 / 819 / 807 / 973 / 1438; 17000 x 2048, 1408 /
// 2432 rows 236 / 277 -> 227 / 281).
bool verify_in_pairs(const disco_ctx* c, int R, int d, bool dev_R, int likely_R) {
    if (dev_R) return d >= 1024 && likely_R > 1024 && VerifyTiling::pairs_possible(R, c->sm_count);
    return VerifyTiling::in_pairs(R, c->V, d, c->sm_count);
}

// CTAs that do nothing but finish a verification in the kernel that projects it (umma_tail.cuh), a warp for each sequence; 0: the
// rest must not get more to do for it, and there is a limit.  (us, 32000 x 5120 head, 11 rows of one sequence, launches one
// after the other: the last CTA to take a ticket finishes 53.5, a CTA of its own 52.3; in a graph 53.3 and 51.9.)
int verify_finishers(const disco_ctx* c, int R, int d, int B) {
    const int n = (B + kUmmaEpiWarps - 1) / kUmmaEpiWarps;
    if (n > 8 || !VerifyTiling::possible(R, c->sm_count - n)) return 0;
    const VerifyTiling all = VerifyTiling::make(R, c->V, d, c->sm_count), less = VerifyTiling::make(R, c->V, d, c->sm_count - n);
    return less.TPC == all.TPC && less.GS == all.GS && less.TRN <= all.TRN + (R <= 128 ? 16 : 0) ? n : 0;   // (one tile: HBM is the bound)
}

// Launch the tcgen05 verification kernel for R hidden rows of width d against the LM head W [V, d].
int launch_umma(disco_ctx* c, const void* W, const void* H, int d, int R, const UmmaParams* fused, cudaStream_t st,
                const int32_t* dev_R = nullptr, int likely_R = 0) {
    UmmaParams p{};
    if (fused) p = *fused;  // verification finished by the main kernel's last CTA
    p.V = c->V;
    p.d = d;
    p.R = R;
    p.dev_R = dev_R;
    const bool lanes = !dev_R && verify_on_lanes(c, R, d);
    const bool wide = lanes && R > kUmmaLaneRows;
    const bool pair = !lanes && verify_in_pairs(c, R, d, dev_R != nullptr, likely_R);
    p.t = pair ? VerifyTiling::make_pairs(R, c->V, d, c->sm_count) : VerifyTiling::make(R, c->V, d, c->sm_count - p.finishers);
    // (with the row count in device memory the kernel derives the tiling)
    p.box_rows = (dev_R ? 256 : p.t.TRN) / (pair ? 2 : 1);
    p.a_rows = lanes ? (R + 15) / 16 * 16 : pair || p.t.MT > 1 ? 128 : (R + 7) / 8 * 8;
    p.a_tiles = !lanes && (dev_R || p.t.GS == 2) ? 2 : 1;
    // The A tile holds a_rows rows.  The MMA still reads 128 rows from its start: what lies behind the tile (other
    // stages of the ring, always inside it) only feeds accumulator lanes nobody reads.
    p.a_bytes = (p.a_rows * 128 + 1023) / 1024 * 1024;
    p.b_bytes = (p.box_rows * 128 + 1023) / 1024 * 1024;
    p.stages = std::max(2, std::min(kUmmaMaxStages, kUmmaRingBytes / (p.a_bytes * p.a_tiles + p.b_bytes)));
    p.status = c->status;
    p.keys = c->keys;
    CUtensorMap tmap_W, tmap_H;
    if (!encode_bf16_2d(c, &tmap_W, W, c->V, d, p.box_rows) || !encode_bf16_2d(c, &tmap_H, H, R, d, p.a_rows))
        return DISCO_ERR_CUDA;
    static KernelSetup setup[7];
    auto kern = pair    ? umma_tail_kernel<false, false, true, false>
                : wide  ? (p.finishers ? umma_tail_kernel<true, true, false, true> : umma_tail_kernel<true, true, false, false>)
                : lanes ? (p.finishers ? umma_tail_kernel<true, false, false, true> : umma_tail_kernel<true, false, false, false>)
                        : (p.finishers ? umma_tail_kernel<false, false, false, true> : umma_tail_kernel<false, false, false, false>);
    const int smem_bytes = lanes ? kUmmaLaneSmemBytes : kUmmaSmemBytes;
    if (!raise_smem_limit(c, setup[pair ? 6 : lanes + wide + (p.finishers ? 3 : 0)], kern, (size_t)smem_bytes, nullptr)) return DISCO_ERR_CUDA;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(dev_R ? (pair ? c->sm_count & ~1 : c->sm_count) : p.t.groups * p.t.CN * (pair ? 2 : 1) + p.finishers));
    cfg.blockDim = dim3(kUmmaThreads);
    cfg.dynamicSmemBytes = (size_t)smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = launch_attributes(c, pair, attr);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tmap_W, tmap_H, p);
    c->launches += 1;
    return cuda_ok(e, "umma_tail_kernel launch") ? DISCO_OK : DISCO_ERR_CUDA;
}

// The batched draft step and its relatives need at most kDbMaxRecords CTAs per tile of rows and 28-bit token ids.
bool draft_batch_possible(const disco_ctx* c, int R) {
    const int MT = (R + 127) / 128;
    return c->encode_tiled != nullptr && MT <= c->sm_count && c->sm_count / MT <= kDbMaxRecords && c->V < (int)kDbNoIndex;
}

// Few hidden rows: the vocabulary on the TMEM lanes.  Up to 32, and beyond 16 only where a CTA has more than 32 vocabulary rows: with
// fewer there is no shared bound, and then the lists of four rows are one warp's work after another (us, 512-wide heads of 4000 /
// 8000, vocabulary on the columns -> on the lanes: 32 rows 9.9 / 11.7 -> 13.5 / 11.7, 16 rows 9.6 / 11.0 -> 9.6 / 9.5, 12 rows 9.5 / 9.8 -> 9.4 /
// 9.2, 4 rows 9.8 / 9.9 -> 9.2 / 9.3; of 1024 x 2000, 4 / 9 / 16 rows 9.8 / 10.0 / 9.7 -> 9.3 / 10.1 / 10.5).
bool draft_few_possible(const disco_ctx* c, int R) {
    return R <= 32 && c->sm_count >= 8 && (R <= 16 || c->V > 32 * (c->sm_count - draft_finishers(c->sm_count, R)));
}

template <bool STATS, int NR>
int launch_draft_few(disco_ctx* c, const void* W, const void* H, int d, int R, float* probs, const DraftFinalParams& f,
                     cudaStream_t st, RecordLayout* layout) {
    DraftBatchParams p{};
    p.V = c->V;
    p.d = d;
    p.R = R;
    p.MT = 1;
    p.finishers = draft_finishers(c->sm_count, R);
    p.CN = c->sm_count - p.finishers;
    p.TPC = std::max(1, (c->V + 128 * p.CN - 1) / (128 * p.CN));
    p.TR = (c->V + p.CN * p.TPC - 1) / (p.CN * p.TPC);
    p.TRN = std::max(16, (p.TR + 15) / 16 * 16);
    p.a_rows = 8 * NR;
    p.a_bytes = p.a_rows * 128;
    p.w_rows = p.TR;
    p.b_bytes = (p.w_rows * 128 + 1023) / 1024 * 1024;
    if ((size_t)R * p.CN > (size_t)128 * c->sm_count || R > c->part_rows) return DISCO_ERR_WORKSPACE;
    auto kern = umma_draft_few_kernel<STATS, NR>;
    static KernelSetup setup;
    size_t dyn_limit = 0;
    if (!raise_smem_limit(c, setup, kern, 0, &dyn_limit)) return DISCO_ERR_CUDA;
    const size_t fixed = draft_few_fixed_smem(NR, f.clf_H);
    // (an MMA reads 128 rows from the start of the last stage of W)
    const int stage_bytes = p.a_bytes + p.b_bytes;
    const size_t least = std::max((size_t)2 * stage_bytes, (size_t)p.b_bytes + 16384);
    if (dyn_limit < fixed + least) return DISCO_ERR_UNSUPPORTED_SHAPE;
    p.stages = (int)std::min<size_t>(kDbMaxStages, (dyn_limit - fixed) / stage_bytes);
    while (p.stages > 2 && fixed + (size_t)(p.stages - 1) * p.b_bytes + 16384 > dyn_limit) --p.stages;
    p.ring_bytes = std::max(p.stages * stage_bytes, (p.stages - 1) * p.b_bytes + 16384);
    p.status = c->status;
    p.part_rec = reinterpret_cast<float4*>(c->stamped_rec);
    p.probs = probs;
    p.bound = c->row_bound;
    p.set_words = (size_t)c->part_rows * kDbBoundStride;
    p.sync = c->ticket + 48;
    CUtensorMap tmap_W, tmap_H;
    if (!encode_bf16_2d(c, &tmap_W, W, c->V, d, p.w_rows) || !encode_bf16_2d(c, &tmap_H, H, R, d, p.a_rows))
        return DISCO_ERR_CUDA;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(p.CN + p.finishers));
    cfg.blockDim = dim3(kDbThreads);
    cfg.dynamicSmemBytes = fixed + p.ring_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = c->pdl ? 1 : 0;
    if (layout) *layout = RecordLayout{p.part_rec, 1, kStampedPieces * p.CN, p.CN, p.TPC * p.TR};
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tmap_W, tmap_H, p, f);
    c->launches += 1;
    return cuda_ok(e, "umma_draft_few_kernel launch") ? DISCO_OK : DISCO_ERR_CUDA;
}

// Launch the batched draft step (STATS: arg-max and statistics only) for R hidden rows of width d against W [V, d].
template <bool STATS>
int launch_draft_batch(disco_ctx* c, const void* W, const void* H, int d, int R, float* probs, const DraftFinalParams& f,
                       cudaStream_t st, RecordLayout* layout) {
    if (draft_few_possible(c, R)) {
        if (R <= 8) return launch_draft_few<STATS, 1>(c, W, H, d, R, probs, f, st, layout);
        if (R <= 16) return launch_draft_few<STATS, 2>(c, W, H, d, R, probs, f, st, layout);
        return launch_draft_few<STATS, 4>(c, W, H, d, R, probs, f, st, layout);
    }
    DraftBatchParams p{};
    p.V = c->V;
    p.d = d;
    p.R = R;
    const bool pair = draft_in_pairs(c->V, d, (R + 127) / 128, probs != nullptr, STATS, c->sm_count);
    const DraftTiling t = DraftTiling::make(c->V, d, R, probs != nullptr, pair, c->sm_count);
    p.MT = t.MT;
    p.finishers = t.finishers;
    p.CN = t.CN;
    p.TPC = t.TPC;
    p.TR = t.TR;
    p.TRN = t.TRN;
    p.a_rows = p.MT > 1 ? 128 : std::max(8, (R + 7) / 8 * 8);
    p.a_bytes = (p.a_rows * 128 + 1023) / 1024 * 1024;
    p.w_rows = pair ? p.TRN / 2 : p.TR;
    if ((size_t)R * p.CN > (size_t)128 * c->sm_count || R > c->part_rows) return DISCO_ERR_WORKSPACE;
    auto kern = pair ? umma_draft_batch_kernel<STATS, true> : umma_draft_batch_kernel<STATS, false>;
    static KernelSetup setup[2];
    size_t dyn_limit = 0;
    if (!raise_smem_limit(c, setup[pair], kern, 0, &dyn_limit)) return DISCO_ERR_CUDA;
    p.all_finish = p.finishers == 0 && R > kDbFinWarps * p.MT * p.CN;
    const int fin_warps = kDbFinWarps + (p.all_finish || p.finishers ? kDbEpiWarps : 0);
    const size_t fixed = 1024 + 512 + kDbXchBytes + (size_t)(fin_warps * kDbFinWords + 128) * 4 +
                         (probs ? kDbEpiWarps * 32 * kDbTurnStride * 4 : 0) + umma_clf_bytes(f.clf_H) + 128;
    // Room for what the MMA takes, or for the box alone where that makes one more stage (us, the former -> the latter: 90 rows of
    // 49152 x 768, five stages -> six, 22.9 -> 22.2; 100 rows of 49152 x 1024, five either way, 25.8 -> 26.2).
    const int roomy = ((pair ? p.TRN / 2 : p.TRN) * 128 + 1023) / 1024 * 1024, close = (p.w_rows * 128 + 1023) / 1024 * 1024;
    auto fit = [&](int b_bytes) {
        return dyn_limit < fixed ? 0 : (int)std::min<size_t>(kDbMaxStages, (dyn_limit - fixed) / (p.a_bytes + b_bytes));
    };
    p.b_bytes = fit(close) > fit(roomy) ? close : roomy;
    p.stages = fit(p.b_bytes);
    if (p.stages < 2) return DISCO_ERR_UNSUPPORTED_SHAPE;
    p.ring_bytes = p.stages * (p.a_bytes + p.b_bytes);
    p.status = c->status;
    p.part_rec = reinterpret_cast<float4*>(c->stamped_rec);
    p.probs = probs;
    p.bound = c->row_bound;
    p.set_words = (size_t)c->part_rows * kDbBoundStride;
    p.sync = c->ticket + 48;
    CUtensorMap tmap_W, tmap_H;
    if (!encode_bf16_2d(c, &tmap_W, W, c->V, d, p.w_rows) || !encode_bf16_2d(c, &tmap_H, H, R, d, p.a_rows))
        return DISCO_ERR_CUDA;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(p.MT * p.CN + p.finishers));
    cfg.blockDim = dim3(kDbThreads);
    cfg.dynamicSmemBytes = fixed + p.ring_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = launch_attributes(c, pair, attr);
    if (layout) *layout = RecordLayout{p.part_rec, 1, kStampedPieces * p.CN, p.CN, p.TPC * p.TR};
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tmap_W, tmap_H, p, f);
    c->launches += 1;
    return cuda_ok(e, "umma_draft_batch_kernel launch") ? DISCO_OK : DISCO_ERR_CUDA;
}


// The draft phase as one persistent kernel (1..4 sequences): see umma_gemv_loop.cuh.
template <int RK>
int launch_gemv_loop_rk(disco_ctx* c, GemvLoopParams& lp, const CUtensorMap& mW, const CUtensorMap& mH, cudaStream_t st) {
    auto kern = umma_gemv_loop_kernel<RK>;
    static KernelSetup setup;
    size_t dyn_limit = 0;
    if (!raise_smem_limit(c, setup, kern, 0, &dyn_limit)) return DISCO_ERR_CUDA;
    GemvParams& g = lp.g;
    const size_t fixed = gemv_loop_fixed_smem_bytes(RK, g.t.clf_H, g.t.d, g.h_rows, g.TRN);
    if (dyn_limit < fixed + 2 * (size_t)g.b_bytes) return DISCO_ERR_UNSUPPORTED_SHAPE;
    g.stages = (int)std::min<size_t>(kGemvMaxStages, (dyn_limit - fixed) / g.b_bytes);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)c->sm_count);
    cfg.blockDim = dim3(kGemvThreads);
    cfg.dynamicSmemBytes = fixed + (size_t)g.stages * g.b_bytes;
    cfg.stream = st;
    // the steps hand over through global memory: every CTA has to be running, which a cooperative launch checks
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = c->pdl ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, mW, mH, lp);
    c->launches += 1;
    return cuda_ok(e, "umma_gemv_loop_kernel launch") ? DISCO_OK : DISCO_ERR_CUDA;
}

bool gemv_loop_possible(const disco_ctx* c, int B, int sl_max, size_t w_step_stride) {
    if (!c->encode_tiled || B > 4 || sl_max > kLoopMaxSteps) return false;
    if (c->path != 0 && c->path != 3) return false;
    if ((c->V + c->sm_count - 1) / c->sm_count > 256 * kGemvMaxTiles) return false;   // the fold's lists
    if (w_step_stride != 0 && w_step_stride != (size_t)c->V * c->d_draft * 2) return false;   // one tensor map over all copies
    if ((long long)c->V * sl_max > 0x7fffffffll) return false;
    return (size_t)((c->d_draft + kUmmaBK - 1) / kUmmaBK) * 8 * 128 <= 48 * 1024;
}

int steps_per_launch(const disco_ctx* c, int B, int sl_max, size_t w_step_stride) {
    if (w_step_stride != 0 || c->path != 0) return 1;
    const int most = std::min(std::min(kMaxGroup, sl_max), c->part_rows / B);
    if (most < 2 || !draft_batch_possible(c, most * B)) return 1;
    return draft_steps_per_launch(c->V, c->d_draft, B, sl_max, most, c->sm_count);
}

int launch_gemv_loop(disco_ctx* c, const TailParams& t, int steps, size_t w_step_stride, cudaStream_t st) {
    GemvLoopParams lp{};
    GemvParams& g = lp.g;
    g.t = t;
    const int grid = c->sm_count;
    if (grid > kGroupMaxRecords) return DISCO_ERR_UNSUPPORTED_SHAPE;
    g.TR = (t.V + grid - 1) / grid;
    g.tiles = (g.TR + 255) / 256;
    g.TRt = (g.TR + g.tiles - 1) / g.tiles;
    g.TRN = (g.TRt + 15) / 16 * 16;
    g.b_bytes = (g.TRN * 128 + 1023) / 1024 * 1024;
    g.h_rows = 8;
    lp.steps = steps;
    lp.w_rows_per_step = w_step_stride ? t.V : 0;
    lp.flags = c->ticket + 64;
    lp.epoch = c->ticket + 128;
    lp.records = reinterpret_cast<float4*>(c->loop_rec);
    CUtensorMap mW, mH;
    if (!encode_bf16_2d(c, &mW, t.W, t.V * (w_step_stride ? steps : 1), t.d, g.TRN) ||
        !encode_bf16_2d(c, &mH, t.H, t.R * steps, t.d, g.h_rows))
        return DISCO_ERR_CUDA;
    if (t.R == 1) return launch_gemv_loop_rk<1>(c, lp, mW, mH, st);
    if (t.R == 2) return launch_gemv_loop_rk<2>(c, lp, mW, mH, st);
    return launch_gemv_loop_rk<4>(c, lp, mW, mH, st);
}

void fill_scratch(const disco_ctx* c, TailParams& p) {
    p.part_rec = reinterpret_cast<float4*>(c->part_rec);
    p.keys = c->keys;
    p.ticket = c->ticket;
    p.status = c->status;
    p.final_stats = c->final_stats;
}

int check_clf(const disco_ctx* c, const disco_clf* clf) {
    if (!clf || !clf->W1 || !clf->b1 || !clf->w2 || !clf->b2) return DISCO_ERR_INVALID_ARG;
    if (clf->H < 1 || clf->H > DISCO_MAX_CLF_HIDDEN) return DISCO_ERR_INVALID_ARG;
    if (clf->H > c->clf_hidden) return DISCO_ERR_WORKSPACE;
    return DISCO_OK;
}

}  // namespace

extern "C" {

const char* disco_strerror(int code) {
    switch (code) {
        case DISCO_OK: return "ok";
        case DISCO_ERR_INVALID_ARG: return "invalid argument (null or misaligned pointer, size out of range)";
        case DISCO_ERR_UNSUPPORTED_SHAPE: return "shape not supported by the kernels";
        case DISCO_ERR_WORKSPACE: return "batch, rows or classifier width beyond what the context was created for";
        case DISCO_ERR_CUDA: return "a CUDA runtime call failed";
        case DISCO_ERR_TIMEOUT: return "a bounded device-side wait ran out";
        case DISCO_ERR_STATIC_LIMIT: return "size beyond the fixed scratch of the allocation-free entry point";
        default: return "unknown disco status";
    }
}

int disco_create(disco_ctx** out, int V, int d_draft, int d_target, int max_batch, int max_rows, int k,
                 int clf_hidden) {
    if (!out) return DISCO_ERR_INVALID_ARG;
    if (V < 1 || d_draft < 8 || d_target < 8 || (d_draft % 8) || (d_target % 8)) return DISCO_ERR_INVALID_ARG;
    if (max_batch < 1 || max_rows < 1 || k != DISCO_TOPK) return DISCO_ERR_INVALID_ARG;
    if (clf_hidden < 1 || clf_hidden > DISCO_MAX_CLF_HIDDEN) return DISCO_ERR_INVALID_ARG;
    if (d_draft > kMaxHidden || d_target > kMaxHidden) return DISCO_ERR_UNSUPPORTED_SHAPE;

    disco_ctx* c = new (std::nothrow) disco_ctx();
    if (!c) return DISCO_ERR_CUDA;
    std::memset(c, 0, sizeof(*c));
    int sms = 0, optin = 0;   // (two attributes: the whole cudaDeviceProp takes milliseconds)
    if (cudaGetDevice(&c->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device) != cudaSuccess) {
        delete c;
        return DISCO_ERR_CUDA;
    }
    c->V = V;
    c->d_draft = d_draft;
    c->d_target = d_target;
    c->max_batch = max_batch;
    c->max_rows = max_rows;
    c->clf_hidden = clf_hidden;
    {
        const char* e = std::getenv("DISCO_PDL");
        c->pdl = !(e && e[0] == '0');
    }
    c->sm_count = sms;
    c->smem_optin = (size_t)optin;

    const int rpc = std::max(1, std::min((V + c->sm_count - 1) / c->sm_count, 2048));
    c->max_grid = (V + rpc - 1) / rpc;
    c->part_rows = std::max(max_batch, max_rows);  // the target rows of a verification with sampling go the same way
    c->part_slots = std::max(c->max_grid, 2 * c->sm_count);
    const size_t slots = (size_t)c->part_rows * c->part_slots;
    {
        cudaDriverEntryPointQueryResult qres;
        void* fn = nullptr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            c->encode_tiled = fn;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &fn, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            c->pointer_attributes = fn;
    }
    // the largest layout is disco_iteration_host's: 6 arrays of max_batch words and 2 of max_rows
    const size_t n_int = (size_t)8 * max_batch + (size_t)3 * max_rows + 64;
    const size_t hid = std::max((size_t)max_batch * d_draft, (size_t)max_rows * d_target) * 2;
    // One device allocation and one pinned one, cut into pieces of 256 bytes; what must start at zero comes first.
    // (A call to the allocator costs tens of microseconds to milliseconds, and there are about twenty pieces.)
    size_t dev_bytes = 0, host_bytes = 0, zero_bytes = 0;
    struct Piece {
        void** p;
        size_t at;
    };
    Piece pieces[32];
    int n_pieces = 0;
    auto device = [&](auto** p, size_t bytes) {
        pieces[n_pieces++] = Piece{reinterpret_cast<void**>(p), dev_bytes};
        dev_bytes += (bytes + 255) & ~(size_t)255;
    };
    device(&c->keys, (size_t)max_rows * sizeof(unsigned long long));
    device(&c->ticket, 1024);
    device(&c->status, 256);
    device(&c->loop_rec, (size_t)4 * c->sm_count * 80);            // no stamp yet
    // R rows take R * (sm_count / ceil(R / 128)) <= 128 * sm_count records
    device(&c->stamped_rec, (size_t)128 * c->sm_count * 80);       // no stamp yet
    device(&c->row_bound, (size_t)2 * c->part_rows * kDbBoundStride * 4);
    zero_bytes = dev_bytes;
    device(&c->part_rec, slots * 64);
    device(&c->final_stats, (size_t)c->part_rows * 2 * sizeof(float));
    device(&c->final_stats2, (size_t)c->part_rows * 2 * sizeof(float));
    device(&c->chain_alive, (size_t)max_batch + 64);
    device(&c->sample_seg_tot, (size_t)max_batch * kSampleMaxSegments * 2 * sizeof(double));
    device(&c->sample_seg_last, (size_t)max_batch * kSampleMaxSegments * 2 * sizeof(int32_t));
    device(&c->sample_tickets, (size_t)max_batch * sizeof(unsigned int));
    device(&c->pack_rows, (size_t)max_rows * d_target * 2);
    // (a fixed-shape verification is bounded by its rows alone, and every sequence has at least one)
    device(&c->pack_off, ((size_t)std::max(max_batch, max_rows) + 1) * sizeof(int32_t));
    device(&c->stage_hidden, hid);
    device(&c->stage_hidden_draft, (size_t)max_rows * d_draft * 2);
    device(&c->stage_dev, (2 * (size_t)max_batch + (size_t)max_rows) * sizeof(int32_t));
    auto pinned = [&](size_t bytes) {
        const size_t at = host_bytes;
        host_bytes += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t at_int = pinned(n_int * sizeof(int32_t));
    const size_t at_float = pinned(((size_t)max_batch * (1 + kNFeat) + max_rows) * sizeof(float));
    const size_t at_byte = pinned((size_t)max_batch * 2 + max_rows + 64);
    void* host_d = nullptr;
    bool ok = cudaMalloc(&c->device_mem, dev_bytes) == cudaSuccess;
    ok = ok && cudaHostAlloc(&c->host_mem, host_bytes, cudaHostAllocMapped) == cudaSuccess;
    ok = ok && cudaHostGetDevicePointer(&host_d, c->host_mem, 0) == cudaSuccess;
    ok = ok && cudaStreamCreateWithFlags(&c->copy_stream, cudaStreamNonBlocking) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&c->copy_done, cudaEventDisableTiming) == cudaSuccess;
    ok = ok && cudaMemset(c->device_mem, 0, zero_bytes) == cudaSuccess;
    if (ok) {
        for (int i = 0; i < n_pieces; ++i) *pieces[i].p = static_cast<char*>(c->device_mem) + pieces[i].at;
        char *h = static_cast<char*>(c->host_mem), *d = static_cast<char*>(host_d);
        c->stage_int_h = reinterpret_cast<int32_t*>(h + at_int), c->stage_int_d = reinterpret_cast<int32_t*>(d + at_int);
        c->stage_float_h = reinterpret_cast<float*>(h + at_float), c->stage_float_d = reinterpret_cast<float*>(d + at_float);
        c->stage_byte_h = reinterpret_cast<uint8_t*>(h + at_byte), c->stage_byte_d = reinterpret_cast<uint8_t*>(d + at_byte);
    }
    ok = ok && cudaDeviceSynchronize() == cudaSuccess;
    if (!ok) {
        disco_destroy(c);
        return DISCO_ERR_CUDA;
    }
    *out = c;
    return DISCO_OK;
}

int disco_destroy(disco_ctx* c) {
    if (!c) return DISCO_ERR_INVALID_ARG;
    cudaFree(c->device_mem);
    if (c->copy_stream) cudaStreamDestroy(c->copy_stream);
    if (c->copy_done) cudaEventDestroy(c->copy_done);
    cudaFreeHost(c->host_mem);
    delete c;
    return DISCO_OK;
}

int disco_last_device_status(disco_ctx* c, int* out) {
    if (!c || !out) return DISCO_ERR_INVALID_ARG;
    // read and clear on the stream the context was last used on: nothing else on the device is waited for
    int v = 0;
    if (cudaMemcpyAsync(&v, c->status, sizeof(int), cudaMemcpyDeviceToHost, c->last_stream) != cudaSuccess ||
        cudaMemsetAsync(c->status, 0, sizeof(int), c->last_stream) != cudaSuccess ||
        cudaStreamSynchronize(c->last_stream) != cudaSuccess)
        return DISCO_ERR_CUDA;
    *out = v;
    return DISCO_OK;
}

int disco_launch_count(disco_ctx* c, long long* out) {
    if (!c || !out) return DISCO_ERR_INVALID_ARG;
    *out = c->launches;
    return DISCO_OK;
}

int disco_test_hooks(disco_ctx* c, long long wait_budget_clocks, int withhold_records) {
    if (!c || wait_budget_clocks < 0) return DISCO_ERR_INVALID_ARG;
    const long long budget = wait_budget_clocks ? wait_budget_clocks : kDefaultWaitBudgetClocks;
    if (cudaMemcpyToSymbol(g_wait_budget_clocks, &budget, sizeof(budget)) != cudaSuccess) return DISCO_ERR_CUDA;
    c->test_stamp_skew = withhold_records ? 0x40000000u : 0u;
    return DISCO_OK;
}

int disco_set_kernel_path(disco_ctx* c, int which) {
    if (!c || which < 0 || which > 3) return DISCO_ERR_INVALID_ARG;
    c->path = which;
    return DISCO_OK;
}

}  // extern "C"

namespace {
// Launch a small follow-up kernel with programmatic stream serialization (it waits with griddepcontrol.wait
// before it reads anything), so that its launch latency hides behind the kernel before it.
template <typename... KArgs, typename... Args>
cudaError_t launch_after(const disco_ctx* c, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                         Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = c->pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// Host memory as the device sees it, if all of [p, p + bytes) is pinned, 16-byte aligned memory of one allocation.
const void* device_view(const disco_ctx* c, const void* p, size_t bytes) {
    if (!c->pointer_attributes || !aligned16(p)) return nullptr;
    unsigned int type = 0;
    unsigned long long dev = 0, start = 0;
    size_t size = 0;
    CUpointer_attribute what[4] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                   CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* where[4] = {&type, &dev, &start, &size};
    using Fn = CUresult (*)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
    const unsigned long long at = reinterpret_cast<unsigned long long>(p);
    if (reinterpret_cast<Fn>(c->pointer_attributes)(4, what, where, at) != CUDA_SUCCESS) return nullptr;
    if (type != CU_MEMORYTYPE_HOST || dev == 0 || (dev & 15u) || at < start || at + bytes > start + size) return nullptr;
    return reinterpret_cast<const void*>(dev);
}

// The end of a *_host entry point, failed or not: its copies read the caller's memory and its kernels the staging buffers, so
// nothing of the call may still be on its way when it returns.
int host_call_done(const disco_ctx* c, int rc, cudaStream_t st, bool used_copy_stream = false) {
    if (rc && used_copy_stream) cudaStreamSynchronize(c->copy_stream);   // (a call that did not fail made st wait for it)
    const bool ok = cudaStreamSynchronize(st) == cudaSuccess;
    return rc ? rc : (ok ? (int)DISCO_OK : (int)DISCO_ERR_CUDA);
}

// Shared body of the LM-head + soft-max passes: B rows of hidden size d against the head W.
//   * nll_sum != null selects the perplexity rule (no classifier; tau is the perplexity bound);
//   * stats_only = 1: arg-max (token, optional) and soft-max statistics only, no classifier: the target
//     rows of a verification with sampling (pos, n_drafted, conf, halt unused);
//   * stats_only = 2: token and features, no classifier: bulk feature extraction (n_drafted, conf, halt unused).
int draft_step_common(disco_ctx* c, const void* W_D, const void* h_D, int d, int B, int max_rows, const int32_t* pos,
                      const int32_t* n_drafted, const uint8_t* active, const disco_clf* clf, float tau,
                      int sl_max, int32_t* token, float* conf, uint8_t* halt, float* feats, float* probs,
                      float* nll_sum, int stats_only, void* stream, bool normalize = true,
                      RecordLayout* layout = nullptr, const ChainLink* chain = nullptr, unsigned int* clear_words = nullptr, int clear_n = 0,
                      float* stats = nullptr) {
    if (!c || !W_D || !h_D) return DISCO_ERR_INVALID_ARG;
    if (!stats_only && !chain && (!pos || !n_drafted)) return DISCO_ERR_INVALID_ARG;
    if (!stats_only && (!token || !conf || !halt)) return DISCO_ERR_INVALID_ARG;
    if (stats_only == 2 && (!pos || !feats)) return DISCO_ERR_INVALID_ARG;
    if (!aligned16(W_D) || !aligned16(h_D)) return DISCO_ERR_INVALID_ARG;
    if (B < 1 || sl_max < 1) return DISCO_ERR_INVALID_ARG;
    if (B > max_rows) return DISCO_ERR_WORKSPACE;
    static const disco_clf no_clf = {nullptr, nullptr, nullptr, nullptr, 0};
    int rc = DISCO_OK;
    if (nll_sum || stats_only) {
        clf = &no_clf;
    } else {
        rc = check_clf(c, clf);
        if (rc) return rc;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    c->last_stream = st;

    TailParams p{};
    p.W = static_cast<const uint16_t*>(W_D);
    p.H = static_cast<const uint16_t*>(h_D);
    p.V = c->V;
    p.d = d;
    p.R = B;
    p.B = B;
    fill_scratch(c, p);
    if (stats) p.final_stats = stats;
    p.stats_only = stats_only;
    p.pos = pos;
    p.n_drafted = n_drafted;
    p.active = active;
    if (chain) p.chain = *chain;
    p.clear_words = clear_words;
    p.clear_n = clear_n;
    p.clf_W1 = clf->W1;
    p.clf_b1 = clf->b1;
    p.clf_w2 = clf->w2;
    p.clf_b2 = clf->b2;
    p.clf_H = clf->H;
    p.tau = tau;
    p.sl_max = sl_max;
    p.token = token;
    p.conf = conf;
    p.halt = halt;
    p.feats = feats;
    p.probs = probs;
    p.nll_sum = nll_sum;
    // The tensor-core kernels serve every batch (us per step in a stream, cold L2: one sequence of 32000 x 768 11.4, 7 of
    // 40011 x 768 14.4, 64 of 32000 x 768 16.5); the CUDA-core streaming kernel is the path without tensor maps.
    const bool use_umma = draft_batch_possible(c, B) && c->path != 1;
    if (use_umma) {
        DraftFinalParams f{};
        f.B = B;
        f.pos = pos;
        f.n_drafted = n_drafted;
        f.active = active;
        f.clf_W1 = clf->W1;
        f.clf_b1 = clf->b1;
        f.clf_w2 = clf->w2;
        f.clf_b2 = clf->b2;
        f.clf_H = clf->H;
        f.tau = tau;
        f.sl_max = sl_max;
        f.token = token;
        f.conf = conf;
        f.halt = halt;
        f.feats = feats;
        f.final_stats = p.final_stats;
        f.nll_sum = nll_sum;
        f.stats_only = stats_only;
        f.test_stamp_skew = c->test_stamp_skew;
        f.clear_words = clear_words;
        f.clear_n = clear_n;
        if (chain) f.chain = *chain;
        rc = stats_only == 1 ? launch_draft_batch<true>(c, W_D, h_D, d, B, probs, f, st, layout)
                             : launch_draft_batch<false>(c, W_D, h_D, d, B, probs, f, st, layout);
        if (rc) return rc;
    } else {
        rc = run_stream<true>(c, p, clf->H, st);
        if (rc) return rc;
        const int slabs = (p.V + p.rows_per_cta - 1) / p.rows_per_cta;
        if (layout) *layout = RecordLayout{p.part_rec, 4, 4 * slabs, slabs, p.rows_per_cta};
    }
    if (probs && normalize) {
        dim3 grid((unsigned)std::min(64, (c->V + 255) / 256), (unsigned)B);
        const cudaError_t e = launch_after(c, normalize_probs_kernel, grid, dim3(256), 0, st, probs,
                                           (const float*)c->final_stats, active, c->V);
        c->launches += 1;
        if (!cuda_ok(e, "normalize_probs_kernel launch")) return DISCO_ERR_CUDA;
    }
    return DISCO_OK;
}

// Verification of R rows for B sequences.  pad == null: packed rows (row_off, or a uniform look-ahead SL);
// pad != null: the fixed-shape layout, R = B * (SL + 1) rows of which the first sl[b] + 1 of each sequence
// count (sl is device memory).
int verify_common(disco_ctx* c, const void* W_T, const void* H_T, const int32_t* draft_ids, const int32_t* row_off,
                  int B, int R, int SL, int32_t* n_accept, int32_t* bonus, int32_t* target_ids,
                  const VerifyPadded* pad, void* stream) {
    if (!aligned16(W_T) || !aligned16(H_T)) return DISCO_ERR_INVALID_ARG;
    if (R > c->max_rows) return DISCO_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    c->last_stream = st;

    TailParams p{};
    p.W = static_cast<const uint16_t*>(W_T);
    p.H = static_cast<const uint16_t*>(H_T);
    p.V = c->V;
    p.d = c->d_target;
    p.R = R;
    p.B = B;
    p.SL = SL;
    fill_scratch(c, p);
    p.draft_ids = draft_ids;
    p.row_off = row_off;
    p.n_accept = n_accept;
    p.bonus = bonus;
    p.target_ids = target_ids;
    if (pad) p.padded = *pad;
    const bool use_umma = c->encode_tiled != nullptr && VerifyTiling::possible(R, c->sm_count) &&
                          (c->path == 2 || (c->path == 0 && R >= 2));
    if (!use_umma) return run_stream<false>(c, p, 0, st);
    // Fixed-shape rows beyond one tile of 128: the projection is no longer free of charge for the rows that do not
    // count, so they are packed first and the tensor-core kernel tiles for the row count it finds on the device.
    const int32_t* dev_R = nullptr;
    const int likely_R = pad ? (int)((long long)B * (SL + 3) / 2) : R;   // look-aheads anything from 1 to SL
    if (pad && R > 128) {
        PackParams pk{};
        pk.H = static_cast<const uint16_t*>(H_T);
        pk.packed = static_cast<uint16_t*>(c->pack_rows);
        pk.sl = pad->sl;
        pk.off = c->pack_off;
        pk.off_user = pad->row_off_out;
        pk.B = B;
        pk.SL = SL;
        pk.d = c->d_target;
        const cudaError_t e = launch_after(c, pack_rows_kernel, dim3((unsigned)(SL + 1), (unsigned)B), dim3(128), 0, st, pk);
        c->launches += 1;
        if (!cuda_ok(e, "pack_rows_kernel launch")) return DISCO_ERR_CUDA;
        H_T = c->pack_rows;
        p.padded.packed_off = c->pack_off;
        p.padded.row_off_out = nullptr;
        dev_R = c->pack_off + B;
    }
    // CTAs of their own finish the job in the same launch where that costs the others nothing (us, a second launch -> finishing
    // CTAs, rows of 2 and 4 a sequence: 17 sequences of 32000 x 2048 26.8 / 26.5 -> 24.7 / 25.1, 32 26.8 / 27.2 -> 24.9 / 26.0, 64 28.7 /
    // 34.8 -> 28.1 / 31.0; 17 of 8000 x 2048 13.6 / 13.3 -> 12.9 / 12.4).  Where it does not: with few sequences the last CTA of the main
    // kernel, whose eight warps take the sequences in turn behind a fence and a ticket; with more a second launch, which hides
    // under the first (us in one / two launches, 32000 x 2048, 5 rows each: 4 sequences 26.9 / 27.3, 8 26.5 / 26.8, 16 29.0 / 28.6, 20
    // 30.2 / 29.7, 32 35.3 / 33.4; 32000 x 5120: 54.6 / 55.1, 55.8 / 56.0, 60.0 / 59.2, 63.2 / 59.6).
    const bool pairs = !verify_on_lanes(c, R, c->d_target) && verify_in_pairs(c, R, c->d_target, false, R);
    // (behind a draft phase, pad: 89.0 us in the other form against 92.4, 11 rows of 32000 x 5120 and steps with a head each)
    const int finishers = dev_R || pairs || pad ? 0 : verify_finishers(c, R, c->d_target, B);
    if (B <= 16 || finishers) {
        UmmaParams fp{};
        fp.fuse_final = 1;
        fp.finishers = finishers;
        fp.ticket = c->ticket + 32;
        fp.draft_ids = draft_ids;
        fp.row_off = row_off;
        fp.B = B;
        fp.SL = p.SL;
        fp.n_accept = n_accept;
        fp.bonus = bonus;
        fp.target_ids = target_ids;
        fp.padded = p.padded;
        return launch_umma(c, W_T, H_T, c->d_target, R, &fp, st, dev_R, likely_R);
    }
    int rc = launch_umma(c, W_T, H_T, c->d_target, R, nullptr, st, dev_R, likely_R);
    if (rc) return rc;
    VerifyFinalParams f{};
    f.keys = c->keys;
    f.draft_ids = draft_ids;
    f.row_off = row_off;
    f.B = B;
    f.SL = p.SL;
    f.R = R;
    f.n_accept = n_accept;
    f.bonus = bonus;
    f.target_ids = target_ids;
    f.status = c->status;
    f.ticket = c->ticket + 16;
    f.padded = p.padded;
    f.dev_R = dev_R;
    const cudaError_t e = launch_after(c, verify_finalize_kernel, dim3((unsigned)((B + 3) / 4)), dim3(128), 0, st, f);
    c->launches += 1;
    return cuda_ok(e, "verify_finalize_kernel launch") ? DISCO_OK : DISCO_ERR_CUDA;
}

}  // namespace

extern "C" {

int disco_draft_step(disco_ctx* c, const void* W_D, const void* h_D, int B, const int32_t* pos,
                     const int32_t* n_drafted, const uint8_t* active, const disco_clf* clf, float tau,
                     int sl_max, int32_t* token, float* conf, uint8_t* halt, float* feats, float* probs,
                     void* stream) {
    if (!c) return DISCO_ERR_INVALID_ARG;
    return draft_step_common(c, W_D, h_D, c->d_draft, B, c->max_batch, pos, n_drafted, active, clf, tau, sl_max, token,
                             conf, halt, feats, probs, nullptr, 0, stream);
}

int disco_draft_step_ppl(disco_ctx* c, const void* W_D, const void* h_D, int B, const int32_t* n_drafted,
                         const uint8_t* active, float* nll_sum, float ppl_max, int sl_max, int32_t* token,
                         float* ppl, uint8_t* halt, void* stream) {
    if (!nll_sum) return DISCO_ERR_INVALID_ARG;
    if (!c) return DISCO_ERR_INVALID_ARG;
    return draft_step_common(c, W_D, h_D, c->d_draft, B, c->max_batch, n_drafted, n_drafted, active, nullptr, ppl_max,
                             sl_max, token, ppl, halt, nullptr, nullptr, nll_sum, 0, stream);
}

int disco_draft_step_sample(disco_ctx* c, const void* W_D, const void* h_D, int B, const int32_t* pos,
                            const int32_t* n_drafted, const uint8_t* active, const disco_clf* clf, float tau,
                            int sl_max, const float* u, int32_t* token, float* p_token, float* conf, uint8_t* halt,
                            float* feats, float* probs, void* stream) {
    if (!c || !u || !probs) return DISCO_ERR_INVALID_ARG;
    RecordLayout rl{};
    int rc = draft_step_common(c, W_D, h_D, c->d_draft, B, c->max_batch, pos, n_drafted, active, clf, tau, sl_max,
                               token, conf, halt, feats, probs, nullptr, 0, stream, false, &rl);
    if (rc) return rc;
    // probs holds the logits: the kernel turns them into y^D and replaces the greedy token by the draw
    DrawRowsParams dp{};
    dp.rec_step = rl.step;
    dp.rec_row = rl.row;
    dp.NP = rl.NP;
    dp.slab = rl.slab;
    // about two CTAs per SM, at least one slab each
    const int seg = std::max(1, std::min(rl.NP, 2 * c->sm_count / B));
    dp.seg_slabs = (rl.NP + seg - 1) / seg;
    dp.V = c->V;
    constexpr int kMaxRows = 65535;   // a grid's second dimension
    for (size_t b0 = 0; b0 < (size_t)B; b0 += kMaxRows) {
        dp.probs = probs + b0 * c->V;
        dp.stats = c->final_stats + 2 * b0;
        dp.recs = rl.recs + b0 * rl.row;
        dp.u = u + b0;
        dp.active = active ? active + b0 : nullptr;
        dp.token = token + b0;
        dp.p_token = p_token ? p_token + b0 : nullptr;
        const dim3 grid((unsigned)((rl.NP + dp.seg_slabs - 1) / dp.seg_slabs), (unsigned)std::min<size_t>(kMaxRows, B - b0));
        const cudaError_t e = launch_after(c, draw_rows_kernel, grid, dim3(kSampleThreads), 0, static_cast<cudaStream_t>(stream), dp);
        c->launches += 1;
        if (!cuda_ok(e, "draw_rows_kernel launch")) return DISCO_ERR_CUDA;
    }
    return DISCO_OK;
}

int disco_verify_sample_ragged(disco_ctx* c, const void* W_T, const void* H_T, const int32_t* draft_ids,
                               const float* draft_probs, const int32_t* row_off, int B, int R,
                               const float* u_accept, const float* u_sample, int32_t* n_accept,
                               int32_t* next_token, float* y_T, int32_t* target_ids, void* stream) {
    if (!c || !W_T || !H_T || !u_sample || !n_accept || !next_token || !y_T) return DISCO_ERR_INVALID_ARG;
    if (B < 1 || R < B) return DISCO_ERR_INVALID_ARG;
    if (R > B && (!draft_ids || !draft_probs || !u_accept)) return DISCO_ERR_INVALID_ARG;
    if (B > c->max_batch || R > c->max_rows) return DISCO_ERR_WORKSPACE;
    if (!row_off && R % B != 0) return DISCO_ERR_INVALID_ARG;
    if (!aligned16(W_T) || !aligned16(H_T)) return DISCO_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // logits and soft-max statistics of all rows by the LM-head pass (which also clears the tickets); one more
    // launch normalises the rows, counts the accepted tokens and draws the next one
    int rc = draft_step_common(c, W_T, H_T, c->d_target, R, c->max_rows, nullptr, nullptr, nullptr, nullptr, 0.f, 1,
                               target_ids, nullptr, nullptr, nullptr, y_T, nullptr, 1, stream, false, nullptr, nullptr,
                               c->sample_tickets, B);
    if (rc) return rc;
    SampleRowsParams sp{};
    sp.y_T = y_T;
    sp.stats = c->final_stats;
    sp.draft_probs = draft_probs;
    sp.draft_ids = draft_ids;
    sp.row_off = row_off;
    sp.u_accept = u_accept;
    sp.u_sample = u_sample;
    sp.B = B;
    sp.SL = row_off ? 0 : (R / B - 1);
    sp.R = R;
    sp.V = c->V;
    // about two CTAs per SM; a row is cut into at most kSampleMaxSegments segments
    sp.SEG = std::max(1, std::min(kSampleMaxSegments, (2 * c->sm_count + R - 1) / R));
    sp.seg_len = ((c->V + sp.SEG - 1) / sp.SEG + 3) & ~3;
    sp.n_accept = n_accept;
    sp.next_token = next_token;
    sp.seg_tot = c->sample_seg_tot;
    sp.seg_last = c->sample_seg_last;
    sp.tickets = c->sample_tickets;
    sp.status = c->status;
    const auto kern = sp.seg_len > kSampleShortWalk ? sample_rows_fused_kernel<true> : sample_rows_fused_kernel<false>;
    const cudaError_t e = launch_after(c, kern, dim3((unsigned)R * sp.SEG), dim3(kSampleThreads), 0, st, sp);
    c->launches += 1;
    return cuda_ok(e, "sample_rows_fused_kernel launch") ? DISCO_OK : DISCO_ERR_CUDA;
}

int disco_extract_features(disco_ctx* c, const void* W_D, const void* H_D, const void* W_T, const void* H_T,
                           const int32_t* pos, int N, float* feats_D, float* feats_T, float* tv, uint8_t* label,
                           int32_t* token_D, int32_t* token_T, float* y_D, float* y_T, void* stream) {
    if (!c || !pos || !feats_D || !feats_T || !tv || !label || !token_D || !token_T || !y_D || !y_T)
        return DISCO_ERR_INVALID_ARG;
    if (N < 1) return DISCO_ERR_INVALID_ARG;
    if (N > c->max_rows) return DISCO_ERR_WORKSPACE;
    // everything both passes will check, before the first of them is enqueued
    if (!W_D || !H_D || !W_T || !H_T) return DISCO_ERR_INVALID_ARG;
    if (!aligned16(W_D) || !aligned16(H_D) || !aligned16(W_T) || !aligned16(H_T)) return DISCO_ERR_INVALID_ARG;
    // the same LM-head pass as a draft step, once per model, without the classifier; y_D and y_T receive the logits
    int rc = draft_step_common(c, W_D, H_D, c->d_draft, N, c->max_rows, pos, nullptr, nullptr, nullptr, 0.f, 1, token_D,
                               nullptr, nullptr, feats_D, y_D, nullptr, 2, stream, false);
    if (rc) return rc;
    rc = draft_step_common(c, W_T, H_T, c->d_target, N, c->max_rows, pos, nullptr, nullptr, nullptr, 0.f, 1, token_T,
                           nullptr, nullptr, feats_T, y_T, nullptr, 2, stream, false, nullptr, nullptr, nullptr, 0,
                           c->final_stats2);
    if (rc) return rc;
    const cudaError_t e = launch_after(c, tv_label_kernel, dim3((unsigned)N), dim3(kFeatThreads), 0, static_cast<cudaStream_t>(stream),
                                       y_D, y_T, (const float*)c->final_stats, (const float*)c->final_stats2,
                                       (const int32_t*)token_D, (const int32_t*)token_T, c->V, tv, label);
    c->launches += 1;
    return cuda_ok(e, "tv_label_kernel launch") ? DISCO_OK : DISCO_ERR_CUDA;
}

int disco_verify_ragged(disco_ctx* c, const void* W_T, const void* H_T, const int32_t* draft_ids,
                        const int32_t* row_off, int B, int R, int32_t* n_accept, int32_t* bonus,
                        int32_t* target_ids, void* stream) {
    if (!c || !W_T || !H_T || !n_accept || !bonus) return DISCO_ERR_INVALID_ARG;
    if (B < 1 || R < B) return DISCO_ERR_INVALID_ARG;
    if (R > B && !draft_ids) return DISCO_ERR_INVALID_ARG;
    return verify_common(c, W_T, H_T, draft_ids, row_off, B, R, row_off ? 0 : (R / B - 1), n_accept, bonus, target_ids,
                         nullptr, stream);
}

int disco_verify(disco_ctx* c, const void* W_T, const void* H_T, const int32_t* draft_ids, int B, int SL,
                 int32_t* n_accept, int32_t* bonus, int32_t* target_ids, void* stream) {
    if (B < 1 || SL < 0) return DISCO_ERR_INVALID_ARG;
    const long long R = (long long)B * (SL + 1);
    if (c && R > c->max_rows) return DISCO_ERR_WORKSPACE;
    return disco_verify_ragged(c, W_T, H_T, draft_ids, nullptr, B, (int)R, n_accept, bonus, target_ids, stream);
}

int disco_draft_loop(disco_ctx* c, const void* W_D, size_t w_step_stride, const void* h_D, int B, const int32_t* pos0,
                     const disco_clf* clf, float tau, int sl_max, const int32_t* sl_forced, int32_t* token,
                     float* conf, uint8_t* halt, float* feats, int32_t* sl, void* stream) {
    if (!c || !W_D || !h_D || !pos0 || !token || !conf || !halt || !sl) return DISCO_ERR_INVALID_ARG;
    if (B < 1 || sl_max < 1) return DISCO_ERR_INVALID_ARG;
    if (!aligned16(W_D) || !aligned16(h_D) || (w_step_stride & 15u)) return DISCO_ERR_INVALID_ARG;
    if (B > c->max_batch) return DISCO_ERR_WORKSPACE;
    int rc = check_clf(c, clf);
    if (rc) return rc;
    const size_t h_step = (size_t)B * c->d_draft * 2;   // bytes of one step's hidden states
    if (h_step & 15u) return DISCO_ERR_INVALID_ARG;
    const int group = steps_per_launch(c, B, sl_max, w_step_stride);
    if (group == 1 && gemv_loop_possible(c, B, sl_max, w_step_stride)) {
        // a handful of sequences: all steps in one persistent kernel
        cudaStream_t st = static_cast<cudaStream_t>(stream);
        c->last_stream = st;
        TailParams p{};
        p.W = static_cast<const uint16_t*>(W_D);
        p.H = static_cast<const uint16_t*>(h_D);
        p.V = c->V;
        p.d = c->d_draft;
        p.R = B;
        p.B = B;
        fill_scratch(c, p);
        p.chain = ChainLink{c->chain_alive, sl, pos0, sl_forced, 1};
        p.clf_W1 = clf->W1;
        p.clf_b1 = clf->b1;
        p.clf_w2 = clf->w2;
        p.clf_b2 = clf->b2;
        p.clf_H = clf->H;
        p.tau = tau;
        p.sl_max = sl_max;
        p.token = token;
        p.conf = conf;
        p.halt = halt;
        p.feats = feats;
        return launch_gemv_loop(c, p, sl_max, w_step_stride, st);
    }
    for (int step = 1; step <= sl_max; step += group) {
        const size_t k = (size_t)(step - 1);
        const int steps = std::min(group, sl_max - step + 1);
        const ChainLink link{c->chain_alive, sl, pos0, sl_forced, step, steps, B};
        rc = draft_step_common(c, static_cast<const char*>(W_D) + k * w_step_stride,
                               static_cast<const char*>(h_D) + k * h_step, c->d_draft, steps * B, c->part_rows, nullptr,
                               nullptr, nullptr, clf, tau, sl_max, token + k * B, conf + k * B, halt + k * B,
                               feats ? feats + k * B * kNFeat : nullptr, nullptr, nullptr, 0, stream, true, nullptr,
                               &link);
        if (rc) return rc;
    }
    return DISCO_OK;
}

int disco_verify_sl(disco_ctx* c, const void* W_T, const void* H_T, const int32_t* draft_ids, long long ids_stride_b,
                    long long ids_stride_j, const int32_t* sl, int B, int sl_max, int32_t* n_accept, int32_t* bonus,
                    int32_t* target_ids, int32_t* row_off, const int32_t* pos0, int32_t* pos_next, void* stream) {
    if (!c || !W_T || !H_T || !sl || !n_accept || !bonus) return DISCO_ERR_INVALID_ARG;
    if (B < 1 || sl_max < 0) return DISCO_ERR_INVALID_ARG;
    if (sl_max > 0 && !draft_ids) return DISCO_ERR_INVALID_ARG;
    if (pos_next && !pos0) return DISCO_ERR_INVALID_ARG;
    const long long R = (long long)B * (sl_max + 1);
    if (R > c->max_rows) return DISCO_ERR_WORKSPACE;
    const VerifyPadded pad{sl, ids_stride_b, ids_stride_j, row_off, pos0, pos_next};
    return verify_common(c, W_T, H_T, draft_ids, nullptr, B, (int)R, sl_max, n_accept, bonus, target_ids, &pad, stream);
}

// late_src (optional): host memory to copy to H_T (late_bytes bytes) on the context's copy stream once the draft
// phase has been enqueued; the verification waits for it.
static int iteration_impl(disco_ctx* c, const void* W_D, size_t w_step_stride, const void* h_D, const void* W_T,
                          const void* H_T, int B, const int32_t* pos0, const disco_clf* clf, float tau, int sl_max,
                          const int32_t* sl_forced, const int32_t* draft_ids, int32_t* token, float* conf, uint8_t* halt,
                          float* feats, int32_t* sl, int32_t* n_accept, int32_t* bonus, int32_t* target_ids,
                          int32_t* row_off, int32_t* pos_next, void* stream, const void* late_src, size_t late_bytes) {
    // everything the second half will check, before the first half is enqueued
    if (!c || !W_T || !H_T || !n_accept || !bonus || !sl) return DISCO_ERR_INVALID_ARG;
    if (!aligned16(W_T) || !aligned16(H_T)) return DISCO_ERR_INVALID_ARG;
    if (B < 1 || sl_max < 1 || (long long)B * (sl_max + 1) > c->max_rows) return B < 1 || sl_max < 1 ? DISCO_ERR_INVALID_ARG : DISCO_ERR_WORKSPACE;
    int rc = disco_draft_loop(c, W_D, w_step_stride, h_D, B, pos0, clf, tau, sl_max, sl_forced, token, conf, halt, feats,
                              sl, stream);
    if (rc) return rc;
    if (late_src &&
        (!cuda_ok(cudaMemcpyAsync(const_cast<void*>(H_T), late_src, late_bytes, cudaMemcpyHostToDevice, c->copy_stream),
                  "cudaMemcpyAsync") ||
         !cuda_ok(cudaEventRecord(c->copy_done, c->copy_stream), "cudaEventRecord") ||
         !cuda_ok(cudaStreamWaitEvent(static_cast<cudaStream_t>(stream), c->copy_done, 0), "cudaStreamWaitEvent")))
        return DISCO_ERR_CUDA;
    if (draft_ids)
        return disco_verify_sl(c, W_T, H_T, draft_ids, sl_max, 1, sl, B, sl_max, n_accept, bonus, target_ids, row_off,
                               pos0, pos_next, stream);
    return disco_verify_sl(c, W_T, H_T, token, 1, B, sl, B, sl_max, n_accept, bonus, target_ids, row_off, pos0,
                           pos_next, stream);
}

int disco_iteration(disco_ctx* c, const void* W_D, size_t w_step_stride, const void* h_D, const void* W_T,
                    const void* H_T, int B, const int32_t* pos0, const disco_clf* clf, float tau, int sl_max,
                    const int32_t* sl_forced, const int32_t* draft_ids, int32_t* token, float* conf, uint8_t* halt,
                    float* feats, int32_t* sl, int32_t* n_accept, int32_t* bonus, int32_t* target_ids,
                    int32_t* row_off, int32_t* pos_next, void* stream) {
    return iteration_impl(c, W_D, w_step_stride, h_D, W_T, H_T, B, pos0, clf, tau, sl_max, sl_forced, draft_ids, token, conf,
                          halt, feats, sl, n_accept, bonus, target_ids, row_off, pos_next, stream, nullptr, 0);
}

int disco_draft_step_host(disco_ctx* c, const void* W_D, const void* h_D_host, int B, const int32_t* pos_host,
                          const int32_t* n_drafted_host, const uint8_t* active_host, const disco_clf* clf,
                          float tau, int sl_max, int32_t* token_host, float* conf_host, uint8_t* halt_host,
                          float* feats_host, void* stream) {
    if (!c || !h_D_host || !pos_host || !n_drafted_host || !token_host || !conf_host || !halt_host)
        return DISCO_ERR_INVALID_ARG;
    if (B < 1) return DISCO_ERR_INVALID_ARG;
    if (B > c->max_batch) return DISCO_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int mb = c->max_batch;
    int32_t* h_pos = c->stage_int_h;
    int32_t* h_nd = h_pos + mb;
    int32_t* h_tok = h_nd + mb;
    float* h_conf = c->stage_float_h;
    float* h_feats = h_conf + mb;
    uint8_t* h_act = c->stage_byte_h;
    uint8_t* h_halt = h_act + mb;
    // host -> device view of the same words
    auto dev_i = [c](int32_t* h) { return c->stage_int_d + (h - c->stage_int_h); };
    auto dev_f = [c](float* h) { return c->stage_float_d + (h - c->stage_float_h); };
    auto dev_b = [c](uint8_t* h) { return c->stage_byte_d + (h - c->stage_byte_h); };
    std::memcpy(h_pos, pos_host, (size_t)B * 4);
    std::memcpy(h_nd, n_drafted_host, (size_t)B * 4);
    if (active_host) std::memcpy(h_act, active_host, (size_t)B);
    if (cudaMemcpyAsync(c->stage_hidden, h_D_host, (size_t)B * c->d_draft * 2, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return DISCO_ERR_CUDA;
    int rc = disco_draft_step(c, W_D, c->stage_hidden, B, dev_i(h_pos), dev_i(h_nd), active_host ? dev_b(h_act) : nullptr,
                              clf, tau, sl_max, dev_i(h_tok), dev_f(h_conf), dev_b(h_halt),
                              feats_host ? dev_f(h_feats) : nullptr, nullptr, stream);
    rc = host_call_done(c, rc, st);
    if (rc) return rc;
    // inactive sequences keep the caller's values: hand back only what the kernel wrote
    for (int b = 0; b < B; ++b) {
        if (active_host && !active_host[b]) continue;
        token_host[b] = h_tok[b];
        conf_host[b] = h_conf[b];
        halt_host[b] = h_halt[b];
        if (feats_host) std::memcpy(feats_host + (size_t)b * kNFeat, h_feats + (size_t)b * kNFeat, kNFeat * 4);
    }
    return DISCO_OK;
}

int disco_verify_ragged_host(disco_ctx* c, const void* W_T, const void* H_T_host, const int32_t* draft_ids_host,
                             const int32_t* row_off_host, int B, int R, int32_t* n_accept_host,
                             int32_t* bonus_host, int32_t* target_ids_host, void* stream) {
    if (!c || !H_T_host || !row_off_host || !n_accept_host || !bonus_host) return DISCO_ERR_INVALID_ARG;
    if (B < 1 || R < B) return DISCO_ERR_INVALID_ARG;
    if (R > B && !draft_ids_host) return DISCO_ERR_INVALID_ARG;
    if (B > c->max_batch || R > c->max_rows) return DISCO_ERR_WORKSPACE;
    // the host can see row_off here, so check it before anything is enqueued
    if (row_off_host[0] != 0 || row_off_host[B] != R) return DISCO_ERR_INVALID_ARG;
    for (int b = 0; b < B; ++b)
        if (row_off_host[b + 1] <= row_off_host[b]) return DISCO_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int mb = c->max_batch, mr = c->max_rows;
    int32_t* h_ids = c->stage_int_h + 3 * (size_t)mb;
    int32_t* h_off = h_ids + mr;
    int32_t* h_nacc = h_off + mb + 1;
    int32_t* h_bonus = h_nacc + mb;
    int32_t* h_tids = h_bonus + mb;
    auto dev_i = [c](int32_t* h) { return c->stage_int_d + (h - c->stage_int_h); };   // device view of the same words
    if (R > B) std::memcpy(h_ids, draft_ids_host, (size_t)(R - B) * 4);
    std::memcpy(h_off, row_off_host, (size_t)(B + 1) * 4);
    if (cudaMemcpyAsync(c->stage_hidden, H_T_host, (size_t)R * c->d_target * 2, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return DISCO_ERR_CUDA;
    int rc = disco_verify_ragged(c, W_T, c->stage_hidden, dev_i(h_ids), dev_i(h_off), B, R, dev_i(h_nacc), dev_i(h_bonus),
                                 target_ids_host ? dev_i(h_tids) : nullptr, stream);
    rc = host_call_done(c, rc, st);
    if (rc) return rc;
    std::memcpy(n_accept_host, h_nacc, (size_t)B * 4);
    std::memcpy(bonus_host, h_bonus, (size_t)B * 4);
    if (target_ids_host) std::memcpy(target_ids_host, h_tids, (size_t)R * 4);
    return DISCO_OK;
}

int disco_iteration_host(disco_ctx* c, const void* W_D, size_t w_step_stride, const void* h_D_host, const void* W_T,
                         const void* H_T_host, int B, const int32_t* pos0_host, const disco_clf* clf, float tau,
                         int sl_max, const int32_t* sl_forced_host, const int32_t* draft_ids_host,
                         int32_t* token_host, float* conf_host, uint8_t* halt_host, int32_t* sl_host,
                         int32_t* n_accept_host, int32_t* bonus_host, int32_t* pos_next_host, void* stream) {
    if (!c || !h_D_host || !H_T_host || !pos0_host || !token_host || !conf_host || !halt_host || !sl_host ||
        !n_accept_host || !bonus_host)
        return DISCO_ERR_INVALID_ARG;
    if (B < 1 || sl_max < 1) return DISCO_ERR_INVALID_ARG;
    const size_t SB = (size_t)sl_max * B, R = (size_t)B * (sl_max + 1);
    if (B > c->max_batch || R > (size_t)c->max_rows) return DISCO_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t mb = (size_t)c->max_batch, mr = (size_t)c->max_rows;
    // pinned, device-mapped staging: pos0 | forced | sl | n_accept | bonus | pos_next (max_batch each), ids | token
    // (max_rows each); conf; halt
    int32_t* h_pos = c->stage_int_h;
    int32_t* h_forced = h_pos + mb;
    int32_t* h_sl = h_forced + mb;
    int32_t* h_nacc = h_sl + mb;
    int32_t* h_bonus = h_nacc + mb;
    int32_t* h_next = h_bonus + mb;
    int32_t* h_ids = h_next + mb;
    int32_t* h_tok = h_ids + mr;
    float* h_conf = c->stage_float_h;
    uint8_t* h_halt = c->stage_byte_h;
    auto dev_i = [c](int32_t* h) { return c->stage_int_d + (h - c->stage_int_h); };
    std::memcpy(h_pos, pos0_host, (size_t)B * 4);
    if (sl_forced_host) std::memcpy(h_forced, sl_forced_host, (size_t)B * 4);
    if (draft_ids_host) std::memcpy(h_ids, draft_ids_host, SB * 4);
    // entries of steps a sequence does not take are not written by the kernels: hand the caller's values back
    std::memcpy(h_tok, token_host, SB * 4);
    std::memcpy(h_conf, conf_host, SB * 4);
    std::memcpy(h_halt, halt_host, SB);
    auto hand_back = [&]() {
        std::memcpy(token_host, h_tok, SB * 4);
        std::memcpy(conf_host, h_conf, SB * 4);
        std::memcpy(halt_host, h_halt, SB);
        std::memcpy(sl_host, h_sl, (size_t)B * 4);
        std::memcpy(n_accept_host, h_nacc, (size_t)B * 4);
        std::memcpy(bonus_host, h_bonus, (size_t)B * 4);
        if (pos_next_host) std::memcpy(pos_next_host, h_next, (size_t)B * 4);
        return (int)DISCO_OK;
    };
    const size_t bytes_D = SB * c->d_draft * 2, bytes_T = R * c->d_target * 2;
    const void *src_D = nullptr, *src_T = nullptr;
    // (not ahead of the persistent draft phase: a cooperative launch starts when all before it has ended, and the engine's second
    // copy runs beside it: 11 rows of 5120 and ten steps of 768 with a head each 141 us, fetched 150)
    const bool fetch = w_step_stride == 0 && bytes_D + bytes_T <= kFetchBytes && (src_D = device_view(c, h_D_host, bytes_D)) != nullptr &&
                       (src_T = device_view(c, H_T_host, bytes_T)) != nullptr;
    if (fetch) {
        // Little to move, all of it pinned: one kernel brings it over, and the draft phase's launch and its first loads of the
        // LM head run meanwhile.
        FetchParams fp{};
        int32_t* dev = c->stage_dev;     // pos0 | forced | ids
        auto part = [&fp](const void* src, void* dst, size_t bytes, unsigned unit) {
            fp.part[fp.n++] = FetchPart{src, dst, (unsigned)(bytes / unit), unit == 16 ? 1u : 0u};
        };
        part(src_D, c->stage_hidden_draft, bytes_D, 16);
        part(src_T, c->stage_hidden, bytes_T, 16);
        part(dev_i(h_pos), dev, (size_t)B * 4, 4);
        if (sl_forced_host) part(dev_i(h_forced), dev + mb, (size_t)B * 4, 4);
        if (draft_ids_host) part(dev_i(h_ids), dev + 2 * mb, SB * 4, 4);
        unsigned pieces = 0;
        for (int i = 0; i < fp.n; ++i) pieces += fp.part[i].pieces;
        cudaError_t e = launch_after(c, fetch_kernel, dim3((pieces + kFetchThreads - 1) / kFetchThreads), dim3(kFetchThreads), 0, st, fp);
        c->launches += 1;
        if (!cuda_ok(e, "fetch_kernel launch")) return DISCO_ERR_CUDA;
        const int rc = iteration_impl(c, W_D, w_step_stride, c->stage_hidden_draft, W_T, c->stage_hidden, B, dev, clf, tau, sl_max,
                                      sl_forced_host ? dev + mb : nullptr, draft_ids_host ? dev + 2 * mb : nullptr,
                                      dev_i(h_tok), c->stage_float_d, c->stage_byte_d, nullptr, dev_i(h_sl), dev_i(h_nacc),
                                      dev_i(h_bonus), nullptr, nullptr, pos_next_host ? dev_i(h_next) : nullptr, stream, nullptr, 0);
        const int end = host_call_done(c, rc, st);
        return end ? end : hand_back();
    }
    // The draft phase needs the draft hidden states only: the (larger) target hidden states are sent once it is
    // enqueued, on a stream of their own, and the verification waits for them.  (Every host entry point returns with its
    // work done, so nothing earlier still reads the staging buffers.)
    if (cudaMemcpyAsync(c->stage_hidden_draft, h_D_host, bytes_D, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return DISCO_ERR_CUDA;
    const int rc = iteration_impl(c, W_D, w_step_stride, c->stage_hidden_draft, W_T, c->stage_hidden, B, dev_i(h_pos), clf, tau,
                            sl_max, sl_forced_host ? dev_i(h_forced) : nullptr, draft_ids_host ? dev_i(h_ids) : nullptr,
                            dev_i(h_tok), c->stage_float_d, c->stage_byte_d, nullptr, dev_i(h_sl), dev_i(h_nacc),
                            dev_i(h_bonus), nullptr, nullptr, pos_next_host ? dev_i(h_next) : nullptr, stream, H_T_host,
                            bytes_T);
    const int end = host_call_done(c, rc, st, true);
    return end ? end : hand_back();
}

}  // extern "C"
