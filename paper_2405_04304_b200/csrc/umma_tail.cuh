// Tensor-core (tcgen05) kernel for greedy verification (two hidden rows and more), and the PTX wrappers that the other
// tensor-core kernels share.
//
//   D[r, v] = sum_k H[r, k] * W[v, k]      r on the 128 TMEM lanes, v on the TMEM columns
//
//   * warp 0   producer: one TMA box of H (A operand, up to 128 rows x 64 k) and one of W (B operand, up
//              to 256 vocabulary rows x 64 k) per stage, 128-byte swizzle, through a ring of
//              shared-memory stages;
//   * warp 1   issues tcgen05.mma (M = 128, N = rows of the vocabulary tile, K = 16 per instruction),
//              accumulating in one of two 256-column TMEM buffers; tcgen05.commit frees the stage;
//   * warps 2+ epilogue: tcgen05.ld 32 columns at a time; every thread owns one hidden row and walks
//              over the vocabulary columns, so the running arg-max lives in its registers: no shuffles,
//              and the logits never leave the chip.  Two warps share each TMEM lane quadrant and
//              split the columns.
//
// With few hidden rows (and some counts just beyond a tile) the operands change places: vocabulary rows on the TMEM lanes,
// hidden rows on the columns, as many as there are in steps of 16.  HBM bounds both forms, but 11 rows on 128 lanes are eight
// times the multiplications that are needed, and a launch that streams HBM for more than some milliseconds runs at the power
// limit: 11 rows, 32000 x 5120 head, one launch after the other: 60.9 us at 1.29 GHz with the hidden rows on the lanes,
// 54.9 us at 1.78 GHz with the vocabulary there (54.2 us either way in a short burst; 51.1 us at the measured copy bandwidth).
//
// A CTA keeps one or two tiles of hidden rows and walks over a contiguous range of vocabulary tiles (VerifyTiling).  CTAs
// that share a vocabulary tile run side by side, so the LM head crosses HBM once and is shared through L2.
// With many rows two CTAs may work as one (cta_group::2, VerifyTiling::make_pairs): the operands' way from L2 is the bound there.
// Results leave the CTA as one atomicMax per row; CTAs of their own finish the job, a warp per sequence, or the last CTA to take
// a ticket, or a small separate kernel (verify_finishers and what follows it in disco_api.cu say which).
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "stream_tail.cuh"  // verify_one_sequence, warp_halt_classifier
#include "group_merge.cuh"

namespace disco {

constexpr int kUmmaMaxStages = 16;
constexpr int kUmmaBK = 64;               // k elements per stage (one 128-byte swizzle span)
constexpr int kUmmaRingBytes = 192 * 1024;  // shared memory for the operand stages
constexpr int kUmmaEpiWarps = 8;
constexpr int kUmmaThreads = (2 + kUmmaEpiWarps) * 32;
constexpr int kUmmaSmemBytes = kUmmaRingBytes + 1024 /*align*/ + 512 /*barriers*/;
constexpr int kUmmaLaneRows = 32;         // hidden rows whose arg-max a thread can hold, with a vocabulary row per lane
constexpr int kUmmaWideRows = 256;        // hidden rows on the columns at most
// ... where an MMA reads whole blocks of 128 vocabulary rows, up to 16 KB past the last stage
constexpr int kUmmaLaneSmemBytes = kUmmaSmemBytes + 16 * 1024;
// shared memory of a staged classifier (draft steps)
inline int umma_clf_bytes(int clf_H) { return (clf_H * (kNFeat + 2) + 4) * 4; }

// How R hidden rows and V vocabulary rows are cut: MT tiles of 128 hidden rows, GS of them (1 or 2) to a CTA; CN CTAs per
// such group share the vocabulary, TPC tiles of TR rows each (MMA width TRN).  The groups of a vocabulary tile run side by
// side: with the whole of H against one vocabulary tile after the other in each CTA, the LM head came from HBM once per
// group (1000 rows, 32000 x 5120 head: 284 us instead of 235).
struct VerifyTiling {
    int MT, GS, groups, CN, TPC, TR, TRN;
    // Every group of tiles needs a CTA: at most two tiles of hidden rows per CTA (37888 rows on 148 SMs).
    __host__ __device__ static bool possible(int R, int grid) { return ((R + 127) / 128 + 1) / 2 <= grid; }
    __host__ __device__ static VerifyTiling make(int R, int V, int d, int grid) {
        VerifyTiling t;
        t.MT = (R + 127) / 128;
        // Two tiles of hidden rows per CTA halve the LM head's traffic from L2 (425 rows, 32000 x 5120 head: 133 -> 120 us;
        // 130 rows, 32000 x 2048: 35 -> 31), but they use both accumulators, so the epilogue does not overlap the next
        // tile's MMAs (1000 rows, 32000 x 768: 39 -> 43), and an odd last tile has its CTAs to itself (300 rows: 105 -> 116).
        // So: two tiles that share every vocabulary tile always; more where the contraction is long and the CTAs' largest
        // share of work grows by at most a twentieth, or where there are more tiles of hidden rows than CTAs.
        const int cn_pairs = grid / ((t.MT + 1) / 2), cn_single = grid / t.MT;
        t.GS = t.MT == 2 || t.MT > grid || (t.MT > 2 && d >= 2048 && cn_pairs * 21 >= cn_single * 40) ? 2 : 1;
        t.groups = (t.MT + t.GS - 1) / t.GS;
        t.CN = grid / t.groups;
        t.TPC = (V + 256 * t.CN - 1) / (256 * t.CN);
        t.TR = (V + t.CN * t.TPC - 1) / (t.CN * t.TPC);
        t.TRN = (t.TR + 15) / 16 * 16;
        return t;
    }
    // Pairs of CTAs (cta_group::2): MT counts tiles of 256 hidden rows, GS of them (1 or 2) to a pair, CN pairs per group.  Of
    // the two the cheaper one by the longer of tensor time and operand traffic (cycles per 64 k; an SM takes in about 61 bytes
    // a cycle), and by the epilogue that GS = 2 does not hide.
    __host__ __device__ static bool pairs_possible(int R, int grid) { return (R + 511) / 512 <= grid / 2; }
    __host__ __device__ static VerifyTiling make_pairs(int R, int V, int d, int grid) {
        VerifyTiling best{};
        long long least = 0;
        const int KB = (d + 63) / 64;
        for (int gs = 1; gs <= 2; ++gs) {
            VerifyTiling t;
            t.MT = (R + 255) / 256;
            t.GS = gs;
            t.groups = (t.MT + gs - 1) / gs;
            t.CN = grid / 2 / t.groups;
            if (t.CN == 0) continue;
            t.TPC = (V + 256 * t.CN - 1) / (256 * t.CN);
            t.TR = (V + t.CN * t.TPC - 1) / (t.CN * t.TPC);
            t.TRN = (t.TR + 15) / 16 * 16;
            const int size = gs < t.MT ? gs : t.MT;
            const int mma = 2 * t.TRN * size, feed = (size * 128 + t.TRN / 2) * 21 / 10;
            const long long cost = (long long)t.TPC * ((long long)KB * (mma > feed ? mma : feed) + (size == 2 ? 1500 : 0));
            if (best.CN == 0 || cost < least) best = t, least = cost;
        }
        return best;
    }
    // Whether pairs are the faster form (us under continuous load, single CTAs -> pairs; few launches in a row differ by as much).
    // They halve the LM head's traffic from L2, but cut the rows into tiles of 256: a CTA's share of the tensor work may not grow by
    // more than a few hundredths.  Then
    //   * a pair with one tile of rows, whose epilogue runs under the next vocabulary tile, beats CTAs with two (32000 x 1024 / 2048 /
    //     5120, 251 rows 23.2 / 39.3 / 95 -> 20.4 / 34.1 / 88; x 2048 / 5120, 650 rows 87 / 202 -> 79 / 193; 4000 x 5120, 512 rows 35.2 ->
    //     24.8), and CTAs with one where it has three vocabulary tiles to gain on (32000 x 1024, 650 / 974 / 2432 rows 47.1 / 59.2 / 133
    //     -> 43.4 / 56.5 / 127, but 8000 x 1024, 512 rows 10.9 -> 12.0);
    //   * a pair with two has its epilogue exposed like a CTA with two, and waits for more (32000 x 2048 / 5120, 1520 rows 156 / 364 -> 162 /
    //     371; against CTAs with one: 49152 x 1024, 428 rows 45.4 -> 49.6, 8000 x 1024, 2432 rows 33.4 -> 39.9).  It pays on a short head
    //     of a long contraction only (4000 / 8000 x 5120, 1520 rows 57 / 109 -> 54 / 105, 4000 x 6144, 2432 rows 113 -> 102).
    __host__ __device__ static bool in_pairs(int R, int V, int d, int grid) {
        if (d < 1024 || R <= 128 || !pairs_possible(R, grid)) return false;
        const VerifyTiling one = make(R, V, d, grid), two = make_pairs(R, V, d, grid);
        auto share = [](const VerifyTiling& t) { return (long long)t.TPC * t.TRN * (t.GS < t.MT ? t.GS : t.MT); };
        if (32 * share(two) > 33 * share(one)) return false;
        return two.GS == 1 ? one.GS == 2 || two.TPC >= 3 : d >= 4096 && V <= 8192 && two.TPC <= 2;
    }
};

struct UmmaParams {
    int V, d, R;
    VerifyTiling t;
    int box_rows;  // rows of the LM-head box
    int a_rows;    // rows of the H box (multiple of 8, <= 128)
    int stages;    // ring depth (<= kUmmaMaxStages); stage s holds one or two A tiles of a_bytes and a B tile of b_bytes
    int a_bytes, b_bytes;  // multiples of 1024
    int a_tiles;   // A tiles a stage has room for
    int* status;
    unsigned long long* keys;  // [R]
    // verification finished inside this kernel by the last CTA (few sequences only)
    int fuse_final;
    unsigned int* ticket;
    int finishers;         // with fuse_final: the grid's last CTAs finish eight sequences each and have no vocabulary of their own
    const int32_t* draft_ids;
    const int32_t* row_off;
    int B, SL;
    int32_t* n_accept;
    int32_t* bonus;
    int32_t* target_ids;
    VerifyPadded padded;   // sl != null: fixed-shape rows, per-sequence look-ahead read from the device
    // Verification whose row count is device memory (rows packed by the kernel before this one): R is then an upper bound,
    // the kernel derives the tiling from *dev_R, and the LM-head box is 256 rows high.
    const int32_t* dev_R;
};

// ---------------------------------------------------------------------------------------------
// PTX wrappers
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void tma_load_2d(uint32_t dst_smem, const CUtensorMap* tmap, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst_smem),
        "l"(tmap), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst_smem, const CUtensorMap* tmap, int c0, int c1, uint64_t* bar) {
    tma_load_2d(smem_addr(dst_smem), tmap, c0, c1, smem_addr(bar));
}
// Bring one box of a tensor map into L2 (no shared-memory destination, nothing to wait for).
__device__ __forceinline__ void tma_prefetch_l2_2d(const CUtensorMap* tmap, int c0, int c1) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(tmap), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* tmap) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst_smem)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) { tc_commit(smem_addr(bar)); }
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// ---- two CTAs of a cluster as one (cta_group::2): 256 rows of the A operand, 128 in each CTA, and a B operand of which each
// CTA holds half; the even CTA (the leader) issues the MMAs for both ----
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// The leader's word at the place of this CTA's one.
__device__ __forceinline__ uint32_t leader_addr(uint32_t smem) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(smem));
    return a;
}
__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// A load into this CTA's shared memory that is counted on the leader's barrier.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst_smem, const CUtensorMap* tmap, int c0, int c1, uint32_t leader_bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst_smem),
        "l"(tmap), "r"(c0), "r"(c1), "r"(leader_bar)
        : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst_smem)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// Arrives at the barrier of this address in both CTAs once the MMAs issued so far are done.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
                 "h"(static_cast<uint16_t>(3))
                 : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                 uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// 32 lanes x 32 consecutive fp32 columns -> 32 registers per thread (the wait names the registers, so that the compiler
// moves nothing that looks at them ahead of it)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                   "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])::"memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// The largest of a warp's numbers, in one instruction.
__device__ __forceinline__ float warp_max_f32(float x) {
    float m;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
    return m;
}

// Shared-memory matrix descriptor: K-major tile, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t umma_smem_desc(const void* tile) {
    uint64_t desc = 0;
    desc |= static_cast<uint64_t>((smem_addr(tile) & 0x3ffffu) >> 4);  // start address
    desc |= static_cast<uint64_t>(1) << 16;                            // leading byte offset (unused with swizzle)
    desc |= static_cast<uint64_t>(1024 >> 4) << 32;                    // stride byte offset
    desc |= static_cast<uint64_t>(1) << 46;                            // descriptor version
    desc |= static_cast<uint64_t>(2) << 61;                            // 128-byte swizzle
    return desc;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = m (256 for a pair of CTAs), N = n.
__device__ __forceinline__ uint32_t umma_idesc(int n, uint32_t m = 128) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | ((m >> 4) << 24);
}

// Draft step, second phase: one warp per sequence merges the per-CTA partial records, forms the
// features of Eq. 2 and runs the halt classifier and the stopping rule.
struct DraftFinalParams {
    int B;
    const int32_t* pos;
    const int32_t* n_drafted;
    const uint8_t* active;
    const float* clf_W1;
    const float* clf_b1;
    const float* clf_w2;
    const float* clf_b2;
    int clf_H;
    float tau;
    int sl_max;
    int32_t* token;
    float* conf;
    uint8_t* halt;
    float* feats;
    float* final_stats;
    float* nll_sum;
    int stats_only;
    ChainLink chain;      // alive != null: this launch is one step of a draft phase chained on the device
    unsigned int test_stamp_skew;   // 0.  Tests: the finishing warps expect a stamp that no CTA writes, so their wait runs out
    // words that the kernel after this one counts in (the tickets of a verification with sampling): cleared here
    unsigned int* clear_words;
    int clear_n;
};

// Vocabulary tile t covers rows [t * TR, min(V, (t + 1) * TR)).  The TMA box and the MMA take TRN >= TR
// rows; the extra rows (the next tile's first rows, or zero fill past V) land in columns the epilogue skips.
// ---------------------------------------------------------------------------------------------
// main kernel
// ---------------------------------------------------------------------------------------------
// VL: vocabulary rows on the TMEM lanes (A operand, two blocks of 128 per tile), at most kUmmaLaneRows hidden rows, which all
// CTAs read as one B operand of 16 or 32 rows.
// WIDE: the same with up to kUmmaWideRows hidden rows; the warp finds the largest logit of a column at once, and the running
// keys live in shared memory.  130 rows, 32000 x 2048: 36.2 -> 32.3 us; 20.5 us at the measured copy bandwidth.
// PAIR: clusters of two CTAs with 256 hidden rows to a tile (VerifyTiling::make_pairs): each loads its own 128 hidden rows and half
// of the LM-head box, the even one issues the MMAs of both.
// FIN: the grid's last p.finishers CTAs finish the sequences (an instance of its own: the code behind the last load comes from memory
// line by line when another kernel ran before, and a verification behind its draft phase lost 3 us to code that it did not use).
template <bool VL, bool WIDE, bool PAIR, bool FIN>
__global__ void __launch_bounds__(kUmmaThreads, 1)
umma_tail_kernel(const __grid_constant__ CUtensorMap tmap_W, const __grid_constant__ CUtensorMap tmap_H,
                 const UmmaParams p) {
    extern __shared__ uint8_t smem_dyn[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
    uint8_t* a_tiles = smem;
    uint8_t* b_tiles = smem + p.stages * p.a_bytes * p.a_tiles;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kUmmaRingBytes);
    uint64_t* empty = full + kUmmaMaxStages;
    uint64_t* tmem_full = empty + kUmmaMaxStages;
    uint64_t* tmem_empty = tmem_full + 2;
    uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(tmem_empty + 2);

    // the next kernel of the stream may begin its prologue; this one touches what its predecessor may
    // have written (hidden states, scratch) only after griddepcontrol.wait
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int KB = (p.d + kUmmaBK - 1) / kUmmaBK;
    // tiling: from the host, or (row count in device memory) derived here by the same rule
    int R = p.R;
    VerifyTiling tl = p.t;
    if (p.dev_R) {
        asm volatile("griddepcontrol.wait;" ::: "memory");   // the count is the predecessor's output
        R = min(max(__ldcg(p.dev_R), 1), p.R);
        tl = PAIR ? VerifyTiling::make_pairs(R, p.V, p.d, (int)gridDim.x) : VerifyTiling::make(R, p.V, p.d, (int)gridDim.x);
    }
    const int rank = PAIR ? (int)cluster_rank() : 0;
    const bool leader = rank == 0;
    const int cta = PAIR ? (int)blockIdx.x >> 1 : (int)blockIdx.x;      // (or pair of CTAs)
    // this CTA: `size` tiles of hidden rows from m_tile on, vocabulary rows v_begin .. v_end - 1 in tiles of TR
    const int m_tile = cta % tl.groups * tl.GS;
    const int size = VL ? 1 : min(tl.GS, tl.MT - m_tile);
    const int slot = cta / tl.groups;
    constexpr int kTileStep = PAIR ? 256 : 128;
    const int h_row = m_tile * kTileStep + rank * 128;                  // the first hidden row of this CTA; its second tile: kTileStep on
    const int v_begin = slot * tl.TPC * tl.TR;
    const int v_end = min(p.V, v_begin + tl.TPC * tl.TR);

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tmem_full[b], 1);
            mbar_init(&tmem_empty[b], PAIR ? 2 * kUmmaEpiWarps : kUmmaEpiWarps);
        }
        fence_mbar_init();
        prefetch_tensormap(&tmap_W);
        prefetch_tensormap(&tmap_H);
    }
    if (warp == 1) {
        if constexpr (PAIR) {
            tmem_alloc_pair(tmem_base_s, 512);
        } else {
            tmem_alloc(tmem_base_s, 512);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    if constexpr (PAIR) cluster_sync();
    else __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_base_s;

    // (VL) columns of a block of 128 vocabulary rows; two blocks per tile, one or two tiles in TMEM
    const int lane_cols = WIDE ? (p.a_rows + 31) & ~31 : kUmmaLaneRows;
    const int lane_bufs = lane_cols <= 128 ? 2 : 1;
    const bool live = slot < tl.CN;   // (CTAs beyond the tiling have nothing to do)

    if (warp == 0) {
        // ------------------------------ producer ------------------------------
        if (live && elect_one()) {
            // A single thread: running addresses and counters, as few instructions per stage as possible.
            const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty), a0 = smem_addr(a_tiles), b0 = smem_addr(b_tiles);
            const uint32_t a_box = (uint32_t)p.a_rows * 128u, w_box = (uint32_t)p.box_rows * 128u;   // bytes of the two boxes
            const uint32_t a_step = (uint32_t)p.a_bytes * p.a_tiles;
            const int k_end = KB * kUmmaBK;
            // (a pair's loads are counted on the leader's barriers)
            const uint32_t count0 = PAIR ? leader_addr(full0) : full0, expected = (PAIR ? 2 : 1) * (w_box + size * a_box);
            const int v_half = PAIR ? rank * (tl.TRN / 2) : 0;
            auto load = [&](uint32_t dst, const CUtensorMap* map, int c0, int c1, int slot) {
                if constexpr (PAIR) tma_load_2d_pair(dst, map, c0, c1, count0 + slot * 8);
                else tma_load_2d(dst, map, c0, c1, count0 + slot * 8);
            };
            // The LM head is never written by this library: its first tiles are requested before the
            // dependency wait, the hidden-state tiles of the same stages right after it.
            int v0 = v_begin;
            const int pre = v0 < v_end ? min(p.stages, KB) : 0;
            for (int n = 0; n < pre; ++n) {
                if (leader) mbar_arrive_expect_tx(full0 + n * 8, expected);
                load(b0 + n * p.b_bytes, &tmap_W, n * kUmmaBK, v0 + v_half, n);
            }
            asm volatile("griddepcontrol.wait;" ::: "memory");
            for (int n = 0; n < pre; ++n) {
                load(a0 + n * a_step, &tmap_H, n * kUmmaBK, h_row, n);
                if (size == 2) load(a0 + n * a_step + p.a_bytes, &tmap_H, n * kUmmaBK, h_row + kTileStep, n);
            }
            int stage = pre == p.stages ? 0 : pre, phase = pre == p.stages ? 1 : 0;
            int k = pre * kUmmaBK;
            uint32_t at_a = a0 + stage * a_step, at_b = b0 + stage * p.b_bytes;
            for (; v0 < v_end; v0 += tl.TR, k = 0) {
                for (; k < k_end; k += kUmmaBK) {
                    mbar_wait(empty0 + stage * 8, phase ^ 1, p.status);
                    if (leader) mbar_arrive_expect_tx(full0 + stage * 8, expected);
                    load(at_b, &tmap_W, k, v0 + v_half, stage);
                    load(at_a, &tmap_H, k, h_row, stage);
                    if (size == 2) load(at_a + p.a_bytes, &tmap_H, k, h_row + kTileStep, stage);
                    at_a += a_step;
                    at_b += p.b_bytes;
                    if (++stage == p.stages) {
                        stage = 0;
                        phase ^= 1;
                        at_a = a0;
                        at_b = b0;
                    }
                }
            }
            if constexpr (PAIR) {   // the leader's arrivals at this CTA's barriers are all in before it leaves
                for (int n = 0; n < p.stages; ++n) {
                    mbar_wait(empty0 + stage * 8, phase ^ 1, p.status);
                    if (++stage == p.stages) stage = 0, phase ^= 1;
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        if (live && leader && elect_one()) {
            const uint32_t idesc = umma_idesc(VL ? p.a_rows : tl.TRN, PAIR ? 256 : 128);
            auto mma = [&](uint32_t d, uint64_t a, uint64_t b, uint32_t accumulate) {
                if constexpr (PAIR) tc_mma_bf16_pair(d, a, b, idesc, accumulate);
                else tc_mma_bf16(d, a, b, idesc, accumulate);
            };
            auto commit = [&](uint32_t bar) {
                if constexpr (PAIR) tc_commit_pair(bar);
                else tc_commit(bar);
            };
            const bool upper = tl.TRN > 128;   // (VL)
            const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty);
            const uint64_t a0 = umma_smem_desc(a_tiles), b0 = umma_smem_desc(b_tiles);
            const uint32_t a_half = (uint32_t)p.a_bytes >> 4, a_step = a_half * p.a_tiles, b_step = (uint32_t)p.b_bytes >> 4;   // descriptor units
            uint64_t a_desc = a0, b_desc = b0;
            int stage = 0, phase = 0;
            // Two tiles of hidden rows use an accumulator each, one alternates between the two.
            int it = 0;
            for (int v0 = v_begin; v0 < v_end; v0 += tl.TR, ++it) {
                const bool alternate = VL ? lane_bufs == 2 : size == 1;
                const int first = alternate ? it & 1 : 0;
                const uint32_t parity = (alternate ? it >> 1 : it) & 1;
                for (int j = 0; j < size; ++j) {
                    if constexpr (PAIR) mbar_wait_cluster(smem_addr(&tmem_empty[first + j]), parity ^ 1u, p.status);
                    else mbar_wait(&tmem_empty[first + j], parity ^ 1u, p.status);
                }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + first * (VL ? 2 * lane_cols : 256);
                for (int kb = 0; kb < KB; ++kb) {
                    mbar_wait(full0 + stage * 8, phase, p.status);
                    tc_fence_after();
                    if constexpr (VL) {
#pragma unroll
                        for (int k = 0; k < kUmmaBK / 16; ++k)
                            tc_mma_bf16(d_tmem, b_desc + 2 * k, a_desc + 2 * k, idesc, (kb | k) != 0);
                        if (upper) {
#pragma unroll
                            for (int k = 0; k < kUmmaBK / 16; ++k)   // 128 rows further on
                                tc_mma_bf16(d_tmem + lane_cols, b_desc + (128 * 128 >> 4) + 2 * k, a_desc + 2 * k, idesc, (kb | k) != 0);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < kUmmaBK / 16; ++k)  // 16 k-elements = 32 bytes = 2 descriptor units
                            mma(d_tmem, a_desc + 2 * k, b_desc + 2 * k, (kb | k) != 0);
                    }
                    if (!VL && size == 2) {
#pragma unroll
                        for (int k = 0; k < kUmmaBK / 16; ++k)
                            mma(d_tmem + 256, a_desc + a_half + 2 * k, b_desc + 2 * k, (kb | k) != 0);
                    }
                    commit(empty0 + stage * 8);
                    a_desc += a_step;
                    b_desc += b_step;
                    if (++stage == p.stages) {
                        stage = 0;
                        phase ^= 1;
                        a_desc = a0;
                        b_desc = b0;
                    }
                }
                for (int j = 0; j < size; ++j) commit(smem_addr(&tmem_full[first + j]));
            }
        }
    } else if (live) {
        // ------------------------------ epilogue ------------------------------
        asm volatile("griddepcontrol.wait;" ::: "memory");  // scratch and outputs belong to the predecessor until now
        const int ew = warp - 2;            // 0 .. kUmmaEpiWarps-1
        const int quad = warp & 3;          // TMEM lane quadrant this warp may read
        const int share = ew >> 2;          // two warps per quadrant split the columns of a tile
        if constexpr (VL && WIDE) {
            // a lane holds one vocabulary row of the tile, a column is a hidden row; the warp's keys are behind the barriers,
            // where MMAs may read (lanes nobody looks at) but nothing is loaded to
            constexpr int kEpiThreads = kUmmaEpiWarps * 32;
            unsigned long long* keys_s = reinterpret_cast<unsigned long long*>(smem + kUmmaRingBytes + 512);
            unsigned long long* mine = keys_s + ew * kUmmaWideRows + lane;
            for (int c = 0; c < lane_cols; c += 32) mine[c] = 0ull;
            const int block_row = share * 128 + quad * 32;
            int it = 0;
            for (int v0 = v_begin; v0 < v_end; v0 += tl.TR, ++it) {
                const int b = lane_bufs == 2 ? it & 1 : 0;
                const int ncols = min(tl.TR, v_end - v0);
                mbar_wait(&tmem_full[b], (lane_bufs == 2 ? it >> 1 : it) & 1, p.status);
                tc_fence_after();
                if (block_row < ncols) {
                    const bool in = block_row + lane < ncols;
#pragma unroll 1
                    for (int c = 0; c < lane_cols; c += 32) {
                        float z[32];
                        tmem_ld32(tmem_base + (2 * b + share) * lane_cols + c + (static_cast<uint32_t>(quad * 32) << 16), z);
                        float top = DISCO_NEG_INF;      // lane i: the largest logit of column i and the lanes that hold it
                        unsigned int who = 0u;
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            const float x = in ? z[i] : DISCO_NEG_INF;
                            const float m = warp_max_f32(x);
                            const unsigned int at = __ballot_sync(kFullMask, x == m);
                            if (lane == i) top = m, who = at;
                        }
                        if (top > DISCO_NEG_INF) {
                            const unsigned long long key = argmax_key(__fadd_rn(top, 0.f), v0 + block_row + __ffs(who) - 1);
                            if (key > mine[c]) mine[c] = key;
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tmem_empty[b]);
            }
            named_barrier_sync(2, kEpiThreads);
            const int r = ew * 32 + lane;               // one result per hidden row and CTA
            if (r < R) {
                unsigned long long key = 0ull;
#pragma unroll
                for (int w = 0; w < kUmmaEpiWarps; ++w) key = max(key, keys_s[w * kUmmaWideRows + r]);
                if (key) atomicMax(p.keys + r, key);
            }
        } else if constexpr (VL) {
            // a thread holds one vocabulary row of the tile, a column is a hidden row
            float best_v[kUmmaLaneRows];
            int best_i[kUmmaLaneRows];
#pragma unroll
            for (int r = 0; r < kUmmaLaneRows; ++r) best_v[r] = DISCO_NEG_INF, best_i[r] = kNoIndex;
            const int tile_row = share * 128 + quad * 32 + lane;
            int it = 0;
            for (int v0 = v_begin; v0 < v_end; v0 += tl.TR, ++it) {
                const int b = it & 1;
                const int ncols = min(tl.TR, v_end - v0);
                mbar_wait(&tmem_full[b], (it >> 1) & 1, p.status);
                tc_fence_after();
                if (share * 128 + quad * 32 < ncols) {
                    float z[32];
                    tmem_ld32(tmem_base + (2 * b + share) * kUmmaLaneRows + (static_cast<uint32_t>(quad * 32) << 16), z);
                    if (tile_row < ncols) {
#pragma unroll
                        for (int r = 0; r < kUmmaLaneRows; ++r)
                            if (z[r] > best_v[r]) best_v[r] = z[r], best_i[r] = v0 + tile_row;
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tmem_empty[b]);
            }
            // one result per hidden row and CTA: the keys of a row side by side in the ring (every load has landed and every MMA
            // is done), a warp per row.  (32 folds in registers one after the other are 13 KB of code that comes from L2 in an
            // iteration: 2 us.)
            unsigned long long* keys_s = reinterpret_cast<unsigned long long*>(smem);
            constexpr int kEpiThreads = kUmmaEpiWarps * 32;
#pragma unroll
            for (int r = 0; r < kUmmaLaneRows; ++r)
                if (r < R) keys_s[r * kEpiThreads + ew * 32 + lane] = best_i[r] != kNoIndex ? argmax_key(__fadd_rn(best_v[r], 0.f), best_i[r]) : 0ull;
            named_barrier_sync(2, kEpiThreads);
#pragma unroll 1
            for (int r = ew; r < R; r += kUmmaEpiWarps) {
                unsigned long long key = 0ull;
#pragma unroll
                for (int i = 0; i < kUmmaEpiWarps; ++i) key = max(key, keys_s[r * kEpiThreads + i * 32 + lane]);
                const uint32_t hi = static_cast<uint32_t>(key >> 32);
                const uint32_t top = __reduce_max_sync(kFullMask, hi);
                const uint32_t low = __reduce_max_sync(kFullMask, hi == top ? static_cast<uint32_t>(key) : 0u);
                if (lane == 0 && top) atomicMax(p.keys + r, static_cast<unsigned long long>(top) << 32 | low);
            }
        } else {
            float best_v[2] = {DISCO_NEG_INF, DISCO_NEG_INF};
            int best_i[2] = {kNoIndex, kNoIndex};
            int it = 0;
            for (int v0 = v_begin; v0 < v_end; v0 += tl.TR, ++it) {
                const int ncols = min(tl.TR, v_end - v0);  // further columns belong to the next tile or lie past V
                const int nchunks = (ncols + 31) >> 5;
                const int c_lo = (nchunks * share + 1) / 2, c_hi = (nchunks * (share + 1) + 1) / 2;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (j >= size) break;
                    const int b = size == 2 ? j : it & 1;
                    mbar_wait(&tmem_full[b], (size == 2 ? it : it >> 1) & 1, p.status);
                    tc_fence_after();
                    if (h_row + j * kTileStep + quad * 32 < R) {
                        for (int c = c_lo; c < c_hi; ++c) {
                            float z[32];
                            tmem_ld32(tmem_base + b * 256 + c * 32 + (static_cast<uint32_t>(quad * 32) << 16), z);
                            const int n = ncols - c * 32;
                            if (n < 32) {
#pragma unroll
                                for (int i = 0; i < 32; ++i)
                                    if (i >= n) z[i] = DISCO_NEG_INF;
                            }
                            float cmax = fmaxf(z[0], z[1]);
#pragma unroll
                            for (int i = 2; i < 32; i += 2) cmax = RegTop10::max3(cmax, z[i], z[i + 1]);
                            // (a chunk seldom holds a new largest logit: its index is looked for only then)
                            if (__any_sync(kFullMask, cmax > best_v[j])) {
                                int at = 0;
#pragma unroll
                                for (int i = 31; i >= 0; --i)
                                    if (z[i] == cmax) at = i;
                                if (cmax > best_v[j]) {
                                    best_v[j] = cmax;
                                    best_i[j] = v0 + c * 32 + at;
                                }
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (PAIR) mbar_arrive_cluster(leader_addr(smem_addr(&tmem_empty[b])));
                        else mbar_arrive(&tmem_empty[b]);
                    }
                }
            }
            // one result per hidden row and CTA
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int row = h_row + j * kTileStep + quad * 32 + lane;
                if (j < size && row < R && best_i[j] != kNoIndex)
                    atomicMax(p.keys + row, argmax_key(__fadd_rn(best_v[j], 0.f), best_i[j]));
            }
        }
        if constexpr (FIN) {
            __threadfence();
            named_barrier_sync(2, kUmmaEpiWarps * 32);
            if (ew == 0 && lane == 0) atomicAdd(p.ticket, 1u);
        } else if (p.fuse_final) {
            // ticket: the last CTA to get here matches the prefixes and clears the keys
            __shared__ int s_last;
            __threadfence();
            named_barrier_sync(2, kUmmaEpiWarps * 32);
            if (ew == 0 && lane == 0) s_last = atomicAdd(p.ticket, 1u) == (unsigned)(tl.groups * tl.CN * (PAIR ? 2 : 1)) - 1u;   // CTAs beyond the tiling take none
            named_barrier_sync(2, kUmmaEpiWarps * 32);
            if (s_last) {
                __threadfence();
                for (int b = ew; b < p.B; b += kUmmaEpiWarps)
                    verify_one_sequence(p.keys, p.draft_ids, p.row_off, p.B, p.SL, R, b, p.n_accept, p.bonus,
                                        p.target_ids, p.status, lane, p.padded);
                if (ew == 0) warp_write_row_offsets(p.padded, p.B, p.SL, lane);
                named_barrier_sync(2, kUmmaEpiWarps * 32);
                for (int r = ew * 32 + lane; r < p.R; r += kUmmaEpiWarps * 32) p.keys[r] = 0ull;
                if (ew == 0 && lane == 0) *p.ticket = 0u;
            }
        }
    } else if constexpr (FIN) {
        // ------------------------------ finishers ------------------------------
        // What does not depend on the keys is read while the others work; then the CTAs that are done are counted.  The others
        // leave at once, so the next launch sets itself up on their SMs meanwhile.  (Blocks start in order, so these CTAs are
        // the last ones; should one start after them, it has an SM of its own to wait for.)
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const int ew = warp - 2, first = (int)gridDim.x - p.finishers;
        const int b0 = ((int)blockIdx.x - first) * kUmmaEpiWarps + ew;
        VerifySeq q{};
        if (b0 < p.B) q = verify_locate(p.draft_ids, p.row_off, p.B, p.SL, R, b0, lane, p.padded);
        if (lane == 0) {
            const long long t0 = clock64();
            for (int polls = 0; ld_relaxed_u32(p.ticket) != (unsigned)first; ++polls) {
                __nanosleep(40);
                if ((polls & 255) == 255 && (*reinterpret_cast<volatile int*>(p.status) == DISCO_ERR_TIMEOUT ||
                                             clock64() - t0 > 64 * kWaitBudgetClocks)) {
                    record_status(p.status, DISCO_ERR_TIMEOUT);
                    break;
                }
            }
            __threadfence();
        }
        __syncwarp();
        if (b0 < p.B) verify_match(q, p.keys, p.draft_ids, b0, p.n_accept, p.bonus, p.target_ids, p.status, lane, p.padded);
        // the last of these CTAs leaves the keys and the counters at zero
        __shared__ int s_clear;
        named_barrier_sync(2, kUmmaEpiWarps * 32);
        if (ew == 0 && lane == 0) s_clear = p.finishers == 1 || atomicAdd(p.ticket + 1, 1u) == (unsigned)p.finishers - 1u;
        named_barrier_sync(2, kUmmaEpiWarps * 32);
        if (s_clear) {
            for (int r = ew * 32 + lane; r < p.R; r += kUmmaEpiWarps * 32) p.keys[r] = 0ull;
            if (ew == 0 && lane == 0) p.ticket[0] = p.ticket[1] = 0u;
        }
    }

    tc_fence_before();
    if constexpr (PAIR) cluster_sync();    // (neither CTA of a pair leaves before the other)
    else __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        if constexpr (PAIR) tmem_dealloc_pair(tmem_base, 512);
        else tmem_dealloc(tmem_base, 512);
    }
}

// ---------------------------------------------------------------------------------------------
// finishing kernels
// ---------------------------------------------------------------------------------------------

// Verification: one warp per sequence decodes the arg-max keys, matches the prefix and picks the
// bonus token.  The last CTA to finish clears the keys for the next call.
struct VerifyFinalParams {
    unsigned long long* keys;
    const int32_t* draft_ids;
    const int32_t* row_off;
    int B, SL, R;
    int32_t* n_accept;
    int32_t* bonus;
    int32_t* target_ids;
    int* status;
    unsigned int* ticket;
    VerifyPadded padded;
    const int32_t* dev_R;   // non-null: the row count is device memory (R is then the upper bound)
};

__global__ void __launch_bounds__(128) verify_finalize_kernel(const VerifyFinalParams p) {
    __shared__ int s_last;
    // launched with programmatic stream serialization: resident early, reading only once its predecessor has completed
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.x * (blockDim.x >> 5) + warp;
    const int R = p.dev_R ? min(max(__ldcg(p.dev_R), 1), p.R) : p.R;
    if (b < p.B)
        verify_one_sequence(p.keys, p.draft_ids, p.row_off, p.B, p.SL, R, b, p.n_accept, p.bonus, p.target_ids,
                            p.status, lane, p.padded);
    if (blockIdx.x == gridDim.x - 1 && warp == (blockDim.x >> 5) - 1) warp_write_row_offsets(p.padded, p.B, p.SL, lane);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int r = threadIdx.x; r < p.R; r += blockDim.x) p.keys[r] = 0ull;  // every reader is done
    if (threadIdx.x == 0) *p.ticket = 0u;
}

}  // namespace disco
