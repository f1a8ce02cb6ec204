// The draft phase of an iteration as ONE persistent kernel, for a handful of sequences (1..4): up to
// sl_max draft steps (Sec. 3: after every draft token the classifier decides whether the next one is
// drafted) without leaving the GPU and without a launch per step.
//
// Each step is a tensor-core GEMV with the vocabulary on the TMEM lanes: the A operand is 128 rows of the LM head, the B
// operand the hidden rows (N = 16), D[v, r].  An MMA of that shape takes 39 cycles against 112 of one with the hidden rows
// on the lanes and 224 vocabulary rows on the columns, and its accumulator has one vocabulary row per thread, which is
// what the fold wants.  What the loop adds:
//   * one CTA per SM stays resident for all steps (cooperative launch: the steps hand over through global
//     memory, so every CTA must be running);
//   * the producer never stops: as soon as the MMAs of step i have released a ring stage it is refilled
//     with the LM head's tiles for step i + 1, while the CTA folds, publishes its record, and the step is
//     decided.  The hidden rows of step i + 1, an input of the call like all others, follow as soon as the MMAs of step i
//     are done with theirs;
//   * the B operand is the one 8-row box of hidden rows read twice over (zero stride between the 8-row groups of the
//     descriptor), so nothing outside it is read;
//   * every warp folds its 32 logits of a hidden row (statistics, arg-max, a descending list of ten); one barrier later a
//     group of warps per sequence ranks the lists' entries that can be among the CTA's ten largest while another of its
//     warps adds up the statistics, and the CTA's record is published in stamped 16-byte pieces: no fence and no counter
//     between the writer and its reader;
//   * CTA 0 finishes the sequences with all eight epilogue warps (group_merge_partials polls the records
//     of the step until all carry its stamp), records which sequences go on, and publishes the decision
//     "continue / stop" in a stamped word that every CTA polls (bounded);
//   * tiles requested ahead for a step that does not take place are awaited before the CTA leaves.
// Every one of these phases is a chain of dependent instructions on a few warps, so the code is written for
// short chains (values through shared memory and independent comparisons instead of shuffle chains, loads
// of a batch in flight before the first use), not for few instructions.
#pragma once

#include "umma_tail.cuh"

namespace disco {

constexpr int kGemvEpiWarps = 8;
constexpr int kGemvThreads = (3 + kGemvEpiWarps) * 32;   // producer, two MMA issuers, epilogue
constexpr int kGemvMaxStages = 16;
constexpr int kGemvMaxTiles = 4;          // tiles of up to 256 vocabulary rows per CTA

struct GemvParams {
    TailParams t;     // V, d, R and everything the fused epilogue needs (scratch, classifier, outputs)
    int TR;           // vocabulary rows per CTA (slab)
    int tiles;        // ceil(TR / 256)
    int TRt;          // vocabulary rows per tile
    int TRN;          // rows of the LM-head box (TRt rounded up to 16, <= 256)
    int b_bytes;      // bytes of one ring stage (TRN * 128, a multiple of 1024)
    int h_rows;       // rows of the hidden-state box (8)
    int stages;       // ring depth (2 .. kGemvMaxStages)
};

constexpr int kLoopMaxSteps = 64;
constexpr unsigned kLoopContinue = 1u, kLoopStop = 2u;
// shared memory of the fold, per sequence: the warps' lists, entry k of warp w at [k * NW + w] (NW warps over all tiles;
// padded with -inf to whole batches of 32), and the warps' statistics
constexpr int kFoldMaxWarps = kGemvEpiWarps * kGemvMaxTiles;
constexpr int kFoldListWords = kTopK * kFoldMaxWarps;
constexpr int kFoldWords = kFoldListWords + 4 * kFoldMaxWarps;
static_assert(kFoldListWords % 32 == 0, "whole batches");

struct GemvLoopParams {
    GemvParams g;          // geometry of one step; g.t: shapes, scratch, classifier, outputs of step 1, chain bookkeeping
    int steps;             // sl_max
    int w_rows_per_step;   // the LM head of step i starts (i - 1) * w_rows_per_step rows into the tensor map (0: one head)
    unsigned int* flags;   // [steps] decision of each step: (stamp << 2) | kLoopContinue / kLoopStop
    unsigned int* epoch;   // launches completed so far; the stamp of this launch is that + 1
    float4* records;       // [sequence][CTA] stamped records of 80 bytes; written by this kernel only, starts zeroed
};

__device__ __forceinline__ void st_relaxed_u32(unsigned int* p, unsigned int v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The hidden rows of one step (rows row0 .. of the map), all k-blocks on one barrier; they stay for the step.
__device__ __forceinline__ void loop_issue_hidden(uint8_t* h_tiles, int h_stride, int KB, const CUtensorMap* tmap_H, int row0,
                                                  uint64_t* h_full) {
    mbar_arrive_expect_tx(h_full, (uint32_t)(KB * h_stride));
    for (int kb = 0; kb < KB; ++kb) tma_load_2d(h_tiles + kb * h_stride, tmap_H, kb * kUmmaBK, row0, h_full);
}

// A wait that is expected to last microseconds (the MMA issuer between two steps): sleep between the tests so
// that the warp does not compete for issue slots.  Bounded like mbar_wait.
__device__ __forceinline__ bool mbar_wait_idle(uint64_t* bar, uint32_t parity, int* status) {
    const long long t0 = clock64();
    for (int polls = 0;; ++polls) {
        if (mbar_try_wait(bar, parity)) return true;
        __nanosleep(64);
        if ((polls & 255) == 255 && ((status && *reinterpret_cast<volatile int*>(status) == DISCO_ERR_TIMEOUT) ||
                                     clock64() - t0 > kWaitBudgetClocks)) {
            record_status(status, DISCO_ERR_TIMEOUT);
            return false;
        }
    }
}

// Result of one hidden row of a step, in shared memory (16 words): m, Z, S, -, the ten largest logits, the arg-max key.
struct RowState {
    float m, Z, S, pad;
    float top[kTopK];
    uint32_t key_lo, key_hi;
};

// RK consecutive accumulator columns: one logit per thread and hidden row
template <int RK>
__device__ __forceinline__ void tmem_ld_rows(uint32_t taddr, float (&z)[RK]) {
    uint32_t r[RK];
    if constexpr (RK == 1)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r[0]) : "r"(taddr) : "memory");
    else if constexpr (RK == 2)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr) : "memory");
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(taddr)
                     : "memory");
    if constexpr (RK == 1)
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0])::"memory");
    else if constexpr (RK == 2)
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1])::"memory");
    else
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3])::"memory");
#pragma unroll
    for (int i = 0; i < RK; ++i) z[i] = __uint_as_float(r[i]);
}

// A warp's 32 logits of one hidden row (lane's vocabulary index v; lanes without one hold -inf), as warp w of NW: its
// list and its statistics (m, Z, S, arg-max key low word) go to `fold`.  warp_vals: 32 words owned by the warp.
__device__ __forceinline__ void warp_fold_row(float val, bool valid, int v, float* fold, int w, int NW, float* warp_vals,
                                              int lane) {
    const uint32_t bits = ordered_bits(val);
    const uint32_t mb = __reduce_max_sync(kFullMask, bits);
    // arg-max of the warp: largest value, lowest index (0: the warp holds no logit)
    const uint32_t klo = __reduce_max_sync(kFullMask, valid && bits == mb ? 0xffffffffu - static_cast<uint32_t>(v) : 0u);
    const int rank = rank_in_warp(val, lane, warp_vals);
    if (rank < kTopK) fold[rank * NW + w] = val;
    const float M = from_ordered_bits(mb);
    float e = 0.f, et = 0.f;
    if (valid) {
        const float t = val - M;
        e = __expf(t);
        et = e * t;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        e += __shfl_xor_sync(kFullMask, e, off);
        et += __shfl_xor_sync(kFullMask, et, off);
    }
    if (lane == 0) *reinterpret_cast<float4*>(fold + kFoldListWords + 4 * w) = make_float4(M, e, et, __uint_as_float(klo));
}

// The warps' results of one hidden row -> the CTA's, by a group of GT threads (whole warps; gt: index in it).  A barrier
// lies before (the warps' results are complete, rs->top is -inf) and after it.
template <int GT>
__device__ __forceinline__ void group_fold_row(const float* fold, int NW, RowState* rs, int gt) {
    const int lane = gt & 31, n = kTopK * NW;
    // ten logits are at or above the largest of the warps' tenth largest
    const float theta = from_ordered_bits(
        __reduce_max_sync(kFullMask, ordered_bits(lane < NW ? fold[(kTopK - 1) * NW + lane] : DISCO_NEG_INF)));
    // (entries that can qualify come first: the warps' largest, then their second largest, ..)
    for (int i = gt; i < n; i += GT) {
        const float x = fold[i];
        if (x >= theta && x > DISCO_NEG_INF) {
            const int r = rank_in_list(fold, n, x, i);
            if (r < kTopK) rs->top[r] = x;
        }
    }
    if (gt >= GT - 32) {
        const float4 q = lane < NW ? *reinterpret_cast<const float4*>(fold + kFoldListWords + 4 * lane)
                                   : make_float4(DISCO_NEG_INF, 0.f, 0.f, 0.f);
        const uint32_t mine = ordered_bits(q.y > 0.f ? q.x : DISCO_NEG_INF);
        const uint32_t Mb = __reduce_max_sync(kFullMask, mine);
        const uint32_t klo = __reduce_max_sync(kFullMask, q.y > 0.f && mine == Mb ? __float_as_uint(q.w) : 0u);
        const float M = from_ordered_bits(Mb);
        // (A warp whose sum is no number may have an infinite logit in its list: the CTA's sum is then no number either, and
        // the reader leaves its record out.)
        float Z = 0.f, S = 0.f;
        if (q.y != 0.f) {
            const float dm = q.x - M;
            const float e = __expf(dm);
            Z = q.y * e;
            S = e * fmaf(dm, q.y, q.z);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            Z += __shfl_xor_sync(kFullMask, Z, off);
            S += __shfl_xor_sync(kFullMask, S, off);
        }
        if (lane == 0) {
            rs->m = M, rs->Z = Z, rs->S = S;
            rs->key_hi = klo ? Mb : 0u, rs->key_lo = klo;
        }
    }
}

// RK: compile-time bound on the sequences (1, 2 or 4); 8 / RK epilogue warps finish each sequence.
template <int RK>
__global__ void __launch_bounds__(kGemvThreads, 1)
umma_gemv_loop_kernel(const __grid_constant__ CUtensorMap tmap_W, const __grid_constant__ CUtensorMap tmap_H,
                      const GemvLoopParams lp) {
    extern __shared__ uint8_t smem_dyn[];
    const GemvParams& g = lp.g;
    const TailParams& p = g.t;
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
    const int KB = (p.d + kUmmaBK - 1) / kUmmaBK;
    const int h_stride = g.h_rows * 128;
    uint8_t* h_tiles = smem;
    uint8_t* w_tiles = smem + KB * h_stride;
    uint8_t* after = w_tiles + g.stages * g.b_bytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(after);
    uint64_t* empty = full + kGemvMaxStages;
    uint64_t* tmem_full = empty + kGemvMaxStages;
    uint64_t* tmem_empty = tmem_full + 2;
    uint64_t* h_full = tmem_empty + 2;
    uint64_t* go_bar = h_full + 1;
    uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(go_bar + 1);
    uint32_t* s_code = tmem_base_s + 2;                       // [kLoopMaxSteps] decision of each step, as this CTA saw it
    RowState* row_s = reinterpret_cast<RowState*>(after + 1024);                 // [RK]
    float* fold_s = reinterpret_cast<float*>(row_s + RK);     // [RK][kFoldWords]
    float* vals_s = fold_s + RK * kFoldWords;                 // [8][32] the warps' logits
    float* group_s = vals_s + kGemvEpiWarps * 32;             // RK x kGroupScratchWords
    float* clf_s = group_s + RK * kGroupScratchWords;
    __shared__ int s_alive;
    __shared__ int s_pos0[4], s_forced[4], s_live[4];         // the finishing CTA's copy of the per-sequence inputs

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int grid = gridDim.x;
    const int B = p.R;
    const int v_begin = blockIdx.x * g.TR;
    const int v_end = min(p.V, v_begin + g.TR);
    const int tiles = v_begin < p.V ? (v_end - v_begin + g.TRt - 1) / g.TRt : 0;
    const int total = tiles * KB;          // LM-head stages of one step
    const bool two = g.TRN > 128;          // a tile has rows beyond the 128 of one MMA

    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], two ? 2 : 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tmem_full[b], two ? 2 : 1);
            mbar_init(&tmem_empty[b], kGemvEpiWarps);
        }
        mbar_init(h_full, 1);
        mbar_init(go_bar, 1);
        fence_mbar_init();
        prefetch_tensormap(&tmap_W);
        prefetch_tensormap(&tmap_H);
    }
    if (warp == 1) {
        tmem_alloc(tmem_base_s, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_base_s;

    if (warp == 0) {
        // ------------------------------ producer ------------------------------
        // One thread requests every LM-head stage of every step.  Its loop keeps running counters (no
        // divisions) and does nothing but test two barriers and issue copies; it sleeps when there is nothing to do.
        if (total > 0 && elect_one()) {
            const uint32_t w_bytes = (uint32_t)g.TRN * 128u;
            int w_step = 0, w_n = 0, w_tile = 0, w_kb = 0;     // the next stage to request: step, stage of the step, tile, k-block
            int w_row = v_begin;                                // first LM-head row of that step's slab in the tensor map
            int w_slot = 0, w_fill = 0;                         // its ring slot, and how often that slot has been filled before
            int ahead_slot = 0, ahead_fill = 0;                 // slot and fill count of the first stage of step w_step
            auto issue_w = [&]() {
                if (w_n == 0) {
                    ahead_slot = w_slot;
                    ahead_fill = w_fill;
                }
                mbar_arrive_expect_tx(&full[w_slot], w_bytes);
                tma_load_2d(w_tiles + w_slot * g.b_bytes, &tmap_W, w_kb * kUmmaBK, w_row + w_tile * g.TRt, &full[w_slot]);
                if (++w_kb == KB) {
                    w_kb = 0;
                    ++w_tile;
                }
                if (++w_n == total) {
                    w_n = 0;
                    w_tile = 0;
                    ++w_step;
                    w_row += lp.w_rows_per_step;
                }
                if (++w_slot == g.stages) {
                    w_slot = 0;
                    ++w_fill;
                }
            };
            // the LM head does not depend on the preceding kernel: the first step's stages are requested at once
            const int pre = min(g.stages, total);
            for (int n = 0; n < pre; ++n) issue_w();
            asm volatile("griddepcontrol.wait;" ::: "memory");
            loop_issue_hidden(h_tiles, h_stride, KB, &tmap_H, 0, h_full);
            int live = 1;                     // steps known to take place
            bool stopped = false;
            const long long t0 = clock64();
            int polls = 0;
            int p_step = 0, p_n = 0;          // the next stage to bring into L2: step, stage of the step
            for (;;) {
                bool progress = false;
                // the decision of step `live` (its hidden rows were requested by the thread that read the decision)
                if (live < lp.steps && mbar_test(go_bar, (live - 1) & 1)) {
                    if (s_code[live - 1] != kLoopContinue) {
                        stopped = true;
                        break;
                    }
                    ++live;
                    progress = true;
                }
                // the next LM-head stage: of a step known to take place, or of the one after it (requested ahead)
                if (w_step < lp.steps && w_step <= live) {
                    if (w_fill == 0 || mbar_test(&empty[w_slot], (w_fill - 1) & 1)) {
                        issue_w();
                        progress = true;
                    }
                } else if (w_step >= lp.steps && live >= lp.steps) {
                    break;                    // everything requested, every step known to take place
                }
                // The ring holds a good half of the next step's slab.  Once that has landed, HBM would idle until the step has
                // been decided: the other half is brought into L2 meanwhile, a box at a time (ten steps, 32000 x 768 head: 124 -> 115 us;
                // 49152 x 768: 185 -> 154).
                if (!progress && w_step == live && w_n > 0) {
                    if (p_step != w_step) p_step = w_step, p_n = w_n;
                    if (p_n < w_n) p_n = w_n;
                    const int last = w_slot == 0 ? g.stages - 1 : w_slot - 1;
                    if (p_n < total && mbar_test(&full[last], (w_slot == 0 ? w_fill - 1 : w_fill) & 1)) {
                        const int tile = p_n / KB, kb = p_n - tile * KB;
                        tma_prefetch_l2_2d(&tmap_W, kb * kUmmaBK, w_row + tile * g.TRt);
                        ++p_n;
                        progress = true;
                    }
                }
                if (!progress) __nanosleep(32);   // leave the issue slots to the warps that compute
                if (!progress && (++polls & 1023) == 0) {
                    if (*reinterpret_cast<volatile int*>(p.status) == DISCO_ERR_TIMEOUT ||
                        clock64() - t0 > kWaitBudgetClocks * (long long)lp.steps) {
                        record_status(p.status, DISCO_ERR_TIMEOUT);
                        stopped = true;
                        break;
                    }
                }
            }
            if (stopped) {
                // Stages requested ahead for the step that does not take place (the one after the `live` steps that
                // did: every stage of those has been consumed): its w_n first stages, or all of them if the next
                // stage to request already belongs to the step after it.  Nothing may still be landing at exit.
                const int n_ahead = w_step == live ? w_n : (w_step > live ? total : 0);
                int slot = ahead_slot, fill = ahead_fill;
                for (int n = 0; n < n_ahead; ++n) {
                    mbar_wait(&full[slot], fill & 1, p.status);
                    if (++slot == g.stages) {
                        slot = 0;
                        ++fill;
                    }
                }
            }
        }
    } else if (warp == 1 || warp == 2 + kGemvEpiWarps) {
        // ------------------------------ MMA issuers ------------------------------
        // MMAs this small are bound by their issue (39 cycles each, and a wait per stage), so the two halves of a tile have a
        // warp each: the first 128 rows of the box, and its last 128 (a multiple of eight rows in).
        const bool first = warp == 1;
        if (total > 0 && (first || two) && elect_one()) {
            const uint32_t idesc = umma_idesc(16);
            const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty);
            const uint64_t w0 = umma_smem_desc(w_tiles);
            const uint64_t h0 = umma_smem_desc(h_tiles) & ~(0x3fffull << 32);   // zero stride between the 8-row groups
            const uint32_t w_step = (uint32_t)g.b_bytes >> 4, h_step = (uint32_t)h_stride >> 4;   // descriptor units
            const uint64_t w_base = w0 + (first ? 0u : (uint32_t)(g.TRN - 128) * 8u);
            uint64_t w_desc = w_base;
            int h_ahead = -1;          // step whose hidden rows were requested and not yet used
            int slot = 0, fill = 0, t_global = 0;
            for (int step0 = 0; step0 < lp.steps; ++step0) {
                if (step0 > 0) {
                    if (!mbar_wait_idle(go_bar, (step0 - 1) & 1, p.status)) break;
                    if (s_code[step0 - 1] != kLoopContinue) break;
                }
                if (!mbar_wait(h_full, step0 & 1, p.status)) break;
                h_ahead = -1;
                tc_fence_after();
                for (int tile = 0; tile < tiles; ++tile, ++t_global) {
                    const int buf = t_global & 1;
                    mbar_wait(&tmem_empty[buf], ((t_global >> 1) & 1) ^ 1, p.status);
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + buf * 32 + (first ? 0 : 16);
                    uint64_t h_desc = h0;
                    for (int kb = 0; kb < KB; ++kb) {
                        mbar_wait(full0 + slot * 8, fill & 1, p.status);
                        tc_fence_after();
#pragma unroll
                        for (int k = 0; k < kUmmaBK / 16; ++k)
                            tc_mma_bf16(d_tmem, w_desc + 2 * k, h_desc + 2 * k, idesc, (kb | k) != 0);
                        tc_commit(empty0 + slot * 8);
                        w_desc += w_step;
                        h_desc += h_step;
                        if (++slot == g.stages) {
                            slot = 0;
                            ++fill;
                            w_desc = w_base;
                        }
                    }
                    tc_commit(&tmem_full[buf]);
                }
                // Once the MMAs of this step are done with the hidden rows, those of the next step are requested, ahead of the
                // decision (if the phase stops here they are awaited before the CTA leaves).
                if (first && step0 + 1 < lp.steps) {
                    mbar_wait(&tmem_full[(t_global - 1) & 1], ((t_global - 1) >> 1) & 1, p.status);
                    loop_issue_hidden(h_tiles, h_stride, KB, &tmap_H, (step0 + 1) * B, h_full);
                    h_ahead = step0 + 1;
                }
            }
            if (h_ahead >= 0) mbar_wait(h_full, h_ahead & 1, p.status);
        }
    } else {
        // ------------------------------ epilogue ------------------------------
        constexpr int BAR_THREADS = kGemvEpiWarps * 32;
        constexpr int GW = kGemvEpiWarps / RK;      // warps that finish one sequence
        const int ew = warp - 2;
        const int quad = warp & 3;
        const int tid = ew * 32 + lane;
        if (p.clf_H > 0 && blockIdx.x == 0) {       // the finishing CTA stages the classifier
            const int Hc = p.clf_H;
            const int n1 = Hc * kNFeat;
            for (int i = tid; i < n1 + 2 * Hc + 1; i += BAR_THREADS) {
                const float* src = i < n1 ? p.clf_W1 + i
                                          : (i < n1 + Hc ? p.clf_b1 + (i - n1)
                                                         : (i < n1 + 2 * Hc ? p.clf_w2 + (i - n1 - Hc) : p.clf_b2));
                cp_async4(clf_s + i, src);
            }
            cp_async_commit();
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        // stamp of this launch: read by every CTA before anything of this launch can advance the word
        const unsigned int launch_stamp = ld_relaxed_u32(lp.epoch) + 1u;
        if (blockIdx.x == 0 && tid < B) {
            s_pos0[tid] = p.chain.pos0[tid];
            s_forced[tid] = p.chain.sl_forced ? p.chain.sl_forced[tid] : 0x7fffffff;
            s_live[tid] = 1;
        }
        cp_async_wait_all();
        // (the padding of the lists is never written again)
        for (int i = tid; i < RK * kFoldWords; i += BAR_THREADS) fold_s[i] = DISCO_NEG_INF;
        named_barrier_sync(1, BAR_THREADS);
        int t_global = 0;
        // this thread's vocabulary row within a tile: 128 per half of the tile's box
        const bool second_half = ew >= 4;
        const int tile_row = quad * 32 + lane + (second_half ? g.TRN - 128 : 0);
        const bool row_ok = second_half ? g.TRN > 128 && tile_row >= 128 : true;
        const int NW = tiles * kGemvEpiWarps;

        for (int step0 = 0; step0 < lp.steps; ++step0) {
            // stamp of this step's records: unique among everything a reader can still find in the buffer
            const uint32_t rec_stamp = (launch_stamp << 6) | (uint32_t)(step0 & 63) | 0x80000000u;
            if (tid < RK * kTopK) row_s[tid / kTopK].top[tid % kTopK] = DISCO_NEG_INF;
            for (int tile = 0; tile < tiles; ++tile, ++t_global) {
                const int buf = t_global & 1;
                const int v0 = v_begin + tile * g.TRt;
                const int ncols = min(g.TRt, v_end - v0);
                mbar_wait(&tmem_full[buf], (t_global >> 1) & 1, p.status);
                tc_fence_after();
                float z[RK];
                tmem_ld_rows<RK>(tmem_base + buf * 32 + (second_half ? 16 : 0) + (static_cast<uint32_t>(quad * 32) << 16), z);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tmem_empty[buf]);
                const bool valid = row_ok && tile_row < ncols;
#pragma unroll
                for (int r = 0; r < RK; ++r)
                    if (r < B)
                        warp_fold_row(valid ? __fadd_rn(z[r], 0.f) : DISCO_NEG_INF, valid, v0 + tile_row, fold_s + r * kFoldWords,
                                      tile * kGemvEpiWarps + ew, NW, vals_s + ew * 32, lane);
            }
            named_barrier_sync(1, BAR_THREADS);   // the warps' results are complete
            const int gb = ew / GW;               // the sequence this warp's group works for
            const int gt = (ew % GW) * 32 + lane;
            if (gb < B) {
                group_fold_row<GW * 32>(fold_s + gb * kFoldWords, NW, row_s + gb, gt);
                named_barrier_sync(2 + gb, GW * 32);
            }
            // ---- the CTA's record of this step for each sequence, in stamped pieces ----
            if (gb < B && gt < kStampedPieces) {
                const int r = gb, piece = gt;
                const RowState* rs = row_s + r;
                float4* dst = lp.records + ((size_t)r * grid + blockIdx.x) * kStampedPieces + piece;
                const float sf = __uint_as_float(rec_stamp);
                float a, b2, c2;
                if (piece == 0) a = rs->m, b2 = rs->Z, c2 = rs->S;
                else if (piece < 4) a = rs->top[3 * piece - 3], b2 = rs->top[3 * piece - 2], c2 = rs->top[3 * piece - 1];
                else a = rs->top[9], b2 = __uint_as_float(rs->key_lo), c2 = __uint_as_float(rs->key_hi);
                store_relaxed_v4(dst, a, b2, c2, sf);
            }
            // ---- CTA 0 finishes the sequences and decides ----
            if (blockIdx.x == 0) {
                if (tid == 0) s_alive = 0;
                named_barrier_sync(1, BAR_THREADS);
                const int b = gb;
                if (b < B) {
                    const bool takes_part = s_live[b] != 0;
                    if (takes_part) {               // uniform over the group
                        const MergedPartials mp =
                            group_merge_partials<GW>(lp.records + (size_t)b * grid * kStampedPieces, grid, rec_stamp,
                                                     p.status, group_s + b * kGroupScratchWords, 2 + b, gt);
                        if (gt < 32) {
                            const size_t at = (size_t)step0 * B;
                            const DraftOutputs o{p.token + at, p.conf + at, p.halt + at,
                                                 p.feats ? p.feats + at * kNFeat : nullptr, p.final_stats, nullptr, 0,
                                                 ChainLink{}};
                            const int Hc = p.clf_H;
                            const bool no_halt = warp_draft_epilogue(
                                mp.st, mp.key, mp.sel, static_cast<float>(s_pos0[b] + step0 + 1), step0 + 1, p.tau,
                                p.sl_max, group_s + b * kGroupScratchWords, clf_s, clf_s + Hc * kNFeat,
                                clf_s + Hc * (kNFeat + 1), clf_s + Hc * (kNFeat + 2), Hc, b, o, lane);
                            if (lane == 0) {
                                // the look-ahead bookkeeping: this CTA finishes every step, so it keeps the flags itself
                                const bool goes_on = s_forced[b] != 0x7fffffff ? (step0 + 1 < s_forced[b]) : no_halt;
                                p.chain.sl[b] = step0 + 1;
                                s_live[b] = goes_on ? 1 : 0;
                                if (goes_on) atomicAdd(&s_alive, 1);
                            }
                        }
                    }
                }
                named_barrier_sync(1, BAR_THREADS);
                if (tid == 0) {
                    const bool last_step = step0 + 1 == lp.steps;
                    const unsigned code = (s_alive > 0 && !last_step) ? kLoopContinue : kLoopStop;
                    // the launch stamp may move on: every CTA has read it (their records of this step were seen)
                    if (code == kLoopStop) *lp.epoch = launch_stamp == 0x00ffffffu ? 0u : launch_stamp;
                    // Nothing in this launch reads what a step wrote except through this word (the outputs are for later
                    // kernels, the records were consumed before the decision): no ordering is needed beside it.
                    st_relaxed_u32(lp.flags + step0, (launch_stamp << 2) | code);
                }
            }
            // ---- every CTA learns the decision ----
            if (tid == 0) {
                unsigned code = 0u;
                const long long t0 = clock64();
                for (int polls = 0;; ++polls) {
                    const unsigned f = ld_relaxed_u32(lp.flags + step0);
                    if ((f >> 2) == launch_stamp) {
                        code = f & 3u;
                        break;
                    }
                    if ((polls & 63) == 63 && (*reinterpret_cast<volatile int*>(p.status) == DISCO_ERR_TIMEOUT ||
                                               clock64() - t0 > kWaitBudgetClocks)) {
                        record_status(p.status, DISCO_ERR_TIMEOUT);
                        code = kLoopStop;
                        break;
                    }
                }
                s_code[step0] = code;
                __threadfence_block();
                mbar_arrive(go_bar);                // the producer and the MMA issuer go on (or leave)
            }
            named_barrier_sync(1, BAR_THREADS);
            if (s_code[step0] != kLoopContinue) break;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

inline size_t gemv_loop_fixed_smem_bytes(int RK, int clf_H, int d, int h_rows, int TRN) {
    size_t b = 1024;                                             // alignment
    b += (size_t)((d + kUmmaBK - 1) / kUmmaBK) * h_rows * 128;   // hidden rows
    b += 1024;                                                   // barriers, TMEM address, decisions
    b += TRN < 128 ? 16384 : 0;                                  // an MMA reads 128 rows from the start of a stage
    b += (size_t)RK * sizeof(RowState);                          // results of the rows
    b += (size_t)(RK * kFoldWords + kGemvEpiWarps * 32) * 4;     // fold
    b += (size_t)RK * kGroupScratchWords * 4;                    // finishing groups
    b += ((size_t)clf_H * (kNFeat + 2) + 4) * 4;                 // classifier parameters
    return b + 128;
}

}  // namespace disco
