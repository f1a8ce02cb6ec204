// Tensor-core draft step for few hidden rows (and the target rows of a small verification with sampling): the work of
// draft_batch.cuh with the operands the other way round,
//
//   D[v, r] = sum_k W[v, k] * H[r, k]      v on the 128 TMEM lanes, r on the TMEM columns
//
// With the hidden rows on the lanes an MMA of 112 vocabulary rows occupies the tensor pipe for 79 cycles whether one row is
// wanted or 128; this way round it is the operand of 128 vocabulary rows that crosses shared memory, 39 cycles at up to 16
// hidden rows.  One row of a 32000 x 768 head: the MMAs of a launch took 5.6 us of 14.6, most of them after the wait for the
// launch before.
//
//   * warp 0      producer: a box of W (up to 128 vocabulary rows x 64 k) and one of H (8 NR rows x 64 k) per stage; the
//                 LM-head boxes of the first stages are requested before the dependency wait;
//   * warp 1      issues tcgen05.mma (M = 128, N = the hidden rows) into one of up to 16 accumulators;
//   * warps 2-9   epilogue: an accumulator goes through shared memory, so that a warp then has a hidden row's logits, four
//                 per lane and tile, of rows warp, warp + 8, ..: partial soft-max sums and arg-max per lane, and the row's
//                 ten largest in lanes 0 - 9;
//   * warps 10-11 and, in the grid's last CTAs, which have no vocabulary, all of 2-11: finish a row each, as in
//                 draft_batch.cuh, whose records, shared bounds and start counter these are.
#pragma once

#include "draft_batch.cuh"

namespace disco {

constexpr int kFewMaxBufs = 16;
constexpr int kFewBarBytes = 768;
constexpr int kFewRankWords = 64;      // per epilogue warp: 32 candidates, the ten largest so far, padding

// The ten largest (lanes 0 .. 9, descending) of those so far and of one candidate per lane (-inf: none).
static __device__ __noinline__ float few_merge_top(float top, float cand, float* sm, int lane) {
    sm[lane] = cand;
    sm[32 + lane] = lane < kTopK ? top : DISCO_NEG_INF;
    __syncwarp();
    const int r_new = cand > DISCO_NEG_INF ? rank_in_list(sm, 42, cand, lane) : kTopK;
    const int r_old = lane < kTopK && top > DISCO_NEG_INF ? rank_in_list(sm, 42, top, 32 + lane) : kTopK;
    __syncwarp();
    if (lane < kTopK) sm[lane] = DISCO_NEG_INF;
    __syncwarp();
    if (r_new < kTopK) sm[r_new] = cand;
    if (r_old < kTopK) sm[r_old] = top;
    __syncwarp();
    const float t = lane < kTopK ? sm[lane] : DISCO_NEG_INF;
    __syncwarp();
    return t;
}

// The same for the lanes of mask alone, their value x above thr: nearly always one or two, which are put in one after the other.
// (Merging 32 at a time whenever one qualified made the CTAs that
// hold a row's largest logits 2 us later than the others.)
static __device__ __noinline__ float few_insert(float top, float x, unsigned mask, float* sm, int lane) {
    if (__popc(mask) > 8) return few_merge_top(top, (mask >> lane) & 1u ? x : DISCO_NEG_INF, sm, lane);
    while (mask) {
        const float v = __shfl_sync(kFullMask, x, __ffs(mask) - 1);
        mask &= mask - 1u;
        const int at = __popc(__ballot_sync(kFullMask, lane < kTopK && top >= v));   // (equal values: behind)
        const float up = __shfl_up_sync(kFullMask, top, 1);
        if (lane < kTopK && lane >= at) top = lane == at ? v : up;
    }
    return top;
}

template <int N>
__device__ __forceinline__ void tmem_ld_few(uint32_t taddr, float (&v)[N]) {
    static_assert(N == 4 || N == 8 || N == 16, "");
    uint32_t r[N];
    if constexpr (N == 4)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
    else if constexpr (N == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "r"(taddr) : "memory");
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                     "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                       "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                     : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < N; ++i) {
        asm volatile("" : "+r"(r[i]));
        v[i] = __uint_as_float(r[i]);
    }
}

// STATS: arg-max and soft-max statistics only (f.stats_only == 1).  NR: hidden rows per epilogue warp, 8 NR at most in all.
template <bool STATS, int NR>
__global__ void __launch_bounds__(kDbThreads, 1)
umma_draft_few_kernel(const __grid_constant__ CUtensorMap tmap_W, const __grid_constant__ CUtensorMap tmap_H,
                      const DraftBatchParams p, const DraftFinalParams f) {
    constexpr int kRows = 8 * NR, N = kRows < 16 ? 16 : kRows;
    constexpr int NB = 512 / N < kFewMaxBufs ? 512 / N : kFewMaxBufs;   // accumulators
    extern __shared__ uint8_t smem_dyn[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
    uint8_t* w_tiles = smem;
    uint8_t* h_tiles = smem + p.stages * p.b_bytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + p.ring_bytes);
    uint64_t* empty = full + kDbMaxStages;
    uint64_t* tmem_full = empty + kDbMaxStages;
    uint64_t* tmem_empty = tmem_full + kFewMaxBufs;
    uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(tmem_empty + kFewMaxBufs);
    uint32_t* s_stamp = tmem_base_s + 2;                      // (as in draft_batch.cuh)
    uint32_t* s_look = tmem_base_s + 4;
    uint32_t* s_live = tmem_base_s + 5;
    float* zt_s = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(full) + kFewBarBytes);   // [2][kRows][128] logits of a tile
    float* rank_s = zt_s + 2 * kRows * 128;
    float* fin_s = rank_s + kDbEpiWarps * kFewRankWords;
    float* clf_s = fin_s + (kDbEpiWarps + kDbFinWarps) * kDbFinWords;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int KB = (p.d + kUmmaBK - 1) / kUmmaBK;
    const int nslot = blockIdx.x;
    const int v_first = nslot * p.TPC * p.TR;                 // this CTA's vocabulary rows: its tiles in sequence
    const int tiles = v_first < p.V ? min(p.TPC, (p.V - v_first + p.TR - 1) / p.TR) : 0;
    const bool chained = !STATS && f.chain.alive != nullptr && f.chain.step > 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < NB; ++b) {
            mbar_init(&tmem_full[b], 1);
            mbar_init(&tmem_empty[b], kDbEpiWarps);
        }
        *s_stamp = 0u;
        *s_live = 0u;
        fence_mbar_init();
        prefetch_tensormap(&tmap_W);
        prefetch_tensormap(&tmap_H);
    }
    if (warp == 1) {
        tmem_alloc(tmem_base_s, 512);
        tmem_relinquish();
    }
    if (warp == 2) {   // (a hint, as in draft_batch.cuh)
        const bool any = !chained || chain_any_live(f.chain, f.chain.B, lane);
        if (lane == 0) *s_look = any ? 1u : 0u;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_base_s;
    const bool looks_live = *s_look != 0u;
    auto step_live = [&]() { return !chained || cold_smem_word(s_live, p.status) == 1u; };

    if (warp == 0) {
        // ------------------------------ producer ------------------------------
        const int total = tiles * KB;
        const uint32_t w_bytes = (uint32_t)p.w_rows * 128u, h_bytes = (uint32_t)kRows * 128u;
        const int pre = looks_live ? min(p.stages, total) : 0;
        const int rot = nslot % KB;       // (every CTA reads the same hidden rows: each starts at another k-block)
        const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty), w0 = smem_addr(w_tiles), h0 = smem_addr(h_tiles);
        const int k_end = KB * kUmmaBK, k_first = rot * kUmmaBK;
        int k = k_first, v0 = v_first, left = KB;      // the next stage to request: k, vocabulary row, k-blocks left of the tile
        auto advance = [&]() {
            k += kUmmaBK;
            if (k == k_end) k = 0;
            if (--left == 0) {
                left = KB;
                v0 += p.TR;
            }
        };
        if (elect_one()) {
            for (int n = 0; n < pre; ++n, advance()) {
                mbar_expect_tx(full0 + n * 8, w_bytes);
                tma_load_2d(w0 + n * p.b_bytes, &tmap_W, k, v0, full0 + n * 8);
            }
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const bool live = step_live();
        if (!live) {
            if (elect_one()) {
                for (int n = 0; n < pre; ++n) mbar_arrive(&full[n]);
                for (int n = 0; n < pre; ++n) mbar_wait(&full[n], 0, p.status);   // nothing may still be landing at exit
            }
        } else if (elect_one()) {
            int kh = k_first;
            for (int n = 0; n < pre; ++n) {
                mbar_arrive_expect_tx(full0 + n * 8, h_bytes);
                tma_load_2d(h0 + n * kRows * 128, &tmap_H, kh, 0, full0 + n * 8);
                kh += kUmmaBK;
                if (kh == k_end) kh = 0;
            }
            int stage = pre == p.stages ? 0 : pre, phase = pre == p.stages ? 1 : 0;
            k = k_first, v0 = v_first, left = KB;      // (the elected thread need not be the one of before)
            for (int n = 0; n < pre; ++n) advance();
            uint32_t at_h = h0 + stage * kRows * 128, at_w = w0 + stage * p.b_bytes;
            for (int n = pre; n < total; ++n, advance()) {
                const uint32_t bar = full0 + stage * 8;
                mbar_wait(empty0 + stage * 8, phase ^ 1, p.status);
                mbar_arrive_expect_tx(bar, w_bytes + h_bytes);
                tma_load_2d(at_w, &tmap_W, k, v0, bar);
                tma_load_2d(at_h, &tmap_H, k, 0, bar);
                at_h += kRows * 128;
                at_w += p.b_bytes;
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1;
                    at_h = h0;
                    at_w = w0;
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        bool live = true;
        if (chained) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            live = chain_any_live(f.chain, f.chain.B, lane);
            if (lane == 0) *reinterpret_cast<volatile uint32_t*>(s_live) = live ? 1u : 2u;
        }
        if (live && elect_one()) {
            const uint32_t idesc = umma_idesc(N);
            const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty);
            // The MMA reads 128 rows from the start of a stage of W: what lies behind a smaller box (shared memory of this CTA,
            // ring_bytes sees to that) only feeds lanes nobody reads.  Eight hidden rows are read twice over.
            const uint64_t a0 = umma_smem_desc(w_tiles);
            const uint64_t b0 = umma_smem_desc(h_tiles) & (NR == 1 ? ~(0x3fffull << 32) : ~0ull);
            const uint32_t a_step = (uint32_t)p.b_bytes >> 4, b_step = (uint32_t)kRows * 128u >> 4;   // descriptor units
            uint64_t a_desc = a0, b_desc = b0;
            int stage = 0, phase = 0;
            for (int t = 0; t < tiles; ++t) {
                const int buf = t % NB;
                mbar_wait(&tmem_empty[buf], ((t / NB) & 1) ^ 1, p.status);
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + buf * N;
                for (int kb = 0; kb < KB; ++kb) {
                    mbar_wait(full0 + stage * 8, phase, p.status);
                    tc_fence_after();
#pragma unroll
                    for (int k = 0; k < kUmmaBK / 16; ++k)
                        tc_mma_bf16(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, (kb | k) != 0);
                    tc_commit(empty0 + stage * 8);
                    a_desc += a_step;
                    b_desc += b_step;
                    if (++stage == p.stages) {
                        stage = 0;
                        phase ^= 1;
                        a_desc = a0;
                        b_desc = b0;
                    }
                }
                tc_commit(&tmem_full[buf]);
            }
        }
    }
    const bool finisher = nslot >= p.CN;
    if (warp >= 2 && warp < 2 + kDbEpiWarps && !finisher) {
        // ------------------------------ epilogue ------------------------------
        const int ew = warp - 2;
        const int quad = warp & 3;              // TMEM lane quadrant this warp may read
        const int share = ew >> 2;              // the two warps of a quadrant split the columns
        const uint32_t t_quad = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + share * 4 * NR;
        float* rank = rank_s + ew * kFewRankWords;
        const bool use_bound = !STATS && (p.TPC > 1 || p.TR > 32);
        const bool defer = tiles > 1;           // a tile's candidates are looked for one tile later, with a better bound
        // (twice: a rehearsal without tiles before the dependency wait, as in draft_batch.cuh)
#pragma unroll 1
        for (int phase = opaque(looks_live ? 0 : 1); phase < 2; phase = opaque(phase + 1)) {
            // Row q of this warp is hidden row ew + 8 q.  m, the largest logit so far, is the warp's; Z, S and the arg-max are
            // the lane's shares; top: lane k < 10 holds the row's k-th largest candidate.
            float m[NR], Z[NR], S[NR], best_v[NR], top[NR], thr[NR], bound_used[NR];
            int best_i[NR];
            bool valid[NR];
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                m[q] = best_v[q] = top[q] = thr[q] = bound_used[q] = DISCO_NEG_INF;
                Z[q] = S[q] = 0.f;
                best_i[q] = (int)kDbNoIndex;
                valid[q] = ew + 8 * q < p.R;
            }
            uint32_t stamp = 1u;
            unsigned int* slots = nullptr;
            if (phase == 0) {
#pragma unroll
                for (int q = 0; q < NR; ++q) m[q] = best_v[q] = static_cast<float>(lane), Z[q] = 1.f;
                if constexpr (!STATS) top[0] = few_insert(top[0], m[0], opaque(1), rank, lane);
            } else {
                asm volatile("griddepcontrol.wait;" ::: "memory");  // scratch and outputs belong to the predecessor until now
                if (!step_live()) break;
                uint32_t seen = 0u;
#pragma unroll
                for (int q = 0; q < NR; ++q) {
                    valid[q] = valid[q] && chain_seq_live(f.chain, f.active, chain_seq(f.chain, ew + 8 * q));
                    seen |= valid[q] ? 1u << q : 0u;
                }
                stamp = db_begin(p, f, ew, s_stamp, seen, lane);
                slots = p.bound + (stamp & 1u) * p.set_words + (size_t)ew * kDbBoundStride;    // row q: 8 q rows on
            }
            const int phase_tiles = phase == 0 ? 0 : tiles;
            float zp[NR][4];                    // the tile before
            float lp[NR];
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                lp[q] = DISCO_NEG_INF;
#pragma unroll
                for (int i = 0; i < 4; ++i) zp[q][i] = DISCO_NEG_INF;
            }
            for (int t = 0; t < phase_tiles; ++t) {
                const int v0 = v_first + t * p.TR, ncols = min(p.TR, p.V - v0);
                mbar_wait(&tmem_full[t % NB], (t / NB) & 1, p.status);
                tc_fence_after();
                float* zt = zt_s + (t & 1) * kRows * 128;
                if (quad * 32 < ncols) {
                    float z[4 * NR];
                    tmem_ld_few<4 * NR>(t_quad + (t % NB) * N, z);
#pragma unroll
                    for (int c = 0; c < 4 * NR; ++c) zt[(share * 4 * NR + c) * 128 + quad * 32 + lane] = z[c];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tmem_empty[t % NB]);
                uint4 sa[NR], sb[NR], sc[NR];   // the rows' bounds, on their way during the statistics
#pragma unroll
                for (int q = 0; q < NR; ++q) {
                    sa[q] = sb[q] = sc[q] = make_uint4(0, 0, 0, 0);
                    if (use_bound && valid[q] && t > 0) {
                        const unsigned int* s = slots + (size_t)8 * q * kDbBoundStride;
                        sa[q] = ld_relaxed_v4_u32(s);
                        sb[q] = ld_relaxed_v4_u32(s + 4);
                        sc[q] = ld_relaxed_v4_u32(s + 8);
                    }
                }
                // (two halves used by turns: a warp writes the next tile's while others still read this one's)
                named_barrier_sync(4, kDbEpiWarps * 32);
                float zc[NR][4], lc[NR];
#pragma unroll
                for (int q = 0; q < NR; ++q) {
                    lc[q] = DISCO_NEG_INF;
#pragma unroll
                    for (int i = 0; i < 4; ++i) zc[q][i] = DISCO_NEG_INF;
                    if (!valid[q]) continue;    // (the whole warp)
                    const float* src = zt + (ew + 8 * q) * 128 + lane;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (lane + 32 * i < ncols) zc[q][i] = src[32 * i];
                    lc[q] = fmaxf(max3f(zc[q][0], zc[q][1], zc[q][2]), zc[q][3]);
                    const float tile_max = warp_max_f32(lc[q]);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (zc[q][i] > best_v[q]) best_v[q] = zc[q][i], best_i[q] = v0 + lane + 32 * i;
                    const float mn = fmaxf(m[q], tile_max);
                    const float dm = fmaxf(m[q] - mn, -1000.f);
                    const float em = ex2_approx(dm * kLog2e);
                    m[q] = mn;
                    float Zc = 0.f, Sc = 0.f;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        // (columns there are none of: finite, far below any logit)
                        const float x = (lane + 32 * i < ncols ? zc[q][i] : -2e38f) - mn;
                        const float e = ex2_approx(x * kLog2e);
                        Zc += e;
                        Sc = fmaf(e, x, Sc);
                    }
                    S[q] = fmaf(em, fmaf(dm, Z[q], S[q]), Sc);
                    Z[q] = fmaf(Z[q], em, Zc);
                    if (p.probs) {
                        float* dst = p.probs + (size_t)(ew + 8 * q) * p.V + v0 + lane;
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (lane + 32 * i < ncols) dst[32 * i] = zc[q][i];
                    }
                    if (use_bound && lane == 0 && (t == 0 || t + 1 < tiles) && tile_max > bound_used[q] && tile_max < -DISCO_NEG_INF)
                        atomicMax(slots + (size_t)8 * q * kDbBoundStride + nslot % kDbBoundSlots, ordered_bits(tile_max + 0.f));
                }
                if constexpr (!STATS) {
                    if (use_bound && (t > 0 || !defer)) {
                        if (t == 0) {
                            for (int k = 0; k < 4; ++k) {   // (not waited for longer: the bound only saves work)
                                bool there = true;
#pragma unroll
                                for (int q = 0; q < NR; ++q) {
                                    if (!valid[q]) continue;
                                    const unsigned int* s = slots + (size_t)8 * q * kDbBoundStride;
                                    sa[q] = ld_relaxed_v4_u32(s);
                                    sb[q] = ld_relaxed_v4_u32(s + 4);
                                    sc[q] = ld_relaxed_v4_u32(s + 8);
                                    there = there && row_bound_of<false>(sa[q], sb[q], sc[q]) > DISCO_NEG_INF;
                                }
                                if (__all_sync(kFullMask, there)) break;
                            }
                        }
#pragma unroll
                        for (int q = 0; q < NR; ++q)    // (lane 0's look: the lanes may have seen different words)
                            if (valid[q])
                                bound_used[q] = fmaxf(bound_used[q], __shfl_sync(kFullMask, row_bound_of<false>(sa[q], sb[q], sc[q]), 0));
                    }
#pragma unroll
                    for (int late = 0; late < 2; ++late) {   // the tile before, then this one if it is the last
                        if (late == 0 ? !(defer && t > 0) : defer && t + 1 < tiles) continue;
#pragma unroll
                        for (int q = 0; q < NR; ++q) {
                            thr[q] = fmaxf(thr[q], bound_used[q]);
                            if (!__any_sync(kFullMask, (late == 0 ? lp[q] : lc[q]) > thr[q])) continue;
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const float x = late == 0 ? zp[q][i] : zc[q][i];
                                const unsigned mask = __ballot_sync(kFullMask, x > thr[q]);
                                if (!mask) continue;
                                top[q] = few_insert(top[q], x, mask, rank, lane);
                                thr[q] = fmaxf(thr[q], __shfl_sync(kFullMask, top[q], kTopK - 1));
                            }
                        }
                    }
#pragma unroll
                    for (int q = 0; q < NR; ++q) {
                        lp[q] = lc[q];
#pragma unroll
                        for (int i = 0; i < 4; ++i) zp[q][i] = zc[q][i];
                    }
                }
            }

            // one record per hidden row and CTA
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                if (!valid[q]) continue;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    Z[q] += __shfl_xor_sync(kFullMask, Z[q], off);
                    S[q] += __shfl_xor_sync(kFullMask, S[q], off);
                }
                const float bv = best_v[q] + 0.f;   // -0 and +0 are the same logit
                const uint32_t ob = ordered_bits(bv), mb = __reduce_max_sync(kFullMask, ob);
                const uint32_t idx = __reduce_min_sync(kFullMask, ob == mb ? (uint32_t)best_i[q] : kDbNoIndex);
                // (statistics that are no numbers: the record is as good as empty)
                const bool numbers = Z[q] > 0.f;
                const float tq = numbers ? top[q] + 0.f : DISCO_NEG_INF;
                const int cnt = !STATS && numbers ? __popc(__ballot_sync(kFullMask, lane < kTopK && tq > DISCO_NEG_INF)) : 0;
                const uint32_t word = ((uint32_t)cnt << 28) | (numbers ? idx : kDbNoIndex);
                // lane 0: m Z S; lane 1: word l0 bound; lanes 2 - 4: three of the list each
                const int from = 3 * lane - 5;
                const float l0 = __shfl_sync(kFullMask, tq, 0);
                float a = __shfl_sync(kFullMask, tq, from & 31), b = __shfl_sync(kFullMask, tq, (from + 1) & 31),
                      c = __shfl_sync(kFullMask, tq, (from + 2) & 31);
                if (lane == 0) a = m[q] + 0.f, b = Z[q], c = S[q];
                if (lane == 1) a = __uint_as_float(word), b = l0, c = bound_used[q];
                if (phase == 1 && lane < (cnt > 4 ? 5 : 3))
                    store_relaxed_v4(p.part_rec + ((size_t)(ew + 8 * q) * kStampedPieces + lane) * p.CN + nslot, a, b, c,
                                     __uint_as_float(stamp));
            }
        }
    }
    if (finisher && warp >= 2) db_finish_dedicated<STATS>(p, f, warp, looks_live, fin_s, clf_s, s_stamp, step_live, lane);

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// Shared memory beside the ring.
inline size_t draft_few_fixed_smem(int NR, int clf_H) {
    return 1024 + kFewBarBytes + (size_t)(2 * 8 * NR * 128 + kDbEpiWarps * kFewRankWords + (kDbEpiWarps + kDbFinWarps) * kDbFinWords) * 4 +
           umma_clf_bytes(clf_H) + 128;
}

}  // namespace disco
