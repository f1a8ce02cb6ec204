// Tensor-core draft step for a batch (and, with other epilogue switches, every other pass over an LM head that wants
// soft-max statistics: the target rows of a verification with sampling, bulk feature extraction).
//
//   D[r, v] = sum_k H[r, k] * W[v, k]      r on the 128 TMEM lanes, v on the TMEM columns
//
//   * warp 0      producer: one TMA box of H (A operand, up to 128 rows x 64 k) and one of W (B operand, one
//                 vocabulary tile x 64 k) per stage; the LM-head boxes of the first stages are requested before the
//                 dependency wait;
//   * warp 1      issues tcgen05.mma (M = 128, N = tile rows) into one of two or four accumulator buffers in TMEM;
//   * warps 2-9   epilogue: every thread owns one hidden row and walks over its share of a tile's columns: soft-max
//                 statistics in registers, and the few logits that can still be among the row's ten largest;
//   * warps 10-11 finish rows: one warp merges the per-CTA records of a hidden row, forms the features of Eq. 2, runs
//                 the halt classifier and the stopping rule.  With one tile of rows (up to 128) the grid's last CTAs do that,
//                 with ten warps each, and have no vocabulary of their own (db_finish_dedicated).
//
// What the design is built around:
//   * The ten largest.  A CTA sees a few hundred columns of each row, so "above this CTA's tenth largest" is no
//     filter (a tenth of all logits pass), and an insertion network fed by it is half of the epilogue.  The rows share a
//     bound instead: twelve words per row, each the largest logit published so far by every twelfth CTA of the grid
//     (atomicMax).  Ten of the twelve groups have a logit at or above the third smallest word, so that is a lower bound
//     of the row's tenth largest logit, at any time and whatever the timing; the final list is exact.  About twenty of a
//     row's logits pass it, over all CTAs.
//   * No waiting on CTAs that may not run.  The finishing warps wait for other CTAs' records, but only once every CTA of
//     the grid has started (a counter); with more than one tile of rows a CTA that is done before that leaves, and the CTA
//     that starts last always finds the counter full, so every row is finished by somebody, with any number of other
//     kernels on the device.  So the launch need not be cooperative, and its prologue and first loads run under the tail of
//     the kernel before it (a cooperative launch was measured to cost 4 - 5 us in a stream).
//   * Code that runs once per launch is fetched from L2 instruction by instruction.  Both the finishing code and what
//     follows the column loop run once for nothing while the first tile is awaited, and the finishing code is short: the
//     wait for the records and what follows it took 12.5 thousand cycles of a launch of 28 (one row of 32000 x 768), now 6
//     of 21.
#pragma once

#include "draft_rules.cuh"
#include "umma_tail.cuh"

namespace disco {

constexpr int kDbThreads = (2 + kDbEpiWarps + kDbFinWarps) * 32;
constexpr int kDbMaxStages = 16;
constexpr int kDbMaxRecords = 160;     // records per row a finishing warp takes in: five per lane
constexpr int kDbXchBytes = 128 * 64;  // states handed between the two warps that share a hidden row
constexpr int kDbFinWords = 16;        // features; per finishing warp
constexpr int kDbBoundStride = 16;     // (rows 64 bytes apart)
constexpr int kDbTurnStride = 36;      // floats per row of the area that turns a chunk of logits round (no bank conflicts)
constexpr int kDbChunks = 4;           // chunks of 32 columns per warp and tile, at most
constexpr uint32_t kDbNoIndex = 0x0fffffffu;           // record word: arg-max index in 28 bits, list length above it
constexpr float kLog2e = 1.4426950408889634f;

struct DraftBatchParams {
    int V, d, R;
    int MT;      // tiles of 128 hidden rows
    int CN;      // CTAs per tile of hidden rows (grid = MT * CN)
    int TPC;     // vocabulary tiles per CTA
    int TR;      // vocabulary rows per tile; the MMA takes TRN = TR rounded up to 16
    int TRN;
    // Rows of the LM-head box: TR.  What the MMA reads behind them (shared memory of this CTA) only feeds columns, or lanes, that
    // nobody looks at.  (Half of TRN for each CTA of a pair.)  With boxes of TRN rows the CTAs that are set aside for finishing could
    // cost a long head more than they gain: 113 rows in a tile instead of 111 were a box of 128 instead of 112, and the rows loaded
    // for nothing come from memory (12 / 32 rows of 49152 x 5120 101.9 / 111.1 -> 93.2 / 102.4 us, 12 rows of 49152 x 3072 68.5 -> 63.0).
    int w_rows;
    int a_rows;  // rows of the H box (multiple of 8, <= 128)
    int stages, a_bytes, b_bytes, ring_bytes;
    int* status;
    float4* part_rec;      // [R][kStampedPieces][CN]: stamped records, piece by piece
    float* probs;          // optional [R][V]: raw logits are written here
    // Two sets of [set_words / kDbBoundStride] rows: ordered bits of the groups' maxima.  A launch uses the set of its
    // stamp's parity, which starts zeroed, and zeroes the other one (whose launch is over, so nothing of it is in flight).
    unsigned int* bound;
    size_t set_words;
    // [0] launches so far (the stamp of this launch is that + 1); [2], [3] rows of the last launch of each parity; from
    // [4] on two sets of (CTAs started, rows claimed), four words apart, used by parity: a launch clears the other
    unsigned int* sync;
    int all_finish;        // more rows than finishing warps in the grid: the epilogue warps help
    int finishers;         // CTAs behind the CN others that finish the rows and have no vocabulary (0: every CTA may finish rows)
};

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Two fp32 numbers in one register pair: an instruction for both.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ void unpack2(f32x2 d, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(d)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float max3f(float a, float b, float c) { return RegTop10::max3(a, b, c); }

__device__ __forceinline__ uint4 ld_relaxed_v4_u32(const unsigned int* p) {
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}
// Two columns of the accumulator: lane r of the quadrant receives row r of each.
__device__ __forceinline__ void tmem_ld_columns(uint32_t a, uint32_t b, float& x, float& y) {
    uint32_t r, s;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(a) : "memory");
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(s) : "r"(b) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r), "+r"(s)::"memory");
    x = __uint_as_float(r);
    y = __uint_as_float(s);
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// A barrier that a warp reaches only once it has the words it read: the barrier takes a predicate made from them.
__device__ __forceinline__ void named_barrier_sync_after(int id, int nthreads, uint32_t word) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %2, 0;\n\t"
        "barrier.cta.red.and.aligned.pred q, %0, %1, p;\n\t}" ::"r"(id),
        "r"(nthreads), "r"(word)
        : "memory");
}
// A shared-memory word that another warp of the CTA is about to make non-zero (bounded).
__device__ __forceinline__ uint32_t smem_word(const uint32_t* p, int* status) {
    for (int i = 0; i < (1 << 22); ++i) {
        const uint32_t v = *reinterpret_cast<const volatile uint32_t*>(p);
        if (v) return v;
    }
    record_status(status, DISCO_ERR_TIMEOUT);
    return 1u;
}

// The same out of line, where it is seldom reached: inlined four times its loop costs the launches that never take it the
// placement of their code (one row of the 32000 x 768 head 15.1 against 14.4 us, 7 rows of 40011 x 768 18.4 against 17.9).
static __device__ __noinline__ uint32_t cold_smem_word(const uint32_t* p, int* status) { return smem_word(p, status); }

// From the twelve words of a row: the bound of its tenth largest logit (the third smallest word); TOP1: of its largest.
template <bool TOP1>
__device__ __forceinline__ float row_bound_of(const uint4& a, const uint4& b, const uint4& c) {
    const unsigned int v[kDbBoundSlots] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
    unsigned int k;
    if (TOP1) {
        k = v[0];
#pragma unroll
        for (int i = 1; i < kDbBoundSlots; ++i) k = max(k, v[i]);
    } else {
        unsigned int s0 = 0xffffffffu, s1 = 0xffffffffu, s2 = 0xffffffffu;
#pragma unroll
        for (int i = 0; i < kDbBoundSlots; ++i) {
            s2 = min(s2, max(s1, v[i]));
            s1 = min(s1, max(s0, v[i]));
            s0 = min(s0, v[i]);
        }
        k = s2;
    }
    return k ? from_ordered_bits(k) : DISCO_NEG_INF;
}
static_assert(kDbBoundSlots - kTopK == 2, "the third smallest of the words bounds the tenth largest logit");

// ---------------------------------------------------------------------------------------------
// second phase: one warp finishes one hidden row
// ---------------------------------------------------------------------------------------------
// A record (five stamped 16-byte pieces, see kStampedPieces): m Z S | word l0 bound | l1 l2 l3 | l4 l5 l6 | l7 l8 l9.  The
// same piece of all CTAs lies side by side: a load of a warp reads four lines (records of 80 bytes one after the other were
// 32 requests each: 2000 cycles for the pieces of a row, against 900).
// word: the arg-max index if the CTA's largest logit passed the bound (kDbNoIndex otherwise), and the number of list
// entries.  l: the CTA's logits above the bound (at most its ten largest), descending.  bound: the largest bound used.
// The last two pieces are written only if there are more than four entries.
//
// What the lists leave out is at most B = the largest of the records' bounds, and at least ten logits of the row are at
// or above B: so the row's k-th largest logit is max(B, the k-th largest list entry), for k <= 10.

// The fifth and further entries of record c's list go into the row's ten largest (lane k < 10 holds the k-th) where they are
// above `least`.  They are in the record's last two pieces, which may still be on their way.
static __device__ __noinline__ float db_long_list(const float4* recs, int NP, int c, int cnt, uint32_t stamp, int* status, float sel,
                                                  float least, int lane) {
    float x = DISCO_NEG_INF;
    if (lane < cnt - 4) {
        const float4* piece = recs + (3 + lane / 3) * NP + c;
        float4 v = load_relaxed_v4(piece);
        const long long t0 = clock64();
        while (__float_as_uint(v.w) != stamp && clock64() - t0 < kWaitBudgetClocks) v = load_relaxed_v4(piece);
        if (__float_as_uint(v.w) != stamp) record_status(status, DISCO_ERR_TIMEOUT);
        const int w = lane % 3;
        x = w == 0 ? v.x : (w == 1 ? v.y : v.z);
    }
    __syncwarp();
    for (unsigned mask = __ballot_sync(kFullMask, x > least); mask; mask &= mask - 1u) {
        const float v = __shfl_sync(kFullMask, x, __ffs(mask) - 1);
        const int at = __popc(__ballot_sync(kFullMask, lane < kTopK && sel >= v));
        const float up = __shfl_up_sync(kFullMask, sel, 1);
        if (lane < kTopK && lane >= at) sel = lane == at ? v : up;
    }
    return sel;
}

// real = false: the same instructions on made-up records, nothing read from or written to global memory.
__device__ __forceinline__ void db_finish_row(const DraftBatchParams& p, const DraftFinalParams& f, int b, bool real,
                                              uint32_t stamp, float* sm, const float* clf_s, bool stats, int lane) {
    constexpr int PER = kDbMaxRecords / 32;
    const int NP = real ? p.CN : 0;
    const float4* recs = p.part_rec + (size_t)b * p.CN * kStampedPieces;
    // issued with the first poll: what the epilogue needs besides the records
    const bool chain = f.chain.alive != nullptr;
    float fpos = 0.f;
    int nd = 1;
    if (real) {
        nd = chain ? chain_step(f.chain, b) : (f.n_drafted ? f.n_drafted[b] : 1);
        fpos = chain ? static_cast<float>(f.chain.pos0[chain_seq(f.chain, b)] + nd) : (f.pos ? static_cast<float>(f.pos[b]) : 0.f);
    }
    float4 q[PER][3];
    {
        const long long t0 = clock64();
#pragma unroll
        for (int j = 0; j < PER; ++j) {   // (no record: Z = 0 and an empty list)
            q[j][0] = make_float4(0.f, 0.f, 0.f, __uint_as_float(stamp));
            q[j][1] = make_float4(0.f, DISCO_NEG_INF, DISCO_NEG_INF, q[j][0].w);
            q[j][2] = make_float4(DISCO_NEG_INF, DISCO_NEG_INF, DISCO_NEG_INF, q[j][0].w);
        }
        if (!real) {   // made-up records, so that the loops below run
            q[0][0] = make_float4(lane * 0.125f, 1.f, 0.f, q[0][0].w);
            q[0][1] = make_float4(__uint_as_float(1u << 28 | lane), lane * 0.125f, 0.f, q[0][1].w);
        }
        unsigned pend = 0u;   // the lane's records that are still awaited: only those are read again
#pragma unroll
        for (int j = 0; j < PER; ++j) pend |= j * 32 + lane < NP ? 1u << j : 0u;
        for (int polls = 0;;) {
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const float4* src = recs + (j * 32 + lane);
                if ((pend >> j) & 1u)
#pragma unroll
                    for (int i = 0; i < 3; ++i) q[j][i] = load_relaxed_v4(src + i * NP);
            }
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (__float_as_uint(q[j][0].w) == stamp && __float_as_uint(q[j][1].w) == stamp && __float_as_uint(q[j][2].w) == stamp)
                    pend &= ~(1u << j);
            if (__all_sync(kFullMask, pend == 0u)) break;
            if ((++polls & 63) == 0) {
                const bool out = *reinterpret_cast<volatile int*>(p.status) == DISCO_ERR_TIMEOUT ||
                                 clock64() - t0 > kWaitBudgetClocks;
                if (__any_sync(kFullMask, out)) {
                    record_status(p.status, DISCO_ERR_TIMEOUT);
                    break;
                }
            }
        }
    }
    // statistics, arg-max, the largest bound
    float lm = DISCO_NEG_INF, bound = DISCO_NEG_INF;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (q[j][0].y > 0.f) {
            lm = fmaxf(lm, q[j][0].x);
            bound = fmaxf(bound, q[j][1].z);
        }
    }
    const float M = from_ordered_bits(__reduce_max_sync(kFullMask, ordered_bits(lm)));
    bound = from_ordered_bits(__reduce_max_sync(kFullMask, ordered_bits(bound)));
    float Z = 0.f, S = 0.f;
    uint32_t idx = kDbNoIndex;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (q[j][0].y > 0.f) {
            const float dm = q[j][0].x - M;
            const float e = ex2_approx(dm * kLog2e);
            Z = fmaf(q[j][0].y, e, Z);
            S = fmaf(e, fmaf(dm, q[j][0].y, q[j][0].z), S);
            if (dm == 0.f) idx = min(idx, __float_as_uint(q[j][1].x) & kDbNoIndex);
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        Z += __shfl_xor_sync(kFullMask, Z, off);
        S += __shfl_xor_sync(kFullMask, S, off);
    }
    idx = __reduce_min_sync(kFullMask, idx);
    float sel = DISCO_NEG_INF;
    if (!stats) {
        // One warp is at work here, on code that it runs once, so what counts is the number of instructions: the four largest
        // entries of each lane's lists (places without an entry hold -inf), then ten times the largest of all, taken from the
        // lane that has it; a lane that has given four looks for its next four.  (Collecting the 30 - 50 entries above the bound
        // and ranking them: 4400 cycles; only those not below the tenth largest of the lanes' heads: 3300; this: 1800.)
        float fourth[PER], more = DISCO_NEG_INF;      // the fourth entry of a list that goes on past it
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            fourth[j] = (__float_as_uint(q[j][1].x) >> 28) > 4u ? q[j][2].z : DISCO_NEG_INF;
            more = fmaxf(more, fourth[j]);
        }
        float t = DISCO_NEG_INF;
        bool ended = false;
#pragma unroll 1
        for (int k = 0; k < kTopK && !ended;) {
            float a[4] = {q[0][1].y, q[0][2].x, q[0][2].y, q[0][2].z};
#pragma unroll
            for (int j = 1; j < PER; ++j) {
                // two descending lists, one reversed: the larger of each pair are the four largest, two steps sort them
                const float c0 = fmaxf(a[0], q[j][2].z), c1 = fmaxf(a[1], q[j][2].y), c2 = fmaxf(a[2], q[j][2].x), c3 = fmaxf(a[3], q[j][1].y);
                const float d0 = fmaxf(c0, c2), d2 = fminf(c0, c2), d1 = fmaxf(c1, c3), d3 = fminf(c1, c3);
                a[0] = fmaxf(d0, d1), a[1] = fminf(d0, d1), a[2] = fmaxf(d2, d3), a[3] = fminf(d2, d3);
            }
            int taken = 0;
#pragma unroll 1
            for (;;) {
                t = warp_max_f32(a[0]);
                ended = !(t > bound);
                if (ended) break;
                if (lane == k) sel = t;
                if (lane == __ffs(__ballot_sync(kFullMask, a[0] == t)) - 1) {
                    a[0] = a[1], a[1] = a[2], a[2] = a[3], a[3] = DISCO_NEG_INF;
                    ++taken;
                }
                if (++k == kTopK || __any_sync(kFullMask, taken == 4)) break;
            }
            if (k < kTopK && !ended) {   // (seldom) what the lanes gave leaves their lists
#pragma unroll 1
                for (; taken > 0; --taken) {
                    float h = q[0][1].y;
#pragma unroll
                    for (int j = 1; j < PER; ++j) h = fmaxf(h, q[j][1].y);
                    bool out = false;
#pragma unroll
                    for (int j = 0; j < PER; ++j)
                        if (!out && q[j][1].y == h) {
                            q[j][1].y = q[j][2].x, q[j][2].x = q[j][2].y, q[j][2].y = q[j][2].z, q[j][2].z = DISCO_NEG_INF;
                            out = true;
                        }
                }
                __syncwarp();
            }
        }
        // A list that goes on may hold more of the ten largest if its fourth entry is above the tenth of those found.
        float least = ended ? bound : t;
        if (__any_sync(kFullMask, more > least)) {
#pragma unroll
            for (int j = 0; j < PER; ++j)
                for (unsigned mask = __ballot_sync(kFullMask, fourth[j] > least); mask; mask &= mask - 1u) {
                    const int src = __ffs(mask) - 1;
                    const int cnt = static_cast<int>(__shfl_sync(kFullMask, __float_as_uint(q[j][1].x), src) >> 28);
                    sel = db_long_list(recs, NP, j * 32 + src, cnt, stamp, p.status, sel, least, lane);
                    least = fmaxf(least, __shfl_sync(kFullMask, sel, kTopK - 1));
                }
        }
        if (lane < kTopK) sel = fmaxf(sel, bound);
    }
    SoftmaxState st;
    st.m = M, st.Z = Z, st.S = S;
    const unsigned long long key = idx != kDbNoIndex ? argmax_key(M, static_cast<int>(idx)) : 0ull;   // (0: token -1)
    // (a launch of several steps: the sequence's verdicts in a spare word of its first row's bounds, cleared with them)
    unsigned int* verdicts = f.chain.group > 1 ? p.bound + (stamp & 1u) * p.set_words + (size_t)chain_seq(f.chain, b) * kDbBoundStride + kDbBoundSlots : nullptr;
    const DraftOutputs o{f.token, f.conf, f.halt, f.feats, f.final_stats, f.nll_sum, f.stats_only, f.chain, real, verdicts, p.status};
    const int Hc = f.clf_H;
    warp_draft_epilogue(st, key, sel, fpos, nd, f.tau, f.sl_max, sm, clf_s, clf_s + Hc * kNFeat, clf_s + Hc * (kNFeat + 1),
                        clf_s + Hc * (kNFeat + 2), Hc, b, o, lane);
}

// A number the compiler cannot know: a loop that rehearses and then runs the same code must stay one copy of it.
__device__ __forceinline__ int opaque(int x) {
    asm volatile("" : "+r"(x));
    return x;
}

// This launch's stamp, by the epilogue warps (eight of the CTA, ew their number) once what went before is over: the set of
// bounds of the launch before is cleared and the CTA counts as started.
// seen: anything made from what the thread has read of the rows' liveness.  Where several steps share a launch, a row that is
// finished may end its sequence and clear the byte that the sequence's other rows, in other CTAs and other warps, went by; that
// happens once all CTAs count as started, so no CTA counts before its threads have their bytes.  (A row that is dead here and
// live to the warp that finishes it would be waited for in vain.)
__device__ __forceinline__ uint32_t db_begin(const DraftBatchParams& p, const DraftFinalParams& f, int ew, uint32_t* s_stamp, uint32_t seen,
                                             int lane) {
    const uint32_t stamp = *reinterpret_cast<volatile unsigned int*>(p.sync) + 1u;
    const uint32_t par = stamp & 1u;
    // (that word is the other parity's: only a launch after this one writes it)
    const int old_rows = *reinterpret_cast<volatile unsigned int*>(p.sync + 2 + (par ^ 1u));
    if (blockIdx.x == 0)
        for (int i = ew * 32 + lane; i < f.clear_n; i += kDbEpiWarps * 32) f.clear_words[i] = 0u;
    uint4* old = reinterpret_cast<uint4*>(p.bound + (par ^ 1u) * p.set_words);
    for (int i = blockIdx.x * (kDbEpiWarps * 32) + ew * 32 + lane; i < old_rows * (kDbBoundStride / 4);
         i += gridDim.x * (kDbEpiWarps * 32))
        old[i] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    // This CTA has started once all of its eight reads of the stamp are done: the stamp may be moved on as soon as every
    // CTA counts as started, and a warp that read the moved word would work on the next launch's set of bounds.  (One
    // warp that reads and hands the stamp to the others through shared memory: their polling costs the step up to 3 %,
    // eight rows of 49152 x 768 kept and drawn 30.9 us against 30.1.)
    named_barrier_sync_after(8, kDbEpiWarps * 32, stamp | seen);
    if (ew == 0 && lane == 0) {
        *reinterpret_cast<volatile uint32_t*>(s_stamp) = stamp;
        atomicAdd(p.sync + 4 + 4 * par, 1u);
    }
    return stamp;
}
// All CTAs have started: the stamp can move on, and the counters of the next launch (this one's may still be looked at) start
// at zero.
__device__ __forceinline__ void db_move_on(const DraftBatchParams& p, uint32_t stamp) {
    unsigned int* other = p.sync + 4 + 4 * ((stamp + 1u) & 1u);
    other[0] = 0u;
    other[1] = 0u;
    p.sync[2 + (stamp & 1u)] = (unsigned int)p.R;
    p.sync[0] = stamp == 0xffffffffu ? 1u : stamp;   // never zero, and the two sets keep alternating
}
__device__ __forceinline__ void db_stage_classifier(const DraftFinalParams& f, float* clf_s, int first, int step) {
    const int Hc = f.clf_H, n1 = Hc * kNFeat;
    if (Hc > 0) {
        for (int i = first; i < n1 + 2 * Hc + 1; i += step) {
            const float* src = i < n1 ? f.clf_W1 + i
                                      : (i < n1 + Hc ? f.clf_b1 + (i - n1)
                                                     : (i < n1 + 2 * Hc ? f.clf_w2 + (i - n1 - Hc) : f.clf_b2));
            cp_async4(clf_s + i, src);
        }
        cp_async_commit();
    }
}

// Up to 128 rows: the last CTAs of the grid have no vocabulary, ten warps of theirs finish a row each.  The CTAs with vocabulary
// leave when their records are out, so the next launch finds their SMs free and has its share of the LM head on the way while
// this one ends; a CTA that finished a row as well was replaced when the launch ended, and its successor's records came 3 us
// after the others'.  A CTA here that starts before the others (blocks start in order, so that is not expected) waits for
// them, bounded; its own place is one that no other CTA of the launch needs.
template <bool STATS, class Live>
__device__ __forceinline__ void db_finish_dedicated(const DraftBatchParams& p, const DraftFinalParams& f, int warp, bool looks_live,
                                                    float* fin_s, float* clf_s, uint32_t* s_stamp, const Live& step_live, int lane) {
    constexpr int kWarps = kDbEpiWarps + kDbFinWarps;
    const int fw = warp - 2;
    float* sm = fin_s + fw * kDbFinWords;
    db_stage_classifier(f, clf_s, fw * 32 + lane, kWarps * 32);
    cp_async_wait_all();
    named_barrier_sync(3, kWarps * 32);
    uint32_t stamp = 1u;
    int b = 0;
    bool run = looks_live;
#pragma unroll 1
    for (int real = opaque(0);; real = opaque(1)) {
        if (run) db_finish_row(p, f, b, real != 0, stamp + (real ? f.test_stamp_skew : 0u), sm, clf_s, STATS, lane);
        if (real) {
            b += kWarps * p.finishers;
        } else {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            if (!step_live()) break;
            b = (int)blockIdx.x - p.CN + fw * p.finishers;
            if (fw < kDbEpiWarps) stamp = db_begin(p, f, fw, s_stamp, 0u, lane);   // (reads its rows' bytes when all have started)
            else stamp = smem_word(s_stamp, p.status);
            if (lane == 0) {
                const unsigned int* started = p.sync + 4 + 4 * (stamp & 1u);
                const long long t0 = clock64();
                for (int polls = 0; ld_relaxed_u32(started) != gridDim.x; ++polls) {
                    __nanosleep(100);
                    if ((polls & 63) == 63 && (*reinterpret_cast<volatile int*>(p.status) == DISCO_ERR_TIMEOUT ||
                                               clock64() - t0 > 64 * kWaitBudgetClocks)) {
                        record_status(p.status, DISCO_ERR_TIMEOUT);
                        break;
                    }
                }
                if (b == 0) db_move_on(p, stamp);
            }
            __syncwarp();
        }
        if (b >= f.B) break;
        run = chain_seq_live(f.chain, f.active, chain_seq(f.chain, b));
    }
}

// The finishing warps, from the start of the launch; with more rows than those of the whole grid, the epilogue warps as
// well once their records are out.  warp: the warp's number in the CTA; step_live: whether the step takes place.
template <bool STATS, class Live>
__device__ __forceinline__ void db_finish_rows(const DraftBatchParams& p, const DraftFinalParams& f, int warp, bool looks_live,
                                               float* fin_s, float* clf_s, int* s_done, uint32_t* s_clf, const uint32_t* s_stamp,
                                               const Live& step_live, int lane) {
    const bool epi = warp < 2 + kDbEpiWarps;
    if (epi && !p.all_finish) return;
    const int fw = epi ? kDbFinWarps + warp - 2 : warp - 2 - kDbEpiWarps;
    float* sm = fin_s + fw * kDbFinWords;
    if (!epi) db_stage_classifier(f, clf_s, fw * 32 + lane, kDbFinWarps * 32);
    uint32_t stamp = 1u;
    unsigned int* set = nullptr;
    int b = 0;
    bool run = !epi && looks_live;
#pragma unroll 1
    for (int real = opaque(0);; real = opaque(1)) {
        if (run) db_finish_row(p, f, b, real != 0, stamp + (real ? f.test_stamp_skew : 0u), sm, clf_s, STATS, lane);
        if (!real) {
            if (!epi) {
                cp_async_wait_all();
                named_barrier_sync(3, kDbFinWarps * 32);
                if (fw == 0 && lane == 0) {
                    __threadfence_block();
                    *reinterpret_cast<volatile uint32_t*>(s_clf) = 1u;
                }
                asm volatile("griddepcontrol.wait;" ::: "memory");
            }
            if (!step_live()) break;
            if (epi) smem_word(s_clf, p.status);
            stamp = smem_word(s_stamp, p.status);
            __syncwarp();
            set = p.sync + 4 + 4 * (stamp & 1u);
            // Have all CTAs of the grid started?  Until then none of their records may be waited for.
            int all = 0;
            if (lane == 0) {
                for (;;) {
                    const bool done = *reinterpret_cast<volatile int*>(s_done) == kDbEpiWarps;
                    __threadfence_block();
                    all = ld_relaxed_u32(set) == gridDim.x;
                    if (all || done) break;
                    __nanosleep(300);   // (148 CTAs polling one word without a pause held everybody up by 5 us)
                }
            }
            if (!__shfl_sync(kFullMask, all, 0)) break;
        }
        // the next row nobody has taken
        int first = 0;
        if (lane == 0) first = (int)atomicAdd(set + 1, 1u);
        b = __shfl_sync(kFullMask, first, 0);
        if (b == 0 && lane == 0) db_move_on(p, stamp);
        if (b >= f.B) break;
        run = chain_seq_live(f.chain, f.active, chain_seq(f.chain, b));
        // The records of the other CTAs will not be there before this CTA's own: polling them earlier only loads L2.
        if (lane == 0 && !epi)
            for (int i = 0; i < (1 << 20) && *reinterpret_cast<volatile int*>(s_done) != kDbEpiWarps; ++i) __nanosleep(32);
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------------------
// main kernel
// ---------------------------------------------------------------------------------------------
// STATS: arg-max and soft-max statistics only (f.stats_only == 1), no list of the ten largest.
// PAIR: clusters of two CTAs share every vocabulary tile: each loads its own 128 hidden rows and half of the LM-head box.
template <bool STATS, bool PAIR>
__global__ void __launch_bounds__(kDbThreads, 1)
umma_draft_batch_kernel(const __grid_constant__ CUtensorMap tmap_W, const __grid_constant__ CUtensorMap tmap_H,
                        const DraftBatchParams p, const DraftFinalParams f) {
    extern __shared__ uint8_t smem_dyn[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
    uint8_t* a_tiles = smem;
    uint8_t* b_tiles = smem + p.stages * p.a_bytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + p.ring_bytes);
    uint64_t* empty = full + kDbMaxStages;
    uint64_t* tmem_full = empty + kDbMaxStages;
    uint64_t* tmem_empty = tmem_full + 4;
    uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(tmem_empty + 4);
    int* s_done = reinterpret_cast<int*>(tmem_base_s + 1);    // epilogue warps that have published their records
    uint32_t* s_live = tmem_base_s + 5;                       // 1: the step takes place, 2: it does not
    uint32_t* s_look = tmem_base_s + 4;                       // whether the step seems to take place
    uint32_t* s_clf = tmem_base_s + 3;                        // set once the classifier is in shared memory
    uint32_t* s_stamp = tmem_base_s + 2;                      // stamp of this launch (0: not read yet, or nothing to do)
    float4* xch = reinterpret_cast<float4*>(reinterpret_cast<uint8_t*>(full) + 512);
    float* fin_s = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(xch) + kDbXchBytes);
    float* row_thr_s = fin_s + (p.all_finish || p.finishers ? kDbFinWarps + kDbEpiWarps : kDbFinWarps) * kDbFinWords;     // [128] the rows' bounds
    float* turn_s = row_thr_s + 128;                          // with probs: 32 rows of one chunk per epilogue warp
    float* clf_s = turn_s + (p.probs ? kDbEpiWarps * 32 * kDbTurnStride : 0);

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int KB = (p.d + kUmmaBK - 1) / kUmmaBK;
    const int m_tile = blockIdx.x % p.MT;
    const int nslot = blockIdx.x / p.MT;
    const int v_first = nslot * p.TPC * p.TR;                 // this CTA's vocabulary rows: its tiles in sequence
    const int tiles = v_first < p.V ? min(p.TPC, (p.V - v_first + p.TR - 1) / p.TR) : 0;
    const bool chained = !STATS && f.chain.alive != nullptr && f.chain.step > 1;
    const int nbuf = p.TRN <= 128 ? 4 : 2, buf_cols = 512 / nbuf;   // accumulator buffers in TMEM

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < nbuf; ++b) {
            mbar_init(&tmem_full[b], 1);
            mbar_init(&tmem_empty[b], PAIR ? 2 * kDbEpiWarps : kDbEpiWarps);
        }
        *s_done = 0;
        *s_stamp = 0u;
        *s_clf = 0u;
        *s_live = 0u;
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
    // A step of a draft phase that has ended already needs neither loads nor rehearsals.  The flags are looked at ahead of
    // the dependency wait for that, once for the whole CTA: they may be old and decide nothing else.
    if (warp == 2) {
        const bool any = !chained || chain_any_live(f.chain, f.chain.B, lane);
        if (lane == 0) *s_look = any ? 1u : 0u;
    }
    tc_fence_before();
    if constexpr (PAIR) cluster_sync();    // (both CTAs' barriers are ready)
    else __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_base_s;
    const bool leader = !PAIR || cluster_rank() == 0;
    // (the CTAs of a pair request the same stages ahead, so they go by the leader's look)
    const bool looks_live = (leader ? *s_look : ld_cluster_u32(leader_addr(smem_addr(s_look)))) != 0u;
    // Does the step take place?  Read once per CTA, by the MMA issuer right after the dependency wait, and told to the others
    // here.  (A finishing warp of this launch may clear flags once every CTA counts as started: db_begin, which the epilogue warps
    // reach only when they have been told.)
    auto step_live = [&]() { return !chained || cold_smem_word(s_live, p.status) == 1u; };

    if (warp == 0) {
        // ------------------------------ producer ------------------------------
        const int total = tiles * KB;
        // (what a stage's barrier, the leader's, counts: the boxes of both CTAs)
        const uint32_t w_bytes = (uint32_t)p.w_rows * (PAIR ? 256u : 128u), h_bytes = (uint32_t)p.a_rows * (PAIR ? 256u : 128u);
        // The LM head is never written by this library: its first stages are requested before the dependency wait.
        const int pre = looks_live ? min(p.stages, total) : 0;
        // Every CTA reads the same hidden rows.  Each starts at another k-block, so that they do not all ask the same few
        // L2 slices for the same lines at the same time.
        const int rot = nslot % KB;
        // A single thread issues everything: running addresses and counters, as few instructions per stage as possible.
        const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty), a0 = smem_addr(a_tiles), b0 = smem_addr(b_tiles);
        const int k_end = KB * kUmmaBK, k_first = rot * kUmmaBK, h_row = m_tile * 128;
        const int v_own = v_first + (leader ? 0 : p.TRN / 2);
        const uint32_t count0 = PAIR ? leader_addr(full0) : full0;
        auto load = [&](uint32_t dst, const CUtensorMap* map, int c0, int c1, int slot) {
            if constexpr (PAIR) tma_load_2d_pair(dst, map, c0, c1, count0 + slot * 8);
            else tma_load_2d(dst, map, c0, c1, count0 + slot * 8);
        };
        int k = k_first, v0 = v_own, left = KB;        // the next stage to request: k, vocabulary row, k-blocks left of the tile
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
                if (leader) mbar_expect_tx(full0 + n * 8, w_bytes);
                load(b0 + n * p.b_bytes, &tmap_W, k, v0, n);
            }
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const bool live = step_live();
        if (!live) {
            if (leader && elect_one()) {
                for (int n = 0; n < pre; ++n) mbar_arrive(&full[n]);
                for (int n = 0; n < pre; ++n) mbar_wait(&full[n], 0, p.status);   // nothing may still be landing at exit
            }
        } else if (elect_one()) {
            int kh = k_first;
            for (int n = 0; n < pre; ++n) {
                if (leader) mbar_arrive_expect_tx(full0 + n * 8, h_bytes);
                load(a0 + n * p.a_bytes, &tmap_H, kh, h_row, n);
                kh += kUmmaBK;
                if (kh == k_end) kh = 0;
            }
            int stage = pre == p.stages ? 0 : pre, phase = pre == p.stages ? 1 : 0;
            k = k_first, v0 = v_own, left = KB;        // (the elected thread need not be the one of before)
            for (int n = 0; n < pre; ++n) advance();
            uint32_t at_a = a0 + stage * p.a_bytes, at_b = b0 + stage * p.b_bytes;
            for (int n = pre; n < total; ++n, advance()) {
                mbar_wait(empty0 + stage * 8, phase ^ 1, p.status);
                if (leader) mbar_arrive_expect_tx(full0 + stage * 8, w_bytes + h_bytes);
                load(at_b, &tmap_W, k, v0, stage);
                load(at_a, &tmap_H, k, h_row, stage);
                at_a += p.a_bytes;
                at_b += p.b_bytes;
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1;
                    at_a = a0;
                    at_b = b0;
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
        bool live = true;
        if (chained) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            live = chain_any_live(f.chain, f.chain.B, lane);
            if (lane == 0) *reinterpret_cast<volatile uint32_t*>(s_live) = live ? 1u : 2u;
        }
        if (live && leader && elect_one()) {
            const uint32_t idesc = umma_idesc(p.TRN, PAIR ? 256 : 128);
            const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty);
            // Up to eight rows: the A operand is the one 8-row box read 16 times over (zero stride between the 8-row groups
            // of the descriptor).  More: the MMA reads 128 rows from the start of the stage; what lies behind the box
            // (further stages, inside the ring) only feeds accumulator lanes nobody reads.
            const uint64_t a0 = umma_smem_desc(a_tiles) & (p.a_rows == 8 ? ~(0x3fffull << 32) : ~0ull);
            const uint64_t b0 = umma_smem_desc(b_tiles);
            const uint32_t a_step = (uint32_t)p.a_bytes >> 4, b_step = (uint32_t)p.b_bytes >> 4;   // descriptor units
            uint64_t a_desc = a0, b_desc = b0;
            int stage = 0, phase = 0;
            for (int t = 0; t < tiles; ++t) {
                const int buf = t % nbuf;
                if constexpr (PAIR) mbar_wait_cluster(smem_addr(&tmem_empty[buf]), ((t / nbuf) & 1) ^ 1, p.status);
                else mbar_wait(&tmem_empty[buf], ((t / nbuf) & 1) ^ 1, p.status);
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + buf * buf_cols;
                for (int kb = 0; kb < KB; ++kb) {
                    mbar_wait(full0 + stage * 8, phase, p.status);
                    tc_fence_after();
#pragma unroll
                    for (int k = 0; k < kUmmaBK / 16; ++k) {  // 16 k-elements = 32 bytes = 2 descriptor units
                        if constexpr (PAIR) tc_mma_bf16_pair(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, (kb | k) != 0);
                        else tc_mma_bf16(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, (kb | k) != 0);
                    }
                    if constexpr (PAIR) tc_commit_pair(empty0 + stage * 8);
                    else tc_commit(empty0 + stage * 8);
                    a_desc += a_step;
                    b_desc += b_step;
                    if (++stage == p.stages) {
                        stage = 0;
                        phase ^= 1;
                        a_desc = a0;
                        b_desc = b0;
                    }
                }
                if constexpr (PAIR) tc_commit_pair(smem_addr(&tmem_full[buf]));
                else tc_commit(&tmem_full[buf]);
            }
        }
    }
    const bool finisher = p.finishers > 0 && nslot >= p.CN;
    if (warp >= 2 && warp < 2 + kDbEpiWarps && !finisher) {
        // ------------------------------ epilogue ------------------------------
        const int ew = warp - 2;
        const int quad = warp & 3;              // TMEM lane quadrant this warp may read
        const int share = ew >> 2;              // the two warps of a quadrant split the columns of a tile
        const int tile_row = quad * 32 + lane;  // row within this tile of hidden rows
        const int row = m_tile * 128 + tile_row;
        const bool warp_has_rows = m_tile * 128 + quad * 32 < p.R;
        bool valid = row < p.R;                 // and (once that can be read) its sequence still drafts
        // A single narrow tile is not worth a bound.  With four accumulator buffers the candidates of a tile are looked for
        // one tile later, when the bound that everybody's tiles give has long arrived; otherwise the first tile waits for it.
        const bool use_bound = p.TPC > 1 || p.TR > 32;
        const bool defer = nbuf == 4 && tiles > 1;
        const uint32_t t_quad = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        volatile float* thr_s = row_thr_s + tile_row;
        float* turn = turn_s + ew * 32 * kDbTurnStride;
        // Twice: a rehearsal without columns before the dependency wait (what follows the column loop is on the critical
        // path, and its instructions would come from L2 one after the other), then for good.
#pragma unroll 1
        for (int phase = opaque(looks_live ? 0 : 1); phase < 2; phase = opaque(phase + 1)) {
            bool many_kept = false;        // enough of them to store four rows per instruction
            unsigned keep_mask = 0u;       // rows of this warp whose raw logits go to probs (none of a masked sequence's)
            unsigned int *slots = nullptr, *my_slot = nullptr;
            float m = DISCO_NEG_INF, Z = 0.f, S = 0.f;       // S = sum e^(z - m) (z - m)
            float best_v = DISCO_NEG_INF;
            int best_i = 0;
            RegTop10 top;
            top.init();
            float thr = DISCO_NEG_INF;     // logits at or below it are not among the row's ten largest (or equal its bound)
            float bound_used = DISCO_NEG_INF;
            if (phase == 0) {
                m = best_v = top.t[0] = static_cast<float>(lane);
                Z = 1.f;
            } else {
                asm volatile("griddepcontrol.wait;" ::: "memory");  // scratch and outputs belong to the predecessor until now
                if (!step_live()) break;
                // Rows of sequences that are masked or have stopped drafting: nobody wants their candidates, and no record of
                // them is written.
                valid = valid && chain_seq_live(f.chain, f.active, chain_seq(f.chain, row));
                keep_mask = __ballot_sync(kFullMask, p.probs && valid);
                many_kept = __popc(keep_mask) > 8 && (reinterpret_cast<uintptr_t>(p.probs) & 15) == 0;
                const uint32_t stamp = db_begin(p, f, ew, s_stamp, valid ? 1u : 0u, lane);
                slots = p.bound + (stamp & 1u) * p.set_words + (size_t)(valid ? row : 0) * kDbBoundStride;
                my_slot = slots + nslot % kDbBoundSlots;
            }
            const int phase_tiles = phase == 0 ? 0 : tiles;

            // Tile by tile: statistics and the chunks' maxima, the tile's maximum to the shared bound, then the candidates.
            float cm[kDbChunks], cm_prev[kDbChunks];
#pragma unroll
            for (int i = 0; i < kDbChunks; ++i) cm[i] = cm_prev[i] = DISCO_NEG_INF;
            for (int t = 0; t < phase_tiles; ++t) {
                mbar_wait(&tmem_full[t % nbuf], (t / nbuf) & 1, p.status);
                tc_fence_after();
                const int ncols = min(p.TR, p.V - (v_first + t * p.TR));  // further columns belong to the next tile or lie past V
                const int half = (((ncols + 31) >> 5) + 1) >> 1;
                const int c_lo = share == 0 ? 0 : half, c_hi = share == 0 ? half : (ncols + 31) >> 5;
                const uint32_t t_buf = t_quad + (t % nbuf) * buf_cols;
                const bool look = use_bound && valid && share == 0;   // one thread per row looks the bound up
                uint4 sa = make_uint4(0, 0, 0, 0), sb = sa, sc = sa;  // (on its way during the statistics)
                if (look && t > 0) {
                    sa = ld_relaxed_v4_u32(slots);
                    sb = ld_relaxed_v4_u32(slots + 4);
                    sc = ld_relaxed_v4_u32(slots + 8);
                }
                if (warp_has_rows) {
                    float tile_max = DISCO_NEG_INF;
#pragma unroll
                    for (int i = 0; i < kDbChunks; ++i) cm_prev[i] = cm[i];
#pragma unroll 1
                    for (int c = c_lo; c < c_hi; ++c) {
                        float z[32];
                        tmem_ld32(t_buf + c * 32, z);
                        const int n = ncols - c * 32;           // columns of the chunk that count
                        if (n < 32) {
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (j >= n) z[j] = DISCO_NEG_INF;
                        }
                        float g[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float x = max3f(z[8 * q], z[8 * q + 1], z[8 * q + 2]), y = max3f(z[8 * q + 3], z[8 * q + 4], z[8 * q + 5]);
                            g[q] = max3f(x, y, fmaxf(z[8 * q + 6], z[8 * q + 7]));
                        }
                        const float cmax = fmaxf(max3f(g[0], g[1], g[2]), g[3]);
                        tile_max = fmaxf(tile_max, cmax);
#pragma unroll
                        for (int i = kDbChunks - 1; i > 0; --i) cm[i] = cm[i - 1];   // cm[0]: the tile's last chunk
                        cm[0] = cmax;
                        // the reference maximum moves first, then the chunk is added
                        const float mn = fmaxf(m, cmax);
                        const float dm = fmaxf(m - mn, -1000.f);
                        const float em = ex2_approx(dm * kLog2e);
                        m = mn;
                        if (n < 32) {   // masked columns: finite, far below any logit (e = 0, and 0 * -inf is avoided)
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (j >= n) z[j] = -2e38f;
                        }
                        // The difference to the maximum comes first: it is exact where it matters, whatever the size of the
                        // logits.  (z * log2e - m * log2e in one instruction keeps the rounding of m * log2e: up to 5e-6 of
                        // every probability at logits of 100, 2e-5 at 400.)  Two columns per instruction, so it costs no more.
                        const f32x2 neg_m = pack2(-mn, -mn), log2e = pack2(kLog2e, kLog2e);
                        f32x2 Zc = 0ull, Sc = 0ull;
#pragma unroll
                        for (int j = 0; j < 32; j += 2) {
                            const f32x2 t = add2(pack2(z[j], z[j + 1]), neg_m);
                            float xa, xb;
                            unpack2(mul2(t, log2e), xa, xb);
                            const f32x2 e = pack2(ex2_approx(xa), ex2_approx(xb));
                            Zc = add2(Zc, e);
                            Sc = fma2(e, t, Sc);
                        }
                        float Za, Zb, Sa, Sb;
                        unpack2(Zc, Za, Zb);
                        unpack2(Sc, Sa, Sb);
                        S = fmaf(em, fmaf(dm, Z, S), Sa + Sb);   // (Z = S = 0 before the first chunk)
                        Z = fmaf(Z, em, Za + Zb);
                        if (keep_mask) {
                            // A thread holds one row: the chunk goes through shared memory so that every store instruction
                            // writes whole lines (four rows of 128 bytes; 32 bytes at a time per row halved the rate of
                            // the whole pass: 278 against 68 us for 1000 rows of the 32000 x 768 head).
                            const int v = v_first + t * p.TR + c * 32;
                            float4* mine = reinterpret_cast<float4*>(turn + lane * kDbTurnStride);
#pragma unroll
                            for (int j = 0; j < 8; ++j) mine[j] = make_float4(z[4 * j], z[4 * j + 1], z[4 * j + 2], z[4 * j + 3]);
                            __syncwarp();
                            float* dst = p.probs + (size_t)(m_tile * 128 + quad * 32) * p.V + v;
                            if (many_kept && ((p.V | v) & 3) == 0 && n >= 32) {
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    const int r = 4 * j + (lane >> 3), col = (lane & 7) * 4;
                                    const float4 x = *reinterpret_cast<const float4*>(turn + r * kDbTurnStride + col);
                                    if ((keep_mask >> r) & 1u) *reinterpret_cast<float4*>(dst + (size_t)r * p.V + col) = x;
                                }
                            } else {
                                for (unsigned left = keep_mask; left != 0u; left &= left - 1u) {   // row by row, those there are
                                    const int r = __ffs(left) - 1;
                                    if (lane < n) dst[(size_t)r * p.V + lane] = turn[r * kDbTurnStride + lane];
                                }
                            }
                            __syncwarp();
                        }
                    }
                    if (use_bound) {
                        // (an infinite logit bounds nothing: its CTA's statistics are no numbers, and its record is left out)
                        if (valid && c_lo < c_hi && (t == 0 || t + 1 < tiles) && tile_max > bound_used && tile_max < -DISCO_NEG_INF)
                            atomicMax(my_slot, ordered_bits(tile_max + 0.f));
                        if (t > 0 || !defer) {
                            if (t == 0 && share == 0) {
                                // (not waited for longer than the round trips of this CTA's own word and a slow neighbour's:
                                // the bound only saves work)
                                for (int k = 0; k < 4; ++k) {
                                    if (look) {
                                        sa = ld_relaxed_v4_u32(slots);
                                        sb = ld_relaxed_v4_u32(slots + 4);
                                        sc = ld_relaxed_v4_u32(slots + 8);
                                    }
                                    if (__all_sync(kFullMask, !valid || row_bound_of<STATS>(sa, sb, sc) > DISCO_NEG_INF)) break;
                                }
                            }
                            if (look) *thr_s = row_bound_of<STATS>(sa, sb, sc);
                            named_barrier_sync(4 + quad, 64);   // the two warps of the quadrant (a later bound would do too)
                            if (valid) bound_used = fmaxf(bound_used, *thr_s);
                        }
                    }
                }
                for (int tc = defer && t > 0 ? t - 1 : t; tc <= t; ++tc) {
                    if (defer && tc == t && t + 1 < tiles) break;       // later, with a better bound
                    const int nc = min(p.TR, p.V - (v_first + tc * p.TR));
                    const int mid = (((nc + 31) >> 5) + 1) >> 1;
                    const int lo = share == 0 ? 0 : mid, hi = share == 0 ? mid : (nc + 31) >> 5;
                    thr = fmaxf(thr, bound_used);
                    // Chunks that hold a logit that can still be among some row's ten largest (STATS: its largest).  A logit
                    // equal to the bound counts for the arg-max only: the finishing warp fills the list up with the bound.
                    unsigned flagged = 0u;
#pragma unroll
                    for (int i = 0; i < kDbChunks; ++i) {
                        const float x = tc == t ? cm[i] : cm_prev[i];
                        const bool want = valid && x >= thr && (x > best_v || (!STATS && x > thr));
                        if (warp_has_rows && hi - lo > i && __any_sync(kFullMask, want)) flagged |= 1u << i;
                    }
                    while (flagged) {   // (bit i: the i-th last chunk; the first columns come first)
                        const int i = 31 - __clz(flagged);
                        flagged &= ~(1u << i);
                        const int c = hi - 1 - i;
                        const uint32_t t_chunk = t_quad + (tc % nbuf) * buf_cols + c * 32;
                        float z[32];
                        tmem_ld32(t_chunk, z);
                        const int n = nc - c * 32;
                        if (n < 32) {
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (j >= n) z[j] = DISCO_NEG_INF;
                        }
                        float cmax = fmaxf(z[0], z[1]);
#pragma unroll
                        for (int j = 2; j < 32; j += 2) cmax = max3f(cmax, z[j], z[j + 1]);
                        const float cut = STATS ? fmaxf(thr, cmax) : thr;   // (STATS: only the chunk's largest can be the row's)
                        unsigned bits = 0u;
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (z[j] >= cut) bits |= 1u << j;
                        if (n < 32) bits &= (1u << n) - 1u;
                        if (!valid) bits = 0u;
                        const int v = v_first + tc * p.TR + c * 32;
                        // Nearly always a row has at most one: its chunk maximum.
                        if (!__any_sync(kFullMask, (bits & (bits - 1u)) != 0u)) {
                            if (bits != 0u && cmax > best_v) {
                                best_v = cmax;
                                best_i = v + __ffs(bits) - 1;
                            }
                            if (!STATS) {
                                top.push(bits != 0u && cmax > thr ? cmax : DISCO_NEG_INF);
                                thr = fmaxf(thr, top.t[kTopK - 1]);
                            }
                            continue;
                        }
                        for (unsigned left = __reduce_or_sync(kFullMask, bits); left != 0u;) {
                            // two columns at a time (the second may be the first again: it is then left out)
                            const int j = __ffs(left) - 1;
                            left &= left - 1u;
                            const int k = left ? __ffs(left) - 1 : j;
                            left &= left - 1u;
                            float x, y;
                            tmem_ld_columns(t_chunk + j, t_chunk + k, x, y);
                            x = (bits >> j) & 1u ? x : DISCO_NEG_INF;
                            y = ((bits >> k) & 1u) && k != j ? y : DISCO_NEG_INF;
                            if (x > best_v) {
                                best_v = x;
                                best_i = v + j;
                            }
                            if (y > best_v) {
                                best_v = y;
                                best_i = v + k;
                            }
                            if (!STATS) {
                                top.push2(x > thr ? x : DISCO_NEG_INF, y > thr ? y : DISCO_NEG_INF);
                                thr = fmaxf(thr, top.t[kTopK - 1]);
                            }
                        }
                    }
                    // this tile's accumulator columns are free again
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (PAIR) mbar_arrive_cluster(leader_addr(smem_addr(&tmem_empty[tc % nbuf])));
                        else mbar_arrive(&tmem_empty[tc % nbuf]);
                    }
                }
            }

            // one record per hidden row and CTA: the warp with share 1 hands its rows' state to the one with share 0
            float4* xrow = xch + tile_row * 4;
            if (share != 0) {
                xrow[0] = make_float4(m, Z, S, __int_as_float(best_i));
                xrow[1] = make_float4(best_v, bound_used, top.t[0], top.t[1]);
                xrow[2] = make_float4(top.t[2], top.t[3], top.t[4], top.t[5]);
                xrow[3] = make_float4(top.t[6], top.t[7], top.t[8], top.t[9]);
            }
            named_barrier_sync(4 + quad, 64);
            if (share == 0 && warp_has_rows) {
                const float4 a = xrow[0], b4 = xrow[1], c4 = xrow[2], d4 = xrow[3];
                // (a share without columns has Z = 0 and m = -inf; a CTA without columns leaves a record with Z = 0)
                const float M = fmaxf(m, a.x);
                const float d1 = Z > 0.f ? m - M : 0.f, d2 = a.y > 0.f ? a.x - M : 0.f;
                const float e1 = ex2_approx(d1 * kLog2e), e2 = ex2_approx(d2 * kLog2e);
                S = e1 * fmaf(d1, Z, S) + e2 * fmaf(d2, a.y, a.z);
                Z = Z * e1 + a.y * e2;
                m = M;
                const int i2 = __float_as_int(a.w);
                if (b4.x > best_v || (b4.x == best_v && i2 < best_i)) {
                    best_v = b4.x;
                    best_i = i2;
                }
                bound_used = fmaxf(bound_used, b4.y);
                uint32_t cnt = 0;
                if (!STATS) {
                    const float theirs[kTopK] = {b4.z, b4.w, c4.x, c4.y, c4.z, c4.w, d4.x, d4.y, d4.z, d4.w};
                    top.merge(theirs);
#pragma unroll
                    for (int k = 0; k < kTopK; ++k) {
                        cnt += top.t[k] > DISCO_NEG_INF ? 1u : 0u;
                        top.t[k] += 0.f;   // -0 and +0 are the same logit
                    }
                }
                // Statistics that are no numbers (logits that are infinite or no numbers themselves): the record is as good as empty.
                if (!(Z > 0.f)) {
                    cnt = 0u;
                    top.init();
                }
                if (valid && phase == 1) {
                    const uint32_t word = (cnt << 28) | (best_v == m && Z > 0.f ? (uint32_t)best_i : kDbNoIndex);
                    float4* rec = p.part_rec + (size_t)row * p.CN * kStampedPieces + nslot;
                    const float sf = __uint_as_float(smem_word(s_stamp, p.status));   // (written microseconds ago)
                    store_relaxed_v4(rec, m + 0.f, Z, S, sf);
                    store_relaxed_v4(rec + p.CN, __uint_as_float(word), top.t[0], bound_used, sf);
                    store_relaxed_v4(rec + 2 * p.CN, top.t[1], top.t[2], top.t[3], sf);
                    if (cnt > 4) {
                        store_relaxed_v4(rec + 3 * p.CN, top.t[4], top.t[5], top.t[6], sf);
                        store_relaxed_v4(rec + 4 * p.CN, top.t[7], top.t[8], top.t[9], sf);
                    }
                }
            }
            __syncwarp();
            if (lane == 0 && phase == 1) {
                __threadfence_block();
                atomicAdd(s_done, 1);
            }
        }
    }
    if (finisher) {
        if (warp >= 2) db_finish_dedicated<STATS>(p, f, warp, looks_live, fin_s, clf_s, s_stamp, step_live, lane);
    } else if (warp >= 2 && p.finishers == 0) {
        db_finish_rows<STATS>(p, f, warp, looks_live, fin_s, clf_s, s_done, s_clf, s_stamp, step_live, lane);
    }

    tc_fence_before();
    // (the CTAs of a pair arrive at each other's barriers: neither leaves before the other)
    if constexpr (PAIR) cluster_sync();
    else __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        if constexpr (PAIR) tmem_dealloc_pair(tmem_base, 512);
        else tmem_dealloc(tmem_base, 512);
    }
}

}  // namespace disco
