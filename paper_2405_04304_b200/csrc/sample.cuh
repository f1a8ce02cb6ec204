// Sampling at temperature 1 (the paper's Table 6 mode): inverse-CDF draws from probability rows that
// the LM-head kernels have left in global memory, and the accept / resample rule of speculative
// sampling (Leviathan et al., named in Sec. 3 as the verification scheme).
//
// Random numbers are inputs: one uniform in [0, 1) per draw.  Running sums are kept in double precision,
// in vocabulary order, so that a draw depends on the probabilities only and not on how the row is split
// over threads (the split changes the rounding of a double sum in its last bits at most).
#pragma once

#include "common.cuh"

namespace disco {

constexpr int kSampleThreads = 512;
constexpr int kSampleWarps = kSampleThreads / 32;

// The last step of a draw: entries [c0, c1) hold the crossing of `target` (the running sum before c0 is `before`); the token is
// written to found[0].  piece_tot: kSampleWarps doubles of shared memory.  Ends without a barrier.
//
// Long ranges (a segment of a row that few CTAs share): consecutive entries per warp, read in whole lines, 256 at a time; the warp
// that holds the crossing goes through its part again.  Bound: the round trips of the 256-entry batches to L2.  (Entries dealt out
// to threads, as below, are 32 lines per load, which only a large L1 survives: the walk of 32000 entries took 31 or 61 us, as the
// SM happened to be configured behind the LM-head kernel.)
template <typename WeightFn>
__device__ __forceinline__ void block_cdf_walk_long(WeightFn w, int c0, int c1, double before, double target, double* piece_tot,
                                                    int* found) {
    constexpr int kRows = 8, kBatch = 32 * kRows;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = ((c1 - c0 + kSampleWarps - 1) / kSampleWarps + 31) & ~31;
    const int p0 = min(c1, c0 + warp * q), p1 = min(c1, p0 + q);
    auto batch = [&](int v0, float (&x)[kRows]) {
#pragma unroll
        for (int k = 0; k < kRows; ++k) x[k] = v0 + 32 * k + lane < p1 ? w(v0 + 32 * k + lane) : 0.f;
    };
    auto warp_sum = [](double x) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(kFullMask, x, off);
        return x;
    };
    double mine = 0.0;
    int last = -1;      // the warp's last entry with weight
    for (int v0 = p0; v0 < p1; v0 += kBatch) {
        float x[kRows];
        batch(v0, x);
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
            mine += static_cast<double>(x[k]);
            if (x[k] > 0.f) last = v0 + 32 * k + lane;
        }
    }
    mine = warp_sum(mine);
    last = __reduce_max_sync(kFullMask, last);
    if (lane == 0) piece_tot[warp] = mine;
    __syncthreads();
    double run = before;
    for (int k = 0; k < warp; ++k) run += piece_tot[k];
    const double end = run + mine;
    if (run <= target && end > target) {   // at most one warp
        int tok = -1;
        for (int v0 = p0; v0 < p1 && tok < 0; v0 += kBatch) {
            float x[kRows];
            batch(v0, x);
            double sum = 0.0;
#pragma unroll
            for (int k = 0; k < kRows; ++k) sum += static_cast<double>(x[k]);
            sum = warp_sum(sum);
            if (!(run + sum > target)) {
                run += sum;
                continue;
            }
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                double incl = static_cast<double>(x[k]);
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const double o = __shfl_up_sync(kFullMask, incl, off);
                    if (lane >= off) incl += o;
                }
                const unsigned hit = __ballot_sync(kFullMask, x[k] > 0.f && run + incl > target);
                if (tok < 0 && hit) tok = v0 + 32 * k + __ffs(hit) - 1;
                run += __shfl_sync(kFullMask, incl, 31);
            }
        }
        if (lane == 0) found[0] = tok >= 0 ? tok : last;   // (sums in another order: the last bit may fall short of the target)
    }
    // ... or that of the whole range may: its last entry with weight
    if (warp == kSampleWarps - 1 && !(end > target)) {
        int sl = -1;
        for (int v0 = c1 - 32; v0 > c0 - 32 && sl < 0; v0 -= 32) {
            const unsigned some = __ballot_sync(kFullMask, v0 + lane >= c0 && w(v0 + lane) > 0.f);
            if (some) sl = v0 + 31 - __clz(some);
        }
        if (lane == 0) found[0] = sl;
    }
}
// Short ranges: a few consecutive entries per thread, a scan over the CTA, and the thread that holds the crossing has its first eight
// entries in registers still.  Up to 5632 entries (sampled verifications of 32000 x 2048, one form -> the other: 43 rows, segments of
// 4572 entries, 46.6 -> 47.9 us; 65 rows, 6400, 52.8 -> 51.8; 126 rows, 10668, 78.3 -> 62.5; 288 rows, 16000, 142 -> 92).
constexpr int kSampleShortWalk = 11 * kSampleThreads;
template <typename WeightFn>
__device__ __forceinline__ void block_cdf_walk(WeightFn w, int c0, int c1, double before, double target,
                                               double* piece_tot, int* found) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int q = (c1 - c0 + kSampleThreads - 1) / kSampleThreads;   // consecutive entries per thread
    const int p0 = min(c1, c0 + t * q), p1 = min(c1, p0 + q);
    // (eight entries at a time, their loads in flight together; the first eight stay in registers for the walk)
    constexpr int kKeep = 8;
    float first[kKeep] = {};
    double mine = 0.0;
    int mylast = -1;
    for (int v0 = p0; v0 < p1; v0 += kKeep) {
        float x[kKeep];
#pragma unroll
        for (int k = 0; k < kKeep; ++k) x[k] = v0 + k < p1 ? w(v0 + k) : 0.f;
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            mine += static_cast<double>(x[k]);
            if (x[k] > 0.f) mylast = v0 + k;
            if (v0 == p0) first[k] = x[k];
        }
    }
    double incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double o = __shfl_up_sync(kFullMask, incl, off);
        if (lane >= off) incl += o;
    }
    if (lane == 31) piece_tot[warp] = incl;
    __syncthreads();
    double pre = before;
#pragma unroll
    for (int k = 0; k < kSampleWarps; ++k)
        if (k < warp) pre += piece_tot[k];
    incl += pre;
    const double excl = incl - mine;
    if (excl <= target && incl > target) {   // at most one thread
        double r2 = excl;
        int tok = -1;
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            if (tok < 0 && p0 + k < p1) {
                r2 += static_cast<double>(first[k]);
                if (r2 > target) tok = p0 + k;
            }
        }
        for (int v = p0 + kKeep; v < p1 && tok < 0; ++v) {
            r2 += static_cast<double>(w(v));
            if (r2 > target) tok = v;
        }
        found[0] = tok >= 0 ? tok : mylast;
    }
    // the scan adds in another order than the totals were: if its last bit falls short of the target, the
    // crossing is the range's last entry with weight
    if (t == kSampleThreads - 1 && !(incl > target)) {
        int sl = -1;
        for (int v = c1 - 1; v >= c0 && sl < 0; --v)
            if (w(v) > 0.f) sl = v;
        found[0] = sl;
    }
}

// Draft side: the row probs[b, :] arrives holding the raw logits left by the LM-head pass; it is turned into the
// distribution y = exp(z - m) / Z in place (m, Z from stats[2b], stats[2b + 1]), and token[b] is drawn from it with u[b];
// p_token[b] = its probability.  Sequences with active[b] == 0 are left untouched.
//
// A row is cut into SEG segments, one CTA each, and no CTA waits for another: the LM-head pass has left a record (m, Z)
// per slab of the vocabulary, in order, so every CTA of a row works out by itself which slab holds u * Z (one warp, beside
// the normalisation), and the CTA whose segment has that slab walks it.  A segment is a whole number of slabs.
// (One CTA per row, staging it in shared memory, took 18 us for 8 rows of 49152; this takes 5.)
struct DrawRowsParams {
    float* probs;             // [B, V]
    const float* stats;       // [B][2]
    const float4* recs;       // records that start with m, Z: NP per row, rec_step * 16 bytes apart, rows rec_row * 16 bytes
    int rec_step, rec_row, NP;
    int slab;                 // vocabulary rows per record
    int seg_slabs;            // slabs per segment
    int V;
    const float* u;           // [B]
    const uint8_t* active;    // [B] or null
    int32_t* token;           // [B]
    float* p_token;           // [B] or null
};
static __global__ void __launch_bounds__(kSampleThreads) draw_rows_kernel(const DrawRowsParams p) {
    __shared__ double piece_tot[kSampleWarps];
    __shared__ double s_before, s_target;
    __shared__ int s_slab, found[1];
    // launched with programmatic stream serialization: resident early, reading only once the LM-head
    // kernel before it has completed
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int t = threadIdx.x, lane = t & 31;
    const int b = blockIdx.y;
    if (p.active && !p.active[b]) return;
    float* y = p.probs + (size_t)b * p.V;
    const float m = p.stats[2 * b], inv_Z = 1.f / p.stats[2 * b + 1];
    const int first_slab = blockIdx.x * p.seg_slabs;
    const int v0 = min(p.V, first_slab * p.slab), v1 = min(p.V, v0 + p.seg_slabs * p.slab);
    if (t < 32) {
        // a few consecutive records per lane, running sums in record order
        const int q = (p.NP + 31) / 32, c0 = min(p.NP, lane * q), c1 = min(p.NP, c0 + q);
        const float4* rec = p.recs + (size_t)b * p.rec_row;
        // (the first few are fetched side by side: a loop of dependent loads is a round trip each)
        constexpr int kAhead = 5;
        float2 mz[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            mz[i] = make_float2(0.f, 0.f);
            if (c0 + i < c1) mz[i] = __ldcg(reinterpret_cast<const float2*>(rec + (size_t)(c0 + i) * p.rec_step));
        }
        auto mass_of = [&](const float2& r) {
            return r.y > 0.f ? static_cast<double>(r.y) * static_cast<double>(expf(r.x - m)) : 0.0;
        };
        double w_first[kAhead];
        double mine = 0.0;
        int last = -1;
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            w_first[i] = mass_of(mz[i]);
            mine += w_first[i];
            if (w_first[i] > 0.0) last = c0 + i;
        }
        auto mass = [&](int c) { return mass_of(__ldcg(reinterpret_cast<const float2*>(rec + (size_t)c * p.rec_step))); };
        for (int c = c0 + kAhead; c < c1; ++c) {
            const double w = mass(c);
            mine += w;
            if (w > 0.0) last = c;
        }
        double incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const double o = __shfl_up_sync(kFullMask, incl, off);
            if (lane >= off) incl += o;
        }
        const double total = __shfl_sync(kFullMask, incl, 31);
        const double target = static_cast<double>(p.u[b]) * total;
        last = __reduce_max_sync(kFullMask, last);
        const bool cross = incl - mine <= target && incl > target;
        const unsigned who = __ballot_sync(kFullMask, cross);
        if (who ? lane == __ffs(who) - 1 : lane == 0) {
            double before = incl - mine;
            int slab = last;               // rounding next to u = 1: the last slab with mass, and its last entry
            if (who) {
                slab = -1;
#pragma unroll
                for (int i = 0; i < kAhead; ++i) {
                    if (slab < 0 && c0 + i < c1) {
                        if (before + w_first[i] > target) slab = c0 + i;
                        else before += w_first[i];
                    }
                }
                for (int c = c0 + kAhead; c < c1 && slab < 0; ++c) {
                    const double w = mass(c);
                    if (before + w > target) slab = c;
                    else before += w;
                }
                if (slab < 0) slab = last;   // (the sums above were added in another order)
            }
            s_slab = slab;
            s_before = who ? before * inv_Z : 0.0;
            s_target = who ? target * inv_Z : 1e300;
            found[0] = -1;
        }
    }
    if (((p.V | v0 | v1) & 3) == 0 && (reinterpret_cast<uintptr_t>(p.probs) & 15) == 0) {
        for (int v = v0 + 4 * t; v < v1; v += 4 * 4 * kSampleThreads) {
            float4 z[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                z[k] = v + 4 * k * kSampleThreads < v1 ? __ldcg(reinterpret_cast<const float4*>(y + v + 4 * k * kSampleThreads))
                                                       : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (v + 4 * k * kSampleThreads < v1)
                    *reinterpret_cast<float4*>(y + v + 4 * k * kSampleThreads) =
                        make_float4(__expf(z[k].x - m) * inv_Z, __expf(z[k].y - m) * inv_Z, __expf(z[k].z - m) * inv_Z,
                                    __expf(z[k].w - m) * inv_Z);
        }
    } else {
        for (int v = v0 + t; v < v1; v += 8 * kSampleThreads) {
            float z[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) z[k] = v + k * kSampleThreads < v1 ? __ldcg(y + v + k * kSampleThreads) : 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (v + k * kSampleThreads < v1) y[v + k * kSampleThreads] = __expf(z[k] - m) * inv_Z;
        }
    }
    __syncthreads();
    const int slab = s_slab;
    if (slab < 0) {   // no mass anywhere
        if (blockIdx.x == 0 && t == 0) {
            p.token[b] = -1;
            if (p.p_token) p.p_token[b] = 0.f;
        }
        return;
    }
    if (slab < first_slab || slab >= first_slab + p.seg_slabs) return;
    const int c0 = slab * p.slab, c1 = min(p.V, c0 + p.slab);
    block_cdf_walk([&](int v) { return __ldcg(y + v); }, c0, c1, s_before, s_target, piece_tot, found);
    __syncthreads();
    if (t == 0) {
        const int tok = found[0];
        p.token[b] = tok;
        if (p.p_token) p.p_token[b] = tok >= 0 ? __ldcg(y + tok) : 0.f;
    }
}

// Verification side.  y_T arrives holding the raw logits of the R target rows (m, Z of row r in stats[2r],
// stats[2r + 1]) and leaves holding the distributions y = exp(z - m) / Z.  Rows r0 .. r1-1 belong to one
// sequence (SL + 1 of them); draft token i was drawn from draft_probs[(i * B + b), :].  Token i is accepted iff
// u_accept * y_D(t_i) < y_T(t_i); n = number accepted before the first rejection.  The next token is drawn with
// u_sample[b] from norm(max(0, y_T[n] - y_D[n])) after a rejection, from y_T[SL] otherwise; a residual without
// mass falls back to y_T[n].  With R = B (no draft tokens) this is a plain draw from each row.
//
// One launch does all of it: CTA (r, s) owns segment s of row r.  It works out n of its sequence itself (a few
// loads), normalises its segment, and, on the row the draw is from, leaves the sums of its segment's weights
// in scratch memory.  The last CTA of a sequence to finish (a ticket per sequence, zeroed by the host before
// the call) picks the segment that holds u * total and walks it.  The acceptance test reads raw logits while
// other CTAs normalise: the SL entries it reads are left raw by their owners and normalised by the last CTA.
constexpr int kSampleMaxSegments = 16;
struct SampleRowsParams {
    float* y_T;                // [R, V]
    const float* stats;        // [R][2]
    const float* draft_probs;  // [steps, B, V] (null when R == B)
    const int32_t* draft_ids;  // [R - B]
    const int32_t* row_off;    // [B + 1] or null (uniform SL)
    const float* u_accept;     // [R - B]
    const float* u_sample;     // [B]
    int B, SL, R, V;
    int SEG, seg_len;          // segments per row (<= kSampleMaxSegments) and their length (a multiple of 4)
    int32_t* n_accept;
    int32_t* next_token;
    double* seg_tot;           // scratch [B][kSampleMaxSegments][2]: weights of the draw, the row itself
    int32_t* seg_last;         // scratch, same shape: last index with positive weight (-1: none)
    unsigned int* tickets;     // [B], zero at launch
    int* status;
};

// LONG: segments of more than kSampleShortWalk entries (an instance of its own: with both walks in one kernel the calls with short
// segments were 1 - 3 % slower).
template <bool LONG>
static __global__ void __launch_bounds__(kSampleThreads, 2) sample_rows_fused_kernel(const SampleRowsParams p) {
    __shared__ double sh[40];
    __shared__ double red[4][kSampleWarps];
    __shared__ int s_b, s_r0, s_r1, s_n, s_skip, s_last, s_lastpos[2];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int r = blockIdx.x / p.SEG, s = blockIdx.x - r * p.SEG;
    const int V = p.V;
    // A chain of round trips to L2 bounds this kernel, so whatever waits for nothing is on its way first: the row's statistics
    // and this CTA's logits.  (Not the draft distribution that the row would be compared with were it the one drawn from: a load from
    // memory that nearly every CTA waits for in vain.  us per call with it -> without, 17000 x 2048, 8 / 26 / 65 / 126 / 323 / 505 rows:
    // 24.4 / 29.5 / 37.7 / 46.3 / 122 / 131 -> 24.2 / 29.1 / 37.4 / 45.3 / 118 / 129; 32000 x 5120: 65.5 / 70.6 / 88.6 / 115 / 269 / 294 ->
    // 64.9 / 70.0 / 87.6 / 113 / 259 / 291.)
    float* y = p.y_T + (size_t)r * V;
    const float m = p.stats[2 * r], Z = p.stats[2 * r + 1];
    const int v_lo = min(V, s * p.seg_len), v_hi = min(V, v_lo + p.seg_len);
    float z_first[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int v = v_lo + t + k * kSampleThreads;
        z_first[k] = v < v_hi ? __ldcg(y + v) : 0.f;
    }
    // malformed offsets are reported once per sequence, by the first CTA of row b
    if (p.row_off && r < p.B && s == 0 && t == 0) {
        const int b = r, r0 = p.row_off[b], r1 = p.row_off[b + 1];
        if (r0 < b || r1 <= r0 || r1 > p.R - (p.B - 1 - b) || (b == 0 && r0 != 0) || (b == p.B - 1 && r1 != p.R)) {
            record_status(p.status, DISCO_ERR_INVALID_ARG);
            p.n_accept[b] = 0;
            p.next_token[b] = -1;
        }
    }
    if (t == 0) {
        s_b = p.row_off ? -1 : r / (p.SL + 1);
        s_r0 = s_b * (p.SL + 1);
        s_r1 = s_r0 + p.SL + 1;
        s_skip = -1;
        s_lastpos[0] = s_lastpos[1] = -1;
    }
    __syncthreads();
    if (p.row_off) {
        for (int b = t; b < p.B; b += kSampleThreads) {
            const int lo = p.row_off[b], hi = p.row_off[b + 1];
            if (lo <= r && r < hi && atomicCAS(&s_b, -1, b) == -1) s_r0 = lo, s_r1 = hi;   // (one of them, if the offsets are malformed)
        }
        __syncthreads();
    }
    const int b = s_b, r0 = s_r0, r1 = s_r1;
    if (b < 0) return;
    if (p.row_off && (r0 < b || r1 <= r0 || r1 > p.R - (p.B - 1 - b) || (b == 0 && r0 != 0) || (b == p.B - 1 && r1 != p.R))) return;
    const int sl = r1 - r0 - 1;
    const float u_draw = p.u_sample[b];
    const float inv_Z = 1.f / Z;
    // the draft distribution this row is compared with if it is the one drawn from (the address is made here: made from n, further
    // down, it costs the kernel its last registers, 8 rows of 17000 x 2048 24.2 -> 25.0 us)
    const float* yD_here = r - r0 < sl ? p.draft_probs + ((size_t)(r - r0) * p.B + b) * V : nullptr;
    // acceptance tests of all positions side by side, then the first that fails
    if (t == 0) s_n = sl;
    __syncthreads();
    int my_tok = -1;          // position t (the first this thread tests): its token and target probability
    float my_pv = 0.f;
    for (int i = t; i < sl; i += kSampleThreads) {
        const int tok = p.draft_ids[r0 - b + i];
        bool pass = false;
        if (tok < 0 || tok >= V) {
            record_status(p.status, DISCO_ERR_INVALID_ARG);
        } else {
            const int row = r0 + i;
            const float pv = expf(__ldcg(p.y_T + (size_t)row * V + tok) - p.stats[2 * row]) * (1.f / p.stats[2 * row + 1]);
            const double pD = p.draft_probs[((size_t)i * p.B + b) * V + tok];
            pass = static_cast<double>(p.u_accept[r0 - b + i]) * pD < static_cast<double>(pv);
            if (row == r) s_skip = tok;      // this entry stays raw until every reader is done
            if (i == t) {
                my_tok = tok;
                my_pv = pv;
            }
        }
        if (!pass) atomicMin(&s_n, i);
    }
    __syncthreads();
    const int n = s_n, skip = s_skip;
    const bool draw_row = r == r0 + n;
    const float* yD = draw_row ? yD_here : nullptr;
    double acc_w = 0.0, acc_y = 0.0;
    int last_w = -1, last_y = -1;
    for (int v0 = v_lo + t; v0 < v_hi; v0 += 8 * kSampleThreads) {
        float z[8], d[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int v = v0 + k * kSampleThreads;
            z[k] = v0 == v_lo + t ? z_first[k] : (v < v_hi ? __ldcg(y + v) : 0.f);
            d[k] = (yD && v < v_hi) ? __ldg(yD + v) : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int v = v0 + k * kSampleThreads;
            if (v < v_hi) {
                const float pv = expf(z[k] - m) * inv_Z;
                if (v != skip) y[v] = pv;
                if (draw_row) {
                    const float w = yD ? fmaxf(0.f, pv - d[k]) : pv;
                    acc_w += static_cast<double>(w);
                    acc_y += static_cast<double>(pv);
                    if (w > 0.f) last_w = max(last_w, v);
                    if (pv > 0.f) last_y = max(last_y, v);
                }
            }
        }
    }
    if (draw_row) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            acc_w += __shfl_xor_sync(kFullMask, acc_w, off);
            acc_y += __shfl_xor_sync(kFullMask, acc_y, off);
            last_w = max(last_w, __shfl_xor_sync(kFullMask, last_w, off));
            last_y = max(last_y, __shfl_xor_sync(kFullMask, last_y, off));
        }
        if (lane == 0) {
            red[0][warp] = acc_w;
            red[1][warp] = acc_y;
            atomicMax(&s_lastpos[0], last_w);
            atomicMax(&s_lastpos[1], last_y);
        }
        __syncthreads();
        if (warp == 0) {
            double tw = lane < kSampleWarps ? red[0][lane] : 0.0, ty = lane < kSampleWarps ? red[1][lane] : 0.0;
#pragma unroll
            for (int off = kSampleWarps / 2; off > 0; off >>= 1) {
                tw += __shfl_xor_sync(kFullMask, tw, off);
                ty += __shfl_xor_sync(kFullMask, ty, off);
            }
            acc_w = tw, acc_y = ty;
        }
        if (t == 0) {
            const double tw = acc_w, ty = acc_y;
            const size_t at = ((size_t)b * kSampleMaxSegments + s) * 2;
            p.seg_tot[at] = tw;
            p.seg_tot[at + 1] = ty;
            p.seg_last[at] = s_lastpos[0];
            p.seg_last[at + 1] = s_lastpos[1];
        }
    }
    // ticket: the last CTA of the sequence finishes it
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = atomicAdd(p.tickets + b, 1u) == (unsigned)((r1 - r0) * p.SEG) - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the entries the acceptance tests read (the first kSampleThreads positions' values are still in registers)
    if (t < sl && my_tok >= 0) p.y_T[(size_t)(r0 + t) * V + my_tok] = my_pv;
    for (int i = t + kSampleThreads; i < sl; i += kSampleThreads) {
        const int tok = p.draft_ids[r0 - b + i];
        if (tok >= 0 && tok < V) {
            const int row = r0 + i;
            float* e = p.y_T + (size_t)row * V + tok;
            *e = expf(__ldcg(e) - p.stats[2 * row]) * (1.f / p.stats[2 * row + 1]);
        }
    }
    __syncthreads();
    // the draw: the segment that holds u * total, then a walk through it
    const float* yn = p.y_T + (size_t)(r0 + n) * V;
    const float* yDn = n < sl ? p.draft_probs + ((size_t)n * p.B + b) * V : nullptr;
    // (the segments' sums are fetched side by side: a loop of dependent global loads would cost a round trip each)
    double* tot = &red[0][0];                                  // [kSampleMaxSegments][2], free again
    int* lastp = reinterpret_cast<int*>(&red[2][0]);           // the same shape
    static_assert(2 * kSampleMaxSegments <= 2 * kSampleWarps, "the sums fit the reduction area");
    if (t < 2 * p.SEG) {
        tot[t] = __ldcg(p.seg_tot + (size_t)b * kSampleMaxSegments * 2 + t);
        lastp[t] = __ldcg(p.seg_last + (size_t)b * kSampleMaxSegments * 2 + t);
    }
    __syncthreads();
    double total = 0.0;
    for (int k = 0; k < p.SEG; ++k) total += tot[2 * k];
    int which = 0;
    if (yDn && !(total > 0.0)) {     // a residual without mass: the row itself
        which = 1;
        total = 0.0;
        for (int k = 0; k < p.SEG; ++k) total += tot[2 * k + 1];
    }
    const double target = static_cast<double>(u_draw) * total;
    int win = -1, lastpos = -1;
    double before = 0.0, run = 0.0;
    for (int k = 0; k < p.SEG; ++k) {
        const double nxt = run + tot[2 * k + which];
        if (win < 0 && nxt > target) {
            win = k;
            before = run;
        }
        run = nxt;
        lastpos = max(lastpos, lastp[2 * k + which]);
    }
    int* found = reinterpret_cast<int*>(sh + 2 * kSampleWarps);
    if (t == 0) found[0] = -1;
    __syncthreads();
    if (win >= 0) {
        const int c0 = min(V, win * p.seg_len), c1 = min(V, c0 + p.seg_len);
        auto walk = [&](auto w) {
            if constexpr (LONG) block_cdf_walk_long(w, c0, c1, before, target, sh + kSampleWarps, found);
            else block_cdf_walk(w, c0, c1, before, target, sh + kSampleWarps, found);
        };
        if (yDn && which == 0) walk([&](int v) { return fmaxf(0.f, __ldcg(yn + v) - __ldg(yDn + v)); });
        else walk([&](int v) { return __ldcg(yn + v); });
    }
    __syncthreads();
    if (t == 0) {
        p.n_accept[b] = n;
        p.next_token[b] = found[0] >= 0 ? found[0] : lastpos;
    }
}

// Bulk feature extraction (App. D): rows n of y_D and y_T arrive holding the raw logits of the two LM-head passes and leave
// holding the distributions y = exp(z - m) / Z (m, Z from the passes' statistics, [N][2] each); per position the
// total-variation distance TV(y^D, y^T) = (1/2) sum_v |y^D_v - y^T_v| and the accepted label (draft arg-max equals
// target arg-max).  One CTA per position: every logit is read once and every probability written once (a normalisation
// pass per model and a pass over both distributions took 213 us for 1000 positions of the 32000-row heads).  Bound: HBM,
// 16 bytes per position and vocabulary row.
constexpr int kFeatThreads = 512;
static __global__ void __launch_bounds__(kFeatThreads)
tv_label_kernel(float* __restrict__ y_D, float* __restrict__ y_T, const float* __restrict__ stats_D,
                const float* __restrict__ stats_T, const int32_t* __restrict__ token_D, const int32_t* __restrict__ token_T,
                int V, float* tv, uint8_t* label) {
    __shared__ double part[kFeatThreads / 32];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int n = blockIdx.x, t = threadIdx.x;
    float* a = y_D + (size_t)n * V;
    float* b = y_T + (size_t)n * V;
    const float mD = stats_D[2 * n], iD = 1.f / stats_D[2 * n + 1], mT = stats_T[2 * n], iT = 1.f / stats_T[2 * n + 1];
    double s = 0.0;
    if ((V & 3) == 0 && ((reinterpret_cast<uintptr_t>(y_D) | reinterpret_cast<uintptr_t>(y_T)) & 15) == 0) {
        constexpr int kBatch = 4;   // 2 x 4 sixteen-byte loads in flight per thread
        const int V4 = V / 4;
        float4* a4 = reinterpret_cast<float4*>(a);
        float4* b4 = reinterpret_cast<float4*>(b);
        for (int v0 = t; v0 < V4; v0 += kBatch * kFeatThreads) {
            float4 x[kBatch], y[kBatch];
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                const int v = v0 + k * kFeatThreads;
                if (v < V4) {
                    x[k] = __ldcg(a4 + v);
                    y[k] = __ldcg(b4 + v);
                }
            }
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                const int v = v0 + k * kFeatThreads;
                if (v < V4) {
                    x[k].x = expf(x[k].x - mD) * iD, x[k].y = expf(x[k].y - mD) * iD, x[k].z = expf(x[k].z - mD) * iD, x[k].w = expf(x[k].w - mD) * iD;
                    y[k].x = expf(y[k].x - mT) * iT, y[k].y = expf(y[k].y - mT) * iT, y[k].z = expf(y[k].z - mT) * iT, y[k].w = expf(y[k].w - mT) * iT;
                    a4[v] = x[k];
                    b4[v] = y[k];
                    s += (static_cast<double>(fabsf(x[k].x - y[k].x)) + static_cast<double>(fabsf(x[k].y - y[k].y))) +
                         (static_cast<double>(fabsf(x[k].z - y[k].z)) + static_cast<double>(fabsf(x[k].w - y[k].w)));
                }
            }
        }
    } else {
        for (int v0 = t; v0 < V; v0 += 8 * kFeatThreads) {
            float x[8], y[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int v = v0 + k * kFeatThreads;
                x[k] = v < V ? __ldcg(a + v) : 0.f;
                y[k] = v < V ? __ldcg(b + v) : 0.f;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int v = v0 + k * kFeatThreads;
                if (v < V) {
                    const float p = expf(x[k] - mD) * iD, q = expf(y[k] - mT) * iT;
                    a[v] = p;
                    b[v] = q;
                    s += static_cast<double>(fabsf(p - q));
                }
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(kFullMask, s, off);
    if ((t & 31) == 0) part[t >> 5] = s;
    __syncthreads();
    if (t == 0) {
        double sum = 0.0;
        for (int w = 0; w < kFeatThreads / 32; ++w) sum += part[w];
        tv[n] = static_cast<float>(0.5 * sum);
        label[n] = token_D[n] == token_T[n] ? 1 : 0;
    }
}

}  // namespace disco
