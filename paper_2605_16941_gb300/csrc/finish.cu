// finish.cu -- the end of a WINO step (sm_103a): merge the score kernel's
// partial softmax records per row, then apply Eq. 4 to the token state.
//
// One warp per row folds the row's partial records (fixed lane order, then a butterfly, so results are bit-for-bit
// reproducible) into
//   argmax   = smallest vocabulary id among the maximal logits,
//   pmax     = max_v p_v = 1 / sum_v exp(l_v - m),
//   ptarget  = p_target = exp(l_t - m) / sum_v exp(l_v - m)    (0 without a target),
// the three statistics Eq. 2 and Eq. 3 use, and on request the entropy
//   H(p)     = -sum_v p_v log p_v = ln Z - sum_v exp(l_v - m) (l_v - m) / Z
// that WINO+'s deferral and sharpening terms use (Sec. 5.3, Eq. 6-7).  In a whole step (wino_step) Eq. 4 follows in
// the same launch:
//   finish_step_kernel, sequences of up to 256 rows: a cluster of CTAs per sequence merges its rows and hands the
//     statistics to its first CTA, which applies Eq. 4;
//   finish_kernel, longer sequences: every CTA adds its merged rows to its sequences' tickets (cleared by the score
//     kernel of the same step), and the CTA that completes a sequence applies Eq. 4.
// Both are launched programmatically: their CTAs start beside the score kernel's and wait (griddepcontrol.wait) for
// its results before touching them; they let the next call's kernels launch at once (those only prefetch W before
// their own griddepcontrol.wait).  They publish the call's status (see StatusWords).
//
// draft_verify_kernel: Eq. 4 alone from caller-supplied statistics
// (wino_draft_verify), one CTA per sequence.
//
// Eq. 4, per sequence, reading the state before the step y^(k-1):
//   draft  (Eq. 2): y_l == MASK and pmax(block row l) > tau1      -> argmax(block row l)
//   verify (Eq. 3): y_l != MASK and p(y_l | shadow row l) < tau2  -> MASK
// and, if no masked position clears tau1 while the block still has a MASK,
// the masked position with the largest pmax (smallest position on ties) is
// drafted: the greedy rule of Eq. 1, which keeps at least one token coming per
// step.  With draft_m > 0 the drafting rule is naive parallel sampling
// instead (Sec. 3): the draft_m masked positions with the largest pmax
// (smallest position first on ties) are drafted, whatever tau1 says.  The
// rules touch disjoint positions (MASK vs not MASK), so the update
// is applied in place in one pass after a CTA-wide reduction.  With
// WINO_OPT_FREEZE_FINISHED a sequence whose block already has no MASK is left
// as it is (its own loop, Sec. 4.2.3, has ended).
#include <algorithm>

#include "fold.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace wino {
namespace {

constexpr float kLn2 = 0.6931471805599453f;
constexpr int kFinishRows = 8;  // rows (warps) per finish_kernel CTA; also the CTA size of draft_verify_kernel
constexpr int kRecInFlight = 5;  // records each lane loads at once (160 per row: two per pair of a 76-pair launch fit)

// Block-wide reduction scratch for eq4_block.
template <int kWarps>
struct Eq4Smem {
    int32_t i0[kWarps], i1[kWarps], i2[kWarps];
    float f0[kWarps];
};

// Dynamic shared memory of a launch with fixed-M drafting: pmax of each masked position, -inf elsewhere.  (Static, every
// finish CTA would take its 4 KB and fewer would fit beside a score CTA, see kScoreSmemMax.)
extern __shared__ float s_conf[];
inline uint32_t conf_bytes(const wino_params &p) { return p.draft_m > 0 ? (uint32_t)p.blk_len * 4u : 0u; }

// Where Eq. 4 finds a sequence's statistics: entry l of argmax and pmax belongs to the row read for a masked position
// l, entry l of ptarget to the row read for a decoded one.
struct SeqStats {
    const int32_t *argmax;
    const float *pmax, *ptarget;
};

// The same from per-row arrays whose first row of the sequence is row `first`.
__device__ __forceinline__ SeqStats seq_stats(const int32_t *argmax, const float *pmax, const float *ptarget,
                                              int64_t first, const wino_params &p)
{
    const bool both = !(p.options & (WINO_OPT_NO_SHADOW | WINO_OPT_COMPACT));  // block rows, then shadow rows
    return SeqStats{argmax + first, pmax + first, ptarget ? ptarget + first + (both ? p.blk_len : 0) : nullptr};
}

// The current tokens of sequence s's block, thread t's positions t, t + 32 * kWarps, ...
template <int kWarps>
__device__ __forceinline__ void load_tokens(const int32_t *tokens, int s, const wino_params &p,
                                            int32_t (&yv)[kMaxBlkLen / (32 * kWarps)])
{
    const int32_t *y = tokens + (int64_t)s * p.seq_len + p.blk_start;
#pragma unroll
    for (int i = 0; i < kMaxBlkLen / (32 * kWarps); ++i) {
        const int l = (int)threadIdx.x + i * 32 * kWarps;
        yv[i] = l < p.blk_len ? y[l] : 0;
    }
}

// Eq. 4 on sequence s, whose block holds the tokens yv, by the whole CTA of kWarps warps.  Every load is issued before any decision so
// the update costs about one memory round trip.  kShared: the statistics are in this CTA's shared memory; otherwise
// they are read through L2, as other CTAs of the same launch may have written them.
template <bool kShared, int kWarps>
__device__ void eq4_block(int s, const int32_t (&yv)[kMaxBlkLen / (32 * kWarps)], const SeqStats st, int32_t *tokens,
                          const wino_params &p, int32_t *counts, int8_t *flags, int32_t status, Eq4Smem<kWarps> &sm)
{
    constexpr int kT = 32 * kWarps;
    constexpr int kPer = kMaxBlkLen / kT;  // positions per thread
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (status != WINO_OK) {  // the scores of this step are invalid: leave the state alone
        if (tid < 3)
            counts[s * 3 + tid] = status;
        return;
    }
    const int L = p.blk_len;
    const int32_t mask = p.mask_id;
    const bool shadow = !(p.options & WINO_OPT_NO_SHADOW);  // WINO+ inference has no verification rows
    int32_t *y = tokens + (int64_t)s * p.seq_len + p.blk_start;

    int32_t av[kPer];
    float pm[kPer], pt[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int l = tid + i * kT;
        if (l < L) {
            av[i] = kShared ? st.argmax[l] : __ldcg(st.argmax + l);
            pm[i] = kShared ? st.pmax[l] : __ldcg(st.pmax + l);
            // 1.0 is never below tau2 <= 1: no re-mask
            pt[i] = !shadow ? 1.0f : (kShared ? st.ptarget[l] : __ldcg(st.ptarget + l));
        }
    }
    // Pass 1: how many masked positions clear tau1, and the most confident masked position.
    int n_clear = 0, n_mask = 0;
    float best = -INFINITY;
    int best_l = INT32_MAX;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int l = tid + i * kT;
        if (l < L && yv[i] == mask) {
            ++n_mask;
            n_clear += (pm[i] > p.tau1);
            if (pm[i] > best) {  // l grows with i: the first maximum keeps the smallest position
                best = pm[i];
                best_l = l;
            }
        }
    }
    n_clear = __reduce_add_sync(0xffffffffu, n_clear);
    n_mask = __reduce_add_sync(0xffffffffu, n_mask);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float b2 = __shfl_xor_sync(0xffffffffu, best, off);
        const int l2 = __shfl_xor_sync(0xffffffffu, best_l, off);
        if (b2 > best || (b2 == best && l2 < best_l)) {
            best = b2;
            best_l = l2;
        }
    }
    if (lane == 0) {
        sm.i0[warp] = n_clear;
        sm.i1[warp] = n_mask;
        sm.i2[warp] = best_l;
        sm.f0[warp] = best;
    }
    __syncthreads();
    n_clear = n_mask = 0;
    best = -INFINITY;
    best_l = INT32_MAX;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        n_clear += sm.i0[w];
        n_mask += sm.i1[w];
        if (sm.f0[w] > best || (sm.f0[w] == best && sm.i2[w] < best_l)) {
            best = sm.f0[w];
            best_l = sm.i2[w];
        }
    }
    __syncthreads();  // the scratch is reused below
    if (n_mask == 0 && (p.options & WINO_OPT_FREEZE_FINISHED)) {  // finished block: its loop has stopped
        if (flags)
            for (int l = tid; l < L; l += kT)
                flags[(int64_t)s * L + l] = 0;
        if (tid < 3)
            counts[s * 3 + tid] = 0;
        return;
    }
    const int fallback = (p.draft_m <= 0 && n_clear == 0 && n_mask > 0) ? best_l : -1;

    // Fixed-M drafting: position l is drafted iff fewer than M masked positions rank before it
    // (larger pmax, or equal pmax and a smaller position).
    bool top[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i)
        top[i] = false;
    if (p.draft_m > 0) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int l = tid + i * kT;
            if (l < L)
                s_conf[l] = (yv[i] == mask) ? pm[i] : -INFINITY;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int l = tid + i * kT;
            if (l < L && yv[i] == mask) {
                int before = 0;
                for (int j = 0; j < L && before < p.draft_m; ++j) {
                    const float c = s_conf[j];
                    before += (c > pm[i]) || (c == pm[i] && j < l);
                }
                top[i] = before < p.draft_m;
            }
        }
        __syncthreads();  // conf is scratch of this sequence only
    }

    // Pass 2: apply Eq. 4 simultaneously.
    int drafted = 0, remasked = 0, left = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int l = tid + i * kT;
        if (l >= L)
            break;
        const int32_t prev = yv[i];
        int32_t next = prev;
        int8_t code = 0;
        if (prev == mask) {
            if (p.draft_m > 0 ? top[i] : (pm[i] > p.tau1 || l == fallback)) {
                next = av[i];
                code = (next == mask) ? 4 : (p.draft_m > 0 ? 5 : (l == fallback ? 2 : 1));
            }
        } else if (shadow && pt[i] < p.tau2) {
            next = mask;
            code = 3;
        }
        if (next != prev) {
            y[l] = next;
            if (p.last_change)  // WINO finalization step bookkeeping (Sec. 5.1)
                p.last_change[(int64_t)s * p.seq_len + p.blk_start + l] = p.step_index;
        }
        drafted += (code == 1 || code == 2 || code == 5);
        remasked += (code == 3);
        left += (next == mask);
        if (flags)
            flags[(int64_t)s * L + l] = code;
    }
    drafted = __reduce_add_sync(0xffffffffu, drafted);
    remasked = __reduce_add_sync(0xffffffffu, remasked);
    left = __reduce_add_sync(0xffffffffu, left);
    if (lane == 0) {
        sm.i0[warp] = drafted;
        sm.i1[warp] = remasked;
        sm.i2[warp] = left;
    }
    __syncthreads();
    if (tid < 3) {
        const int32_t *src = tid == 0 ? sm.i0 : (tid == 1 ? sm.i1 : sm.i2);
        int32_t v = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w)
            v += src[w];
        counts[s * 3 + tid] = v;
    }
    __syncthreads();  // the scratch may be reused for the next sequence
}

// Whether the caller's active-sequence list names no sequence of the batch for the a-th scored sequence.
__device__ __forceinline__ bool bad_entry(const wino_params &p, int64_t a)
{
    return p.active_seq && (p.active_seq[a] < 0 || p.active_seq[a] >= p.n_seq);
}

// A row's merged softmax state.
struct Merged {
    float m, s, tl, u;
    int32_t idx;
};

// Merge the records of rows row[0 .. kU) (negative: no row) by a warp, kK records per row, lane and round in flight.
// Fixed lane order, then a butterfly.  The record of the pair whose tiles hold the row's target carries its logit, the
// others -inf.
template <int kU, int kK, bool kEntropy>
__device__ __forceinline__ void merge_rows(const FinishArgs &a, const int64_t (&row)[kU], Merged (&o)[kU])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < kU; ++u)
        o[u] = Merged{-INFINITY, 0.f, -INFINITY, 0.f, INT32_MAX};
    for (int j0 = 0; j0 < a.G; j0 += 32 * kK) {
        float4 r[kU][kK];
#pragma unroll
        for (int u = 0; u < kU; ++u)
#pragma unroll
            for (int i = 0; i < kK; ++i) {
                const int j = j0 + lane + 32 * i;
                r[u][i] = (row[u] >= 0 && j < a.G) ? __ldcg(a.part + row[u] * a.G + j)
                                                   : make_float4(-INFINITY, 0.f, __int_as_float(INT32_MAX), -INFINITY);
            }
#pragma unroll
        for (int u = 0; u < kU; ++u)
#pragma unroll
            for (int i = 0; i < kK; ++i) {
                const int j = j0 + lane + 32 * i;
                if (kEntropy)
                    combine_u(o[u].m, o[u].s, o[u].u, o[u].idx, r[u][i].x, r[u][i].y,
                              (row[u] >= 0 && j < a.G) ? __ldcg(a.part_u + row[u] * a.G + j) : 0.f,
                              __float_as_int(r[u][i].z));
                else
                    combine(o[u].m, o[u].s, o[u].idx, r[u][i].x, r[u][i].y, __float_as_int(r[u][i].z));
                o[u].tl = fmaxf(o[u].tl, r[u][i].w);
            }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const float m2 = __shfl_xor_sync(0xffffffffu, o[u].m, off);
            const float s2 = __shfl_xor_sync(0xffffffffu, o[u].s, off);
            const int32_t i2 = __shfl_xor_sync(0xffffffffu, o[u].idx, off);
            o[u].tl = fmaxf(o[u].tl, __shfl_xor_sync(0xffffffffu, o[u].tl, off));
            if (kEntropy)
                combine_u(o[u].m, o[u].s, o[u].u, o[u].idx, m2, s2, __shfl_xor_sync(0xffffffffu, o[u].u, off), i2);
            else
                combine(o[u].m, o[u].s, o[u].idx, m2, s2, i2);
        }
}

// The three statistics of a merged row; invalid ones (status != WINO_OK) are -1 and NaN.
struct RowStats {
    int32_t argmax;
    float pmax, ptarget;
};
__device__ __forceinline__ RowStats row_stats(const Merged &o, int32_t status)
{
    if (status != WINO_OK)
        return RowStats{-1, __int_as_float(0x7fc00000), __int_as_float(0x7fc00000)};
    return RowStats{o.idx, 1.0f / o.s, (o.tl > -INFINITY) ? ptx::ex2((o.tl - o.m) * kLog2e) / o.s : 0.0f};
}

__device__ __forceinline__ void store_row(const FinishArgs &a, int64_t row, const RowStats &x)
{
    a.argmax[row] = x.argmax;
    a.pmax[row] = x.pmax;
    a.ptarget[row] = x.ptarget;
}

// Publish the call's outcome; every thread of every CTA calls it with the `current` word it read.  Without a failure
// nobody writes that word, and the first CTA stores the outcome (a bad active-sequence entry is the only error left).
// After a failure the last CTA to come here also clears the word, which every CTA has then read.
__device__ __forceinline__ void publish_status(const FinishArgs &a, int32_t status, int64_t n_scored_seq)
{
    if (status == WINO_OK) {
        if (blockIdx.x == 0 && threadIdx.x < 32) {
            bool bad = false;
            if (a.tokens && a.p.active_seq)
                for (int64_t i = threadIdx.x; i < n_scored_seq; i += 32)
                    bad |= bad_entry(a.p, i);
            bad = __any_sync(0xffffffffu, bad);
            if (threadIdx.x == 0)
                a.status->last = bad ? (int32_t)WINO_ERR_ARG : (int32_t)WINO_OK;
        }
        return;
    }
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&a.status->finished, 1u) == gridDim.x - 1) {
        __threadfence();
        a.status->finished = 0;
        a.status->last = atomicExch(&a.status->current, (int32_t)WINO_OK);
    }
}

// The end of a step whose sequences have at most kClusterSeqRows rows: a cluster of up to 8 CTAs per sequence.  Its
// warps merge the sequence's rows and hand the statistics to the first CTA's shared memory; behind one cluster barrier
// that CTA applies Eq. 4, whose tokens it has loaded meanwhile.
// What bounds it is latency: dependent round trips to L2 and barriers after the score kernel's last CTA.  The 8-warp CTAs
// are small enough to start beside the row-block kernel's and wait there: 9.5 -> 8.5 us for the tiny step in a CUDA graph
// against 64 registers and 4.3 KB of shared memory, both changed at once.  The 48 registers cost spills (36 bytes with 8
// warps, 28 with 16); a step in a graph with 48 / 56 (12 and 24 bytes) / 64 (none): 6.60 / 6.77 / 6.43 us (d = 64, V = 1000, N = 64),
// 12.43 / 12.58 / 12.13 (d = 512, V = 32000, N = 128).  Beside the vocabulary-major kernel the CTAs do not fit (168
// registers a thread there); with 160 there they do, and nothing is gained: 149.4 -> 149.5 us (64 rows), 226.8 -> 227.3
// (300), 25.4 -> 25.4 (333 rows, d = 1024, V = 32000, where finish_kernel follows).
// Handing over through global memory (finish_kernel: one CTA per 8 rows, fences, a ticket per sequence, the statistics
// read back) costs about 3 us more, but merges more rows at once.  us per step, finish_kernel -> here: 64 rows 9.2 ->
// 7.9 (d = 64, V = 1000), 151.0 -> 147.8 (d = 4096, V = 126464); 128 rows 9.3 -> 8.5.  Above 128 rows with 16 warps per
// CTA instead of 8: 192 rows 12.3 -> 11.6, 256 rows 11.9 -> 11.5 (d = 256, V = 20000; with 8 warps 13.0).  512 rows took
// 13.4 against 10.3, so longer sequences stay with finish_kernel.
template <int kWarps>
__global__ void __maxnreg__(48) finish_step_kernel(const FinishArgs a)
{
    ptx::grid_dep_launch_dependents();  // the next call may start streaming its H and W
    __shared__ Eq4Smem<kWarps> sm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();
    const int seq = (int)blockIdx.x / a.cluster, R = a.seq_rows;
    // dynamic shared memory: [fixed-M scratch | argmax[R] | pmax[R] | ptarget[R]]
    int32_t *s_argmax = reinterpret_cast<int32_t *>(s_conf + (a.p.draft_m > 0 ? a.p.blk_len : 0));
    float *s_pmax = reinterpret_cast<float *>(s_argmax + R), *s_ptarget = s_pmax + R;
    ptx::cluster_sync();  // the first CTA has started: its shared memory may be written
    ptx::grid_dep_wait();
    const int32_t status = *reinterpret_cast<const volatile int32_t *>(&a.status->current);
    int32_t yv[kMaxBlkLen / (32 * kWarps)];
    int s = -1;
    if (rank == 0 && !bad_entry(a.p, seq)) {
        s = a.p.active_seq ? a.p.active_seq[seq] : seq;
        load_tokens<kWarps>(a.tokens, s, a.p, yv);
    }
    const int64_t first = (int64_t)seq * R;
    const int stride = a.cluster * kWarps;
    auto hand_over = [&](int r, const Merged &o) {  // row r of the sequence, by lane 0
        const RowStats x = row_stats(o, status);
        store_row(a, first + r, x);
        ptx::st_shared_cluster_u32(ptx::mapa(ptx::smem_u32(s_argmax + r), 0), (uint32_t)x.argmax);
        ptx::st_shared_cluster_u32(ptx::mapa(ptx::smem_u32(s_pmax + r), 0), __float_as_uint(x.pmax));
        ptx::st_shared_cluster_u32(ptx::mapa(ptx::smem_u32(s_ptarget + r), 0), __float_as_uint(x.ptarget));
    };
    int r = (int)rank * kWarps + warp;
    if (R <= stride) {  // one row per warp
        if (r < R) {
            Merged o[1];
            merge_rows<1, kRecInFlight, false>(a, {first + r}, o);
            if (lane == 0)
                hand_over(r, o[0]);
        }
    } else {
        for (; r < R; r += 2 * stride) {
            const int r2 = r + stride;
            Merged o[2];
            merge_rows<2, 3, false>(a, {first + r, r2 < R ? first + r2 : -1}, o);
            if (lane == 0) {
                hand_over(r, o[0]);
                if (r2 < R)
                    hand_over(r2, o[1]);
            }
        }
    }
    __syncwarp();
    ptx::cluster_sync();  // the statistics are in the first CTA's shared memory
    if (s >= 0)
        eq4_block<true, kWarps>(s, yv, seq_stats(s_argmax, s_pmax, s_ptarget, 0, a.p), a.tokens, a.p, a.counts, a.flags, status,
                        sm);
    publish_status(a, status, a.N / R);
}

// Eq. 4 at the end of finish_kernel: the CTA that merges the last rows of a sequence updates that sequence.
__device__ void eq4_tail(const FinishArgs &a, int64_t row0, int32_t status, int32_t *s_done, int32_t &s_ndone,
                         Eq4Smem<kFinishRows> &sm)
{
    __syncthreads();
    const int64_t per_seq = a.seq_rows;
    if (threadIdx.x == 0) {
        int32_t nd = 0;
        const int64_t rend = min(row0 + kFinishRows, (int64_t)a.N);
        for (int64_t r = row0; r < rend;) {
            const int64_t sq = r / per_seq;
            const int64_t send = min((sq + 1) * per_seq, rend);
            const int32_t cnt = (int32_t)(send - r);
            if (atomicAdd(&a.tickets[sq], cnt) + cnt == per_seq)
                s_done[nd++] = (int32_t)sq;
            r = send;
        }
        s_ndone = nd;
        __threadfence();
    }
    __syncthreads();
    const int nd = s_ndone;
    for (int i = 0; i < nd; ++i) {
        const int sq = s_done[i];
        if (bad_entry(a.p, sq))
            continue;  // no update (the status says so)
        const int s = a.p.active_seq ? a.p.active_seq[sq] : sq;
        int32_t yv[kMaxBlkLen / (32 * kFinishRows)];
        load_tokens<kFinishRows>(a.tokens, s, a.p, yv);
        eq4_block<false, kFinishRows>(s, yv, seq_stats(a.argmax, a.pmax, a.ptarget, sq * per_seq, a.p), a.tokens, a.p, a.counts,
                         a.flags, status, sm);
    }
}

// Rows without a state update (wino_score_rows), and the end of a step with longer sequences: one warp per row.  As
// finish_step_kernel, it is bound by latency; without a state update it neither fences nor counts its CTAs (333 rows at
// d = 1024, V = 32000: 28.2 -> 26.5 us per call).
__global__ void __launch_bounds__(kFinishRows * 32, 5) finish_kernel(const FinishArgs a)
{
    ptx::grid_dep_launch_dependents();  // the next call may start streaming its H and W
    __shared__ int32_t s_done[kFinishRows];
    __shared__ int32_t s_ndone;
    __shared__ Eq4Smem<kFinishRows> sm;
    const int64_t row0 = (int64_t)blockIdx.x * kFinishRows;
    const int64_t row = row0 + (threadIdx.x >> 5);
    ptx::grid_dep_wait();
    const int32_t status = *reinterpret_cast<const volatile int32_t *>(&a.status->current);
    if (row < a.N) {
        Merged o[1];
        if (a.entropy)
            merge_rows<1, kRecInFlight, true>(a, {row}, o);
        else
            merge_rows<1, kRecInFlight, false>(a, {row}, o);
        if ((threadIdx.x & 31) == 0) {
            store_row(a, row, row_stats(o[0], status));
            if (a.entropy)  // H = ln Z - (u ln 2) / Z, with u in log2 units
                a.entropy[row] = status == WINO_OK ? (ptx::lg2(o[0].s) - o[0].u / o[0].s) * kLn2
                                                   : __int_as_float(0x7fc00000);
            if (a.tokens)
                __threadfence();  // publish this row before the CTA signals its ticket
        }
    }
    if (a.tokens)
        eq4_tail(a, row0, status, s_done, s_ndone, sm);
    publish_status(a, status, a.tokens ? a.N / a.seq_rows : 0);
}

// Eq. 4 alone, one CTA per sequence.
__global__ void __launch_bounds__(kFinishRows * 32)
    draft_verify_kernel(int32_t *tokens, const int32_t *argmax, const float *pmax, const float *ptarget,
                        const wino_params p, int32_t *counts, int8_t *flags)
{
    __shared__ Eq4Smem<kFinishRows> sm;
    const int s = blockIdx.x;
    const int64_t rows = ((p.options & (WINO_OPT_NO_SHADOW | WINO_OPT_COMPACT)) ? 1 : 2) * (int64_t)p.blk_len;
    int32_t yv[kMaxBlkLen / (32 * kFinishRows)];
    load_tokens<kFinishRows>(tokens, s, p, yv);
    eq4_block<false, kFinishRows>(s, yv, seq_stats(argmax, pmax, ptarget, s * rows, p), tokens, p, counts, flags, WINO_OK, sm);
}

// Row compaction: one CTA per position copies the one row Eq. 4 will read -- the block row of a masked
// position, the shadow row of a decoded one -- with 16-byte loads (d % 8 == 0).
__global__ void __launch_bounds__(256) gather_compact_kernel(const uint4 *__restrict__ H, uint4 *__restrict__ Hc,
                                                             const int32_t *__restrict__ tokens, const wino_params p,
                                                             int64_t vec_per_row)
{
    ptx::grid_dep_launch_dependents();  // the score kernel may set up now; it waits for these rows itself
    ptx::grid_dep_wait();  // the token state may still be being written by the previous step
    const int64_t r = blockIdx.x;  // = s * L + l
    const int64_t s = r / p.blk_len, l = r - s * p.blk_len;
    const bool masked = tokens[s * p.seq_len + p.blk_start + l] == p.mask_id;
    const uint4 *src = H + ((2 * s + (masked ? 0 : 1)) * p.blk_len + l) * vec_per_row;
    uint4 *dst = Hc + r * vec_per_row;
    for (int64_t i = threadIdx.x; i < vec_per_row; i += blockDim.x)
        dst[i] = __ldg(src + i);
}

// Active-sequence gather: one CTA per scored row copies the row of a listed sequence (row r of the
// gathered layout belongs to the a-th listed sequence s) into the workspace with 16-byte loads, and
// writes the row's target: the current token of the position a shadow row verifies, else -1 (MASK or
// a block row), so that the score kernel reads the gathered rows with explicit targets.
__global__ void __launch_bounds__(256) gather_active_kernel(const uint4 *__restrict__ H, uint4 *__restrict__ Hc,
                                                            int32_t *__restrict__ target,
                                                            const int32_t *__restrict__ tokens, const wino_params p,
                                                            int64_t vec_per_row)
{
    ptx::grid_dep_launch_dependents();  // the score kernel waits for these rows itself
    ptx::grid_dep_wait();  // the token state may still be being written by the previous step
    const bool shadow = !(p.options & WINO_OPT_NO_SHADOW);
    const bool compact = (p.options & WINO_OPT_COMPACT) != 0;
    const int64_t L = p.blk_len;
    const int64_t per_seq = (shadow && !compact) ? 2 * L : L;
    const int64_t r = blockIdx.x;
    const int64_t a = r / per_seq, j = r - a * per_seq;
    const int64_t s = p.active_seq[a];
    uint4 *dst = Hc + r * vec_per_row;
    if (s < 0 || s >= p.n_seq) {  // a bad entry of the caller's list: read nothing (the finish kernel reports it)
        for (int64_t i = threadIdx.x; i < vec_per_row; i += blockDim.x)
            dst[i] = make_uint4(0, 0, 0, 0);
        if (threadIdx.x == 0)
            target[r] = -1;
        return;
    }
    const int64_t l = (j < L) ? j : j - L;
    const int32_t y = tokens[s * p.seq_len + p.blk_start + l];
    // kind of the row: the shadow row for j >= L; with compaction, the row Eq. 4 reads for this position
    const int kind = !shadow ? 0 : (compact ? (y == p.mask_id ? 0 : 1) : (j < L ? 0 : 1));
    const int64_t src_row = shadow ? (2 * s + kind) * L + l : s * L + l;
    const uint4 *src = H + src_row * vec_per_row;
    for (int64_t i = threadIdx.x; i < vec_per_row; i += blockDim.x)
        dst[i] = __ldg(src + i);
    if (threadIdx.x == 0)
        target[r] = (kind == 1 && y != p.mask_id) ? y : -1;
}

}  // namespace

cudaError_t launch_gather_compact(const uint16_t *H, uint16_t *Hc, const int32_t *tokens, const wino_params &p,
                                  int64_t d, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((int64_t)p.n_seq * p.blk_len));
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gather_compact_kernel, reinterpret_cast<const uint4 *>(H),
                              reinterpret_cast<uint4 *>(Hc), tokens, p, d / 8);
}

cudaError_t launch_gather_active(const uint16_t *H, uint16_t *Hc, int32_t *target, const int32_t *tokens,
                                 const wino_params &p, int64_t rows, int64_t d, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)rows);
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gather_active_kernel, reinterpret_cast<const uint4 *>(H),
                              reinterpret_cast<uint4 *>(Hc), target, tokens, p, d / 8);
}

cudaError_t launch_finish(FinishArgs a, cudaStream_t stream)
{
    const wino_params &p = a.p;
    a.seq_rows = a.tokens ? (int32_t)rows_per_seq(p) : 0;
    const bool clusters = a.tokens && a.seq_rows <= kClusterSeqRows;
    const int warps = clusters && a.seq_rows > 128 ? 16 : kFinishRows;
    a.cluster = clusters ? std::min(8, (a.seq_rows + warps - 1) / warps) : 1;  // 8: the portable most
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters ? (unsigned)(a.N / a.seq_rows * a.cluster)
                                : (unsigned)((a.N + kFinishRows - 1) / kFinishRows));
    cfg.blockDim = dim3((unsigned)warps * 32);
    cfg.dynamicSmemBytes = (a.tokens ? conf_bytes(p) : 0) + (clusters ? 12u * (uint32_t)a.seq_rows : 0);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)a.cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = clusters ? 2 : 1;
    if (!clusters)
        return cudaLaunchKernelEx(&cfg, finish_kernel, a);
    return warps == 16 ? cudaLaunchKernelEx(&cfg, finish_step_kernel<16>, a)
                       : cudaLaunchKernelEx(&cfg, finish_step_kernel<8>, a);
}

cudaError_t launch_draft_verify(int32_t *tokens, const int32_t *argmax, const float *pmax, const float *ptarget,
                                const wino_params &p, int32_t *counts, int8_t *flags, cudaStream_t stream)
{
    draft_verify_kernel<<<p.n_seq, kFinishRows * 32, conf_bytes(p), stream>>>(tokens, argmax, pmax, ptarget, p, counts, flags);
    return cudaGetLastError();
}

}  // namespace wino
