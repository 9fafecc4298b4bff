// score_vmajor.cu -- the score kernel with the vocabulary on the M side of the MMA (sm_103a).
//
// Same results as score.cu (see there for what is computed and why), for row counts that do not fill 256-row
// blocks.  score.cu multiplies blocks of 256 rows of H by vocabulary tiles; every row count is padded to a
// multiple of 256 in MMA time, shared-memory reads and staged bytes.  Here a CTA pair's MMA has M = 256
// vocabulary rows (128 per CTA; bn of them used, as in score.cu's tiles) and N = hw rows of H, a multiple of 16
// or 32 up to 256, one or two accumulators per vocabulary tile: up to 512 rows of H share each staged W slice, and
// the padding is at most 31 rows per group.  Up to about 200 rows the MMAs take a fraction of the time of the W
// stream, which then runs at the copy bandwidth (152.4 us for 1.036 GB at N = 32, 6.8 TB/s; score.cu 157.0 us).
// From there on the W stream and the MMAs bound it together, and over longer times the board's power (N = 300: W at
// 80 % of the copy rate with the tensor pipe busy 77 % of the cycles; N = 1024: busy 96 %).
//
// The accumulator then has the vocabulary along the TMEM lanes and the rows of H along the columns, so a
// thread's TMEM load gives 32 different rows' logits of one vocabulary entry.  The epilogue transposes each
// 32 x 32 block through 4 KB of shared memory per warp (XOR-swizzled 16-byte groups: conflict-free both ways),
// after which lane j holds 32 consecutive vocabulary entries of row j and folds them as score.cu does.  Each
// thread keeps the running state of its rows (up to 8) in registers across all of the pair's tiles; the four
// lane quarters of a CTA are merged once at the end, one record per (row, CTA).
//
// Roles (320 threads): warp 0 TMA producer, warp 1 TMEM + MMA issuer (leader), warps 2-9 epilogue: two warps per
// TMEM lane quarter, on alternate 32-column chunks.  With two accumulators per tile the second one's MMAs of a
// tile's first ring stages are deferred until the epilogue has read it (polled per K slice, so the staged slices
// are held no longer than needed).  Waits, abort and drain, programmatic launch, status and timeline are those of
// score.cu.
#include <mutex>

#include "fold.cuh"
#include "internal.h"
#include "ptx.cuh"
#include "wait.cuh"

namespace wino {
namespace {

constexpr uint16_t kBothCtas = 0x3;
constexpr int kPrefetchSlices = 4;  // K slices of the first W tile prefetched into L2 before the grid wait
constexpr int kVmEpiWarps = 8;
constexpr int kVmThreads = 64 + 32 * kVmEpiWarps;
constexpr int kMaxChunks = 4;  // 32-column chunks of one accumulator (256 columns) per epilogue warp

// The split and the choice between the two score kernels: estimated ns on the busiest pair, fitted to measured calls of
// both.  Per tile and K slice, from 24 K slices on (long enough for the board's power limit) and below:
//   one accumulator    190 + 0.75 hw,                   204 + 0.22 hw;
//   two                60 + 1.4 w and 4 w per tile,     1.25 w - 12 and 8 w per tile, w = hw[0] + hw[1];
//   score.cu           0.95 (bn + 144) and 700 per tile, 1.75 (bn - 55) and 607 per tile;
// here the epilogue (540 for two 32-column chunks, one per warp of a quarter) if that is longer, plus a third of the
// shorter of the two for one accumulator below 24 K slices; and the last tile's epilogue.
// us per call of wino_score_rows, score.cu -> here (groups), both on the same inputs in turn, d = 4096, V = 126464:
// N = 288 275 -> 202 (1), 320 285 -> 221 (1), 384 292 -> 272 (1), 448 297 -> 284 (2), 512 303 -> 313 (2), 576 465 -> 373 (2),
// 640 471 -> 422 (2), 768 483 -> 459 (3), 896 570 -> 549 (4), 1024 576 -> 598 (4), 1280 815 -> 775 (5), 1664 1177 -> 1068 (4),
// 2048 1214 -> 1198 (8; stays with score.cu); d = 1664, V = 64677: 310 67.3 -> 54.7 (1); d = 576, V = 103363: 308 48.8 ->
// 36.7 (2); d = 512, V = 54379: 1298 66.1 -> 59.5 (6); d = 448, V = 54533: 373 24.5 -> 23.9 (2); d = 256, V = 64000: 384 18.9 ->
// 24.7 (2; stays).
// Of 48 random shapes (N = 49 to 2048, d = 320 to 4096, V = 19456 to 134400) the choice sent 29 here, all with more than
// 256 rows: 0.90 of score.cu's time (geometric mean; 0.77 at N = 304, d = 2112, V = 121643 to 1.06 at N = 907, d = 448,
// V = 65313), six of them 1.6 to 6.3 % slower than score.cu, and 1.01 of the best split's of either kernel.
// Up to 256 rows (one row block) both kernels follow the W stream.  This one wins where score.cu's mostly
// empty boxes of H hold it up (N = 32, d = 1024 33.8 -> 26.6; N = 64 27.0 -> 27.6) and where the W stream is long
// enough for the power limit to bite (N = 128: d = 3072, V = 126464 124.7 -> 123.0; d = 4096 163.8 -> 159.0; but d = 4096,
// N = 208 177.4 -> 183.6, and d = 2048, V = 64000, N = 128 48.0 -> 48.4).  Of the 14 random shapes of 49 to 256 rows, all with
// score.cu, five would have been 12 to 32 % faster here (49 to 112 rows, d = 576 to 960): the line at
// kVmShortRows lies low for such heads.
constexpr int kVmCappedSlices = 24;
constexpr int kVmShortRows = 48;                        // always here (with a vocabulary for every pair's records)
constexpr int kVmMinSlices = 5;                         // K slices per tile: below, latencies that the estimates leave out
constexpr int64_t kVmLongHead = int64_t(1) << 28;       // V * d from which one row block may come here, 512 MiB of W
constexpr int64_t kRowOneBlockSliceNs = 356;            // a K slice of score.cu's tile of a single row block there
constexpr int kVmMaxGroups = 8;
constexpr int kVmEvenTileRows = 192;  // rows per group up to which the W stream, not the MMAs, sets the time: tiles are
                                      // then narrowed to split the vocabulary evenly over the pairs (V = 126464 on 76
                                      // pairs: 240; N = 300, MMA-bound: 242 us with 240, 236 with 256)
constexpr uint32_t kTransBytes = kVmEpiWarps * 32 * 32 * 4;

struct alignas(8) VmBarriers {
    uint64_t full[kVmMaxStages];       // leader: both CTAs' copies of a stage landed
    uint64_t empty[kVmMaxStages];      // both: the stage's MMAs are done (multicast commit)
    uint64_t tmem_full[kVmMaxSlots];   // both: accumulator i holds a finished tile (multicast commit)
    uint64_t tmem_empty[kVmMaxSlots];  // leader: all 16 epilogue warps of the pair have read accumulator i
    uint64_t mma_done;                 // leader: every MMA issued has completed
    uint32_t tmem_base;
    int32_t abort;
};
static_assert(sizeof(VmBarriers) <= kVmBarrierBytes, "barrier block must fit its reserve");

// Item i of the pair at column `col` of its group: vocabulary tile vt, accumulators [h0, h1).  Rounds of whole tiles
// col, col + G, ...; in a last round that would leave at least half of the pairs idle (ScoreArgs::split), a tile's two
// accumulators go to two pairs (V = 126464 on 76 pairs: 6.5 tiles a pair instead of 7; us per step at d = 4096, N = 288
// 215.5 -> 209.5, 300 222.5 -> 217.5, 384 275.3 -> 270.3, steady state; 352 in 20-step regions 229 -> 219).
struct VmItem {
    int vt, h0, h1;
};
__device__ __forceinline__ bool vm_item(const ScoreArgs &a, int col, int i, VmItem &it)
{
    const int full = a.n_vt / a.G, rem = a.n_vt - full * a.G;
    const bool half = a.split && i == full;
    it.vt = i * a.G + (half ? col >> 1 : col);
    it.h0 = half ? col & 1 : 0;
    it.h1 = half ? it.h0 + 1 : (a.hw[1] > 0 ? 2 : 1);
    return half ? col < 2 * rem : it.vt < a.n_vt;
}

// Running state of one row in one thread (the four partial sums of a fold are added up after each fold).
struct ColState {
    float m, s, tlog, u;
    int32_t am;
};

template <bool kEntropy>
__device__ __forceinline__ void fold_col(ColState &c, float (&x)[32], int v, int cvalid, int tgt)
{
    RowState r{c.m, c.s, 0.f, 0.f, 0.f, c.tlog, c.u, 0.f, 0.f, 0.f, c.am};
    fold32<kEntropy>(r, x, v, cvalid, tgt);
    c.m = r.m;
    c.s = (r.s0 + r.s1) + (r.s2 + r.s3);
    if (kEntropy)
        c.u = (r.u0 + r.u1) + (r.u2 + r.u3);
    c.tlog = r.tlog;
    c.am = r.am;
}

template <bool kEntropy>
__global__ void __launch_bounds__(kVmThreads, 1)
    score_vmajor_kernel(const __grid_constant__ CUtensorMap tmH, const __grid_constant__ CUtensorMap tmW,
                        const ScoreArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;  // swizzle atoms need 1024-B alignment
    uint8_t *const ring_ptr = smem_raw + (ring - raw);
    const uint32_t ring_bytes = (uint32_t)a.stages * a.stage_bytes;
    float *const trans = reinterpret_cast<float *>(ring_ptr + ring_bytes);
    VmBarriers *bars = reinterpret_cast<VmBarriers *>(ring_ptr + ring_bytes + kTransBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();  // 0: leader (issues the MMAs), 1: peer
    const bool leader = rank == 0;
    const int pair = blockIdx.x >> 1;
    uint64_t *const tl = a.timeline ? a.timeline + (size_t)blockIdx.x * kTimelineWords : nullptr;
    float4 pend[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};  // see score.cu
    float pend_u[2] = {0.f, 0.f};
    int64_t pend_idx[2] = {-1, -1};
    if (tl && threadIdx.x == 0)
        tl[0] = ptx::globaltimer_ns();

    const int S = a.stages;
    const int hw0 = a.hw[0], hw1 = a.hw[1], slots = a.slots;  // hw1 = 0: one accumulator per tile
    const int hrows = (hw0 + hw1) >> 1;  // rows of H this CTA stages per K slice
    const int half_bn = a.bn >> 1;      // vocabulary rows this CTA stages per tile
    auto sA = [&](int s) { return ring + (uint32_t)s * a.stage_bytes; };
    auto sB = [&](int s, int h) { return sA(s) + kVmStageBytesW + (uint32_t)(h * (hw0 >> 1)) * 128u; };
    auto full = [&](int s) { return ptx::smem_u32(&bars->full[s]); };
    auto empty = [&](int s) { return ptx::smem_u32(&bars->empty[s]); };
    auto tfull = [&](int i) { return ptx::smem_u32(&bars->tmem_full[i]); };
    auto tempty = [&](int i) { return ptx::smem_u32(&bars->tmem_empty[i]); };
    const uint32_t mma_done = ptx::smem_u32(&bars->mma_done);

    // Set-up that touches no global memory overlaps the previous kernel (programmatic launch).
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            ptx::mbar_init(full(s), 1);
            ptx::mbar_init(empty(s), 1);
        }
        for (int i = 0; i < kVmMaxSlots; ++i) {
            ptx::mbar_init(tfull(i), 1);
            ptx::mbar_init(tempty(i), 2 * kVmEpiWarps);  // the epilogue warps of both CTAs
        }
        ptx::mbar_init(mma_done, 1);
        bars->abort = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 0 && lane == 0) {
        ptx::prefetch_tensormap(&tmH);
        ptx::prefetch_tensormap(&tmW);
    }
    if (warp == 1) {
        ptx::tmem_alloc_pair(ptx::smem_u32(&bars->tmem_base), kTmemCols);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before();
    ptx::cluster_sync();  // barriers and TMEM address of both CTAs are now visible to both
    ptx::tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    const uint32_t peer_tmem = ptx::ld_shared_cluster_u32(ptx::mapa(ptx::smem_u32(&bars->tmem_base), rank ^ 1u));
    const bool tmem_ok = (peer_tmem == tmem);
    if (tl && threadIdx.x == 0)
        tl[1] = ptx::globaltimer_ns();
    ptx::grid_dep_launch_dependents();

    const int grp = pair % a.n_groups;  // rows [grp * (hw0 + hw1), ...) of H
    const int col = pair / a.n_groups;  // vocabulary tiles col, col + G, ...
    const int row0 = grp * (hw0 + hw1);

    if (warp >= 2 || !tmem_ok) {
        ptx::grid_dep_wait();
        if (tl && threadIdx.x == 64)
            tl[3] = ptx::globaltimer_ns();
        if (threadIdx.x >= 64)
            for (int i = blockIdx.x * (32 * kVmEpiWarps) + (int)threadIdx.x - 64; i < a.n_tickets;
                 i += gridDim.x * (32 * kVmEpiWarps))
                a.tickets[i] = 0;
    }
    if (!tmem_ok) {
        // nothing to do: the status word reports the failed allocation check
    } else if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (both CTAs)
        if (ptx::elect_one()) {
            auto w_x = [&](int kb) { return a.w_panels ? 0 : kb * kBK; };
            auto w_y = [&](int kb, int v) { return a.w_panels ? kb * a.V + v : v; };
            for (int kb = 0; kb < min(a.n_kb, kPrefetchSlices); ++kb)
                ptx::tma_prefetch_2d(&tmW, w_x(kb), w_y(kb, col * a.bn + (int)rank * half_bn));
            ptx::grid_dep_wait();
            const uint64_t pol_h = ptx::policy_evict_last();    // H is re-read for every tile
            const uint64_t pol_w = ptx::policy_evict_normal();  // W is shared by the row groups
            const uint32_t stage_tx = 2u * 128u * (uint32_t)(half_bn + hrows);  // both CTAs' copies
            int stage = 0;
            uint32_t phase = 0;
            int64_t issued = 0;
            bool aborted = false;
            VmItem it;
            for (int i = 0; !aborted && vm_item(a, col, i, it); ++i) {
                for (int kb = 0; kb < a.n_kb; ++kb) {
                    if (!wait_bounded(empty(stage), phase ^ 1u, &bars->abort)) {
                        aborted = true;
                        break;
                    }
                    const uint32_t bar = ptx::mapa(full(stage), 0);  // the leader's stage barrier
                    if (leader)
                        ptx::mbar_arrive_expect_tx(full(stage), stage_tx);
                    ptx::tma_load_2d_pair(sA(stage), &tmW, bar, w_x(kb), w_y(kb, it.vt * a.bn + (int)rank * half_bn),
                                          pol_w);
                    ptx::tma_load_2d_pair(sB(stage, 0), &tmH, bar, kb * kBK, row0 + (int)rank * hrows, pol_h);
                    if (tl && issued == 0)
                        tl[2] = ptx::globaltimer_ns();
                    ++issued;
                    if (++stage == S) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (aborted && leader) {
                // Let every copy already issued (by either CTA) land before the pair's shared memory goes away.
                for (int s = 0; s < S && s < issued; ++s)
                    wait_drain(full(s), (uint32_t)((issued - 1 - s) / S) & 1u);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (leader)
        if (leader && ptx::elect_one()) {
            const uint32_t idesc0 = ptx::idesc_bf16_f32(kPairM, (uint32_t)hw0);
            const uint32_t idesc1 = ptx::idesc_bf16_f32(kPairM, (uint32_t)hw1);
            int tiles = 0;
            int stage = 0;
            uint32_t phase = 0;
            // accumulators are used in turn: `slot` for the next use, after `round` uses of each before it
            int slot = 0;
            uint32_t round = 0;
            bool aborted = false;
            auto issue = [&](int acc, int s, int h, int kb) {  // 4 x K16 from stage s into accumulator acc
                const uint64_t da = ptx::sdesc_kmajor_sw128(sA(s));
                const uint64_t db = ptx::sdesc_kmajor_sw128(sB(s, h));
                const uint32_t dst = tmem + (uint32_t)(acc * hw0);
                const uint32_t idesc = h ? idesc1 : idesc0;
#pragma unroll
                for (int k = 0; k < kBK / 16; ++k)  // +32 B along K per MMA = +2 in the encoded address
                    ptx::mma_bf16_pair(dst, da + 2u * k, db + 2u * k, idesc, (kb | k) != 0);
            };
            VmItem it;
            for (int i = 0; !aborted && vm_item(a, col, i, it); ++i) {
                const bool both = it.h1 - it.h0 == 2;
                const int acc0 = slot;
                const uint32_t par0 = (round & 1u) ^ 1u;
                if (++slot == slots) {
                    slot = 0;
                    ++round;
                }
                const int acc1 = slot;  // with both accumulators of a tile
                const uint32_t par1 = (round & 1u) ^ 1u;
                if (both && ++slot == slots) {
                    slot = 0;
                    ++round;
                }
                // the epilogue has read the accumulator's previous use
                if (!wait_bounded<true>(tempty(acc0), par0, &bars->abort)) {
                    aborted = true;
                    break;
                }
                ptx::tc_fence_after();
                bool second = !both;        // the second accumulator is free (or not used)
                int held = 0;               // K slices whose second-accumulator MMAs have not been issued: [0, held)
                const int s0 = stage;
                for (int kb = 0; kb < a.n_kb; ++kb) {
                    if (!wait_bounded(full(stage), phase, &bars->abort)) {
                        aborted = true;
                        break;
                    }
                    issue(acc0, stage, it.h0, kb);
                    if (both && kb == a.n_kb - 1)  // accumulator 0 is done: its epilogue need not wait for 1
                        ptx::mma_commit_pair_multicast(tfull(acc0), kBothCtas);
                    if (second) {
                        if (both)
                            issue(acc1, stage, 1, kb);
                        ptx::mma_commit_pair_multicast(empty(stage), kBothCtas);
                    } else {
                        ++held;
                        if (held == S || kb == a.n_kb - 1) {  // no stage or slice left to run ahead on
                            if (!wait_bounded<true>(tempty(acc1), par1, &bars->abort)) {
                                aborted = true;
                                break;
                            }
                            second = true;
                        } else {
                            second = ptx::mbar_test_wait_cluster(tempty(acc1), par1);
                        }
                        if (second) {
                            ptx::tc_fence_after();
                            int sj = s0;
                            for (int j = 0; j < held; ++j) {
                                issue(acc1, sj, 1, j);
                                ptx::mma_commit_pair_multicast(empty(sj), kBothCtas);
                                if (++sj == S)
                                    sj = 0;
                            }
                        }
                    }
                    if (++stage == S) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (aborted)
                    break;
                // the item's last commit (see score.cu)
                ptx::mma_commit_pair_multicast(tfull(both ? acc1 : acc0), kBothCtas);
                tiles += it.h0 == 0;
            }
            // No MMA may still be writing either CTA's TMEM when it is released.
            ptx::mma_commit_pair(mma_done);
            wait_drain(mma_done, 0);
            if (tl) {
                tl[4] = ptx::globaltimer_ns();
                tl[7] = (uint64_t)ptx::smid() << 32 | (uint32_t)tiles;
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
        const int q = warp & 3;           // this warp may only read TMEM lanes [32q, 32q + 32)
        const int sel = (warp - 2) >> 2;  // which of the quarter's two warps: chunks of parity sel ^ accumulator
        const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
        float *const tb = trans + (warp - 2) * 1024;
        auto chunk_of = [&](int h, int i) { return 2 * i + (sel ^ h); };
        // The row of H behind column c of accumulator h: CTA 0 staged the first half of the columns, CTA 1 the others.
        auto row_of = [&](int h, int c) {
            const int half = (h ? hw1 : hw0) >> 1, hi = c >= half ? 1 : 0;
            return row0 + hi * hrows + h * (hw0 >> 1) + c - hi * half;
        };
        ColState st[2 * kMaxChunks];
        int32_t tgt[2 * kMaxChunks];
        uint32_t live = 0;  // chunks with a row of H in them (warp-uniform)
#pragma unroll
        for (int k = 0; k < 2 * kMaxChunks; ++k) {
            const int h = k / kMaxChunks, c = chunk_of(h, k % kMaxChunks) * 32 + lane;
            const int row = row_of(h, c);
            const bool mine = c < (h ? hw1 : hw0) && row < a.N;
            st[k] = ColState{-INFINITY, 0.f, -INFINITY, 0.f, 0};
            tgt[k] = mine ? row_target(a.ts, row, a.V) : -1;
            if (__any_sync(0xffffffffu, mine))
                live |= 1u << k;
        }
        int use = 0, n_uses = 0;  // accumulators read, and of all of the pair's items
        VmItem it;
        for (int i = 0; vm_item(a, col, i, it); ++i)
            n_uses += it.h1 - it.h0;
        bool aborted = false;
        for (int i = 0; !aborted && vm_item(a, col, i, it); ++i) {
            const int v0 = it.vt * a.bn + (int)rank * half_bn + q * 32;  // vocabulary id of this warp's first lane
            const int nvalid = min(half_bn - q * 32, a.V - v0);       // valid lanes from there (may be <= 0)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h < it.h0 || h >= it.h1 || aborted)
                    continue;
                const int slot = use % slots;
                int ok = 1;
                if (lane == 0)
                    ok = wait_bounded(tfull(slot), (uint32_t)(use / slots) & 1u, &bars->abort);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                ptx::tc_fence_after();
                if (!ok) {
                    aborted = true;
                    continue;
                }
                // Accumulator fully read by this warp: tell the leader's MMA warp.  Sent once the warp's last chunk is in
                // registers, before its fold: with two accumulators per tile the MMAs wait for it (d = 4096,
                // V = 126464, N = 352 258.3 -> 255.6 us per step, 600 402 -> 399; with one, no change).
                // Not sent where the MMA warp does not wait for it (see score.cu's closing barrier).
                auto release = [&] {
                    if (use + slots >= n_uses)
                        return;
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0)
                        ptx::mbar_arrive_cluster_relaxed(ptx::mapa(tempty(slot), 0));
                };
                const uint32_t mine = nvalid > 0 ? live >> (h * kMaxChunks) & ((1u << kMaxChunks) - 1u) : 0u;
                if (!mine)
                    release();
                if (nvalid > 0) {
#pragma unroll
                    for (int c = 0; c < kMaxChunks; ++c) {
                        const int k = h * kMaxChunks + c;
                        if (!(live >> k & 1u))
                            continue;
                        float x[32];
                        ptx::tmem_ld_32x32b_x32(lanes + (uint32_t)(slot * hw0 + chunk_of(h, c) * 32), x);
                        ptx::tmem_ld_wait();
                        if (mine >> (c + 1) == 0)
                            release();  // the warp's last chunk is in registers
                        // transpose: row j (of the chunk), vocabulary lane l at j * 32 + ((l / 4) ^ (j % 8)) * 4 + l % 4
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            tb[j * 32 + ((((lane >> 2) ^ (j & 7)) << 2) | (lane & 3))] = x[j];
                        __syncwarp();
#pragma unroll
                        for (int g = 0; g < 8; ++g) {
                            const float4 t = *reinterpret_cast<const float4 *>(tb + lane * 32 + ((g ^ (lane & 7)) << 2));
                            x[4 * g] = t.x;
                            x[4 * g + 1] = t.y;
                            x[4 * g + 2] = t.z;
                            x[4 * g + 3] = t.w;
                        }
                        __syncwarp();  // before the next chunk's stores
                        fold_col<kEntropy>(st[k], x, v0, nvalid, tgt[k]);
                    }
                }
                ++use;
            }
        }
        if (tl && !leader && warp == 2 && lane == 0)
            tl[4] = ptx::globaltimer_ns();
        // Merge the four lane quarters of every row in the ring, which is free: the last accumulator's MMAs have
        // completed, and with them every copy they read.  (After an abort the records are not used.)
        float4 *const rec = reinterpret_cast<float4 *>(ring_ptr);
        float *const rec_u = reinterpret_cast<float *>(ring_ptr + 4 * kVmMaxRows * sizeof(float4));
#pragma unroll
        for (int k = 0; k < 2 * kMaxChunks; ++k) {
            if (!(live >> k & 1u))
                continue;
            const int h = k / kMaxChunks, c = h * kBN + chunk_of(h, k % kMaxChunks) * 32 + lane;
            rec[q * kVmMaxRows + c] = make_float4(st[k].m, st[k].s, __int_as_float(st[k].am), st[k].tlog);
            if (kEntropy)
                rec_u[q * kVmMaxRows + c] = st[k].u;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kVmEpiWarps) : "memory");
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int c = (int)threadIdx.x - 64, row = row_of(i, c);  // column c of accumulator i
            if (c >= (i ? hw1 : hw0) || row >= a.N)
                continue;
            float m = -INFINITY, s = 0.f, u = 0.f, t = -INFINITY;
            int32_t am = INT32_MAX;
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
                const float4 r = rec[qq * kVmMaxRows + i * kBN + c];
                if (kEntropy)
                    combine_u(m, s, u, am, r.x, r.y, rec_u[qq * kVmMaxRows + i * kBN + c], __float_as_int(r.z));
                else
                    combine(m, s, am, r.x, r.y, __float_as_int(r.z));
                t = fmaxf(t, r.w);
            }
            pend[i] = make_float4(m, s, __int_as_float(am), t);
            pend_u[i] = u;
            pend_idx[i] = (int64_t)row * (2 * a.G) + 2 * col + (int)rank;
        }
    }

    // Neither CTA releases TMEM, or exits, while its peer may still use the pair's TMEM or barriers (see score.cu).
    ptx::tc_fence_before();
    __syncthreads();
    if (tl && threadIdx.x == 0)
        tl[5] = ptx::globaltimer_ns();
    const bool gave_up = *reinterpret_cast<volatile int32_t *>(&bars->abort) != 0;
    if (gave_up)
        ptx::cluster_arrive_release();
    else
        ptx::cluster_arrive_relaxed();
#pragma unroll
    for (int i = 0; i < 2; ++i)
        if (pend_idx[i] >= 0) {
            a.part[pend_idx[i]] = pend[i];
            if (kEntropy)
                a.part_u[pend_idx[i]] = pend_u[i];
        }
    if (threadIdx.x == 64) {
        // Warp 2 has passed griddepcontrol.wait: a failure recorded now belongs to this call (see score.cu).
        if (!tmem_ok)
            atomicExch(&a.status->current, (int32_t)WINO_ERR_UNSUPPORTED);
        else if (gave_up)
            atomicExch(&a.status->current, (int32_t)WINO_ERR_DEVICE_TIMEOUT);
    }
    ptx::cluster_wait_acquire();
    ptx::tc_fence_after();
    if (gave_up)
        settle_peer_arrivals();
    if (warp == 1)
        ptx::tmem_dealloc_pair(tmem, kTmemCols);
    if (tl && threadIdx.x == 0)
        tl[6] = ptx::globaltimer_ns();
}

}  // namespace

namespace {

// The split over n_groups row groups: each group of pairs owns hw[0] + hw[1] consecutive rows of H and, as in
// score.cu, walks the vocabulary tiles side by side.  Two records per pair (one per CTA) and row.  False when it
// cannot run with that many groups.
bool vm_split(int64_t N, int64_t n_kb, int64_t V, int max_units, int32_t records_cap, int32_t n_groups, VmSchedule *out)
{
    VmSchedule s{};
    const int64_t rows = (N + n_groups - 1) / n_groups;
    if (rows > kVmMaxRows || n_groups > max_units)
        return false;
    s.n_groups = n_groups;
    // accumulator widths: multiples of 32 up to 128, of 16 above; the first one no narrower than the second
    const int32_t n16 = (int32_t)((rows + 15) / 16);
    s.hw[0] = rows > kBN ? (n16 + 1) / 2 * 16 : (rows > 128 ? n16 * 16 : (n16 + 1) / 2 * 32);
    s.hw[1] = rows > kBN ? n16 / 2 * 16 : 0;
    if ((int64_t)(s.hw[0] + s.hw[1]) * (n_groups - 1) >= N)
        return false;  // the last group would own no rows
    // the epilogue reads whole 32-column chunks: up to 16 columns past the last accumulator
    const int32_t slots = ((int32_t)kTmemCols - s.hw[0] % 32) / s.hw[0];
    s.slots = slots < kVmMaxSlots ? slots : kVmMaxSlots;
    const int64_t g = max_units / n_groups;
    if (2 * g > records_cap || 2 * g > kMaxRecordsPerRow)
        return false;  // a vocabulary too small for two records from every pair
    const int64_t tiles = ((V + kBN - 1) / kBN + g - 1) / g;  // on the busiest pair, at the widest tile
    int64_t bn = kBN;
    if (n_groups == 1 && rows <= kVmEvenTileRows) {
        bn = ((V + tiles * g - 1) / (tiles * g) + 15) / 16 * 16;
        bn = bn < kMinBN ? kMinBN : bn;
    }
    s.bn = (int32_t)bn;
    s.n_vt = (int32_t)((V + bn - 1) / bn);
    s.G = (int32_t)(g < s.n_vt ? g : s.n_vt);
    const int64_t w = s.hw[0] + s.hw[1], chunks = (s.hw[0] + 31) / 32 + (s.hw[1] + 31) / 32;
    const int64_t epilogue = (chunks + 1) / 2 * 540, rem = s.n_vt % s.G;
    const bool two = s.hw[1] > 0, capped = n_kb >= kVmCappedSlices;
    const int64_t mma = two ? (capped ? n_kb * (60 + w * 7 / 5) + 4 * w : n_kb * (w * 5 / 4 - 12) + 8 * w)
                            : n_kb * (capped ? 190 + w * 3 / 4 : 204 + w * 2 / 9);
    int64_t tile = mma > epilogue ? mma : epilogue;
    if (!two && !capped)
        tile += (mma < epilogue ? mma : epilogue) / 3;
    s.split = two && rem > 0 && 2 * rem <= s.G;
    s.cost = epilogue + tiles * tile - (s.split ? tile * 3 / 10 : 0);
    s.stage_bytes = kVmStageBytesW + (uint32_t)((s.hw[0] + s.hw[1]) / 2) * 128u;
    const uint32_t fit = kVmRingCapacity / s.stage_bytes;
    s.stages = (int32_t)(fit < (uint32_t)kVmMaxStages ? fit : (uint32_t)kVmMaxStages);
    *out = s;
    return true;
}

}  // namespace

bool score_vmajor_schedule(int64_t N, int64_t d, int64_t V, int max_units, int32_t records_cap,
                           const ScoreSchedule &rows, VmSchedule *out)
{
    const int64_t n_kb = (d + kBK - 1) / kBK;
    bool found = false;
    const int32_t most = N <= kPairM ? 1 : kVmMaxGroups;  // one row block is bound by the W stream: no second reader
    for (int32_t g = 1; g <= most; ++g) {
        VmSchedule s;
        if (vm_split(N, n_kb, V, max_units, records_cap, g, &s) && (!found || s.cost < out->cost)) {
            *out = s;
            found = true;
        }
    }
    if (!found || N <= kVmShortRows)
        return found;
    if (n_kb < kVmMinSlices)
        return false;
    const int64_t blocks = (N + kPairM - 1) / kPairM;
    const int64_t row_tiles = (blocks + rows.n_groups - 1) / rows.n_groups * ((rows.n_vt + rows.G - 1) / rows.G);
    if (blocks == 1)
        return V * d >= kVmLongHead && out->cost < row_tiles * n_kb * kRowOneBlockSliceNs;
    const int64_t row_tile = n_kb >= kVmCappedSlices ? n_kb * 380 * (rows.bn + 144) / 400 + 700
                                                     : n_kb * 352 * (rows.bn - 55) / 201 + 607;
    return out->cost < row_tiles * row_tile + 5 * rows.bn;
}

cudaError_t launch_score_vmajor(const CUtensorMap &tmH, const CUtensorMap &tmW, const ScoreArgs &a, bool entropy,
                                cudaStream_t stream)
{
    static std::mutex mu;
    static bool done[64];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return cudaErrorUnknown;
    {
        std::lock_guard<std::mutex> g(mu);
        if (!done[dev]) {
            for (auto *k : {score_vmajor_kernel<false>, score_vmajor_kernel<true>}) {
                const cudaError_t e =
                    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kScoreSmemMax);
                if (e != cudaSuccess)
                    return e;
            }
            done[dev] = true;
        }
    }
    // The ring must hold the stages and, at the end, the row records; the TMEM columns the accumulators.
    const uint64_t ring = (uint64_t)a.stages * a.stage_bytes;
    if (a.stages < 2 || a.stages > kVmMaxStages || ring > kVmRingCapacity || ring < kVmMaxRows * 4 * 20 ||
        a.hw[0] % 16 != 0 || a.hw[1] % 16 != 0 || a.hw[0] < 32 || a.hw[0] > kBN || a.hw[1] < 0 || a.hw[1] > a.hw[0] ||
        a.slots < 2 || a.slots > kVmMaxSlots || a.slots * a.hw[0] + a.hw[0] % 32 > (int32_t)kTmemCols ||
        a.bn % 16 != 0 || a.bn > kPairM || a.stage_bytes != kVmStageBytesW + (uint32_t)((a.hw[0] + a.hw[1]) / 2) * 128u)
        return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = score_launch_config((unsigned)(2 * a.n_groups * a.G), kVmThreads,
                                                 vmajor_smem_bytes((uint32_t)ring), stream, attr);
    return entropy ? cudaLaunchKernelEx(&cfg, score_vmajor_kernel<true>, tmH, tmW, a)
                   : cudaLaunchKernelEx(&cfg, score_vmajor_kernel<false>, tmH, tmW, a);
}

}  // namespace wino
