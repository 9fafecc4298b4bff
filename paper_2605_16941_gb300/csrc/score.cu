// score.cu -- fused LM-head GEMM + full-vocabulary softmax statistics (sm_103a).
//
// For every scored row h_n the method needs three numbers of the model's
// distribution p(. | Y~) = softmax_v(<h_n, w_v>) over the whole vocabulary
// (Eq. 2 and Eq. 3 of the WINO paper): argmax_v p, max_v p and p(target).
// The logits never leave the chip: each CTA pair computes logit tiles of 256
// rows x bn vocabulary columns with 2-SM tensor-core MMAs
// (tcgen05.mma.cta_group::2, bf16 x bf16 -> fp32 in TMEM, M = 256 split
// 128/128 over the two SMs, N = bn <= 256), and eight epilogue warps per CTA
// fold each tile straight out of TMEM into a running per-row state (max, sum
// of exp, argmax, target logit) that lives in registers across all of the
// pair's vocabulary tiles of that row block.  One partial record per
// (row, pair) goes to the workspace; finish.cu merges them.
//
// Row counts that leave much of their 256-row blocks empty, and a few others, go to the vocabulary-major kernel
// instead (score_vmajor.cu; the rule is score_vmajor_schedule).
//
// Two modes (ScoreArgs::two, chosen per launch by score_schedule):
//   single tiles, for shapes bound by the W stream from HBM (one 256-row
//     block): the two accumulators alternate between consecutive tiles, so
//     the epilogue of one tile overlaps the MMAs of the next, and the ring has
//     up to 7 stages, the most W bytes in flight per SM;
//   passes, for tensor-bound shapes: a stage holds three 16 KB slots and
//     feeds both accumulators, a quarter fewer bytes delivered per SM and MMA
//     than single tiles.  A group of pairs that owns two or more row blocks
//     takes them two at a time (row-pair sweeps): the two blocks' H slices
//     and one tile's W slice, so every W slice staged serves both blocks and
//     the group streams W from HBM once per two blocks.  A block left without
//     a partner is swept alone (tile-pair sweeps): its H slice and the slices
//     of two tiles.  The accumulators then fill TMEM, so a pass's MMAs into
//     the first accumulator start as soon as the epilogue has read it, and
//     its MMAs into the second accumulator for the first ring stages are
//     deferred until the epilogue has read that one too (the stages are
//     released after those).
//
// Kernel structure (persistent, clusters of 2 CTAs = one SM pair, 320 threads each):
//   warp 0  TMA producer (both CTAs): per K slice, its 128 rows of H (of one
//           or two row blocks) and its bn/2 of the (one or two) tiles' W rows
//           into the ring; both CTAs' copies complete on the LEADER's stage
//           barrier;
//   warp 1  TMEM allocation (both CTAs, all 512 columns) and, in the leader
//           only, the MMA issuer: 4 x (M256 Nbn K16) per stage and tile,
//           committing stage release and accumulator-ready to both CTAs
//           (multicast);
//           Both of these roles run in one thread of their warp, chosen by
//           elect.sync: behind a branch on the lane index the compiler cannot
//           know that the operands of tcgen05.mma, tcgen05.commit and the
//           copies are warp-uniform, and issuing a K slice's MMAs then took
//           longer than the MMAs themselves.  Branch on the lane index and a
//           shuffle per wait, then elect.sync (us per step, 20-step regions;
//           d = 4096, V = 126464): N = 64 168 -> 156, N = 256
//           179 -> 166, N = 2048 1092 -> 1070; d = 1024, V = 64000, N = 2048
//           247 -> 201;
//   warps 2-9 epilogue (both CTAs): two warps per TMEM lane quarter, on the
//           even and the odd 32-column chunks of every tile; one thread per row
//           (TMEM lane) and warp.  Online softmax over its chunks, then release
//           of the accumulator to the leader's MMA warp.  At the end of a sweep
//           the second warp's row states are merged into the first one's.
//           The epilogue is latency-bound in a single warp per scheduler (25-30
//           cycles per column against 5 instructions), and a pass's MMAs wait
//           for it.  One warp per quarter, then two with the packed fold of
//           fold.cuh and accumulator 0 handed over before accumulator 1 is
//           done (us per step, V = 64000, N = 2048): d = 256 107 -> 74, d = 1024
//           200 -> 182; d = 4096, V = 126464 1195 -> 1173; three or four warps
//           per quarter: 72 / 73, 182 / 183, no change.  That was with a release
//           at cluster scope in every accumulator release, a memory barrier that
//           held each warp for about as long as a chunk's fold; with a relaxed
//           arrival d = 256 73.4 -> 58.3, d = 1024 168.7 -> 165.5.
// Work split: see ScoreArgs in internal.h.
//
// Every mbarrier wait is bounded (kWaitLimitNs): on expiry the CTA raises an
// abort flag and drains its in-flight copies and MMAs (again bounded); both
// CTAs then meet at the closing cluster barrier before TMEM is released, and
// the CTA records WINO_ERR_DEVICE_TIMEOUT in the call's status word.
//
// Optional timeline (ScoreArgs::timeline, diagnostics only): per CTA,
// globaltimer stamps [0] entry, [1] set-up done (barriers, TMEM), [2] first
// TMA issue, [3] griddepcontrol.wait returned in the epilogue, [4] last MMA
// completed (leader) or last tile read (peer), [5] all roles done, [6] exit;
// [7] = SM id << 32 | tiles of the pair.
#include <mutex>

#include "fold.cuh"
#include "internal.h"
#include "ptx.cuh"
#include "wait.cuh"

namespace wino {
namespace {

constexpr uint16_t kBothCtas = 0x3;
constexpr int kPrefetchSlices = 4;   // K slices of the first W tile prefetched into L2 before the grid wait

struct alignas(8) Barriers {
    uint64_t full[kMaxStages];   // leader: both CTAs' copies of a stage landed
    uint64_t empty[kMaxStages];  // both: the stage's MMAs are done (multicast commit)
    uint64_t tmem_full[2];       // both: accumulator i holds a finished tile (multicast commit)
    uint64_t tmem_empty[2];      // leader: every epilogue warp of the pair has read accumulator i
    uint64_t mma_done;           // leader: every MMA issued has completed
    uint32_t tmem_base;
    int32_t abort;
};
static_assert(sizeof(Barriers) <= 256, "barrier block must fit its reserve");

// Fold this warp's share of the nvalid first columns of one accumulator (32 TMEM lanes from tbase), vocabulary ids
// v0 ..: every kEpiPerQuarter-th 32-column chunk from chunk `sel` on.
template <bool kEntropy>
__device__ __forceinline__ void fold_tile(RowState &r, uint32_t tbase, int sel, int v0, int nvalid, int tgt)
{
#pragma unroll 1
    for (int c = sel * 32; c < nvalid; c += 32 * kEpiPerQuarter) {
        float x[32];
        ptx::tmem_ld_32x32b_x32(tbase + (uint32_t)c, x);
        ptx::tmem_ld_wait();
        fold32<kEntropy>(r, x, v0 + c, nvalid - c, tgt);
    }
}

// One row's state as the other epilogue warps of its lane quarter hand it over.
struct RowPart {
    float m[kBM], s[kBM], tlog[kBM], u[kBM];
    int32_t am[kBM];
};
static_assert(2 * (kEpiPerQuarter - 1) * sizeof(RowPart) == kMergeBytes, "merge scratch");

// kTwo: passes (ScoreArgs::two == 1: row-pair and tile-pair sweeps), else single tiles.
template <bool kEntropy, bool kTwo>
__global__ void __launch_bounds__(kScoreThreads, 1)
    score_kernel(const __grid_constant__ CUtensorMap tmH, const __grid_constant__ CUtensorMap tmW,
                 const ScoreArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;  // swizzle atoms need 1024-B alignment
    const uint32_t ring_bytes = (uint32_t)a.stages * a.stage_bytes;
    Barriers *bars = reinterpret_cast<Barriers *>(smem_raw + (ring - raw) + ring_bytes + (kTwo ? kMergeBytes : 0u));
    // Scratch for merging a row's states at the end of a sweep.  Single tiles have one sweep per launch, at whose end
    // the ring is free.
    RowPart *const parts = reinterpret_cast<RowPart *>(smem_raw + (ring - raw) + (kTwo ? ring_bytes : 0u));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();  // 0: leader (issues the MMAs), 1: peer
    const bool leader = rank == 0;
    const int pair = blockIdx.x >> 1;
    uint64_t *const tl = a.timeline ? a.timeline + (size_t)blockIdx.x * kTimelineWords : nullptr;
    // The records of an epilogue thread's last sweep (one row, or two in a row-pair sweep) are stored after
    // this CTA's arrival on the closing cluster barrier, so that the barrier's release does not wait for them.
    float4 pend[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    float pend_u[2] = {0.f, 0.f};
    int64_t pend_idx[2] = {-1, -1};
    if (tl && threadIdx.x == 0)
        tl[0] = ptx::globaltimer_ns();

    const int S = a.stages;
    const uint32_t wb = stage_bytes_w(a.bn);
    auto sA = [&](int s) { return ring + (uint32_t)s * a.stage_bytes; };
    auto sB = [&](int s, int t) { return sA(s) + kStageBytesA + (uint32_t)t * wb; };
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
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(tfull(i), 1);
            ptx::mbar_init(tempty(i), 2 * kEpiWarps);  // the epilogue warps of both CTAs
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
        // Both CTAs of the pair take part in the pair allocation, which reserves the same columns in
        // both SMs; the address check below refuses to run if the two CTAs were given different ones.
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

    // Programmatic launch: everything above overlapped the grid before us.  Whatever that grid is (the
    // previous WINO call's finish kernel, or a kernel of the caller's that wrote H), its writes are only
    // visible after griddepcontrol.wait, so every role waits before its first global access; the producer
    // first prefetches the start of its first W tile into L2, which is safe before the wait (L2 is coherent).
    ptx::grid_dep_launch_dependents();

    const int grp = pair % a.n_groups;  // 256-row blocks grp, grp + n_groups, ...
    const int col = pair / a.n_groups;  // vocabulary tiles col, col + G, ...
    // Sweeps over the pair's vocabulary tiles.  Single tiles: one sweep per row block, one tile per item.
    // Passes: row blocks mb and mb + n_groups together (row-pair sweep: item = one tile of both blocks, so
    // each W slice staged serves both and the group reads W once per two blocks), or a block left without
    // a partner alone (tile-pair sweep: item = tiles vt and vt + G of that block).
    const int mb_step = kTwo ? 2 * a.n_groups : a.n_groups;
    const int vstep = kTwo ? 2 * a.G : a.G;  // tiles per item of a single-tile or tile-pair sweep

    if (warp >= 2 || !tmem_ok) {
        ptx::grid_dep_wait();
        if (tl && threadIdx.x == 64)
            tl[3] = ptx::globaltimer_ns();
        if (threadIdx.x >= 64)
            for (int i = blockIdx.x * (32 * kEpiWarps) + (int)threadIdx.x - 64; i < a.n_tickets;
                 i += gridDim.x * (32 * kEpiWarps))
                a.tickets[i] = 0;
    }
    if (!tmem_ok) {
        // nothing to do: the status word reports the failed allocation check
    } else if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (both CTAs)
        if (ptx::elect_one()) {
            const int half_bn = a.bn >> 1;  // W rows each CTA stages per tile
            // W map coordinates of (K slice kb, vocabulary row v): (64 kb, v) in row-major W, (0, kb V + v) in the
            // panel copy
            auto w_x = [&](int kb) { return a.w_panels ? 0 : kb * kBK; };
            auto w_y = [&](int kb, int v) { return a.w_panels ? kb * a.V + v : v; };
            if (grp < a.n_mb)
                for (int kb = 0; kb < min(a.n_kb, kPrefetchSlices); ++kb)
                    ptx::tma_prefetch_2d(&tmW, w_x(kb), w_y(kb, col * a.bn + (int)rank * half_bn));
            ptx::grid_dep_wait();
            const uint64_t pol_h = ptx::policy_evict_last();    // H is re-read for every item
            const uint64_t pol_w = ptx::policy_evict_normal();  // W is shared by the row-block groups
            int stage = 0;
            uint32_t phase = 0;
            int64_t issued = 0;  // stages filled so far
            bool aborted = false;
            for (int mb = grp; mb < a.n_mb && !aborted; mb += mb_step) {
                const int mb2 = mb + a.n_groups;  // partner row block of a row-pair sweep
                const bool rows2 = kTwo && mb2 < a.n_mb;
                for (int vt = col; vt < a.n_vt && !aborted; vt += rows2 ? a.G : vstep) {
                    const bool two = kTwo && (rows2 || vt + a.G < a.n_vt);
                    // both CTAs' copies: H, the tile's W, and the partner block's H or the second tile's W
                    const uint32_t stage_tx = 2u * (kStageBytesA + wb + (rows2 ? kStageBytesA : (two ? wb : 0u)));
                    for (int kb = 0; kb < a.n_kb; ++kb) {
                        if (!wait_bounded(empty(stage), phase ^ 1u, &bars->abort)) {
                            aborted = true;
                            break;
                        }
                        const uint32_t bar = ptx::mapa(full(stage), 0);  // the leader's stage barrier
                        if (leader)
                            ptx::mbar_arrive_expect_tx(full(stage), stage_tx);
                        ptx::tma_load_2d_pair(sA(stage), &tmH, bar, kb * kBK, mb * kPairM + (int)rank * kBM, pol_h);
                        ptx::tma_load_2d_pair(sB(stage, 0), &tmW, bar, w_x(kb),
                                              w_y(kb, vt * a.bn + (int)rank * half_bn), pol_w);
                        if (rows2)
                            ptx::tma_load_2d_pair(sB(stage, 1), &tmH, bar, kb * kBK,
                                                  mb2 * kPairM + (int)rank * kBM, pol_h);
                        else if (two)
                            ptx::tma_load_2d_pair(sB(stage, 1), &tmW, bar, w_x(kb),
                                                  w_y(kb, (vt + a.G) * a.bn + (int)rank * half_bn), pol_w);
                        if (tl && issued == 0)
                            tl[2] = ptx::globaltimer_ns();
                        ++issued;
                        if (++stage == S) {
                            stage = 0;
                            phase ^= 1u;
                        }
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
            const uint32_t idesc = ptx::idesc_bf16_f32(kPairM, (uint32_t)a.bn);
            int tiles = 0;
            int stage = 0;
            uint32_t phase = 0;
            int item = 0;  // items issued so far
            bool last_two = true;  // whether the last item used both accumulators
            bool aborted = false;
            auto wait_acc_free = [&](int i, uint32_t uses) -> bool {  // the epilogue has read use uses-1 of acc i
                const bool ok = wait_bounded<true>(tempty(i), (uses & 1u) ^ 1u, &bars->abort);
                ptx::tc_fence_after();
                return ok;
            };
            auto issue = [&](int acc, uint32_t a_smem, uint32_t b_smem, int kb) {  // 4 x K16 from one stage
                const uint64_t da = ptx::sdesc_kmajor_sw128(a_smem);
                const uint64_t db = ptx::sdesc_kmajor_sw128(b_smem);
#pragma unroll
                for (int k = 0; k < kBK / 16; ++k)  // +32 B along K per MMA = +2 in the encoded address
                    ptx::mma_bf16_pair(tmem + (uint32_t)acc * kBN, da + 2u * k, db + 2u * k, idesc, (kb | k) != 0);
            };
            for (int mb = grp; mb < a.n_mb && !aborted; mb += mb_step) {
                const bool rows2 = kTwo && mb + a.n_groups < a.n_mb;
                // accumulator 1 of a pass: the partner block's H (third slot) x the tile's W, or this block's
                // H x the second tile's W (third slot)
                auto issue1 = [&](int s, int kb) {
                    issue(1, rows2 ? sB(s, 1) : sA(s), rows2 ? sB(s, 0) : sB(s, 1), kb);
                };
                for (int vt = col; vt < a.n_vt && !aborted; vt += rows2 ? a.G : vstep, ++item) {
                    const bool two = kTwo && (rows2 || vt + a.G < a.n_vt);
                    // single tiles: item i uses accumulator i & 1 for the (i >> 1)-th time;
                    // passes: item i uses both accumulators for the i-th time
                    const int acc0 = kTwo ? 0 : (item & 1);
                    const uint32_t uses0 = kTwo ? (uint32_t)item : (uint32_t)(item >> 1);
                    if (!wait_acc_free(acc0, uses0)) {
                        aborted = true;
                        break;
                    }
                    const int defer = two ? min(S, a.n_kb) : 0;  // stages whose second-accumulator MMAs wait
                    const int s0 = stage;
                    for (int kb = 0; kb < a.n_kb; ++kb) {
                        if (!wait_bounded(full(stage), phase, &bars->abort)) {
                            aborted = true;
                            break;
                        }
                        issue(acc0, sA(stage), sB(stage, 0), kb);
                        if (kTwo && kb == a.n_kb - 1)  // accumulator 0 is done: its epilogue need not wait for 1
                            ptx::mma_commit_pair_multicast(tfull(0), kBothCtas);
                        if (kb < defer) {
                            if (kb == defer - 1) {  // the second accumulator is needed now
                                if (!wait_acc_free(1, (uint32_t)item)) {
                                    aborted = true;
                                    break;
                                }
                                int sj = s0;
                                for (int j = 0; j < defer; ++j) {
                                    issue1(sj, j);
                                    ptx::mma_commit_pair_multicast(empty(sj), kBothCtas);
                                    if (++sj == S)
                                        sj = 0;
                                }
                            }
                        } else {
                            if (two)
                                issue1(stage, kb);
                            ptx::mma_commit_pair_multicast(empty(stage), kBothCtas);
                        }
                        if (++stage == S) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                    if (aborted)
                        break;
                    // The epilogue waits for both accumulators of every pass, or for the tile's one.  This commit is
                    // the item's last: whoever has waited for it has the stage barriers' arrivals behind it as well,
                    // assuming that the arrivals of one thread's successive commits reach a CTA in their order (PTX
                    // states that each follows the MMAs issued before its commit, not an order among them).
                    ptx::mma_commit_pair_multicast(tfull(kTwo ? 1 : acc0), kBothCtas);
                    tiles += two ? 2 : 1;
                    last_two = two;
                }
            }
            // The release of accumulator 1 that no later item has waited for (see the closing barrier).
            if (kTwo && !aborted && !last_two && item > 1)
                wait_acc_free(1, (uint32_t)(item - 1));
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
        // ------------------------------------------------------------ epilogue (warps 2.., both CTAs)
        const int q = warp & 3;           // this warp may only read TMEM lanes [32q, 32q + 32)
        const int sel = (warp - 2) >> 2;  // which of the quarter's warps
        const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
        int item = 0;
        bool aborted = false;
        auto take = [&](int i, uint32_t uses) -> bool {  // wait for use `uses` of accumulator i
            int ok = 1;
            if (lane == 0)
                ok = wait_bounded(tfull(i), uses & 1u, &bars->abort);
            ok = __shfl_sync(0xffffffffu, ok, 0);
            ptx::tc_fence_after();
            return ok != 0;
        };
        // Items of this pair, and how many later an accumulator is used again.
        int n_items = 0;
        for (int mb = grp; mb < a.n_mb; mb += mb_step) {
            const int step = (kTwo && mb + a.n_groups < a.n_mb) ? a.G : vstep;
            n_items += (a.n_vt - col + step - 1) / step;
        }
        const int reuse = kTwo ? 1 : 2;
        // Accumulator i fully read by this warp: tell the leader's MMA warp, if it waits for that (see the closing barrier).
        auto release = [&](int i) {
            if (item + reuse >= n_items)
                return;
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0)
                ptx::mbar_arrive_cluster_relaxed(ptx::mapa(tempty(i), 0));
        };
        auto epilogue_sync = [&] { asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory"); };
        const RowState r0{-INFINITY, 0.f, 0.f, 0.f, 0.f, -INFINITY, 0.f, 0.f, 0.f, 0.f, 0};
        for (int mb = grp; mb < a.n_mb; mb += mb_step) {
            const int mb2 = mb + a.n_groups;
            const bool rows2 = kTwo && mb2 < a.n_mb;
            const int64_t in_block = (int)rank * kBM + q * 32 + lane;
            const int64_t row = (int64_t)mb * kPairM + in_block;
            const int64_t row2 = rows2 ? (int64_t)mb2 * kPairM + in_block : (int64_t)a.N;  // a.N: no row
            const int32_t tgt = (row < a.N) ? row_target(a.ts, row, a.V) : -1;
            const int32_t tgt2 = (row2 < a.N) ? row_target(a.ts, row2, a.V) : -1;
            RowState r = r0, r2 = r0;  // r2: the partner block's row in a row-pair sweep
            for (int vt = col; vt < a.n_vt && !aborted; vt += rows2 ? a.G : vstep, ++item) {
                const int acc0 = kTwo ? 0 : (item & 1);
                const uint32_t uses0 = kTwo ? (uint32_t)item : (uint32_t)(item >> 1);
                if (!take(acc0, uses0)) {
                    aborted = true;
                    break;
                }
                fold_tile<kEntropy>(r, lanes + (uint32_t)acc0 * kBN, sel, vt * a.bn, min(a.bn, a.V - vt * a.bn), tgt);
                release(acc0);
                if (kTwo) {
                    if (!take(1, (uint32_t)item)) {
                        aborted = true;
                        break;
                    }
                    const int vt1 = vt + a.G;
                    if (rows2)
                        fold_tile<kEntropy>(r2, lanes + kBN, sel, vt * a.bn, min(a.bn, a.V - vt * a.bn), tgt2);
                    else if (vt1 < a.n_vt)
                        fold_tile<kEntropy>(r, lanes + kBN, sel, vt1 * a.bn, min(a.bn, a.V - vt1 * a.bn), tgt);
                    release(1);
                }
            }
            // Merge the states of the quarter's warps into the first one's.  (Every warp of the CTA comes here as
            // often, aborted or not; after an abort the records are not used.)
            if (sel > 0)
#pragma unroll
                for (int i = 0; i < (kTwo ? 2 : 1); ++i) {
                    RowPart &p = parts[(sel - 1) * 2 + i];
                    const RowState &x = i ? r2 : r;
                    const int k = q * 32 + lane;
                    p.m[k] = x.m;
                    p.s[k] = (x.s0 + x.s1) + (x.s2 + x.s3);
                    p.tlog[k] = x.tlog;
                    p.am[k] = x.am;
                    if (kEntropy)
                        p.u[k] = (x.u0 + x.u1) + (x.u2 + x.u3);
                }
            epilogue_sync();
            if (sel == 0)
#pragma unroll
                for (int i = 0; i < (kTwo ? 2 : 1); ++i) {
                    if (pend_idx[i] >= 0) {  // the previous sweep's records, then this sweep's become pending
                        a.part[pend_idx[i]] = pend[i];
                        if (kEntropy)
                            a.part_u[pend_idx[i]] = pend_u[i];
                    }
                    const RowState &x = i ? r2 : r;
                    float m = x.m, s = (x.s0 + x.s1) + (x.s2 + x.s3), t = x.tlog, u = (x.u0 + x.u1) + (x.u2 + x.u3);
                    int32_t am = x.am;
#pragma unroll
                    for (int j = 0; j < kEpiPerQuarter - 1; ++j) {
                        const RowPart &p = parts[j * 2 + i];
                        const int k = q * 32 + lane;
                        if (kEntropy)
                            combine_u(m, s, u, am, p.m[k], p.s[k], p.u[k], p.am[k]);
                        else
                            combine(m, s, am, p.m[k], p.s[k], p.am[k]);
                        t = fmaxf(t, p.tlog[k]);
                    }
                    pend[i] = make_float4(m, s, __int_as_float(am), t);
                    pend_u[i] = u;
                    const int64_t rr = i ? row2 : row;
                    pend_idx[i] = rr < a.N ? rr * a.G + col : -1;
                }
            if (kTwo)
                epilogue_sync();  // before the next sweep's states overwrite the scratch
        }
        if (tl && !leader && warp == 2 && lane == 0)
            tl[4] = ptx::globaltimer_ns();
    }

    // Neither CTA releases TMEM, or exits, while its peer may still use the pair's TMEM or barriers.  No memory access
    // needs ordering by this barrier unless a wait gave up: every arrival sent to the leader's barriers has been
    // waited for (for the peer's stage barriers see the item's last commit).  The release it then does without held every launch's end: us per step in a CUDA graph 6.9 -> 6.6
    // (d = 64, V = 1000, N = 64), 13.05 -> 12.56 (d = 512, V = 32000, N = 128).
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
        // Warp 2 has passed griddepcontrol.wait, so the previous call's finish kernel, which clears the
        // status word, has completed: a failure recorded now belongs to this call.
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

// Choose the mode, the tile width bn and the number of row-block groups.  One 256-row block is bound by the
// W stream from HBM: single tiles (the most bytes in flight).  More rows are tensor-bound: passes (fewer bytes
// delivered per MMA; row-pair sweeps where a group owns more than one row block).  Then: fewest vocabulary columns on the busiest pair plus a per-tile or
// per-pass overhead, the widest tile, fewest passes over W (more groups).  A width below kBN pays when the
// vocabulary then splits evenly over the pairs: V = 126464 on 76 pairs is 494 tiles of 256 (7 on the
// busiest pair, 6.5 on average) but 527 tiles of 240 (7 on 71 pairs).
constexpr int32_t kPassMinRowBlocks = 2;  // fewest 256-row blocks that use passes
static_assert(kPassMinRowBlocks <= 2, "single tiles merge their row states in the ring, which is free after one sweep only");

ScoreSchedule score_schedule(int32_t n_mb, int64_t V, int max_units, int32_t records_cap)
{
    constexpr int64_t kTileOverheadCols = 16;  // single tiles: H re-staged per tile, in columns
    constexpr int64_t kPassOverheadCols = 32;  // passes: the epilogue the next pass partly waits for
    const int32_t two = n_mb >= kPassMinRowBlocks ? 1 : 0;
    ScoreSchedule best{kBN, (int32_t)((V + kBN - 1) / kBN), 1, 1, two, 2, 0};
    int64_t best_cost = -1;
    const int32_t top = n_mb < max_units ? n_mb : max_units;
    for (int32_t bn = kBN; bn >= kMinBN; bn -= 16) {
        const int64_t n_vt = (V + bn - 1) / bn;
        for (int32_t groups = top; groups >= 1; --groups) {
            int64_t g = max_units / groups;
            g = g < n_vt ? g : n_vt;
            g = g < records_cap ? g : records_cap;
            g = g < kMaxRecordsPerRow ? g : kMaxRecordsPerRow;
            g = g < 1 ? 1 : g;
            const int64_t tiles = (n_vt + g - 1) / g;  // on the busiest pair, per row block
            const int64_t per_mb = two ? tiles * bn + ((tiles + 1) / 2) * kPassOverheadCols
                                       : tiles * (bn + kTileOverheadCols);
            const int64_t cost = (int64_t)((n_mb + groups - 1) / groups) * per_mb;
            if (best_cost < 0 || cost < best_cost) {
                best_cost = cost;
                best.bn = bn;
                best.n_vt = (int32_t)n_vt;
                best.n_groups = groups;
                best.G = (int32_t)g;
            }
        }
    }
    // A pass stage has a third slot: the second tile's W, or in a row-pair sweep (a group with more than
    // one row block) the partner block's H.
    const uint32_t wb = stage_bytes_w(best.bn);
    const uint32_t capacity = two ? kPassRingCapacity : kRingCapacity;
    const bool row_pairs = two && n_mb > best.n_groups;
    best.stage_bytes = kStageBytesA + wb + (two ? (row_pairs && wb < kStageBytesA ? kStageBytesA : wb) : 0u);
    const uint32_t fit = capacity / best.stage_bytes;
    best.stages = (int32_t)(fit < (uint32_t)kMaxStages ? fit : (uint32_t)kMaxStages);
    return best;
}

cudaLaunchConfig_t score_launch_config(unsigned grid, unsigned threads, uint32_t smem, cudaStream_t stream,
                                       cudaLaunchAttribute (&attr)[2])
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

namespace {

// Per-device one-time set-up: shared-memory opt-in and the number of co-resident pairs.
int configure_device()
{
    static std::mutex mu;
    static int pairs[64];
    static bool done[64];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return -1;
    std::lock_guard<std::mutex> g(mu);
    if (!done[dev]) {
        for (auto *k : {score_kernel<false, false>, score_kernel<false, true>, score_kernel<true, false>,
                        score_kernel<true, true>})
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit) !=
                cudaSuccess)
                return -1;
        cudaLaunchAttribute attr[2];
        // Any launch's shared memory exceeds half an SM's, so one CTA per SM whatever the ring size.
        cudaLaunchConfig_t cfg = score_launch_config(2, kScoreThreads, kSmemLimit, nullptr, attr);
        cfg.numAttrs = 1;  // the cluster shape is what matters for the occupancy query
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, score_kernel<false, true>, &cfg) != cudaSuccess || clusters < 1)
            return -1;
        pairs[dev] = clusters;
        done[dev] = true;
    }
    return pairs[dev];
}

}  // namespace

int score_max_pairs() { return configure_device(); }

cudaError_t launch_score(const CUtensorMap &tmH, const CUtensorMap &tmW, const ScoreArgs &a, bool entropy,
                         cudaStream_t stream)
{
    if (configure_device() < 1)
        return cudaErrorUnknown;
    // The ring must hold what the producer stages: a pass's third slot takes an H box (16 KB) in a row-pair
    // sweep, which the launch has when a group owns more than one row block.
    const uint32_t wb = stage_bytes_w(a.bn);
    if (!a.two && a.n_mb > a.n_groups)
        return cudaErrorInvalidValue;  // a second sweep's copies would run into the merge scratch
    const uint32_t third = a.two ? (a.n_mb > a.n_groups && wb < kStageBytesA ? kStageBytesA : wb) : 0u;
    if (a.stages < 2 || a.stages > kMaxStages || a.stage_bytes < kStageBytesA + wb + third ||
        a.stage_bytes % 1024u != 0 || (uint64_t)a.stages * a.stage_bytes > (a.two ? kPassRingCapacity : kRingCapacity) ||
        (uint64_t)a.stages * a.stage_bytes < kMergeBytes)
        return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = score_launch_config((unsigned)(2 * a.n_groups * a.G), kScoreThreads,
                                                 score_smem_bytes(a.two != 0, (uint32_t)a.stages * a.stage_bytes), stream,
                                                 attr);
    if (entropy)
        return a.two ? cudaLaunchKernelEx(&cfg, score_kernel<true, true>, tmH, tmW, a)
                     : cudaLaunchKernelEx(&cfg, score_kernel<true, false>, tmH, tmW, a);
    return a.two ? cudaLaunchKernelEx(&cfg, score_kernel<false, true>, tmH, tmW, a)
                 : cudaLaunchKernelEx(&cfg, score_kernel<false, false>, tmH, tmW, a);
}

}  // namespace wino
