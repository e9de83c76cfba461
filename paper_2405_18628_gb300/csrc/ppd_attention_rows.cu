// ppd_attention_rows.cu -- tree-masked attention of the PPD verification step
// for trees of 65..512 tokens on sm_103a (paper Section 3 step (1): tree
// attention over the candidate tree; Section 4.1: every tree token attends to
// the cached prefix, its tree ancestors and itself).
//
// With more than 64 tree tokens the queries fill the tensor core's M side, so
// this kernel keeps one query per TMEM lane (queries zero-padded to 128).  Per
// block of 128 queries and tile of 128 keys:
//
//   S  = Q * K_tile^T          tcgen05.mma, M = 128 queries, N = 128 keys, K = D
//   P  = exp2(S*scale*log2e - m)   four softmax warps, one query row per thread;
//                              P is split into bf16 hi + lo and written back to
//                              TMEM over the scores it came from
//   O += P_hi * V + P_lo * V   tcgen05.mma with A read from TMEM, M = 128
//                              queries, N = D, two products per 16 keys
//
// A CTA runs two such streams, each with its own scores, output accumulator and
// softmax warps (warps 0-3 and 4-7), and the tensor core alternates between
// them: PV and the next S of one stream execute while the other stream's
// softmax runs.  The bound is the tensor pipe, 3 x 512 cycles per block and
// tile (D = 128), or HBM for trees of up to 128 tokens.  One stream with three
// score buffers, issued from one lane's branch, kept the pipe 43 % busy: the
// softmax and its hand-offs took longer than the pipe's work for a tile, and
// the issue of a tcgen05.mma ~100 cycles.  Steps at D = 128, from that form to this
// one: 32 x 32 slices, 285 tokens over 1500 keys 541 -> 430 us (its pipe time is 245);
// 96 tokens over 4096 keys (40 x 40 slices) 628 -> 561 us, 0.94 of the measured copy
// rate; eight ragged sequences of up to 16384 keys with 128 tokens (4 x 32 slices
// each) 1046 -> 885 us, the longest queue's share of the bytes taking 870.
// Measured on the way: probabilities handed over in one piece per tile, 5 %
// slower on 285 tokens; the softmax unrolled over a tile with its scores in
// registers, 606 us there (instruction fetch).  What the streams work on:
//
//   a pair job     two blocks of 128 queries of one (layer, sequence, head)
//                  slice, one per stream; every K and V tile is loaded once and
//                  read by both
//   a single job   one block; its tiles go to the streams in turn, and the two
//                  partial softmax states are merged at the job's end (a row's
//                  two accumulators sit in the same TMEM lane)
//
// Trees of 65-128 tokens are single jobs, 129-256 pair jobs, 385-512 two pair
// jobs a slice; 257-384 tokens are a pair and a single job, done by two groups
// of CTAs side by side so that the second reader of a slice finds it in L2.
// Launches with few slices take single jobs throughout (plan_rows).
//
// A thread owns a whole query row: the running maximum and the row sum are
// registers and no vote or exchange is needed.  The maximum is lazy: it moves
// only when a score exceeds it by more than 2^16, and the warp then rescales
// its rows of O (the PV product of the tile before is complete by then: the
// tensor pipe executes one thread's products in order, and the wait for S(i)
// covers everything issued before it).  The tree mask is a 128-bit ancestor
// bitset per tile and thread, built from the parent array in registers.
//
// The K and V tiles share one ring of shared-memory slots, loaded in the order
// the products consume them: K0 V0 K1 V1 ... for pair jobs, K0 K1 V0 K2 V1 ...
// for single jobs (an SM's copies land roughly in issue order, so a tile
// queued ahead of its turn would hold back the one needed first).
//
// The sharing of units among CTAs, the fused step's side warp and the merges of
// partial states are those of the kernel for trees of up to 64 tokens
// (ppd_attention.cu).  Warp roles (384 threads): warps 0-7 softmax, 8 TMA producer,
// 9 and 10 the streams' MMA issuers (9 owns TMEM), 11 the fused step's side work.
#include "ppd_attention_common.cuh"

#include <cmath>

namespace ppd {

template <int D_>
struct RowsLayout {
    static constexpr int D = D_;
    static constexpr int KT = 128;                         // keys per tile
    static constexpr int M = 128;                          // query rows per block (zero-padded)
    static constexpr int DCH = D / 64;                     // 64-column groups along D
    static constexpr uint32_t GROUP_BYTES = 128 * 128;     // 128 rows of 64 bf16
    static constexpr uint32_t TILE_BYTES = KT * D * 2;
    static constexpr uint32_t Q_BYTES = M * D * 2;
    static constexpr int QS = 2;                           // Q slots: one per stream, or two jobs' deep
    static constexpr int RS = (D == 64) ? 10 : 5;          // slots of the K/V tile ring

    static constexpr uint32_t OFF_Q = 0;
    static constexpr uint32_t OFF_R = OFF_Q + QS * Q_BYTES;
    static constexpr uint32_t OFF_BAR = OFF_R + RS * TILE_BYTES;
    static constexpr int B_QFULL = 0;
    static constexpr int B_QEMPTY = B_QFULL + QS;
    static constexpr int B_FULL = B_QEMPTY + QS;    // [RS] tile landed
    static constexpr int B_EMPTY = B_FULL + RS;     // [RS] every product that reads the slot is done
    static constexpr int B_SFULL = B_EMPTY + RS;    // [2] scores of the stream's tile in TMEM
    static constexpr int B_PFULL = B_SFULL + 2;     // [2][2] its probabilities, keys 0-63 and 64-127, in TMEM (4 warps)
    static constexpr int B_DONE = B_PFULL + 4;      // [2] the stream's last PV product of a job complete
    static constexpr int B_OFREE = B_DONE + 2;      // [2] a stream's output of a job read back from TMEM (8 arrivals)
    static constexpr int B_DRAIN = B_OFREE + 2;
    static constexpr int B_TURN = B_DRAIN + 1;      // [2] the other issuer is done with its turn
    static constexpr int NBAR = B_TURN + 2;
    static constexpr uint32_t OFF_TMEMPTR = OFF_BAR + NBAR * 8;
    static constexpr uint32_t OFF_ABORT = OFF_TMEMPTR + 4;
    static constexpr uint32_t OFF_X = (OFF_ABORT + 4 + 15) & ~15u;   // [2][M] (maximum, sum) per stream and row
    static constexpr uint32_t OFF_RANGE = OFF_X + 2 * M * 8;         // WorkRange
    static constexpr uint32_t OFF_SEQ = OFF_RANGE + ((sizeof(WorkRange) + 15) & ~15u);   // order of the sequences
    static constexpr uint32_t SMEM_BYTES = OFF_SEQ + kSplitMaxB;
    // TMEM columns: S_A | S_B (128 each; P is written over S) | O_A | O_B (D each)
    static constexpr uint32_t T_S = 0, T_O = 256, TMEM_COLS = 512;
    // floats between the rows of a partial state in shared memory: lanes hold
    // neighbouring rows, so their 16-byte stores spread over the banks
    static constexpr int C_PITCH = D + 4;
    static_assert(M * C_PITCH * 4 <= RS * TILE_BYTES, "a partial state fits over the ring");

    static_assert(SMEM_BYTES <= 232448, "shared memory budget");
    static_assert((OFF_R | Q_BYTES | TILE_BYTES) % 1024 == 0, "1024-byte aligned operand tiles");
};

// One job of a CTA: tiles [j0, j1) of a block of 128 queries (qb), or of the
// two blocks qb and qb + 1 (pair).
struct RowsJob {
    UnitInfo ui;   // n_tiles: the job's tiles, the tree tiles past its last query left out
    int j0, j1;
    bool pair;
};

// Does this CTA take pair jobs (all its jobs are of one kind)?
template <bool RANGE>
PPD_DEV bool rows_pair_cta(const AttnParams &p)
{
    return !RANGE && p.pairs && (p.n_qb != 3 || (int)blockIdx.x < p.pair_grid);
}

// Walks a CTA's jobs in order (every role walks the same sequence).  Whole
// jobs round-robin: single jobs (n_qb 1), pair jobs (n_qb 2, or 4 with two a
// slice); with n_qb 3 the first p.pair_grid CTAs take the slices' pairs and
// the others their third blocks.  RANGE (either split): single jobs, the CTA's range
// of tiles.
template <bool RANGE, bool RAGGED = false>
struct RowsIter {
    SegIter<RANGE, RAGGED> seg;
    int x, step, n, per;
    bool pair;
    PPD_DEV RowsIter(const AttnParams &p, const WorkRange &w) : seg(w)
    {
        const int c = (int)blockIdx.x, G = (int)gridDim.x;
        pair = rows_pair_cta<RANGE>(p);
        x = c;
        step = G;
        per = p.n_qb;   // jobs a slice
        if (p.pairs) {
            per = p.n_qb == 4 ? 2 : 1;
            if (p.n_qb == 3) {
                x = pair ? c : c - p.pair_grid;
                step = pair ? p.pair_grid : G - p.pair_grid;
            }
        }
        n = p.n_units / p.n_qb * per;
    }
    PPD_DEV bool next(const AttnParams &p, RowsJob &j)
    {
        if (RANGE) {
            Seg s;
            if (!seg.next(p, s)) return false;
            j.ui = s.ui;
            j.j0 = s.j0;
            j.j1 = s.j1;
            j.pair = false;
            return true;
        }
        int job = x;
        if (RAGGED && seg.seq) job = ragged_job(p, seg.seq, x, step, n, per);
        if (job < 0 || job >= n) return false;
        x += step;
        const int slice = job / per, i = job - slice * per;
        const int qb = pair ? 2 * i : (p.pairs ? p.n_qb - 1 : i);
        j.ui = unit_info(p, slice * p.n_qb + qb);
        // a query's ancestors come before it: no tree tile past the job's last block
        j.ui.n_tiles = j.ui.n_pref + qb + (pair ? 2 : 1);
        j.j0 = 0;
        j.j1 = j.ui.n_tiles;
        j.pair = pair;
        return true;
    }
};

// prefetch_first_tiles for whole jobs: the first `n` prefix tiles of this CTA's first
// job in round-robin order.
template <bool RANGE>
PPD_DEV void rows_prefetch(const AttnParams &p, int lane, const CUtensorMap *kc, const CUtensorMap *vc,
                           int dch, int n)
{
    if (RANGE) {
        prefetch_first_tiles<RANGE>(p, lane, kc, vc, dch, n);
        return;
    }
    const WorkRange none{};
    const RowsIter<RANGE> it(p, none);
    if (lane != 0 || it.x >= it.n) return;
    const int lbh = it.x / it.per;
    const int P = min(max(ld_relaxed_gpu_s32(p.prefix_len + (lbh / p.H) % p.B), 0), p.S_max);
    for (int j = 0; j < min(n, (P + 127) >> 7); ++j) {
        for (int c = 0; c < dch; ++c) {
            tma_prefetch_l2_3d(kc, c * 64, j * 128, lbh);
            tma_prefetch_l2_3d(vc, c * 64, j * 128, lbh);
        }
    }
}

// MODE: whole jobs round-robin (0), the work split (1), the cluster split (2),
// whole jobs with the longest sequences first (3).
template <int D, int MODE>
__global__ void __launch_bounds__(384, 1)
tree_attention_rows_kernel(const __grid_constant__ CUtensorMap map_q,
                           const __grid_constant__ CUtensorMap map_kc,
                           const __grid_constant__ CUtensorMap map_vc,
                           const __grid_constant__ CUtensorMap map_kt,
                           const __grid_constant__ CUtensorMap map_vt, const AttnParams p)
{
    using Lay = RowsLayout<D>;
    using Pos = RingPos<Lay::RS>;
    constexpr bool SPLIT = MODE == 1, RANGE = MODE == 1 || MODE == 2, RAGGED = MODE == 3;
    extern __shared__ __align__(1024) uint8_t smem[];
    if (smem_addr(smem) & 1023u) {
        if (threadIdx.x == 0 && p.dev_status)
            for (int b = 0; b < p.B; ++b) p.dev_status[b] = kErrUnsupported;
        return;
    }

    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + Lay::OFF_BAR);
    uint32_t *tmem_ptr = reinterpret_cast<uint32_t *>(smem + Lay::OFF_TMEMPTR);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + Lay::OFF_ABORT);
    float2 *xs = reinterpret_cast<float2 *>(smem + Lay::OFF_X);
    float2 *cs = reinterpret_cast<float2 *>(smem);   // cluster split: [M] over the Q slots, free by then

    const int warp = warp_uniform((int)threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int T = p.T;

    const bool pair_cta = rows_pair_cta<RANGE>(p);
    if (threadIdx.x == 0) {
        for (int i = 0; i < Lay::NBAR; ++i) {
            uint32_t count = 1;
            if (i >= Lay::B_PFULL && i < Lay::B_PFULL + 4) count = 4;
            // both issuers pass every ring position, and both read a single job's Q block
            if (i >= Lay::B_EMPTY && i < Lay::B_EMPTY + Lay::RS) count = 2;
            if (!pair_cta && i >= Lay::B_QEMPTY && i < Lay::B_QEMPTY + Lay::QS) count = 2;
            if (i == Lay::B_DRAIN) count = 2;
            if (i >= Lay::B_OFREE && i < Lay::B_OFREE + 2) count = 8;
            mbar_init(bars + i, count);
        }
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 9) {
        tmem_alloc(tmem_ptr, Lay::TMEM_COLS);
        tmem_relinquish();
    }
    if (warp == 8 && lane == 0) {
        // the tensor maps are kernel parameters: fetch them before any wait
        tma_prefetch_map(&map_q);
        tma_prefetch_map(&map_kc);
        tma_prefetch_map(&map_vc);
        tma_prefetch_map(&map_kt);
        tma_prefetch_map(&map_vt);
    }
    // in a chain of programmatic launches the inputs may come from the preceding
    // grid: everything above overlapped it, nothing below reads before it is done
    // (the first K/V tiles are only asked of L2 before)
    if (p.pdl_wait) {
        if (warp == 8) rows_prefetch<RANGE>(p, lane, &map_kc, &map_vc, Lay::DCH, 3);
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    WorkRange *wr_s = reinterpret_cast<WorkRange *>(smem + Lay::OFF_RANGE);
    if (warp == 8) {
        const WorkRange w = plan_range(p, lane, RAGGED ? smem + Lay::OFF_SEQ : nullptr);   // whole units round-robin without p.split
        if (lane == 0) {
            *wr_s = w;
            if (SPLIT) p.split_rec[blockIdx.x].u = -1;   // no cut unit recorded yet
        }
    }
    // the merge of cut units, or the next call of a chain (a dependent launch),
    // may be scheduled now; it waits for this grid to complete
    if (SPLIT || p.pdl_wait) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_ptr;
    const WorkRange &wr = *wr_s;

    if (warp == 11) {
        // ------------------------------------------------------------ fused-step side work
        if (p.fused) fused_side_warp<false>(p, wr, lane, abort_flag);
        else if (p.set_status) status_warp(p, lane);
        if (p.late_wait) pdl_wait();
    } else if (warp == 8) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            // slices of three or four blocks stay in L2 for their later readers; two single
            // blocks of a slice are read side by side (with the normal policy too: 32 slices
            // of 2048 keys, 200 tokens, 18.8 us a call either way, 40 of 4096 38.9 -> 39.6)
            const uint64_t pol = p.n_qb > 2 ? l2_policy_evict_normal() : l2_policy_evict_first();
            Pos pos;
            int n_tiles = 0, n_q0 = 0, n_q1 = 0;   // copies issued: ring tiles, Q blocks per slot
            auto load = [&](const CUtensorMap *map, int row, int lbh) {
                // a fresh barrier counts as past its odd phase: the first round never waits
                mbar_wait(bars + Lay::B_EMPTY + pos.slot, pos.phase ^ 1u, abort_flag);
                if (!*abort_flag) {
                    uint64_t *full = bars + Lay::B_FULL + pos.slot;
                    mbar_arrive_expect_tx(full, Lay::TILE_BYTES);
#pragma unroll
                    for (int c = 0; c < Lay::DCH; ++c)
                        tma_load_3d(smem + Lay::OFF_R + pos.slot * Lay::TILE_BYTES + c * Lay::GROUP_BYTES, map,
                                    full, c * 64, row, lbh, pol);
                    ++n_tiles;
                }
                pos.advance();
            };
            auto load_q = [&](int qs, uint32_t parity, int qb, int lbh) {
                mbar_wait(bars + Lay::B_QEMPTY + qs, parity ^ 1u, abort_flag);
                if (!*abort_flag) {
                    // rows T..127 of the box lie beyond the tensor and arrive as zeros
                    mbar_arrive_expect_tx(bars + Lay::B_QFULL + qs, Lay::Q_BYTES);
#pragma unroll
                    for (int c = 0; c < Lay::DCH; ++c)
                        tma_load_3d(smem + Lay::OFF_Q + qs * Lay::Q_BYTES + c * Lay::GROUP_BYTES, &map_q,
                                    bars + Lay::B_QFULL + qs, c * 64, qb * Lay::M, lbh, pol);
                    n_q0 += qs == 0;
                    n_q1 += qs == 1;
                }
            };
            // V tiles of a single job trail their K tiles by two: their coordinates
            int v_row[2] = {0, 0}, v_lbh[2] = {0, 0};
            bool v_tree[2] = {false, false};
            int g = 0, k = 0;
            RowsIter<RANGE, RAGGED> it(p, wr);
            for (RowsJob jb; it.next(p, jb); ++k) {
                const UnitInfo &ui = jb.ui;
                if (!jb.pair) load_q(k & 1, (uint32_t)(k >> 1) & 1u, ui.qb, ui.lbh);
                for (int j = jb.j0; j < jb.j1; ++j, ++g) {
                    const bool tree = (j >= ui.n_pref);
                    const int row = (tree ? j - ui.n_pref : j) * Lay::KT;
                    if (jb.pair) {
                        load(tree ? &map_kt : &map_kc, row, ui.lbh);
                        load(tree ? &map_vt : &map_vc, row, ui.lbh);
                        // the Q slots are free once the job before has its last scores:
                        // its first tiles are queued ahead of that wait
                        if (j == jb.j0) {
                            load_q(0, (uint32_t)k & 1u, ui.qb, ui.lbh);
                            load_q(1, (uint32_t)k & 1u, ui.qb + 1, ui.lbh);
                        }
                        continue;
                    }
                    if (g & 1) {
                        if (g >= 2) load(v_tree[1] ? &map_vt : &map_vc, v_row[1], v_lbh[1]);
                        v_row[1] = row;
                        v_lbh[1] = ui.lbh;
                        v_tree[1] = tree;
                    } else {
                        if (g >= 2) load(v_tree[0] ? &map_vt : &map_vc, v_row[0], v_lbh[0]);
                        v_row[0] = row;
                        v_lbh[0] = ui.lbh;
                        v_tree[0] = tree;
                    }
                    load(tree ? &map_kt : &map_kc, row, ui.lbh);
                }
            }
            if (!it.pair) {
                for (int e = max(0, g - 2); e < g; ++e)
                    load((e & 1 ? v_tree[1] : v_tree[0]) ? &map_vt : &map_vc, e & 1 ? v_row[1] : v_row[0],
                         e & 1 ? v_lbh[1] : v_lbh[0]);
            }
            if (*abort_flag) {
                // let every copy already issued land before the CTA can exit
                for (int i = max(0, n_tiles - Lay::RS); i < n_tiles; ++i)
                    mbar_wait_drain(bars + Lay::B_FULL + i % Lay::RS, (i / Lay::RS) & 1);
                if (n_q0 > 0) mbar_wait_drain(bars + Lay::B_QFULL + 0, (n_q0 - 1) & 1);
                if (n_q1 > 0) mbar_wait_drain(bars + Lay::B_QFULL + 1, (n_q1 - 1) & 1);
            }
        }
    } else if (warp == 9 || warp == 10) {
        // ------------------------------------------------------------ MMA issuers
        // one warp per stream: the whole warp walks the tiles and waits, one elected lane
        // issues.  (One warp for both left the tensor pipe idle at every wait: its queue
        // holds two to three products.)  Both warps pass every position of the ring in
        // order, also those of the other stream's tiles, and a slot is refilled when both
        // have: a wait on a barrier's parity is then never more than one phase behind.
        const uint32_t s = (uint32_t)warp - 9u;
        const uint32_t idesc_qk = make_idesc_bf16(128, 128, 0, 0);
        const uint32_t idesc_pv = make_idesc_bf16(128, D, 0, 1);
        const uint32_t t_s = warp_uniform(tmem_base) + Lay::T_S + s * 128u, t_o = warp_uniform(tmem_base) + Lay::T_O + s * D;
        const uint64_t dq0 = make_smem_desc(warp_uniform(smem_addr(smem + Lay::OFF_Q)), 16, 1024);
        const uint64_t dk0 = make_smem_desc(warp_uniform(smem_addr(smem + Lay::OFF_R)), 16, 1024);
        const uint64_t dv0 = make_smem_desc(warp_uniform(smem_addr(smem + Lay::OFF_R)), Lay::GROUP_BYTES, 1024);

        Pos pos;                                  // next ring position
        bool pend = false;                        // a tile's PV product is still to be issued
        bool p_first = false, p_last = false;     // the tile's place among the stream's of its job
        int p_job = -1;                           // its job, counting those with tiles of the stream
        uint32_t p_par = 0;
        bool dead = false;                        // the CTA gave up: keep the control flow, issue nothing

        // The streams take turns, a tile's PV and the next scores at a time: A, B, A, ...
        // (Free-running they fall into step and their softmaxes coincide.)  A warp waits
        // for everything else first.
        uint32_t turn = 0;
        auto take_turn = [&]() {
            if (s == 1 || turn > 0) mbar_wait(bars + Lay::B_TURN + s, (turn - 1u + s) & 1u, abort_flag);
            ++turn;
        };

        // A position that only the other stream's products read.
        auto pass = [&]() {
            mbar_wait(bars + Lay::B_FULL + pos.slot, pos.phase, abort_flag);
            if (elect_one()) mbar_arrive(bars + Lay::B_EMPTY + pos.slot);
            __syncwarp();
            pos.advance();
        };

        // O += P_hi V + P_lo V for the pending tile, as its halves of 64 keys arrive.  Per
        // 32 keys the probability columns hold 8 columns of hi pairs for keys 0..15, 8 for
        // keys 16..31, then the lo pairs in the same order.  A job's first PV product
        // overwrites O: it waits until the softmax warps have read back the output of the
        // stream's job before (one phase of the barrier for each job with tiles of the
        // stream, so the wait is never more than one phase behind).
        auto issue_pv = [&](bool flush) {
            mbar_wait(bars + Lay::B_FULL + pos.slot, pos.phase, abort_flag);
            if (p_first && p_job >= 1) mbar_wait(bars + Lay::B_OFREE + s, (uint32_t)(p_job - 1) & 1u, abort_flag);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                mbar_wait(bars + Lay::B_PFULL + 2 * s + half, p_par, abort_flag);
                if (half == 0 && !flush) take_turn();
                tc_fence_after();
                if (elect_one()) {
                    if (!dead) {
                        const uint64_t b0 = desc_advance(dv0, pos.slot * Lay::TILE_BYTES);
#pragma unroll
                        for (int kk = 4 * half; kk < 4 * half + 4; ++kk) {
                            const uint64_t b = desc_advance(b0, kk * 2048);
                            const uint32_t a_hi = t_s + 32u * (kk >> 1) + 8u * (kk & 1);
                            umma_bf16_ta(t_o, a_hi, b, idesc_pv, (p_first && kk == 0) ? 0u : 1u);
                            umma_bf16_ta(t_o, a_hi + 16u, b, idesc_pv, 1u);
                        }
                    }
                    if (half == 1) {
                        umma_commit(bars + Lay::B_EMPTY + pos.slot);
                        if (p_last) umma_commit(bars + Lay::B_DONE + s);
                    }
                }
                __syncwarp();
            }
            pos.advance();
            p_par ^= 1u;
            pend = false;
        };

        // S = Q K^T of one tile, after the stream's pending PV product (which reads the
        // probabilities that the new scores replace: one thread's products execute in the
        // order they are issued).  first, last: the tile among the stream's of the job.
        auto issue_s = [&](int qs, bool first, bool last) {
            mbar_wait(bars + Lay::B_FULL + pos.slot, pos.phase, abort_flag);
            tc_fence_after();
            if (elect_one()) {
                if (!dead) {
                    const uint64_t a0 = desc_advance(dq0, qs * Lay::Q_BYTES);
                    const uint64_t b0 = desc_advance(dk0, pos.slot * Lay::TILE_BYTES);
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint32_t off = (kk >> 2) * Lay::GROUP_BYTES + (kk & 3) * 32;
                        umma_bf16(t_s, desc_advance(a0, off), desc_advance(b0, off), idesc_qk, kk > 0 ? 1u : 0u);
                    }
                }
                mbar_arrive(bars + Lay::B_TURN + (s ^ 1u));   // the turn is over
                umma_commit(bars + Lay::B_SFULL + s);
                umma_commit(bars + Lay::B_EMPTY + pos.slot);
                if (last) umma_commit(bars + Lay::B_QEMPTY + qs);
            }
            __syncwarp();
            pos.advance();
            pend = true;
            p_first = first;
            p_last = last;
            if (first) ++p_job;
        };

        RowsIter<RANGE, RAGGED> it(p, wr);
        const bool pair = it.pair;
        int g = 0, k = 0;   // tiles and jobs of the CTA so far
        for (RowsJob jb;; ++k) {
            const int n = warp_uniform(it.next(p, jb) ? jb.j1 - jb.j0 : 0);
            if (n == 0) break;
            if (pair) {
                // K0 V0 K1 V1 ...; the job's last tile holds no key that a query of its first
                // block may see (n >= 2), so stream A stops one tile earlier
                for (int i = 0; i < n; ++i) {
                    if (pend) issue_pv(false);
                    else take_turn();
                    if (s == 0 && i == n - 1) {
                        if (elect_one()) mbar_arrive(bars + Lay::B_TURN + 1);
                        __syncwarp();
                        pass();
                        pass();
                        continue;
                    }
                    if (i == 0) {
                        mbar_wait(bars + Lay::B_QFULL + s, (uint32_t)k & 1u, abort_flag);
                        dead = warp_uniform(*abort_flag) != 0;
                    }
                    issue_s((int)s, i == 0, i == (s == 0 ? n - 2 : n - 1));
                }
            } else {
                // K0 K1 V0 K2 V1 ...: tile e of all jobs is preceded by the V of tile e - 2
                const int qs = k & 1, i0 = (g ^ (int)s) & 1;
                auto q_wait = [&]() {
                    mbar_wait(bars + Lay::B_QFULL + qs, (uint32_t)(k >> 1) & 1u, abort_flag);
                    dead = warp_uniform(*abort_flag) != 0;
                };
                for (int i = 0; i < n; ++i) {
                    if (((i ^ i0) & 1) == 0) {
                        if (pend) issue_pv(false);
                        else take_turn();
                        if (i == i0) q_wait();
                        issue_s(qs, i == i0, i + 2 >= n);
                    } else {
                        if (g + i >= 2) pass();
                        pass();
                    }
                }
                if (i0 >= n) {   // none of the job's tiles is this stream's
                    q_wait();
                    if (elect_one()) mbar_arrive(bars + Lay::B_QEMPTY + qs);
                    __syncwarp();
                }
                g += n;
            }
        }
        if (pair) {
            if (pend) issue_pv(true);
        } else {
            for (int e = max(0, g - 2); e < g; ++e) {
                if ((e & 1) == (int)s) issue_pv(true);
                else pass();
            }
        }
        if (elect_one()) umma_commit(bars + Lay::B_DRAIN);
        __syncwarp();
        mbar_wait_drain(bars + Lay::B_DRAIN, 0);
    } else {
        // ------------------------------------------------------------ softmax warps
        const int s = warp >> 2;                 // stream
        const int q = (warp & 3) * 32 + lane;    // query row of the block, and TMEM lane
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_s = tmem_base + lane_off + Lay::T_S + s * 128u;
        const uint32_t t_os = tmem_base + lane_off + Lay::T_O + s * D;
        const float sl2 = p.scale_log2;
        const uint64_t sl2x2 = pack2(sl2, sl2);
        const bool vec_out = (reinterpret_cast<uintptr_t>(p.out) & 15u) == 0;
        const bool out32 = (reinterpret_cast<uintptr_t>(p.out) & 31u) == 0;
        constexpr int NW = kMaxTree / 32;

        float m = -INFINITY;    // running maximum of the row (log2 units)
        float l = 0.f;          // its row sum
        // bit i of anc[w]: tree node 32w + i is an ancestor of (or is) this thread's query
        // (indexed at run time, so it stays out of the registers)
        uint32_t anc[NW] = {};
        int cur_key = -1;
        int g = 0;              // tiles of the CTA's jobs so far
        uint32_t s_par = 0, d_par = 0;   // phase parities: scores; bit x: stream x's jobs done

        // Probabilities of 32 keys from their raw scores r against the maximum, split
        // into bf16 hi + lo and stored over the scores.
        auto emit = [&](auto bits_c, const uint32_t (&r)[32], uint32_t bits, uint64_t negm, uint32_t t_dst,
                        uint64_t (&sum)[2]) {
            constexpr bool BITS = decltype(bits_c)::value != 0;
            uint32_t w[32];
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
                const uint64_t d = fma2(pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), sl2x2, negm);
                float d0, d1;
                unpack2(d, d0, d1);
                if (BITS) {
                    d0 = ((bits >> e) & 1u) ? d0 : -INFINITY;
                    d1 = ((bits >> (e + 1)) & 1u) ? d1 : -INFINITY;
                }
                const float p0 = ex2(d0), p1 = ex2(d1);
                const uint64_t pp = pack2(p0, p1);
                sum[(e >> 1) & 1] = add2(sum[(e >> 1) & 1], pp);
                split_bf16x2(pp, p0, p1, w[e >> 1], w[16 + (e >> 1)]);
            }
            tmem_st32(t_dst, w);
        };

        // Largest of 32 raw scores (the visible ones) and mx.
        auto chunk_max = [&](auto bits_c, const uint32_t (&r)[32], uint32_t bits, float mx) {
            constexpr bool BITS = decltype(bits_c)::value != 0;
            float a = mx, b = -INFINITY;
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
                float v[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    v[x] = __uint_as_float(r[e + x]);
                    if (BITS) v[x] = ((bits >> (e + x)) & 1u) ? v[x] : -INFINITY;
                }
                a = max3(a, v[0], v[1]);
                b = max3(b, v[2], v[3]);
            }
            return fmaxf(a, b);
        };

        // Half of a tile's probabilities (and any rescaled O) are in TMEM.
        auto p_ready = [&](int half) {
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bars + Lay::B_PFULL + 2 * s + half);
        };

        // One tile of the stream: scores in TMEM to probabilities in TMEM.
        auto softmax_tile = [&](auto bits_c, const uint32_t (&bits)[4], bool first) {
            constexpr bool BITS = decltype(bits_c)::value != 0;
            uint32_t r[4][32];
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(t_s + 32 * c, r[c]);
            float mx = -INFINITY;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                tmem_wait_ld(r[c]);
                mx = chunk_max(bits_c, r[c], bits[c], mx);
            }
            mx *= sl2;   // sl2 > 0
            const bool up = mx > m + 16.f || (first && mx > m);
            float alpha = 1.f;
            if (up) {
                alpha = ex2(m - mx);   // 0 from -inf
                m = mx;
            }
            if (!first && __any_sync(0xffffffffu, up)) {
                // rescale this row of O: the PV product of the stream's tile before is
                // complete (it was issued before these scores' product)
                tc_fence_after();
#pragma unroll 1
                for (int ch = 0; ch < D / 16; ++ch) {
                    uint32_t o[16];
                    tmem_ld16(t_os + ch * 16, o);
                    tmem_wait_ld(o);
#pragma unroll
                    for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                    tmem_st16(t_os + ch * 16, o);
                }
                l *= alpha;
            }
            const uint64_t negm = pack2(-m, -m);
            uint64_t sum[2] = {0ull, 0ull};
            // the scores are read again, half a tile at a time in one rolled loop: unrolled
            // over the tile, the code of eight warps at different places did not fit the
            // instruction caches
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                const uint32_t t_h = t_s + 64u * (uint32_t)half;
                uint32_t ra[32], rb[32];
                tmem_ld32(t_h, ra);
                tmem_ld32(t_h + 32, rb);
                const uint32_t b0 = BITS && half ? bits[2] : bits[0], b1 = BITS && half ? bits[3] : bits[1];
                tmem_wait_ld(ra);
                tmem_wait_ld(rb);
                emit(bits_c, ra, b0, negm, t_h, sum);
                emit(bits_c, rb, b1, negm, t_h + 32, sum);
                p_ready(half);
            }
            float l0, l1;
            unpack2(add2(sum[0], sum[1]), l0, l1);
            l += l0 + l1;
        };

        // 32 output values of row `orow` at `scale`.
        auto store32 = [&](float *dst, const uint32_t (&r)[32], float scale) {
            if (out32) {
#pragma unroll
                for (int e = 0; e < 32; e += 8) st_global_v8(dst + e, r + e, scale);
            } else if (vec_out) {
#pragma unroll
                for (int e = 0; e < 32; e += 4)
                    *reinterpret_cast<float4 *>(dst + e) =
                        make_float4(__uint_as_float(r[e]) * scale, __uint_as_float(r[e + 1]) * scale,
                                    __uint_as_float(r[e + 2]) * scale, __uint_as_float(r[e + 3]) * scale);
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) dst[e] = __uint_as_float(r[e]) * scale;
            }
        };

        auto wait_done = [&](int st) {
            mbar_wait(bars + Lay::B_DONE + st, (d_par >> st) & 1u, abort_flag);
            d_par ^= 1u << st;
        };
        auto o_free = [&](int st, uint32_t n) {   // this warp has read stream st's output (n arrivals)
            if (lane == 0) mbar_arrive_n(bars + Lay::B_OFREE + st, n);
        };

        // End of a pair job: this stream's block of 128 rows.
        auto finish_pair = [&](const RowsJob &jb) {
            const int qg = (jb.ui.qb + s) * Lay::M + q;
            if (qg < T && p.lse) p.lse[(size_t)jb.ui.lbh * T + qg] = (m + lg2(l)) * 0.69314718055994530942f;
            const float linv = rcp(l);
            float *orow = p.out + ((size_t)jb.ui.lbh * T + qg) * D;
            wait_done(s);
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < D; c += 64) {
                uint32_t r0[32], r1[32];
                tmem_ld32(t_os + c, r0);
                tmem_ld32(t_os + c + 32, r1);
                tmem_wait_ld(r0);
                tmem_wait_ld(r1);
                if (c + 64 == D) {
                    tc_fence_before();
                    __syncwarp();
                    o_free(s, 2);
                }
                if (qg < T) {
                    store32(orow + c, r0, linv);
                    store32(orow + c + 32, r1, linv);
                }
            }
        };

        // End of a single job: the row's two partial states (one per stream) merged;
        // this thread writes half of the row, stream A's the first D / 2 columns.  `st0`:
        // the stream of the job's first tile, `both`: the other one had tiles too.
        auto finish_single = [&](const RowsJob &jb, int st0, bool both, int slot) {
            named_bar_sync(1, 256);   // the job before is done with the exchange
            xs[s * Lay::M + q] = make_float2(m, l);
            named_bar_sync(1, 256);
            const float2 xo = xs[(s ^ 1) * Lay::M + q];
            const float mt = fmaxf(m, xo.x);
            // a stream without tiles, or whose tiles hide every key from this row, has
            // weight 0; its accumulator may hold anything then
            const float w_own = m == -INFINITY ? 0.f : ex2(m - mt);
            const float w_oth = xo.x == -INFINITY ? 0.f : ex2(xo.x - mt);
            const float lt = w_own * l + w_oth * xo.y;
            const int qg = jb.ui.qb * Lay::M + q;
            const bool whole = !RANGE || (SPLIT && jb.j0 == 0 && jb.j1 == jb.ui.n_tiles);
            const float inv = whole ? rcp(lt) : 1.f;
            float *dst;
            if (whole) {
                if (s == 0 && qg < T && p.lse)
                    p.lse[(size_t)jb.ui.lbh * T + qg] = (mt + lg2(lt)) * 0.69314718055994530942f;
                dst = p.out + ((size_t)jb.ui.lbh * T + qg) * D;
            } else if (MODE == 2) {
                // this CTA's part for the cluster: rows over the ring (every copy has landed,
                // and the waits below cover every product that reads it)
                if (s == 0) cs[q] = make_float2(mt, lt);
                dst = reinterpret_cast<float *>(smem + Lay::OFF_R) + q * Lay::C_PITCH;
            } else {
                // a part of a cut unit: the unnormalised row, its maximum and its sum
                float *base = p.split_part + (size_t)slot * split_slot_floats(D);
                if (s == 0 && qg < T) {
                    base[(size_t)kSplitRows * D + q] = mt;
                    base[(size_t)kSplitRows * D + kSplitRows + q] = lt;
                }
                dst = base + (size_t)q * D;
            }
            dst += s * (D / 2);
            const bool live = qg < T;
            const float fa = (s == 0 ? w_own : w_oth) * inv, fb = (s == 0 ? w_oth : w_own) * inv;
            const bool has_a = both || st0 == 0, has_b = both || st0 == 1;
            if (has_a) wait_done(0);
            if (has_b) wait_done(1);
            tc_fence_after();
            const uint32_t t_o = tmem_base + lane_off + Lay::T_O + (uint32_t)s * (D / 2);
#pragma unroll
            for (int c = 0; c < D / 2; c += 32) {
                uint32_t r0[32] = {}, r1[32] = {};
                if (has_a) tmem_ld32(t_o + c, r0);
                if (has_b) tmem_ld32(t_o + D + c, r1);
                tmem_wait_ld(r0);
                tmem_wait_ld(r1);
                if (c + 32 == D / 2) {
                    tc_fence_before();
                    __syncwarp();
                    if (has_a) o_free(0, 1);
                    if (has_b) o_free(1, 1);
                }
                if (live) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        const float a = fa != 0.f ? __uint_as_float(r0[e]) * fa : 0.f;
                        r0[e] = __float_as_uint(fb != 0.f ? fmaf(__uint_as_float(r1[e]), fb, a) : a);
                    }
                    if (MODE == 2) {
#pragma unroll
                        for (int e = 0; e < 32; e += 4)
                            st_shared_v4(smem_addr(dst + c + e), r0[e], r0[e + 1], r0[e + 2], r0[e + 3]);
                    } else {
                        store32(dst + c, r0, 1.f);
                    }
                }
            }
        };

        RowsIter<RANGE, RAGGED> it(p, wr);
        int k = 0;
        for (RowsJob jb; it.next(p, jb); ++k) {
            const UnitInfo &ui = jb.ui;
            const int qb = ui.qb + (jb.pair ? s : 0);
            const int qg = qb * Lay::M + q;   // this thread's tree token
            if (ui.b * p.n_qb + qb != cur_key) {
#pragma unroll
                for (int w = 0; w < NW; ++w) anc[w] = 0;
                if (qg < T) {
                    int a = qg;
                    while (true) {
                        anc[a >> 5] |= 1u << (a & 31);
                        const int pa = ld_input(p.parent + (size_t)ui.b * T + a);
                        if (pa < 0 || pa >= a) break;   // the root, or a malformed tree
                        a = pa;
                    }
                }
                cur_key = ui.b * p.n_qb + qb;
            }

            const int n = jb.j1 - jb.j0;
            const int st0 = g & 1;   // single job: the stream of its first tile
            // this stream's tiles of the job: all of a pair's, every other one of a single's
            // (stream A's queries see nothing of a pair's last tree tile)
            const int n_s = jb.pair && s == 0 ? n - 1 : n;
            for (int i = jb.pair ? 0 : (s ^ st0); i < n_s; i += jb.pair ? 1 : 2) {
                const int j = jb.j0 + i;
                const bool tree = (j >= ui.n_pref);
                const int n_valid = tree ? T : min(Lay::KT, ui.P - j * Lay::KT);
                const bool first = i < (jb.pair ? 1 : 2);
                mbar_wait(bars + Lay::B_SFULL + s, s_par, abort_flag);
                s_par ^= 1u;
                tc_fence_after();
                if (!tree && n_valid == Lay::KT) {
                    const uint32_t all[4] = {~0u, ~0u, ~0u, ~0u};
                    softmax_tile(kind_t<0>{}, all, first);
                } else {
                    uint32_t bits[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int left = n_valid - 32 * c;
                        bits[c] = left >= 32 ? ~0u : (left > 0 ? (1u << left) - 1u : 0u);
                        if (tree) bits[c] = anc[4 * (j - ui.n_pref) + c];
                    }
                    // V rows of invisible keys in a partial prefix tile may be NaN: zero them
                    // (each stream of a pair before its own product)
                    if (!tree) {
                        const int e = g + i;
                        int pos;   // the V tile's place in the ring order
                        if (jb.pair) pos = 2 * e + 1;
                        else pos = (RANGE && e == wr.n_tiles - 1) ? 2 * e + 1 : 2 * e + 2;
                        const int vs = pos % Lay::RS;
                        mbar_wait(bars + Lay::B_FULL + vs, (uint32_t)(pos / Lay::RS) & 1u, abort_flag);
                        if (q >= n_valid) {
                            const uint32_t vrow = smem_addr(smem + Lay::OFF_R + vs * Lay::TILE_BYTES) + q * 128u;
#pragma unroll
                            for (int c = 0; c < Lay::DCH; ++c)
#pragma unroll
                                for (int x = 0; x < 8; ++x)
                                    st_shared_v4(vrow + c * Lay::GROUP_BYTES + x * 16, 0u, 0u, 0u, 0u);
                        }
                        fence_proxy_async_smem();
                    }
                    softmax_tile(kind_t<1>{}, bits, first);
                }
            }
            g += n;

            if (jb.pair) {
                finish_pair(jb);
            } else {
                int slot = 0;
                if (SPLIT && !(jb.j0 == 0 && jb.j1 == ui.n_tiles)) {
                    // a part: slot 2c for the range's first segment, 2c + 1 for its last
                    const int u = ui.lbh * p.n_qb + ui.qb;
                    slot = 2 * (int)blockIdx.x + (u == wr.u_first ? 0 : 1);
                    // the part holding the unit's first tile records it for the merge
                    if (jb.j0 == 0 && threadIdx.x == 0)
                        p.split_rec[blockIdx.x] =
                            SplitRecord{wr.x_first + (wr.n_tiles - it.seg.left) - jb.j1, wr.n_shared, u, ui.n_tiles};
                }
                finish_single(jb, st0, n >= 2, slot);
            }
            m = -INFINITY;
            l = 0.f;
        }
    }

    if (MODE == 2) {
        cluster_sync();
        bool unused = false;
        if (warp < 8) {
            const int u = (int)blockIdx.x / p.cluster;
            const int lbh = u / p.n_qb, qb = u - lbh * p.n_qb;
            unused = cluster_merge<2>(p, wr.parts, smem_addr(smem) + Lay::OFF_R, Lay::C_PITCH * 4, smem_addr(cs), D,
                          (int)blockIdx.x - u * p.cluster, min(Lay::M, T - qb * Lay::M),
                          (size_t)lbh * T + (size_t)qb * Lay::M, threadIdx.x, 256);
        }
        __syncwarp();
        cluster_leave(unused);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*abort_flag && threadIdx.x == 0) {
        for (int b = 0; b < p.B; ++b) {
            if (p.dev_status) atomicMax(p.dev_status + b, (int)kErrTimeout);
            if (p.fused) atomicMax(p.fs.status + b, (int)kErrTimeout);
        }
    }
    if (warp == 9) tmem_dealloc(tmem_base, Lay::TMEM_COLS);
}

template <int D>
static cudaError_t launch_rows_t(const AttnMaps &m, const AttnParams &p, int num_sms,
                                 bool programmatic, cudaStream_t stream)
{
    static std::atomic<uint64_t> configured[4] = {{0}, {0}, {0}, {0}};
    if (whole_ragged(p))
        return launch_attention_grid(tree_attention_rows_kernel<D, 3>, RowsLayout<D>::SMEM_BYTES, 384,
                                     configured[3], m, p, num_sms, programmatic, stream);
    if (p.cluster > 1)
        return launch_attention_grid(tree_attention_rows_kernel<D, 2>, RowsLayout<D>::SMEM_BYTES, 384,
                                     configured[2], m, p, num_sms, programmatic, stream);
    if (p.split)
        return launch_attention_grid(tree_attention_rows_kernel<D, 1>, RowsLayout<D>::SMEM_BYTES, 384,
                                     configured[1], m, p, num_sms, programmatic, stream);
    return launch_attention_grid(tree_attention_rows_kernel<D, 0>, RowsLayout<D>::SMEM_BYTES, 384,
                                 configured[0], m, p, num_sms, programmatic, stream);
}

cudaError_t launch_tree_attention_rows(const AttnMaps &m, const AttnParams &p, int D, int num_sms,
                                       bool programmatic, cudaStream_t stream)
{
    if (D == 128) return launch_rows_t<128>(m, p, num_sms, programmatic, stream);
    return launch_rows_t<64>(m, p, num_sms, programmatic, stream);
}

}  // namespace ppd
