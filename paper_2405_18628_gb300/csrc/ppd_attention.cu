// ppd_attention.cu -- tree-masked attention of the PPD verification step on
// sm_103a (paper Section 3 step (1): tree attention over the candidate tree;
// Section 4.1: every tree token attends to the cached prefix, its tree
// ancestors and itself).
//
// One persistent CTA per SM walks a list of (layer, sequence, head) units.  A
// unit streams its KV prefix in tiles of 128 keys and finishes with one tile
// holding the tree's own keys.  Per tile:
//
//   S^T = K_tile * Q^T     tcgen05.mma, M = 128 keys, N = T_pad queries, K = D
//                          (keys on the M side, so a 64-token tree wastes no
//                          tensor-core rows), accumulated in TMEM
//   P   = exp2(S*scale*log2e - m)   by the softmax warpgroups, one key row per
//                          thread, split into bf16 hi + lo parts (P = hi + lo to
//                          2^-18) and written to shared memory
//   O^T += V^T * [P_hi | P_lo]^T    one tcgen05.mma, M = D, N = 2*T_pad, K = 128
//
// This kernel serves trees of up to 64 tokens (padded to TP = 32 or 64 columns);
// larger trees fill the tensor core's M side with queries and run the
// query-row kernel (ppd_attention_rows.cu).  Warp roles: two softmax warpgroups,
// each owning half of the query columns, then the TMA producer, the MMA issuer and
// TMEM owner, and the fused step's argmax / acceptance / compaction.  Four
// warpgroups of a quarter each gain 3 % on long slices of D = 64 with TP = 64 (8 x 16
// slices of 8000 keys: 302 against 292 us) but leave 96 registers a thread, too few
// for the side warp: 30 x 16 slices of 1000 keys, 40 tokens, 439 against 510 us.
//
// Bound: HBM for long slices (32 x 32 slices of 2048 keys: 177.6 us for 1.17 GB,
// 0.97 of the measured copy rate); for short ones the chain of a tile -- scores,
// softmax, hand-over -- and the unit's two ends.  What shortened it, measured
// together on that case, on 24 x 16 slices of 512 keys and on 4 x 80 x 16 slices
// of 350-700 keys (D = 64, T = 32): 184.7 -> 177.6, 36.3 -> 32, 307 -> 195 us:
// products issued from warp-uniform code (ppd_device.cuh, elect_one); two fp32
// operations per instruction; all of a thread's scores in one TMEM load; a
// unit's first tile without the exact maximum; ancestor sets by shuffles,
// without barriers; at D = 64 rings of 4 and 6 tiles instead of 2.
//
// The running row maximum m is lazy.  A unit starts from the scores of its
// first key, which every query sees: no larger than the true maximum.  Each
// tile is done with the current m, and only if a score exceeds m by more than
// 2^16 does it take the exact path -- a cross-lane maximum, a rescale of O and
// of the row sums, and recomputed probabilities.  The
// tree mask is an ancestor bitset built from the parent array; rows beyond
// the prefix (which may hold anything, NaN included) are masked by select
// and their V rows are zeroed in shared memory before the PV product.  O is
// double-buffered in TMEM and a unit's output is read back only after the
// next unit's first tile, so the stream of tiles never waits for a unit's
// last PV product.  Launches with fewer units than SMs share units among CTAs
// (ppd_attention_common.cuh): by clusters, whose CTAs merge their partial states
// through distributed shared memory, or by the work split, merged by a grid of
// its own (split_merge_kernel).
#include "ppd_attention_common.cuh"

#include <cmath>
#include <type_traits>

namespace ppd {

template <int D_, int TP_>
struct AttnLayout {
    static constexpr int D = D_;
    static constexpr int TP = TP_;                // query columns (the tree padded to 32 or 64)
    static constexpr int KT = 128;                // keys per tile
    static constexpr int DCH = D / 64;            // 64-column (128-byte) groups along D
    static constexpr int NWG = 2;                 // softmax warpgroups
    static constexpr int NC = TP / NWG;           // query columns of each
    static constexpr int SW = 4 * NWG;            // softmax warps; then producer, issuer, side warp
    static constexpr int THREADS = (SW + 3) * 32;
    static constexpr uint32_t GROUP_BYTES = KT * 128;   // one column group of a tile
    static constexpr uint32_t TILE_BYTES = KT * D * 2;
    static constexpr uint32_t Q_GROUP_BYTES = TP * 128;
    static constexpr uint32_t Q_BYTES = TP * D * 2;
    static constexpr uint32_t P_BYTES = (2 * TP / 64) * GROUP_BYTES;   // [hi | lo] columns
    static constexpr int OB = 2;                          // O accumulators in TMEM
    static constexpr int QS = 2;                          // Q buffers
    // When a tile's probabilities fit in its own K slot, free once S^T = K Q^T is
    // done, they need no tiles of their own.
    static constexpr bool P_IN_K = P_BYTES <= TILE_BYTES;
    static constexpr int PS = P_IN_K ? 0 : 2;             // dedicated P tiles
    static constexpr int PB = 2;                          // P full/free barrier pairs
    static constexpr int KS = D == 128 ? 3 : (P_IN_K ? 6 : 4);   // K tile ring
    static constexpr int VS = KS;                         // V tile ring

    static constexpr uint32_t OFF_Q = 0;
    static constexpr uint32_t OFF_P = OFF_Q + QS * Q_BYTES;
    static constexpr uint32_t OFF_K = OFF_P + PS * P_BYTES;
    static constexpr uint32_t OFF_V = OFF_K + KS * TILE_BYTES;
    static constexpr uint32_t OFF_BAR = OFF_V + VS * TILE_BYTES;
    // barrier indices
    static constexpr int B_QFULL = 0;
    static constexpr int B_QEMPTY = B_QFULL + QS;
    static constexpr int B_KFULL = B_QEMPTY + QS;
    static constexpr int B_KEMPTY = B_KFULL + KS;
    static constexpr int B_VFULL = B_KEMPTY + KS;
    static constexpr int B_VEMPTY = B_VFULL + VS;
    static constexpr int B_SFULL = B_VEMPTY + VS;
    static constexpr int B_PFULL = B_SFULL + 2;   // also: the tile's scores are read
    static constexpr int B_PFREE = B_PFULL + PB;
    static constexpr int B_DRAIN = B_PFREE + PB;
    static constexpr int NBAR = B_DRAIN + 1;
    static constexpr uint32_t OFF_TMEMPTR = OFF_BAR + NBAR * 8;
    static constexpr uint32_t OFF_ABORT = OFF_TMEMPTR + 4;
    static constexpr uint32_t OFF_NM = (OFF_ABORT + 4 + 15) & ~15u;   // [TP] minus the running maxima
    static constexpr uint32_t OFF_LINV = OFF_NM + TP * 4;         // [OB][TP] 1 / row sums (row sums of a partial)
    static constexpr uint32_t OFF_PMX = OFF_LINV + OB * TP * 4;   // [OB][TP] maxima of a partial
    static constexpr uint32_t OFF_RED = OFF_PMX + OB * TP * 4;    // [NWG][4][NC] reduction scratch
    static constexpr uint32_t OFF_RANGE = (OFF_RED + NWG * 4 * NC * 4 + 15) & ~15u;   // WorkRange
    static constexpr uint32_t OFF_SEQ = OFF_RANGE + ((sizeof(WorkRange) + 15) & ~15u);   // order of the sequences
    static constexpr uint32_t SMEM_BYTES = OFF_SEQ + kSplitMaxB;
    // TMEM columns: S0 | S1 | O0 (hi | lo) | O1 (hi | lo)
    static constexpr uint32_t T_S = 0, T_O = 2 * TP;
    static constexpr uint32_t TMEM_COLS = TP == 64 ? 512 : 256;

    static_assert(SMEM_BYTES <= 232448, "shared memory budget");
    static_assert((OFF_P | OFF_K | OFF_V) % 1024 == 0, "1024-byte aligned operand tiles");
    static_assert((2 + 2 * OB) * TP <= TMEM_COLS, "TMEM budget");
    static_assert(NC == 16 || NC == 32, "query columns of a softmax thread");
};

// MODE: whole units round-robin (0), the work split (1), the cluster split (2),
// whole units with the longest sequences first (3).
template <int D, int TP, int MODE>
__global__ void __launch_bounds__(AttnLayout<D, TP>::THREADS, 1)
tree_attention_kernel(const __grid_constant__ CUtensorMap map_q,
                      const __grid_constant__ CUtensorMap map_kc,
                      const __grid_constant__ CUtensorMap map_vc,
                      const __grid_constant__ CUtensorMap map_kt,
                      const __grid_constant__ CUtensorMap map_vt, const AttnParams p)
{
    using Lay = AttnLayout<D, TP>;
    using KPos = RingPos<Lay::KS>;
    using VPos = RingPos<Lay::VS>;
    constexpr bool SPLIT = MODE == 1, RANGE = MODE == 1 || MODE == 2, RAGGED = MODE == 3;
    constexpr int NC = Lay::NC;
    using Cols = uint32_t[Lay::NC];   // a softmax thread's scores of one tile
    extern __shared__ __align__(1024) uint8_t smem[];
    // The swizzled operand tiles need a 1024-byte aligned base; the check is
    // uniform over the CTA, before any barrier.
    if (smem_addr(smem) & 1023u) {
        if (threadIdx.x == 0 && p.dev_status)
            for (int b = 0; b < p.B; ++b) p.dev_status[b] = kErrUnsupported;
        return;
    }

    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + Lay::OFF_BAR);
    uint32_t *tmem_ptr = reinterpret_cast<uint32_t *>(smem + Lay::OFF_TMEMPTR);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + Lay::OFF_ABORT);

    const int warp = warp_uniform((int)threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int T = p.T;

    if (threadIdx.x == 0) {
        for (int i = 0; i < Lay::NBAR; ++i) {
            uint32_t count = 1;
            if (i >= Lay::B_PFULL && i < Lay::B_PFULL + Lay::PB) count = Lay::SW;
            mbar_init(bars + i, count);
        }
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == Lay::SW + 1) {
        tmem_alloc(tmem_ptr, Lay::TMEM_COLS);
        tmem_relinquish();
    }
    if (warp == Lay::SW && lane == 0) {
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
        if (warp == Lay::SW) prefetch_first_tiles<RANGE>(p, lane, &map_kc, &map_vc, Lay::DCH, 3);
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    WorkRange *wr_s = reinterpret_cast<WorkRange *>(smem + Lay::OFF_RANGE);
    if (warp == Lay::SW) {
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

    if (warp == Lay::SW + 2) {
        // ------------------------------------------------------------ fused-step side work
        if (p.fused) fused_side_warp<true>(p, wr, lane, abort_flag);
        else if (p.set_status) status_warp(p, lane);
        if (p.late_wait) pdl_wait();
    } else if (warp == Lay::SW) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const uint64_t pol = l2_policy_evict_first();
            KPos kp;
            VPos vp;
            int g = 0, k = 0;
            SegIter<RANGE, RAGGED> it(wr);
            for (Seg sg; it.next(p, sg); ++k) {
                const UnitInfo &ui = sg.ui;
                const int u = sg.u;
                const int qs = k & 1;
                // a fresh barrier counts as past its odd phase: the first round never waits
                mbar_wait(bars + Lay::B_QEMPTY + qs, ((k >> 1) & 1) ^ 1, abort_flag);
                if (!*abort_flag) {
                    mbar_arrive_expect_tx(bars + Lay::B_QFULL + qs, Lay::Q_BYTES);
#pragma unroll
                    for (int c = 0; c < Lay::DCH; ++c)
                        tma_load_3d(smem + Lay::OFF_Q + qs * Lay::Q_BYTES + c * Lay::Q_GROUP_BYTES,
                                    &map_q, bars + Lay::B_QFULL + qs, c * 64, 0, u, pol);
                }
                for (int j = sg.j0; j < sg.j1; ++j, ++g) {
                    const bool tree = (j == ui.n_pref);
                    const int row = tree ? 0 : j * Lay::KT;
                    mbar_wait(bars + Lay::B_KEMPTY + kp.slot, kp.phase ^ 1u, abort_flag);
                    if (!*abort_flag) {
                        mbar_arrive_expect_tx(bars + Lay::B_KFULL + kp.slot, Lay::TILE_BYTES);
#pragma unroll
                        for (int c = 0; c < Lay::DCH; ++c)
                            tma_load_3d(smem + Lay::OFF_K + kp.slot * Lay::TILE_BYTES + c * Lay::GROUP_BYTES,
                                        tree ? &map_kt : &map_kc, bars + Lay::B_KFULL + kp.slot, c * 64,
                                        row, u, pol);
                    }
                    kp.advance();
                    mbar_wait(bars + Lay::B_VEMPTY + vp.slot, vp.phase ^ 1u, abort_flag);
                    if (!*abort_flag) {
                        mbar_arrive_expect_tx(bars + Lay::B_VFULL + vp.slot, Lay::TILE_BYTES);
#pragma unroll
                        for (int c = 0; c < Lay::DCH; ++c)
                            tma_load_3d(smem + Lay::OFF_V + vp.slot * Lay::TILE_BYTES + c * Lay::GROUP_BYTES,
                                        tree ? &map_vt : &map_vc, bars + Lay::B_VFULL + vp.slot, c * 64,
                                        row, u, pol);
                    }
                    vp.advance();
                }
            }
            if (*abort_flag) {
                // let every copy already issued land before the CTA can exit
                for (int i = max(0, g - Lay::KS); i < g; ++i)
                    mbar_wait_drain(bars + Lay::B_KFULL + i % Lay::KS, (i / Lay::KS) & 1);
                for (int i = max(0, g - Lay::VS); i < g; ++i)
                    mbar_wait_drain(bars + Lay::B_VFULL + i % Lay::VS, (i / Lay::VS) & 1);
                for (int i = max(0, k - Lay::QS); i < k; ++i)
                    mbar_wait_drain(bars + Lay::B_QFULL + i % Lay::QS, (i / Lay::QS) & 1);
            }
        }
    } else if (warp == Lay::SW + 1) {
        // ------------------------------------------------------------ MMA issuer
        // the whole warp walks the tiles and waits; one elected lane issues
        constexpr uint32_t idesc_qk = make_idesc_bf16(128, TP, 0, 0);
        constexpr uint32_t idesc_pv = make_idesc_bf16(128, 2 * TP, 1, 1);
        const uint32_t tmem = warp_uniform(tmem_base);
        const uint32_t s0 = warp_uniform(smem_addr(smem));
        // V^T as the A operand: M = D spans the tile's 64-column groups.  With
        // D = 64 both M halves read the same group (rows 64..127 of O^T repeat
        // rows 0..63 and are ignored).
        constexpr uint32_t v_lbo = (D == 128) ? Lay::GROUP_BYTES : 0u;
        const uint64_t dq0 = make_smem_desc(s0 + Lay::OFF_Q, 16, 1024);
        const uint64_t dk0 = make_smem_desc(s0 + Lay::OFF_K, 16, 1024);
        const uint64_t dv0 = make_smem_desc(s0 + Lay::OFF_V, v_lbo, 1024);
        const uint64_t dp0 = make_smem_desc(s0 + (Lay::P_IN_K ? Lay::OFF_K : Lay::OFF_P), Lay::GROUP_BYTES, 1024);

        VPos vp;
        KPos pk;            // K slot of the tile whose PV product comes next
        int gp = 0;         // that tile
        auto issue_pv = [&](bool first, uint32_t t_o) {
            const int ps = gp & 1;
            mbar_wait(bars + Lay::B_VFULL + vp.slot, vp.phase, abort_flag);
            mbar_wait(bars + Lay::B_PFULL + ps, (gp >> 1) & 1, abort_flag);
            tc_fence_after();
            const bool dead = warp_uniform(*abort_flag) != 0;
            if (elect_one()) {
                if (!dead) {
                    // descriptors built once; each 16-key step moves 2048 bytes on
                    const uint64_t a0 = desc_advance(dv0, vp.slot * Lay::TILE_BYTES);
                    const uint64_t b0 = desc_advance(dp0, Lay::P_IN_K ? pk.slot * Lay::TILE_BYTES : ps * Lay::P_BYTES);
#pragma unroll
                    for (int kk = 0; kk < Lay::KT / 16; ++kk)
                        umma_bf16(t_o, desc_advance(a0, kk * 2048), desc_advance(b0, kk * 2048), idesc_pv,
                                  (first && kk == 0) ? 0u : 1u);
                }
                umma_commit(bars + Lay::B_PFREE + ps);
                umma_commit(bars + Lay::B_VEMPTY + vp.slot);
                if (Lay::P_IN_K) umma_commit(bars + Lay::B_KEMPTY + pk.slot);
            }
            __syncwarp();
            vp.advance();
            pk.advance();
            ++gp;
        };

        // Tiles are issued as S(g), PV(g-1) across unit boundaries, so the next
        // unit's first scores are under way before this unit's last PV product.
        KPos kp;
        int g = 0, k = 0;
        bool prev_first = false;
        uint32_t prev_to = 0;
        SegIter<RANGE, RAGGED> it(wr);
        for (Seg sg;; ++k) {
            const int n = warp_uniform(it.next(p, sg) ? sg.j1 - sg.j0 : 0);
            if (n == 0) break;
            const int qs = k & 1;
            const uint32_t t_o = tmem + Lay::T_O + (uint32_t)(k & 1) * 2 * TP;
            mbar_wait(bars + Lay::B_QFULL + qs, (k >> 1) & 1, abort_flag);
            for (int j = 0; j < n; ++j, ++g) {
                const int sb = g & 1;
                // (the score buffer is free: tile g - 2's PV product, issued before, waited
                // for its probabilities)
                mbar_wait(bars + Lay::B_KFULL + kp.slot, kp.phase, abort_flag);
                tc_fence_after();
                const bool dead = warp_uniform(*abort_flag) != 0;
                if (elect_one()) {
                    if (!dead) {
                        const uint64_t a0 = desc_advance(dk0, kp.slot * Lay::TILE_BYTES);
                        const uint64_t b0 = desc_advance(dq0, qs * Lay::Q_BYTES);
                        const uint32_t d_s = tmem + Lay::T_S + sb * TP;
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk) {
                            const uint32_t koff = (kk >> 2) * Lay::GROUP_BYTES + (kk & 3) * 32;
                            const uint32_t qoff = (kk >> 2) * Lay::Q_GROUP_BYTES + (kk & 3) * 32;
                            umma_bf16(d_s, desc_advance(a0, koff), desc_advance(b0, qoff), idesc_qk,
                                      kk > 0 ? 1u : 0u);
                        }
                    }
                    umma_commit(bars + Lay::B_SFULL + sb);
                    if (!Lay::P_IN_K) umma_commit(bars + Lay::B_KEMPTY + kp.slot);
                    if (j == n - 1) umma_commit(bars + Lay::B_QEMPTY + qs);
                }
                __syncwarp();
                kp.advance();
                if (g > 0) issue_pv(prev_first, prev_to);
                prev_first = (j == 0);
                prev_to = t_o;
            }
        }
        if (g > 0) issue_pv(prev_first, prev_to);
        // all MMAs finished before TMEM can be released
        if (elect_one()) umma_commit(bars + Lay::B_DRAIN);
        __syncwarp();
        mbar_wait_drain(bars + Lay::B_DRAIN, 0);
    } else {
        // ------------------------------------------------------------ softmax warpgroups
        const int wg = warp >> 2;
        const int wq = warp & 3;
        const int t = wq * 32 + lane;           // key row of S^T, and d of O^T
        const int q0 = wg * NC;                 // first query column of this warpgroup
        const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
        // this thread's row of the probability tile (128-byte swizzled atoms): its hi and
        // lo columns' 16-byte chunks
        const uint32_t p_row = smem_addr(smem) + (Lay::P_IN_K ? Lay::OFF_K : Lay::OFF_P) +
                               (uint32_t)(t >> 3) * 1024u + (uint32_t)(t & 7) * 128u;
        const uint32_t p_swz = (uint32_t)(t & 7);
        const float sl2 = p.scale_log2;
        const uint64_t sl2x2 = pack2(sl2, sl2);
        float *nm = reinterpret_cast<float *>(smem + Lay::OFF_NM) + q0;           // [NC]
        float *red = reinterpret_cast<float *>(smem + Lay::OFF_RED) + wg * 4 * NC;   // [4][NC]
        float *linv = reinterpret_cast<float *>(smem + Lay::OFF_LINV) + q0;       // [OB][TP]
        float *pmx = reinterpret_cast<float *>(smem + Lay::OFF_PMX) + q0;         // [OB][TP]
        float2 *ml = reinterpret_cast<float2 *>(smem + Lay::OFF_PMX) + q0;        // cluster split: [TP] over pmx

        uint64_t lacc[NC / 2];   // this key row's share of every owned query's row sum, in pairs
#pragma unroll
        for (int c = 0; c < NC / 2; ++c) lacc[c] = 0ull;
        uint32_t dbits = 0;   // bit c: key t (tree node t) is visible to query q0 + c
        int cur_b = -1;
        int g = 0;
        KPos kp;
        VPos vp;
        int cur_k = 0;        // this CTA's unit counter (selects the O accumulator)
        // a finished segment whose output still sits in TMEM; a partial one (a
        // unit cut by the work split) goes to its slot instead of the output
        // pend_f: bit 0 a segment is pending, bit 1 it is partial, bit 2 it was
        // the range's first segment, bit 3 its O accumulator
        int pend_f = 0, pend_u = 0, pend_g = 0;

        // Probabilities of this thread's key row for its NC query columns from its raw
        // scores r, against the current running maxima, exponents clamped at 64 so
        // nothing overflows before a rescale.  STORE: split into bf16 hi + lo, store
        // into the probability tile at byte offset `pbuf` and add to lacc.  UNDO: subtract the
        // same values from lacc again (bit-identical to an earlier STORE with the same
        // maxima).  Returns the largest unclamped exponent.
        auto emit = [&](auto bits_c, auto undo_c, const Cols &r, uint32_t bits, uint32_t pbuf) {
            constexpr bool BITS = decltype(bits_c)::value != 0;
            constexpr bool UNDO = decltype(undo_c)::value != 0;
            float maxd = -INFINITY;
#pragma unroll
            for (int h = 0; h < NC; h += 8) {
                const ulonglong2 na = *reinterpret_cast<const ulonglong2 *>(nm + h);
                const ulonglong2 nb = *reinterpret_cast<const ulonglong2 *>(nm + h + 4);
                const uint64_t nmv[4] = {na.x, na.y, nb.x, nb.y};
                uint32_t hw[4], lw[4];
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    float d0, d1;
                    unpack2(fma2(pack2(__uint_as_float(r[h + e]), __uint_as_float(r[h + e + 1])), sl2x2, nmv[e >> 1]),
                            d0, d1);
                    if (BITS) {
                        d0 = ((bits >> (h + e)) & 1u) ? d0 : -INFINITY;
                        d1 = ((bits >> (h + e + 1)) & 1u) ? d1 : -INFINITY;
                    }
                    maxd = max3(maxd, d0, d1);
                    const float p0 = ex2(fminf(d0, 64.f)), p1 = ex2(fminf(d1, 64.f));
                    if (UNDO) {
                        lacc[(h + e) >> 1] = add2(lacc[(h + e) >> 1], pack2(-p0, -p1));
                    } else {
                        const uint64_t pp = pack2(p0, p1);
                        lacc[(h + e) >> 1] = add2(lacc[(h + e) >> 1], pp);
                        split_bf16x2(pp, p0, p1, hw[e >> 1], lw[e >> 1]);
                    }
                }
                if (!UNDO) {
                    const int ch = q0 + h, cl = TP + q0 + h;   // hi and lo columns
                    const uint32_t ah = p_row + pbuf + (uint32_t)(ch >> 6) * Lay::GROUP_BYTES +
                                        ((((uint32_t)(ch & 63) >> 3) ^ p_swz) << 4);
                    const uint32_t al = p_row + pbuf + (uint32_t)(cl >> 6) * Lay::GROUP_BYTES +
                                        ((((uint32_t)(cl & 63) >> 3) ^ p_swz) << 4);
                    st_shared_v4(ah, hw[0], hw[1], hw[2], hw[3]);
                    st_shared_v4(al, lw[0], lw[1], lw[2], lw[3]);
                }
            }
            return maxd;
        };
        using store_t = kind_t<0>;
        using undo_t = kind_t<1>;

        auto load_cols = [&](uint32_t taddr, Cols &r) {   // then tmem_wait_ld
            if constexpr (NC == 32) tmem_ld32(taddr, r);
            else tmem_ld16(taddr, r);
        };

        // A score jumped past its column's maximum by more than 2^16: the optimistic
        // contributions are taken back out of the row sums; every column's maximum
        // over the 128 key rows is a warp max (redux) combined across the four warps;
        // the row sums, and O unless this is the unit's first tile, are rescaled; the
        // probabilities are recomputed.
        auto exact_tile = [&](auto bits_c, const Cols &r, uint32_t bits, uint32_t pbuf, bool first) {
            constexpr bool BITS = decltype(bits_c)::value != 0;
            (void)emit(bits_c, undo_t{}, r, bits, pbuf);
#pragma unroll
            for (int e = 0; e < NC; ++e) {
                const bool vis = !BITS || ((bits >> e) & 1u) != 0;
                const float mx = warp_max(vis ? __uint_as_float(r[e]) * sl2 : -INFINITY);
                if (lane == e) red[wq * NC + e] = mx;
            }
            named_bar_sync(1 + wg, 128);
            if (t < NC) {
                const float tm = fmaxf(fmaxf(red[t], red[NC + t]), fmaxf(red[2 * NC + t], red[3 * NC + t]));
                const float old = -nm[t];
                const float nw = fmaxf(old, tm);
                nm[t] = -nw;
                red[t] = (nw == old) ? 1.f : ex2(old - nw);   // alpha
            }
            named_bar_sync(1 + wg, 128);
            if (!first) {
                // the PV product of the previous tile must have landed first
                mbar_wait(bars + Lay::B_PFREE + ((g - 1) & 1), ((g - 1) >> 1) & 1, abort_flag);
                tc_fence_after();
            }
            const uint32_t t_o = tmem_base + lane_off + Lay::T_O + (uint32_t)(cur_k & 1) * 2 * TP + q0;
#pragma unroll
            for (int h = 0; h < NC; h += 8) {
                float a[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) a[e] = red[h + e];
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    float l0, l1;
                    unpack2(lacc[(h + e) >> 1], l0, l1);
                    lacc[(h + e) >> 1] = pack2(l0 * a[e], l1 * a[e + 1]);
                }
                if (first) continue;   // uniform
#pragma unroll
                for (int part = 0; part < 2; ++part) {
                    uint32_t o[8];
                    tmem_ld8(t_o + part * TP + h, o);
                    tmem_wait_ld(o);
#pragma unroll
                    for (int e = 0; e < 8; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * a[e]);
                    tmem_st8(t_o + part * TP + h, o);
                }
            }
            if (!first) tmem_wait_st();
            (void)emit(bits_c, store_t{}, r, bits, pbuf);
        };

        // O (hi + lo) of a finished unit's accumulator: one head-dim element per thread,
        // this warpgroup's queries in order, through `put(query column, value)`.
        auto read_o = [&](int ob, int g_last, auto put) {
            mbar_wait(bars + Lay::B_PFREE + (g_last & 1), (g_last >> 1) & 1, abort_flag);
            tc_fence_after();
            if (wq * 32 < D) {
                const uint32_t t_o = tmem_base + lane_off + Lay::T_O + (uint32_t)ob * 2 * TP + q0;
                Cols rh, rl;
                load_cols(t_o, rh);
                load_cols(t_o + TP, rl);
                tmem_wait_ld(rh);
                tmem_wait_ld(rl);
#pragma unroll
                for (int e = 0; e < NC; ++e)
                    if (q0 + e < T) put(e, __uint_as_float(rh[e]) + __uint_as_float(rl[e]));
            }
            tc_fence_before();
        };

        // The pending segment: a whole unit's output times the reciprocal row sums, or the
        // partial state of a cut one into its slot (O unnormalised, each query's running
        // maximum and row sum).
        const size_t slot_floats = split_slot_floats(D);
        auto flush_pending = [&]() {
            const int ob = (pend_f >> 3) & 1;
            if (!SPLIT || !(pend_f & 2)) {
                const float *li = linv + ob * TP;
                float *orow = p.out + ((size_t)pend_u * T + q0) * D + t;
                read_o(ob, pend_g, [&](int e, float v) { orow[(size_t)e * D] = v * li[e]; });
            } else {
                float *base = p.split_part + (size_t)(2 * (int)blockIdx.x + ((pend_f & 4) ? 0 : 1)) * slot_floats;
                read_o(ob, pend_g, [&](int e, float v) { base[(size_t)(q0 + e) * D + t] = v; });
                if (t < NC && q0 + t < T) {
                    base[(size_t)kSplitRows * D + q0 + t] = pmx[ob * TP + t];
                    base[(size_t)kSplitRows * D + kSplitRows + q0 + t] = linv[ob * TP + t];
                }
            }
        };

        int k = 0;
        SegIter<RANGE, RAGGED> it(wr);
        for (Seg sg; it.next(p, sg); ++k) {
            const UnitInfo &ui = sg.ui;
            const int u = sg.u;
            cur_k = k;
            const int ob = k & 1;
            // a new sequence's tree: this warp's parents, two nodes a lane (used after the
            // unit's first tile is on its way)
            const bool new_tree = ui.b != cur_b;
            cur_b = ui.b;
            int par[2] = {-1, -1};
            if (new_tree) {
#pragma unroll
                for (int x = 0; x < TP / 32; ++x)
                    if (lane + 32 * x < T) par[x] = ld_input(p.parent + (size_t)ui.b * T + lane + 32 * x);
            }

            for (int j = sg.j0; j < sg.j1; ++j, ++g) {
                const bool tree = (j == ui.n_pref);
                const bool first = (j == sg.j0);
                const int n_valid = tree ? T : min(Lay::KT, ui.P - j * Lay::KT);
                const bool masked = tree || n_valid < Lay::KT;
                const int sb = g & 1;
                const int ps = g & 1;
                if (first && new_tree) {
                    // ancestor sets by shuffles: lane c walks up from query q0 + c, then every
                    // lane collects its key's bit of each set
                    uint64_t anc = 0;
                    int a = lane < NC && q0 + lane < T ? q0 + lane : -1;
                    while (__any_sync(0xffffffffu, a >= 0)) {
                        if (a >= 0) anc |= 1ull << a;
                        const int i = a < 0 ? 0 : a;
                        int pa = __shfl_sync(0xffffffffu, par[0], i & 31);
                        if (TP > 32) {
                            const int hi = __shfl_sync(0xffffffffu, par[1], i & 31);
                            if (i >= 32) pa = hi;
                        }
                        a = (a > 0 && pa >= 0 && pa < a) ? pa : -1;   // strictly upwards: ends
                    }
                    dbits = 0;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const uint32_t lo = __shfl_sync(0xffffffffu, (uint32_t)anc, c);
                        const uint32_t hi = TP > 32 ? __shfl_sync(0xffffffffu, (uint32_t)(anc >> 32), c) : 0u;
                        const uint32_t w = t < 32 ? lo : hi;
                        if (t < T && ((w >> (t & 31)) & 1u)) dbits |= 1u << c;
                    }
                }
                mbar_wait(bars + Lay::B_SFULL + sb, (g >> 1) & 1, abort_flag);
                tc_fence_after();
                const uint32_t t_s = tmem_base + lane_off + Lay::T_S + sb * TP + q0;
                const uint32_t pbuf = Lay::P_IN_K ? kp.slot * Lay::TILE_BYTES : (uint32_t)ps * Lay::P_BYTES;
                Cols r;
                load_cols(t_s, r);
                // a dedicated probability tile is free once the PV product of tile
                // g - PS is done; a K slot is free as soon as S(g) is (waited above)
                if constexpr (!Lay::P_IN_K) mbar_wait(bars + Lay::B_PFREE + ps, ((g >> 1) & 1) ^ 1, abort_flag);
                tmem_wait_ld(r);
                if (first) {
                    // a unit starts with the scores of the tile's first key (visible to every
                    // query: a prefix key, or the root) as its maxima: none is above the
                    // true one, and the tile's vote catches any that is too far below
                    if (t == 0) {
#pragma unroll
                        for (int e = 0; e < NC; ++e) nm[e] = -(__uint_as_float(r[e]) * sl2);
                    }
                    named_bar_sync(1 + wg, 128);
                }
                // Done optimistically with the current running maxima; when a score
                // exceeds its maximum by more than 2^16, again by the exact path.
                const uint32_t bits = tree ? dbits : (t < n_valid ? 0xffffffffu : 0u);
                if (!masked) {
                    const float maxd = emit(kind_t<0>{}, store_t{}, r, bits, pbuf);
                    if (named_bar_or(1 + wg, 128, maxd > 16.f)) exact_tile(kind_t<0>{}, r, bits, pbuf, first);
                } else {
                    const float maxd = emit(kind_t<1>{}, store_t{}, r, bits, pbuf);
                    if (named_bar_or(1 + wg, 128, maxd > 16.f)) exact_tile(kind_t<1>{}, r, bits, pbuf, first);
                }

                // V rows of invisible keys in a partial prefix tile may be NaN: zero them
                if (!tree && masked && wg == 0) {
                    mbar_wait(bars + Lay::B_VFULL + vp.slot, vp.phase, abort_flag);
                    if (t >= n_valid) {
                        const uint32_t vrow = smem_addr(smem + Lay::OFF_V + vp.slot * Lay::TILE_BYTES) + t * 128u;
#pragma unroll
                        for (int c = 0; c < Lay::DCH; ++c)
#pragma unroll
                            for (int x = 0; x < 8; ++x)
                                st_shared_v4(vrow + c * Lay::GROUP_BYTES + x * 16, 0u, 0u, 0u, 0u);
                    }
                }
                kp.advance();
                vp.advance();
                fence_proxy_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bars + Lay::B_PFULL + ps);

                // the previous segment's output, once this segment's first tile is on its way
                if (first && pend_f) {
                    flush_pending();
                    pend_f = 0;
                }
            }

            // ------------------------------------------ unit end: row sums, LSE
            {
                named_bar_sync(1 + wg, 128);   // every thread is done reading alpha and the maxima
#pragma unroll
                for (int c = 0; c < NC; c += 16) {
                    float v[16];
#pragma unroll
                    for (int e = 0; e < 16; e += 2) unpack2(lacc[(c + e) >> 1], v[e], v[e + 1]);
                    const float s = warp_transpose_reduce16(v, lane, OpAdd());
                    if (!(lane & 1)) red[wq * NC + c + (lane >> 1)] = s;
                }
                named_bar_sync(1 + wg, 128);
                if (t < NC) {
                    const float l = red[t] + red[NC + t] + red[2 * NC + t] + red[3 * NC + t];
                    const float m = -nm[t];
                    if (!RANGE || (SPLIT && seg_whole(sg))) {
                        if (p.lse && q0 + t < T) p.lse[(size_t)u * T + q0 + t] = (m + lg2(l)) * 0.69314718055994530942f;
                        linv[ob * TP + t] = rcp(l);
                    } else if (MODE == 2) {
                        ml[t] = make_float2(m, l);
                    } else {
                        linv[ob * TP + t] = l;
                        pmx[ob * TP + t] = m;
                    }
                }
#pragma unroll
                for (int c = 0; c < NC / 2; ++c) lacc[c] = 0ull;
                pend_u = u;
                pend_g = g - 1;
                pend_f = 1 | (ob << 3);
                if (SPLIT && !seg_whole(sg)) {
                    // a part: slot 2c for the range's first segment, 2c + 1 for its last
                    pend_f |= 2 | (sg.u == wr.u_first ? 4 : 0);
                    // the part holding the unit's first tile records it for the merge
                    if (sg.j0 == 0 && threadIdx.x == 0)
                        p.split_rec[blockIdx.x] = SplitRecord{wr.x_first + (wr.n_tiles - it.left) - sg.j1, wr.n_shared, u, ui.n_tiles};
                }
            }
        }
        if (MODE == 2) {
            // this CTA's part of the unit for the cluster: O rows over the K ring (every
            // copy has landed and every product that reads it is done), maxima and sums
            // where the segment's end left them
            if (pend_f) {
                float *st = reinterpret_cast<float *>(smem + Lay::OFF_K);
                read_o(0, pend_g, [&](int e, float v) { st[(q0 + e) * D + t] = v; });
            }
        } else if (pend_f) {
            named_bar_sync(1 + wg, 128);   // the row sums are in shared memory
            flush_pending();
        }
    }

    if (MODE == 2) {
        cluster_sync();
        bool unused = false;
        if (warp < Lay::SW) {
            const int u = (int)blockIdx.x / p.cluster;
            unused = cluster_merge<1>(p, wr.parts, smem_addr(smem) + Lay::OFF_K, D * 4, smem_addr(smem) + Lay::OFF_PMX,
                          D, (int)blockIdx.x - u * p.cluster, T, (size_t)u * T, threadIdx.x, Lay::SW * 32);
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
    if (warp == Lay::SW + 1) tmem_dealloc(tmem_base, Lay::TMEM_COLS);
}

// The merge of the units cut by the work split: blockIdx.x is an attention
// CTA (gridDim.x = the attention grid), blockIdx.y a block of 256 / (D / 8)
// rows of the unit that CTA recorded; each thread merges 8 columns of a row,
// once the attention grid has completed.
__global__ void __launch_bounds__(256) split_merge_kernel(const AttnParams p, int D)
{
    // a next grid launched as a programmatic dependent may start at once; it
    // waits for this grid to complete before it reads or writes anything
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const SplitRecord r = p.split_rec[blockIdx.x];
    if (r.u < 0) return;
    const int per_row = D / 8;
    const int rows_per_block = (int)blockDim.x / per_row;
    const int lbh = r.u / p.n_qb, qb = r.u - lbh * p.n_qb;
    const int n_rows = min(kSplitRows, p.T - qb * kSplitRows);
    const int row = (int)blockIdx.y * rows_per_block + (int)threadIdx.x / per_row;
    if (row >= n_rows) return;
    const SplitParts sp = split_parts(r.n_shared, r.off, r.n_tiles);
    split_merge_chunk(p.split_part, p.out, p.lse, sp, r.n_shared, (int)gridDim.x,
                      (size_t)lbh * p.T + (size_t)qb * kSplitRows, row, ((int)threadIdx.x % per_row) * 8, D);
}

cudaError_t launch_split_merge(const AttnParams &p, int D, int grid, cudaStream_t stream)
{
    const int rows_per_block = 256 / (D / 8);
    const int rows = p.T < kSplitRows ? p.T : kSplitRows;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, (unsigned)((rows + rows_per_block - 1) / rows_per_block));
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, split_merge_kernel, p, D);
}

template <int D, int TP>
static cudaError_t launch_tree_attention_t(const AttnMaps &m, const AttnParams &p, int num_sms,
                                           bool programmatic, cudaStream_t stream)
{
    using Lay = AttnLayout<D, TP>;
    static std::atomic<uint64_t> configured[4] = {{0}, {0}, {0}, {0}};
    if (whole_ragged(p))
        return launch_attention_grid(tree_attention_kernel<D, TP, 3>, Lay::SMEM_BYTES, Lay::THREADS,
                                     configured[3], m, p, num_sms, programmatic, stream);
    if (p.cluster > 1)
        return launch_attention_grid(tree_attention_kernel<D, TP, 2>, Lay::SMEM_BYTES, Lay::THREADS,
                                     configured[2], m, p, num_sms, programmatic, stream);
    if (p.split)
        return launch_attention_grid(tree_attention_kernel<D, TP, 1>, Lay::SMEM_BYTES, Lay::THREADS,
                                     configured[1], m, p, num_sms, programmatic, stream);
    return launch_attention_grid(tree_attention_kernel<D, TP, 0>, Lay::SMEM_BYTES, Lay::THREADS,
                                 configured[0], m, p, num_sms, programmatic, stream);
}

// Asked of one attention kernel for all of them: each takes a whole SM, so the
// answer only depends on how the device groups its SMs.
int max_attention_clusters(int size)
{
    static std::atomic<int> cache[64][kMaxCluster + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    if (dev < 0 || dev >= 64 || size < 1 || size > kMaxCluster) return 0;
    return asked_once(cache[dev][size], [&] {
        using Lay = AttnLayout<128, 64>;
        auto kern = tree_attention_kernel<128, 64, 2>;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)size);
        cfg.blockDim = dim3(Lay::THREADS);
        cfg.dynamicSmemBytes = Lay::SMEM_BYTES;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)size;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Lay::SMEM_BYTES) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            return -1;
        }
        return n;
    });
}

cudaError_t launch_tree_attention(const AttnMaps &m, const AttnParams &p, int D, int num_sms,
                                  bool programmatic, cudaStream_t stream)
{
    cudaError_t e;
    if (p.T_pad > 64) e = launch_tree_attention_rows(m, p, D, num_sms, programmatic, stream);
    else if (D == 128 && p.T_pad == 64) e = launch_tree_attention_t<128, 64>(m, p, num_sms, programmatic, stream);
    else if (D == 128) e = launch_tree_attention_t<128, 32>(m, p, num_sms, programmatic, stream);
    else if (p.T_pad == 64) e = launch_tree_attention_t<64, 64>(m, p, num_sms, programmatic, stream);
    else e = launch_tree_attention_t<64, 32>(m, p, num_sms, programmatic, stream);
    if (e != cudaSuccess || !p.split) return e;
    return launch_split_merge(p, D, attention_grid(p, num_sms), stream);
}

}  // namespace ppd
