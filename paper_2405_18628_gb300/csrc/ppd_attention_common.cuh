// ppd_attention_common.cuh -- pieces shared by the two tree-attention kernels
// (ppd_attention.cu for trees of up to 64 tokens, ppd_attention_rows.cu for
// 65..512): the unit walk and the two ways to share a unit among CTAs (work split
// and clusters) with their merges, drain waits and the fused step's side warp.
#pragma once

#include "ppd_accept.cuh"
#include "ppd_device.cuh"
#include "ppd_kernels.h"

#include <algorithm>
#include <atomic>
#include <type_traits>

namespace ppd {

// A (layer, sequence, head) unit: its sequence, clamped prefix length and tiles
// (prefix tiles of 128 keys, then one tile of the tree's own keys).
struct UnitInfo {
    int lbh, qb, b, P, P_raw, n_pref, n_tiles;
};

// Unit u = (layer, sequence, head) slice lbh and block qb of its query rows
// (slices of trees over 128 tokens split their queries into blocks of 128).
template <bool SKIP = false>
PPD_DEV UnitInfo unit_info(const AttnParams &p, int u)
{
    UnitInfo ui;
    // SKIP: no division that says nothing (every role does this between two units;
    // short slices gain 1 %, the query-row kernel's loops lose 2 %)
    ui.lbh = SKIP && p.n_qb == 1 ? u : u / p.n_qb;
    ui.qb = u - ui.lbh * p.n_qb;
    ui.b = SKIP && p.B == 1 ? 0 : (ui.lbh / p.H) % p.B;
    ui.P_raw = ld_input(p.prefix_len + ui.b);
    ui.P = min(max(ui.P_raw, 0), p.S_max);
    ui.n_pref = (ui.P + 127) >> 7;
    ui.n_tiles = ui.n_pref + p.n_tt;
    return ui;
}

// ------------------------------------------------------------------ work split
//
// Units are taken round-robin (CTA c: units c, c+G, c+2G, ...), whole, unless there
// are fewer units than CTAs.  With p.cluster > 1 every unit then has a cluster of
// CTAs (plan_cluster, cluster_merge).  With p.split (the clusters that fit would be
// too small) all units are shared out by their key tiles: the
// tiles (unit u's tiles 0..n_tiles(u)-1, units in order) go to the CTAs in
// equal contiguous ranges (CTA c: tiles [c*N/G, (c+1)*N/G)).  A unit cut by a
// range boundary is done in parts, one per CTA; each part leaves its partial
// softmax state (the unnormalised O rows, the running maximum and the row sum
// of every query) in a slot of its CTA, and the CTA holding the unit's first
// tile leaves a record of it.  Once the launch is complete a second, small
// grid merges every recorded unit, so nothing in the attention grid waits
// for, or counts, other CTAs.

struct WorkRange {
    int rr_units;            // units taken whole, round-robin (all, or none)
    int u_first, j_first;    // first unit and tile of this CTA's range (split)
    int n_tiles;             // tiles in the range (0: none)
    int u_last;              // last unit the range touches
    long long x_first;       // index of the range's first tile
    long long n_shared;        // tiles shared out by the split
    const uint8_t *seq;      // not null: whole jobs go longest sequence first, in this order
    int parts;               // cluster split: the CTAs of the cluster with tiles, the first ones
};

// Whole jobs (n in all, `per` a slice) go to `step` queues round-robin, queue x
// getting x, x + step, ...  With sequences of different lengths they are taken
// longest sequence first, rounds alternating in direction (the last, partial one
// forward), so that a queue's long and short jobs add up: eight sequences of
// 66-128 tiles over 152 SMs leave the longest queue 5 % above the mean instead of
// 16 %.  ragged_job: the job at round-robin position i (< rounds * step) then, or
// -1.  An instantiation of its own (batches of 2 to kSplitMaxB): the test alone, in
// the loops of every role, cost single sequences 3 %.
PPD_DEV int ragged_job(const AttnParams &p, const uint8_t *seq, int i, int step, int n, int per)
{
    const int r = i / step, x = i - r * step, rounds = (n + step - 1) / step;
    const int j = r * step + (((rounds - 1 - r) & 1) ? step - 1 - x : x);
    if (r >= rounds || j >= n) return -1;
    const int per_layer = p.H * per, per_seq = p.L * per_layer;
    const int b = seq[j / per_seq], rest = j % per_seq;
    return (rest / per_layer * p.B + b) * per_layer + rest % per_layer;
}

// First shared tile of CTA c, and the CTA holding shared tile x.
PPD_DEV long long split_start(int c, long long N, int G) { return (long long)c * N / G; }
PPD_DEV int split_cta_of(long long x, long long N, int G) { return (int)(((x + 1) * G + N - 1) / N) - 1; }

// This CTA's share of its cluster's unit (the cluster split): no lane needs another's.
template <bool kHint = false>
PPD_DEV WorkRange plan_cluster(const AttnParams &p)
{
    WorkRange w{};
    const int c = (int)blockIdx.x;
    w.u_first = w.u_last = c / p.cluster;
    const int32_t *P = p.prefix_len + w.u_first / (p.H * p.n_qb) % p.B;
    const int nt = ((min(max(kHint ? ld_relaxed_gpu_s32(P) : ld_input(P), 0), p.S_max) + 127) >> 7) + p.n_tt;
    const int r = c - w.u_first * p.cluster;
    w.parts = min(p.cluster, nt);
    if (r < w.parts) {
        w.j_first = r * nt / w.parts;
        w.n_tiles = (r + 1) * nt / w.parts - w.j_first;
    }
    return w;
}

// This CTA's work, computed by one whole warp (every lane gets the result).
// The tiles of one layer's block of sequence b number H * n_qb * (n_pref(b) +
// n_tt); lanes hold sequences b = lane and lane + 32.
// seq: kSplitMaxB bytes of shared memory for the order of the sequences (whole
// jobs; null: always round-robin).  kHint: the prefix
// lengths are read through L2 because they may still be changing (a plan
// made before the wait of a chained launch, used for prefetch hints only).
template <bool kHint = false>
PPD_DEV WorkRange plan_range(const AttnParams &p, int lane, uint8_t *seq = nullptr)
{
    if (p.cluster > 1) return plan_cluster<kHint>(p);
    WorkRange w{};
    const int G = (int)gridDim.x, c = (int)blockIdx.x;
    // no range of tiles unless one is found below
    w.u_first = p.n_units;
    w.u_last = -1;
    w.n_tiles = 0;
    w.rr_units = p.split ? 0 : p.n_units;   // units taken whole, round-robin
    w.seq = nullptr;
    const unsigned full = 0xffffffffu;
    const int per_b = p.H * p.n_qb;
    auto nt_of = [&](int b) {
        const int P = min(max(kHint ? ld_relaxed_gpu_s32(p.prefix_len + b) : ld_input(p.prefix_len + b), 0),
                          p.S_max);
        return ((P + 127) >> 7) + p.n_tt;
    };
    if (w.rr_units > 0) {
        if (!seq || p.B < 2 || p.B > kSplitMaxB || p.n_units <= G) return w;
        // sequences by falling tile count, the lower index first among equals
        const int t0 = lane < p.B ? nt_of(lane) : -1, t1 = lane + 32 < p.B ? nt_of(lane + 32) : -1;
        int r0 = 0, r1 = 0;
        bool equal = true;
        for (int b = 0; b < p.B; ++b) {
            const int t = b < 32 ? __shfl_sync(full, t0, b) : __shfl_sync(full, t1, b - 32);
            r0 += t > t0 || (t == t0 && b < lane);
            r1 += t > t1 || (t == t1 && b < lane + 32);
            equal = equal && t == __shfl_sync(full, t0, 0);
        }
        if (equal) return w;
        if (lane < p.B) seq[r0] = (uint8_t)lane;
        if (lane + 32 < p.B) seq[r1] = (uint8_t)(lane + 32);
        w.seq = seq;
        return w;
    }
    const int w0 = lane < p.B ? per_b * nt_of(lane) : 0;
    const int w1 = lane + 32 < p.B ? per_b * nt_of(lane + 32) : 0;
    int s0 = w0, s1 = w1;   // inclusive prefix sums over b
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(full, s0, o);
        const int x = __shfl_up_sync(full, s1, o);
        if (lane >= o) {
            s0 += a;
            s1 += x;
        }
    }
    s1 += __shfl_sync(full, s0, 31);
    const long long per_layer = __shfl_sync(full, s1, 31);
    const long long N = per_layer * p.L;
    // unit and tile of global tile x (0 <= x < N)
    auto locate = [&](long long x, int &u, int &j) {
        const int l = (int)(x / per_layer);
        const int r = (int)(x - (long long)l * per_layer);
        const unsigned m0 = __ballot_sync(full, lane < p.B && s0 > r);
        int b, incl, wt;
        if (m0) {
            b = __ffs(m0) - 1;
            incl = __shfl_sync(full, s0, b);
            wt = __shfl_sync(full, w0, b);
        } else {
            const unsigned m1 = __ballot_sync(full, lane + 32 < p.B && s1 > r);
            const int bl = m1 ? __ffs(m1) - 1 : 0;
            b = bl + 32;
            incl = __shfl_sync(full, s1, bl);
            wt = __shfl_sync(full, w1, bl);
        }
        const int rb = r - (incl - wt);   // tile offset within the block of sequence b
        const int nt = wt / per_b;
        const int idx = rb / nt;
        j = rb - idx * nt;
        u = (l * p.B + b) * per_b + idx;
    };
    w.n_shared = N;
    const long long gs = split_start(c, w.n_shared, G), ge = split_start(c + 1, w.n_shared, G);
    w.x_first = gs;
    w.n_tiles = (int)(ge - gs);
    if (ge > gs) {
        int jl;
        locate(gs, w.u_first, w.j_first);
        locate(ge - 1, w.u_last, jl);
    }
    return w;
}

// Before the wait of a chained launch (one warp, all lanes): ask L2 for the
// first `n` K and V prefix tiles of this CTA's work, from a plan made with
// prefix lengths that may still be changing.  Only a hint -- nothing is
// written to shared memory and nothing waits on it; the real loads follow the
// wait with the plan remade -- so the preceding grid's work overlaps the
// first tiles' trip from HBM.  Tree tiles are skipped (in a model the
// preceding grids write them).  Whole units go in index order here, also where
// the work then takes the longest sequences first: L2 serves every CTA, so a tile
// helps whichever CTA streams it, and working that order out costs time before the
// hint (calls of 8 sequences of up to 4096 keys, 32 heads, 64 tokens: 76.5 us like
// this, 77.4 in the order of the work, 78.4 without the hint).
template <bool SPLIT>
PPD_DEV void prefetch_first_tiles(const AttnParams &p, int lane, const CUtensorMap *kc,
                                  const CUtensorMap *vc, int dch, int n)
{
    const WorkRange w = plan_range<true>(p, lane);
    if (lane != 0) return;
    int u = SPLIT ? w.u_first : (int)blockIdx.x;
    int j = SPLIT ? w.j_first : 0;
    int left = SPLIT ? w.n_tiles : n;
    for (int k = 0; k < n && left > 0 && u < p.n_units; ++k, --left) {
        const int lbh = u / p.n_qb;
        const int b = (lbh / p.H) % p.B;
        const int P = min(max(ld_relaxed_gpu_s32(p.prefix_len + b), 0), p.S_max);
        const int n_pref = (P + 127) >> 7;
        if (j < n_pref) {
            for (int c = 0; c < dch; ++c) {
                tma_prefetch_l2_3d(kc, c * 64, j * 128, lbh);
                tma_prefetch_l2_3d(vc, c * 64, j * 128, lbh);
            }
            ++j;
        } else {   // the unit's tree tiles: on to the next unit
            u = SPLIT ? u + 1 : u + (int)gridDim.x;
            j = 0;
        }
    }
}

// Position in a ring of tile slots: slot and the parity of its current phase.
template <int RS>
struct RingPos {
    int slot = 0;
    uint32_t phase = 0;
    PPD_DEV void advance()
    {
        if (++slot == RS) {
            slot = 0;
            phase ^= 1u;
        }
    }
};

// One stretch of a unit's tiles [j0, j1) processed by this CTA.
struct Seg {
    UnitInfo ui;
    int u, j0, j1;
};

// Walks this CTA's segments in order (every role of the CTA walks the same
// sequence): whole units round-robin, or (SPLIT) its range of tiles, `left`
// counting the range's tiles not yet handed out.
template <bool SPLIT, bool RAGGED = false>
struct SegIter {
    int u, j0, left;       // whole units: the next round-robin position; else the range's next unit
    const uint8_t *seq;
    PPD_DEV explicit SegIter(const WorkRange &w)
    {
        u = SPLIT ? w.u_first : (int)blockIdx.x;
        j0 = SPLIT ? w.j_first : 0;
        left = SPLIT ? w.n_tiles : 0;
        seq = RAGGED ? w.seq : nullptr;
    }
    PPD_DEV bool next(const AttnParams &p, Seg &s)
    {
        if (!SPLIT) {
            int unit = u;
            if (RAGGED && seq) unit = ragged_job(p, seq, u, (int)gridDim.x, p.n_units, 1);
            if (unit < 0 || unit >= p.n_units) return false;
            s.ui = unit_info<true>(p, unit);
            s.u = unit;
            s.j0 = 0;
            s.j1 = s.ui.n_tiles;
            u += (int)gridDim.x;
            return true;
        }
        if (left <= 0 || u >= p.n_units) return false;
        s.ui = unit_info<true>(p, u);
        s.u = u;
        s.j0 = j0;
        s.j1 = min(s.ui.n_tiles, j0 + left);
        if (s.j1 <= j0) {   // cannot happen with a consistent plan; never loop on it
            left = 0;
            return false;
        }
        left -= s.j1 - j0;
        ++u;
        j0 = 0;
        return true;
    }
};

// Does the CTA process all of the segment's unit?
PPD_DEV bool seg_whole(const Seg &s) { return s.j0 == 0 && s.j1 == s.ui.n_tiles; }

// The parts of a cut unit: the CTAs c_a..c_b whose ranges are not empty (a
// launch with fewer tiles than CTAs leaves some ranges empty).  Part c's slot
// is 2c for the first segment of its range and 2c + 1 for the last (only c_a
// can hold the unit in its last segment).
struct SplitParts {
    int c_a, c_b, slot_a, n_parts;
};

PPD_DEV bool split_nonempty(int c, long long N, int G) { return split_start(c + 1, N, G) > split_start(c, N, G); }

PPD_DEV SplitParts split_parts(long long N, long long off, int n_tiles)
{
    SplitParts sp;
    const int G = (int)gridDim.x;
    sp.c_a = split_cta_of(off, N, G);
    sp.c_b = split_cta_of(off + n_tiles - 1, N, G);
    sp.slot_a = 2 * sp.c_a + (split_start(sp.c_a, N, G) < off ? 1 : 0);
    sp.n_parts = 0;
    for (int c = sp.c_a; c <= sp.c_b; ++c) sp.n_parts += split_nonempty(c, N, G) ? 1 : 0;
    return sp;
}

PPD_DEV int split_slot(const SplitParts &sp, int c) { return c == sp.c_a ? sp.slot_a : 2 * c; }

// Floats of one partial-state slot: kSplitRows rows of D, their maxima, their sums.
PPD_DEV size_t split_slot_floats(int D) { return (size_t)kSplitRows * (D + 2); }

// Merge the partial states of a cut unit whose parts have all arrived: slot
// row r (output row out_row0 + r), columns [c0, c0 + 8), by one thread.  One
// pass over the parts with a running maximum M: part c enters with weight
// 2^(m_c - M), earlier sums are rescaled when M grows; the output is the
// weighted sum of the parts' O rows over the weighted sum of their row sums.
// The parts are read eight at a time, every load of a batch issued before any
// is used, so a batch costs one round trip to L2.
static __device__ __forceinline__ void split_merge_chunk(const float *split_part, float *out, float *lse,
                                                         const SplitParts &sp, long long N, int G,
                                                         size_t out_row0, int r, int c0, int D)
{
    constexpr int PB = 8;   // parts per batch
    const size_t sf = split_slot_floats(D);
    const bool dense = N >= G;   // no empty ranges
    float M = -INFINITY, Ls = 0.f;
    float acc[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) acc[x] = 0.f;
    for (int cb = sp.c_a; cb <= sp.c_b; cb += PB) {
        float mc[PB], lc[PB];
        float4 v[PB][2];
#pragma unroll
        for (int y = 0; y < PB; ++y) {
            const int c = cb + y;
            const bool live = c <= sp.c_b && (dense || split_nonempty(c, N, G));
            const float *b_ = split_part + (size_t)split_slot(sp, live ? c : sp.c_a) * sf;
            mc[y] = live ? __ldcg(b_ + (size_t)kSplitRows * D + r) : -INFINITY;
            lc[y] = live ? __ldcg(b_ + (size_t)kSplitRows * D + kSplitRows + r) : 0.f;
            const float4 *o4 = reinterpret_cast<const float4 *>(b_ + (size_t)r * D + c0);
            v[y][0] = live ? __ldcg(o4) : make_float4(0.f, 0.f, 0.f, 0.f);
            v[y][1] = live ? __ldcg(o4 + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int y = 0; y < PB; ++y) {
            if (mc[y] == -INFINITY) continue;   // absent, or the part saw no key of this row
            const float Mn = fmaxf(M, mc[y]);
            const float so = ex2(M - Mn);       // 0 while M = -inf
            const float w = ex2(mc[y] - Mn);
            Ls = fmaf(Ls, so, w * lc[y]);
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                acc[4 * x] = fmaf(acc[4 * x], so, w * v[y][x].x);
                acc[4 * x + 1] = fmaf(acc[4 * x + 1], so, w * v[y][x].y);
                acc[4 * x + 2] = fmaf(acc[4 * x + 2], so, w * v[y][x].z);
                acc[4 * x + 3] = fmaf(acc[4 * x + 3], so, w * v[y][x].w);
            }
            M = Mn;
        }
    }
    const float inv = 1.f / Ls;
    float *dst = out + (out_row0 + r) * D + c0;
    if ((reinterpret_cast<uintptr_t>(out) & 15u) == 0) {
        reinterpret_cast<float4 *>(dst)[0] = make_float4(acc[0] * inv, acc[1] * inv, acc[2] * inv, acc[3] * inv);
        reinterpret_cast<float4 *>(dst)[1] = make_float4(acc[4] * inv, acc[5] * inv, acc[6] * inv, acc[7] * inv);
    } else {
#pragma unroll
        for (int x = 0; x < 8; ++x) dst[x] = acc[x] * inv;
    }
    if (c0 == 0 && lse) lse[out_row0 + r] = (M + lg2(Ls)) * 0.69314718055994530942f;
}

// The end of a cluster split: the first `parts` CTAs of the cluster have left their
// partial states in shared memory -- unnormalised O rows at `o` (`pitch` bytes apart),
// each row's (maximum, sum) at `ml` (maximum -inf: no key seen, the row of O may hold
// anything) -- and all threads have passed a cluster_sync().  CTA `rank` merges its
// share of the n_rows rows, 4 X columns per thread at a time (four of each X-th of the
// row, so that a warp reads whole lines), every value of kParts parts loaded before
// any is used.  The code runs once or twice a launch and mostly waits for its own
// instructions (a first pass takes 1.1 us, a second 0.35), so it is kept short: all
// kMaxCluster parts in one go took 32 calls of 32 slices, 64 tokens, 433 us instead of
// 421.  Returns true when a part had weight 0 in a row of this thread's, so that its O
// values, unused, may still be on their way.  X = 2 pays with many rows (the query-row
// kernel: 16 calls of 64 units, 200 tokens, 343 -> 326 us), X = 1 keeps more threads
// busy with few.
template <int X>
PPD_DEV bool cluster_merge(const AttnParams &p, int parts, uint32_t o, uint32_t pitch, uint32_t ml, int D,
                           int rank, int n_rows, size_t out_row0, int tid, int n_threads)
{
    constexpr int kParts = 4;
    const int n = p.cluster, per_row = D / (4 * X);
    const int r0 = rank * n_rows / n, r1 = (rank + 1) * n_rows / n;
    const bool vec_out = (reinterpret_cast<uintptr_t>(p.out) & 15u) == 0;
    bool unused = false;
    for (int i = tid; i < (r1 - r0) * per_row; i += n_threads) {
        const int row = r0 + i / per_row, col = 4 * (i % per_row);   // and D / X further
        float M = -INFINITY, Ls = 0.f, acc[4 * X] = {};
#pragma unroll 1
        for (int c0 = 0; c0 < parts; c0 += kParts) {
            float2 s[kParts];
            float4 v[kParts][X];
            float Mn = M;
#pragma unroll
            for (int c = 0; c < kParts; ++c) {
                s[c] = make_float2(-INFINITY, 0.f);
                if (c0 + c < parts) {
                    s[c] = ld_cluster_v2(cluster_map(ml + row * 8, c0 + c));
                    const uint32_t a = cluster_map(o + row * pitch + col * 4, c0 + c);
#pragma unroll
                    for (int x = 0; x < X; ++x) v[c][x] = ld_cluster_v4(a + x * (4 * D / X));
                }
            }
#pragma unroll
            for (int c = 0; c < kParts; ++c) {
                Mn = fmaxf(Mn, s[c].x);
                unused |= c0 + c < parts && s[c].x == -INFINITY;
            }
            const float f = M == -INFINITY ? 0.f : ex2(M - Mn);
            M = Mn;
            Ls *= f;
#pragma unroll
            for (int x = 0; x < 4 * X; ++x) acc[x] *= f;
#pragma unroll
            for (int c = 0; c < kParts; ++c) {
                if (c0 + c >= parts || s[c].x == -INFINITY) continue;
                const float w = ex2(s[c].x - M);
                Ls = fmaf(w, s[c].y, Ls);
#pragma unroll
                for (int x = 0; x < X; ++x) {
                    acc[4 * x] = fmaf(w, v[c][x].x, acc[4 * x]);
                    acc[4 * x + 1] = fmaf(w, v[c][x].y, acc[4 * x + 1]);
                    acc[4 * x + 2] = fmaf(w, v[c][x].z, acc[4 * x + 2]);
                    acc[4 * x + 3] = fmaf(w, v[c][x].w, acc[4 * x + 3]);
                }
            }
        }
        const float inv = 1.f / Ls;
        float *dst = p.out + (out_row0 + row) * D + col;
        if (vec_out) {
#pragma unroll
            for (int x = 0; x < 4 * X; x += 4)
                *reinterpret_cast<float4 *>(dst + x / 4 * (D / X)) =
                    make_float4(acc[x] * inv, acc[x + 1] * inv, acc[x + 2] * inv, acc[x + 3] * inv);
        } else {
#pragma unroll
            for (int x = 0; x < 4 * X; ++x) dst[x / 4 * (D / X) + x % 4] = acc[x] * inv;
        }
        if (col == 0 && p.lse) p.lse[out_row0 + row] = (M + lg2(Ls)) * 0.69314718055994530942f;
    }
    return unused;
}

// The barrier before the cluster's CTAs leave: no shared memory that a peer reads
// goes away.  A thread that has used every value it loaded has no load under way and
// arrives without waiting for its output's stores (with a release, 16 calls of four
// slices, 64 tokens, took 118 us instead of 111); other warps arrive with release.
PPD_DEV void cluster_leave(bool unused)
{
    if (__any_sync(0xffffffffu, unused)) cluster_sync();
    else cluster_sync_exit();
}

// The statuses of an attention call that is not part of a fused step, by one
// spare warp per CTA: sequence b by CTA b mod grid, a malformed tree before a
// prefix length outside the cache.  Every status gets its one plain store here,
// at the start of the grid; only a CTA whose waits ran out, seconds later,
// raises it again (atomicMax).
PPD_DEV void status_warp(const AttnParams &p, int lane)
{
    for (int b = blockIdx.x; b < p.B; b += gridDim.x) {
        bool bad = false;
        for (int i = lane; i < p.T; i += 32) {
            const int pa = ld_input(p.parent + (size_t)b * p.T + i);
            bad |= i == 0 ? pa != -1 : (pa < 0 || pa >= i);
        }
        bad = __any_sync(0xffffffffu, bad);
        const int P = ld_input(p.prefix_len + b);
        if (lane == 0) p.dev_status[b] = bad ? kErrTree : (P < 0 || P > p.S_max ? kErrCapacity : kOk);
    }
}

PPD_DEV void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c),
                 "r"(d)
                 : "memory");
}

// Time-bounded wait that ignores the abort flag (used only to drain copies
// still in flight after an abort, before the CTA exits).
PPD_DEV void mbar_wait_drain(uint64_t *bar, uint32_t parity)
{
    const uint32_t a = smem_addr(bar);
    const uint64_t t0 = global_timer();
    while (!mbar_try_wait(a, parity))
        if (global_timer() - t0 > kWaitLimitNs) return;
}

template <int K>
using kind_t = std::integral_constant<int, K>;

// Mask kinds of a tile: every key visible (a full prefix tile), keys t < n_valid
// visible (the last, partial prefix tile), or the tree-ancestor mask.
enum : int { kMaskNone = 0, kMaskRows = 1, kMaskTree = 2 };

// One warp's partial top-1 of columns [lo, hi) of the logits row x, and with
// kStats the softmax statistics of the same columns at scale stat_k; lane 0
// holds the result.  Four 16-byte loads per lane (2 KB per warp) are in
// flight at a time: deeper bursts of loads from this warp slow the softmax
// warps that share its SM sub-partition more than they gain.
template <bool kStats>
PPD_DEV void warp_logit_partial(const float *x, int lo, int hi, bool vec, float stat_k, int lane,
                                float &bv, int &bi, SoftStats &st)
{
    bv = -INFINITY;
    bi = INT_MAX;
    st = SoftStats{};
    auto take4 = [&](const float4 &f, int base) {
        consider(f.x, base, bv, bi);
        consider(f.y, base + 1, bv, bi);
        consider(f.z, base + 2, bv, bi);
        consider(f.w, base + 3, bv, bi);
        if (kStats) stats_add4(st, f.x * stat_k, f.y * stat_k, f.z * stat_k, f.w * stat_k);
    };
    if (vec) {
        const float4 *x4 = reinterpret_cast<const float4 *>(x);
        const int n4_hi = hi >> 2;
        int i = (lo >> 2) + lane;
        for (; i + 3 * 32 < n4_hi; i += 4 * 32) {
            float4 f[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) f[k] = __ldcs(x4 + i + k * 32);
#pragma unroll
            for (int k = 0; k < 4; ++k) take4(f[k], 4 * (i + k * 32));
        }
        for (; i < n4_hi; i += 32) take4(__ldcs(x4 + i), 4 * i);
    } else {
        for (int i = lo + lane; i < hi; i += 32) {
            const float v = __ldcs(x + i);
            consider(v, i, bv, bi);
            if (kStats) stats_add4(st, v * stat_k, -INFINITY, -INFINITY, -INFINITY);
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float ov = __shfl_down_sync(0xffffffffu, bv, off);
        const int oi = __shfl_down_sync(0xffffffffu, bi, off);
        consider(ov, oi, bv, bi);
        if (kStats) {
            SoftStats o;
            o.m = __shfl_down_sync(0xffffffffu, st.m, off);
            o.s = __shfl_down_sync(0xffffffffu, st.s, off);
            o.t = __shfl_down_sync(0xffffffffu, st.t, off);
            stats_merge(st, o);
        }
    }
}

// In-grid argmax of the fused step: this CTA's chunks of the [B*T][splits]
// partial grid (chunk c by CTA c mod grid), then its flag.  Each lane fences
// its own writes before the warp barrier, so lane 0's release covers them all.
PPD_DEV void side_argmax_chunks(const AttnParams &p, unsigned long long tag, int lane)
{
    const FusedStep &f = p.fs;
    const int S = f.splits;
    const long long n_chunks = (long long)p.B * p.T * S;
    for (long long c = blockIdx.x; c < n_chunks; c += gridDim.x) {
        const long long row = c / S;
        const int lo = (int)(c - row * S) * f.chunk;
        const int hi = min(f.V, lo + f.chunk);
        const float *x = f.logits + row * (long long)f.V;
        float bv;
        int bi;
        SoftStats st;
        if (f.typical) warp_logit_partial<true>(x, lo, hi, f.vec != 0, f.stat_k, lane, bv, bi, st);
        else warp_logit_partial<false>(x, lo, hi, f.vec != 0, 0.f, lane, bv, bi, st);
        if (lane == 0) {
            f.part_val[c] = bv;
            f.part_idx[c] = bi;
            if (f.typical) {
                float *ps = f.part_stats + 3 * c;
                ps[0] = st.m;
                ps[1] = st.s;
                ps[2] = st.t;
            }
        }
    }
    __threadfence();
    __syncwarp();
    if (lane == 0 && (int)blockIdx.x != f.withhold_cta) st_release_gpu(f.ready + blockIdx.x, tag);
}

// Wait until every CTA of the grid has published `tag` (bounded: raises the
// CTA's abort flag and returns false after f.wait_limit_ns, or at once when the
// flag is already up; lane 0 takes that decision for the whole warp, so no
// lane leaves while others still shuffle).  Only CTA 0 reads the per-CTA flags; once all are up
// it advances the epoch for the next call and publishes `tag` in all_ready,
// the one word the other CTAs poll (from one lane, with a backoff), so the
// waits add little to the L2 traffic of the attention stream.
PPD_DEV bool side_wait_all(const AttnParams &p, unsigned long long tag, int lane,
                           volatile int *abort_flag)
{
    const FusedStep &f = p.fs;
    const int G = (int)gridDim.x;
    const uint64_t t0 = global_timer();
    bool done = false;
    while (true) {
        if (blockIdx.x == 0) {
            bool ok = true;
            for (int c = lane; c < G; c += 32) ok = ok && ld_acquire_gpu(f.ready + c) == tag;
            done = __all_sync(0xffffffffu, ok);
        } else {
            done = __shfl_sync(0xffffffffu, lane == 0 && ld_acquire_gpu(f.all_ready) == tag, 0);
        }
        if (done) break;
        const bool give_up = __shfl_sync(
            0xffffffffu, lane == 0 && (*abort_flag || global_timer() - t0 > f.wait_limit_ns), 0);
        if (give_up) {
            if (lane == 0) *abort_flag = 1;
            return false;
        }
        __nanosleep(blockIdx.x == 0 ? 200 : 1000);
    }
    __syncwarp();
    __threadfence();
    if (blockIdx.x == 0 && lane == 0) {
        st_relaxed_gpu(f.epoch, tag);
        st_release_gpu(f.all_ready, tag);
    }
    return true;
}

// Side work of the fused verification step, done by one extra warp of every CTA
// while the other warps stream attention.  Once the argmax partials are
// complete -- the preceding grid's (griddepcontrol.wait), or with in_grid the
// ones the side warps of all CTAs compute first (side_argmax_chunks, then
// side_wait_all) -- for every sequence b this CTA touches, or is designated to
// report (b mod grid), the warp combines the node argmax from the partial
// maxima, decides acceptance, writes the sequence's outputs if designated, and
// copies the accepted tree K/V rows of this CTA's own (layer, sequence, head)
// slices into the cache.  Attention only reads cache rows below each prefix,
// so the copies never race with it.  Scratch (parent copies, top-1 tokens,
// path) lives in a per-CTA slice of the workspace.  Kept out of line so that
// its code does not reshape the register allocation of the attention loops.
template <bool kSmallTree>
static __device__ __noinline__ void fused_side_warp(const AttnParams &p, const WorkRange &wr, int lane,
                                                    volatile int *abort_flag)
{
    const FusedStep &f = p.fs;
    unsigned long long tag = 0;
    bool have_all = false;
    if (f.in_grid) {
        tag = __shfl_sync(0xffffffffu, lane == 0 ? ld_relaxed_gpu(f.epoch) + 1ull : 0ull, 0);
        side_argmax_chunks(p, tag, lane);
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        have_all = true;
    }
    // the units whose first tile this CTA streams (its round-robin units and the
    // units starting in its range) compact their slices here
    const int t_lo = wr.u_first + (wr.j_first > 0 ? 1 : 0), t_hi = wr.n_tiles > 0 ? wr.u_last : -1;
    auto owns_first_tile = [&](auto fn) {
        for (int u = (int)blockIdx.x; u < wr.rr_units; u += (int)gridDim.x)
            if (fn(u)) return;
        for (int u = t_lo; u <= t_hi; ++u)
            if (fn(u)) return;
    };
    const int T = p.T, B = p.B, S = f.splits;
    int *s_par = f.scratch + (size_t)blockIdx.x * kSideScratchInts;
    int *top = s_par + kAcceptScratchInts;
    int *path = top + kMaxTree;
    float *s_lse = reinterpret_cast<float *>(path + kMaxTree);
    float *s_ent = s_lse + kMaxTree;
    const int chunks = f.row_bytes >> 4;
    for (int b = 0; b < B; ++b) {
        const bool designated = (b % (int)gridDim.x) == (int)blockIdx.x;
        bool has_unit = false;
        owns_first_tile([&](int u) {
            has_unit = ((u / p.n_qb / p.H) % B) == b && u % p.n_qb == 0;
            return has_unit;
        });
        if (!designated && !has_unit) continue;
        if (!have_all) {
            if (!side_wait_all(p, tag, lane, abort_flag)) return;
            have_all = true;
        }
        // node r's top-1 token from its partials (with typical acceptance also its
        // log-sum-exp and entropy)
        auto row_top = [&](int r, float &lse_r, float &ent_r) {
            const size_t base = ((size_t)b * T + r) * S;
            float bv = -INFINITY;
            int bi = INT_MAX;
            if ((S & 3) == 0) {
                // 16-byte loads, up to 16 partials in flight (the arrays are 256-byte
                // aligned and a row's partials start at a multiple of 4)
                const float4 *v4 = reinterpret_cast<const float4 *>(f.part_val + base);
                const int4 *i4 = reinterpret_cast<const int4 *>(f.part_idx + base);
                for (int k0 = 0; k0 < S / 4; k0 += 4) {
                    float4 v[4];
                    int4 ix[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (k0 + j < S / 4) {
                            v[j] = __ldcg(v4 + k0 + j);
                            ix[j] = __ldcg(i4 + k0 + j);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (k0 + j < S / 4) {
                            consider(v[j].x, ix[j].x, bv, bi);
                            consider(v[j].y, ix[j].y, bv, bi);
                            consider(v[j].z, ix[j].z, bv, bi);
                            consider(v[j].w, ix[j].w, bv, bi);
                        }
                    }
                }
            } else {
#pragma unroll 8
                for (int k = 0; k < S; ++k) consider(__ldcg(f.part_val + base + k), __ldcg(f.part_idx + base + k), bv, bi);
            }
            if (f.typical) stats_finish(combine_stats(f.part_stats, (int64_t)b * T + r, S), lse_r, ent_r);
            return bi;
        };
        const int32_t *par_b = p.parent + (size_t)b * T;
        const int32_t *tok_b = f.cand_tokens + (size_t)b * T;
        const int P = ld_input(p.prefix_len + b);
        AcceptResult res;
        // the accepted path: in registers (lane j % 32, slot j / 32) for trees of up
        // to 64 nodes, else in the scratch
        int path_r[2] = {-1, -1};
        constexpr bool small = kSmallTree;   // the key-row kernel's trees: T <= 64
        if constexpr (small) {
            int top_r[2] = {0, 0};
            float lse_r[2] = {0.f, 0.f}, ent_r[2] = {0.f, 0.f};
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int r = lane + 32 * k;
                if (r < T) {
                    top_r[k] = row_top(r, lse_r[k], ent_r[k]);
                    if (designated) f.argmax_out[(size_t)b * T + r] = top_r[k];
                }
            }
            if (f.typical) {
                const float *x = f.logits + (size_t)b * T * f.V;
                res = accept_warp_small(
                    top_r,
                    [&](int, int pa, int tk) {
                        const float pt = expf(ld_input(x + (size_t)pa * f.V + tk) * f.inv_temp - node_value(lse_r, pa));
                        return pt > fminf(f.epsilon, f.delta * expf(-node_value(ent_r, pa)));
                    },
                    par_b, tok_b, P, T, f.V, p.S_max, lane, path_r);
            } else {
                res = accept_warp_small(
                    top_r, [&](int, int pa, int tk) { return tk == node_value(top_r, pa); }, par_b, tok_b, P,
                    T, f.V, p.S_max, lane, path_r);
            }
            if (designated) {
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if (lane + 32 * k < T) f.path[(size_t)b * T + lane + 32 * k] = path_r[k];
            }
        } else {
            for (int r = lane; r < T; r += 32) {
                top[r] = row_top(r, s_lse[r], s_ent[r]);
                if (designated) f.argmax_out[(size_t)b * T + r] = top[r];
            }
            __syncwarp();
            const auto top_of = [&](int n) { return top[n]; };
            res = f.typical
                      ? accept_warp_typical(top_of, f.logits + (size_t)b * T * f.V,
                                            [&](int n) { return s_lse[n]; }, [&](int n) { return s_ent[n]; },
                                            f.inv_temp, f.epsilon, f.delta, par_b, tok_b, P, T, f.V, p.S_max,
                                            lane, s_par, path)
                      : accept_warp(top_of, par_b, tok_b, P, T, f.V, p.S_max, lane, s_par, path);
            if (designated)
                for (int i = lane; i < T; i += 32) f.path[(size_t)b * T + i] = path[i];
        }
        if (designated && lane == 0) {
            f.accept_len[b] = res.n_acc;
            f.next_token[b] = res.next_token;
            f.new_prefix_len[b] = res.new_prefix_len;
            atomicMax(f.status + b, res.status);
        }
        if (has_unit && res.n_acc > 0) {
            // cache rows [P_b, P_b + n_acc) <- the accepted tree rows
            const int n = res.n_acc;
            // each slice once: by the CTA holding the first tile of its first query block
            owns_first_tile([&](int u) {
                const int lbh = u / p.n_qb;
                if (u % p.n_qb != 0 || ((lbh / p.H) % B) != b) return false;
                // four 16-byte pieces of K and of V per lane loaded before any is
                // stored, so a slice's rows cost one round trip
                for (int w0 = 0; w0 < n * chunks; w0 += 4 * 32) {
                    uint4 kx[4], vx[4];
                    size_t dof[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int w = w0 + u * 32 + lane;
                        const bool in = w < n * chunks;
                        const int j = in ? w / chunks : 0, c = w - j * chunks;
                        const int src = small ? node_value(path_r, j) : (in ? path[j] : 0);
                        if (in) {
                            const size_t so = ((size_t)lbh * T + src) * f.row_bytes + (size_t)c * 16;
                            dof[u] = ((size_t)lbh * p.S_max + P + j) * f.row_bytes + (size_t)c * 16;
                            kx[u] = ld_input(reinterpret_cast<const uint4 *>(f.k_tree + so));
                            vx[u] = ld_input(reinterpret_cast<const uint4 *>(f.v_tree + so));
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (w0 + u * 32 + lane < n * chunks) {
                            *reinterpret_cast<uint4 *>(f.k_cache + dof[u]) = kx[u];
                            *reinterpret_cast<uint4 *>(f.v_cache + dof[u]) = vx[u];
                        }
                    }
                }
                return false;
            });
        }
        __syncwarp();
    }
}

// Launch one of the persistent attention kernels: one CTA per SM (at most one
// per unit, or with the work split at most one per tile and kSplitMaxGrid) of
// `threads` threads, `smem` bytes of dynamic shared memory, with programmatic
// stream serialization when asked, and as a cooperative launch (all CTAs
// resident at once, or the launch fails) when the fused step's side warps
// compute the argmax in-grid.  The shared-memory opt-in is set once per
// device.
template <class Kern>
cudaError_t launch_attention_grid(Kern kern, uint32_t smem, int threads,
                                  std::atomic<uint64_t> &configured,
                                  const AttnMaps &m, const AttnParams &p, int num_sms,
                                  bool programmatic, cudaStream_t stream)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? (1ull << dev) : 0ull;
    if (!bit || !(configured.load(std::memory_order_acquire) & bit)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit, std::memory_order_acq_rel);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)attention_grid(p, num_sms));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[3];
    unsigned n_attr = 0;
    if (p.cluster > 1) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = (unsigned)p.cluster;
        attr[n_attr].val.clusterDim.y = 1;
        attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    if (programmatic) {
        attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
        ++n_attr;
    }
    if (p.fused && p.fs.in_grid) {
        // the side warps wait for one another's flags: every CTA must be resident
        attr[n_attr].id = cudaLaunchAttributeCooperative;
        attr[n_attr].val.cooperative = 1;
        ++n_attr;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n_attr;
    return cudaLaunchKernelEx(&cfg, kern, m.q, m.kc, m.vc, m.kt, m.vt, p);
}

}  // namespace ppd

