// ppd_kernels.h -- internal launch interface between the C-ABI layer
// (ppd_api.cu) and the kernels.  Not part of the public API.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

namespace ppd {

// A bounded device-side wait gives up after this many nanoseconds of %globaltimer.
constexpr uint64_t kWaitLimitNs = 4000000000ull;

// Tensor maps of the attention operands (bf16, 128-byte swizzle, boxes of
// 64 columns): Q [LBH][T][D] (box rows T_pad), cache K/V [LBH][S_max][D] and
// tree K/V [LBH][T][D] (box rows 128).
struct AttnMaps {
    CUtensorMap q, kc, vc, kt, vt;
};

// The fused verification step's side work (see ppd_attention_common.cuh):
// argmax partials (from the preceding grid, or with in_grid computed by the
// side warps themselves), acceptance, and compaction of the CTA's own
// (layer, sequence, head) slices.
struct FusedStep {
    float *part_val;             // [B*T*splits] partial maxima
    int32_t *part_idx;
    int splits;
    // in_grid != 0: no preceding grid; the side warps compute the partial
    // maxima themselves while the other warps stream K/V.  Chunk c of the
    // [B*T][splits] partial grid is computed by CTA c mod grid; a CTA
    // publishes ready[cta] = tag once its chunks are written, where tag =
    // *epoch + 1 read at its start.  CTA 0 waits until every flag equals tag,
    // then sets *epoch = tag and *all_ready = tag; the other CTAs read
    // partials once *all_ready equals their tag.  Every call has a fresh tag,
    // so no flag needs zeroing.
    int in_grid;
    unsigned long long wait_limit_ns;   // the grid-wide wait gives up after this long
    int withhold_cta;            // diagnostics: this CTA never publishes its flag (-1: none)
    int chunk;                   // logits per chunk (multiple of 4 when vec)
    int vec;                     // 16-byte loads of the logits
    float stat_k;                // log2(e) / temperature (typical acceptance)
    unsigned long long *epoch;   // [1]
    unsigned long long *all_ready;   // [1]
    unsigned long long *ready;   // [grid]
    const int32_t *cand_tokens;  // [B,T]
    int32_t *argmax_out;         // [B,T]
    int32_t *accept_len;         // [B]
    int32_t *path;               // [B,T]
    int32_t *next_token;         // [B]
    int32_t *new_prefix_len;     // [B]
    int32_t *status;             // [B]: zeroed by the grid before (the argmax grid, or with
                                 // in_grid a one-block reset), then raised with atomicMax
    uint8_t *k_cache, *v_cache;  // raw cache storage
    const uint8_t *k_tree, *v_tree;
    int row_bytes;               // D * element size
    int V;
    int *scratch;                // [grid][kSideScratchInts] per-CTA scratch of the side warp
    // typical acceptance (typical != 0): partial softmax statistics from the
    // preceding grid, the logits for p(token), and the rule's parameters
    int typical;
    float *part_stats;           // [B*T*splits][3]
    const float *logits;         // [B,T,V]
    float inv_temp, epsilon, delta;
};

// Largest tree (nodes) of the verification step, and the per-warp scratch
// that acceptance needs: parents, then one 32-bit word per 32 nodes of pass bits.
constexpr int kMaxTree = 512;
constexpr int kAcceptScratchInts = kMaxTree + kMaxTree / 32;

// Per-CTA scratch of the fused step's side warp: acceptance scratch, top-1
// tokens, path, and (typical acceptance) each node's log-sum-exp and entropy.
constexpr int kSideScratchInts = kAcceptScratchInts + 4 * kMaxTree + 8;

struct AttnParams {
    const int32_t *prefix_len;  // [B]
    const int32_t *parent;      // [B,T]
    float *out;                 // [L,B,H,T,D]
    float *lse;                 // [L,B,H,T] or null
    int32_t *dev_status;        // [B] or null (main-loop errors; null in the fused step)
    int L, B, H, T, T_pad, S_max, n_units;
    int n_qb;                   // query blocks of 128 per (layer, sequence, head) slice
    int n_tt;                   // tree-key tiles of 128 per slice
    int pairs;                  // query-row kernel: two blocks of queries of a slice are one job
    int pair_grid;              // with n_qb 3: the CTAs that take the slices' pairs
    float scale_log2;           // softmax scale * log2(e)
    // Work split: split != 0 shares all units out by their key tiles (launches with
    // fewer units than CTAs, B <= kSplitMaxB); units cut by a range
    // boundary leave partial softmax states in split_part, merged afterwards by
    // launch_split_merge from the per-CTA records in split_rec.
    int split;
    float *split_part;          // [2 * grid][kSplitRows * (D + 2)] partial states
    struct SplitRecord *split_rec;   // [grid]
    // Cluster split: cluster > 1 gives every unit a cluster of that many CTAs, each an
    // equal share of its tiles; their partial states are merged through distributed
    // shared memory.
    int cluster;
    int set_status;             // the attention grid writes every sequence's dev_status itself
    int fused;                  // run the end phase below
    FusedStep fs;
    // Launched as a programmatic dependent of the preceding grid (a chain of
    // ppd_tree_attention calls): the setup that reads no input overlaps that
    // grid, then every thread waits for it before reading any input.
    int pdl_wait;
    // Launched as a programmatic dependent of grids whose results it does not read
    // (a step of more than 64 sequences): a spare warp waits for them, so that this
    // grid's completion says that they are complete too.
    int late_wait;
};

// Work split limits: batch size (the per-CTA range search holds the batch in
// two warp-wide registers), CTAs, and query rows of a partial state.
constexpr int kSplitMaxB = 64;
constexpr int kSplitMaxGrid = 256;
constexpr int kSplitRows = 128;

// CTAs of a cluster at most (the portable size).
constexpr int kMaxCluster = 8;

// Clusters of `size` attention CTAs (one per SM) the current device can hold at
// once; 0 when it cannot be asked.
int max_attention_clusters(int size);

// A number >= 0 asked for once: kept in `slot` (plus one; 0: not known yet).  An `ask`
// that fails (a negative answer) counts as 0 this time and is asked again the next.
template <class Ask>
inline int asked_once(std::atomic<int> &slot, Ask ask)
{
    const int got = slot.load(std::memory_order_relaxed);
    if (got > 0) return got - 1;
    const int n = ask();
    if (n < 0) return 0;
    slot.store(n + 1, std::memory_order_relaxed);
    return n;
}

// The unit a CTA has to have merged: it holds the unit's first tile and its
// range ends inside the unit (u = -1: none).  off: the unit's tile 0 among
// the launch's tiles; n_shared: their number.
struct SplitRecord {
    long long off, n_shared;
    int u, n_tiles;
};

// Jobs of a launch without a split: its units, or with p.pairs (n_qb 2 to 4)
// one, two -- a pair and a single block -- and two jobs a slice.
inline long long whole_jobs(const AttnParams &p)
{
    if (!p.pairs) return p.n_units;
    const long long slices = p.n_units / p.n_qb;
    return p.n_qb == 2 ? slices : 2 * slices;
}

// Whether the query-row kernel's whole jobs are pairs of query blocks, and for
// n_qb 3 the split of the CTAs between pairs and single blocks: the choice with
// the shortest longest queue.  A pair counts as 2 n + 4 and a single block next
// to it as n + 4.5 tiles of 128 x 128 with n prefix tiles (S_max standing in for
// the device-side prefix lengths): three tree tiles each, and the end of a job,
// which only a pair's other stream overlaps.  Without pairs every block streams
// its keys itself: 15 % more a tile (L2), but twice the jobs, so it is the
// choice for launches with few slices (16 x 32 calls of 32 slices, 285 tokens
// over 1500 keys: pairs 36.6 us a call, single blocks 30.1).
inline void plan_rows(AttnParams &p, int num_sms)
{
    p.pairs = 0;
    if (p.T_pad <= 64 || p.n_qb < 2) return;
    const long long S = p.n_units / p.n_qb, G = num_sms, n = (p.S_max + 127) / 128;
    const long long single_all = (23 * (2 * n + 9)) * ((p.n_units + G - 1) / G);   // in 1/40 tiles
    long long best = -1;
    int grid = 0;
    if (p.n_qb == 3) {
        const long long Gp = G < 2 * S ? G : 2 * S;
        for (long long g = 1; g < Gp; ++g) {
            const long long a = (4 * n + 8) * ((S + g - 1) / g), b = (2 * n + 9) * ((S + Gp - g - 1) / (Gp - g));
            const long long t = a > b ? a : b;
            if (best < 0 || t <= best) {
                best = t;
                grid = (int)g;
            }
        }
    } else {
        const long long jobs = p.n_qb == 2 ? S : 2 * S;
        best = (4 * n + 8) * ((jobs + G - 1) / G);
    }
    if (best < 0 || 20 * best > single_all) return;
    p.pairs = 1;
    p.pair_grid = grid;
}

// Whether the launch takes whole jobs of several sequences, whose lengths (known
// to the device alone) may differ.
inline bool whole_ragged(const AttnParams &p)
{
    return p.B > 1 && p.B <= kSplitMaxB && !p.split && p.cluster <= 1;
}

// CTAs of an attention launch: one per SM, at most one per job (with the
// work split: at most one per tile, and kSplitMaxGrid).
inline int attention_grid(const AttnParams &p, int num_sms)
{
    long long grid = num_sms;
    if (p.cluster > 1) return p.n_units * p.cluster;
    if (p.split) {
        const long long max_tiles = (long long)p.n_units * ((p.S_max + 127) / 128 + p.n_tt);
        grid = grid < kSplitMaxGrid ? grid : kSplitMaxGrid;
        grid = grid < max_tiles ? grid : max_tiles;
    } else {
        const long long jobs = whole_jobs(p);
        grid = grid < jobs ? grid : jobs;
    }
    return (int)grid;
}

// Merge the partial states of every cut unit of the attention launch just
// enqueued (one CTA per attention CTA, `grid` of them), after it completes.
cudaError_t launch_split_merge(const AttnParams &p, int D, int grid, cudaStream_t stream);

// Batches up to this size run the fused step (one grid, or an argmax grid then
// the attention grid).
constexpr int kFusedMaxB = 64;

// Dispatches on the padded tree size: up to 64 tokens the key-row kernel
// (ppd_attention.cu), 65..512 the query-row kernel (ppd_attention_rows.cu).
cudaError_t launch_tree_attention(const AttnMaps &m, const AttnParams &p, int D, int num_sms,
                                  bool programmatic, cudaStream_t stream);
cudaError_t launch_tree_attention_rows(const AttnMaps &m, const AttnParams &p, int D, int num_sms,
                                       bool programmatic, cudaStream_t stream);

// A kernel launch as a programmatic dependent of the stream's previous grid (it
// may start before that grid completes; the kernel waits with pdl_wait()), in
// clusters of `cluster` (1 1 1: none).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(void (*kern)(KArgs...), dim3 grid, dim3 block, dim3 cluster,
                                  cudaStream_t stream, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 1;
    if (cluster.x * cluster.y * cluster.z > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = cluster.x;
        attr[1].val.clusterDim.y = cluster.y;
        attr[1].val.clusterDim.z = cluster.z;
        cfg.numAttrs = 2;
    }
    cfg.attrs = attr;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// Splits per node row of the argmax: about 512 blocks over all rows, chunks of
// at least 2048 logits, at most 64 splits.
inline int argmax_split_count(int64_t rows, int V)
{
    if (rows <= 0) return 1;
    int64_t want = (512 + rows - 1) / rows;
    int64_t cap = V / 2048;
    if (cap > 64) cap = 64;
    if (cap < 1) cap = 1;
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    return (int)want;
}

// Node argmax in two steps: per-(row, split) partial maxima, then a combine.
// part_stats (3 floats per partial) non-null: also the softmax statistics at
// `temperature` (typical acceptance).
cudaError_t launch_argmax_partials(const float *logits, int64_t rows, int V, int splits,
                                   float *part_val, int32_t *part_idx, float *part_stats,
                                   float temperature, int32_t *zero_status, int n_zero,
                                   cudaStream_t stream);
// The same partials from `grid` blocks of 512 threads (one warp per chunk at a
// time): the fused step's argmax grid on the SMs of its attention grid's last,
// partial round.
cudaError_t launch_argmax_narrow(const float *logits, int64_t rows, int V, int splits, int grid,
                                 float *part_val, int32_t *part_idx, float *part_stats,
                                 float temperature, int32_t *zero_status, int n_zero,
                                 cudaStream_t stream);
cudaError_t launch_argmax_combine(const float *part_val, const int32_t *part_idx, int64_t rows,
                                  int splits, int32_t *argmax_out, cudaStream_t stream);

struct AcceptArgs {
    const int32_t *cand_tokens;  // [B,T]
    const int32_t *parent;       // [B,T]
    const int32_t *prefix_len;   // [B]
    int32_t *accept_len;         // [B]
    int32_t *path;               // [B,T]
    int32_t *next_token;         // [B]
    int32_t *new_prefix_len;     // [B]
    int32_t *dev_status;         // [B]
    int T, V, S_max;
};

cudaError_t launch_accept_path(const int32_t *argmax, const AcceptArgs &a, int B,
                               cudaStream_t stream);

// Node argmax in one grid, a cluster of CTAs per row; with lse_out also the
// natural-log log-sum-exp and entropy of softmax(row / temperature).
cudaError_t launch_node_argmax(const float *logits, int64_t rows, int V, float temperature,
                               int32_t *argmax_out, float *lse_out, float *ent_out, cudaStream_t stream);

// argmax, natural-log log-sum-exp and entropy per row from stats partials.
cudaError_t launch_node_stats_combine(const float *part_val, const int32_t *part_idx,
                                      const float *part_stats, int64_t rows, int splits,
                                      int32_t *argmax_out, float *lse_out, float *ent_out,
                                      cudaStream_t stream);

cudaError_t launch_typical_accept(const float *logits, const float *lse, const float *ent,
                                  const int32_t *argmax, const AcceptArgs &a, int B,
                                  float temperature, float epsilon, float delta,
                                  cudaStream_t stream);

// chained: as a programmatic dependent of the stream's previous grid.
cudaError_t launch_kv_compact(void *k_cache, void *v_cache, const void *k_tree,
                              const void *v_tree, const int32_t *path,
                              const int32_t *accept_len, const int32_t *prefix_len, int L,
                              int B, int H, int T, int D, int S_max, int elem_bytes,
                              cudaStream_t stream, bool chained = true);

// Next-step candidate tree: at most this many guesses per depth.
constexpr int kNextMaxK = 16;
constexpr int kNextMaxEpt = 128;
constexpr int kNextMaxSplit = 8;    // CTAs (a cluster) sharing one row's columns

cudaError_t launch_next_tree(const float *logits, const int32_t *parent, const int32_t *cand,
                             const int32_t *path, const int32_t *accept_len,
                             const int32_t *next_token, int B, int T, int V, int n_states,
                             int T_next, const int32_t *tmpl_parent, const int32_t *tmpl_rank, int K,
                             int n_ept, int ept_mean, int32_t *topk, int32_t *kstate, float *lse,
                             int num_sms, int32_t *next_parent, int32_t *next_cand,
                             int32_t *next_state, int32_t *status, cudaStream_t stream);

// fp32 -> bf16 copies (round to nearest even) of n tensors [lbh][rows][D]; of a
// `cache` tensor only the rows below the sequence's prefix length.  chained: as
// a programmatic dependent of the stream's previous grid.
struct RoundArgs {
    struct Tensor {
        const float *src;
        uint16_t *dst;
        int rows;
        int cache;
    } t[5];
    const int32_t *prefix_len;
    int n, B, H, D;
};
cudaError_t launch_round_bf16(const RoundArgs &r, int64_t lbh, bool chained, cudaStream_t stream);

// Zero `n` status words once the preceding grid has completed, as a
// programmatic dependent launch that lets the next grid launch at once.
cudaError_t launch_zero_status(int32_t *status, int n, cudaStream_t stream);

cudaError_t launch_selftest_umma(const CUtensorMap &ma, const CUtensorMap &mb, const void *a_raw,
                                 const void *b_raw, float *d, int mode, int N, cudaStream_t stream);

}  // namespace ppd
