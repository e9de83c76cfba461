// ppd_next.cu -- next-step candidate tree of the PPD decode loop (paper
// Section 3 step (1): the prompt tokens appended to a guess token predict the
// tokens that follow it; Section 3, Ensemble Prompt Tokens: each prompt
// position holds n_ept tokens, the j-th seeing only the j-th of the positions
// before it, and the guess comes from the average of their logits -- or, in
// the formula the section gives, of their probabilities; Appendix,
// Definition of tree states: the next tree takes state T_k, whose candidate
// subtree is at most k deep, k being the number of prompt positions left
// below the accepted token).
//
// The log-sum-exp and top-K kernels first find, per (sequence, chain position
// d), the n_ept prompt chains below the accepted end node (find_chains: each node's
// lowest-index prompt child by a shared-memory minimum, one node per thread;
// the end node's prompt children ranked by ballots; each chain walked through
// those links).  The probability mode then takes each chain row's log-sum-exp
// (next_lse_kernel, one block a row).  next_topk_kernel ranks the averaged
// logits (or sum_j exp(x_j - lse_j), the probability mean without its 1/n_ept,
// which no ranking sees) of each row with a cluster of up to kNextMaxSplit CTAs
// and next_assemble_kernel, one block per sequence, fills the state's template
// with the root token and the guesses.
//
// All of it is latency: the rows of four sequences with four chains each are 6
// MB, about a microsecond of HBM, behind dependent loads (which rows?) and the
// selection.  Selecting costs three block barriers a batch of 8192 columns,
// whatever the values: every warp's K-th largest lane maximum (K rounds of one
// redux) is a lower bound of the K-th best, the largest of those bounds leaves
// a few dozen candidates, and a candidate's place is the number of better ones.
// Insertion into per-thread lists, with the merges of lists in grids of their
// own, took 48.2 us there (one box; 12.0 now).
#include "ppd.h"
#include "ppd_accept.cuh"
#include "ppd_device.cuh"
#include "ppd_kernels.h"

#include <climits>

namespace ppd {

constexpr int kTopkThreads = 512;                  // one tree node per thread (T <= 512)
constexpr int kTopkWarps = kTopkThreads / 32;
constexpr int kBatch = 4;                          // 16-byte loads in flight per row and thread
constexpr int kEach = 4 * kBatch;                  // columns per thread and batch
constexpr float kLog2e = 1.4426950408889634f;
static_assert(kMaxTree <= kTopkThreads, "find_chains takes one tree node per thread");

// A call's kernels form a chain of programmatic launches, and so do calls one
// after the other: each kernel waits for the previous grid before it reads an
// input.  The kernels in front of next_assemble_kernel let it start only once
// their own wait is over, so it may read the call's inputs (the template) ahead
// of its wait for their results.

// Running log-sum-exp of a row: maximum m, sum s of exp(x - m) over the finite
// entries, and whether a NaN or +inf was seen.  -inf entries add nothing and
// every exponent is a difference <= 0, so nothing overflows.
struct LseAcc {
    float m, s;
    int bad;
};

PPD_DEV void lse_add(LseAcc &a, float x)
{
    if (isnan(x) || x == INFINITY) {
        a.bad = 1;
    } else if (x > a.m) {
        a.s = a.s * exp2f((a.m - x) * kLog2e) + 1.f;
        a.m = x;
    } else if (x > -INFINITY) {
        a.s += exp2f((x - a.m) * kLog2e);
    }
}

PPD_DEV void lse_merge(LseAcc &a, float om, float os, int ob)
{
    const float nm = fmaxf(a.m, om);
    if (nm > -INFINITY)
        a.s = (a.m > -INFINITY ? a.s * exp2f((a.m - nm) * kLog2e) : 0.f) +
              (om > -INFINITY ? os * exp2f((om - nm) * kLog2e) : 0.f);
    a.m = nm;
    a.bad |= ob;
}

// Merge across the lanes of a warp (every lane ends with the total).
PPD_DEV void lse_warp(LseAcc &a)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, a.m, off);
        const float os = __shfl_xor_sync(0xffffffffu, a.s, off);
        const int ob = __shfl_xor_sync(0xffffffffu, a.bad, off);
        lse_merge(a, om, os, ob);
    }
}

// An entry of a ranking as one integer, larger = earlier: NaN first, then the
// larger value (-0 = +0), then the lower index (< 2^31).  Never 0.
PPD_DEV uint32_t rank_key(float x)
{
    if (x != x) return 0xFFFFFFFFu;
    const uint32_t u = x == 0.f ? 0u : __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
PPD_DEV unsigned long long rank_entry(uint32_t key, int i) { return (unsigned long long)key << 32 | (uint32_t)~i; }
PPD_DEV int entry_index(unsigned long long e) { return (int)~(uint32_t)e; }

// The n_ept prompt chains below sequence b's accepted end node, for chain
// position d (one block of kTopkThreads threads, T <= kTopkThreads): each
// node's lowest-index prompt child (a later node) by a shared-memory minimum,
// one node per thread; the end node's prompt children ranked by ballots; each
// chain walked through those links.  Leaves in c the chains' nodes at
// position d and the state k (0 with fewer than n_ept heads, else the
// shortest chain capped at n_states - 1); ends with a block barrier.
struct ChainSmem {
    int fc[kMaxTree];
    int head[kNextMaxEpt], len[kNextMaxEpt], node[kNextMaxEpt];
    int wcnt[kTopkWarps];
    int nh, k;
};

PPD_DEV void find_chains(ChainSmem &c, const int32_t *parent, const int32_t *cand,
                         const int32_t *path, const int32_t *accept_len, int b, int d, int T,
                         int n_states, int n_ept)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cap = n_states - 1;
    const int32_t *par = parent + (size_t)b * T;
    const int32_t *tok = cand + (size_t)b * T;
    int pa = -1, tk = 0;
    if (tid < T) {
        pa = __ldcg(par + tid);
        tk = __ldcg(tok + tid);
    }
    const int n = __ldcg(accept_len + b);
    const int e = (n >= 1 && n <= T) ? __ldcg(path + (size_t)b * T + n - 1) : -1;
    for (int i = tid; i < T; i += kTopkThreads) c.fc[i] = INT_MAX;
    __syncthreads();
    bool head = false;
    if (tid < T) {
        if (tk == -1 && pa >= 0 && pa < tid) atomicMin(c.fc + pa, tid);
        head = tk == -1 && e >= 0 && e < T && pa == e && tid > e;
    }
    const unsigned hm = __ballot_sync(0xffffffffu, head);
    if (lane == 0) c.wcnt[warp] = __popc(hm);
    __syncthreads();
    int rank = __popc(hm & ((1u << lane) - 1u));
    for (int w = 0; w < warp; ++w) rank += c.wcnt[w];
    if (head && rank < n_ept) c.head[rank] = tid;
    if (tid == 0) {
        int cnt = 0;
        for (int w = 0; w < kTopkWarps; ++w) cnt += c.wcnt[w];
        c.nh = min(cnt, n_ept);
    }
    __syncthreads();
    // each chain's length (capped) and its node at position d, one thread a chain
    if (c.nh == n_ept) {
        for (int j = tid; j < n_ept; j += kTopkThreads) {
            int cur = c.head[j], len = 1, node = d == 1 ? cur : -1;
            while (len < cap) {
                const int nx = c.fc[cur];
                if (nx == INT_MAX) break;
                cur = nx;
                ++len;
                if (len == d) node = cur;
            }
            c.len[j] = len;
            c.node[j] = node;
        }
    }
    __syncthreads();
    if (tid == 0) {
        int k = 0;
        if (c.nh == n_ept) {
            k = cap;
            for (int j = 0; j < n_ept; ++j) k = min(k, c.len[j]);
        }
        c.k = k;
    }
    __syncthreads();
}

// ln sum_v exp(x_j[v]) of chain row j = blockIdx.z at position d of sequence b
// (probability mode): an online maximum and sum per thread, merged over the
// block; NaN when the row holds a NaN or +inf, or only -inf.  Written to
// lse[(b * (n_states - 1) + d - 1) * kNextMaxEpt + j].
__global__ void __launch_bounds__(kTopkThreads)
next_lse_kernel(const float *logits, const int32_t *parent, const int32_t *cand,
                const int32_t *path, const int32_t *accept_len, int T, int V, int n_states,
                int n_ept, int vec, float *lse)
{
    __shared__ ChainSmem cs;
    __shared__ float s_m[kTopkWarps], s_s[kTopkWarps];
    __shared__ int s_b[kTopkWarps];
    const int b = blockIdx.x, d = blockIdx.y + 1, j = blockIdx.z;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_wait();
    pdl_release();
    find_chains(cs, parent, cand, path, accept_len, b, d, T, n_states, n_ept);
    if (d > cs.k) return;   // uniform over the block
    const float *x = logits + ((size_t)b * T + cs.node[j]) * V;
    LseAcc acc{-INFINITY, 0.f, 0};
    if (vec) {
        const int V4 = V >> 2;
        for (int v4 = tid; v4 < V4; v4 += kBatch * kTopkThreads) {
            float4 xs[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                xs[q] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                if (v4 + q * kTopkThreads < V4) xs[q] = ld_input(reinterpret_cast<const float4 *>(x) + v4 + q * kTopkThreads);
            }
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                lse_add(acc, xs[q].x);
                lse_add(acc, xs[q].y);
                lse_add(acc, xs[q].z);
                lse_add(acc, xs[q].w);
            }
        }
    } else {
        for (int v = tid; v < V; v += kTopkThreads) lse_add(acc, ld_input(x + v));
    }
    lse_warp(acc);
    if (lane == 0) {
        s_m[warp] = acc.m;
        s_s[warp] = acc.s;
        s_b[warp] = acc.bad;
    }
    __syncthreads();
    if (warp == 0) {
        LseAcc a{-INFINITY, 0.f, 0};
        if (lane < kTopkWarps) a = LseAcc{s_m[lane], s_s[lane], s_b[lane]};
        lse_warp(a);
        if (lane == 0)
            lse[((size_t)b * (n_states - 1) + d - 1) * kNextMaxEpt + j] =
                (a.bad || a.m == -INFINITY) ? NAN : a.m + logf(a.s);
    }
}

// Top-K (K <= kNextMaxK) of the averaged logits (ept_mean 0) or probabilities
// (ept_mean 1) at chain position d (1-based) of sequence b, in ranking order,
// into topk[(b * (n_states - 1) + d - 1) * K ...]: one cluster, CTA z taking
// columns [z * chunk, (z + 1) * chunk).  Position 1 also writes the state k of
// its sequence to kstate[b].  vec: rows may be read as float4 (chunk is then a
// multiple of 4).  kChains: ensemble chains whose loads are in flight together.
template <int kChains>
__global__ void __launch_bounds__(kTopkThreads)
next_topk_kernel(const float *logits, const int32_t *parent, const int32_t *cand,
                 const int32_t *path, const int32_t *accept_len, int T, int V, int n_states, int K,
                 int n_ept, int ept_mean, int vec, int chunk, const float *lse, int32_t *topk,
                 int32_t *kstate)
{
    // a warp has at most K lanes above its own bound, so at most this many candidates
    constexpr int kMaxCand = kTopkWarps * kNextMaxK * kEach;
    __shared__ ChainSmem cs;
    __shared__ float s_lse[kNextMaxEpt];
    __shared__ unsigned long long s_bound[kTopkWarps], s_list[2][kNextMaxK], s_cand[kMaxCand];
    __shared__ int s_n;
    const int b = blockIdx.x;
    const int d = blockIdx.y + 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    pdl_wait();   // the inputs, the log-sum-exps, and the previous call's readers of topk and kstate
    pdl_release();
    find_chains(cs, parent, cand, path, accept_len, b, d, T, n_states, n_ept);
    if (tid == 0 && d == 1 && blockIdx.z == 0) kstate[b] = cs.k;
    if (d > cs.k) return;   // uniform over the cluster
    auto row = [&](int j) { return logits + ((size_t)b * T + cs.node[j]) * V; };
    const bool probs = ept_mean == 1 && n_ept > 1;
    const int c0 = (int)blockIdx.z * chunk, c1 = min(V, c0 + chunk);   // this CTA's columns

    // ---- probability mode: the chain rows' log-sum-exps (next_lse_kernel)
    if (probs) {
        for (int j = tid; j < n_ept; j += kTopkThreads)
            s_lse[j] = __ldcg(lse + ((size_t)b * (n_states - 1) + d - 1) * kNextMaxEpt + j);
    }
    if (tid < kNextMaxK) s_list[0][tid] = 0;
    if (tid == 0) s_n = 0;
    __syncthreads();

    const float n_f = (float)n_ept;
    int cur = 0;   // the list of the batches before
    const int step = vec ? kEach * kTopkThreads : kBatch * kTopkThreads;
    for (int first = c0; first < c1; first += step) {
        // ---- this thread's columns: element e is column col(e), ascending in e
        const int base = first + (vec ? 4 * tid : tid);
        auto col = [&](int e) { return base + (vec ? (e >> 2) * 4 * kTopkThreads + (e & 3) : e * kTopkThreads); };
        float sc[kEach];
        if (vec) {
            float4 a[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q) a[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            // the EPT average is summed in chain order, then divided once (IEEE); the
            // probabilities are summed in chain order, a NaN lse_j making every score NaN
            // (the loads of kChains chains are in flight together)
            for (int j0 = 0; j0 < n_ept; j0 += kChains) {
                float4 fj[kChains][kBatch];
#pragma unroll
                for (int y = 0; y < kChains; ++y) {
                    if (j0 + y >= n_ept) break;
                    const float *x = row(j0 + y);
#pragma unroll
                    for (int q = 0; q < kBatch; ++q) {
                        fj[y][q] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (col(4 * q) < c1) fj[y][q] = __ldcs(reinterpret_cast<const float4 *>(x + col(4 * q)));
                    }
                }
#pragma unroll
                for (int y = 0; y < kChains; ++y) {
                    if (j0 + y >= n_ept) break;
                    const float l = probs ? s_lse[j0 + y] : 0.f;
#pragma unroll
                    for (int q = 0; q < kBatch; ++q) {
                        float4 f = fj[y][q];
                        if (probs) {
                            f.x = exp2f((f.x - l) * kLog2e);
                            f.y = exp2f((f.y - l) * kLog2e);
                            f.z = exp2f((f.z - l) * kLog2e);
                            f.w = exp2f((f.w - l) * kLog2e);
                        }
                        if (j0 + y == 0) {
                            a[q] = f;
                        } else {
                            a[q].x += f.x;
                            a[q].y += f.y;
                            a[q].z += f.z;
                            a[q].w += f.w;
                        }
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                sc[4 * q] = a[q].x;
                sc[4 * q + 1] = a[q].y;
                sc[4 * q + 2] = a[q].z;
                sc[4 * q + 3] = a[q].w;
            }
        } else {
#pragma unroll
            for (int e = 0; e < kEach; ++e) sc[e] = 0.f;
            for (int j = 0; j < n_ept; ++j) {
                const float *x = row(j);
                const float l = probs ? s_lse[j] : 0.f;
#pragma unroll
                for (int e = 0; e < kBatch; ++e) {
                    float f = col(e) < c1 ? __ldcs(x + col(e)) : 0.f;
                    if (probs) f = exp2f((f - l) * kLog2e);
                    sc[e] = j == 0 ? f : sc[e] + f;
                }
            }
        }
        const bool mean = !probs && n_ept > 1;
        uint32_t key[kEach];
        uint32_t bk = 0;   // the thread's best
        int bi = INT_MAX;
#pragma unroll
        for (int e = 0; e < kEach; ++e) {
            const bool live = (vec || e < kBatch) && col(e) < c1;
            key[e] = live ? rank_key(mean ? sc[e] / n_f : sc[e]) : 0u;
            if (key[e] > bk) {
                bk = key[e];
                bi = col(e);
            }
        }

        // ---- the warp's K-th best lane: at least K entries are as good
        unsigned long long bound = 0;
        for (int r = 0; r < K; ++r) {
            const uint32_t m = __reduce_max_sync(0xffffffffu, bk);
            if (m == 0) {   // fewer than K lanes hold anything
                bound = 0;
                break;
            }
            const bool top = bk == m;
            int i = bi;
            if (__popc(__ballot_sync(0xffffffffu, top)) > 1) i = __reduce_min_sync(0xffffffffu, top ? bi : INT_MAX);
            const bool win = top && bi == i;
            if (r == K - 1) bound = __shfl_sync(0xffffffffu, rank_entry(m, bi), __ffs(__ballot_sync(0xffffffffu, win)) - 1);
            if (win) bk = 0;
        }
        if (lane == 0) s_bound[warp] = bound;
        __syncthreads();
        // ---- the candidates: at least as good as every bound, better than the list's last
        unsigned long long least = s_list[cur][K - 1] + 1;
#pragma unroll
        for (int w = 0; w < kTopkWarps; ++w) least = s_bound[w] > least ? s_bound[w] : least;
        const uint32_t least_key = (uint32_t)(least >> 32);
#pragma unroll
        for (int e = 0; e < kEach; ++e) {
            if (key[e] >= least_key && key[e] != 0 && rank_entry(key[e], col(e)) >= least)
                s_cand[atomicAdd(&s_n, 1)] = rank_entry(key[e], col(e));
        }
        if (tid < kNextMaxK) s_list[cur ^ 1][tid] = 0;
        __syncthreads();
        // ---- each entry's place is the number of better ones
        const int n = s_n;
        for (int x = tid; x < n + K; x += kTopkThreads) {
            const unsigned long long mine = x < n ? s_cand[x] : s_list[cur][x - n];
            int place = 0;
            for (int y = 0; y < n; ++y) place += s_cand[y] > mine;
            for (int y = 0; y < K; ++y) place += s_list[cur][y] > mine;
            if (mine != 0 && place < K) s_list[cur ^ 1][place] = mine;
        }
        __syncthreads();
        if (tid == 0) s_n = 0;
        cur ^= 1;
    }

    // ---- the cluster's lists: CTA 0 places every entry among all of them
    if (cur == 1 && tid < K) s_list[0][tid] = s_list[1][tid];
    __syncthreads();
    cluster_sync();
    if (blockIdx.z == 0) {
        const int n = (int)gridDim.z * K;   // <= 128 entries
        unsigned long long *all = s_cand;
        if (tid < n) all[tid] = ld_cluster_u64(cluster_map(smem_addr(&s_list[0][0]) + (uint32_t)tid % K * 8, tid / K));
        __syncthreads();
        if (tid < n) {
            const unsigned long long mine = all[tid];
            int place = 0;
            for (int y = 0; y < n; ++y) place += all[y] > mine;
            if (mine != 0 && place < K)
                topk[((size_t)b * (n_states - 1) + d - 1) * K + place] = entry_index(mine);
        }
    }
    cluster_sync_exit();   // no CTA leaves while CTA 0 reads its list
}

// One block per sequence: state, template checks, and the next tree.  The
// templates (all states', when they fit) are in shared memory before the wait
// for the states and guesses.
constexpr int kAsmThreads = 256;
constexpr int kAsmEntries = 4096;

__global__ void __launch_bounds__(kAsmThreads)
next_assemble_kernel(const int32_t *path, const int32_t *accept_len, const int32_t *next_token, int T,
                     int n_states, int T_next, const int32_t *tmpl_parent, const int32_t *tmpl_rank,
                     int K, const int32_t *topk, const int32_t *kstate, int32_t *next_parent,
                     int32_t *next_cand, int32_t *next_state, int32_t *status, int early)
{
    __shared__ int16_t s_par[kAsmEntries], s_rank[kAsmEntries];   // clamped: every valid value fits
    const int b = blockIdx.x, tid = threadIdx.x;
    const int total = n_states * T_next;
    const bool all = early && total <= kAsmEntries;
    auto clamp16 = [](int v) { return (int16_t)max(-2, min(v, 32767)); };
    auto load = [&](int first, int n) {   // through L2: ahead of the wait, no earlier line of L1 will do
        for (int i = tid; i < n; i += kAsmThreads) {
            s_par[i] = clamp16(ld_relaxed_gpu_s32(tmpl_parent + first + i));
            s_rank[i] = clamp16(ld_relaxed_gpu_s32(tmpl_rank + first + i));
        }
    };
    if (!early) pdl_wait();
    pdl_release();
    if (all) load(0, total);
    if (early) pdl_wait();   // the states and the guesses (and, of a call's only grid, the inputs)
    const int n = __ldcg(accept_len + b), nt = __ldcg(next_token + b);
    bool bad = !(n >= 1 && n <= T && nt >= 0);
    int k = 0;
    if (!bad) {
        const int e = __ldcg(path + (size_t)b * T + n - 1);
        bad = !(e >= 0 && e < T);
        if (!bad && n_states > 1) k = __ldcg(kstate + b);
    }
    if (!all) load(k * T_next, T_next);
    __syncthreads();
    const int16_t *tp = s_par + (all ? k * T_next : 0), *tr = s_rank + (all ? k * T_next : 0);
    int32_t *np = next_parent + (size_t)b * T_next;
    int32_t *nc = next_cand + (size_t)b * T_next;
    // template checks: parents before their children, ranks below K
    for (int i = tid; i < T_next && !bad; i += kAsmThreads) {
        if (i == 0) bad |= tp[0] != -1;
        else bad |= tp[i] < 0 || tp[i] >= i || tr[i] >= K;
    }
    bad = __syncthreads_or(bad);
    // each candidate's depth: only candidates above it, at most k of them with itself
    int tok[2] = {-1, -1};   // T_next <= 512: two nodes a thread
    if (!bad) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int i = tid + x * kAsmThreads;
            if (i >= T_next) continue;
            if (i == 0) {
                tok[x] = nt;
            } else if (tr[i] >= 0) {
                int depth = 0;
                bool ok = true;
                for (int a = i; a > 0; a = tp[a]) {
                    ok &= tr[a] >= 0;
                    ++depth;
                }
                if (!ok || depth > k) bad = true;
                else tok[x] = __ldcg(topk + ((size_t)b * (n_states - 1) + depth - 1) * K + tr[i]);
            }
        }
    }
    bad = __syncthreads_or(bad);
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int i = tid + x * kAsmThreads;
        if (i >= T_next) continue;
        np[i] = bad ? -1 : tp[i];
        nc[i] = bad ? -1 : tok[x];
    }
    if (tid == 0) {
        next_state[b] = bad ? -1 : k;
        status[b] = bad ? kErrTree : kOk;
    }
}

cudaError_t launch_next_tree(const float *logits, const int32_t *parent, const int32_t *cand,
                             const int32_t *path, const int32_t *accept_len,
                             const int32_t *next_token, int B, int T, int V, int n_states,
                             int T_next, const int32_t *tmpl_parent, const int32_t *tmpl_rank, int K,
                             int n_ept, int ept_mean, int32_t *topk, int32_t *kstate, float *lse,
                             int num_sms, int32_t *next_parent, int32_t *next_cand,
                             int32_t *next_state, int32_t *status, cudaStream_t stream)
{
    if (n_states > 1) {
        const int vec = (V % 4 == 0) && ((reinterpret_cast<uintptr_t>(logits) & 15) == 0);
        // each row shared by a cluster, about two CTAs per SM in all, no CTA without columns
        const long long rows = (long long)B * (n_states - 1);
        int n_split = (int)((2LL * num_sms + rows - 1) / rows);
        n_split = n_split < 1 ? 1 : (n_split > kNextMaxSplit ? kNextMaxSplit : n_split);
        int chunk = (V + n_split - 1) / n_split;
        chunk = (chunk + 3) & ~3;
        n_split = (V + chunk - 1) / chunk;
        const unsigned cap = (unsigned)(n_states - 1);
        cudaError_t e;
        if (ept_mean == 1 && n_ept > 1) {
            e = launch_chained(next_lse_kernel, dim3((unsigned)B, cap, (unsigned)n_ept), dim3(kTopkThreads),
                               dim3(1), stream, logits, parent, cand, path, accept_len, T, V, n_states,
                               n_ept, vec, lse);
            if (e != cudaSuccess) return e;
        }
        // Four chains' loads in flight take 118 registers, one CTA per SM: where the grid
        // fits that way (clusters of eight find places on about 3/4 of the SMs), it hides
        // more latency (4 sequences, V 32000, 4 chains: 14.2 -> 12.2 us; 13.4 with two),
        // beyond that the second CTA is worth more (16 sequences, V 50257: 115 us with
        // four, 64.7 with two, 65.2 with one).
        auto *kern = n_ept == 1 ? next_topk_kernel<1>
                     : 4 * rows * n_split <= 3LL * num_sms ? next_topk_kernel<4> : next_topk_kernel<2>;
        e = launch_chained(kern, dim3((unsigned)B, cap, (unsigned)n_split), dim3(kTopkThreads),
                           dim3(1, 1, (unsigned)n_split), stream, logits, parent, cand, path, accept_len, T,
                           V, n_states, K, n_ept, ept_mean, vec, chunk, (const float *)lse, topk, kstate);
        if (e != cudaSuccess) return e;
    }
    return launch_chained(next_assemble_kernel, dim3((unsigned)B), dim3(kAsmThreads), dim3(1), stream, path,
                          accept_len, next_token, T, n_states, T_next, tmpl_parent, tmpl_rank, K,
                          (const int32_t *)topk, (const int32_t *)kstate, next_parent, next_cand,
                          next_state, status, n_states > 1 ? 1 : 0);
}

}  // namespace ppd
