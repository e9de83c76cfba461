"""Every plan of the attention inside the fused step, steps of more than 64 sequences
with attention grids that are over long before the acceptance, chains of programmatic
launches replayed from CUDA graphs, and outputs that allow no wide stores, against the
fp64 oracle.  Each case states the plan it is meant for, so that it cannot move to
another one unnoticed."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_18628_gb300 import ppd
from paper_2405_18628_gb300 import workloads as W

from test_gpu_fused_modes import _check, _form, _inputs, _ref, _run
from test_gpu_parity import assert_attn_close, i32, run_attention, tensors
from test_gpu_typical import DELTA, EPS, TEMP, _margins_clear

pytestmark = pytest.mark.gpu

SPLIT, WHOLE, PAIRS = 1, 0, 16


def _plan(w, workspace=True, one_grid=False):
    return ppd.ppd_attention_plan(w.L, w.B, w.H, w.T, w.D, w.S_max, workspace, one_grid)


def _wl(seed, L, B, H, D, P, T, V, **kw):
    base = dict(n_cand=max(1, (T + 3) // 4), max_depth=5, chains="fill3", match_rate=0.7, seed=seed)
    base.update(kw)
    return W.Workload("plans", L=L, B=B, H=H, D=D, P=P, T=T, V=V, **base)


# ----------------------------------------------------------------------------- plans of the fused step

# workload, prefix lengths, the plan with an argmax grid first (form 1) and with the argmax
# in the attention grid (form 2, which rules clusters out)
FUSED = {
    # 80 slices: no cluster fits, the key tiles are shared out and merged by a grid
    "split_keyrow": (_wl(601, 1, 2, 40, 64, 2000, 40, 301), [2000, 1900], SPLIT, SPLIT),
    "split_rows": (_wl(602, 1, 2, 40, 64, 3000, 100, 248), [3000, 1411], SPLIT, SPLIT),
    # few slices: clusters; without them 25 parts a slice, fewer tiles than SMs (SMs with
    # none), several query blocks and parts of tree tiles alone
    "cluster_keyrow": (_wl(603, 1, 1, 30, 128, 832, 64, 1000), [787], 4, WHOLE),
    "cluster_rows": (_wl(604, 1, 2, 9, 128, 1308, 100, 248), [1308, 513], 6, SPLIT),
    "two_slices": (_wl(610, 1, 1, 2, 128, 3000, 64, 500), [3000], 7, SPLIT),
    "few_tiles": (_wl(611, 1, 2, 3, 128, 4056, 40, 300), [100, 5], 7, SPLIT),
    "few_tiles_t200": (_wl(612, 1, 2, 1, 128, 900, 200, 120), [900, 33], 6, SPLIT),
    "few_tiles_t512": (_wl(613, 1, 1, 1, 64, 300, 512, 100), [300], 6, SPLIT),
    # one sequence, more slices than SMs: pairs of query blocks; 285 tokens run pairs and
    # third blocks in two groups of SMs
    "pairs_t200": (_wl(605, 1, 1, 160, 64, 300, 200, 248), [300], PAIRS, PAIRS),
    "pairs_t285": (_wl(606, 1, 1, 160, 64, 300, 285, 192), [257], PAIRS, PAIRS),
    "pairs_t400": (_wl(607, 1, 1, 160, 64, 140, 400, 120), [140], PAIRS, PAIRS),
    # the same of two sequences of different lengths
    "ragged_pairs_t285": (_wl(608, 1, 2, 80, 64, 300, 285, 192), [300, 100], PAIRS, PAIRS),
    # single blocks, one sequence
    "whole_t100": (_wl(609, 1, 1, 160, 64, 300, 100, 248), [300], WHOLE, WHOLE),
}


@pytest.mark.parametrize("fused_form", [1, 2])
@pytest.mark.parametrize("case", sorted(FUSED))
def test_fused_step_of_every_plan(cuda_device, case, fused_form):
    w, pl, *plans = FUSED[case]
    plan = plans[fused_form - 1]
    assert _plan(w, one_grid=fused_form == 2) == plan
    prev = ppd.ppd_set_verify_step_form(fused_form)
    try:
        assert _form(w) == fused_form
        # the merge grid of the work split is one launch more
        assert ppd.ppd_verify_step_launches(w.L, w.B, w.H, w.T, w.D, w.V, w.S_max) == 2 + (plan == SPLIT)
        s, t = _inputs(w, pl)
        g, bufs = _run(w, s, t, cuda_device)
    finally:
        ppd.ppd_set_verify_step_form(prev)
    ref = _ref(s, t)
    _check(w, s, t, g, bufs, ref, f"{case} form {fused_form}")
    assert (ref["accept_len"] >= 1).all()


# ----------------------------------------------------------------------------- clusters of every size

@pytest.mark.parametrize("T,D", [(40, 64), (64, 128), (100, 64), (128, 128)])
@pytest.mark.parametrize("size,slices,tiles", [(2, 60, 9), (3, 40, 9), (4, 30, 8), (5, 24, 10), (6, 18, 12),
                                               (7, 12, 14), (8, 10, 16)])
def test_clusters_of_every_size(cuda_device, size, slices, tiles, T, D):
    """One call of `slices` slices whose cache holds `tiles` tiles with the tree's, both
    kernels; one sequence fills its cache but for the tree, the other leaves some of its
    cluster's CTAs without tiles."""
    P = 128 * (tiles - 1) - T
    w = _wl(681 + size, 1, 2, slices // 2, D, P, T, 16)
    assert _plan(w) == _plan(w, workspace=False) == size
    pl = np.asarray([P, 129], np.int32)
    s = W.make_step_inputs(w, prefix_len=pl)
    t = tensors(w, prefix_len=pl)
    out, lse, st = run_attention({k: v.to(cuda_device) for k, v in t.items()}, pl, s.parent, cuda_device)
    ref, ref_lse, _, _ = oracle.tree_attention(t["q"], t["k_cache"], t["v_cache"], t["k_tree"], t["v_tree"], pl,
                                               s.parent)
    assert (st == 0).all()
    assert_attn_close(out.cpu().numpy().reshape(ref.shape), ref, f"clusters of {size}")
    np.testing.assert_allclose(lse.cpu().numpy().reshape(ref_lse.shape), ref_lse, rtol=0, atol=1e-3)


# ----------------------------------------------------------------------------- more than 64 sequences

LARGE = {
    # logits that outweigh a tiny attention by far: its grid is done long before the
    # acceptance, and the compaction must wait for both
    "keyrow": (_wl(621, 1, 70, 1, 64, 3, 16, 32000, max_depth=3), False),
    "keyrow_typical": (_wl(622, 1, 66, 2, 128, 5, 33, 8000), True),
    "rows": (_wl(623, 1, 66, 1, 64, 4, 100, 8000), False),
    "keyrow_f32": (_wl(624, 1, 65, 1, 64, 3, 16, 20000, max_depth=3, dtype="f32"), False),
    "rows_f32": (_wl(625, 1, 65, 1, 64, 2, 70, 4000, dtype="f32"), False),
}


class _Step:
    """A step of more than 64 sequences with its buffers, run as often as asked."""

    def __init__(self, w, typical, seed, dev):
        self.w, self.typical, self.dev = w, typical, dev
        self.pl = np.random.default_rng(w.seed).integers(0, w.P + 1, size=w.B).astype(np.int32)
        self.s, self.t = _inputs(w, self.pl, seed=seed)
        if typical:
            # guesses, thresholds and logits apart by more than rounding: taken seed by seed
            while not _margins_clear(self.ref()):
                seed += 1
                self.s, self.t = _inputs(w, self.pl, seed=seed)
        self.g = {k: v.to(dev) for k, v in self.t.items()}
        self.pre, self.par = i32(self.s.prefix_len, dev), i32(self.s.parent, dev)
        self.cand, self.logits = i32(self.s.cand_tokens, dev), torch.from_numpy(self.s.logits).to(dev)
        dt = ppd.PPD_F32 if w.dtype == "f32" else ppd.PPD_BF16
        self.bufs = ppd.StepBuffers(w.L, w.B, w.H, w.T, w.D, w.V, w.S_max, dt, device=dev, with_lse=True)

    def ref(self):
        args = (self.t["q"], self.t["k_cache"], self.t["v_cache"], self.t["k_tree"], self.t["v_tree"],
                self.s.prefix_len, self.s.parent, self.s.cand_tokens, self.s.logits)
        if self.typical:
            return oracle.verify_step_typical(*args, TEMP, EPS, DELTA)
        return oracle.verify_step(*args)

    def enqueue(self, stream=None):
        g, b = self.g, self.bufs
        args = (g["q"], g["k_cache"], g["v_cache"], g["k_tree"], g["v_tree"], self.pre, self.par, self.cand,
                self.logits)
        outs = (b.out, b.argmax, b.accept_len, b.path, b.next_token, b.new_prefix_len, b.dev_status, b.workspace)
        if self.typical:
            ppd.ppd_verify_step_typical(*args, TEMP, EPS, DELTA, *outs, lse=b.lse, stream=stream)
        else:
            ppd.ppd_verify_step(*args, *outs, lse=b.lse, stream=stream)

    def reset(self):
        """Caches as given, and outputs of no earlier call in the buffers."""
        for k in ("k_cache", "v_cache"):
            self.g[k].copy_(self.t[k])
        b = self.bufs
        b.out.fill_(float("nan"))
        for k in ("argmax", "accept_len", "path", "next_token", "new_prefix_len", "dev_status"):
            getattr(b, k).fill_(-99)

    def check(self, ref, what):
        b = self.bufs
        assert_attn_close(b.out.cpu().numpy().reshape(ref["out"].shape), ref["out"], what)
        np.testing.assert_array_equal(b.argmax.cpu().numpy(), ref["argmax"], err_msg=what)
        for k in ("accept_len", "path", "next_token", "new_prefix_len"):
            np.testing.assert_array_equal(getattr(b, k).cpu().numpy(), ref[k], err_msg=f"{what} {k}")
        np.testing.assert_array_equal(b.dev_status.cpu().numpy(), ref["status"], err_msg=what)
        bits = torch.int16 if self.w.dtype == "bf16" else torch.int32
        for k in ("k_cache", "v_cache"):
            got = self.g[k].cpu().view(bits).numpy()
            np.testing.assert_array_equal(got, ref[k].view(got.dtype), err_msg=f"{what} {k}")


def _capture(fn):
    """A CUDA graph of what fn(stream) enqueues."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        fn(side)                                  # warm-up outside the capture
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        fn(side)
    torch.cuda.synchronize()
    return graph


@pytest.mark.parametrize("case", sorted(LARGE))
def test_large_batch_compaction_waits_for_the_acceptance(cuda_device, case):
    w, typical = LARGE[case]
    assert _form(w) == 0
    st = _Step(w, typical, w.seed, cuda_device)
    ref = st.ref()
    assert (ref["accept_len"] >= 1).all() and (ref["accept_len"] > 1).any()
    st.reset()
    torch.cuda.synchronize()
    st.enqueue()
    torch.cuda.synchronize()
    st.check(ref, f"{case} in a stream")
    graph = _capture(st.enqueue)
    for rep in range(3):
        st.reset()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        st.check(ref, f"{case} replay {rep}")


# ----------------------------------------------------------------------------- a decode loop in a graph

@pytest.mark.parametrize("B,H,D,T,V", [(2, 8, 64, 48, 8192),      # clusters, key-row kernel
                                       (3, 4, 128, 96, 4001),     # clusters, query-row kernel, scalar loads
                                       (2, 90, 64, 32, 2048)])    # whole slices, ragged lengths
def test_chain_of_two_steps_replayed(cuda_device, B, H, D, T, V):
    """Two steps as a decode loop enqueues them, in one CUDA graph: the attention layer by
    layer, top-1 tokens, acceptance, compaction and the next tree, then the attention of
    that tree over the grown cache with the new prefix lengths, and its acceptance and
    compaction.  Every grid after the first starts while those before it still run, and
    reads what they write.  Replays with other logits, guesses and lengths."""
    dev, L, K, n_states, S_max = cuda_device, 2, 4, 4, 700 + 2 * T
    w = _wl(641 + B, L, B, H, D, 700, T, V)
    g = torch.Generator().manual_seed(B * 1000 + T)
    mk = lambda *shape: torch.randn(shape, generator=g).bfloat16()   # noqa: E731
    qs, kts, vts = ([mk(L, B, H, T, D) for _ in range(2)] for _ in range(3))
    kc0, vc0 = mk(L, B, H, S_max, D), mk(L, B, H, S_max, D)
    tp, tr = W.make_tree_templates(n_states, T, K, np.random.default_rng(T))
    new = lambda *shape: torch.zeros(shape, dtype=torch.int32, device=dev)   # noqa: E731
    dq, dkt, dvt = ([x.to(dev) for x in xs] for xs in (qs, kts, vts))
    kc, vc = kc0.to(dev), vc0.to(dev)
    logits = [torch.zeros(B, T, V, device=dev) for _ in range(2)]
    pre = [new(B), new(B), new(B)]
    par, cand = [new(B, T), new(B, T)], [new(B, T), new(B, T)]
    out = [torch.zeros(L, B, H, T, D, device=dev) for _ in range(2)]
    top, path = [new(B, T), new(B, T)], [new(B, T), new(B, T)]
    acc, nxt = [new(B), new(B)], [new(B), new(B)]
    st_attn, st_acc, st_next, state = [new(L, B), new(L, B)], [new(B), new(B)], new(B), new(B)
    ws = ppd.workspace(1, B, H, T, D, V, S_max, device=dev)
    nws = torch.zeros(max(256, ppd.load().ppd_next_tree_workspace_bytes(B, n_states, K)), dtype=torch.uint8,
                      device=dev)
    tpd, trd = i32(tp, dev), i32(tr, dev)

    def enqueue(stream):
        for i in range(2):
            for l in range(L):
                sl = slice(l, l + 1)
                ppd.ppd_tree_attention(dq[i][sl], kc[sl], vc[sl], dkt[i][sl], dvt[i][sl], pre[i], par[i], out[i][sl],
                                       st_attn[i][l], workspace=ws, stream=stream)
            ppd.ppd_node_argmax(logits[i], top[i], ws, stream=stream)
            ppd.ppd_accept_path(top[i], cand[i], par[i], pre[i], V, S_max, acc[i], path[i], nxt[i], pre[i + 1],
                                st_acc[i], stream=stream)
            ppd.ppd_kv_compact(kc, vc, dkt[i], dvt[i], path[i], acc[i], pre[i], stream=stream)
            if i == 0:
                ppd.ppd_next_tree(logits[0], par[0], cand[0], path[0], acc[0], nxt[0], tpd, trd, K, par[1], cand[1],
                                  state, st_next, workspace=nws, stream=stream)

    def fill(seed):
        """Host inputs and the oracle's results of both steps."""
        pl = np.random.default_rng(seed).integers(1, 701, size=B).astype(np.int32)
        s = W.make_step_inputs(w, seed=seed, prefix_len=pl)
        x1 = W.make_step_inputs(w, seed=seed + 500).logits
        r0 = oracle.verify_step(qs[0], kc0, vc0, kts[0], vts[0], pl, s.parent, s.cand_tokens, s.logits)
        n = oracle.next_tree(s.logits, s.parent, s.cand_tokens, r0["path"], r0["accept_len"], r0["next_token"], tp, tr, K)
        assert (r0["status"] == 0).all() and (n["status"] == 0).all()
        # the second step's top tokens follow its guesses here and there
        for b in range(B):
            for i in range(1, T, 2):
                if n["next_cand"][b, i] >= 0:
                    x1[b, n["next_parent"][b, i], n["next_cand"][b, i]] = 50.0 + i
        r1 = oracle.verify_step(qs[1], _bf16(r0["k_cache"]), _bf16(r0["v_cache"]), kts[1], vts[1],
                                r0["new_prefix_len"], n["next_parent"], n["next_cand"], x1)
        kc.copy_(kc0)
        vc.copy_(vc0)
        pre[0].copy_(i32(pl, dev))
        par[0].copy_(i32(s.parent, dev))
        cand[0].copy_(i32(s.cand_tokens, dev))
        logits[0].copy_(torch.from_numpy(s.logits))
        logits[1].copy_(torch.from_numpy(x1))
        for x in (*top, *path, *acc, *nxt, pre[1], pre[2], par[1], cand[1], *st_attn, *st_acc, st_next, state):
            x.fill_(-7)
        return r0, n, r1

    fill(1)
    graph = _capture(enqueue)
    deeper = 0
    for seed in (2, 3, 4):
        r0, n, r1 = fill(seed)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for i, r in enumerate((r0, r1)):
            what = f"seed {seed} step {i}"
            assert (st_attn[i] == 0).all(), what
            assert_attn_close(out[i].cpu().numpy().reshape(r["out"].shape), r["out"], what)
            for got, k in ((top[i], "argmax"), (acc[i], "accept_len"), (path[i], "path"), (nxt[i], "next_token"),
                           (pre[i + 1], "new_prefix_len"), (st_acc[i], "status")):
                np.testing.assert_array_equal(got.cpu().numpy(), r[k], err_msg=f"{what} {k}")
        for got, k in ((par[1], "next_parent"), (cand[1], "next_cand"), (state, "next_state"), (st_next, "status")):
            np.testing.assert_array_equal(got.cpu().numpy(), n[k], err_msg=f"seed {seed} {k}")
        for got, k in ((kc, "k_cache"), (vc, "v_cache")):
            np.testing.assert_array_equal(got.cpu().view(torch.int16).numpy().view(np.uint16), r1[k],
                                          err_msg=f"seed {seed} {k}")
        deeper += int((r1["accept_len"] > 1).sum())
    assert deeper > 0


def _bf16(bits):
    return torch.from_numpy(np.ascontiguousarray(bits).view(np.int16)).view(torch.bfloat16)


# ----------------------------------------------------------------------------- alignment of the output

@pytest.mark.parametrize("offset", [1, 2, 4])       # floats: 4, 8 and 16 bytes off a 512-byte boundary
@pytest.mark.parametrize("L,B,H,T,D,prefix,plan", [
    (1, 1, 10, 64, 128, [1856], 8),                  # clusters, key-row kernel
    (1, 2, 9, 100, 64, [1308, 513], 6),              # clusters, query-row kernel
    (1, 2, 40, 40, 64, [2000, 1900], SPLIT),         # the merge grid
    (1, 2, 40, 100, 64, [3000, 1411], SPLIT),        # the query-row kernel's
    (1, 1, 160, 33, 64, [129], WHOLE),               # key-row kernel
    (1, 1, 160, 100, 128, [300], WHOLE),             # single jobs
    (1, 1, 160, 200, 128, [129], PAIRS),             # pair jobs
])
def test_outputs_off_alignment(cuda_device, L, B, H, T, D, prefix, plan, offset):
    """out needs 4-byte alignment only: the wide stores of every path have a narrow form."""
    w = _wl(661 + T, L, B, H, D, max(prefix), T, 16)
    assert _plan(w) == plan
    pl = np.asarray(prefix, np.int32)
    s = W.make_step_inputs(w, prefix_len=pl)
    t = tensors(w, prefix_len=pl)
    g = {k: v.to(cuda_device) for k, v in t.items()}
    n = L * B * H * T * D
    buf = torch.full((n + 64,), float("nan"), device=cuda_device)
    assert buf.data_ptr() % 512 == 0
    out = buf[offset:offset + n].view(L, B, H, T, D)
    st = torch.full((B,), -7, dtype=torch.int32, device=cuda_device)
    ws = ppd.workspace(L, B, H, T, D, 1, w.S_max, device=cuda_device)
    ppd.ppd_tree_attention(g["q"], g["k_cache"], g["v_cache"], g["k_tree"], g["v_tree"], i32(pl, cuda_device),
                           i32(s.parent, cuda_device), out, st, workspace=ws)
    torch.cuda.synchronize()
    ref, _, _, _ = oracle.tree_attention(t["q"], t["k_cache"], t["v_cache"], t["k_tree"], t["v_tree"], pl, s.parent)
    assert (st == 0).all()
    assert_attn_close(out.cpu().numpy().reshape(ref.shape), ref, f"plan {plan} offset {offset}")
    rest = torch.cat([buf[:offset], buf[offset + n:]])
    assert torch.isnan(rest).all()                   # nothing written around it
