"""GPU tests of calls at the edges of what the entry points take, each compared with the ordinary form of the same call."""
from dataclasses import replace

import numpy as np
import pytest

from synth import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _vb():
    from paper_2606_12243_b200 import binding
    return binding


def _engine(wl, **kw):
    from paper_2606_12243_b200.engine import Engine
    eng = Engine(wl, fill_context="device", **kw)
    eng.set_inputs(W.step_inputs(wl))
    return eng


def _shifted(t):
    """The same values one element off a 16-byte boundary."""
    s = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)[1:].view(t.shape).copy_(t)
    assert s.data_ptr() % 16 != 0
    return s


def _step(eng, model, cache, batch, nodes):
    vb = _vb()
    slim, full, res = eng.logits_buffer(), eng.logits_buffer(), vb.alloc_result(batch, nodes)
    vb.verify_step(model, cache, eng.draft, eng.params(), slim, full, res)
    torch.cuda.synchronize()
    assert vb.get_stats(model).device_status == 0
    return [slim, full, res.tier, res.n_acc, res.path, res.out_tok, res.n_emit, res.judge, res.corr_src]


# ---------------------------------------------------------------------------------------------
# arrays that need not be aligned beyond their element
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("name,batch,head_dim,one", [("c1_tiny", None, None, 1), ("mini_7b", None, None, 1), ("mini_7b", 8, None, 1), ("mini_7b", None, 64, 1),
                                                     ("c1_tiny", None, None, 0), ("mini_7b", None, None, 0)])
def test_gains_and_caches_need_no_alignment(name, batch, head_dim, one, monkeypatch):
    """Norm gains at an odd float offset (a pass in one launch, fp32 and bf16; pair GEMM from 48 rows on; unfused bf16 path; fp32 path launch
    by launch, one-CTA GEMM), and where no tensor map is built over them (fp32, head_dim 64) caches at an odd element: same bits as
    aligned."""
    monkeypatch.setenv("VIASD_ONE_LAUNCH", str(one))
    vb = _vb()
    base = W.get(name)
    wl = replace(base, batch=batch or base.batch, shape=replace(base.shape, head_dim=head_dim or base.shape.head_dim))
    eng = _engine(wl)
    state = [t.clone() for t in (eng.k_full, eng.v_full, eng.k_slim, eng.v_slim, eng.len, eng.pending, eng.tokens, eng.len_full)]
    n0 = vb.launch_count()
    want = _step(eng, eng.model, eng.cache, wl.batch, wl.n_nodes)
    assert (vb.launch_count() - n0 == 4) == (one == 1 and batch is None and head_dim is None)      # pass, statistics, walk, commit
    layers = [{k: _shifted(v) if k.startswith("norm") else v for k, v in l.items()} for l in eng.layers]
    ws = torch.empty_like(eng.workspace)
    assert ws.data_ptr() % 256 == 0
    mask = [int(l in eng.routed) for l in range(wl.shape.n_layers)]
    model = vb.init_model(eng.cfg, eng.embed, eng.lm_head, _shifted(eng.final_norm), layers, mask, ws)
    if wl.shape.dtype == "f32" or wl.shape.head_dim == 64:
        state[:4] = [_shifted(t) for t in state[:4]]
    got = _step(eng, model, vb.make_cache(*state), wl.batch, wl.n_nodes)
    for w, g in zip(want, got):
        assert torch.equal(w, g)
    for w, g in zip((eng.k_full, eng.v_full, eng.k_slim, eng.v_slim, eng.len, eng.pending, eng.tokens), state):
        assert torch.equal(w, g)


# ---------------------------------------------------------------------------------------------
# a wait that expires
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("name,batch", [("mini_7b", 1), ("mini_13b", 8)])
def test_expired_wait_leaves_a_usable_handle(name, batch):
    """One arrival counter is off (as after a failure): the tile it belongs to gives up its wait after its limit, the pass ends,
    the status says so, and the next pass on the same handle computes what it did before.  One-CTA and pair GEMM."""
    vb = _vb()
    base = W.get(name)
    # one layer, k = 2048: the first tile of the O and down projections is split among CTAs
    wl = replace(base, batch=batch, shape=replace(base.shape, n_layers=1, d_model=2048, d_ff=2048), n_routed=1)
    eng = _engine(wl)
    want, got = eng.logits_buffer(), eng.logits_buffer()
    n0 = vb.launch_count()
    vb.full_forward(eng.model, eng.cache, eng.draft, want)
    torch.cuda.synchronize()
    assert vb.launch_count() - n0 > 1                          # (not a small model's pass in one)
    # the counters are the workspace's last piece
    s = wl.shape
    n = 4 * (max(s.vocab, s.n_heads * s.head_dim + 2 * s.n_kv_heads * s.head_dim, s.d_ff) // 64 + 8)
    at = eng.workspace.numel() - (n + 255) // 256 * 256
    counters = eng.workspace[at:at + n].view(torch.int32)
    assert int(counters.abs().max()) == 0
    counters[0] = 1 << 20                                      # the first arrival wraps it: one is missing
    vb.full_forward(eng.model, eng.cache, eng.draft, got)
    torch.cuda.synchronize()
    assert vb.get_stats(eng.model).device_status == vb.VIASD_EDEVICE
    vb.full_forward(eng.model, eng.cache, eng.draft, got)
    torch.cuda.synchronize()
    assert torch.equal(want, got) and int(counters.abs().max()) == 0


@pytest.mark.parametrize("word", [0, 1, 2])
@pytest.mark.parametrize("name", ["c1_tiny", "mini_7b"])
def test_wrong_counter_of_a_pass_in_one_launch_costs_one_pass(name, word):
    """The same for a small model's pass in one launch: a barrier's counter is off (its wait gives up, the status says so), or an
    attention pair's (nobody merges that pair, or too early); the next pass, and the one behind it, compute what the first did."""
    vb = _vb()
    wl = W.get(name)
    eng = _engine(wl)
    out = eng.logits_buffer()

    def run():
        n0 = vb.launch_count()
        vb.full_forward(eng.model, eng.cache, eng.draft, out)
        torch.cuda.synchronize()
        assert vb.launch_count() - n0 == 1
        return out.clone()

    want = run()
    # in front of the workspace's last piece: a line that says which set is next, and two sets of whole lines
    s, line = wl.shape, 32
    words = 2 + min(2 * wl.batch * s.n_heads * 4, s.n_heads * 4 + s.n_kv_heads * 64)
    words = -(-words // line) * line
    last = 4 * (max(s.vocab, s.n_heads * s.head_dim + 2 * s.n_kv_heads * s.head_dim, s.d_ff) // 64 + 8)
    n = 4 * (line + 2 * words)
    at = eng.workspace.numel() - (last + 255) // 256 * 256 - (n + 255) // 256 * 256
    counters = eng.workspace[at:at + n].view(torch.int32)
    which = int(counters[0])
    assert which in (0, 1) and int(counters[1:].abs().max()) == 0
    counters[line + which * words + word] = 1 << 20            # the first arrival wraps it: one is missing
    bad = run()
    if word < 2:
        assert vb.get_stats(eng.model).device_status == vb.VIASD_EDEVICE
    else:
        assert not torch.equal(bad, want)
    for _ in range(2):
        assert torch.equal(run(), want) and int(counters[1:].abs().max()) == 0


# ---------------------------------------------------------------------------------------------
# a node whose gate row does not exist
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("phases", [(3,), (1, 2)])
@pytest.mark.parametrize("mode,bad", [("greedy", -1), ("greedy", 99), ("sampling", 8)])
def test_node_without_a_gate_row_goes_to_the_full_verifier(phases, mode, bad):
    """prow outside [0, R): recorded, and the node is judged by q, never accepted outright; alone or with the walk."""
    vb = _vb()
    wl = replace(W.get("mini_7b"), mode=mode)
    eng = _engine(wl)
    prow = eng.prow.clone()
    prow[2] = bad
    draft = vb.make_draft(eng.draft_tok, eng.parent, prow, eng.inputs.n_prows, eng.drafter_logits)
    g = torch.Generator(device="cuda").manual_seed(5)
    slim, full = (torch.randn(eng.logits_buffer().shape, device="cuda", generator=g) for _ in range(2))
    results = []
    for d in (eng.draft, draft):
        r = vb.alloc_result(wl.batch, wl.n_nodes)
        for phase in phases:
            # every token is accepted outright where its gate row exists
            vb.tier_accept(eng.model, d, eng.params(log_tau_lo=-1e9, log_tau_hi=-1e9), slim, full, phase, r)
        torch.cuda.synchronize()
        results.append((r, vb.get_stats(eng.model).device_status))
    (good, s0), (r, s1) = results
    assert s0 == 0 and int(good.n_acc[0]) == wl.n_nodes and s1 == vb.VIASD_EDEVICE
    assert r.tier[0].tolist() == [2 if n == 2 else 0 for n in range(wl.n_nodes)]
    assert r.conf[0, 2].item() == -float("inf") and int(r.judge[0, 2]) >> 4 == 2


# ---------------------------------------------------------------------------------------------
# one sweep for both verifiers on the GEMM for many rows
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("batch,nodes", [(7, 6), (5, 12), (2, 63)])
def test_one_sweep_of_many_rows_is_the_two_passes(batch, nodes):
    """49, 65 and 128 rows per verifier, routed layers 98 (one sub-tile), 130 (the second stream begins inside a sub-tile) and
    256 (a full launch): logits and caches bit for bit those of the separate passes; 128 as the option's value means 128."""
    vb = _vb()
    base = W.get("mini_13b")
    wl = replace(base, batch=batch, ctx=70, parent=W.chain(nodes))
    eng = _engine(wl)
    slim, full, res = eng.logits_buffer(), eng.logits_buffer(), vb.alloc_result(batch, nodes)
    caches = (eng.k_full, eng.v_full, eng.k_slim, eng.v_slim)
    before, pending = [t.clone() for t in caches], eng.pending.clone()
    vb.full_forward(eng.model, eng.cache, eng.draft, full)
    vb.slim_forward(eng.model, eng.cache, eng.draft, slim)
    torch.cuda.synchronize()
    want = [t.clone() for t in (full, slim, *caches)]
    launches = []
    for option in (-1, 128):
        for t, b in zip(caches, before):
            t.copy_(b)
        eng.len.fill_(wl.ctx)
        eng.pending.copy_(pending)
        vb.set_option(eng.model, "dual_max_rows", option)
        n0 = vb.launch_count()
        # nothing is accepted, so the commit moves no row
        vb.verify_step(eng.model, eng.cache, eng.draft, eng.params(log_tau_lo=1e9, log_tau_hi=1e9, log_acc_rel=(1e9, 1e9, 1e9)), slim, full, res)
        torch.cuda.synchronize()
        launches.append(vb.launch_count() - n0)
        for w, t in zip(want, (full, slim, *caches)):
            assert torch.equal(w, t)
    assert vb.get_stats(eng.model).device_status == 0 and int(res.n_acc.sum()) == 0
    assert (launches[0] < launches[1]) == (2 * batch * (nodes + 1) > 128)


# ---------------------------------------------------------------------------------------------
# precision of attention with many query rows per kv head
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("nodes,ctx", [(63, 900), (32, 2500)])
def test_attention_of_many_rows_is_as_precise_as_fp32(nodes, ctx):
    """256 and 132 query rows per kv head, on a model whose logits are the normalised attention output: one layer, embeddings
    that are exact in bf16 and small, an identity as output projection and head, no feed-forward.  The output goes through
    two bf16 pairs (2.2e-6 each, rms); fp32 arithmetic adds 1e-6, queries and weights as pairs would add 3e-6 and more."""
    vb = _vb()
    H, Hkv, hd, M, B = 8, 2, 128, nodes + 1, 2
    d, V, ff, N = H * hd, H * hd, 128, nodes
    g = torch.Generator(device="cuda").manual_seed(7)
    rnd = lambda *shape, s=1.0: (torch.randn(*shape, device="cuda", generator=g) * s).bfloat16()
    eye, zero, ones = torch.eye(d, device="cuda").bfloat16(), torch.zeros(ff, d, device="cuda").bfloat16(), torch.ones(d, device="cuda")
    wq, wk, wv = rnd(H * hd, d, s=0.04), rnd(Hkv * hd, d, s=0.04), rnd(Hkv * hd, d, s=0.04)
    embed = rnd(V, d, s=2.0 ** -14)
    layer = dict(wq=wq, wk=wk, wv=wv, wo=eye, wg=zero, wu=zero, wd=zero.T.contiguous(), norm1=ones, norm2=ones)
    max_ctx = ctx + M + 5
    cfg = vb.make_config(1, d, H, Hkv, hd, ff, V, "bf16", B, max_ctx, M, rms_eps=0.0)
    ws = torch.empty(vb.workspace_bytes(cfg, 1), dtype=torch.uint8, device="cuda")
    model = vb.init_model(cfg, embed, eye, ones, [layer], [1], ws)
    kc, vc = rnd(1, B, Hkv, max_ctx, hd, s=1.3), rnd(1, B, Hkv, max_ctx, hd, s=1.3)
    ints = lambda *s: torch.randint(0, V, s, dtype=torch.int32, device="cuda", generator=g)
    pending, tok = ints(B), ints(B, N)
    cache = vb.make_cache(kc, vc, kc.clone(), vc.clone(), torch.full((B,), ctx, dtype=torch.int32, device="cuda"), pending)
    parent = torch.arange(-1, N - 1, dtype=torch.int32, device="cuda")
    logits = torch.empty(B, M, V, device="cuda")
    vb.full_forward(model, cache, vb.make_draft(tok, parent, parent, 0, None), logits)
    torch.cuda.synchronize()
    assert vb.get_stats(model).device_status == 0
    e = embed[torch.cat([pending[:, None], tok], 1).long()].double()
    a = e * torch.rsqrt((e * e).mean(-1, keepdim=True))
    q = (a @ wq.double().T).view(B, M, H, hd)
    pos = (ctx + torch.arange(M, device="cuda")).double()[:, None] * 1e4 ** (-2 * torch.arange(hd // 2, device="cuda").double() / hd)
    c, s = torch.cos(pos)[None, :, None], torch.sin(pos)[None, :, None]
    q = torch.cat([q[..., :64] * c - q[..., 64:] * s, q[..., 64:] * c + q[..., :64] * s], -1)
    n = ctx + M                                                # the block's own rows as the cache holds them
    keys, values = kc[0, :, :, :n].double().repeat_interleave(H // Hkv, 1), vc[0, :, :, :n].double().repeat_interleave(H // Hkv, 1)
    score = torch.einsum("bmhd,bhkd->bhmk", q, keys) / hd ** 0.5
    hidden = torch.ones(M, n, dtype=torch.bool, device="cuda").triu(ctx + 1)
    out = torch.einsum("bhmk,bhkd->bmhd", score.masked_fill(hidden, -np.inf).softmax(-1), values).reshape(B, M, d)
    h = e + out
    want = h * torch.rsqrt((h * h).mean(-1, keepdim=True))
    rel = float((logits.double() - want).norm() / want.norm())
    assert rel < 4.2e-6, rel


# ---------------------------------------------------------------------------------------------
# many rejections at one position
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("vocab,team,nodes,alpha,beta", [(4099, 1, 40, 0.0, 1.0), (4100, 1, 25, 0.1, 0.8), (33000, 8, 40, 0.0, 1.0), (20003, 2, 17, 0.0, 1.3)])
def test_star_of_rejected_children(vocab, team, nodes, alpha, beta):
    """A star of children, all unlikely under their judges, half of them judged by either: the rejections of one position are
    written out every eighth time and replayed between; vocabularies of every alignment, one CTA and several.  The last
    child is likely, so that a test after many rejections passes too.  Decisions against the oracle under the margin rule."""
    from oracle import tiers
    from tests import parity_util as PU
    vb = _vb()
    base = W.get("mini_8b_tree")
    wl = replace(base, batch=4, ctx=8, parent=tuple([-1] * nodes), shape=replace(base.shape, vocab=vocab, n_layers=1), n_routed=1)
    eng = _engine(wl)
    vb.set_option(eng.model, "accept_team", team)
    si = eng.inputs
    rng = np.random.default_rng(vocab)
    B, M, V = wl.batch, wl.rows, vocab
    near = np.repeat(si.drafter_logits[:, :1], M, axis=1)
    slim = (near + rng.standard_normal((B, M, V))).astype(np.float32)
    full = (near + rng.standard_normal((B, M, V))).astype(np.float32)
    for b in range(B):
        for n in range(nodes):
            d = 12.0 if n == nodes - 1 and b % 2 else -6.0
            slim[b, 0, si.draft_tok[b, n]] += d
            full[b, 0, si.draft_tok[b, n]] += d
    d = tiers.tier_rule(si.drafter_logits, si.draft_tok, si.prow, 0.0, 0.0)[1].ravel()
    lo, hi = float(np.median(d)), 1.0                          # nothing is accepted outright
    res = vb.alloc_result(B, nodes)
    p = eng.params(log_tau_lo=lo, log_tau_hi=hi, mode=1, alpha=alpha, beta=beta)
    vb.tier_accept(eng.model, eng.draft, p, torch.from_numpy(slim).cuda(), torch.from_numpy(full).cuda(), 3, res)
    torch.cuda.synchronize()
    tier, _ = tiers.tier_rule(si.drafter_logits, si.draft_tok, si.prow, lo, hi)
    assert np.array_equal(res.tier.cpu().numpy(), tier)
    P = tiers.Params(mode="sampling", temperature=wl.temperature, seed=wl.seed, alpha=alpha, beta=beta)
    seqs = tiers.resolve(si.draft_tok, wl.parent, si.prow, tier, si.drafter_logits, slim, full, P)
    assert int(((res.judge & 3) == 2).sum()) >= 9 * B          # folded in every sequence
    pinned, total, whole = PU.compare_resolution(seqs, res.n_acc.cpu().numpy(), res.path.cpu().numpy(), res.out_tok.cpu().numpy(),
                                                 res.n_emit.cpu().numpy(), res.corr_src.cpu().numpy(), eps_row=2.5e-5)
    PU.assert_pinned(f"star of {nodes}, vocabulary {vocab}", pinned, total, whole, B, 0.85, 3)
    assert vb.get_stats(eng.model).device_status == 0 and eng.guards_intact()


# ---------------------------------------------------------------------------------------------
# precision of the verification cost
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("vocab,temperature", [(32000, 1.0), (50257, 0.7), (152064, 1.0), (152064, 1.3)])
def test_cost_is_as_precise_as_its_sums(vocab, temperature):
    """Relative error of a row's cost, rms over rows: the fp32 sums over its vocabulary (2e-7 to 3e-7 rms, measured; any other
    order shows as much), not the last bit of a logarithm of the order of ten, which shifts every margin of a row (7e-7)."""
    vb = _vb()
    g = torch.Generator(device="cuda").manual_seed(11)
    judge = torch.randn(64, vocab, device="cuda", generator=g) * 1.3
    prop = judge + torch.randn(64, vocab, device="cuda", generator=g) * 0.4
    got, _ = vb.kl_cost(judge, prop, temperature=temperature)
    t = float(np.float32(temperature))
    lq, lp = (judge.double() / t).log_softmax(1), (prop.double() / t).log_softmax(1)
    d = (lp - lq).clamp(min=0)
    want = (lp.exp() * d).sum(1) + (lq.exp() * d).sum(1)
    err = (got.double() - want) / want
    assert float(err.pow(2).mean().sqrt()) < 4.5e-7, float(err.pow(2).mean().sqrt())


# ---------------------------------------------------------------------------------------------
# fp32 products at the sizes where the features per warp change (148 SMs: 1776, 2368 and 4736 outputs)
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("rows,n,k", [(9, 1775, 72), (9, 1777, 64), (5, 2367, 40), (8, 2369, 40), (13, 3001, 40), (4, 4735, 136), (9, 4738, 64)])
def test_fp32_product_by_features_per_warp(rows, n, k):
    vb = _vb()
    g = torch.Generator(device="cuda").manual_seed(3)
    x, w = torch.randn(rows, k, device="cuda", generator=g), torch.randn(n, k, device="cuda", generator=g) * 0.05
    y = torch.full((rows, n), float("nan"), device="cuda")
    vb.gemm(x, w, y, torch.empty(vb.gemm_scratch_bytes(rows, n, k), dtype=torch.uint8, device="cuda"))
    want = x.double() @ w.double().T
    # exact products, fp32 accumulation of k terms
    assert float((y.double() - want).abs().max()) <= 2e-6 * np.sqrt(k) * float(want.abs().max()) + 1e-6


# ---------------------------------------------------------------------------------------------
# a step that will be refused
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("dual_max", [-1, 0])
@pytest.mark.parametrize("what", ["no drafter rows", "too many drafter rows", "no place for the path"])
def test_refused_step_runs_nothing(dual_max, what):
    """Arguments that the walk refuses are refused before either verifier has run, in one sweep or in turn."""
    vb = _vb()
    wl = W.get("mini_7b")
    eng = _engine(wl)
    vb.set_option(eng.model, "dual_max_rows", dual_max)
    n_prows = {"no drafter rows": 0, "too many drafter rows": 65}.get(what, eng.inputs.n_prows)
    draft = vb.make_draft(eng.draft_tok, eng.parent, eng.prow, n_prows, eng.drafter_logits)
    res = vb.alloc_result(wl.batch, wl.n_nodes)
    if what == "no place for the path":
        res.path = None
    before = [t.clone() for t in (eng.k_full, eng.k_slim, eng.len)]
    n0 = vb.launch_count()
    with pytest.raises(vb.ViasdError) as e:
        vb.verify_step(eng.model, eng.cache, draft, eng.params(conf_source=1), eng.logits_buffer(), eng.logits_buffer(), res)
    torch.cuda.synchronize()
    assert e.value.code == vb.VIASD_EINVAL and vb.launch_count() == n0
    assert all(torch.equal(a, b) for a, b in zip(before, (eng.k_full, eng.k_slim, eng.len)))


# ---------------------------------------------------------------------------------------------
# caches that have never been written past the block
# ---------------------------------------------------------------------------------------------
@pytest.mark.parametrize("name,nodes,kernel,one", [("mini_7b", 8, "mma", 1), ("mini_7b", 8, "tk", 1), ("mini_8b_tree", 26, "tc", 1), ("mini_8b_tree", 40, "tc", 1),
                                                   ("mini_32b_b3", 5, "tk", 1), ("mini_32b_b3", 5, "tc", 1), ("c1_tiny", 4, "auto", 1), ("c1_tiny", 4, "auto", 0),
                                                   ("mini_7b", 8, "auto", 1), ("mini_8b_tree_greedy", 5, "auto", 1)])
@pytest.mark.parametrize("ctx", [0, 116, 245, 333])
def test_nothing_past_the_block_is_read_into_the_result(name, nodes, kernel, one, ctx):
    """NaN in every slot past the block's: same bits as with zeros there, whatever 16-, 32-, 64- or 128-key group the block ends in;
    with kernel "auto" in one launch, or (one: 0) launch by launch."""
    vb = _vb()
    base = W.get(name)
    eng = _engine(replace(base, ctx=ctx, parent=W.chain(nodes), shape=replace(base.shape, n_layers=2), n_routed=1), extra_ctx=140)
    vb.set_option(eng.model, "attention_kernel", kernel)
    vb.set_option(eng.model, "one_launch", one)
    eng.len.fill_(ctx)
    n0 = vb.launch_count()
    got = []
    for fill in (0.0, float("nan")):
        for t in (eng.k_full, eng.v_full):
            t[:, :, :, ctx:] = fill
        out = eng.logits_buffer()
        vb.full_forward(eng.model, eng.cache, eng.draft, out)
        torch.cuda.synchronize()
        got.append(out)
    assert torch.isfinite(got[1]).all() and torch.equal(*got)
    assert (vb.launch_count() - n0 == 2) == (kernel == "auto" and one == 1)


# ---------------------------------------------------------------------------------------------
# a context that does not hold the one launch of a small model's pass
# ---------------------------------------------------------------------------------------------
_NO_ROOM = """
import sys
sys.path.insert(0, {root!r})
from dataclasses import replace
import torch
from paper_2606_12243_b200 import binding as vb
vb.LIB_PATH = {lib!r}
from paper_2606_12243_b200.engine import Engine
from synth import workloads as W

for name, policy in (("c1_tiny", 0), ("mini_7b", 0), ("mini_13b", 0), ("mini_7b", 1)):
    wl = W.get(name)
    outs = []
    for one in (1, 0):
        eng = Engine(wl, fill_context="device", max_query=wl.rows + (18 if policy else 0))
        eng.set_inputs(W.step_inputs(wl))
        vb.set_option(eng.model, "one_launch", one)
        vb.set_timing(eng.model, True)
        sl, fl, f2, s2, res = *(eng.logits_buffer().zero_() for _ in range(4)), vb.alloc_result(wl.batch, wl.n_nodes)
        n0 = vb.launch_count()
        vb.full_forward(eng.model, eng.cache, eng.draft, f2)
        vb.slim_forward(eng.model, eng.cache, eng.draft, s2)
        # (every token is the full verifier's to judge: the routed step's pass runs)
        vb.verify_step(eng.model, eng.cache, eng.draft, eng.params(policy=policy, log_tau_lo=1e9, log_tau_hi=1e9), sl, fl, res)
        torch.cuda.synchronize()
        stats = vb.get_stats(eng.model)
        assert stats.device_status == 0 and stats.full_ran
        timing = vb.get_timing(eng.model)
        outs.append(([vb.launch_count() - n0] + [v["launches"] for v in timing.values() if isinstance(v, dict)],
                     [t.clone() for t in (sl, fl, f2, s2, eng.k_full, eng.v_full, eng.k_slim, eng.v_slim, eng.len, eng.pending, res.out_tok, res.n_acc)]))
    assert outs[0][0] == outs[1][0], (name, policy, outs[0][0], outs[1][0])
    assert all(torch.equal(a, b) for a, b in zip(outs[0][1], outs[1][1])), (name, policy)
"""


def test_pass_without_room_goes_launch_by_launch(tmp_path):
    """The driver refuses the cooperative launch (in a context with a share of the SMs, say): the library with that launcher replaced by
    one that always answers so computes, launches and counts what it does with the option off - step, single passes, routed step."""
    import os
    import subprocess
    import sys
    from paper_2606_12243_b200 import build as B
    B.build()
    stub, obj, lib = tmp_path / "stub.cu", tmp_path / "stub.o", tmp_path / "libviasd_no_room.so"
    stub.write_text("""
        #include "common.cuh"
        bool small_pass_takes(const viasd_model *m, const viasd_cache *, int, int, bool) { return m->opt.one_launch; }
        int launch_small_pass(viasd_model *, const viasd_cache *, const viasd_draft *, int, int, float *, float *, cudaStream_t) { return SMALL_PASS_NO_ROOM; }
        """)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.check_call([B.NVCC, *B.FLAGS, "-I", B.CSRC, "-c", str(stub), "-o", str(obj)])
    others = [os.path.join(B.OBJ, f[:-3] + ".o") for f in B._sources() if f != "small_pass.cu"]
    subprocess.check_call([B.NVCC, "-shared", "-o", str(lib), str(obj), *others, "-lcuda"])
    code = _NO_ROOM.format(root=root, lib=str(lib))
    subprocess.run([sys.executable, "-c", code], check=True, timeout=300, cwd=root)
