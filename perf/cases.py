"""What this framework is measured on: the calls a speculative-decoding server makes of it, over their real range.

A case is a dict of plain values.  ``kind`` names the call:
  step     viasd_verify_step (one decoding cycle; ``steps`` > 1: that many in a row, the cache growing as tokens are committed)
  prefill  one chunk of a prompt through both verifiers and into both caches (full forward, slim forward, commit)
  accept   viasd_tier_accept on logits at hand (a server that runs the forward passes itself)
  score    viasd_kl_cost and viasd_region_mass over a window of decoding positions (mask search, threshold calibration)
  gemm     the stand-alone projection viasd_gemm
Models have the layer shapes of the benchmark workloads; the number of layers is what lets a state fit the card three
times, every layer doing the same work.  Weights are N(0, 0.02), drafter logits N(0, 2) with 3 added on each drafted
token, thresholds at the 40th and 75th percentile of drafter confidence (75 % of the drafted tokens need a verifier).
"""
import math

import torch

from paper_2606_12243_b200 import binding as vb

TINY = dict(d_model=256, heads=4, kv_heads=4, head_dim=64, d_ff=1024, vocab=1024, dtype="f32")
MINI = dict(d_model=512, heads=4, kv_heads=4, head_dim=128, d_ff=1408, vocab=2048, dtype="bf16")
MINI_GQA = dict(d_model=512, heads=4, kv_heads=1, head_dim=128, d_ff=1536, vocab=4096, dtype="bf16")
S7B = dict(d_model=4096, heads=32, kv_heads=32, head_dim=128, d_ff=11008, vocab=32000, dtype="bf16")
S8B = dict(d_model=4096, heads=32, kv_heads=8, head_dim=128, d_ff=14336, vocab=128256, dtype="bf16")
S13B = dict(d_model=5120, heads=40, kv_heads=40, head_dim=128, d_ff=13824, vocab=32000, dtype="bf16")
S32B = dict(d_model=5120, heads=40, kv_heads=8, head_dim=128, d_ff=27648, vocab=152064, dtype="bf16")


def _step(name, shape, layers, routed, batch, ctx, draft, mode="greedy", gate="drafter", policy=0, steps=1):
    c = dict(kind="step", layers=layers, routed=routed, batch=batch, ctx=ctx, draft=draft, mode=mode, gate=gate, policy=policy,
             steps=steps, **shape)
    return dict(name=name, **c) if name else c


def _prefill(name, shape, layers, routed, batch, ctx, chunk):
    c = dict(kind="prefill", layers=layers, routed=routed, batch=batch, ctx=ctx, draft="chain%d" % (chunk - 1), **shape)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # smallest: a toy-sized fp32 model, one sequence; nothing but latency
        _step("step_tiny_f32", TINY, 2, 1, 1, 128, "chain4"),
        # a drafter-sized bf16 verifier (an embedded or test deployment), one sequence; latency of the bf16 path
        _step("step_mini_bf16", MINI, 4, 2, 1, 300, "chain8"),
        # one user of a 7B model, the usual chain draft, greedy
        _step("step_7b_b1", S7B, 32, 16, 1, 1024, "chain8"),
        # one user of an 8B model with a tree draft, sampling (the benchmark's default workload)
        _step("step_8b_tree_b1", S8B, 32, 12, 1, 2048, "tree26", mode="sampling"),
        # the same with four users batched: 108 rows per verifier
        _step("step_8b_tree_b4", S8B, 32, 12, 4, 2048, "tree26", mode="sampling"),
        # eight users with long contexts and no grouped heads: half of the bytes are the KV cache
        _step("step_13b_b8", S13B, 20, 10, 8, 4096, "chain6"),
        # a full batch on the largest model, the slim verifier's own confidence as the gate (Algorithm 2)
        _step("step_32b_b16", S32B, 16, 8, 16, 4096, "chain5", gate="slim"),
        # six cycles of the routed execution policy with the thresholds it is for (most tokens in tiers 0 and 1)
        _step("routed_7b_6steps", S7B, 32, 16, 1, 1024, "chain8", policy=1, steps=6),
        # a chunk in the middle of eight users' prompts: the path's other direction, and its largest call
        _prefill("prefill_8b_b8", S8B, 32, 12, 8, 960, 64),
        # the decision alone, sixteen users with trees, on logits at hand
        dict(name="accept_tree_b16", kind="accept", batch=16, draft="tree26", vocab=128256, mode="sampling"),
        # scoring a layer mask over a window of positions; an odd number of rows
        dict(name="score_1021x152064", kind="score", rows=1021, vocab=152064, smooth=False),
        # one projection on its own, an odd number of rows
        dict(name="gemm_41x13824x5120", kind="gemm", rows=41, n=13824, k=5120),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    """One more case: any model shape, batch, context, draft and option of the ranges above."""
    most = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= most and _state_bytes(c) < 48e9:
            return c


def _draw(rng):
    kind = rng.choices(["step", "prefill", "accept", "score", "gemm"], [12, 3, 2, 2, 2])[0]
    if kind == "accept":
        return dict(kind=kind, batch=_log_int(rng, 1, 16), draft=rng.choice(["chain5", "chain8", "tree7", "tree26"]),
                    vocab=rng.choice([32000, 50257, 128256, 152064]), mode=rng.choice(["greedy", "sampling"]))
    if kind == "score":
        return dict(kind=kind, rows=_log_int(rng, 5, 1021), vocab=rng.choice([32000, 50257, 128256, 152064]),
                    smooth=rng.random() < 0.25)
    if kind == "gemm":
        return dict(kind=kind, rows=_log_int(rng, 1, 256), n=8 * _log_int(rng, 40, 16000), k=8 * _log_int(rng, 64, 2048))
    size = rng.random()
    if size < 0.15 and kind == "step":
        shape, layers = dict(TINY, d_model=rng.choice([192, 256, 384]), d_ff=rng.choice([680, 1024])), rng.randint(1, 4)
    elif size < 0.3 and kind == "step":
        shape, layers = dict(rng.choice([MINI, MINI_GQA])), rng.randint(2, 6)
    else:
        shape, layers = dict(rng.choice([S7B, S8B, S13B, S32B])), rng.randint(4, 16)
    batch, ctx, routed = _log_int(rng, 1, 16), _log_int(rng, 65, 4096), max(1, int(layers * rng.uniform(0.25, 0.75)))
    if kind == "prefill":
        return _prefill("", shape, layers, routed, batch, ctx, rng.choice([17, 33, 48, 64]))
    policy = 1 if shape["dtype"] == "bf16" and shape["heads"] == shape["kv_heads"] and rng.random() < 0.2 else 0
    draft = rng.choice(["chain3", "chain5", "chain6", "chain8", "tree7"] + ([] if policy else ["tree26", "tree26"]))
    return _step("", shape, layers, routed, batch, ctx, draft, rng.choice(["greedy", "sampling"]),
                 rng.choice(["drafter", "slim"]), policy, 4 if policy else 1)


# ---- what a case needs -------------------------------------------------------------------------------------------
def _tree(draft):
    """Parents of the draft's nodes (-1: child of the pending token), parents first."""
    if draft.startswith("chain"):
        return list(range(-1, int(draft[5:]) - 1))
    if draft == "tree7":
        return [-1, -1, -1, 0, 0, 3, 1]
    par = [-1] * 4 + [i for i in range(4) for _ in range(3)] + [4 + 3 * i for i in range(4) for _ in range(2)] + [16, 24]
    assert draft == "tree26" and len(par) == 26
    return par


def _prows(parent):
    """Which drafter row each node was drawn from: one row per distinct parent, in order of appearance."""
    order = {}
    return [order.setdefault(p, len(order)) for p in parent], len(order)


def _lens(c):
    """Committed lengths: the users of a batch are not equally far."""
    return [max(c["ctx"] - (37 * b) % 128, c["ctx"] // 2) for b in range(c["batch"])]


def _layer_params(c):
    d, hd = c["d_model"], c["head_dim"]
    return 2 * d * c["heads"] * hd + 2 * d * c["kv_heads"] * hd + 3 * d * c["d_ff"] + 2 * d


REPLAY = 18            # committed tokens the routed policy can replay


def _state_bytes(c):
    if c["kind"] in ("step", "prefill"):
        es = 4 if c["dtype"] == "f32" else 2
        kv = (c["layers"] + c["routed"]) * 2 * c["batch"] * c["kv_heads"] * (c["ctx"] + 600) * c["head_dim"]
        return (c["layers"] * _layer_params(c) + 2 * c["vocab"] * c["d_model"] + kv) * es
    return work(c)["bytes"]


def _cost(c):
    w = work(c)
    return max(w["bytes"], w["flops"] / 200)


def work(case):
    c = case
    if c["kind"] == "gemm":
        return {"bytes": 2 * (c["rows"] + c["n"]) * c["k"] + 4 * c["rows"] * c["n"], "flops": 2 * c["rows"] * c["n"] * c["k"]}
    if c["kind"] == "score":                                  # both calls read both rows
        return {"bytes": 2 * 2 * c["rows"] * c["vocab"] * 4, "flops": 30 * c["rows"] * c["vocab"]}
    parent = _tree(c["draft"])
    rows, (_, n_prows) = c["batch"] * (len(parent) + 1), _prows(parent)
    if c["kind"] == "accept":                                 # each logits row once
        return {"bytes": (2 * rows + c["batch"] * n_prows) * c["vocab"] * 4, "flops": 5 * (2 * rows + c["batch"] * n_prows) * c["vocab"]}
    es = 4 if c["dtype"] == "f32" else 2
    both = c["layers"] + c["routed"]                          # layer passes; a routed layer's weights serve both verifiers
    weights = (c["layers"] * _layer_params(c) + c["vocab"] * c["d_model"]) * es
    kv_row = 2 * c["kv_heads"] * c["head_dim"] * es
    kv = both * kv_row * (sum(_lens(c)) + rows)
    logits = 2 * 2 * rows * c["vocab"] * 4 if c["kind"] == "step" else 2 * rows * c["vocab"] * 4     # written, and read by the walk
    flops = 2 * rows * (both * _layer_params(c) + 2 * c["vocab"] * c["d_model"]) \
        + both * 4 * (len(parent) + 1) * (sum(_lens(c)) + rows) * c["heads"] * c["head_dim"]
    tier = c["batch"] * n_prows * c["vocab"] * 4 if c["kind"] == "step" else 0
    if c.get("policy") == 1:
        # the slim verifier in every step, the full verifier in a tenth of them
        part = (c["routed"] * _layer_params(c) + c["vocab"] * c["d_model"]) * es + c["routed"] * kv_row * (sum(_lens(c)) + rows)
        full = weights + c["layers"] * kv_row * (sum(_lens(c)) + rows)
        return {"bytes": c["steps"] * (part + logits // 2 + tier) + max(1.0, 0.1 * c["steps"]) * full,
                "flops": c["steps"] * 2 * rows * (c["routed"] * _layer_params(c) + c["vocab"] * c["d_model"])}
    return {"bytes": weights + kv + logits + tier + 2 * rows * c["d_model"] * es, "flops": flops}


def tolerance(case):
    """About four times what the same call shows with its sums in another order (attention kernels and key ranges swapped,
    norms unfused) or against 64 bits; single values of bf16 caches may round the other way, and a near-tie may fall so."""
    if case["kind"] == "accept":                              # fp32 differences of fp32 logits, and decisions on them
        return {"rel": 1e-6, "differ": 0.01}
    if case["kind"] == "score":                               # fp32 sums over a vocabulary: 8e-7
        return {"rel": 3e-6, "max": 1e-5}
    if case["kind"] == "gemm":                                # exact products, fp32 sums over k: 3.3e-6
        return {"rel": 1.3e-5, "max": 5e-5}
    if case["dtype"] == "f32":                                # fp32 sums throughout
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    return {"rel": 1.2e-3, "max": 0.032, "differ": 0.01}      # activations as bf16 pairs, bf16 caches: 3e-4, one bf16 step


# ---- states ------------------------------------------------------------------------------------------------------
class _State:
    pass


def _normal(g, shape, sigma, dtype=torch.float32):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, sigma, generator=g)


def _ints(values):
    return torch.tensor(values, dtype=torch.int32, device="cuda")


def _model(s, c, g, max_query, max_ctx):
    """Weights, caches with a committed context, and the handle: what a server sets up once."""
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    d, hd, ff, V, L = c["d_model"], c["head_dim"], c["d_ff"], c["vocab"], c["layers"]
    qd, kvd = c["heads"] * hd, c["kv_heads"] * hd
    w = lambda n, k: _normal(g, (n, k), 0.02 if d >= 1024 else 0.05, dt)
    gain = lambda: 1.0 + _normal(g, (d,), 0.05)
    layers = [dict(wq=w(qd, d), wk=w(kvd, d), wv=w(kvd, d), wo=w(d, qd), wg=w(ff, d), wu=w(ff, d), wd=w(d, ff), norm1=gain(),
                   norm2=gain()) for _ in range(L)]
    cfg = vb.make_config(L, d, c["heads"], c["kv_heads"], hd, ff, V, c["dtype"], c["batch"], max_ctx, max_query)
    routed = sorted({i * L // c["routed"] for i in range(c["routed"])})
    s.workspace = torch.zeros(vb.workspace_bytes(cfg, len(routed)), dtype=torch.uint8, device="cuda")
    s.model = vb.init_model(cfg, w(V, d), w(V, d), gain(), layers, [int(l in routed) for l in range(L)], s.workspace)
    kv = lambda n: _normal(g, (n, c["batch"], c["kv_heads"], max_ctx, hd), 0.02 * math.sqrt(d) if d >= 1024 else 1.0, dt)
    s.kv = [kv(L), kv(L), kv(len(routed)), kv(len(routed))]
    lens = _lens(c)
    pending = torch.randint(0, V, (c["batch"],), generator=g, device="cuda", dtype=torch.int32)
    s.marks0 = torch.stack([_ints(lens), pending, _ints(lens)])          # len, pending, len_full
    s.marks = s.marks0.clone()
    tokens = torch.randint(0, V, (c["batch"], max_ctx), generator=g, device="cuda", dtype=torch.int32)
    s.cache = vb.make_cache(*s.kv, s.marks[0], s.marks[1], tokens, s.marks[2])
    # the part of the caches that a call may write, from the shortest sequence's end on
    s.written = [t[:, :, :, min(lens):] for t in s.kv]


def _draft(c, g, parent):
    """Draft tokens of a batch with the drafter's logits: N(0, 2), 3 added on every drafted token."""
    prow, R = _prows(parent)
    B, N, V = c["batch"], len(parent), c["vocab"]
    base = torch.randint(0, V, (B, 1), generator=g, device="cuda")
    tok = ((base + torch.arange(N, device="cuda") * 7919) % V).to(torch.int32)        # siblings differ
    logits = _normal(g, (B, R, V), 2.0)
    b = torch.arange(B, device="cuda")[:, None].expand(B, N)
    logits[b, torch.tensor(prow, device="cuda").expand(B, N), tok.long()] += 3.0
    return vb.make_draft(tok, _ints(parent), _ints(prow), R, logits)


def _thresholds(g, V, lo_q, hi_q):
    """Quantiles of the drafter's relative confidence over a sample of its rows."""
    rows = _normal(g, (256, V), 2.0)
    rows[:, 0] += 3.0
    d = rows[:, 0] - rows.max(dim=1).values
    return [float(x) for x in torch.quantile(d, torch.tensor([lo_q, hi_q], device="cuda"))]


def _params(c, g, seed):
    lo, hi = _thresholds(g, c["vocab"], *((0.05, 0.5) if c.get("policy") else (0.40, 0.75)))
    slim = c.get("gate") == "slim"
    return [vb.make_params(lo, hi, mode=int(c["mode"] == "sampling"), seed=seed, step=i, policy=c.get("policy", 0),
                           conf_source=int(slim), strict_break=int(slim)) for i in range(c.get("steps", 1))]


def _answers(s, r):
    return [r.tier, r.conf, r.n_acc, r.path, r.out_tok, r.n_emit, r.judge, r.corr_src]


def prepare(case, seed):
    c, s = case, _State()
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s.kind = c["kind"]
    if s.kind == "gemm":
        s.x, s.w = _normal(g, (c["rows"], c["k"]), 1.0, torch.bfloat16), _normal(g, (c["n"], c["k"]), 0.02, torch.bfloat16)
        s.y = torch.empty((c["rows"], c["n"]), dtype=torch.float32, device="cuda")
        s.scratch = torch.empty(vb.gemm_scratch_bytes(c["rows"], c["n"], c["k"]), dtype=torch.uint8, device="cuda")
        return s
    if s.kind == "score":
        # the slim verifier's logits are near the full verifier's
        s.judge = _normal(g, (c["rows"], c["vocab"]), 1.3)
        s.proposal = s.judge + _normal(g, (c["rows"], c["vocab"]), 0.4)
        s.margin, s.tau = int(c["smooth"]), _thresholds(g, c["vocab"], 0.40, 0.75)
        return s
    parent = _tree(c["draft"])
    B, N = c["batch"], len(parent)
    M = N + 1
    if s.kind == "accept":
        # the decision needs a handle of the right vocabulary; the passes run elsewhere
        _model(s, dict(TINY, dtype="bf16", head_dim=128, heads=2, kv_heads=2, vocab=c["vocab"], layers=1, routed=1, batch=B, ctx=64), g, M, 128)
        s.draft = _draft(c, g, parent)
        drafter, prow = s.draft._keep[3], _prows(parent)[0]
        row_of = {p + 1: r for p, r in zip(parent, prow)}                # block row -> the drafter row of its children
        near = drafter[:, [row_of.get(i, 0) for i in range(M)]]
        s.slim, s.full = near + _normal(g, near.shape, 1.0), near + _normal(g, near.shape, 1.0)
        s.params, s.result = _params(c, g, seed), vb.alloc_result(B, N)
        return s
    policy = c.get("policy", 0)
    _model(s, c, g, M + (REPLAY if policy else 0), c["ctx"] + M * c.get("steps", 1) + REPLAY + 64)
    s.drafts = [_draft(c, g, parent) for _ in range(c.get("steps", 1))]
    s.slim = torch.zeros((B, M, c["vocab"]), dtype=torch.float32, device="cuda")
    s.full = torch.zeros_like(s.slim)
    s.results = [vb.alloc_result(B, N) for _ in s.drafts]
    if s.kind == "prefill":                                   # the whole chunk is accepted as it is
        r = s.results[0]
        r.n_acc.fill_(N)
        r.n_emit.fill_(N)
        r.path.copy_(torch.arange(N, device="cuda").expand(B, N))
        r.out_tok[:, :N] = s.drafts[0]._keep[0]
    else:
        s.params = _params(c, g, seed)
    return s


def run(state):
    s = state
    if s.kind == "gemm":
        vb.gemm(s.x, s.w, s.y, s.scratch)
        return s.y
    if s.kind == "score":
        cost, total = vb.kl_cost(s.judge, s.proposal, margin=s.margin, tau=0.5)
        mass, mean = vb.region_mass(s.judge, s.proposal, s.tau[1], s.tau[0])
        return cost, total, mass, mean
    if s.kind == "accept":
        vb.tier_accept(s.model, s.draft, s.params[0], s.slim, s.full, 3, s.result)
        return _answers(s, s.result)
    s.marks.copy_(s.marks0)                                   # rolls the caches back to the committed context
    if s.kind == "prefill":
        vb.full_forward(s.model, s.cache, s.drafts[0], s.full)
        vb.slim_forward(s.model, s.cache, s.drafts[0], s.slim)
        vb.kv_commit(s.model, s.cache, s.drafts[0], s.results[0])
        return [s.full, s.slim, s.marks] + s.written
    for draft, params, result in zip(s.drafts, s.params, s.results):
        vb.verify_step(s.model, s.cache, draft, params, s.slim, s.full, result)
    return [s.full, s.slim, s.marks] + s.written + [a for r in s.results for a in _answers(s, r)]
