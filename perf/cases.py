"""Cases for timing the verification library through its public entry points.

A case is one pass of something a serving program does: a whole verification step (plan, attention
layer by layer, acceptance, compaction), one attention call, one acceptance call, one contemplate-token
embedding.  Sizes are those of the workloads in paper_2603_08899_b200/inputs.py and of the parity
tests, or generic ones in between.  Inputs follow inputs.py: N(0,1) queries, keys and values, random
breadth-first draft trees, full-vocabulary logits, draft tokens drawn from the draft rows.

Steps come in two forms, as programs use them: eager calls, and a captured CUDA graph that is replayed
(buffers stay where they are, their contents change).  With "append" the pass first writes the
step's own K/V rows behind each prefix, layer by layer, as a serving loop over this library does; without
it the rows are in the cache already (written by the producer of K and V).
"""
import math

import numpy as np
import torch

from paper_2603_08899_b200 import binding as cb
from paper_2603_08899_b200 import inputs
from paper_2603_08899_b200.step import VerifyStep

PAGE = 128
DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32, "e4m3": torch.float8_e4m3fn}
BYTES = {"bf16": 2, "fp32": 4, "e4m3": 1}


def _step(name=None, **kw):
    c = dict(kind="step", B=1, L=32, Hq=32, Hkv=8, D=128, T=60, C=4, S=16, V=128256, lo=4096, hi=4096, tree="random",
             kv="bf16", logits="bf16", sigma=3.0, draft="noise", temperature=1.0, rule="ratio", graph=True, append=False,
             paged=False)
    c.update(kw)
    return dict(c, name=name) if name else c


def _attention(name=None, **kw):
    c = dict(kind="attention", B=4, Hq=32, Hkv=8, D=128, T=60, C=4, S=16, lo=500, hi=4000, tree="random", kv="bf16",
             own_plan=True)
    c.update(kw)
    return dict(c, name=name) if name else c


def _accept(name=None, **kw):
    c = dict(kind="accept", B=16, T=60, C=4, V=128256, tree="random", logits="bf16", sigma=3.0, draft="noise",
             temperature=1.0, rule="ratio")
    c.update(kw)
    return dict(c, name=name) if name else c


def _embed(name=None, **kw):
    c = dict(kind="embed", B=8, H_in=12288, H_out=4096, n_expert=64, k_expert=2, dtype="bf16", bias=True, renormalize=False)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest step: 8-node chain, fp32, head dim 64, vocabulary 1000: host work and launches
        _step("tiny_step", L=1, Hq=4, Hkv=2, D=64, T=8, C=2, S=2, V=1000, lo=256, hi=256, tree="chain", kv="fp32",
              logits="fp32", sigma=2.0, draft="independent", graph=False),
        # interactive decoding of one user, groups of three query heads, calls made one by one
        _step("llama3b_step_eager", L=28, Hq=24, lo=2048, hi=2048, draft="independent", graph=False),
        # interactive decoding of one user, the step replayed as a graph
        _step("llama8b_step"),
        # the same with one contemplate row per draft node (120 query rows) at temperature 0.7
        _step("llama8b_2t_step", C=60, temperature=0.7),
        # one user, long prefix, greedy decoding
        _step("qwen4b_greedy_step", L=36, V=151936, lo=8192, hi=8192, temperature=0.0),
        # a small server: eight users of odd, short prefixes in a paged cache, typical tree (30 nodes and a contemplate
        # row each), rows appended layer by layer, row statistics on demand
        _step("batch8_paged_step", B=8, T=30, C=30, lo=101, hi=3001, rule="lazy", append=True, paged=True),
        # a full server: 32 users, ragged prefixes 512..16384 (sixteen of the layers: a pass returns the whole cache)
        _step("batch32_step", B=32, L=16, lo=512, hi=16384),
        # the same over an 8-bit cache, the rows quantised as they are appended
        _step("batch32_e4m3_step", B=32, L=16, lo=512, hi=16384, kv="e4m3", append=True),
        # one layer, groups of eight query heads
        _attention("attention_g8", Hq=64),
        # one layer, head dim 64
        _attention("attention_d64", B=2, D=64, lo=1500, hi=2500),
        # sample-and-match acceptance of a batch, largest vocabulary, peaked logits
        _accept("accept_match", V=151936, sigma=5.0, rule="match"),
        # contemplate-token embedding from the concatenated hidden states of three layers
        _embed("con_embedding"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rows(rng):
    """Tree rows and contemplate rows: a few each, a whole tree with a few, or one contemplate row per node."""
    T = rng.choice([_log(rng, 2, 64), 30, 60, rng.randint(40, 64)])
    C = rng.choice([T, min(T, 4), rng.randint(0, T)])
    return T, C


def draw(rng):
    kind = rng.choice(["one", "one", "one", "batch", "batch", "attention", "attention", "accept", "accept", "embed"])
    T, C = _rows(rng)
    V = rng.choice([128256, 151936, 32000, rng.randint(1000, 200000)])
    temperature = rng.choice([1.0, 0.7, 0.0])
    tree = "chain" if rng.random() < 0.1 else "random"
    if kind == "one":
        lo = _log(rng, 64, 16384)
        return _step(L=rng.randint(16, 36), Hq=rng.choice([8, 24, 32]), T=T, C=C, S=rng.choice([0, 16, 16]), V=V, lo=lo, hi=lo, tree=tree,
                     draft=rng.choice(["noise", "independent"]), temperature=temperature, rule=rng.choice(["ratio", "ratio", "lazy", "match"]),
                     graph=rng.random() < 0.6, append=rng.random() < 0.4, paged=rng.random() < 0.3)
    if kind == "batch":
        B = _log(rng, 2, 32)
        hi = _log(rng, 300, 12000)
        return _step(B=B, L=rng.randint(4, 16), Hq=rng.choice([24, 32]), T=T, C=min(C, T), V=V, lo=max(1, hi // 20), hi=hi, tree=tree,
                     kv=rng.choice(["bf16", "bf16", "e4m3"]), temperature=temperature, rule=rng.choice(["ratio", "lazy", "match"]),
                     graph=rng.random() < 0.6, append=rng.random() < 0.6, paged=rng.random() < 0.5)
    if kind == "attention":
        hi = _log(rng, 100, 6000)
        kv = rng.choice(["bf16", "bf16", "bf16", "fp32"])
        D = rng.choice([64, 128])
        Hkv = rng.choice([2, 4, 8])
        G = rng.choice([1, 2, 4, 7, 8])
        return _attention(B=rng.randint(1, 6), Hq=Hkv * G, Hkv=Hkv, D=D, T=T, C=C, lo=max(1, hi // 8), hi=hi, tree=tree, kv=kv,
                          own_plan=rng.random() < 0.5)
    if kind == "accept":
        return _accept(B=_log(rng, 1, 32), T=T, C=C, V=V, tree=tree, logits=rng.choice(["bf16", "bf16", "fp32"]),
                       sigma=rng.uniform(2.0, 6.0), temperature=temperature, rule=rng.choice(["ratio", "lazy", "match"]))
    H = rng.choice([2560, 4096, 3072, 8 * rng.randint(100, 600)])
    n = _log(rng, 4, 256)
    return _embed(B=_log(rng, 1, 64), H_in=3 * H, H_out=H, n_expert=n, k_expert=min(n, rng.randint(1, 8)),
                  dtype=rng.choice(["bf16", "bf16", "fp32"]), bias=rng.random() < 0.5, renormalize=rng.random() < 0.5)


# ------------------------------------------------------------------------------------ inputs
def _lengths(case):
    """Prefix lengths: a property of the case, not of the seed, so that every seed is the same amount of work."""
    r = np.random.default_rng([case["B"], case["lo"], case["hi"]])
    return torch.from_numpy(r.integers(case["lo"], case["hi"] + 1, size=case["B"]).astype(np.int32))


def _config(case, seed):
    return inputs.VerifyConfig(
        "case", B=case["B"], L=case.get("L", 1), Hq=case.get("Hq", 4), Hkv=case.get("Hkv", 1), D=case.get("D", 64), T=case["T"], C=case["C"],
        S=case.get("S", 0), V=case.get("V", 32), prefix=(case.get("lo", 1), case.get("hi", 1)), tree=case["tree"],
        kv_dtype=DTYPES[case.get("kv", "bf16")], logit_dtype=DTYPES[case.get("logits", "bf16")], sigma_logit=case.get("sigma", 1.0),
        draft=case.get("draft", "noise"), temperatures=(case.get("temperature", 1.0),), seed=seed % 2_000_003)


class _State:
    pass


def _trees(s, cfg):
    parent, owner = inputs.trees(cfg)
    s.parent_host = parent
    s.parent, s.owner = parent.cuda(), owner.cuda() if cfg.C else None


def _cache(s, case, cfg):
    """Packed or paged pools of all layers, K and V each as one tensor [L, slots, Hkv, D], and the rows to append."""
    plen = _lengths(case)
    seq_start, n_slots = inputs.cache_layout(cfg, plen)
    s.block_table, s.max_pages = None, 0
    if case.get("paged"):
        need = [(int(p) + cfg.R + PAGE - 1) // PAGE for p in plen]
        order = np.random.default_rng([cfg.seed, 77]).permutation(sum(need) + 3).astype(np.int32)
        s.max_pages = max(need)
        table = np.zeros((cfg.B, s.max_pages), np.int32)
        at = 0
        for b, n in enumerate(need):
            table[b, :n] = order[at:at + n]
            at += n
        s.block_table = torch.from_numpy(table).cuda()
        n_slots = (sum(need) + 3) * PAGE
    s.n_slots = n_slots
    s.seq_start, s.plen = seq_start.cuda(), plen.cuda()
    fp8 = cfg.kv_dtype == torch.float8_e4m3fn
    q_type, kv_type = (torch.bfloat16, torch.uint8) if fp8 else (cfg.kv_dtype, cfg.kv_dtype)
    L = cfg.L
    s.q = torch.empty((L, cfg.B, cfg.R, cfg.Hq, cfg.D), dtype=q_type, device="cuda")
    s.out = torch.zeros_like(s.q)
    s.k = torch.empty((L, n_slots, cfg.Hkv, cfg.D), dtype=kv_type, device="cuda")
    s.v = torch.empty_like(s.k)
    s.ks = torch.empty((L, cfg.S, cfg.Hkv, cfg.D), dtype=kv_type, device="cuda") if cfg.S else None
    s.vs = torch.empty_like(s.ks) if cfg.S else None
    s.scales = []
    for l in range(L):
        t = inputs.layer_tensors(cfg, l, n_slots, device="cuda")
        s.q[l].copy_(t["q"])
        s.k[l].copy_(t["k_cache"])
        s.v[l].copy_(t["v_cache"])
        if cfg.S:
            s.ks[l].copy_(t["k_soft"])
            s.vs[l].copy_(t["v_soft"])
        if fp8:
            s.scales.append((t["k_scale"], t["v_scale"]))
    if case.get("append"):
        g = torch.Generator(device="cuda")
        g.manual_seed(cfg.seed + 5)
        s.rows = torch.randn((2, L, cfg.B, cfg.R, cfg.Hkv, cfg.D), generator=g, device="cuda", dtype=q_type)


def _logits(s, case, cfg):
    s.tl, s.dl = inputs.logits(cfg, device="cuda")
    s.tokens = inputs.draft_tokens(cfg, s.parent_host, s.dl, case["temperature"]).cuda()
    s.uniforms = inputs.uniforms(cfg).cuda()


def _prepare_step(case, seed):
    s, cfg = _State(), _config(case, seed)
    _trees(s, cfg)
    _cache(s, case, cfg)
    _logits(s, case, cfg)
    s.step = VerifyStep(cfg, s.n_slots)
    if s.block_table is not None:
        cb.confu_set_paging(s.step.ctx, s.block_table, s.max_pages)
    L = range(cfg.L)
    s.step.bind([s.q[l] for l in L], [s.k[l] for l in L], [s.v[l] for l in L], [s.ks[l] for l in L] if cfg.S else None,
                [s.vs[l] for l in L] if cfg.S else None, [s.out[l] for l in L], s.seq_start, s.plen, s.parent, s.owner, s.tl, s.dl,
                s.tokens, s.uniforms, kv_scales=s.scales or None)
    s.case = case
    if case["graph"]:
        _step_calls(s)                       # once outside the capture
        s.replay = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.replay):
            _step_calls(s)
    return s


def _step_calls(s):
    case, st = s.case, s.step
    if not case["append"] and case["rule"] == "ratio":
        st.run(case["temperature"])
        return
    if case["append"]:
        st.run_plan()
        for l in range(case["L"]):
            if s.scales:
                cb.confu_set_kv_scales(st.ctx, *s.scales[l])
            cb.confu_kv_append(st.ctx, st.dims, s.rows[0, l], s.rows[1, l], s.k[l], s.v[l], s.seq_start, s.plen)
            cb.confu_tree_attention(st.ctx, st.dims, s.q[l], s.k[l], s.v[l], s.n_slots, s.seq_start, s.plen,
                                    s.ks[l] if s.ks is not None else None, s.vs[l] if s.vs is not None else None, None, None, st.plan,
                                    s.out[l], None, st.status)
    else:
        st.run_attention()
    if case["rule"] == "match":
        cb.confu_tree_accept_match(st.ctx, case["B"], case["T"], case["C"], case["V"], s.tl.dtype, s.tl, s.tokens, s.parent, s.owner,
                                   s.uniforms if case["temperature"] > 0 else None, case["temperature"], st.accept_len, st.path,
                                   st.next_token, st.future_row, st.counters, st.status)
    else:
        st.run_accept(case["temperature"], 1 | (cb.ACCEPT_LAZY if case["rule"] == "lazy" else 0))
    st.run_compact()


def _prepare_attention(case, seed):
    s, cfg = _State(), _config(case, seed)
    _trees(s, cfg)
    _cache(s, case, cfg)
    s.ctx = cb.confu_create(0)
    s.dims = cb.make_dims(cfg.B, cfg.Hq, cfg.Hkv, cfg.D, cfg.T, cfg.C, cfg.S, cfg.kv_dtype)
    s.ws = torch.empty(cb.confu_workspace_bytes(s.ctx, s.dims), dtype=torch.uint8, device="cuda")
    cb.confu_set_workspace(s.ctx, s.ws)
    s.lse = torch.zeros((cfg.B, cfg.R, cfg.Hq), dtype=torch.float32, device="cuda")
    s.status = torch.zeros(cfg.B, dtype=torch.int32, device="cuda")
    s.plan = None
    if not case["own_plan"]:
        s.plan = torch.empty(cb.confu_plan_bytes(s.ctx, s.dims), dtype=torch.uint8, device="cuda")
        cb.confu_tree_plan(s.ctx, s.dims, s.seq_start, s.plen, s.parent, s.owner, s.plan, s.status)
    return s


def _prepare_accept(case, seed):
    s, cfg = _State(), _config(case, seed)
    s.case = case
    _trees(s, cfg)
    _logits(s, case, cfg)
    s.ctx = cb.confu_create(0)
    B, i32 = cfg.B, dict(dtype=torch.int32, device="cuda")
    s.ws = torch.empty(cb.confu_accept_workspace_bytes(B, cfg.T, cfg.V), dtype=torch.uint8, device="cuda")
    s.status, s.accept_len, s.next_token, s.future_row = (torch.zeros(B, **i32) for _ in range(4))
    s.path, s.counters = torch.zeros((B, cb.MAX_DEPTH + 1), **i32), torch.zeros((B, 4), **i32)
    return s


def _prepare_embed(case, seed):
    s = _State()
    s.case, dt = case, DTYPES[case["dtype"]]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def randn(*shape, std=1.0):
        return (torch.randn(shape, generator=g, device="cuda") * std).to(dt)

    s.hidden = randn(case["B"], case["H_in"])
    s.router_w = randn(case["n_expert"], case["H_in"], std=2.0 / math.sqrt(case["H_in"]))
    s.router_b = randn(case["n_expert"]) if case["bias"] else None
    s.experts = randn(case["n_expert"], case["H_out"])
    s.out = torch.zeros((case["B"], case["H_out"]), dtype=dt, device="cuda")
    s.sel = torch.zeros((case["B"], case["k_expert"]), dtype=torch.int32, device="cuda")
    s.gate = torch.zeros((case["B"], case["k_expert"]), dtype=torch.float32, device="cuda")
    s.status = torch.zeros(case["B"], dtype=torch.int32, device="cuda")
    s.ctx = cb.confu_create(0)
    return s


def prepare(case, seed):
    s = {"step": _prepare_step, "attention": _prepare_attention, "accept": _prepare_accept, "embed": _prepare_embed}[case["kind"]](case, seed)
    s.kind = case["kind"]
    return s


# ------------------------------------------------------------------------------------ one pass
def run(s):
    if s.kind == "step":
        if s.case["graph"]:
            s.replay.replay()
        else:
            _step_calls(s)
        st = s.step
        # the attention outputs and decisions of the step, and the cache it has updated in place
        return {"out": s.out, "accept_len": st.accept_len, "path": st.path, "next_token": st.next_token, "future_row": st.future_row,
                "counters": st.counters, "new_prefix_len": st.new_prefix_len, "status": st.status, "k": s.k, "v": s.v}
    if s.kind == "attention":
        cb.confu_tree_attention(s.ctx, s.dims, s.q[0], s.k[0], s.v[0], s.n_slots, s.seq_start, s.plen,
                                s.ks[0] if s.ks is not None else None, s.vs[0] if s.vs is not None else None,
                                s.parent, s.owner, s.plan, s.out[0], s.lse, s.status)
        return {"out": s.out, "lse": s.lse, "status": s.status}
    if s.kind == "accept":
        c = s.case
        args = (s.accept_len, s.path, s.next_token, s.future_row, s.counters)
        sampled = c["temperature"] > 0
        if c["rule"] == "match":
            cb.confu_tree_accept_match(s.ctx, c["B"], c["T"], c["C"], c["V"], s.tl.dtype, s.tl, s.tokens, s.parent, s.owner,
                                       s.uniforms if sampled else None, c["temperature"], *args, s.status)
        else:
            cb.confu_tree_accept(s.ctx, c["B"], c["T"], c["C"], c["V"], s.tl.dtype, s.tl, s.dl if sampled else None, s.tokens, s.parent,
                                 s.owner, s.uniforms if sampled else None, c["temperature"],
                                 1 | (cb.ACCEPT_LAZY if c["rule"] == "lazy" else 0), *args, s.ws, s.status)
        return {"accept_len": s.accept_len, "path": s.path, "next_token": s.next_token, "future_row": s.future_row,
                "counters": s.counters, "status": s.status}
    c = s.case
    cb.confu_con_embedding(s.ctx, s.hidden, s.router_w, s.router_b, s.experts, c["k_expert"], c["renormalize"], s.out, s.sel, s.gate, s.status)
    return {"out": s.out, "sel": s.sel, "gate": s.gate, "status": s.status}


# ------------------------------------------------------------------------------------ what a pass cannot do without
def _accept_bytes(case):
    """Every row of the target matrix (and of the draft matrix when sampling) by the rule's default form; with statistics
    on demand and by the match rule the rows of a short walk, two nodes."""
    row = case["V"] * BYTES[case["logits"]] * case["B"]
    if case["rule"] == "match":
        return 2 * row
    mats = 2 if case["temperature"] > 0 else 1
    return mats * row * (min(2, case["T"]) if case["rule"] == "lazy" else case["T"])


def work(case):
    if case["kind"] == "embed":
        e = BYTES[case["dtype"]]
        out = case["B"] * case["H_out"] * e
        read = (case["B"] + case["n_expert"]) * case["H_in"] * e + min(case["n_expert"], case["B"] * case["k_expert"]) * case["H_out"] * e
        return {"bytes": read + out, "flops": 2.0 * case["B"] * (case["n_expert"] * case["H_in"] + case["k_expert"] * case["H_out"])}
    if case["kind"] == "accept":
        n = _accept_bytes(case)
        return {"bytes": n, "flops": 3.0 * n / BYTES[case["logits"]]}
    plen = [int(p) for p in _lengths(case)]
    R, e = case["T"] + case["C"], BYTES[case["kv"]]
    row = case["Hkv"] * case["D"] * e                       # K or V of one slot
    io = 2 * len(plen) * R * case["Hq"] * case["D"] * (2 if case["kv"] == "e4m3" else e)
    layer = 2 * row * (sum(plen) + len(plen) * R + case["S"]) + io
    keys = sum(case["T"] * (p + 4) + case["C"] * (p + 5 + case["S"]) for p in plen)         # a tree row sees about four tree rows
    flops = 4.0 * keys * case["Hq"] * case["D"]
    if case["kind"] == "attention":
        return {"bytes": layer, "flops": flops}
    if case["append"]:
        layer += 2 * len(plen) * R * case["Hkv"] * case["D"] * ((2 if case["kv"] == "e4m3" else e) + e)
    return {"bytes": case["L"] * layer + _accept_bytes(case), "flops": case["L"] * flops}


def tolerance(case):
    if case["kind"] == "accept":
        return "exact"
    kind = case["dtype"] if case["kind"] == "embed" else case["kv"]
    return {"bf16": {"rel": 1e-2}, "fp32": {"rel": 1e-5}, "e4m3": {"rel": 3e-2}}[kind]
