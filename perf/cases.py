"""The work that a user of this framework has it do, as timed cases.

Every case is one pass through `paper_2510_26577_b200.binding.CastContext`, called the way a decoding loop calls it
(one context per engine, device tensors in, device tensors out, nothing captured, nothing synchronised):

  step       one whole draft-and-verify step: tree build, every layer's verification attention, acceptance, compaction
  tree       the draft tree alone: begin, H expansion layers, rerank
  attention  the verification attention of some layers of the target model on a given batch of trees
  draft      the draft model's attention while the tree grows: the rows of one tree layer per call
  accept     what follows the target's forward at temperature 0: greedy acceptance and compaction of all layers
  sample     the same at temperature > 0: accept-or-resample and compaction

Shapes are those of `workloads.CONFIGS`, of the tests and of the paper's hyper-parameters, or generic ones around them.
"""
import numpy as np
import torch

from paper_2510_26577_b200 import binding

DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}
SIZE = {"f32": 4, "bf16": 2}
STD = 3.0  # standard deviation of the logits' bulk

# Cost tables on a grid of 512 positions x 128 tokens: a slowly rising latency in context and in verified tokens.
GRID, ROWS, COLS, SLOPE = 512, 64, 128, 1.4e-4


def _case(kind, name=None, **kw):
    c = {} if name is None else {"name": name}
    c.update(kind=kind, **kw)
    return c


def _logits(vocab, logits, depth, top_k, total, sizing="fixed"):
    return {"vocab": vocab, "logits": logits, "depth": depth, "top_k": top_k, "total": total, "sizing": sizing}


def _cache(layers, dtype, q_heads, kv_heads, head_dim, page, lo, hi):
    return {"layers": layers, "kv": dtype, "q_heads": q_heads, "kv_heads": kv_heads, "head_dim": head_dim, "page": page,
            "prefix_lo": lo, "prefix_hi": hi}


def listed():
    return [
        # a toy model in 32 bits, as in a smoke test or on a developer's first run: launches and latency only
        _case("step", "step_tiny_f32", batch=1, **_logits(4096, "f32", 4, 4, 16), **_cache(2, "f32", 8, 8, 64, 0, 256, 256)),
        # one interactive user of an 8B model: all 32 layers, fixed tree of 60 tokens
        _case("step", "step_b1", batch=1, **_logits(128256, "f32", 6, 10, 60), **_cache(32, "bf16", 32, 8, 128, 0, 2048, 2048)),
        # a moderately loaded server: 16 ragged sequences in a paged cache, tree sizes from the cost model, 8 of the layers
        _case("step", "step_b16_paged", batch=16, **_logits(128256, "f32", 6, 8, 64, "cost"),
              **_cache(8, "bf16", 32, 8, 128, 16, 512, 4096)),
        # the paper's own hyper-parameters at batch 1 (depth 13, top 12, 72 tokens), half-precision draft logits,
        # all three sizing rules on: a long chain of small launches
        _case("tree", "tree_b1_deep", batch=1, **_logits(32000, "bf16", 13, 12, 72, "all")),
        # the largest batch: the logits of a draft layer are hundreds of megabytes
        _case("tree", "tree_b64", batch=64, **_logits(128256, "f32", 6, 8, 64, "cost")),
        # the verification attention of a loaded server: 64 ragged paged sequences with small trees, bound by the cache
        _case("attention", "attention_b64", batch=64, total=12, ragged=True, **_cache(2, "bf16", 32, 8, 128, 16, 512, 4096)),
        # wide trees on a 70B model's heads, contiguous cache: bound by the tensor cores
        _case("attention", "attention_wide", batch=8, total=128, ragged=False, **_cache(4, "bf16", 64, 8, 128, 0, 4096, 4096)),
        # long context, a GQA group of seven
        _case("attention", "attention_long", batch=4, total=96, ragged=False, **_cache(2, "bf16", 28, 4, 128, 16, 32768, 32768)),
        # heads of 64 dimensions (small models), ragged sequences
        _case("attention", "attention_d64", batch=8, total=48, ragged=True, **_cache(4, "bf16", 32, 8, 64, 16, 512, 2048)),
        # the one-layer draft model's attention, layer after layer of the growing tree
        _case("draft", "draft_b4", batch=4, depth=6, top_k=8, **_cache(1, "bf16", 32, 8, 128, 16, 512, 4096)),
        # the end of a greedy step of a server with half-precision target logits: acceptance, then all 32 layers' caches
        _case("accept", "accept_b16", batch=16, **_logits(128256, "bf16", 6, 8, 24), **_cache(32, "bf16", 32, 8, 128, 16, 128, 1024)),
        # the end of a step at temperature 0.8
        _case("sample", "sample_b16", batch=16, temperature=0.8, **_logits(128256, "f32", 6, 8, 24),
              **_cache(32, "bf16", 32, 8, 128, 16, 128, 1024)),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(lo * (hi / lo) ** rng.random())))


def _draw_once(rng):
    kind = rng.choice(["step", "tree", "attention", "attention", "draft", "accept", "sample"])
    batch = _log_int(rng, 1, 64)
    top_k = rng.randint(2, 16)
    lg = _logits(rng.choice([32000, 50257, 128256, 152064, _log_int(rng, 4096, 152064), _log_int(rng, 4096, 152064) | 1]),
                 rng.choice(["f32", "bf16"]), rng.randint(3, 13), top_k, rng.randint(8, 128), rng.choice(["fixed", "cost", "all"]))
    kv = "f32" if rng.random() < 0.15 else "bf16"
    group = rng.choice([1, 2, 4, 4, 7, 8])
    kv_heads = rng.choice([1, 2, 4, 8, 8])
    head_dim = 64 if kv == "f32" or rng.random() < 0.25 else 128
    hi = _log_int(rng, 64, 32768)
    lo = hi if rng.random() < 0.3 else max(1, hi // rng.randint(2, 8))
    ca = _cache(_log_int(rng, 1, 32), kv, group * kv_heads, kv_heads, head_dim, rng.choice([0, 8, 16, 16, 32, 64]), lo, hi)
    if kind == "tree":
        return _case(kind, batch=batch, **lg)
    if kind == "attention":
        return _case(kind, batch=batch, total=_log_int(rng, 4, 128), ragged=rng.random() < 0.5, **ca)
    if kind == "draft":
        ca["layers"] = 1
        return _case(kind, batch=batch, depth=rng.randint(3, 9), top_k=min(top_k, 12), **ca)
    if kind in ("accept", "sample"):
        lg["sizing"] = "fixed"
        ca["prefix_lo"], ca["prefix_hi"] = min(lo, 1024), min(hi, 1024)
    if kind == "sample":
        return _case(kind, batch=batch, temperature=rng.choice([0.5, 0.8, 1.0, 1.2]), **lg, **ca)
    return _case(kind, batch=batch, **lg, **ca)


def _cost(case):
    """A rough cost, for the bound on drawn cases: bytes, or operations at what the type's units do per byte of memory."""
    w = work(case)
    per = 15 if case.get("kv") == "f32" else 50 if case.get("head_dim") == 64 else 200
    room = _cache_bytes(case) + _logit_rows(case) * case.get("vocab", 0) * SIZE[case.get("logits", "f32")]
    return max(w["bytes"], w["flops"] / per), room


def draw(rng):
    most = max(_cost(c)[0] for c in listed())
    while True:
        c = _draw_once(rng)
        cost, room = _cost(c)
        if cost <= most and room <= 8e9:
            return c


# ---------------------------------------------------------------------------------------------------- inputs
def _generators(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g, np.random.Generator(np.random.Philox(seed))


def _randn(shape, dtype, gen, std=1.0):
    x = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32 if std != 1.0 else DTYPE[dtype])
    return x if std == 1.0 else x.mul_(std).to(DTYPE[dtype])


def _draft_logits(case, gen, rows):
    """A draft head's logits: a Gaussian bulk and one likely token per row (probability about 0.3 to 0.9)."""
    shape = (case["batch"], rows, case["vocab"])
    x = torch.randn(shape, generator=gen, device="cuda").mul_(STD)
    likely = torch.randint(0, case["vocab"], shape[:2] + (1,), generator=gen, device="cuda")
    odds = torch.rand(shape[:2] + (1,), generator=gen, device="cuda") * 3.2 - 0.9
    x.scatter_(2, likely, odds + float(np.log(case["vocab"]) + STD * STD / 2))
    return x.to(DTYPE[case["logits"]])


def _trees(case, rng, depth, n_tree):
    """Random rooted trees in creation order: tokens, parents, depths [B, total] and ancestor masks (host arrays)."""
    B, cap, vocab = case["batch"], case["total"], case.get("vocab", 32000)
    tokens, parent, level = (np.full((B, cap), -1, np.int32) for _ in range(3))
    anc = np.zeros((B, cap, (cap + 31) // 32), np.uint32)
    for b in range(B):
        tok = (rng.integers(vocab) + np.arange(cap) * rng.integers(1, vocab // 128)) % vocab  # distinct, so siblings differ
        for t in range(int(n_tree[b])):
            p = -1 if t == 0 else int(min(rng.integers(0, t), rng.integers(0, t)))  # early nodes have more children
            while p >= 0 and level[b, p] >= depth:
                p = parent[b, p]
            tokens[b, t], parent[b, t], level[b, t] = tok[t], p, 0 if p < 0 else level[b, p] + 1
            if p >= 0:
                anc[b, t] = anc[b, p]
            anc[b, t, t >> 5] |= np.uint32(1 << (t & 31))
    return tokens, parent, level, anc


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _int(*shape):
    return torch.zeros(shape, dtype=torch.int32, device="cuda")


def _capacity(case, tokens):
    """Positions reserved per sequence, in whole pages."""
    unit = case["page"] or 1
    return -(-(case["prefix_hi"] + tokens) // unit) * unit


def _cache_bytes(case):
    if "layers" not in case:
        return 0
    return 2 * case["layers"] * case["batch"] * _capacity(case, 128) * case["kv_heads"] * case["head_dim"] * SIZE[case["kv"]]


def _logit_rows(case):
    """Logit rows that a state of the case holds."""
    draft = case["batch"] * case["depth"] * case["top_k"] if case["kind"] in ("step", "tree") else 0
    target = case["batch"] * case["total"] if case["kind"] in ("step", "accept", "sample") else 0
    return draft + (2 * target if case["kind"] == "sample" else target)


class State:
    pass


def _context(case, s, early):
    sizing = case.get("sizing", "fixed")
    kw = dict(max_batch=case["batch"], vocab=case.get("vocab", 32000), top_k=case.get("top_k", 8),
              max_depth=case.get("depth", 8), total_token=s.total, max_tree=s.total)
    if sizing != "fixed":
        kw.update(enable_bp=1, enable_dr=1)
    if sizing == "all":
        kw.update(enable_dp=1)
    s.ctx = binding.CastContext(**kw)
    if sizing != "fixed":
        B, n = case["batch"], np.arange(1, COLS + 1, dtype=np.float64)[None, :]
        c = (np.arange(1, ROWS + 1, dtype=np.float64) * GRID)[:, None]
        target = 1.0 + 0.25 * B * c / (64.0 * 4096.0) + SLOPE * B * n
        s.ctx.cast_set_cost_tables(B, GRID, ROWS, COLS, target, 0.05 * target)
    if early:  # a decoding loop: between two layers' attention nothing writes the tree, the lengths or the prefix rows
        s.ctx.cast_set_attention_early_reads(True)


def _prepare_cache(case, s, gen, rng, tokens):
    B, nl, unit = case["batch"], case["layers"], case["page"] or 1
    positions = _capacity(case, tokens)
    s.seq_cap, s.pages, s.table = positions // unit, 0, None
    if case["page"]:
        s.pages = B * s.seq_cap
        s.table = _dev(rng.permutation(s.pages).astype(np.int32).reshape(B, s.seq_cap))
    shape = (nl, s.pages, unit) if case["page"] else (nl, B, positions)
    shape += (case["kv_heads"], case["head_dim"])
    s.k, s.v = _randn(shape, case["kv"], gen), _randn(shape, case["kv"], gen)
    s.stride = s.k[0].numel() * s.k.element_size()
    s.kv0 = _dev(rng.integers(case["prefix_lo"], case["prefix_hi"] + 1, B).astype(np.int32))
    s.kv_len = s.kv0.clone()


def _prepare_queries(case, s, gen):
    s.q = _randn((case["layers"], case["batch"], s.total, case["q_heads"], case["head_dim"]), case["kv"], gen)
    s.out = torch.zeros_like(s.q)
    s.ctx.cast_reserve_attention(s.q.dtype, case["batch"], case["q_heads"], case["kv_heads"], case["head_dim"], case["page"],
                                 s.seq_cap)


def _prepare_tree(case, s, gen):
    B, H, K = case["batch"], case["depth"], case["top_k"]
    s.draft = [_draft_logits(case, gen, K) for _ in range(H)]
    s.root = torch.randint(0, case["vocab"], (B,), generator=gen, device="cuda", dtype=torch.int32)
    s.next_tokens, s.next_rows, s.next_count = _int(H, B, K), _int(H, B, K), _int(H, 1)
    s.tokens, s.parent, s.depth, s.pool_idx = (_int(B, s.total) for _ in range(4))
    s.anc, s.n_tree = _int(B, s.total, s.ctx.words), _int(B)
    s.scores = torch.zeros((B, s.total), dtype=torch.float64, device="cuda")


def _prepare_given_trees(case, s, rng, n_tree):
    tokens, parent, level, anc = _trees(case, rng, case.get("depth", 8), n_tree)
    s.tokens, s.parent, s.depth, s.anc = _dev(tokens), _dev(parent), _dev(level), _dev(anc.view(np.int32))
    s.n_tree = _dev(n_tree.astype(np.int32))
    return tokens, parent


def _prepare_accept(case, s):
    B, H = case["batch"], case["depth"]
    s.accept_len, s.accept_path, s.bonus = _int(B), _int(B, H + 1), _int(B)


def _favour_children(logits, tokens, parent, rng, chosen_only):
    """Raise the logits of children's tokens at their parents' rows: of all children, eldest highest, as in a draft head's
    rows, or (chosen_only) of one child of about seven nodes in ten, as where the target agrees with the draft."""
    at = []
    for b in range(tokens.shape[0]):
        kids = {}
        for t in range(1, tokens.shape[1]):
            if parent[b, t] >= 0:
                kids.setdefault(int(parent[b, t]), []).append(t)
        for p, cs in kids.items():
            if not chosen_only:
                at += [(b, p, tokens[b, c], STD * 5.5 - 0.5 * j) for j, c in enumerate(cs)]
            elif rng.random() < 0.7:
                c = cs[min(int(rng.geometric(0.6)) - 1, len(cs) - 1)]
                at.append((b, p, tokens[b, c], STD * 6.5))
    if at:
        b, p, t, v = (np.array(x) for x in zip(*at))
        logits[_dev(b), _dev(p), _dev(t).long()] = _dev(v).to(logits.dtype)


def prepare(case, seed):
    gen, rng = _generators(seed)
    kind, B = case["kind"], case["batch"]
    s = State()
    s.case = case
    s.total = 1 + (case["depth"] - 1) * case["top_k"] if kind == "draft" else case["total"]
    case = dict(case, total=s.total)
    _context(case, s, early=kind in ("step", "attention"))
    if kind in ("step", "tree"):
        _prepare_tree(case, s, gen)
    if kind == "tree":
        s.kv_len = _dev(rng.integers(512, 4097, B).astype(np.int32))
        return s
    _prepare_cache(case, s, gen, rng, s.total)
    if kind == "step":
        _prepare_queries(case, s, gen)
        _prepare_accept(case, s)
        s.target = _randn((B, s.total, case["vocab"]), case["logits"], gen, STD)
        _build_tree(s)  # once, for the tree whose tokens the target is made to agree with
        _favour_children(s.target, s.tokens.cpu().numpy(), s.parent.cpu().numpy(), rng, chosen_only=True)
    elif kind == "attention":
        n = rng.integers(max(1, s.total // 2), s.total + 1, B) if case["ragged"] else np.full(B, s.total)
        _prepare_given_trees(case, s, rng, n)
        _prepare_queries(case, s, gen)
    elif kind == "draft":
        _prepare_given_trees(case, s, rng, np.full(B, s.total))
        _prepare_queries(case, s, gen)
        ends = [1 + i * case["top_k"] for i in range(case["depth"])]  # tokens up to and including every layer
        s.ends = [_int(B).fill_(e) for e in ends]
        s.starts = [_int(B).fill_(e) for e in [0] + ends[:-1]]
    else:
        tokens, parent = _prepare_given_trees(case, s, rng, np.full(B, s.total))
        _prepare_accept(case, s)
        shape = (B, s.total, case["vocab"])
        if kind == "accept":
            s.target = _randn(shape, case["logits"], gen, STD)
            _favour_children(s.target, tokens, parent, rng, chosen_only=True)
        else:
            draft = torch.randn(shape, generator=gen, device="cuda").mul_(STD)
            _favour_children(draft, tokens, parent, rng, chosen_only=False)
            target = torch.randn(shape, generator=gen, device="cuda").mul_(0.7).add_(draft)
            s.target, s.draft = target.to(DTYPE[case["logits"]]), draft.to(DTYPE[case["logits"]])
            s.u_accept, s.u_bonus = _dev(rng.uniform(1e-12, 1 - 1e-12, (B, s.total))), _dev(rng.uniform(1e-12, 1 - 1e-12, B))
            s.ctx.cast_accept_stochastic_plan(s.target.dtype)
    return s


# ---------------------------------------------------------------------------------------------------- one pass
def _build_tree(s):
    ctx = s.ctx
    ctx.cast_step_begin(s.case["batch"], s.root, s.kv_len)
    for i in range(s.case["depth"]):
        ctx.cast_tree_expand(i + 1, s.draft[i], s.next_tokens[i], s.next_rows[i], s.next_count[i])
    ctx.cast_select_nodes(s.tokens, s.parent, s.depth, s.anc, s.pool_idx, s.scores, s.n_tree)
    return {"next_tokens": s.next_tokens, "next_rows": s.next_rows, "next_count": s.next_count, "tokens": s.tokens,
            "parent": s.parent, "depth": s.depth, "anc": s.anc, "pool_idx": s.pool_idx, "scores": s.scores, "n_tree": s.n_tree}


def _attend(s):
    c = s.case
    for layer in range(c["layers"]):
        s.ctx.cast_tree_attention(s.q[layer], s.k[layer], s.v[layer], c["batch"], c["q_heads"], c["kv_heads"], c["head_dim"],
                                  c["page"], s.table, s.seq_cap, s.pages, s.kv_len, s.anc, s.n_tree, 0.0, s.out[layer])
    return {"attention": s.out}


def _finish(s):
    c = s.case
    if c["kind"] == "sample":
        s.ctx.cast_accept_stochastic(s.target, s.draft, c["batch"], c["temperature"], s.tokens, s.parent, s.n_tree, s.u_accept,
                                     s.u_bonus, s.accept_len, s.accept_path, s.bonus)
    else:
        s.ctx.cast_accept(s.target, c["batch"], s.tokens, s.parent, s.depth, s.anc, s.n_tree, s.accept_len, s.accept_path,
                          s.bonus)
    s.ctx.cast_compact_kv(s.k, s.v, c["batch"], c["layers"], s.stride, c["kv_heads"], c["head_dim"], c["page"], s.table,
                          s.seq_cap, s.pages, s.accept_path, s.accept_len, s.kv_len)
    return {"accept_len": s.accept_len, "accept_path": s.accept_path, "bonus": s.bonus, "kv_len": s.kv_len, "k": s.k, "v": s.v}


def run(s):
    c = s.case
    if c["kind"] == "tree":
        return _build_tree(s)
    if c["kind"] == "attention":
        return _attend(s)
    if c["kind"] == "draft":
        for end, start in zip(s.ends, s.starts):
            s.ctx.cast_tree_attention_rows(s.q[0], s.k[0], s.v[0], c["batch"], c["q_heads"], c["kv_heads"], c["head_dim"],
                                           c["page"], s.table, s.seq_cap, s.pages, s.kv_len, s.anc, end, start, 0.0, s.out[0])
        return {"attention": s.out}
    s.kv_len.copy_(s.kv0)  # compaction advances the lengths in place: a pass starts from the same prefix as the one before
    if c["kind"] == "step":
        return {**_build_tree(s), **_attend(s), **_finish(s)}
    return _finish(s)


# ---------------------------------------------------------------------------------------------------- bounds
def _tree_rows(case):
    """Draft rows that are read per sequence: the root's, then those of the retained nodes (with these logits the cost rule
    keeps a layer's full width; depth pruning ends most trees after eight layers or so)."""
    layers = min(case["depth"], 8) if case["sizing"] == "all" else case["depth"]
    return 1 + (layers - 1) * case["top_k"]


def _attention_work(case, tokens, calls):
    """Of `calls` layers: each sequence's keys and values, queries and outputs once; two products per visible pair."""
    B, prefix = case["batch"], (case["prefix_lo"] + case["prefix_hi"]) / 2
    size, row = SIZE[case["kv"]], case["head_dim"]
    return {"bytes": calls * B * size * row * (2 * (prefix + tokens) * case["kv_heads"] + 2 * tokens * case["q_heads"]),
            "flops": calls * B * 4 * tokens * case["q_heads"] * row * (prefix + 4)}


def work(case):
    kind, B = case["kind"], case["batch"]
    parts = []
    if kind in ("step", "tree"):
        parts.append({"bytes": B * _tree_rows(case) * case["vocab"] * SIZE[case["logits"]], "flops": 0})
    if kind == "draft":
        parts.append(_attention_work(case, case["top_k"], case["depth"]))
    if kind == "attention":
        parts.append(_attention_work(case, case["total"] * (0.75 if case["ragged"] else 1.0), case["layers"]))
    tokens = case.get("total", 0)
    if kind == "step":
        tokens = tokens if case["sizing"] == "fixed" else min(tokens, 1100 / B)  # what these cost tables let a batch verify
        parts.append(_attention_work(case, tokens, case["layers"]))
    if kind in ("step", "accept", "sample"):
        rows = tokens if kind != "sample" else 2 * min(4, case["depth"])  # sampling reads the accepted path's rows only
        moved = 2 * case["layers"] * 3 * case["kv_heads"] * case["head_dim"] * SIZE[case["kv"]]  # about three rows each
        parts.append({"bytes": B * (rows * case["vocab"] * SIZE[case["logits"]] + 2 * moved), "flops": 0})
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def tolerance(case):
    if case["kind"] in ("accept", "sample"):
        return "exact"  # comparisons, fp64 sampling and copies of cache rows
    if case["kind"] != "tree" and case["kv"] == "bf16":
        return {"rel": 1e-2}
    return {"rel": 1e-5}  # log-values over an fp32 log-sum-exp; 32-bit attention
