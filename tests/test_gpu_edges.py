"""The edges of single kernels' tilings and dispatch rules: first and last elements of unaligned rows, remainders of
tiles, the smallest and largest sizes of a range. Each against the CPU oracle or a plain statement of the result."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2510_26577_b200 import build
    build.build()
    from paper_2510_26577_b200 import binding as b
    b.load_library()
    return b


def _ints(a):
    return torch.tensor(a, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V", [5, 4096, 4099, 16385, 50257, 65537])
def test_accept_winner_at_the_ends_of_unaligned_rows(binding, dtype, V):
    """A star of N - 1 children under the root: the root's row and every other row have their maximum at the first or the
    last token, at a chunk's or vector's edge, twice (the lower id wins), or nowhere (all -inf: token 0)."""
    N = 12
    g = torch.Generator(device="cuda").manual_seed(V)
    logits = torch.randn((1, N, V), generator=g, device="cuda").to(dtype)
    where = [0, V - 1, 1, V - 2, V // 2, min(7, V - 1), min(8, V - 1), (V // 8) * 8 - 1 if V > 8 else 0]
    want = []
    for t in range(N):
        if t < len(where):
            logits[0, t, where[t]] = 30.0
            want.append(where[t])
        elif t == len(where):  # two equal maxima
            logits[0, t, V - 1] = logits[0, t, V // 3] = 30.0
            want.append(V // 3)
        elif t == len(where) + 1:
            logits[0, t] = float("-inf")
            want.append(0)
        else:
            want.append(int(logits[0, t].float().argmax()) if t != N - 1 else -1)
    logits[0, N - 1] = logits[0, N - 1].abs().neg()  # a zero of either sign at the top
    logits[0, N - 1, V - 1], logits[0, N - 1, V // 4] = 0.0, -0.0
    want[N - 1] = V // 4
    got = []
    for t in range(N):  # the bonus token of a one-node tree is the argmax of its row
        ctx = binding.CastContext(max_batch=1, vocab=V, top_k=1, max_depth=2, total_token=1, max_tree=1)
        n, p, b = _ints([0]), _ints([[0, 0, 0]]), _ints([0])
        ctx.cast_accept(logits[:, t:t + 1].contiguous() if t % 2 else logits[:, t:t + 1], 1, _ints([[0]]), _ints([[-1]]), None,
                        None, _ints([1]), n, p, b)
        assert ctx.cast_poll_status()[0] == 0
        got.append(int(b.item()))
    assert got == want


@pytest.mark.parametrize("Hkv,D,dtype", [(1, 64, torch.bfloat16), (3, 64, torch.float32), (8, 128, torch.bfloat16),
                                         (8, 128, torch.float32), (5, 8, torch.bfloat16)])
@pytest.mark.parametrize("path", [[0], [0, 1, 2], [0, 2, 3], [0, 1, 2, 3, 5, 9, 11, 12, 13, 20, 21, 22, 23, 24, 25, 26, 30]])
def test_compaction_of_whole_position_rows(binding, Hkv, D, dtype, path):
    """Row widths from a few vectors to several CTAs, paths of one node, in place, overlapping, and of the largest depth."""
    H, NL, page, cap = 16, 3, 4, 16
    ctx = binding.CastContext(max_batch=2, vocab=100, top_k=2, max_depth=H, total_token=32, max_tree=32)
    g = torch.Generator(device="cuda").manual_seed(1)
    shape = (NL, 2 * cap, page, Hkv, D)
    k, v = (torch.randn(shape, generator=g, device="cuda").to(dtype) for _ in range(2))
    table = torch.randperm(2 * cap, generator=torch.Generator().manual_seed(2)).to(torch.int32).view(2, cap)
    kv_len = [9, 0]
    ref = [x.clone() for x in (k, v)]
    rows = lambda b, pos: (int(table[b, pos // page]), pos % page)
    for x in ref:
        old = x.clone()
        for b in range(2):
            for j, src in enumerate(path):
                x[(slice(None),) + rows(b, kv_len[b] + j)] = old[(slice(None),) + rows(b, kv_len[b] + src)]
    lens = _ints(kv_len)
    full = path + [-1] * (H + 1 - len(path))
    ctx.cast_compact_kv(k, v, 2, NL, k[0].numel() * k.element_size(), Hkv, D, page, table.cuda(), cap, 2 * cap,
                        _ints([full, full]), _ints([len(path) - 1] * 2), lens)
    assert ctx.cast_poll_status()[0] == 0
    assert torch.equal(k, ref[0]) and torch.equal(v, ref[1])
    assert lens.tolist() == [x + len(path) for x in kv_len]


def _attention_reference(q, k, v, page, table, kv_len, anc, n_tree, first=None):
    """fp64 softmax attention on the device, one sequence at a time (rows outside [first, n_tree) stay NaN)."""
    B, _, Hq, D = q.shape
    out = torch.full(q.shape, float("nan"), dtype=torch.float64, device="cuda")
    for b in range(B):
        N, L = int(n_tree[b]), int(kv_len[b])
        pos = torch.arange(L + N, device="cuda")
        idx = (table[b].long()[pos // page] * page + pos % page) if page else b * k.shape[1] + pos
        kk, vv = (x.reshape(-1, x.shape[-2], D)[idx].double().repeat_interleave(Hq // x.shape[-2], 1) for x in (k, v))
        s = torch.einsum("thd,phd->htp", q[b, :N].double(), kk) / D ** 0.5
        j = torch.arange(N, device="cuda")
        vis = ((anc[b, :N][:, j // 32] >> (j % 32)[None, :]) & 1).bool()
        s[:, :, L:] = s[:, :, L:].masked_fill(~vis[None], float("-inf"))
        f = 0 if first is None else int(first[b])
        out[b, f:N] = torch.einsum("htp,phd->thd", s.softmax(-1), vv)[f:]
    return out


def _random_trees(rng, B, cap, n_tree):
    anc = np.zeros((B, cap, (cap + 31) // 32), np.uint32)
    for b in range(B):
        for t in range(n_tree[b]):
            if t:
                anc[b, t] = anc[b, int(rng.integers(max(0, t - 6), t))]
            anc[b, t, t // 32] |= np.uint32(1 << (t % 32))
    return torch.from_numpy(anc.view(np.int32)).cuda()


def _attend(binding, rng, B, cap, n_tree, Hq, Hkv, D, page, kv, dtype=torch.bfloat16, gain=1.0, first=None, early=False,
            beyond=None, budget=None):
    """Device output and fp64 reference of one call. `beyond`: what the query rows past a tree hold; `budget`: total_token, where
    it is not the trees' capacity."""
    g = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 30)))
    unit = page or 1
    seq = -(-(max(kv) + cap) // unit)
    k, v = (torch.randn((B * seq, page, Hkv, D) if page else (B, seq, Hkv, D), generator=g, device="cuda").to(dtype)
            for _ in range(2))
    table = torch.randperm(B * seq, generator=g, device="cuda").to(torch.int32).view(B, seq) if page else None
    q = (torch.randn((B, cap, Hq, D), generator=g, device="cuda") * gain).to(dtype)
    if beyond is not None:
        for b, n in enumerate(n_tree):
            q[b, n:] = beyond
    anc, nt, kv_len = _random_trees(rng, B, cap, n_tree), _ints(n_tree), _ints(kv)
    ctx = binding.CastContext(max_batch=B, vocab=100, top_k=2, max_depth=4, total_token=budget or cap, max_tree=cap)
    ctx.cast_reserve_attention(dtype, B, Hq, Hkv, D, page, seq)
    if early:
        ctx.cast_set_attention_early_reads(True)
    out = torch.full_like(q, float("nan"))
    args = (q, k, v, B, Hq, Hkv, D, page, table, seq, B * seq if page else 0, kv_len, anc, nt)
    for _ in range(2 if early else 1):
        if first is None:
            ctx.cast_tree_attention(*args, 0.0, out)
        else:
            ctx.cast_tree_attention_rows(*args, _ints(first), 0.0, out)
    assert ctx.cast_poll_status()[0] == 0
    return out, _attention_reference(q, k, v, page, table, kv, anc, n_tree, first)


@pytest.mark.parametrize("B,cap,Hq,Hkv,page,kv", [
    (1, 1, 1, 1, 0, [0]), (1, 33, 8, 8, 0, [63]), (2, 128, 4, 1, 16, [64, 1]), (3, 32, 14, 2, 8, [65, 700, 0]),
    (1, 60, 32, 8, 16, [2048]), (4, 128, 64, 8, 0, [1500, 1400, 90, 1536]), (40, 12, 32, 8, 64, [37 * i for i in range(40)]),
    (5, 48, 16, 4, 32, [5000, 10, 3000, 64, 128])])
def test_attention_of_64_dims_rounds_only_its_output(binding, B, cap, Hq, Hkv, page, kv):
    """bf16 heads of 64 dims: the probabilities enter the second product with 16 bits, the partials of KV splits are fp32:
    the result is the exact one rounded to bf16 (2^-9 of the value) but for what the scores' fp32 sums leave."""
    rng = np.random.default_rng(B * 1000 + cap)
    n_tree = [int(rng.integers(max(1, cap // 2), cap + 1)) for _ in range(B)]
    for gain, first in ((1.0, None), (6.0, None), (1.0, [n // 3 for n in n_tree])):
        got, want = _attend(binding, rng, B, cap, n_tree, Hq, Hkv, 64, page, kv, gain=gain, first=first)
        keep = ~want.isnan()
        assert torch.equal(got.isnan(), ~keep)
        err = (got.double() - want)[keep].abs() - want[keep].abs() * 2.0 ** -8
        assert float(err.max()) < 2e-5 * gain


@pytest.mark.parametrize("V", [17, 8193, 32768, 32769, 65537, 131073, 155648, 155649, 196609])
@pytest.mark.parametrize("B,dtype,shift", [(1, torch.float32, 0.0), (12, torch.bfloat16, 0.0), (2, torch.float32, -2000.0),
                                           (10, torch.float32, 900.0)])
def test_stochastic_accept_at_the_steps_of_its_dispatch(binding, V, B, dtype, shift):
    """Vocabularies at the ends of a segment size, batches below and above what clusters of 16 cover at once, logits so far
    from zero that exp(logit / T) leaves fp64's range. A root with two children, the first of which has one."""
    from oracle import stochastic_accept
    rng = np.random.default_rng(V + B)
    N, H, T = 4, 3, 0.9
    g = torch.Generator(device="cuda").manual_seed(V)
    parent = np.tile(np.array([-1, 0, 0, 1], np.int32), (B, 1))
    tokens = np.stack([rng.permutation(V)[:N] if V > N else np.arange(N) for _ in range(B)]).astype(np.int32)
    draft = torch.randn((B, N, V), generator=g, device="cuda") * 3
    for b in range(B):
        for t, p in ((1, 0), (2, 0), (3, 1)):
            draft[b, p, int(tokens[b, t])] = 15.0 - t
    target = draft + 0.5 * torch.randn(draft.shape, generator=g, device="cuda") + shift
    target, draft = target.to(dtype), (draft + shift).to(dtype)
    n_tree = np.full(B, N, np.int32)
    ua, ub = rng.uniform(0.01, 0.99, (B, N)), rng.uniform(0.01, 0.99, B)
    ctx = binding.CastContext(max_batch=B, vocab=V, top_k=2, max_depth=H, total_token=N, max_tree=N)
    dev = lambda a: torch.from_numpy(a).cuda()
    n, path, bonus = _ints([0] * B), _ints([[0] * (H + 1)] * B), _ints([0] * B)
    ctx.cast_accept_stochastic(target, draft, B, T, dev(tokens), dev(parent), dev(n_tree), dev(ua), dev(ub), n, path, bonus)
    assert ctx.cast_poll_status()[0] == 0
    want_n, want_path, want_bonus, margin = stochastic_accept(target.double().cpu().numpy(), draft.double().cpu().numpy(), tokens,
                                                              parent, n_tree, H, T, ua, ub)
    clear = margin > 1e-11
    assert clear.any()
    for got, want in ((n, want_n), (path, want_path), (bonus, want_bonus)):
        assert np.array_equal(got.cpu().numpy()[clear], want[clear])


@pytest.mark.parametrize("V,B", [(4099, 1), (40000, 1), (128256, 1), (152064, 2), (190000, 1), (100001, 12), (128256, 12),
                                 (152064, 12)])
@pytest.mark.parametrize("dtype,T,top", [(torch.float32, 0.9, None), (torch.bfloat16, 1.3, None), (torch.float32, 0.7, 640.0),
                                         (torch.float32, 0.9, 689.9)])
def test_stochastic_accept_mixes_logits_within_and_beyond_the_limits(binding, V, B, dtype, T, top):
    """Groups of logits that hold what exp(logit / T) takes without a range test and what it does not: tokens that are ruled
    out (-inf), hardly possible ones (-1e4 T) and, with `top`, two likely ones at top * T, just inside the limit (their sum
    asks for the second evaluation or just does not). Segments of every size the kernel is compiled for."""
    from oracle import stochastic_accept
    rng = np.random.default_rng(V + B)
    N, H = 4, 3
    g = torch.Generator(device="cuda").manual_seed(V + B)
    parent = np.tile(np.array([-1, 0, 0, 1], np.int32), (B, 1))
    tokens = np.stack([rng.permutation(V)[:N] for _ in range(B)]).astype(np.int32)
    draft = torch.randn((B, N, V), generator=g, device="cuda") * 3
    target = draft + 0.5 * torch.randn(draft.shape, generator=g, device="cuda")
    for x, share, value in ((target, 1e-3, float("-inf")), (target, 1e-4, -1e4 * T), (draft, 1e-4, -1e4 * T)):
        x[torch.rand(x.shape, generator=g, device="cuda") < share] = value
    for b in range(B):
        for t, p in ((1, 0), (2, 0), (3, 1)):
            draft[b, p, int(tokens[b, t])] = 15.0 - t
            target[b, p, int(tokens[b, t])] = 14.0 - t
        if top is not None:
            target[b, :, V // 3] = top * T
            target[b, :, V - 1] = (top - 0.5) * T
    target, draft = target.to(dtype), draft.to(dtype)
    n_tree = np.full(B, N, np.int32)
    ua, ub = rng.uniform(0.01, 0.99, (B, N)), rng.uniform(0.01, 0.99, B)
    ctx = binding.CastContext(max_batch=B, vocab=V, top_k=2, max_depth=H, total_token=N, max_tree=N)
    dev = lambda a: torch.from_numpy(a).cuda()
    n, path, bonus = _ints([0] * B), _ints([[0] * (H + 1)] * B), _ints([0] * B)
    ctx.cast_accept_stochastic(target, draft, B, T, dev(tokens), dev(parent), dev(n_tree), dev(ua), dev(ub), n, path, bonus)
    assert ctx.cast_poll_status()[0] == 0
    want_n, want_path, want_bonus, margin = stochastic_accept(target.double().cpu().numpy(), draft.double().cpu().numpy(), tokens,
                                                              parent, n_tree, H, T, ua, ub)
    clear = margin > 1e-11
    assert clear.any()
    for got, want in ((n, want_n), (path, want_path), (bonus, want_bonus)):
        assert np.array_equal(got.cpu().numpy()[clear], want[clear])


def _sample_at_root(binding, target, draft, T, tokens, ua, ub):
    """Trees of a root and tokens.shape[1] - 1 children: accepted lengths, paths and bonus tokens, and the oracle's with margins."""
    from oracle import stochastic_accept
    B, N, V = target.shape
    parent = np.tile(np.array([-1] + [0] * (N - 1), np.int32), (B, 1))
    n_tree = np.full(B, N, np.int32)
    ctx = binding.CastContext(max_batch=B, vocab=V, top_k=2, max_depth=2, total_token=N, max_tree=N)
    dev = lambda a: torch.from_numpy(a).cuda()
    n, path, bonus = _ints([0] * B), _ints([[0] * 3] * B), _ints([0] * B)
    ctx.cast_accept_stochastic(target, draft, B, T, dev(tokens), dev(parent), dev(n_tree), dev(ua), dev(ub), n, path, bonus)
    assert ctx.cast_poll_status()[0] == 0
    want = stochastic_accept(target.double().cpu().numpy(), draft.double().cpu().numpy(), tokens, parent, n_tree, 2, T, ua, ub)
    return [x.cpu().numpy() for x in (n, path, bonus)], want[:3], want[3]


@pytest.mark.parametrize("V,B", [(4099, 8), (40000, 8), (128256, 5), (128256, 12), (200001, 4)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("top_p,top_q", [(32.0, -7.0), (-7.0, 32.0)])
def test_stochastic_accept_of_rows_far_apart(binding, V, B, dtype, top_p, top_q):
    """Temperature 0.05, one row's top logits at 32 (a sum of 1e278) and the other's at -7 (1e-61), each way round: both sums
    are within fp64's range, their quotient is not. The children are the tokens that the target likes least, to be rejected.
    The last vocabulary is one whose segments are not cached."""
    rng = np.random.default_rng(V + B)
    T, hot = 0.05, np.stack([rng.permutation(V)[:8] for _ in range(B)])
    rows = np.empty((2, B, 3, V))
    for x, top in zip(rows, (top_p, top_q)):
        x[:] = top - rng.uniform(4, 40, x.shape)
        step = 2.0 ** -2 if top > 0 else 2.0 ** -5  # (as fine as bf16 has them there)
        for b in range(B):
            x[b][:, hot[b]] = top - step * (rng.permutation(8) // 3)
    target, draft = (torch.from_numpy(x).to(dtype).cuda() for x in rows)
    t0, d0 = (np.take_along_axis(x[:, 0].double().cpu().numpy(), hot, 1) / T for x in (target, draft))
    worst = np.argsort(t0 - d0, axis=1)[:, :2]
    tokens = np.concatenate([np.zeros((B, 1)), np.take_along_axis(hot, worst, 1)], 1).astype(np.int32)
    ua, ub = rng.uniform(0.95, 0.999, (B, 3)), rng.uniform(0.01, 0.99, B)
    got, want, margin = _sample_at_root(binding, target, draft, T, tokens, ua, ub)
    clear = margin > 1e-9
    assert clear.sum() >= B // 2 and (want[0][clear] == 0).any()
    for g, w in zip(got, want):
        assert np.array_equal(g[clear], w[clear])


@pytest.mark.parametrize("V,B", [(4099, 64), (40000, 64), (128256, 4), (128256, 24), (200001, 16)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_stochastic_accept_of_rows_with_all_mass_on_one_token(binding, V, B, dtype):
    """Both rows of the root hold all their mass on the same token; the child is another one, with e^-60 of the draft's mass and
    none of the target's, and is rejected. What is left of P_T - P_D is 0 or the last bits of it: the bonus token is that token."""
    for seed in range(6):
        rng = np.random.default_rng(V + 1000 * seed)
        target, draft = (torch.full((B, 2, V), float("-inf"), dtype=dtype, device="cuda") for _ in range(2))
        at = np.stack([1 + rng.permutation(V - 1)[:2] for _ in range(B)])
        rows, hot, child = torch.arange(B, device="cuda"), torch.from_numpy(at[:, 0]).cuda(), torch.from_numpy(at[:, 1]).cuda()
        top = torch.from_numpy(rng.uniform(-5, 20, (2, B))).cuda().to(dtype)
        target[rows, 0, hot], draft[rows, 0, hot] = top[0], top[1]
        draft[rows, 0, child] = top[1] - 60.0
        tokens = np.stack([np.zeros(B), at[:, 1]], 1).astype(np.int32)
        got, want, _ = _sample_at_root(binding, target, draft, 1.0, tokens, rng.uniform(0.1, 0.9, (B, 2)), rng.uniform(0.1, 0.9, B))
        assert np.array_equal(want[2], at[:, 0])
        for g, w in zip(got, want):
            assert np.array_equal(g, w)


@pytest.mark.parametrize("V,B", [(65536, 8), (128256, 4), (128256, 24)])
@pytest.mark.parametrize("T", [0.05, 0.8, 3.0])
def test_stochastic_accept_exponentials_to_fp64_rounding(binding, V, B, T):
    """Two tokens of about equal mass, logits up to 600 T on either side of zero, all others 60 nats and more below (1e-22 of the
    mass): u just below the first one's share gives that token, just above it the second. The share is known to 40 digits. An
    exponential is off by 2^-52 (its table entry) + 2^-53 (its last step) + 0.011 * 2^-52 (the polynomial), the two sums, their
    folds, the scale and the goal by some ten roundings of 2^-53: 4e-15 is twice all that. An argument that carries its own
    rounding, as next to padding (which these vocabularies have at the end only), would be off by up to 600 * 2^-53 = 7e-14."""
    from decimal import Decimal, getcontext
    getcontext().prec = 40
    rng = np.random.default_rng(V + B)
    top = np.linspace(-600, 600, B) + rng.uniform(-5, 5, B)
    x = ((top[:, None] - rng.uniform(60, 80, (B, V))) * T).astype(np.float32)
    at = np.sort(np.stack([1 + rng.permutation(V * 9 // 10)[:2] for _ in range(B)]), axis=1)
    below, above = np.empty(B), np.empty(B)
    for b in range(B):
        x[b, at[b]] = (top[b] + rng.uniform(0, 1, 2)) * T
        first, second = (Decimal(float(v)) / Decimal(T) for v in x[b, at[b]])
        share = 1 / (1 + (second - first).exp())
        below[b], above[b] = (float(share * (1 + s * Decimal(4e-15))) for s in (-1, 1))
    x = x[:, None]
    target = torch.from_numpy(x).cuda()
    tokens, ua = np.zeros((B, 1), np.int32), np.full((B, 1), 0.5)
    for ub, want in ((below, at[:, 0]), (above, at[:, 1])):
        got, _, _ = _sample_at_root(binding, target, target, T, tokens, ua, ub)
        assert np.array_equal(got[2], want)


@pytest.mark.parametrize("logits", ["f32", "bf16"])
@pytest.mark.parametrize("V", [33, 8191, 16385, 32769, 65529, 131073, 262147])
@pytest.mark.parametrize("kind", ["random", "rising", "constant", "one_block", "few_finite"])
def test_tree_layer_at_the_edges_of_the_sweep(binding, logits, V, kind):
    """Vocabularies around the buffers' sizes (unaligned rows), values that overflow the candidate lists: a row that rises with
    the token, equal logits everywhere, all large logits in one thread's reach, hardly more finite ones than K."""
    from helpers import assert_tree_equal, gpu_tree, oracle_tree
    B, K, H = 2, 16, 2
    g = torch.Generator().manual_seed(V)
    dt = torch.bfloat16 if logits == "bf16" else torch.float32
    layers = []
    for _ in range(H):
        x = torch.randn((B, K, V), generator=g) * 3
        if kind == "rising":
            x = x.sort(-1).values
        elif kind == "constant":
            x = torch.full_like(x, -1.5)
        elif kind == "one_block":
            x[..., V // 2:V // 2 + 16] += torch.arange(16) * 0.5 + 40.0
        elif kind == "few_finite":
            keep = torch.zeros(V, dtype=torch.bool)
            keep[torch.randperm(V, generator=g)[:K + 1]] = True
            x[..., ~keep] = float("-inf")
        layers.append(x.to(dt))
    kw = dict(vocab=V, top_k=K, max_depth=H, total_token=40, max_tree=40)
    root, kv = torch.tensor([1, 2], dtype=torch.int32), torch.tensor([5, 6], dtype=torch.int32)
    want = oracle_tree(kw, None, root, kv, layers)
    ctx = binding.CastContext(max_batch=B, **kw)
    assert_tree_equal(gpu_tree(ctx, root.cuda(), kv.cuda(), [x.cuda() for x in layers]), want)


@pytest.mark.parametrize("dtype,D,page", [(torch.float32, 64, 16), (torch.float32, 128, 0), (torch.bfloat16, 128, 128)])
@pytest.mark.parametrize("B,cap,Hq,Hkv,kv", [(1, 1, 1, 1, [0]), (1, 32, 4, 1, [6000]), (2, 33, 6, 2, [1000, 3]), (3, 9, 8, 8, [64, 63, 500]),
                                             (64, 5, 8, 8, [(i * 29) % 300 for i in range(64)])])
def test_cuda_core_attention_merges(binding, dtype, D, page, B, cap, Hq, Hkv, kv):
    """One split, up to sixteen (merged by the last CTA), more (a kernel of its own), splits without tiles; windows."""
    rng = np.random.default_rng(B * 100 + cap)
    n_tree = [int(rng.integers(max(1, cap // 2), cap + 1)) for _ in range(B)]
    for first in (None, [n // 2 for n in n_tree]):
        got, want = _attend(binding, rng, B, cap, n_tree, Hq, Hkv, D, page, kv, dtype=dtype, first=first)
        keep = ~want.isnan()
        assert torch.equal(got.isnan(), ~keep)
        tol = 1e-5 if dtype == torch.float32 else 1e-5 + want[keep].abs() * 2.0 ** -8
        assert bool(((got.double() - want)[keep].abs() <= tol).all())


@pytest.mark.parametrize("dtype,page", [(torch.float32, 16), (torch.float32, 0), (torch.bfloat16, 128), (torch.bfloat16, 16)])
@pytest.mark.parametrize("Hq,kv", [(4, 70), (4, 2000), (1, 9)])
def test_attention_reports_a_tree_beyond_total_token(binding, dtype, page, Hq, kv):
    """n_tree of total_token, one more and max_tree, on the CUDA cores (splits merged by the last CTA or by a kernel of its
    own) and the tensor cores: BAD_TREE names the sequence, the rows of the first total_token tokens come, the rest stay."""
    B, cap, total, D = 3, 64, 40, 64
    rng = np.random.default_rng(kv)
    g = torch.Generator(device="cuda").manual_seed(kv)
    seq = -(-(kv + cap) // page) if page else kv + cap
    k, v = (torch.randn((B * seq, page, 1, D) if page else (B, seq, 1, D), generator=g, device="cuda").to(dtype) for _ in range(2))
    table = torch.arange(B * seq, device="cuda", dtype=torch.int32).view(B, seq) if page else None
    q = torch.randn((B, cap, Hq, D), generator=g, device="cuda").to(dtype)
    anc = _random_trees(rng, B, cap, [cap] * B)
    ctx = binding.CastContext(max_batch=B, vocab=100, top_k=2, max_depth=4, total_token=total, max_tree=cap)
    ctx.cast_reserve_attention(dtype, B, Hq, 1, D, page, seq)
    want = _attention_reference(q, k, v, page, table, [kv] * B, anc, [total] * B)
    for n_tree, status in (([total] * 3, (0, None)), ([total, total + 1, total], (6, 1)), ([total, 5, cap], (6, 2))):
        out = torch.full_like(q, float("nan"))
        ctx.cast_tree_attention(q, k, v, B, Hq, 1, D, page, table, seq, B * seq if page else 0, _ints([kv] * B), anc,
                                _ints(n_tree), 0.0, out)
        st, detail = ctx.cast_poll_status()
        assert st == status[0] and (st == 0 or detail == status[1])
        for b in range(B):
            n = min(n_tree[b], total)
            assert out[b, n:].isnan().all()
            # (a token sees its ancestors, all of them before it: the rows of a cut tree are those of the whole one)
            # (tolerances as above: fp32 sums, the output's rounding, two bf16 terms of P on the tensor cores)
            tol = 1e-5 if dtype == torch.float32 else 2e-5 + want[b, :n].abs() * 2.0 ** -8
            assert bool(((out[b, :n].double() - want[b, :n]).abs() <= tol).all())


def _early_setup(binding, B, cap, Hq, Hkv, D, page, kv, dtype=torch.bfloat16, share=None):
    """A context with the early-read promise and one layer's inputs: its attention call, and the state the call reads.
    share: another such context, its lengths and its tree sizes, to be used here too."""
    rng = np.random.default_rng(Hq * D)
    g = torch.Generator(device="cuda").manual_seed(Hq * D)
    seq = -(-(max(kv) + 2 * cap) // page)
    k, v = (torch.randn((B * seq, page, Hkv, D), generator=g, device="cuda").to(dtype) for _ in range(2))
    table = torch.randperm(B * seq, generator=g, device="cuda").to(torch.int32).view(B, seq)
    q = torch.randn((B, cap, Hq, D), generator=g, device="cuda").to(dtype)
    anc = _random_trees(rng, B, cap, [cap] * B)
    if share is None:
        ctx = binding.CastContext(max_batch=B, vocab=100, top_k=2, max_depth=4, total_token=cap, max_tree=cap)
        ctx.cast_set_attention_early_reads(True)
        kv_len, n_tree = _ints(kv), _ints([cap] * B)
    else:
        ctx, kv_len, n_tree = share
    ctx.cast_reserve_attention(dtype, B, Hq, Hkv, D, page, seq)

    def call(first=None):
        out = torch.full_like(q, float("nan"))
        a = (q, k, v, B, Hq, Hkv, D, page, table, seq, B * seq, kv_len, anc, n_tree)
        ctx.cast_tree_attention(*a, 0.0, out) if first is None else ctx.cast_tree_attention_rows(*a, _ints(first), 0.0, out)
        return out

    def check(out):
        want = _attention_reference(q, k, v, page, table, kv_len.tolist(), anc, n_tree.tolist())
        live = ~want.isnan()
        assert torch.equal(out.isnan(), ~live)
        # P in bf16 (a term of the sum off by 2^-9 of itself, all of them by no more than that of max |v|), then the output
        assert float((out.double() - want)[live].abs().max()) <= 2.0 ** -9 * float(v.abs().max()) + 2.0 ** -8 * float(want[live].abs().max())
        assert ctx.cast_poll_status()[0] == 0

    def compact(path):
        full = path + [-1] * (5 - len(path))
        ctx.cast_compact_kv(k, v, B, 1, k.numel() * k.element_size(), Hkv, D, page, table, seq, B * seq, _ints([full] * B),
                            _ints([len(path) - 1] * B), kv_len)
    return ctx, call, check, compact, kv_len, n_tree


@pytest.mark.parametrize("between", ["window", "f32"])
def test_a_call_between_does_not_keep_an_old_work_list(binding, between):
    """Under the early-read promise: attention, a compaction (which moves the lengths), a call that takes no work list
    - a draft's window, a 32-bit layer - and the first attention again: it must see the new lengths."""
    ctx, call, check, compact, kv_len, n_tree = _early_setup(binding, 2, 8, 8, 2, 128, 16, [40, 700])
    check(call())
    check(call())
    compact([0, 2, 3])
    assert kv_len.tolist() == [43, 703]
    if between == "window":
        call(first=[3, 4])
    else:
        x = torch.zeros((2, 8, 4, 64), device="cuda")
        ctx.cast_reserve_attention(torch.float32, 2, 4, 1, 64, 0, 16)
        c = torch.zeros((2, 16, 1, 64), device="cuda")
        ctx.cast_tree_attention(x, c, c, 2, 4, 1, 64, 0, None, 16, 0, _ints([1, 2]), _ints([[[1]] * 8] * 2), n_tree, 0.0, x.clone())
    check(call())


@pytest.mark.parametrize("Hq,Hkv,D", [(8, 2, 64), (14, 2, 128), (8, 2, 128)])
def test_shapes_outside_the_early_reads_ignore_the_promise(binding, Hq, Hkv, D):
    """The header's shapes (128 dims, a group size that divides 128) take a reused work list, and a caller that changes the
    lengths by itself says so; the other shapes see such a change without being told."""
    ctx, call, check, _, kv_len, n_tree = _early_setup(binding, 2, 8, Hq, Hkv, D, 16, [40, 700])
    check(call())
    for lengths, sizes in (([9, 64], [8, 5]), ([500, 7], [1, 8])):
        kv_len.copy_(_ints(lengths))
        n_tree.copy_(_ints(sizes))
        if D == 128 and 128 % (Hq // Hkv) == 0:
            ctx.cast_set_attention_early_reads(True)
        torch.cuda.synchronize()
        check(call())
        check(call())


@pytest.mark.parametrize("B,Hq,Hkv,D,page,positions", [(1, 32, 8, 128, 16, 4096), (8, 32, 8, 128, 0, 4096), (2, 16, 4, 64, 16, 1024)])
def test_the_fallback_of_a_tensor_core_shape_stays_small(binding, B, Hq, Hkv, D, page, positions):
    """bf16 keys and values on 16-byte boundaries that are not the tensor path's 128 go to the CUDA cores: the workspace
    reserved for that is a few megabytes (two CTAs per SM of 17 KB partials, whole 2 MB pages), and the call runs with it."""
    cap = 60
    rng = np.random.default_rng(B)
    unit = page or 1
    seq = positions // unit
    g = torch.Generator(device="cuda").manual_seed(B)
    shape = (B * seq, page, Hkv, D) if page else (B, seq, Hkv, D)
    n = int(np.prod(shape))
    k, v = (torch.randn(n + 8, generator=g, device="cuda").to(torch.bfloat16)[8:].view(shape) for _ in range(2))
    assert k.data_ptr() % 128 == 16
    table = torch.randperm(B * seq, generator=g, device="cuda").to(torch.int32).view(B, seq) if page else None
    q = torch.randn((B, cap, Hq, D), generator=g, device="cuda").to(torch.bfloat16)
    n_tree = [cap - 7 * (b % 3) for b in range(B)]
    kv = [int(x) for x in rng.integers(1, positions - cap, B)]
    anc = _random_trees(rng, B, cap, n_tree)
    ctx = binding.CastContext(max_batch=B, vocab=100, top_k=2, max_depth=4, total_token=cap, max_tree=cap)
    out = torch.full_like(q, float("nan"))
    args = (B, Hq, Hkv, D, page)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx.cast_reserve_attention(q.dtype, *args, seq)
    assert before - torch.cuda.mem_get_info()[0] <= 8 << 20
    ctx.cast_tree_attention(q, k, v, *args, table, seq, B * seq if page else 0, _ints(kv), anc, _ints(n_tree), 0.0, out)
    assert ctx.cast_poll_status()[0] == 0
    want = _attention_reference(q, k, v, page, table, kv, anc, n_tree)
    live = ~want.isnan()
    assert torch.equal(out.isnan(), ~live)
    assert bool(((out.double() - want)[live].abs() <= 1e-5 + want[live].abs() * 2.0 ** -8).all())


def test_a_list_of_a_shape_outside_the_promise_is_not_trusted_inside(binding):
    """64-dim heads, a change of the lengths that need not be announced there, and a layer of 128-dim heads of the same
    call shape: it decodes its own list."""
    ctx, call64, check64, _, kv_len, n_tree = _early_setup(binding, 2, 8, 8, 2, 64, 16, [40, 700])
    _, call128, check128, _, _, _ = _early_setup(binding, 2, 8, 8, 2, 128, 16, [40, 700], share=(ctx, kv_len, n_tree))
    check64(call64())
    kv_len.copy_(_ints([333, 12]))
    n_tree.copy_(_ints([4, 8]))
    torch.cuda.synchronize()
    check128(call128())
    check64(call64())


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B,Hkv,G,cap,longest", [
    (38, 8, 1, 24, 1100), (40, 8, 2, 17, 1000), (38, 8, 4, 33, 1024), (64, 8, 8, 19, 1030), (64, 5, 16, 9, 1200),
    (38, 8, 64, 4, 1100), (38, 8, 128, 2, 1100), (38, 8, 4, 24, 1024), (64, 8, 8, 12, 1030), (64, 5, 16, 6, 1200),
    (40, 8, 64, 1, 1100), (3, 2, 4, 20, 9000), (3, 2, 4, 40, 9000), (38, 8, 4, 33, 300)])
def test_query_rows_past_the_tree_are_left_out(binding, D, B, Hkv, G, cap, longest):
    """Where the largest tree fills three quarters of a row block at most, launches without clusters copy the boxes of queries
    that hold live rows and fill the rest with zeros; the tree sizes run over the edges of the boxes, and what lies past the
    trees is NaN. The cases whose budget is above that, the cluster of (3, 2, 4) and the short sequences of the last one take whole
    row blocks. Two bf16 roundings, of the probabilities and of the output: 2^-9 of |v|'s maximum each."""
    rng = np.random.default_rng(B + G)
    n_tree = [1 + i % cap for i in range(B)]
    kv = [longest] + [int(x) for x in rng.integers(0, 200, B - 1)]
    for first in (None, [n // 2 for n in n_tree]):
        got, want = _attend(binding, rng, B, cap, n_tree, Hkv * G, Hkv, D, 16, kv, first=first, beyond=float("nan"))
        keep = ~want.isnan()
        assert torch.equal(got.isnan(), ~keep)
        assert float((got.double() - want)[keep].abs().max()) < 2.0 ** -8 * 6


@pytest.mark.parametrize("mode", ["default", "early", "rows"])
@pytest.mark.parametrize("D,B,Hkv,G,cap,page", [(128, 24, 8, 4, 24, 16), (128, 33, 8, 1, 96, 0), (128, 20, 8, 8, 12, 32),
                                                (128, 30, 5, 16, 6, 16), (128, 23, 8, 32, 3, 16), (64, 24, 8, 4, 24, 16),
                                                (64, 38, 4, 2, 48, 0)])
def test_live_query_rows_of_blocks_in_pieces(binding, D, B, Hkv, G, cap, page, mode):
    """Ragged sequences with somewhat more row blocks than half of a wave's slots: the long ones are cut and merged through the
    workspace, every piece with its live query rows alone; with early reads Q comes behind the first tiles, and a window's rows
    start inside the tree. The partials' half precision adds 2^-11 of |v|'s maximum to two bf16 roundings of 2^-9."""
    slots = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert slots < 2 * B * Hkv < 2 * slots and cap * G <= 96  # one block each, no clusters
    n_tree = [1 + (i * 5) % cap for i in range(B)]
    kv = [100 + 6000 * i // B for i in range(B)]
    first = [n // 3 for n in n_tree] if mode == "rows" else None
    got, want = _attend(binding, np.random.default_rng(B + G), B, cap, n_tree, Hkv * G, Hkv, D, page, kv, first=first,
                        early=mode == "early", beyond=float("nan"))
    keep = ~want.isnan()
    assert torch.equal(got.isnan(), ~keep)
    assert float((got.double() - want)[keep].abs().max()) < 2.25 * 2.0 ** -9 * 6


@pytest.mark.parametrize("B,cap,Hq,Hkv,page,sizes,kv", [
    (24, 64, 16, 8, 16, None, [6000] * 24),                              # 192 equal items on 296 slots
    (9, 128, 16, 4, 0, [128] * 9, [9000, 100, 64, 1, 2000, 300, 63, 65, 4000]),  # one sequence much longer than the rest
    (40, 96, 16, 8, 16, None, [20 + 13 * i for i in range(39)] + [9000]),  # unsplit, the items fill more than a wave
    (9, 128, 16, 4, 16, [5, 128, 17, 1, 90, 64, 33, 128, 2], [9000, 100, 64, 1, 9000, 300, 63, 8999, 4000]),
    (16, 64, 32, 8, 16, None, [2048] * 16)])                             # items that are left as they are
def test_items_that_fill_their_waves_badly(binding, B, cap, Hq, Hkv, page, sizes, kv):
    """Equal long items on too many slots, one long sequence among short ones, more items than a wave, with the early-read
    promise. Two bf16 roundings, of the probabilities and of the output, and the partials' in half precision where a row block is
    split: 2^-9, 2^-9 and 2^-11 of |v|'s maximum."""
    rng = np.random.default_rng(B + cap)
    n_tree = sizes or [cap] * B
    got, want = _attend(binding, rng, B, cap, n_tree, Hq, Hkv, 128, page, kv, early=True)
    keep = ~want.isnan()
    assert torch.equal(got.isnan(), ~keep)
    assert float((got.double() - want)[keep].abs().max()) < 2.25 * 2.0 ** -9 * 6


@pytest.mark.parametrize("B,cap,Hq,Hkv,largest,kv", [
    (24, 64, 16, 8, 64, [6000] * 24),                          # 192 equal items on 296 slots, each one piece
    (8, 48, 64, 8, 46, [14000] * 7 + [9000]),                  # three row blocks per sequence and head
    (24, 128, 32, 8, 30, [6000 + 20 * i for i in range(24)]),  # trees far under the budget: more waves launched than they need
    (20, 128, 32, 8, 60, [300 * i + 7 for i in range(20)])])   # the same, ragged, more items than a wave
def test_launches_without_clusters_cut_by_the_trees_alone(binding, B, cap, Hq, Hkv, largest, kv):
    """How a row block is split, and so how its sums are rounded (a block in one piece is not, before the output), depends on the
    trees and lengths, not on the early-read promise or on the waves that the budget has launched: the same bits."""
    n_tree = [largest - i % 3 for i in range(B)]
    outs = []
    for early, budget in ((False, cap), (True, cap), (False, largest), (True, largest)):
        got, want = _attend(binding, np.random.default_rng(B), B, cap, n_tree, Hq, Hkv, 128, 16, kv, early=early, budget=budget)
        outs.append(torch.stack([got[b, :largest - 2] for b in range(B)]))
    keep = ~want.isnan()
    assert float((got.double() - want)[keep].abs().max()) < 2.25 * 2.0 ** -9 * 6
    for other in outs[1:]:
        assert torch.equal(outs[0], other)
