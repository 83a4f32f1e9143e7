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
