"""The softmax over all positions where its tile pipeline can go wrong: fewer tiles than ring stages, a ring
that wraps, a last tile of one position, and scores that keep growing, so that rows have to raise the
reference of their exponentials (and rescale what they have summed) many times."""
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


def _bound(C, US, V, wq, wk, wv, score, value):
    """Per output element.  P in bf16: 2^-9 of sum p |value|, its sum unrounded; O in bf16: 2^-9 of it.  The products
    behind scores and output have operands of two bf16 halves (2^-17 each): a score is off by 2^-16 of the sum of its
    products' sizes, a weight by twice that, the output by 2^-14 of sum p |US| |V^T W_V| (three products, fp32 sums)."""
    v = V.double()
    p = torch.softmax(score, -1)
    off = ((C.double().abs() @ (wq @ wk.T @ v).abs()) @ US.double().abs().transpose(1, 2)).amax(-1, keepdim=True)
    products = US.double().abs() @ (v.transpose(1, 2) @ wv).abs()
    return (2.0 ** -8 + 2.0 ** -15 * off) * (p @ value.abs()) + 2.0 ** -14 * (p @ products)


@pytest.mark.parametrize("growth", [0.0, 60.0, "last"])
@pytest.mark.parametrize("d,r", [(64, 16), (64, 32), (64, 64), (128, 16), (128, 32), (128, 64)])
def test_tiles_and_growing_scores(d, r, growth):
    g = torch.Generator().manual_seed(d + r)
    B = 2
    V = torch.linalg.qr(torch.randn(B, d, r, generator=g))[0].contiguous()
    W = [(torch.randn(d, d, generator=g) * d ** -0.5).bfloat16() for _ in range(3)]
    for N in (r, 127, 128, 129, 256, 384, 385, 513, 900, 1025):
        M = 1 + N % 260
        C = (torch.randn(B, M, d, generator=g) * d ** -0.5).bfloat16()
        US = torch.randn(B, N, r, generator=g)
        if growth == "last":              # half of the candidates look at the last position almost alone
            US[:, -1] *= 40
        else:
            US *= 1 + growth * torch.arange(N)[:, None] / N
        US = US.bfloat16()
        buf = torch.full((B * M * d + 64,), float("nan"), dtype=torch.bfloat16, device="cuda")
        O = buf[: B * M * d].view(B, M, d)
        solar.factored_softmax_attention_fwd(*(t.cuda() for t in (C, US, V, *W)), 1.0, O=O)
        torch.cuda.synchronize()
        wq, wk, wv = (w.double() for w in W)
        H = US.double() @ V.double().transpose(1, 2)
        value = H @ wv
        score = (C.double() @ wq) @ (H @ wk).transpose(1, 2)
        ref = torch.softmax(score, -1) @ value
        assert float(((O.double().cpu() - ref).abs() / _bound(C, US, V, wq, wk, wv, score, value)).max()) <= 1, (N, M)
        assert bool(torch.isnan(buf[B * M * d:]).all()), (N, M)


def _ranges(B, M, N, d, r, workspace_bytes):
    """How many ranges the positions are split into (flash_split): wanted, and as the workspace allows; where their
    counters lie, and how many there are."""
    up = lambda x: -(-x // 256) * 256
    tiles, items = -(-N // 128), B * -(-M // 128)
    counters = B * (2 * up(4 * d * r) + 2 * up(2 * 2 * 64 * d))
    part = counters + up(4 * items)
    k = min(148 * (2 if (d == 64 and r <= 32) or r == 16 else 1) // items, tiles // 4)
    while k > 1 and k * k > 9 * tiles:
        k -= 1
    wanted = max(k, 1)
    k = max(1, min(wanted, max(0, workspace_bytes - part) // (items * (r + 2) * 512)))
    per = lambda n: -(-tiles // -(-tiles // n))
    return per(wanted), per(k), counters, items


@pytest.mark.parametrize("B,M,N,d,r", [(1, 100, 5000, 64, 32), (1, 128, 20000, 64, 16), (2, 300, 3000, 64, 64), (1, 1, 4097, 128, 64),
                                       (3, 129, 1025, 128, 16), (1, 140, 1024, 128, 32)])
def test_positions_split_over_ctas(B, M, N, d, r):
    g = torch.Generator().manual_seed(N + M)
    V = torch.linalg.qr(torch.randn(B, d, r, generator=g))[0].contiguous()
    W = [(torch.randn(d, d, generator=g) * d ** -0.5).bfloat16() for _ in range(3)]
    C = (torch.randn(B, M, d, generator=g) * d ** -0.5).bfloat16()
    wq, wk, wv = (w.double() for w in W)
    for growth in (0.0, 40.0):
        # the largest scores in the middle: the ranges' references differ either way
        at = 1 - (2 * torch.arange(N) / N - 1).abs()
        US = (torch.randn(B, N, r, generator=g) * (1 + growth * at[:, None])).bfloat16()
        args = [t.cuda() for t in (C, US, V, *W)]
        ws = solar.alloc_workspace(B, M, N, d, r, torch.bfloat16)
        ws.fill_(0xFF)
        got = [solar.factored_softmax_attention_fwd(*args, 1.0, workspace=ws) for _ in range(3)]
        small = solar.alloc_workspace(B, M, r, d, r, torch.bfloat16)          # room for the operands: one range
        one = solar.factored_softmax_attention_fwd(*args, 1.0, workspace=small)
        torch.cuda.synchronize()
        # the split happens: every item's ranges have been counted
        wanted, ranges, at_bytes, items = _ranges(B, M, N, d, r, ws.numel())
        assert ws[at_bytes: at_bytes + 4 * items].view(torch.int32).tolist() == [ranges] * items
        assert 2 <= ranges <= wanted
        large = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")       # room for all the ranges wanted
        most = solar.factored_softmax_attention_fwd(*args, 1.0, workspace=large)
        assert large[at_bytes: at_bytes + 4 * items].view(torch.int32).tolist() == [wanted] * items
        assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
        H = US.double() @ V.double().transpose(1, 2)
        value = H @ wv
        score = (C.double() @ wq) @ (H @ wk).transpose(1, 2)
        ref = torch.softmax(score, -1) @ value
        for x in (got[0], one, most):
            assert float(((x.double().cpu() - ref).abs() / _bound(C, US, V, wq, wk, wv, score, value)).max()) <= 1, growth
