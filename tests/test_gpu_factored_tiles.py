"""The softmax over all positions where its tile pipeline can go wrong: fewer tiles than ring stages, a ring
that wraps, a last tile of one position, and scores that keep growing, so that rows have to raise the
reference of their exponentials (and rescale what they have summed) many times."""
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("growth", [0.0, 60.0])
@pytest.mark.parametrize("d,r", [(64, 16), (64, 32), (64, 64), (128, 16), (128, 32), (128, 64)])
def test_tiles_and_growing_scores(d, r, growth):
    g = torch.Generator().manual_seed(d + r)
    B = 2
    V = torch.linalg.qr(torch.randn(B, d, r, generator=g))[0].contiguous()
    W = [(torch.randn(d, d, generator=g) * d ** -0.5).bfloat16() for _ in range(3)]
    for N in (r, 127, 128, 129, 256, 384, 385, 513, 900, 1025):
        M = 1 + N % 260
        C = (torch.randn(B, M, d, generator=g) * d ** -0.5).bfloat16()
        US = (torch.randn(B, N, r, generator=g) * (1 + growth * torch.arange(N)[:, None] / N)).bfloat16()
        buf = torch.full((B * M * d + 64,), float("nan"), dtype=torch.bfloat16, device="cuda")
        O = buf[: B * M * d].view(B, M, d)
        solar.factored_softmax_attention_fwd(*(t.cuda() for t in (C, US, V, *W)), 1.0, O=O)
        torch.cuda.synchronize()
        wq, wk, wv = (w.double() for w in W)
        H = US.double() @ V.double().transpose(1, 2)
        value = H @ wv
        score = (C.double() @ wq) @ (H @ wk).transpose(1, 2)
        ref = torch.softmax(score, -1) @ value
        # P in bf16 (2^-9 of sum p |value|), O in bf16 (2^-9 of it); scores to 2^-16 of their size: a weight to
        # 2 * 2^-16 max|score|
        bound = (2.0 ** -8 + 2.0 ** -15 * float(score.abs().max())) * float(value.abs().max())
        assert float((O.double().cpu() - ref).abs().max()) <= bound, (N, M)
        assert bool(torch.isnan(buf[B * M * d:]).all()), (N, M)


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
        assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
        H = US.double() @ V.double().transpose(1, 2)
        value = H @ wv
        score = (C.double() @ wq) @ (H @ wk).transpose(1, 2)
        ref = torch.softmax(score, -1) @ value
        bound = (2.0 ** -8 + 2.0 ** -15 * float(score.abs().max())) * float(value.abs().max())       # as above
        for x in (got[0], one):
            assert float((x.double().cpu() - ref).abs().max()) <= bound, growth
