"""The FFMA kernels at the edges of their tiles: rows per stage and per slice of the Gram pass, rows per
CTA and token counts of the attention, against double precision."""
import numpy as np
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d", [32, 64, 128])
def test_gram_rows(d, dtype):
    g = torch.Generator().manual_seed(d)
    for N in (1, 2, 31, 32, 33, 55, 56, 57, 99, 100, 101, 127) + ((128, 129, 1000, 2049) if dtype == torch.float32 else ()):
        B = 3
        H = torch.randn(B, N, d, generator=g).to(dtype)
        ws = solar.alloc_workspace(B, 1, N, d, 1, dtype); ws.fill_(0xFF)
        solar.gram_partials(H.cuda(), ws)
        torch.cuda.synchronize()
        P = solar.gram_splits(B, N, d, dtype)
        G = ws[: B * P * d * d * 4].view(torch.float32).view(B, P, d, d).double().sum(1).cpu()
        ref = H.double().transpose(1, 2) @ H.double()
        # an entry is a sum of N products: at most N roundings of 2^-24 of sum |h_i h_j| <= max diagonal entry
        bound = (N + 2) * 2.0 ** -24 * ref.diagonal(dim1=1, dim2=2).amax()
        assert float((G - ref).abs().max()) <= bound, N
        assert torch.equal(G, G.transpose(1, 2))


@pytest.mark.parametrize("flags", [0, solar.FLAG_NO_SOFTMAX])
@pytest.mark.parametrize("d,dtype", [(32, torch.float32), (32, torch.bfloat16), (64, torch.float32), (128, torch.float32)])
def test_attention_rows_and_tokens(d, dtype, flags):
    g = torch.Generator().manual_seed(d)
    Wq, Wk, Wv = ((torch.randn(d, d, generator=g) * d ** -0.5).to(dtype) for _ in range(3))
    for r in sorted({1, 7, 8, 9, 16, 17, 24, 25, 32} | ({33, 40, 41, 48, 49, 63, 64} if d > 32 else set())):
        for M in (1, 127, 128, 129, 300):
            B = 2
            C = (torch.randn(B, M, d, generator=g) * d ** -0.5).to(dtype)
            V = torch.linalg.qr(torch.randn(B, d, r, generator=g))[0].contiguous()
            S = torch.rand(B, r, generator=g) * 10 + 1
            O = solar.svd_attention_fwd(*(t.cuda() for t in (C, S, V, Wq, Wk, Wv)), d ** -0.5, flags)
            torch.cuda.synchronize()
            A = (V.double() * S.double()[:, None]).transpose(1, 2)
            P = d ** -0.5 * (C.double() @ Wq.double()) @ (A @ Wk.double()).transpose(1, 2)
            P = P if flags else torch.softmax(P, -1)
            ref = P @ (A @ Wv.double())
            tol = 1e-5 if dtype == torch.float32 else 2.0 ** -8      # fp32 sums of up to 3 d products; bf16 output rounding
            assert float((O.cpu().double() - ref).abs().max()) <= tol * float(ref.abs().max()), (r, M)


@pytest.mark.parametrize("d,dtype", [(32, torch.float32), (32, torch.bfloat16), (64, torch.float32), (128, torch.float32)])
def test_infinite_candidates_without_softmax(d, dtype):
    """A row with an infinity: infinite scores on the tokens there are, nothing from the padded ones."""
    g = torch.Generator().manual_seed(d)
    B, M = 2, 9
    Wq, Wk, Wv = ((torch.randn(d, d, generator=g) * d ** -0.5).to(dtype) for _ in range(3))
    for r in (1, 2, 3, 7, 8, 15):
        C = (torch.randn(B, M, d, generator=g) * d ** -0.5).to(dtype)
        C[0, 4, 5] = float("inf")
        C[1, 0, 0] = -float("inf")
        V = torch.linalg.qr(torch.randn(B, d, r, generator=g))[0].contiguous()
        S = torch.rand(B, r, generator=g) * 10 + 1
        O = solar.svd_attention_fwd(*(t.cuda() for t in (C, S, V, Wq, Wk, Wv)), d ** -0.5, solar.FLAG_NO_SOFTMAX).cpu()
        A = (V.double() * S.double()[:, None]).transpose(1, 2)
        P = C.double() @ (d ** -0.5 * Wq.double() @ (A @ Wk.double()).transpose(1, 2))       # scores through T
        ref = P @ (A @ Wv.double())
        assert torch.equal(torch.isnan(O), torch.isnan(ref)), r
        assert torch.equal(torch.isinf(O), torch.isinf(ref)), r
        assert torch.equal(O[torch.isinf(O)] > 0, ref[torch.isinf(ref)] > 0), r
        assert r > 2 or bool(torch.isinf(O).any()), r
