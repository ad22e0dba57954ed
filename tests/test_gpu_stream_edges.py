"""The clusters of the Gram pass.  The streaming kernels of the left factor and of the backward pass where their layouts change: output
rows of one, two and four swizzle spans and rows that end inside a warp's 32; token counts around 32,
where the probabilities' shared-memory rows widen."""
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
def test_left_factor_rows(d):
    g = torch.Generator().manual_seed(d)
    for r in (8, 15, 16, 24, 32, 40, 48, 56, 64):
        for N in (128, 129, 159, 160, 161, 385):
            H = torch.randn(3, N, d, generator=g).bfloat16()
            V = torch.linalg.qr(torch.randn(3, d, r, generator=g))[0].contiguous()
            buf = torch.full((3 * N * r + 64,), float("nan"), dtype=torch.bfloat16, device="cuda")
            solar.project_us(H.cuda(), V.cuda(), buf[: 3 * N * r].view(3, N, r))
            torch.cuda.synchronize()
            ref = H.double() @ V.double()
            got = buf[: 3 * N * r].view(3, N, r).cpu().double()
            # one rounding to bf16 (2^-9 of the value) and 2^-16 halves of V
            assert float((got - ref).abs().max()) <= 2.0 ** -8 * float(ref.abs().max()), (r, N)
            assert bool(torch.isnan(buf[3 * N * r:]).all())


@pytest.mark.parametrize("d", [64, 128])
def test_left_factor_rows_of_whole_16_bytes_are_stored_as_such(d):
    """A width that TMA does not store takes about as long as the next one that it does (2-byte stores: four to
    seven times as long)."""
    H = torch.randn(16, 8192, d, device="cuda").bfloat16()
    us = {}
    for r in (40, 56, 64):
        V, US = torch.randn(16, d, r, device="cuda"), torch.empty(16, 8192, r, dtype=H.dtype, device="cuda")
        best = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                solar.project_us(H, V, US)
            b.record()
            b.synchronize()
            best.append(a.elapsed_time(b))
        us[r] = min(best)
    assert max(us[40], us[56]) <= 2.5 * us[64], us


@pytest.mark.parametrize("d", [64, 128])
def test_history_gradient_rows(d):
    g = torch.Generator().manual_seed(2 * d)
    B, r = 2, 40
    for N in (128, 161, 300):
        H = torch.randn(B, N, d, generator=g).bfloat16().cuda()
        V = torch.linalg.qr(torch.randn(B, d, r, generator=g))[0].contiguous().cuda()
        S = (torch.arange(r, 0, -1).float() + 3).repeat(B, 1).cuda()
        dS, dV = torch.randn(B, r, generator=g).cuda(), torch.randn(B, d, r, generator=g).cuda()
        dH = torch.empty_like(H)
        solar.svd_backward(H, S, V, dS, dV, dH, solar.alloc_backward_workspace(B, 1, N, d, r, H.dtype))
        torch.cuda.synchronize()
        s, v = S.double(), V.double()
        D = s[:, :, None] ** 2 - s[:, None, :] ** 2
        X = torch.where(D == 0, torch.zeros_like(D), 1 / D) * (dV.double().transpose(1, 2) @ v)
        K = v @ ((torch.diag_embed(dS.double()) + s[:, :, None] * (X + X.transpose(1, 2))) / s[:, :, None]) @ v.transpose(1, 2)
        ref = H.double() @ K
        assert float((dH.double() - ref).abs().max()) <= 2.0 ** -7 * float(ref.abs().max()), N


@pytest.mark.parametrize("r", [1, 16, 17, 31, 32, 33, 48, 64])
def test_attention_gradients_by_token_count(r):
    g = torch.Generator().manual_seed(r)
    B, M, d = 2, 300, 64
    C, dO = ((torch.randn(B, M, d, generator=g) * d ** -0.5).bfloat16() for _ in range(2))
    W = [(torch.randn(d, d, generator=g) * d ** -0.5).bfloat16() for _ in range(3)]
    V = torch.linalg.qr(torch.randn(B, d, r, generator=g))[0].contiguous()
    S = torch.rand(B, r, generator=g) * 4 + 1
    ws = solar.alloc_backward_workspace(B, M, r, d, r, C.dtype, "cuda")
    ws.fill_(0xFF)
    got = solar.svd_attention_bwd(*(t.cuda() for t in (C, S, V, *W)), d ** -0.5, dO.cuda(), ws)
    torch.cuda.synchronize()
    x = [t.double().requires_grad_() for t in (C, S, V, *W)]
    A = (x[2] * x[1][:, None]).transpose(1, 2)
    O = torch.softmax(d ** -0.5 * (x[0] @ x[3]) @ (A @ x[4]).transpose(1, 2), -1) @ (A @ x[5])
    O.backward(dO.double())
    for name, a, b in zip(("dC", "dWq", "dWk", "dWv", "dS", "dV"), got, [x[i].grad for i in (0, 3, 4, 5, 1, 2)]):
        # dC: one rounding to bf16; the fp32 outputs: products of bf16 halves, about 2^-16 each
        tol = 2.0 ** -7 if name == "dC" else 2e-4
        assert float((a.cpu().double() - b).abs().max()) <= tol * max(float(b.abs().max()), 1e-3), name


@pytest.mark.parametrize("B,N,slices,parts", [(2, 8192, 64, 16), (8, 16384, 16, 4), (16, 8190, 8, 2), (1, 40000, 63, 21), (9, 16300, 16, 8), (15, 16384, 9, 3),
                                              (16, 16384, 9, 9), (3, 1000, 8, 2), (1, 130, 2, 1)])
def test_partial_matrices_of_clustered_slices(B, N, slices, parts):
    d = 128
    H = torch.randn(B, N, d, generator=torch.Generator().manual_seed(N)).bfloat16().cuda()
    assert (solar.gram_slices(B, N, d, H.dtype), solar.gram_splits(B, N, d, H.dtype)) == (slices, parts)
    ws = solar.alloc_workspace(B, 1, N, d, 1, H.dtype).fill_(0xFF)
    solar.gram_partials(H, ws)
    torch.cuda.synchronize()
    got = ws[: B * parts * d * d * 4].view(torch.float32).view(B, parts, d, d).double()
    rows = -(-(-(-N // 128)) // slices) * 128 * (slices // parts)          # rows of a partial: whole tiles of 128
    for p in range(parts):
        x = H[:, p * rows: (p + 1) * rows].double()
        ref = x.transpose(1, 2) @ x
        # a sum of `rows` exact products in fp32: at most one rounding (or truncation) of 2^-23 of the sum per product
        assert float((got[:, p] - ref).abs().max()) <= x.shape[1] * 2.0 ** -23 * float(ref.abs().max()), p
