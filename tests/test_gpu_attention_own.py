"""Attention on kept factors where every CTA makes its user's operands (d = 64, r <= 32, few CTAs)
against the projection kernel followed by the attention kernel: the same bits, with and without softmax, at the
edges of the token and candidate tiles and of the rule itself."""
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,M,r", [(1, 1, 1), (1, 127, 15), (3, 128, 16), (3, 129, 17), (2, 300, 31), (8, 640, 32), (8, 3000, 27),
                                   (111, 256, 8), (111, 257, 24), (2, 130, 33)])
@pytest.mark.parametrize("flags", [0, solar.FLAG_NO_SOFTMAX])
def test_one_launch_equals_two(B, M, r, flags):
    d, gen = 64, torch.Generator(device="cuda")
    gen.manual_seed(B * 1000 + M + r)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    C, W = (rn(B, M, d) / 8).bfloat16(), [(rn(d, d) / 8).bfloat16() for _ in range(3)]
    V = torch.linalg.qr(rn(B, d, r))[0].contiguous()
    S = (rn(B, r).abs().sort(dim=1, descending=True).values * 5.0).contiguous()
    S[0, r // 2:] = 0.0                                      # tokens of zero singular values stay
    ws = solar.alloc_workspace(B, M, 128, d, r, torch.bfloat16)
    ws.fill_(0xff)
    one = solar.svd_attention_fwd(C, S, V, *W, d ** -0.5, flags, workspace=ws)
    again, two = torch.empty_like(C), torch.empty_like(C)
    solar.attn_apply(C, r, flags, again, ws)                 # on the operands that the call left
    ws.fill_(0xff)
    solar.attn_prepare(S, V, *W, d ** -0.5, ws)
    solar.attn_apply(C, r, flags, two, ws)
    torch.cuda.synchronize()
    assert torch.equal(one, two) and torch.equal(again, two)
