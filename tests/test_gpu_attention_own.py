"""Attention on kept factors where every CTA makes its user's operands (d = 64, r <= 32, few CTAs)
against the projection kernel followed by the attention kernel: the same bits, with and without softmax, at the
edges of the token and candidate tiles and of the rule itself; and which of the two a call takes."""
import ctypes

import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def no_slice_limit():
    old = solar.set_slice_limit(0)
    yield
    solar.set_slice_limit(old)


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


def _kernels(B, M, r, d=64, dtype=torch.bfloat16):
    """Kernels that a call launches: the nodes of a graph that holds it alone."""
    C, W = torch.zeros(B, M, d, device="cuda", dtype=dtype), [torch.zeros(d, d, device="cuda", dtype=dtype)] * 3
    S, V = torch.zeros(B, r, device="cuda"), torch.zeros(B, d, r, device="cuda")
    ws, O = solar.alloc_workspace(B, M, 128, d, r, dtype), torch.empty_like(C)
    solar.svd_attention_fwd(C, S, V, *W, 1.0, 0, O=O, workspace=ws)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        solar.svd_attention_fwd(C, S, V, *W, 1.0, 0, O=O, workspace=ws)
    n = ctypes.c_size_t(0)
    nodes = ctypes.CDLL("libcudart.so.12").cudaGraphGetNodes
    assert nodes(ctypes.c_void_p(g.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("B,M,r,limit,kernels", [
    (1, 1, 1, 0, 1), (3, 129, 17, 0, 1), (8, 640, 32, 0, 1), (8, 3000, 27, 0, 1), (111, 256, 8, 0, 1), (222, 128, 32, 0, 1),
    (223, 128, 32, 0, 2), (111, 257, 24, 0, 2),              # more than 222 CTAs
    (2, 130, 33, 0, 2),                                      # r > 32
    (8, 640, 32, 2, 2)])                                     # other requests want the SMs
def test_which_form_a_call_takes(B, M, r, limit, kernels):
    solar.set_slice_limit(limit)
    assert _kernels(B, M, r) == kernels


def test_other_sizes_and_types_take_two_launches():
    assert _kernels(2, 130, 8, d=128) == 2 and _kernels(2, 130, 8, d=32) == 2 and _kernels(2, 130, 8, dtype=torch.float32) == 2
