"""The forward pass under CUDA-graph replay and on several streams at once gives exactly what
the plain calls give (the kernels keep no state; lanes differ only in their workspaces), and
random shapes agree with the oracle."""
import numpy as np
import pytest
import torch

import oracle as o
from paper_2603_02561_b200 import solar
from paper_2603_02561_b200 import workloads as wl

import parity_harness as ph

pytestmark = pytest.mark.gpu


def _inputs(w):
    inp = wl.generate(w)
    H = ph.to_device(inp["H"], w.dtype); C = ph.to_device(inp["C"], w.dtype)
    Wq, Wk, Wv = (ph.to_device(inp[k], w.dtype) for k in ("Wq", "Wk", "Wv"))
    return inp, H, C, Wq, Wk, Wv


def test_graph_replay_and_concurrent_streams_match_plain_calls():
    w = wl.CONFIGS["c2"].with_(B=6, N=1500, M=300)
    inp, H, C, Wq, Wk, Wv = _inputs(w)
    O_ref, S_ref, V_ref = solar.forward(H, C, Wq, Wk, Wv, w.r, inp["scale"])
    torch.cuda.synchronize()

    lanes = []
    for _ in range(3):
        lanes.append(dict(st=torch.cuda.Stream(), S=torch.empty_like(S_ref), V=torch.empty_like(V_ref),
                          O=torch.full_like(O_ref, float("nan")),
                          ws=solar.alloc_workspace(w.B, w.M, w.N, w.d, w.r, H.dtype)))
    main = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(main):
        with torch.cuda.graph(g, stream=main, capture_error_mode="relaxed"):
            fork = torch.cuda.Event(); fork.record(main)
            for ln in lanes:
                ln["st"].wait_event(fork)
                for _ in range(2):     # twice per lane: the second pass reuses a dirty workspace
                    solar.lowrank_factor(H, w.r, S=ln["S"], V=ln["V"], workspace=ln["ws"], stream=ln["st"])
                    solar.svd_attention_fwd(C, ln["S"], ln["V"], Wq, Wk, Wv, inp["scale"], 0, O=ln["O"],
                                            workspace=ln["ws"], stream=ln["st"])
                j = torch.cuda.Event(); j.record(ln["st"]); main.wait_event(j)
        for _ in range(3):
            g.replay()
    torch.cuda.synchronize()
    for ln in lanes:
        assert torch.equal(ln["S"], S_ref) and torch.equal(ln["V"], V_ref) and torch.equal(ln["O"], O_ref)


@pytest.mark.parametrize("seed", range(6))
def test_random_shapes_agree_with_the_oracle(seed):
    g = np.random.default_rng(1000 + seed)
    dtype = ["bf16", "f32"][seed % 2]
    d = int(g.choice([32, 64, 128]))
    r = int(g.integers(1, min(d, 64) + 1))
    B = int(g.integers(1, 4)); N = int(g.integers(r, 900)); M = int(g.integers(1, 300))
    rank = int(min(d, r + g.integers(0, 4)))
    w = wl.Workload(f"rnd{seed}", dtype, B, N, d, r, M, "product_noise", rank=rank,
                    noise_var=float(10.0 ** g.uniform(-4, -2)), seed_index=50 + seed)
    inp = wl.generate(w)
    got = ph.run_gpu(w, inp)
    assert np.all(got["info"] == 0)
    for k in range(B):
        res = ph.compare_user(w, inp, got, k)
        assert res["o_err"] <= ph.TOL[dtype], (w, k, res["o_err"])


@pytest.mark.parametrize("d,dtype", [(32, torch.float32), (32, torch.bfloat16), (64, torch.float32), (64, torch.bfloat16), (128, torch.float32)])
def test_outputs_of_a_call_are_inputs_of_the_next(d, dtype):
    """Calls that start while the one before is draining, each reading what that one writes: the attention's
    output as candidates, gradients as factors, through the whole calls and the single stages."""
    g = torch.Generator().manual_seed(d)
    B, M, N, r = 4, 500, 600, 12
    C0, dO = ((torch.randn(B, M, d, generator=g) * d ** -0.5).to(dtype).cuda() for _ in range(2))
    H = (torch.randn(B, N, r, generator=g) @ torch.randn(B, r, d, generator=g) + 0.1 * torch.randn(B, N, d, generator=g)).to(dtype).cuda()
    W = [(torch.randn(d, d, generator=g) * d ** -0.5).to(dtype).cuda() for _ in range(3)]
    ws, bws = solar.alloc_workspace(B, M, N, d, r, dtype), solar.alloc_backward_workspace(B, M, N, d, r, dtype)

    def chain(wait):
        out = []

        def done(*t):
            out.extend(x.clone() for x in t if wait)               # (a copy would stand between the calls)
            if wait:
                torch.cuda.synchronize()
            else:
                out.extend(t)
        S, V = solar.lowrank_factor(H, r, workspace=ws); done(S, V)
        C = C0
        for _ in range(3):
            C = solar.svd_attention_fwd(C, S, V, *W, d ** -0.5, workspace=ws); done(C)
        grads = solar.svd_attention_bwd(C, S, V, *W, d ** -0.5, dO, bws); done(*grads)
        O = torch.empty_like(C)
        solar.attn_prepare(grads[4], grads[5], *W, 0.3, ws)        # S and V from the kernel just before
        solar.attn_apply(C, r, 0, O, ws); done(O)
        P = torch.empty_like(C)
        solar.attn_apply(O, r, 0, P, ws); done(P)
        dH = torch.empty_like(H)
        solar.svd_backward(H, S, V, grads[4], grads[5], dH, bws, eps_rel=1e-6); done(dH)
        torch.cuda.synchronize()
        return out

    ref = chain(True)
    for _ in range(5):
        for a, b in zip(chain(False), ref):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
