"""Where the tridiagonal reduction stops early (a history of rank R ends it near step R): R at the
edges of the kernel's stages of live columns, of its warps' rows, and at the very end of the matrix."""
import numpy as np
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [32, 64, 128])
def test_the_reduction_may_stop_at_any_step(d):
    rng = np.random.default_rng(d)
    ranks = sorted({R for e in range(8, d + 1, 8) for R in (e - 1, e, e + 1) if 2 <= R <= d} | {1, 2, d - 2, d - 1, d})
    B, N = len(ranks), 300
    H = np.empty((B, N, d), np.float32)
    sv = np.zeros((B, d))
    for b, R in enumerate(ranks):
        U, _ = np.linalg.qr(rng.standard_normal((N, R)))
        W, _ = np.linalg.qr(rng.standard_normal((d, R)))
        sv[b, :R] = 3.0 - 2.0 * np.arange(R) / R        # no two close to each other, none small
        H[b] = (U * sv[b, :R]) @ W.T
    for r in (1, min(d, 32), min(d, 64)):
        keep = [b for b, R in enumerate(ranks) if R >= r]
        Hd = torch.from_numpy(H[keep]).cuda()
        info = torch.full((len(keep),), -1, dtype=torch.int32, device="cuda")
        S, V = solar.lowrank_factor(Hd, r, info=info)
        torch.cuda.synchronize()
        S, V = S.cpu().numpy().astype(np.float64), V.cpu().numpy().astype(np.float64)
        assert torch.all(info == 0)
        # the bounds the eigensolver's other tests use for fp32 histories
        assert np.abs(S - sv[keep, :r]).max() <= 1e-5 * 3.0
        assert np.abs(np.einsum("bki,bkj->bij", V, V) - np.eye(r)).max() <= 2e-5
        G = np.einsum("bni,bnj->bij", H[keep].astype(np.float64), H[keep].astype(np.float64))
        assert np.abs(G @ V - V * (S ** 2)[:, None, :]).max() <= 2e-5 * 9.0
