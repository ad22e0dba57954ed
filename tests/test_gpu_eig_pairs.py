"""Two CTAs per user (r > 32, few users): batches that mix users whose fp32 chain is enough with users whose
gaps need the fp64 one, all-zero and non-finite users among them, against the same users alone under a
slice limit, where a user has one CTA and runs the chains one after the other."""
import numpy as np
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,r,B", [(64, 33, 1), (64, 64, 7), (128, 33, 5), (128, 64, 8), (64, 40, 74), (64, 40, 75)])
def test_mixed_batch_equals_one_cta_per_user(d, r, B):
    rng = np.random.default_rng(d + r + B)
    N = 300
    H = np.zeros((B, N, d), np.float32)
    for b in range(B):
        kind = b % 5
        U, _ = np.linalg.qr(rng.standard_normal((N, d)))
        W, _ = np.linalg.qr(rng.standard_normal((d, d)))
        sig = {0: np.arange(1, d + 1) ** -2.0, 1: np.linspace(2, 1, d), 2: np.zeros(d), 3: np.linspace(2, 1, d), 4: np.arange(1, d + 1) ** -1.5}[kind]
        H[b] = (U * sig) @ W.T
        if kind == 3:
            H[b, 3, 5] = np.nan
    Hd = torch.from_numpy(H).cuda()
    out = []
    for limit in (0, 64):
        old = solar.set_slice_limit(limit)
        try:
            ws = solar.alloc_workspace(B, 1, N, d, r, torch.float32)
            S = torch.empty(B, r, device="cuda"); V = torch.empty(B, d, r, device="cuda")
            info = torch.full((B,), -1, dtype=torch.int32, device="cuda"); taken = torch.zeros_like(info)
            solar.gram_partials(Hd, ws)
            for _ in range(3):
                solar.eig_from_partials_ex(B, N, d, r, torch.float32, solar.ROUTE_AUTO, S, V, info, taken, ws)
            torch.cuda.synchronize()
        finally:
            solar.set_slice_limit(old)
        out.append([t.cpu() for t in (S, V, info, taken)])
    for a, b in zip(out[0], out[1]):
        assert torch.equal(torch.nan_to_num(a), torch.nan_to_num(b)), (out[0][2:], out[1][2:])
    assert any((t & 0xffff) == (2 | (1 << 8)) for t in out[0][3].tolist())       # fp64 chain
    assert B == 1 or any((t & 0xff) == 3 for t in out[0][3].tolist())            # fp32 chain
