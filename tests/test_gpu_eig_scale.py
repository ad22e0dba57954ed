"""Histories of very small and very large scale: the eigensolver works on the Gram matrix times a power of two,
so its route, vectors and relative residuals are those of the same histories at scale one, to the ends of
the range in which the Gram matrix itself is normal."""
import numpy as np
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


def _factor(H, r):
    """S, V, route word and the Gram matrices (fp64 sums of the partials that the eigensolver reads)."""
    B, N, d = H.shape
    ws = solar.alloc_workspace(B, 1, N, d, r, H.dtype)
    S = torch.empty(B, r, device="cuda"); V = torch.empty(B, d, r, device="cuda")
    info = torch.full((B,), -1, dtype=torch.int32, device="cuda"); taken = torch.zeros_like(info)
    solar.gram_partials(H, ws)
    parts = solar.gram_splits(B, N, d, H.dtype)
    G = ws[: B * parts * d * d * 4].view(torch.float32).reshape(B, parts, d, d).double().sum(1)
    solar.eig_from_partials_ex(B, N, d, r, H.dtype, solar.ROUTE_AUTO, S, V, info, taken, ws)
    torch.cuda.synchronize()
    assert info.tolist() == [0] * B
    return S.double(), V.double(), taken.tolist(), G


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("d", [32, 64, 128])
def test_the_scale_of_the_histories_does_not_matter(d, dtype):
    rng = np.random.default_rng(d)
    N, r, H = 300, 8, []
    for noise in (0.3, 0.1, 0.02, 0.002):                     # ends of the reduction on tails of several lengths
        U, _ = np.linalg.qr(rng.standard_normal((N, d)))
        W, _ = np.linalg.qr(rng.standard_normal((d, d)))
        s = noise * (2.0 - np.arange(d) / d)
        s[:r] = 3.0 - 2.0 * np.arange(r) / r                  # no two close to each other
        H.append((U * s) @ W.T)
    H = torch.from_numpy(np.stack(H)).cuda().to(dtype)
    S1, V1, _, _ = _factor(H, r)
    for e in (-60, -58, -56, -52, 52, 56, 60):                # largest entries of G: 2^-120 .. 2^122
        S, V, taken, G = _factor((H.double() * 2.0 ** e).to(dtype), r)
        S, G = S * 2.0 ** -e, G * 4.0 ** -e
        assert [t & 0xFF for t in taken] == [3] * len(taken) and [(t >> 24) & 0xFF for t in taken] == [0] * len(taken), \
            [hex(t & 0xFFFFFFFF) for t in taken]
        if e > 0:                                             # nothing underflows: the same bits
            assert torch.equal(S, S1) and torch.equal(V, V1)
        # a backward stable chain of fp32 sums: a few 2^-24 of the largest eigenvalue
        lam1 = float((S1 ** 2).max())
        assert float((G @ V - V * (S ** 2)[:, None, :]).norm(dim=1).max()) <= 16 * 2.0 ** -24 * lam1
