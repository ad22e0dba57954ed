"""Spectra whose gaps are too small for the fp32 tridiagonal chain: the fp64 chain answers (route 2
with detail 1), with singular values, vectors and residuals at the accuracy of the Gram matrix."""
import numpy as np
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,r", [(32, 9), (32, 32), (64, 31), (64, 64), (128, 32), (128, 33), (128, 64)])
def test_graded_spectra_take_the_double_precision_chain(d, r):
    rng = np.random.default_rng(d + r)
    B, N = 3, 400
    sig = np.arange(1, d + 1) ** -2.0
    H = np.empty((B, N, d), np.float32)
    for b in range(B):
        U, _ = np.linalg.qr(rng.standard_normal((N, d)))
        W, _ = np.linalg.qr(rng.standard_normal((d, d)))
        H[b] = (U * sig) @ W.T
    Hd = torch.from_numpy(H).cuda()
    ws = solar.alloc_workspace(B, 1, N, d, r, torch.float32)
    S = torch.empty(B, r, device="cuda"); V = torch.empty(B, d, r, device="cuda")
    info = torch.full((B,), -1, dtype=torch.int32, device="cuda"); taken = torch.zeros_like(info)
    solar.gram_partials(Hd, ws)
    solar.eig_from_partials_ex(B, N, d, r, torch.float32, solar.ROUTE_AUTO, S, V, info, taken, ws)
    torch.cuda.synchronize()
    assert info.tolist() == [0] * B
    assert [t & 0xffff for t in taken.tolist()] == [2 | (1 << 8)] * B, [hex(t) for t in taken.tolist()]
    S, V = S.cpu().numpy().astype(np.float64), V.cpu().numpy().astype(np.float64)
    for b in range(B):
        G = H[b].astype(np.float64).T @ H[b].astype(np.float64)
        lam, vec = np.linalg.eigh(G)
        lam, vec = lam[::-1], vec[:, ::-1]
        # the kernel's Gram matrix carries fp32 rounding errors of a few 2^-24 lambda_1
        eps = 16 * 2.0 ** -24 * lam[0]
        assert np.all(np.abs(S[b] ** 2 - lam[:r]) <= eps)
        assert np.abs(V[b].T @ V[b] - np.eye(r)).max() <= 2e-5
        assert np.linalg.norm(G @ V[b] - V[b] * lam[:r], axis=0).max() <= 2e-5 * lam[0]
        # first-order perturbation: the sine of the angle to the exact vector is at most |dG| / gap
        gap = np.minimum(np.abs(np.diff(lam, prepend=np.inf))[:r], np.abs(np.diff(lam, append=-np.inf))[:r])
        sine = np.sqrt(np.maximum(0.0, 1 - np.abs(np.sum(V[b] * vec[:, :r], axis=0)).clip(0, 1) ** 2))
        clear = gap > 8 * eps
        assert clear[0] and np.all(sine[clear] <= 2 * eps / gap[clear] + 2e-3), (sine[clear], eps / gap[clear])


@pytest.mark.parametrize("kind", ["rank r/2", "orthogonal columns"])
@pytest.mark.parametrize("d,r", [(64, 16), (64, 32), (64, 64), (128, 16), (128, 64)])
def test_eigenvalues_apart_by_rounding_errors_only(d, r, kind):
    """Kept eigenvalues that are zero, or all the same, but for the rounding errors of the Gram matrix: the
    minors of T - lambda I shrink by those errors from row to row, and the fp64 chain has to follow them."""
    rng = np.random.default_rng(d + 3 * r)
    B, N = 6, 1000
    H = np.empty((B, N, d), np.float32)
    for b in range(B):
        if kind == "rank r/2":
            H[b] = rng.standard_normal((N, r // 2)) @ rng.standard_normal((r // 2, d))
        else:
            H[b] = np.linalg.qr(rng.standard_normal((N, d)))[0] * np.sqrt(N)
    ws = solar.alloc_workspace(B, 1, N, d, r, torch.float32)
    S = torch.empty(B, r, device="cuda"); V = torch.empty(B, d, r, device="cuda")
    info = torch.full((B,), -1, dtype=torch.int32, device="cuda"); taken = torch.zeros_like(info)
    solar.gram_partials(torch.from_numpy(H).cuda(), ws)
    solar.eig_from_partials_ex(B, N, d, r, torch.float32, solar.ROUTE_AUTO, S, V, info, taken, ws)
    torch.cuda.synchronize()
    assert info.tolist() == [0] * B
    assert [t & 0xffff for t in taken.tolist()] == [2 | (1 << 8)] * B, [hex(t & 0xffffffff) for t in taken.tolist()]
    S, V = S.cpu().numpy().astype(np.float64), V.cpu().numpy().astype(np.float64)
    for b in range(B):
        G = H[b].astype(np.float64).T @ H[b].astype(np.float64)
        lam = np.linalg.eigvalsh(G)[::-1]
        eps = 16 * 2.0 ** -24 * lam[0]                 # the kernel's Gram matrix: a few 2^-24 lambda_1
        assert np.all(np.abs(S[b] ** 2 - lam[:r]) <= eps)
        assert np.abs(V[b].T @ V[b] - np.eye(r)).max() <= 2e-5
        assert np.linalg.norm(G @ V[b] - V[b] * lam[:r], axis=0).max() <= 2e-5 * lam[0]
