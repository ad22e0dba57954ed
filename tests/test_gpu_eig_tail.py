"""Where the tridiagonal reduction ends because the kept vectors do not reach the rows behind (a history of
rank R plus noise, whose remaining rows stay far above the rounding level): R at the edges of the kernel's
stages of live columns and near the end of the matrix, noise from just above the rounding level to a
twentieth of the smallest kept singular value, and R below r, where nothing may end early on the noise."""
import numpy as np
import pytest
import torch

from paper_2603_02561_b200 import solar

pytestmark = pytest.mark.gpu


def _histories(d, ranks, noises, N, seed):
    rng = np.random.default_rng(seed)
    H = []
    for R in ranks:
        for noise in noises:
            U, _ = np.linalg.qr(rng.standard_normal((N, d)))
            W, _ = np.linalg.qr(rng.standard_normal((d, d)))
            s = noise * (2.0 - np.arange(d) / d)                  # the noise directions are apart from each other too
            s[:R] = 3.0 - 2.0 * np.arange(R) / R
            H.append((U * s) @ W.T)
    return np.stack(H).astype(np.float32)


@pytest.mark.parametrize("d", [32, 64, 128])
def test_the_reduction_may_end_on_a_tail(d):
    ranks = sorted({R for e in range(8, d, 16) for R in (e - 1, e, e + 1)} | {2, d - 12, d - 9, d - 7, d - 4, d - 2})
    H = _histories(d, ranks, (0.05, 3e-3, 1e-4), 300, d)
    exact = [np.linalg.svd(h.astype(np.float64), full_matrices=False) for h in H]
    for r in sorted({1, 8, min(d, 32) - 3, min(d, 64) - 3}):
        keep = [i for i in range(len(H)) if ranks[i // 3] >= r]
        info = torch.full((len(keep),), -1, dtype=torch.int32, device="cuda")
        S, V = solar.lowrank_factor(torch.from_numpy(H[keep]).cuda(), r, info=info)
        torch.cuda.synchronize()
        S, V = S.cpu().numpy().astype(np.float64), V.cpu().numpy().astype(np.float64)
        assert torch.all(info == 0)
        # the bounds of the test of the reduction's other early end
        assert np.abs(S - np.stack([exact[i][1][:r] for i in keep])).max() <= 1e-5 * 3.0
        assert np.abs(np.einsum("bki,bkj->bij", V, V) - np.eye(r)).max() <= 2e-5
        G = np.einsum("bni,bnj->bij", H[keep].astype(np.float64), H[keep].astype(np.float64))
        assert np.abs(G @ V - V * (S ** 2)[:, None, :]).max() <= 2e-5 * 9.0


@pytest.mark.parametrize("d,R,r", [(64, 8, 16), (64, 16, 17), (128, 20, 32), (32, 4, 8)])
def test_a_tail_that_holds_kept_directions_is_reduced_too(d, R, r):
    H = _histories(d, [R], (0.05, 0.02), 300, 7 * d + r)
    S, V = solar.lowrank_factor(torch.from_numpy(H).cuda(), r)
    S = S.cpu().numpy().astype(np.float64)
    for b in range(len(H)):
        # fp32 Gram matrix: eigenvalues to 2^-22 of the largest (9), singular values of the noise (0.02 and more) to
        # 9 * 2^-22 / (2 * 0.02) = 5.4e-5
        assert np.abs(S[b] - np.linalg.svd(H[b].astype(np.float64), compute_uv=False)[:r]).max() <= 5.4e-5


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d", [32, 64, 128])
def test_where_the_reduction_ends(d, dtype):
    """The fp32 chain itself certifies every one of these users (the default route would hide a wrong end behind
    the chains that follow it), and T has as many rows as the tail asks for."""
    ranks = sorted({R for e in range(8, d, 16) for R in (e - 1, e, e + 1)} | {2, d - 12, d - 9, d - 7, d - 4, d - 2})
    noises = (0.05, 3e-3, 1e-4)
    # Behind row R the bound on what a kept vector leaves falls, from row to row, by the coupling of two noise rows (about a
    # quarter of the spread of their eigenvalues, 3 noise^2) over x / 2; it starts once the trace of the rest is below x / 2, for
    # the largest noise at d = 128 (0.7, against kept eigenvalues from 1) only some rows further on.  2^-28 in the
    # end: three to thirteen rows.
    slack = (16, 12, 10)
    H = torch.from_numpy(_histories(d, ranks, noises, 300, d)).cuda().to(dtype)
    for r in sorted({1, 8, min(d, 32) - 3, min(d, 64) - 3}):
        keep = [i for i in range(len(H)) if ranks[i // 3] >= r]
        B = len(keep)
        S, V = torch.empty(B, r, device="cuda"), torch.empty(B, d, r, device="cuda")
        info = torch.full((B,), -1, dtype=torch.int32, device="cuda")
        taken = torch.full_like(info, -1)
        ws = solar.alloc_workspace(B, 1, 300, d, r, dtype)
        solar.gram_partials(H[keep].contiguous(), ws)
        parts = solar.gram_splits(B, 300, d, dtype)
        G = ws[: B * parts * d * d * 4].view(torch.float32).reshape(B, parts, d, d).double().sum(1)
        solar.eig_from_partials_ex(B, 300, d, r, dtype, solar.ROUTE_AUTO, S, V, info, taken, ws)
        for i, word in zip(keep, taken.tolist()):
            R, tag = ranks[i // 3], (ranks[i // 3], noises[i % 3], r, hex(word & 0xFFFFFFFF))
            assert word & 0xFF == 3 and (word >> 24) & 0xFF == 0, tag
            rows = (word >> 8) & 0xFF
            assert R < rows <= d, tag
            if R + slack[i % 3] < d:
                assert rows <= R + slack[i % 3], tag
        assert torch.all(info == 0)
        # what the end leaves is below the rounding of the chain: a few 2^-24 of the largest eigenvalue (9), and far below
        # what the certificate lets pass
        left = (G @ V.double() - V.double() * (S.double() ** 2)[:, None, :]).norm(dim=1)
        assert float(left.max()) <= 32 * 2.0 ** -24 * 9.0, r


def test_a_noise_direction_that_is_kept_keeps_its_rows():
    """One of the noise directions is among the kept ones: the rest still holds as much as it, and T goes through."""
    H = torch.from_numpy(_histories(64, [16], (0.05, 0.02), 300, 7 * 64 + 17)).cuda()
    S, V = torch.empty(2, 17, device="cuda"), torch.empty(2, 64, 17, device="cuda")
    taken = torch.full((2,), -1, dtype=torch.int32, device="cuda")
    ws = solar.alloc_workspace(2, 1, 300, 64, 17, torch.float32)
    solar.gram_partials(H, ws)
    solar.eig_from_partials_ex(2, 300, 64, 17, torch.float32, solar.ROUTE_AUTO, S, V, None, taken, ws)
    assert [t & 0xFFFF for t in taken.tolist()] == [3 | (64 << 8)] * 2, [hex(t) for t in taken.tolist()]
