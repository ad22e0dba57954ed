"""The certificate's condition on the rows that the tridiagonal reduction leaves out (csrc/eig_rest.cuh, compiled
for the host) on reductions that are ended, wrongly, at every row: an end that loses a kept eigenvalue may pass
the residuals and the traces, never this condition; ends on a decoupled tail and of rank-deficient matrices pass all."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_02561_b200", "csrc")


@pytest.fixture(scope="module")
def keeps_result(tmp_path_factory):
    d = tmp_path_factory.mktemp("rest")
    (d / "cuda_runtime.h").write_text("#define __host__\n#define __device__\n#define __forceinline__ inline\n")
    (d / "rest.cpp").write_text('#include "eig_rest.cuh"\nextern "C" int keeps(float rest, float trace, float theta_last) '
                                "{ return solar::rest_keeps_result(rest, trace, theta_last); }\n")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{d}", f"-I{CSRC}", "-o", str(d / "rest.so"), str(d / "rest.cpp")],
                   check=True)
    fn = ctypes.CDLL(str(d / "rest.so")).keeps
    fn.argtypes, fn.restype = [ctypes.c_float] * 3, ctypes.c_int
    return lambda *a: bool(fn(*a))


def _steps(G):
    """Householder tridiagonalisation: yields (k, T of the rows 0 .. k, coupling of row k, trace of the rows behind)."""
    A, d = G.copy(), len(G)
    for k in range(d - 1):
        x = A[k + 1:, k].copy()
        a = -np.copysign(np.linalg.norm(x), x[0])
        v = x.copy(); v[0] -= a
        if np.linalg.norm(v) > 1e-14 * np.trace(G):
            P = np.eye(d); P[k + 1:, k + 1:] -= 2.0 * np.outer(v, v) / (v @ v)
            A = P @ A @ P
        yield k, A[: k + 1, : k + 1], abs(A[k + 1, k]), np.trace(A[k + 1:, k + 1:])


def _ends(G, r):
    """Per wrong end: do the residuals and traces pass (bf16 bounds), does it lose a kept eigenvalue, the condition's arguments."""
    lam, tr = np.linalg.eigvalsh(G)[::-1], np.trace(G)
    for k, T, e, rest in _steps(G):
        if k < r - 1:
            continue
        th, y = np.linalg.eigh(T)
        th, y = th[::-1][:r], y[:, ::-1][:, :r]
        gap = np.minimum(np.abs(np.diff(th, prepend=np.inf)), np.abs(np.diff(th, append=-np.inf)))
        residuals = np.all(e * np.abs(y[-1]) <= np.maximum(1e-3 * gap, 64 * 2.0 ** -24 * th[0]))
        traces = abs(np.trace(T) + rest - tr) <= 1e-4 * tr
        yield residuals and traces, np.any(np.abs(th - lam[:r]) > 1e-3 * lam[0]), (rest, tr, th[-1])


def _turned(rng, lam):
    Q = np.linalg.qr(rng.standard_normal((len(lam), len(lam))))[0]
    return (Q * lam) @ Q.T


@pytest.mark.parametrize("r", [1, 4, 8])
def test_an_end_that_loses_a_kept_eigenvalue_is_refused(keeps_result, r):
    rng = np.random.default_rng(r)
    wrong_and_certified_without = 0
    for first in (8, 12, 20):
        # two groups of columns that are orthogonal to each other; T decouples behind the first, which holds small eigenvalues
        G = np.zeros((32, 32))
        G[:first, :first] = _turned(rng, np.linspace(1.0, 0.3, first))
        G[first:, first:] = _turned(rng, np.linspace(3.0, 0.1, 32 - first))
        for certified, lost, args in _ends(G, r):
            wrong_and_certified_without += certified and lost
            assert not (certified and lost and keeps_result(*args)), args
    assert wrong_and_certified_without >= 3


@pytest.mark.parametrize("r,rank,noise", [(8, 8, 1e-3), (8, 8, 3e-2), (5, 8, 1e-4), (8, 4, 0.0), (1, 3, 0.0)])
def test_a_sound_end_is_accepted(keeps_result, r, rank, noise):
    rng = np.random.default_rng(rank)
    lam = np.concatenate([np.linspace(3.0, 1.0, rank), noise ** 2 * np.linspace(2.0, 1.0, 32 - rank)])
    accepted = [k for k, (certified, lost, args) in enumerate(_ends(_turned(rng, lam), r)) if certified and keeps_result(*args)]
    assert accepted and accepted[0] <= max(rank - r, 0) + 8          # from a few rows behind the rank on
    assert not keeps_result(float("nan"), 1.0, 1.0) and not keeps_result(1.0, 1.0, float("nan"))
