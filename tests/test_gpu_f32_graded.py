"""The FP32 path on matrices whose entries differ by many orders of magnitude.

An iterate is stored as an FP16 hi/lo pair of its values times a power of two, the largest
that keeps the iterate's norm within FP16 (2^15 for X_0), so an entry of X_0 = X / lam~ is
rounded to at worst a step of 2^-39 however small it is.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2507_09165_gb300 import binding as b  # noqa: E402

from _bars import TOL_F  # noqa: E402

DEV = torch.device("cuda")
COEFS, POST = oracle.schedules.schedule("single")


def _wigner(n, seed):
    G = np.random.default_rng(seed).standard_normal((n, n))
    return (G + G.T) / (2.0 * math.sqrt(n))


def _errors(X):
    """(result, exact filter output) in FP64, each projected in the call that the caller makes."""
    X = X.astype(np.float32)
    X = np.triu(X) + np.triu(X, 1).T
    n = X.shape[0]
    Xd = torch.from_numpy(X).to(DEV)
    single, batched = torch.empty_like(Xd), torch.empty_like(Xd)
    info = torch.zeros(b.INFO_BYTES, dtype=torch.uint8, device=DEV)
    binfo = torch.zeros(b.INFO_BYTES, dtype=torch.uint8, device=DEV)
    b.psd_project_ex(n, Xd, n, single, n, "fp32", info)
    b.psd_project_batched(1, b.block_descs([(n, Xd, n, batched, n, binfo)]), "fp32")
    torch.cuda.synchronize()
    lam, Q = np.linalg.eigh(X.astype(np.float64))
    for o, i in ((single, info), (batched, binfo)):
        d = b.info_from_bytes(i.cpu().numpy())
        assert d["status"] == 0
        F = oracle.filter_from_eig(lam, Q, d["lambda_bound"], COEFS, POST)
        yield o.cpu().numpy().astype(np.float64), F


@pytest.mark.parametrize("n", [300, 1000])
def test_graded_matrix(n):
    d = np.logspace(0, -6, n)
    for o, F in _errors(_wigner(n, n) * d[:, None] * d[None, :]):
        assert oracle.rel_err(o, F) <= TOL_F["fp32"]


@pytest.mark.parametrize("m", [100, 333])
def test_block_far_below_the_bound(m):
    # X = diag(A, B) with B at 1e-8 of the bound, where the filter is linear: X_T = K X_0 with
    # K = prod a_t / s_t.  A rounding of X_0's entries, at most 2^-40 each and evenly spread, so
    # 2^-40 / sqrt 3 in the mean, reaches B's part of the result through X_0 and through X_T, and the later
    # iterates' roundings add about a third to it: relative to ||B||_F / 2 that is
    # 2 * 1.35 K sqrt(m) 2^-40 / sqrt 3, and the result itself is rounded to FP32.
    K = float(np.prod([c[0] / s for c, s in zip(COEFS, POST)]))
    X = np.zeros((2 * m, 2 * m))
    X[:m, :m] = _wigner(m, m)
    X[m:, m:] = _wigner(m, m + 1) * 1e-8
    for o, F in _errors(X):
        assert oracle.rel_err(o, F) <= TOL_F["fp32"]
        assert oracle.rel_err(o[m:, m:], F[m:, m:]) <= 2.7 * K * math.sqrt(m) * 2.0 ** -40 / math.sqrt(3.0) + 2.0 ** -24
