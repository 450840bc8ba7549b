"""Rounding errors of the FP64 gain solve against extended precision: about
those of a Cholesky factorisation and substitutions in FP64, also for fewer
observations than members, where S has many eigenvalues of one beside large
ones (conditions of 1e3 and 1e10)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_10091_gb300 import mgenkf
    return mgenkf


def _gain(Y, Z, sigma, t):
    """T = (I + Y Y^T / sigma^2)^-1 Y Z^T / sigma^2 in the type t, one product at a time."""
    Y, Z, s2 = Y.astype(t), Z.astype(t), t(sigma) ** 2
    n = len(Y)
    S, X = np.zeros((n, n), t), np.zeros((n, n + 1), t)
    for k in range(Y.shape[1]):
        S += np.outer(Y[:, k], Y[:, k])
        X += np.outer(Y[:, k], Z[:, k])
    A, X = np.eye(n, dtype=t) + S / s2, X / s2
    L = np.zeros_like(A)
    for k in range(n):
        L[k, k] = np.sqrt(A[k, k])
        L[k + 1:, k] = A[k + 1:, k] / L[k, k]
        A[k + 1:, k + 1:] -= np.outer(L[k + 1:, k], L[k + 1:, k])
    for k in range(n):
        X[k] /= L[k, k]
        X[k + 1:] -= np.outer(L[k + 1:, k], X[k])
    for k in range(n - 1, -1, -1):
        X[k] /= L[k, k]
        X[:k] -= np.outer(L[k, :k], X[k])
    return X.T


# the errors of two FP64 solves of one system differ by their roundings: over
# three systems their ratio stays within a third (plain L D L^T and
# substitutions in place of Cholesky: 0.98 to 1.02); with inverses of L or of its
# diagonal blocks it was 1.6 to 4.5
@pytest.mark.parametrize("n,sigma", [(32, 0.05), (32, 1e-5), (100, 0.05), (100, 1e-5), (128, 1e-5)])
def test_errors_are_those_of_cholesky(M, n, sigma):
    import torch
    if np.finfo(np.longdouble).nmant < 60:
        pytest.skip("no extended precision")
    ny, ratios = n // 3, []
    for seed in range(3):
        rng = np.random.default_rng([seed, n])
        Y, Z = rng.standard_normal((n, ny)) / np.sqrt(n), rng.standard_normal((n + 1, ny))
        T = torch.zeros((n + 1, n), dtype=torch.float64, device="cuda")
        info = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        M.mgk_gain_ensemble_noalloc(torch.tensor(Y, device="cuda"), torch.tensor(Z, device="cuda"), n, ny, sigma, T,
                                    info)
        assert int(info.item()) == 0
        exact = _gain(Y, Z, sigma, np.longdouble)

        def err(x):
            return float(np.sqrt(np.sum((x - exact) ** 2)))

        ratios.append(err(T.cpu().numpy()) / err(_gain(Y, Z, sigma, np.float64)))
    print(n, sigma, ratios)
    assert np.exp(np.mean(np.log(ratios))) <= 4 / 3
