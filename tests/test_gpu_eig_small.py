"""The truncations' eigensolver at the sizes where its kernels change (register tridiagonalisation up to 32, 64 and 96
rows, shared and global memory above) against LAPACK: graded and very steep spectra, spectra with equal and with nearly equal wanted
eigenvalues, k up to n.  Tolerances as for the eigensolver elsewhere: eigenvalues and residuals within 64 n eps ||A||,
orthonormality 1e-12."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _matrix(n, kind, seed):
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    if kind == "steep":  # entries down to 1e-200: squares and their products leave the range of FP64
        D = 10.0 ** (-100.0 * np.arange(n) / max(n - 1, 1))
        A = D[:, None] * ((q * rng.uniform(0.1, 1.0, n)) @ q.T) * D
        return (A + A.T) / 2
    lam = {"graded": 10.0 ** (-12.0 * np.arange(n) / max(n - 1, 1)),
           "pairs": np.repeat(np.linspace(1.0, 0.1, (n + 1) // 2), 2)[:n],
           "near": 1.0 - 1e-13 * np.arange(n),
           "rank2": np.where(np.arange(n) < 2, 1.0 + np.arange(n), 0.0)}[kind]
    A = (q * lam) @ q.T
    return (A + A.T) / 2


@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 64, 65, 96, 97, 160])
@pytest.mark.parametrize("kind", ["graded", "pairs", "near", "rank2", "steep"])
def test_sizes(ctx, n, kind):
    k = min(n, 33)
    A = np.stack([_matrix(n, kind, s) for s in range(2)])
    w, V = ctx.sym_eig(torch.as_tensor(A, device="cuda"), k)
    w, V = w.cpu().numpy(), V.cpu().numpy()
    for b in range(2):
        ref = np.linalg.eigvalsh(A[b])[::-1][:k]
        tol = 64 * n * np.finfo(float).eps * np.abs(np.linalg.eigvalsh(A[b])).max()
        assert np.abs(w[b] - ref).max() <= tol
        assert np.abs(A[b] @ V[b] - V[b] * w[b]).max() <= tol
        assert np.abs(V[b].T @ V[b] - np.eye(k)).max() <= 1e-12
