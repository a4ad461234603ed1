"""The blocked Cholesky-inverse against elimination column by column.

A matrix that is one leaf is its own root: the application is A^-1 = X^T X with
X = L^-1 of the kernel.  Its error against the inverse in higher precision may be
no larger than that of the textbook elimination (columns one after another,
substitution for X) in the same precision, emulated in numpy, up to the spread of
a mean over the matrices; 1.5 covers that spread and the product X^T X.  The
spectra are graded, condition 1e5, where a block's explicit inverse in the place
of a substitution shows (a factor of 2 at sizes just above one block).  Sizes: the
edges of the 16-column blocks, of the thread counts and of the FP64 clusters.
"""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

COUNT = 32


def _matrices(m, dtype):
    rng = np.random.default_rng(m)
    lam = 10.0 ** (-5.0 * np.arange(m) / max(m - 1, 1))
    out = np.empty((COUNT, m, m))
    for q in range(COUNT):
        Q = np.linalg.qr(rng.standard_normal((m, m)))[0]
        A = (Q * lam) @ Q.T
        out[q] = (0.5 * (A + A.T)).astype(dtype)
    return out


def _chol_inverse(A, dtype):
    """X^T X, X = L^-1, column by column in `dtype`, all matrices together."""
    W = np.array(A, dtype=dtype)
    n, m, _ = W.shape
    L = np.zeros_like(W)
    for j in range(m):
        L[:, j, j] = np.sqrt(W[:, j, j])
        L[:, j + 1:, j] = W[:, j + 1:, j] / L[:, j, j, None]
        W[:, j + 1:, j + 1:] -= L[:, j + 1:, j, None] * L[:, None, j + 1:, j]
    X = np.zeros_like(W)
    for i in range(m):
        r = np.zeros((n, m), dtype=dtype)
        r[:, i] = 1
        for p in range(i):
            r -= L[:, i, p, None] * X[:, p]
        X[:, i] = r / L[:, i, i, None]
    M = np.zeros_like(W)
    for k in range(m):
        M += X[:, k, :, None] * X[:, k, None, :]
    return M


@pytest.mark.parametrize("m", [8, 16, 17, 31, 32, 33, 49, 97, 128, 160])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_error_is_that_of_elimination_column_by_column(prec, m):
    torch = need_gpu()
    from paper_1611_03189_gb300 import _lib

    dtype, high = (np.float32, np.float64) if prec == "f32" else (np.float64, np.longdouble)
    A = _matrices(m, dtype)
    exact = _chol_inverse(A, high)
    plain = _chol_inverse(A, dtype)
    rp = torch.arange(0, m * m + 1, m, dtype=torch.int32, device="cuda")
    ci = torch.arange(m, dtype=torch.int32, device="cuda").repeat(m)
    eye = torch.eye(m, dtype=torch.float64, device="cuda")
    errs = []
    for q in range(COUNT):
        G = _lib.Factor(rp, ci, torch.as_tensor(A[q].reshape(-1).copy(), device="cuda"), np.arange(m, dtype=np.int32),
                        np.array([0, m], dtype=np.int32), 0.0, 0, 1 if prec == "f32" else 0)
        Z = torch.cat([G.apply(eye[c:c + 32].contiguous()) for c in range(0, m, 32)]).cpu().numpy()
        errs.append(float(np.linalg.norm((Z - exact[q]).astype(np.float64)) / np.linalg.norm(exact[q].astype(np.float64))))
        G.close()
    ref = [float(np.linalg.norm((plain[q] - exact[q]).astype(np.float64)) / np.linalg.norm(exact[q].astype(np.float64)))
           for q in range(COUNT)]
    assert np.mean(errs) <= 1.5 * np.mean(ref), (np.mean(errs), np.mean(ref))
