"""Columns of the Gram matrix with a small tail beside a large first entry.

Four super nodes of m unknowns in a chain; eliminating two couples the other two by
S = G^(1/2) (scaled), so each of those is truncated with the Gram matrix G.  G's leading
2 x 2 block [[d, d - delta], [d - delta, d]] has the eigenvalue delta, equal to G_22, and a
coupling t of the two splits them to delta -+ t / 2^(1/2): one lies above the threshold, one
below.  t is 2e-4 (FP64: 1.2e-8) of the entry d - delta beside it in the column, so a
tridiagonalisation that forms |tail|^2 as a difference of rounded squares can drop it
and keep both.  Every d is a case of its own.  Expected: the ranks of LoRaSp by
definition, sigma > eps ||S||.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def check(m, prec):
    import torch

    from paper_1611_03189_gb300 import _lib

    rel = 2e-4 if prec == 1 else 1.2e-8
    for d in np.linspace(0.52, 0.92, 9):
        t = rel * d
        delta = 1.1 * t / np.sqrt(2)
        G = np.diag(np.r_[d, d, delta, np.linspace(0.3, 0.4, m - 3)])
        G[0, 1] = G[1, 0] = d - delta
        G[0, 2] = G[2, 0] = t
        lam, V = np.linalg.eigh(G)
        S = (V * np.sqrt(np.maximum(lam, 0.0))) @ V.T
        eps = np.sqrt(0.55 * t / np.sqrt(2) / lam[-1])
        want = int((lam > eps * eps * lam[-1]).sum())
        assert want == m - 1
        n = 4 * m
        A = 4.0 * np.eye(n)
        for i, B in ((0, S), (1, np.eye(m)), (2, S)):
            r, c = slice(i * m, i * m + m), slice(i * m + m, i * m + 2 * m)
            A[r, c] = B
            A[c, r] = B.T
        rows, cols = np.nonzero(A)
        rp = np.searchsorted(rows, np.arange(n + 1)).astype(np.int32)
        F = _lib.Factor(torch.as_tensor(rp, device="cuda"), torch.as_tensor(cols.astype(np.int32), device="cuda"),
                        torch.as_tensor(A[rows, cols], device="cuda"), np.arange(n, dtype=np.int32),
                        np.arange(0, n + 1, m // 2, dtype=np.int32), eps, 0, prec)
        k = F.ranks(3)
        assert (k >= 0).any() and all(int(x) == want for x in k if x >= 0), (m, prec, d, k, want)
        F.close()


@pytest.mark.parametrize("prec", [1, 0], ids=["f32", "f64"])
@pytest.mark.parametrize("m", [20, 130, 300])
def test_on_chip(m, prec):
    need_gpu()
    check(m, prec)


def test_step_kernels():
    need_gpu()
    code = f"""
import sys
sys.path.insert(0, {os.path.dirname(HERE)!r})
sys.path.insert(0, {HERE!r})
import test_gpu_small_tails as T
for m in (20, 130):
    for prec in (1, 0):
        T.check(m, prec)
print('ok')
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                       env=dict(os.environ, HS_TRI_CLUSTER="0"))
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]
