"""Paths that only some sizes or settings take, forced and compared.

Several preserved vectors through the step kernels and the smallest clusters; FP32
nodes between 1025 and 2048 unknowns (step kernels with a 16-CTA tail, the widest
warps of the products with Q) element by element; the rank decision of nodes beyond
shared memory; recorded solve iterations under another tolerance and iteration limit.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle import hsolver as H
from paper_1611_03189_gb300 import problems as P

from gpu_util import elem, gpu_factor, need_gpu, oracle_factor

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("cluster", ["0", "1", "2"], ids=["steps", "cta", "cluster"])
def test_several_vectors_on_every_tridiagonalisation(cluster):
    need_gpu()
    code = f"""
import sys
sys.path.insert(0, {os.path.dirname(HERE)!r})
sys.path.insert(0, {HERE!r})
import test_gpu_multi_phi as T
for name in ("poisson32 3 eigenvectors", "poisson64 projection 4"):
    for eps in (1e-1, 1e-2):
        T.check_case(name, eps, fp32=(eps == 1e-1))
print('ok')
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                       env=dict(os.environ, HS_EIG_SMALL_MAX="8", HS_TRI_CLUSTER=cluster))
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]


@pytest.mark.parametrize("ab", [(40, 26), (41, 38)], ids=lambda ab: str(ab[0] * ab[1]))
@pytest.mark.parametrize("variant", [H.LORASP, H.GC_CONSTANT])
def test_fp32_application_of_large_nodes(ab, variant):
    torch = need_gpu()
    a, b = ab
    pb = P.make_problem((4 * a, b), P.coef_lognormal((4 * a, b), 0.5, 3), levels=3)
    F = oracle_factor(pb, 1e-2, variant)
    G = gpu_factor(pb, 1e-2, variant, prec=1)
    assert G.info()["max_super"] >= a * b
    B = P.rhs(pb.n, 5, nrhs=2)
    z = G.apply(torch.as_tensor(B.T.copy(), device="cuda")).cpu().numpy().T
    assert elem(z, H.apply(F, B)) <= 1e-3


def test_rank_of_nodes_beyond_shared_memory():
    """FP32 nodes of 8400 unknowns: T and Z stay in global memory.  Two of four nodes
    in a chain are coupled by the diagonal matrix S alone, so the ranks are counts."""
    torch = need_gpu()
    from paper_1611_03189_gb300 import _lib

    m = 8400
    s = np.r_[np.linspace(1.0, 0.5, m // 2), np.linspace(2e-3, 1e-3, m - m // 2)]
    s = s[np.random.default_rng(1).permutation(m)]
    i = np.arange(m)
    one = np.ones(m)
    rows = np.concatenate([np.arange(4 * m), i, m + i, 2 * m + i, m + i, 2 * m + i, 3 * m + i])
    cols = np.concatenate([np.arange(4 * m), m + i, 2 * m + i, 3 * m + i, i, m + i, 2 * m + i])
    vals = np.concatenate([4.0 * np.ones(4 * m), s, one, s, s, one, s])
    import scipy.sparse as sp

    A = sp.csr_matrix((vals, (rows, cols)))
    A.sort_indices()
    F = _lib.Factor(torch.as_tensor(A.indptr.astype(np.int32), device="cuda"),
                    torch.as_tensor(A.indices.astype(np.int32), device="cuda"),
                    torch.as_tensor(A.data, device="cuda"), np.arange(4 * m, dtype=np.int32),
                    np.arange(0, 4 * m + 1, m // 2, dtype=np.int32), 1e-2, H.LORASP, 1)
    k = F.ranks(3)
    assert (k >= 0).any() and all(int(x) == m // 2 for x in k if x >= 0), k
    b = torch.as_tensor(P.rhs(4 * m, 3), device="cuda")
    x, it, rr, _ = F.pcg(b)
    assert rr[0] <= 1.01e-10 and it[0] <= 6, (it, rr)
    F.close()


@pytest.mark.parametrize("shape", [(16, 16), (61, 47)])
def test_recorded_iterations_hold_nothing_of_a_call(shape):
    """A factorization's first iterations are launched directly, later ones replayed:
    after enough solves at one tolerance every call still keeps to its own."""
    torch = need_gpu()
    from paper_1611_03189_gb300 import _lib

    pb = P.poisson2d(*shape, leaf_size=16)
    G = gpu_factor(pb, 0.3, H.LORASP)
    bd = torch.as_tensor(P.rhs(pb.n, 3), device="cuda")
    _, it, _, _ = G.pcg(bd, rtol=1e-3)
    n0 = int(it[0])
    assert n0 >= 1
    for _ in range(12 // n0 + 2):   # past the direct ones
        _, it, _, _ = G.pcg(bd, rtol=1e-3)
        assert int(it[0]) == n0
    _, it, rr, code = G.pcg(bd, rtol=1e-10)
    assert code == _lib.HS_OK and rr[0] <= 1.01e-10 and int(it[0]) > n0
    n1 = int(it[0])
    _, it, rr, code = G.pcg(bd, rtol=1e-10, maxit=n1 - 1, raise_on_fail=False)
    assert code == _lib.HS_ERR_NO_CONVERGENCE and int(it[0]) == n1 - 1 and rr[0] > 1e-10
    _, it, rr, code = G.pcg(bd, rtol=1e-3)
    assert code == _lib.HS_OK and int(it[0]) == n0
    G.close()
