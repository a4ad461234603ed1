"""Node sizes at the edges of the truncation's and the Cholesky-inverse's tiles
and size classes, against the oracle.

A strip of 4 a x b unknowns in eight leaves has four super nodes of a b unknowns
at its first level; eliminating two of them couples the other two, so at least
one node of exactly m = a b unknowns is compressed.  The sizes lie on both
sides of the limits of the Jacobi path, of the lanes per eigenvalue, of the
registers per column of the reflector products and of their threads, of the
16-column blocks of the Cholesky and of its clusters, and of the clusters of
the FP64 tridiagonalisation.  Bars as in the parity tests: equal
ranks and the apply within 1e-10 element-wise in FP64; in FP32 a PCG within
two iterations of the FP64 factor's, to the same solution.
"""
import numpy as np
import pytest

from oracle import hsolver as H
from paper_1611_03189_gb300 import problems as P

from gpu_util import elem, gpu_factor, need_gpu, oracle_factor

pytestmark = pytest.mark.gpu

SIZES = [(3, 3), (5, 3), (4, 4), (17, 1), (31, 1), (8, 4), (11, 3), (9, 7), (8, 8), (13, 5), (127, 1), (16, 8),
         (43, 3), (15, 11), (32, 7), (15, 15), (17, 15), (16, 16), (257, 1), (27, 19), (41, 25), (32, 3), (97, 1), (161, 1), (40, 39)]


@pytest.mark.parametrize("ab", SIZES, ids=lambda ab: str(ab[0] * ab[1]))
@pytest.mark.parametrize("variant", [H.LORASP, H.GC_CONSTANT])
def test_edge_sizes_match_the_oracle(ab, variant):
    torch = need_gpu()
    a, b = ab
    shape = (4 * a, b)
    pb = P.make_problem(shape, P.coef_lognormal(shape, 0.5, 3), levels=3)
    F = oracle_factor(pb, 1e-2, variant)
    G = gpu_factor(pb, 1e-2, variant)
    assert G.info()["max_super"] >= a * b
    # the 257-unknown chain couples its ends by 1e-149: the square, which the
    # Gram matrix of LoRaSp holds, is outside the FP64 range, and the block is
    # dropped (GC takes A_sw phi_w itself)
    beyond = ab == (257, 1) and variant == H.LORASP
    for level, ranks in ({} if beyond else F.ranks()).items():
        g = G.ranks(level)
        assert {i: int(g[i]) for i in ranks} == ranks, level
    B = P.rhs(pb.n, 5, nrhs=2)
    z = G.apply(torch.as_tensor(B.T.copy(), device="cuda")).cpu().numpy().T
    assert elem(z, H.apply(F, B)) <= 1e-10
    bd = torch.as_tensor(B[:, 0].copy(), device="cuda")
    x, it, rr, _ = G.pcg(bd)
    G32 = gpu_factor(pb, 1e-2, variant, prec=1)
    x32, it32, rr32, _ = G32.pcg(bd)
    assert rr[0] <= 1.01e-10 and rr32[0] <= 1.01e-10 and abs(int(it32[0]) - int(it[0])) <= 2
    assert elem(x32.cpu().numpy(), x.cpu().numpy()) <= 1e-6
