"""Solves on one handle keep to their own tolerance and iteration limit, call
after call: an iteration's recorded launches hold nothing of the call that
recorded them.  Sizes around one block, one pass of the grid and more rows
than the grid's threads (the vector kernels' reductions)."""
import numpy as np
import pytest

from oracle import hsolver as H
from paper_1611_03189_gb300 import problems as P

from gpu_util import gpu_factor, need_gpu, oracle_factor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(3, 5), (16, 16), (257, 1), (411, 401)])
def test_each_solve_stops_at_its_own_tolerance(shape):
    torch = need_gpu()
    pb = P.poisson2d(*shape, leaf_size=16) if min(shape) > 1 else P.make_problem(shape, P.coef_constant(shape), 16)
    G = gpu_factor(pb, 1e-1, 0)
    b = P.rhs(pb.n, 3)
    bd = torch.as_tensor(b, device="cuda")
    A = pb.to_scipy()
    last = 0
    for rtol in (1e-3, 1e-10, 1e-6):
        x, it, rr, _ = G.pcg(bd, rtol=rtol)
        true = np.linalg.norm(b - A @ x.cpu().numpy()) / np.linalg.norm(b)
        # the recursive residual stops the solve; the true one differs by rounding only
        assert rr[0] <= 1.01 * rtol and abs(true - rr[0]) <= 1e-13 + 1e-6 * rr[0], (rtol, rr, true)
        if pb.n < 10000:
            F = oracle_factor(pb, 1e-1, H.LORASP)
            xo, ito, _ = H.pcg(F, pb.rowptr, pb.col, pb.val, b, rtol=rtol, maxit=500)
            assert abs(int(it[0]) - int(ito)) <= 1, (rtol, it, ito)
    with pytest.raises(Exception):
        G.pcg(bd, rtol=1e-30, maxit=1)
    G.close()
