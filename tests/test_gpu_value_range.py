"""The truncation does not depend on the scale of the matrix.

A times a power of two has the ranks of A, and its preconditioner is that of A
divided by the power.  At 2^-46 (FP32; 2^-440 FP64) the squares of the well-separated
blocks' entries are far below any absolute floor near 1e-30 and their fourth powers
below the type's range; at 2^46 (2^440) the fourth powers are above it.  Bars: equal
ranks, the application within the parity tests' 1e-3 (FP32 factor) and 1e-10 (FP64).
"""
import numpy as np
import pytest

from oracle import hsolver as H
from paper_1611_03189_gb300 import problems as P

from gpu_util import elem, gpu_factor, need_gpu, oracle_factor

pytestmark = pytest.mark.gpu


def _problem():
    # super nodes of 24 unknowns at the leaves, ranks that add up to other sizes above
    return P.diffusion2d(48, 1.0, 3, leaf_size=12)


@pytest.mark.parametrize("power", [-46, 46])
@pytest.mark.parametrize("variant", [H.LORASP, H.GC_CONSTANT])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_ranks_and_application_follow_the_scale(prec, variant, power):
    torch = need_gpu()
    p = 1 if prec == "f32" else 0
    scale = 2.0 ** (power if prec == "f32" else power * 440 // 46)
    pb = _problem()
    b = torch.as_tensor(P.rhs(pb.n, 5, nrhs=2).T.copy(), device="cuda")
    G = gpu_factor(pb, 1e-2, variant, prec=p)
    z = G.apply(b).cpu().numpy()
    ranks = [G.ranks(level) for level in range(2, pb.levels + 1)]
    x, it, _, _ = G.pcg(b)
    assert sum(int((r > 16).sum()) for r in ranks) > 0 and G.info()["max_super"] > 32
    pb.val = pb.val * scale
    S = gpu_factor(pb, 1e-2, variant, prec=p)
    for level, r in zip(range(2, pb.levels + 1), ranks):
        assert np.array_equal(S.ranks(level), r), level
    assert elem((S.apply(b).cpu().numpy() * scale).T, z.T) <= (1e-3 if p else 1e-10)
    y, its, _, _ = S.pcg(b)
    assert np.abs(its - it).max() <= 1
    assert elem((y * scale).cpu().numpy().T, x.cpu().numpy().T) <= 1e-6


def test_a_chain_coupled_by_the_square_root_of_the_range_keeps_its_rank():
    """A chain of 257 unknowns couples its ends by 1e-149, whose square the Gram
    matrix holds: a normal FP64 number, and the block has rank one."""
    need_gpu()
    shape = (4 * 257, 1)
    pb = P.make_problem(shape, P.coef_lognormal(shape, 0.5, 3), levels=3)
    F = oracle_factor(pb, 1e-2, H.LORASP)
    G = gpu_factor(pb, 1e-2, H.LORASP)
    for level, ranks in F.ranks().items():
        g = G.ranks(level)
        assert {i: int(g[i]) for i in ranks} == ranks, level
