"""The apply's launches over many right-hand-side counts and odd node sizes.

The forward and backward launches pass 1, 2, 4, 8 or 16 right-hand sides at a
time, with 16-byte loads when the chunk is full and aligned.  Every count must
match the oracle (FP64, within 1e-10 element-wise: both sides apply the same
operator with backward-stable steps) and each column must have the bits of the
column applied alone.
"""
import numpy as np
import pytest

from oracle import hsolver as H
from paper_1611_03189_gb300 import problems as P

from gpu_util import elem, gpu_factor, need_gpu, oracle_factor

pytestmark = pytest.mark.gpu

PROBLEMS = {
    "edge": lambda: P.poisson2d(33, 21, leaf_size=8),       # neighbours alive at elimination: none to few
    "ragged3d": lambda: P.poisson3d(11, 7, 9, leaf_size=24),
    "tiny": lambda: P.poisson2d(5, 4, leaf_size=3),
}


@pytest.mark.parametrize("name", sorted(PROBLEMS))
@pytest.mark.parametrize("nbr", [1, 2])
def test_columns_match_the_oracle_and_their_own_solo_bits(name, nbr):
    torch = need_gpu()
    from paper_1611_03189_gb300 import _lib
    from gpu_util import to_dev

    pb = PROBLEMS[name]()
    F = H.factor(pb.n, pb.rowptr, pb.col, pb.val, pb.perm, pb.leaf_ptr, 1e-2, H.GC_CONSTANT, nbr_dist=nbr)
    B = P.rhs(pb.n, 7, nrhs=33)
    zo = H.apply(F, B)
    for prec in (_lib.HS_PREC_F64, _lib.HS_PREC_F32):
        G = _lib.Factor(*to_dev(pb), pb.perm, pb.leaf_ptr, 1e-2, _lib.HS_GC_CONSTANT, prec, nbr_dist=nbr)
        R = torch.as_tensor(B.T.copy(), device="cuda")
        solo = torch.stack([G.apply(R[j]) for j in range(33)])
        if prec == _lib.HS_PREC_F64:
            assert elem(solo.cpu().numpy().T, zo) <= 1e-10
        for nrhs in (2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 20, 32, 33):
            z = G.apply(R[:nrhs].contiguous())
            assert torch.equal(z, solo[:nrhs]), (prec, nrhs)
        G.close()
