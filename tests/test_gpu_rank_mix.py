"""The rank decision of a node does not depend on the other nodes of its launch.

Small and large nodes in one wave of a batch: the large ones' Z = Q^T X with four
preserved vectors does not fit shared memory (FP64 from 1761 unknowns on), which
moves only theirs out of it, with the recurrences that go with that.  At tolerances
around one where its ranks change the small problem has the ranks, and the bits,
that it has alone.
"""
import numpy as np
import pytest

from oracle import hsolver as H
from paper_1611_03189_gb300 import problems as P

from gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu


def _strip(a, b, seed):
    shape = (4 * a, b)
    return P.make_problem(shape, P.coef_lognormal(shape, 0.5, seed), levels=3)


def _ranks(f):
    return np.concatenate([f.ranks(level) for level in (2, 3)])


@pytest.mark.parametrize("side", [(16, 5)])
def test_small_nodes_beside_large_ones_keep_their_ranks_and_bits(side):
    torch = need_gpu()
    from paper_1611_03189_gb300 import _lib

    pbs = [_strip(*side, 1), _strip(60, 30, 2)]
    rng = np.random.default_rng(5)
    Xs = [rng.standard_normal((pb.n, 4)) for pb in pbs]
    args = [to_dev(pb) + (pb.perm, pb.leaf_ptr) for pb in pbs]

    def factors(count, eps):
        fs, status = _lib.factor_batch(args[:count], eps, H.GC_USER, 0, phis=Xs[:count])
        assert list(status) == [0] * count
        return fs

    def alone(eps):
        f, = factors(1, eps)
        r = _ranks(f)
        f.close()
        return r

    # a tolerance at which the small problem's ranks change, to the last bits
    lo, hi = 1e-4, 1e-1
    low = alone(lo)
    while hi - lo > 4e-16 * hi:
        mid = 0.5 * (lo + hi)
        if np.array_equal(alone(mid), low):
            lo = mid
        else:
            hi = mid
    b = torch.as_tensor(P.rhs(pbs[0].n, 5, nrhs=2).T.copy(), device="cuda")
    for j in range(-3, 4):
        eps = lo * (1.0 + j * 2.2e-16)
        one, two = factors(1, eps), factors(2, eps)
        assert two[1].info()["max_super"] > 1760
        assert np.array_equal(_ranks(one[0]), _ranks(two[0])), j
        assert torch.equal(one[0].apply(b), two[0].apply(b)), j
        for f in one + two:
            f.close()
