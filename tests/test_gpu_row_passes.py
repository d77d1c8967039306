"""Sigma product at the sizes where its row passes can go wrong, against the oracle: one, just
one, and several ranges of staged strings; row blocks (16 or 32 rows) with and without a remainder;
groups of lists (8) and parts (16) that are empty, partial and full; the coefficient table in shared
memory (norb <= 42) and in global memory."""
import pytest

from gpu_common import SIGMA_FP64_RTOL, SIGMA_MIXED_RTOL, rel_maxnorm
from paper_2601_16637_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# 232,448 - 1,024 bytes of shared memory hold 1,808 lines of 128 bytes; norb 29: 407 of them are the table
CASES = [
    (29, 10, 1401, 33), (29, 10, 1402, 31),  # one range exactly; two ranges
    (29, 10, 17, 2803),                      # three ranges on the other side
    (44, 3, 1809, 16), (44, 15, 47, 130),    # coefficients in global memory, one and two ranges
    (42, 4, 948, 15), (43, 4, 948, 15),      # last norb with the table staged, first without; two ranges, one
    (64, 5, 40, 530), (58, 4, 33, 2500),     # orbital pairs of the alpha-beta pass in two parts
    (12, 4, 1, 129), (12, 4, 7, 128), (12, 4, 9, 32), (12, 4, 16, 1), (10, 3, 120, 17),
]


@pytest.fixture(scope="module")
def torch():
    import torch as t

    assert t.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_16637_gb300 import build

    build.build()
    return t


@pytest.mark.parametrize("norb,nel,nA,nB", CASES)
def test_sigma_at_range_and_block_edges(torch, norb, nel, nA, nB):
    from oracle import oracle as O
    from paper_2601_16637_gb300 import binding as B

    wl = W.make("rows", norb, nel, nel, nA, nB, 0.3, 1000 * norb + nA + nB)
    o = O.Oracle.from_workload(wl)
    x = W.random_vector(nA * nB, 3)
    ref = o.sigma(x)[0]
    o.close()
    with B.SBD.from_workload(wl) as g:
        xd = torch.from_numpy(x[0]).cuda()
        for prec, tol in (("fp64", SIGMA_FP64_RTOL), ("f32x2", SIGMA_FP64_RTOL), ("mixed", SIGMA_MIXED_RTOL)):
            got = g.sigma(xd.float() if prec == "mixed" else xd, prec)
            again = g.sigma(xd.float() if prec == "mixed" else xd, prec)
            assert torch.equal(got, again), prec
            assert rel_maxnorm(got.cpu().numpy(), ref) <= tol, prec
    # a second handle orders lists of equal length as it likes: the sums must not depend on it
    with B.SBD.from_workload(wl) as g:
        assert torch.equal(got, g.sigma(xd.float(), "mixed"))

