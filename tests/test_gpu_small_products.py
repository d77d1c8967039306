"""Small products: the row passes' form for few strings (up to 768, one range of lists) and the beta pass
without transposes (up to 2^17 determinants), at both sides of either line, against the oracle, and bit
for bit against the batched product, which always transposes."""
import pytest

from gpu_common import SIGMA_FP64_RTOL, SIGMA_MIXED_RTOL, rel_maxnorm
from paper_2601_16637_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [
    (2, 1, 2, 2), (12, 4, 1, 7), (12, 4, 7, 1), (12, 4, 17, 33), (8, 4, 70, 61),
    (12, 4, 495, 264), (12, 4, 495, 265),                # 130,680 and 131,175 determinants
    (16, 5, 768, 31), (16, 5, 769, 31), (16, 5, 31, 768), (16, 5, 31, 769),
    (46, 5, 45, 70), (64, 3, 130, 129),                  # sums of integrals in global memory
]


@pytest.mark.parametrize("norb,nel,nA,nB", CASES)
def test_small_products(norb, nel, nA, nB):
    import torch

    from oracle import oracle as O
    from paper_2601_16637_gb300 import binding as B

    wl = W.make("small", norb, nel, nel, nA, nB, 0.2, 13 * norb + nA + nB)
    o = O.Oracle.from_workload(wl)
    x = W.random_vector(nA * nB, 9)
    ref = o.sigma(x)[0]
    o.close()
    with B.SBD.from_workload(wl) as g:
        xd = torch.from_numpy(x[0]).cuda()
        for prec, tol in (("fp64", SIGMA_FP64_RTOL), ("f32x2", SIGMA_FP64_RTOL), ("mixed", SIGMA_MIXED_RTOL)):
            xp = xd.float() if prec == "mixed" else xd
            got = g.sigma(xp, prec)
            assert rel_maxnorm(got.cpu().numpy(), ref) <= tol, prec
            many = torch.full_like(got, float("nan"))
            B.sbd_sigma_batched([g.handle], [xp], [many], prec)
            assert torch.equal(got, many), prec
