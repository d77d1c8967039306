"""Two-operand alpha-beta pass (inside whole products) where its forms change, against the oracle: one, two
and four lanes to a list (pairs), a row of C that does not fit shared memory (FP64 and pairs from 28,129 columns
at norb 20), and the FP32 form, which runs where the column-stationary pass does not fit (from about 28,500
columns: staged; 57,000: not staged)."""
import pytest

from gpu_common import SIGMA_FP64_RTOL, SIGMA_MIXED_RTOL, rel_maxnorm
from paper_2601_16637_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [
    (24, 8, 40, 40, 0.35), (24, 8, 33, 150, 0.35), (24, 8, 21, 700, 0.35),  # skewed lists, few slices: 4, 4, 2 lanes
    (10, 4, 7, 210, 0.0), (12, 4, 5, 495, 0.0),                             # equal lists: 2 lanes, 1 lane
    (20, 7, 3, 28128, 0.1), (20, 7, 3, 28129, 0.1),                         # last staged, first unstaged row of FP64
    (20, 7, 3, 28700, 0.1), (20, 7, 2, 57000, 0.05),                        # FP32 form staged, not staged
]


@pytest.mark.parametrize("norb,nel,nA,nB,lam", CASES)
def test_products_where_the_alpha_beta_pass_changes_form(norb, nel, nA, nB, lam):
    import torch

    from oracle import oracle as O
    from paper_2601_16637_gb300 import binding as B

    wl = W.make("ab", norb, nel, nel, nA, nB, lam, 77 * norb + nB)
    o = O.Oracle.from_workload(wl)
    x = W.random_vector(nA * nB, 5)
    ref = o.sigma(x)[0]
    o.close()
    with B.SBD.from_workload(wl) as g:
        xd = torch.from_numpy(x[0]).cuda()
        for prec, tol in (("fp64", SIGMA_FP64_RTOL), ("f32x2", SIGMA_FP64_RTOL), ("mixed", SIGMA_MIXED_RTOL)):
            xp = xd.float() if prec == "mixed" else xd
            got = g.sigma(xp, prec)
            assert rel_maxnorm(got.cpu().numpy(), ref) <= tol, prec
            assert torch.equal(got, g.sigma(xp, prec)), prec
