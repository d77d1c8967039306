"""Products over several ranges of lists: both sides of one and two ranges with the table of sums in shared
memory (norb 43 is the last whose table takes no more than half of it) and in global memory (norb 44), orbital
pairs of the alpha-beta pass in up to eight parts, and the batched product against the single one where its
instances differ in all of these."""
import pytest

from gpu_common import SIGMA_FP64_RTOL, SIGMA_MIXED_RTOL, rel_maxnorm
from paper_2601_16637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# 1,808 lines of 128 bytes: 904 of them the table at norb 43; one of them zero at norb 44
@pytest.mark.parametrize("norb,nel,nA,nB", [(43, 4, 904, 17), (43, 4, 905, 17), (44, 4, 17, 1807), (44, 4, 17, 1808),
                                            (64, 4, 3, 20000), (64, 4, 2, 24500)])  # four and eight parts
def test_products_at_range_and_part_edges(norb, nel, nA, nB):
    import torch

    from oracle import oracle as O
    from paper_2601_16637_gb300 import binding as B

    wl = W.make("ranges", norb, nel, nel, nA, nB, 0.1, 7 * norb + nA + nB)
    o = O.Oracle.from_workload(wl)
    x = W.random_vector(nA * nB, 4)
    ref = o.sigma(x)[0]
    o.close()
    with B.SBD.from_workload(wl) as g:
        xd = torch.from_numpy(x[0]).cuda()
        for prec, tol in (("fp64", SIGMA_FP64_RTOL), ("f32x2", SIGMA_FP64_RTOL), ("mixed", SIGMA_MIXED_RTOL)):
            got = g.sigma(xd.float() if prec == "mixed" else xd, prec)
            assert rel_maxnorm(got.cpu().numpy(), ref) <= tol, prec


@pytest.mark.parametrize("shapes", [[(29, 10, 17, 2803), (58, 4, 33, 2500), (6, 2, 5, 7), (44, 4, 1808, 16)],
                                    [(64, 4, 3, 20000), (12, 4, 40, 30), (1, 1, 1, 1), (58, 4, 300, 250)]])
@pytest.mark.parametrize("prec", ["fp64", "f32x2", "mixed"])
def test_batched_product_over_ranges_and_parts_is_the_single_one(shapes, prec):
    import torch

    from paper_2601_16637_gb300 import binding as B

    gs, xs, single, many = [], [], [], []
    try:
        for k, (norb, nel, nA, nB) in enumerate(shapes):
            gs.append(B.SBD.from_workload(W.make("batch", norb, nel, nel, nA, nB, 0.1, 50 + k)))
            x = torch.from_numpy(W.random_vector(nA * nB, k)[0]).cuda()
            xs.append(x.float() if prec == "mixed" else x)
            many.append(torch.full((nA * nB,), float("nan"), dtype=torch.float64, device="cuda"))
        # the two-operand pass of every instance with as many rows per item as the batch has room for
        rows = 2 if max(s[3] for s in shapes) < 10000 else 1
        B.sbd_sigma_batched([g.handle for g in gs], xs, many, prec, rows)
        for g, x, m, s in zip(gs, xs, many, shapes):
            single = torch.full_like(m, float("nan"))
            if rows == 1 and prec != "mixed" and s[3] < 10000:  # the single product stages two rows here
                B.sbd_sigma_batched([g.handle], [x], [single], prec, 1)
            else:
                single = g.sigma(x, prec)
            assert torch.equal(single, m), s
    finally:
        for g in gs:
            g.close()
