"""Rounding error of the FP32-pair product on short excitation lists.

Root mean square error over the product's root mean square, against the FP64 product (which has its
own tests against the oracle; the oracle's sums run one after the other, and their error of 1.5e-15
would hide what is measured here), for 300 x 300 strings at norb 24 and 350 x 600 at norb 26 (lists of
a few dozen entries).  The bound is what the pair product had when eight partial sums were kept per
list, 0.93e-15 and 1.04e-15, with the FP64 product's own error (about 0.4e-15) added in quadrature.
"""
import numpy as np
import pytest

from paper_2601_16637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norb,nel,nA,nB,bound", [(24, 8, 300, 300, 1.0e-15), (26, 9, 350, 600, 1.1e-15)])
def test_pair_product_error(norb, nel, nA, nB, bound):
    import torch

    from paper_2601_16637_gb300 import binding as B

    err = []
    for seed in range(4):
        wl = W.make("pair", norb, nel, nel, nA, nB, 0.35, 900 + seed)
        with B.SBD.from_workload(wl) as g:
            w = []
            for spin in (0, 1):
                s = g.sorted_strings(spin)
                tot = sum(p * ((s >> np.uint64(p)) & np.uint64(1)).astype(np.float64) for p in range(norb))
                w.append(np.exp(-0.06 * (tot - tot.min())))
            x = np.random.default_rng(seed).standard_normal((nA, nB)) * w[0][:, None] * w[1][None, :]
            x = (x / np.linalg.norm(x)).reshape(-1)
            xd = torch.from_numpy(x).cuda()
            got, ref = (g.sigma(xd, p).cpu().numpy() for p in ("f32x2", "fp64"))
        err.append(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    assert np.sqrt(np.mean(np.square(err))) <= bound, err
