"""An amplitude that is no finite number reaches the outputs that are connected to it and no others.

The lists of the row passes and of the two-operand alpha-beta pass are padded; a padding entry must
not multiply an amplitude outside its list (0 x inf is a NaN).  Sparse random sets give lists that are
empty beside longer ones of their group; the amplitude sits at the first string of each staged range,
where padding pointed before, and at a string inside one.
"""
import numpy as np
import pytest

from paper_2601_16637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _level(strings, s):
    return np.array([bin(int(x) ^ int(s)).count("1") // 2 for x in strings])


# (norb, nel, nA, nB, lam): several ranges on the beta side, on the alpha side, integrals' sums in global memory
@pytest.mark.parametrize("norb,nel,nA,nB,lam", [(29, 10, 17, 2803, 0.02), (24, 6, 2500, 19, 0.05), (46, 6, 23, 1900, 0.02),
                                                (12, 4, 9, 150, 0.1)])
@pytest.mark.parametrize("prec", ["fp64", "mixed", "f32x2"])
def test_infinite_amplitude_reaches_only_connected_outputs(norb, nel, nA, nB, lam, prec):
    import torch

    from paper_2601_16637_gb300 import binding as B

    wl = W.make("inf", norb, nel, nel, nA, nB, lam, 31 * norb + nB)
    with B.SBD.from_workload(wl) as g:
        A, Bs = g.sorted_strings(0), g.sorted_strings(1)
        base = W.random_vector(nA * nB, 7)[0].reshape(nA, nB)
        n = max(nA, nB)
        marks = sorted({0, -(-n // 2), -(-n // 3), 2 * -(-n // 3), n // 5} & set(range(n)))
        for m in marks:
            ja, jb = (m, nB // 2) if nA > nB else (nA // 2, m)
            x = base.copy()
            x[ja, jb] = np.inf
            la, lb = _level(A, A[ja]), _level(Bs, Bs[jb])
            apart = la[:, None] + lb[None, :] > 2
            if prec == "mixed":  # the alpha-beta pass has one fixed-point scale per row: rows with a single to ja are NaN
                apart &= (la > 1)[:, None]
            xd = torch.from_numpy(x.reshape(-1)).cuda()
            got = g.sigma(xd.float() if prec == "mixed" else xd, prec).cpu().numpy().reshape(nA, nB)
            assert np.isfinite(got[apart]).all(), (m, int((~np.isfinite(got[apart])).sum()))
            assert not np.isfinite(got[ja, jb])
