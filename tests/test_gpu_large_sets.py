"""Excitation tables of sets at the tile edges of the prefix sums (one CTA up to 16,384 strings, tiles of
8,192 above), and of sets whose windows of 32 strings mostly hold no excitation, against a count in numpy."""
import numpy as np
import pytest

from paper_2601_16637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16384, 16385, 24576, 24577])
def test_tables_at_scan_tile_edges(n):
    from paper_2601_16637_gb300 import binding as B

    wl = W.make("large", 30, 6, 6, n, 1, 0.05, n)
    with B.SBD.from_workload(wl) as g:
        s = g.sorted_strings(0)
        cnt = {1: np.zeros(n, dtype=np.int64), 2: np.zeros(n, dtype=np.int64)}
        for a in range(0, n, 1024):
            pc = np.bitwise_count(s[a:a + 1024, None] ^ s[None, :])
            for kind in (1, 2):
                cnt[kind][a:a + 1024] = (pc == 2 * kind).sum(1)
        for kind in (1, 2):
            ptr, tgt, _, _ = B.sbd_tables(g.handle, 0, kind)
            assert np.array_equal(ptr, np.concatenate([[0], np.cumsum(cnt[kind])])), kind
            i = np.repeat(np.arange(n), cnt[kind])
            assert np.all(np.bitwise_count(s[i] ^ s[tgt]) == 2 * kind)
            assert np.all((np.diff(tgt) > 0) | (np.diff(i) > 0))
