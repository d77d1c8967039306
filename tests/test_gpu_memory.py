"""Device memory that handles, block plans and engine jobs hold: instances that fit a byte budget keep fitting it."""
import numpy as np
import pytest

from paper_2601_16637_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2601_16637_gb300 import binding

    binding.load()
    return binding


def test_sparse_set_of_many_orbitals_holds_no_dense_tables(B):
    # no two of these strings are a single excitation apart: besides the integrals (8 bytes each, and 4 for
    # each two pairs of orbitals) and two vectors, only lists proportional to the strings
    rng = np.random.default_rng(1)
    norb, n, m = 64, 20000, 64
    h, eri, _ = _integrals(norb)

    def strings(k):
        occ = np.argsort(rng.random((k, norb)), axis=1)[:, :32].astype(np.uint64)
        return np.unique((np.uint64(1) << occ).sum(1, dtype=np.uint64))

    A, Bs = strings(n), strings(m)
    with B.SBD(norb, 32, 32, h, eri, A, Bs) as g:
        assert all(B.sbd_table_size(g.handle, s, 1) == 0 for s in (0, 1))
        npair = norb * (norb - 1) // 2
        assert g.memory() <= 8 * norb**4 + 4 * npair**2 + 16 * A.size * Bs.size + 400 * (A.size + Bs.size)


def _integrals(norb):
    rng = np.random.default_rng(3)
    b = rng.standard_normal((4, norb, norb)) * 0.1
    b = b + b.transpose(0, 2, 1)
    h = b[0] + np.diag(-2.0 + 0.1 * np.arange(norb))
    return h, np.einsum("kpq,krs->pqrs", b, b), rng


def test_handle_fits_the_budget_it_used_to(B):
    # 2,000 x 2,000 strings at norb 58: 2.68e8 bytes with lists padded per string, a third copy of
    # their values and FP32 integrals of all index quadruples
    wl = W.make("budget", 58, 19, 19, 2000, 2000, 0.35, 5)
    with B.SBD.from_workload(wl, hbm_budget_bytes=270_000_000) as g:
        assert g.memory() <= 270_000_000


def test_refused_allocation_of_a_block_plan_leaves_the_handle_as_it_was(B):
    import torch

    wl = W.make("plan", 14, 4, 4, 120, 90, 0.3, 8)
    state = {"left": None}

    def alloc(ctx, nbytes, stream):
        if state["left"] is not None:
            state["left"] -= 1
            if state["left"] < 0:
                return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0))

    def free(ctx, ptr, stream):
        torch.cuda.caching_allocator_delete(int(ptr))

    opts = B.sbd_default_options()
    fa, ff = B.ALLOC_FN(alloc), B.FREE_FN(free)
    opts.alloc, opts.free = fa, ff
    h = B.sbd_create(wl.norb, 4, 4, wl.h, wl.eri, wl.A, wl.B, opts, 0)
    try:
        nA, nB = B.sbd_dims(h)
        x = torch.from_numpy(W.random_vector(nA * nB, 2)[0]).cuda()
        ref, out = torch.empty_like(x), torch.empty_like(x)
        B.sbd_sigma(h, x, ref, 1, "fp64", 0)
        torch.cuda.synchronize()
        held, refused = B.sbd_memory(h), 0
        while True:
            state["left"] = refused
            try:
                plan = B.sbd_block_plan_create(h, 0, nA, 0, nA)
                break
            except B.SbdError as e:
                assert e.code == -5
                refused += 1
                state["left"] = None
                assert B.sbd_memory(h) == held
                B.sbd_sigma(h, x, out, 1, "fp64", 0)
                torch.cuda.synchronize()
                assert torch.equal(out, ref)
        state["left"] = None
        assert refused >= 10
        out.zero_()
        B.sbd_sigma_block(plan, x, out, "fp64", 0)
        torch.cuda.synchronize()
        assert float((out - ref).abs().max()) <= 1e-14 * float(ref.abs().max())
        B.sbd_block_plan_destroy(plan)
    finally:
        state["left"] = None
        B.sbd_destroy(h)
        torch.cuda.synchronize()


def test_block_plans_fit_the_budget_they_used_to(B):
    # 3,001 x 4,003 strings at norb 40, the two plans of one of two ranks: 4.96e8 bytes when the handle kept ordered
    # lists of both spins and no range lists
    wl = W.make("plans", 40, 13, 13, 3001, 4003, 0.35, 5)
    with B.SBD.from_workload(wl, hbm_budget_bytes=500_000_000) as g:
        plans = [B.sbd_block_plan_create(g.handle, 0, 1500, *j) for j in ((0, 1500), (1500, 3001))]
        assert g.memory() <= 496_000_000
        for p in plans:
            B.sbd_block_plan_destroy(p)


def test_engine_jobs_fit_the_budget_they_used_to(B):
    # two jobs of 1,500 x 2,000 strings at norb 58 held 1.225e9 bytes before the range lists
    wl = W.make("jobs", 58, 19, 19, 1500, 2000, 0.35, 5)
    with B.Engine(max_slots=2, max_subspace=6, max_iter=4, max_norb=58, max_strings=2000, rows_per_item=4,
                  hbm_budget_bytes=1_235_000_000) as e:
        for _ in range(2):
            e.submit(wl, tol=1e-8)
        e.step()
        st = e.stats()
        assert st["active"] == 2 and st["requeued"] == 0, st
