"""What the performance of this library is measured on: its own calls over their real range.

Every case goes through the public Python entry points (paper_2601_16637_gb300.binding), as a
program that diagonalises selected spaces calls them:

  sigma    one or more products sigma = H c on a handle that the program keeps (FP64, FP32 pairs,
           mixed precision): the call a Davidson loop outside the library makes
  batched  the mixed products of several handles in one launch sequence
  create   the ingestion of one job: sort, validate, excitation tables, diagonal
  solve    a Davidson solve to convergence on a kept handle
  engine   jobs of uneven size submitted to the batched engine and run under an iteration cap

Sizes are those of workloads.py: the norb = 8 full space, the norb = 16 and norb = 29
configurations, the batched instances (norb 16-26, 500-5,000 strings) and the serving jobs
(norb 24-58, 300-20,000 strings).  Inputs follow the same recipe (one- and two-electron integrals,
Gumbel-top-k strings), drawn on the GPU from the seed alone.  Amplitudes are normal deviates that
decay with the excitation level of the determinant, as eigenvectors and Krylov vectors of this
problem do.

The mixed product has FP32 accuracy by definition (FP32 amplitudes and integrals); the program keeps
it, like its input vector, in FP32, and eigenvectors are kept in FP32 too.  Energies, FP64 and
FP32-pair products stay FP64.
"""
import math

import numpy as np
import torch

from paper_2601_16637_gb300 import binding as B

# ---------------------------------------------------------------------------------------------
# the cases


def listed():
    return [
        # the product of the 1.0e8-determinant single solve: the largest call of the benchmark
        dict(name="sigma-mixed-29o-10000", kind="sigma", norb=29, nel=10, nA=10000, nB=10000, lam=0.25,
             precision="mixed", nvec=1),
        # the product of a serving job with many orbitals: long integral tables, sparse lists
        dict(name="sigma-mixed-58o-5003", kind="sigma", norb=58, nel=19, nA=5003, nB=5003, lam=0.35,
             precision="mixed", nvec=1),
        # a mid-sized batched instance, odd and unequal sets
        dict(name="sigma-mixed-20o-1703x2381", kind="sigma", norb=20, nel=7, nA=1703, nB=2381, lam=0.35,
             precision="mixed", nvec=1),
        # the smallest serving jobs: launches and latency count
        dict(name="sigma-mixed-24o-300", kind="sigma", norb=24, nel=8, nA=300, nB=300, lam=0.35,
             precision="mixed", nvec=1),
        # the plain FP64 configuration with three roots: a block of three vectors
        dict(name="sigma-fp64-16o-2000-x3", kind="sigma", norb=16, nel=5, nA=2000, nB=2000, lam=0.35,
             precision="fp64", nvec=3),
        # the FP64 product of the norb = 29 workload (reference solves, checks of mixed results)
        dict(name="sigma-fp64-29o-4001x3607", kind="sigma", norb=29, nel=10, nA=4001, nB=3607, lam=0.25,
             precision="fp64", nvec=1),
        # the FP32-pair product: the defect-correction product of mixed solves
        dict(name="sigma-f32x2-29o-6000", kind="sigma", norb=29, nel=10, nA=6000, nB=6000, lam=0.25,
             precision="f32x2", nvec=1),
        # the products of several small instances in one launch sequence
        dict(name="batched-mixed-8", kind="batched", count=8, smin=500, smax=2500, lam=0.35),
        # ingestion of one large job
        dict(name="create-29o-10000x8009", kind="create", norb=29, nel=10, nA=10000, nB=8009, lam=0.25),
        # a full mixed-precision solve of one root of an instance of ordinary size
        dict(name="solve-mixed-24o-1201x1150", kind="solve", norb=24, nel=8, nA=1201, nB=1150, lam=0.35,
             precision="mixed", nroots=1, tol=1e-8, max_subspace=24),
        # the smallest solve, FP64, the tolerance of its configuration (with equal full sets the largest
        # component would come in pairs, and the sign of the vector would be open)
        dict(name="solve-fp64-8o-70x61", kind="solve", norb=8, nel=4, nA=70, nB=61, lam=0.0,
             precision="fp64", nroots=1, tol=1e-10, max_subspace=0),
        # jobs of uneven size in the engine; the iteration cap of a service with a latency target
        dict(name="engine-6", kind="engine", count=6, smin=500, smax=2500, lam=0.35, max_iter=24),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sigma", "sigma", "sigma", "sigma", "batched", "create", "solve", "engine"])
    if kind == "sigma":
        precision = rng.choice(["mixed", "mixed", "fp64", "f32x2"])
        norb = rng.choice([16, 20, 24, 26, 29, 32, 40, 48, 58])
        nel = min(int(round(norb / 3)), 10) if norb < 32 else int(round(norb / 3))
        top = {"mixed": 8000, "fp64": 2500, "f32x2": 5000}[precision]
        nmax = min(top, math.comb(norb, nel))
        nA, nB = _loguniform(rng, 300, nmax), _loguniform(rng, 300, nmax)
        return dict(kind=kind, norb=norb, nel=nel, nA=nA, nB=nB, lam=0.25 if norb == 29 else 0.35,
                    precision=precision, nvec=rng.choice([1, 1, 2, 3]) if nA * nB < 4e6 else 1)
    if kind == "batched":
        lo = rng.randint(300, 800)
        return dict(kind=kind, count=rng.randint(2, 10), smin=lo, smax=lo + rng.randint(100, 2000), lam=0.35)
    if kind == "create":
        norb = rng.choice([16, 20, 24, 29, 40, 48])
        nel = min(int(round(norb / 3)), 10) if norb < 32 else int(round(norb / 3))
        nmax = min(8000, math.comb(norb, nel))
        return dict(kind=kind, norb=norb, nel=nel, nA=_loguniform(rng, 300, nmax), nB=_loguniform(rng, 300, nmax),
                    lam=0.25 if norb == 29 else 0.35)
    if kind == "solve":
        precision = rng.choice(["mixed", "mixed", "fp64", "f32x2"])
        norb = rng.choice([16, 20, 24, 26])
        nmax = 500 if precision == "fp64" else 1000
        return dict(kind=kind, norb=norb, nel=int(round(norb / 3)), nA=_loguniform(rng, 150, nmax),
                    nB=_loguniform(rng, 150, nmax), lam=0.35, precision=precision, nroots=1, tol=1e-8,
                    max_subspace=rng.choice([0, 16, 24]))
    lo = rng.randint(300, 800)
    return dict(kind=kind, count=rng.randint(2, 6), smin=lo, smax=lo + rng.randint(100, 1200), lam=0.35,
                max_iter=rng.randint(16, 28))


# ---------------------------------------------------------------------------------------------
# inputs, from the seed alone (the recipe of workloads.py, drawn on the GPU)

_all = {}  # (norb, nel) -> every string of the full space, where it is enumerated


def _enumerate(norb, nel):
    if (norb, nel) not in _all:
        level = {0: torch.zeros(1, dtype=torch.int64, device="cuda")}
        for m in range(norb):
            nxt = {}
            for k in range(max(0, nel - (norb - m - 1)), min(nel, m + 1) + 1):
                parts = ([level[k]] if k in level else []) + ([level[k - 1] | (1 << m)] if k - 1 in level else [])
                nxt[k] = torch.cat(parts)
            level = nxt
        _all[(norb, nel)] = level[nel]
    return _all[(norb, nel)]


def _orbital_sum(s, norb):
    tot = torch.zeros(s.shape, dtype=torch.float64, device=s.device)
    for p in range(norb):
        tot += p * ((s >> p) & 1)
    return tot


def _strings(norb, nel, k, lam, gen):
    """k distinct strings in draw order, log-weight -lam * (sum of occupied indices), aufbau included."""
    total = math.comb(norb, nel)
    if k >= total:
        s = _enumerate(norb, nel)
        return s[torch.randperm(total, generator=gen, device="cuda")]
    if total <= 1 << 26:
        s = _enumerate(norb, nel)
        u = torch.rand(total, generator=gen, device="cuda", dtype=torch.float64).clamp_(1e-300, 1 - 1e-16)
        out = s[torch.topk(-lam * _orbital_sum(s, norb) - torch.log(-torch.log(u)), k).indices]
    else:
        out = torch.zeros(0, dtype=torch.int64, device="cuda")
        logw = -lam * torch.arange(norb, dtype=torch.float64, device="cuda")
        while out.numel() < k:
            u = torch.rand(2 * k, norb, generator=gen, device="cuda", dtype=torch.float64).clamp_(1e-300, 1 - 1e-16)
            occ = torch.topk(logw - torch.log(-torch.log(u)), nel, dim=1).indices
            out = torch.cat([out, (torch.ones_like(occ) << occ).sum(1)])
            uniq, inv = torch.unique(out, return_inverse=True)
            first = torch.full((uniq.numel(),), out.numel(), dtype=torch.int64, device="cuda")
            first.scatter_reduce_(0, inv, torch.arange(out.numel(), device="cuda"), "amin")
            out = out[torch.sort(first).values]
        out = out[:k].clone()
    aufbau = (1 << nel) - 1
    if not bool((out == aufbau).any()):
        out[-1] = aufbau
    return out


def _integrals(norb, gen):
    def normal(n):
        return torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)

    p = torch.arange(norb, device="cuda", dtype=torch.float64)
    h = torch.triu(normal((norb, norb)) * 0.05 * torch.exp(-(p[:, None] - p[None, :]).abs() / 4), 1)
    h = h + h.T + torch.diag(-2.0 + 0.15 * p)
    b = torch.triu(normal((2 * norb, norb, norb)) * 0.12)
    b = (b + torch.triu(b, 1).transpose(1, 2)).reshape(2 * norb, norb * norb)
    return h.contiguous(), (b.T @ b).reshape(norb, norb, norb, norb).contiguous()


def _instance(norb, nelA, nelB, nA, nB, lam, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    h, eri = _integrals(norb, gen)
    return dict(norb=norb, nelA=nelA, nelB=nelB, h=h, eri=eri, A=_strings(norb, nelA, nA, lam, gen),
                B=_strings(norb, nelB, nB, lam, gen), gen=gen)


def _amplitudes(inst, nvec, dtype):
    """Normalised vectors in sorted-string order that decay with the determinant's excitation level."""
    wa, wb = (torch.exp(-0.06 * (s - s.min())) for s in
              (_orbital_sum(torch.sort(inst[x]).values, inst["norb"]) for x in "AB"))
    out = torch.empty(nvec, wa.numel() * wb.numel(), dtype=dtype, device="cuda")
    for v in range(nvec):
        x = torch.randn(wa.numel(), wb.numel(), generator=inst["gen"], device="cuda")
        x = x * wa.float()[:, None] * wb.float()[None, :]
        x = x / torch.linalg.vector_norm(x)
        if dtype == torch.float64:  # digits below FP32 too
            x = x.double() * (1 + 1e-7 * torch.rand(x.shape, generator=inst["gen"], device="cuda",
                                                     dtype=torch.float64))
        out[v] = x.reshape(-1)
    return out


def _many(case, seed):
    """The uneven instances of a batched or engine case: norb and string counts as in the batched workload."""
    rng = np.random.default_rng([7, case["count"], case["smin"], case["smax"]])
    out = []
    for i in range(case["count"]):
        norb = int(rng.choice([16, 20, 24, 26]))
        nel = int(round(norb / 3))
        full = math.comb(norb, nel)
        nA, nB = (min(int(rng.integers(case["smin"], case["smax"] + 1)), full) for _ in "AB")
        out.append((norb, nel, nel, nA, nB, case["lam"], 1000 * seed + i))
    return out


def _one(case, seed):
    return _instance(case["norb"], case["nel"], case["nel"], case["nA"], case["nB"], case["lam"], seed)


def _handle(inst, **kw):
    return B.SBD(inst["norb"], inst["nelA"], inst["nelB"], inst["h"], inst["eri"], inst["A"], inst["B"], **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batched":
        g, c, out = [], [], []
        for spec in _many(case, seed):
            inst = _instance(*spec)
            g.append(_handle(inst))
            c.append(_amplitudes(inst, 1, torch.float32)[0])
            out.append(torch.empty(c[-1].numel(), dtype=torch.float64, device="cuda"))
        return dict(kind=kind, g=g, c=c, out=out)
    if kind == "engine":
        jobs = []
        for spec in _many(case, seed):
            i = _instance(*spec)
            jobs.append((i["norb"], i["nelA"], i["nelB"], i["h"].cpu().numpy(), i["eri"].cpu().numpy(),
                         i["A"].cpu().numpy().view(np.uint64), i["B"].cpu().numpy().view(np.uint64)))
        return dict(kind=kind, jobs=jobs, max_iter=case["max_iter"])
    inst = _one(case, seed)
    if kind == "create":
        return dict(kind=kind, inst=inst)
    if kind == "solve":
        return dict(kind=kind, g=_handle(inst, max_subspace=case["max_subspace"]), nroots=case["nroots"],
                    tol=case["tol"], precision=case["precision"])
    f32 = case["precision"] == "mixed"
    c = _amplitudes(inst, case["nvec"], torch.float32 if f32 else torch.float64)
    return dict(kind=kind, g=_handle(inst), c=c, precision=case["precision"],
                out=torch.empty(c.shape, dtype=torch.float64, device="cuda"))


def run(state):
    kind = state["kind"]
    if kind == "sigma":
        s = state["g"].sigma(state["c"], state["precision"], out=state["out"])
        return s.float() if state["precision"] == "mixed" else s
    if kind == "batched":
        B.sbd_sigma_batched([g.handle for g in state["g"]], state["c"], state["out"], "mixed")
        return [s.float() for s in state["out"]]
    if kind == "create":
        with _handle(state["inst"]) as g:
            out = dict(diagonal=g.diagonal())
            for spin in (0, 1):  # what has a size known beforehand; the lists' lengths vary with the strings
                out[f"strings{spin}"] = g.sorted_strings(spin).view(np.int64)
                out[f"elements{spin}"] = g.string_elements(spin, 0)
                out[f"entries{spin}"] = [B.sbd_table_size(g.handle, spin, kind) for kind in (1, 2)]
        return out
    if kind == "solve":
        r = state["g"].davidson(nroots=state["nroots"], tol=state["tol"], precision=state["precision"])
        return dict(energies=r.energies, vectors=r.vectors.float())
    ms = max(max(j[5].size, j[6].size) for j in state["jobs"])
    with B.Engine(max_slots=len(state["jobs"]), max_subspace=20, max_iter=state["max_iter"],
                  max_norb=max(j[0] for j in state["jobs"]), max_strings=ms, schedule="lockstep") as e:
        ids = [e.submit(*j, tol=1e-8, keep_vector=True) for j in state["jobs"]]
        e.run()
        energies, vectors = np.array([e.result(i)["energy"] for i in ids]), []
        for i, j in zip(ids, state["jobs"]):
            v = torch.empty(j[5].size * j[6].size, dtype=torch.float64, device="cuda")
            B.sbd_engine_vector(e.engine, i, v)
            vectors.append(v.float())
    return dict(energies=energies, vectors=vectors)


# ---------------------------------------------------------------------------------------------
# the same numbers in 64 bits from plain torch: string algebra, Slater-Condon elements, products


def _popcount(x):
    x = x - ((x >> 1) & 0x5555555555555555)
    x = (x & 0x3333333333333333) + ((x >> 2) & 0x3333333333333333)
    x = (x + (x >> 4)) & 0x0F0F0F0F0F0F0F0F
    return ((x * 0x0101010101010101) >> 56) & 0x7F


def _pairs(s, pc):
    """(i, j) with popcount(s_i ^ s_j) == pc, in ascending order."""
    out, step = [], max(1, (1 << 25) // s.numel())
    for a in range(0, s.numel(), step):
        ij = (_popcount(s[a:a + step, None] ^ s[None, :]) == pc).nonzero()
        ij[:, 0] += a
        out.append(ij)
    return torch.cat(out).T


def _lowest(x):
    return _popcount((x & -x) - 1)


def _between(ket, a, b):
    one = torch.ones_like(ket)
    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
    return 1 - 2 * (_popcount(ket & ((one << hi) - 1) & ~((one << (lo + 1)) - 1)) & 1)


def _occupation(s, norb):
    return torch.stack([((s >> p) & 1) for p in range(norb)], 1).double()


class _Spin:
    """Same-spin matrix elements of one sorted string set."""

    def __init__(self, s, norb, h, eri, doubles=True):
        self.n, self.occ = s.numel(), _occupation(s, norb)
        i, j = _pairs(s, 2)
        x = s[i] ^ s[j]
        p, q = _lowest(x & s[i]), _lowest(x & s[j])
        self.i, self.j, self.p, self.q = i, j, p, q
        self.sign = _between(s[j], p, q).double()
        d = torch.einsum("pqkk->pqk", eri) - torch.einsum("pkkq->pqk", eri)
        self.single = torch.empty_like(self.sign)
        for a in range(0, i.numel(), 1 << 20):
            w = slice(a, a + (1 << 20))
            self.single[w] = self.sign[w] * (h[p[w], q[w]] + (d[p[w], q[w]] * self.occ[j[w]]).sum(1))
        jk = torch.einsum("ppqq->pq", eri) - torch.einsum("pqqp->pq", eri)
        self.diag = self.occ @ torch.diagonal(h) + 0.5 * ((self.occ @ jk) * self.occ).sum(1)
        if not doubles:
            return
        i, j = _pairs(s, 4)
        x = s[i] ^ s[j]
        a, b = x & s[i], x & s[j]
        p1, q1 = _lowest(a), _lowest(b)
        p2, q2 = _lowest(a & (a - 1)), _lowest(b & (b - 1))
        one = torch.ones_like(q2)
        ph = _between(s[j], q2, p2) * _between(s[j] ^ (one << q2) ^ (one << p2), q1, p1)
        v = ph * (eri[p1, q1, p2, q2] - eri[p1, q2, p2, q1])
        self.h = torch.sparse_coo_tensor(torch.stack([torch.cat([i, self.i]), torch.cat([j, self.j])]),
                                         torch.cat([v, self.single]), (self.n, self.n)).coalesce().to_sparse_csr()


def _diagonal(sa, sb, eri):
    return sa.diag[:, None] + sb.diag[None, :] + sa.occ @ torch.einsum("ppqq->pq", eri) @ sb.occ.T


def _spins(inst, doubles=True):
    return [_Spin(torch.sort(inst[x]).values, inst["norb"], inst["h"], inst["eri"], doubles) for x in "AB"]


class _Sigma:
    """c -> H c in FP64.  Works on c transposed ([nB][nA]) so that the columns of one orbital pair are rows."""

    def __init__(self, inst):
        self.sa, self.sb = sa, sb = _spins(inst)
        norb, self.eri = inst["norb"], inst["eri"]
        self.hd = _diagonal(sa, sb, self.eri)
        jd = torch.einsum("pqkk->pqk", self.eri)
        self.groups = []
        code = torch.maximum(sb.p, sb.q) * norb + torch.minimum(sb.p, sb.q)
        order = torch.argsort(code, stable=True)
        at = [0] + torch.cumsum(torch.bincount(code, minlength=norb * norb), 0).tolist()
        eye = torch.arange(sa.n, device="cuda")
        for rs in range(norb * norb):
            if at[rs + 1] == at[rs]:
                continue
            e, (r, s) = order[at[rs]:at[rs + 1]], divmod(rs, norb)
            self.groups.append((sb.i[e], sb.j[e], sb.sign[e], r, s))
        # the alpha operators of one beta pair: singles with (pq|rs), the diagonal with sum_k (kk|rs)
        idx = torch.stack([torch.cat([sa.i, eye]), torch.cat([sa.j, eye])])
        tag = torch.sparse_coo_tensor(idx, torch.arange(1, idx.shape[1] + 1, device="cuda", dtype=torch.float64),
                                      (sa.n, sa.n)).coalesce()
        self.perm = tag.values().long() - 1
        csr = tag.to_sparse_csr()
        self.crow, self.col = csr.crow_indices(), csr.col_indices()
        self.jd = jd

    def __call__(self, c):
        sa, sb = self.sa, self.sb
        out = self.hd * c
        out += torch.mm(sa.h, c)
        ct = c.T.contiguous()
        ot = torch.mm(sb.h, ct)
        for i, j, t, r, s in self.groups:
            v = torch.cat([sa.sign * self.eri[sa.p, sa.q, r, s], sa.occ @ self.jd[r, s]])[self.perm]
            m = torch.sparse_csr_tensor(self.crow, self.col, v, (sa.n, sa.n))
            ot.index_add_(0, i, torch.mm(m, (ct[j] * t[:, None]).T).T.contiguous())
        out += ot.T
        del ot, ct
        # alpha singles with the beta diagonal
        for a in range(0, sa.i.numel(), 4096):
            w = slice(a, a + 4096)
            k = sa.sign[w, None] * (self.jd[sa.p[w], sa.q[w]] @ sb.occ.T)
            out.index_add_(0, sa.i[w], k * c[sa.j[w]])
        return out


def _exact_solve(inst, nroots):
    """The lowest eigenpairs by block Davidson with full orthogonalisation, to a residual of 1e-11."""
    H = _Sigma(inst)
    shape, n = H.hd.shape, H.hd.numel()
    hd = H.hd.reshape(-1)
    lowest = torch.topk(-hd, nroots).indices
    V = torch.zeros(n, nroots, dtype=torch.float64, device="cuda")
    V[lowest, torch.arange(nroots)] = 1.0
    W = torch.stack([H(V[:, k].reshape(shape)).reshape(-1) for k in range(nroots)], 1)
    u = e = None
    for _ in range(400):
        e, y = torch.linalg.eigh(V.T @ W)
        e, y = e[:nroots], y[:, :nroots]
        u, r = V @ y, W @ y - (V @ y) * e
        if float(torch.linalg.vector_norm(r, dim=0).max()) < 1e-11:
            break
        if V.shape[1] >= 60:
            k = torch.linalg.eigh(V.T @ W)[1][:, :20]
            V, W = V @ k, W @ k
        for j in range(nroots):
            d = hd - e[j]
            t = r[:, j] / torch.where(d.abs() < 1e-4, torch.full_like(d, 1e-4), d)
            for _ in range(2):
                t = t - V @ (V.T @ t)
                t = t / torch.linalg.vector_norm(t)
            V = torch.cat([V, t[:, None]], 1)
            W = torch.cat([W, H(t.reshape(shape)).reshape(-1, 1)], 1)
    big = u.abs().argmax(0)
    return e, u * torch.sign(u[big, torch.arange(nroots)])


def exact(case, seed):
    kind = case["kind"]
    if kind == "engine":
        return None  # capped iterations: the outputs are no eigenpairs
    if kind == "batched":
        out = []
        for spec in _many(case, seed):
            inst = _instance(*spec)
            c = _amplitudes(inst, 1, torch.float32)
            out.append(_Sigma(inst)(c[0].double().reshape(inst["A"].numel(), -1)).reshape(-1))
        return out
    inst = _one(case, seed)
    if kind == "create":
        sa, sb = _spins(inst, doubles=False)
        out = dict(diagonal=_diagonal(sa, sb, inst["eri"]).reshape(-1))
        for k, sp in enumerate((sa, sb)):
            out[f"elements{k}"] = sp.diag.cpu().numpy()
        return out
    if kind == "solve":
        if case["nA"] * case["nB"] > 2_000_000:
            return None  # minutes of plain torch
        e, u = _exact_solve(inst, case["nroots"])
        return dict(energies=e.cpu().numpy(), vectors=u.T.contiguous())
    c = _amplitudes(inst, case["nvec"], torch.float32 if case["precision"] == "mixed" else torch.float64)
    H = _Sigma(inst)
    out = torch.empty(c.shape, dtype=torch.float64, device="cuda")
    for v in range(c.shape[0]):
        out[v] = H(c[v].double().reshape(case["nA"], -1)).reshape(-1)
    return out


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without

_counts = {}


def _list_sizes(norb, nel, n, lam):
    """Singles and doubles inside one string set (of one seed; they hardly vary with it)."""
    key = (norb, nel, n, lam)
    if key not in _counts:
        s = _strings(norb, nel, n, lam, torch.Generator(device="cuda").manual_seed(1))
        c = [0, 0]
        step = max(1, (1 << 25) // n)
        for a in range(0, n, step):
            pc = _popcount(s[a:a + step, None] ^ s[None, :])
            c[0] += int((pc == 2).sum())
            c[1] += int((pc == 4).sum())
        _counts[key] = c
    return _counts[key]


def _sigma_work(norb, nel, nA, nB, lam, in_bytes):
    (sa, da), (sb, db) = _list_sizes(norb, nel, nA, lam), _list_sizes(norb, nel, nB, lam)
    # one multiply-add per connected determinant pair; each amplitude read and each product written once
    return (in_bytes + 8) * nA * nB, 2.0 * (nA * nB + nA * (sb + db) + nB * (sa + da) + sa * sb)


def work(case):
    kind = case["kind"]
    if kind in ("sigma", "solve"):
        b, f = _sigma_work(case["norb"], case["nel"], case["nA"], case["nB"], case["lam"],
                           4 if case["precision"] == "mixed" else 8)
        # a solve takes at least some dozens of products, whatever the method; each on a new vector
        m = 30 * case["nroots"] if kind == "solve" else case["nvec"]
        return {"bytes": m * b, "flops": m * f}
    if kind == "create":
        t = sum(sum(_list_sizes(case["norb"], case["nel"], n, case["lam"])) for n in (case["nA"], case["nB"]))
        # the diagonal, and per excitation a target and an FP64 element
        return {"bytes": 8.0 * case["nA"] * case["nB"] + 12.0 * t,
                "flops": float(case["nA"] * case["nB"] * case["nel"])}
    b = f = 0.0
    for norb, nel, _, nA, nB, lam, _ in _many(case, 0):
        bi, fi = _sigma_work(norb, nel, nA, nB, lam, 4)
        m = case["max_iter"] if kind == "engine" else 1
        b, f = b + m * bi, f + m * fi
    return {"bytes": b, "flops": f}
