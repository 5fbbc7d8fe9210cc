"""Which engine a plan's options select: the tuner's cases, explicit defaults, launch counts."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
import workloads as wl

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def sm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1710_10899_gb300 as pkg
    pkg.load_library()
    return pkg


@pytest.mark.parametrize("n,m", [(12, 2), (20, 8), (50, 24)])
def test_ring_rows_have_patterns_of_their_own(n, m):
    a = wl.ring_spd(n, m, seed=m)
    d = np.zeros((n, n))
    for j in range(n):
        d[j, a.colind[a.rowptr[j]:a.rowptr[j + 1]]] = a.vals[a.rowptr[j]:a.rowptr[j + 1]]
    assert (a.row_sizes() == m).all() and np.array_equal(d, d.T)
    rows = {tuple(a.colind[a.rowptr[j]:a.rowptr[j + 1]]) for j in range(n)}
    # (two entries a row: a row and its antipode have the same two)
    assert len(rows) == (n if m > 2 else n // 2)
    assert np.linalg.eigvalsh(d)[0] > 0.1


@pytest.mark.gpu
@pytest.mark.parametrize("m", [8, 32, 48])
@pytest.mark.parametrize("name", ["small", "sync", "tcgen05"])
def test_tuner_measures_the_engine_it_names(sm, name, m):
    """Every row runs alone through the coupled iteration on the tensor cores: p GEMMs of ten slice products per
    iteration and row (the Krylov engine executes none, rows that share a job execute them once)."""
    from paper_1710_10899_gb300 import tune
    if name == "small" and m > sm.SUBMAT_SMALL_MAX_M:
        return
    a = wl.ring_spd(304, m, seed=m)
    plan = sm.submat_plan(a.rowptr, a.colind, 2, precision="mixed", **tune.ENGINES[name])
    sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"), sync=True)
    rep = plan.report()
    assert rep["flops_tensor"] == pytest.approx(rep["iters_sum"] * 2 * 10 * 2 * m ** 3, rel=1e-12)
    assert rep["iters_sum"] >= a.n and plan.engine_launches() == 3


@pytest.mark.gpu
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("sign", [-1, 1])
def test_small_engine_takes_its_rows(sm, p, sign):
    """Orders 1..27 on the small-submatrix engine (a step limit other than the default keeps the coupled
    iteration), with the same bar as every mixed row."""
    a = wl.overlap_small()
    plan = sm.submat_plan(a.rowptr, a.colind, p, precision="mixed", root_sign=sign, small_max_m=32, k_max=41)
    y = sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"), sync=True).cpu().numpy()
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, p, sign=sign)
    err = [np.linalg.norm(y[s:e] - ref[s:e]) / np.linalg.norm(ref[s:e]) for s, e in zip(a.rowptr[:-1], a.rowptr[1:])]
    rep = plan.report()
    assert max(err) <= 1e-6 and rep["flops_tensor"] > 0 and rep["n_notspd"] == 0


@pytest.mark.gpu
@pytest.mark.parametrize("precision,tol", [("mixed", 1e-4), ("fp64", 1e-7)])
@pytest.mark.parametrize("p", [1, 2])
def test_a_default_given_explicitly_is_the_default(sm, precision, tol, p):
    """Every option that steers the coupled iteration, given with its default: the same launches and bits."""
    a = wl.overlap_small(n=400)
    v = torch.tensor(a.vals, device="cuda")
    plan = sm.submat_plan(a.rowptr, a.colind, p, precision=precision)
    ref = sm.submat_invroot(plan, v, sync=True).clone()
    for kw in (dict(k_max=40), dict(tol=tol), dict(refine_steps=2 if p == 1 else 0), dict(kappa_max=100.0),
               dict(small_max_m=plan.small_max_m), dict(sync_max_m=plan.sync_max_m)):
        other = sm.submat_plan(a.rowptr, a.colind, p, precision=precision, **kw)
        assert other.engine_launches() == plan.engine_launches(), kw
        assert torch.equal(sm.submat_invroot(other, v, sync=True), ref), kw
    steered = sm.submat_plan(a.rowptr, a.colind, p, precision=precision, k_max=41)
    assert not torch.equal(sm.submat_invroot(steered, v, sync=True), ref)


@pytest.mark.gpu
@pytest.mark.parametrize("twins,shared", [(1, False), (60, True)])
def test_groups_from_one_row_in_ten_on(sm, twins, shared):
    """Neighbouring rows of one pattern share a tcgen05 job only where enough rows do: the GEMMs are counted
    once a job, so without groups the executed flops are p 10 / (p + 1) of the method's."""
    r = wl.ring_spd(300, 200, seed=5)
    a = sp.csr_matrix((r.vals, r.colind, r.rowptr), shape=(r.n, r.n))
    twin = np.repeat(np.arange(r.n), np.where(np.arange(r.n) < twins, 2, 1))     # row i twice for i < twins
    a = a[twin][:, twin].tolil()
    for i in np.nonzero(twin[1:] == twin[:-1])[0]:
        a[i, i + 1] = a[i + 1, i] = 0.1
    a = (a + sp.diags(np.full(a.shape[0], 0.5))).tocsr()
    a.sort_indices()
    plan = sm.submat_plan(a.indptr.astype(np.int32), a.indices.astype(np.int32), 2)
    y = sm.submat_invroot(plan, torch.tensor(a.data, device="cuda"), sync=True).cpu().numpy()
    rep = plan.report()
    ratio = rep["flops_tensor"] / rep["flops_alg"] / (20.0 / 3.0)
    assert rep["n_fallback"] == 0 and (ratio < 0.95 if shared else abs(ratio - 1.0) < 1e-12)
    rows = list(range(0, a.shape[0], 37))
    ref = oracle.invroot(a.indptr, a.indices, a.data, 2, rows=rows)
    for j in rows:
        s = slice(a.indptr[j], a.indptr[j + 1])
        assert np.linalg.norm(y[s] - ref[s]) <= 1e-6 * np.linalg.norm(ref[s])
