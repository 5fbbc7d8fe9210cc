"""The Krylov engine (one column of the root by Lanczos) against the oracle and against the
coupled iteration, at the edges of its size classes, and the rows it has to leave to others.

Bars.  FP64: p kappa m eps = 3 * 9 * 250 * 2.2e-16 < 2e-12.  Double-float: products carry an
error near 2^-45 of a row's norm, so m kappa 2^-45 = 192 * 9 * 2.8e-14 < 1e-10.
"""
import numpy as np
import pytest
import scipy.linalg as sl

import oracle
import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one below, at and above each class edge, and the orders around a 32-entry block edge
ORDERS = [1, 2, 5, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 160, 191, 192, 193, 225, 250]


@pytest.fixture(scope="module")
def sm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1710_10899_gb300 as pkg
    pkg.load_library()
    return pkg


def blocks(orders, seed):
    rng = np.random.default_rng(seed)
    mats = []
    for n in orders:
        q = rng.standard_normal((n, n))
        mats.append(q @ q.T / n + 0.5 * np.eye(n))
    return wl.dense_to_csr(sl.block_diag(*mats),
                           keep=sl.block_diag(*[np.ones((n, n), bool) for n in orders]))


def row_err(a, y, ref, rows):
    return max(float(np.linalg.norm(y[a.rowptr[j]:a.rowptr[j + 1]] - ref[a.rowptr[j]:a.rowptr[j + 1]]) /
                     np.linalg.norm(ref[a.rowptr[j]:a.rowptr[j + 1]])) for j in rows)


def forward(sm, a, p, **kw):
    plan = sm.submat_plan(a.rowptr, a.colind, p, **kw)
    y = sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"), sync=True)
    return y.cpu().numpy(), plan.report()


@pytest.mark.parametrize("p,sign", [(1, -1), (2, -1), (3, -1), (1, 1), (2, 1), (3, 1), (7, -1)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_orders(sm, precision, p, sign):
    orders = ORDERS if precision == "fp64" else [n for n in ORDERS if n <= 192]
    a = blocks(orders, seed=p)
    rows = sorted({int(r) for s, n in zip(np.cumsum([0] + orders), orders)
                   for r in (s, s + n // 2, s + n - 1)})
    y, rep = forward(sm, a, p, precision=precision, root_sign=sign)
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, p, rows=rows, sign=sign)
    # the mixed path's largest order on this engine falls with p (the slices' exponent bias);
    # the tcgen05 engine's rows keep its own bar
    top = 250 if precision == "fp64" else {1: 192, 2: 192, 3: 144}.get(p, 1)
    m = a.row_sizes()
    bar = 2e-12 if precision == "fp64" else 1e-10
    assert row_err(a, y, ref, [j for j in rows if m[j] <= top]) <= bar
    assert row_err(a, y, ref, rows) <= (bar if precision == "fp64" else 1e-6)
    assert rep["n_notspd"] == 0 and rep["n_fallback"] == 0 and rep["n_rows"] == a.n
    # an explicit step limit keeps the coupled iteration: the two paths agree
    z, _ = forward(sm, a, p, precision=precision, root_sign=sign, k_max=39)
    assert row_err(a, z, y, range(a.n)) <= (1e-10 if precision == "fp64" else 1e-6)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("p,sign", [(2, -1), (1, 1)])
def test_indefinite_part_out_of_reach(sm, precision, p, sign):
    """A negative eigenvalue in a part of the submatrix that e_pos is not coupled to (stored
    zeros) is found all the same: every row of that pattern is refused."""
    n = 40
    dense = np.eye(n) * 2.0 + np.diag(np.full(n - 1, 0.3), 1) + np.diag(np.full(n - 1, 0.3), -1)
    dense[25, 25] = -1.0
    dense[25, :25] = dense[:25, 25] = dense[25, 26:] = dense[26:, 25] = 0.0
    dense[24, 26] = dense[26, 24] = 0.0
    a = wl.dense_to_csr(dense, keep=np.ones((n, n), bool))
    plan = sm.submat_plan(a.rowptr, a.colind, p, precision=precision, root_sign=sign)
    out = torch.zeros(a.nnz, dtype=torch.float64, device="cuda")
    with pytest.raises(sm.SubmatError) as ei:
        sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"), out, sync=True)
    assert ei.value.name == "SUBMAT_ENOTSPD"
    assert torch.isnan(out).all()


@pytest.mark.parametrize("kappa", [300.0, 1e5])
def test_wide_spectra(sm, kappa):
    """Condition numbers of the wide quadrature rule (300) and beyond the engine's limit (1e5,
    left to the coupled iteration).  The submatrix is well scaled, so FP64 keeps
    m kappa eps = 60 * 1e5 * 2.2e-16 < 2e-9 of the column."""
    rng = np.random.default_rng(3)
    q, _ = np.linalg.qr(rng.standard_normal((60, 60)))
    s = (q * np.geomspace(1.0 / kappa, 1.0, 60)) @ q.T
    a = wl.dense_to_csr(0.5 * (s + s.T), keep=np.ones((60, 60), bool))
    y, rep = forward(sm, a, 2, precision="fp64")
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, 2)
    assert row_err(a, y, ref, range(a.n)) <= (1e-11 if kappa < 1e3 else 2e-9)
    assert rep["n_notspd"] == 0


def test_extreme_scales(sm):
    """Powers of two on the values scale the result exactly: the engine works on the
    submatrix over its largest diagonal entry."""
    a = blocks([20, 70, 150], seed=9)
    y, _ = forward(sm, a, 2, precision="fp64")
    for e in (-200, 200):
        b = wl.CSR(a.n, a.rowptr, a.colind, a.vals * 2.0 ** e)
        z, rep = forward(sm, b, 2, precision="fp64")
        np.testing.assert_allclose(z * 2.0 ** (e // 2), y, rtol=1e-15)
        assert rep["n_fallback"] == 0


@pytest.mark.parametrize("p,sign", [(1, -1), (2, -1), (3, -1), (1, 1), (2, 1), (3, 1)])
@pytest.mark.parametrize("deterministic", [False, True])
def test_adjoint_orders(sm, p, sign, deterministic):
    """The Krylov adjoint at the class edges, with a zero cotangent on one block, against the
    oracle gradient (bar as for the Jacobi adjoint)."""
    orders = [1, 2, 31, 32, 33, 64, 65, 97, 129, 193, 250]
    a = blocks(orders, seed=20 + p)
    w = wl.random_on_pattern(a, seed=5)
    lo = sum(n * n for n in orders[:4])
    w[lo:lo + 33 * 33] = 0.0
    plan = sm.submat_plan(a.rowptr, a.colind, p, root_sign=sign, grad_deterministic=deterministic)
    sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"))
    g = sm.submat_invroot_backward(plan, torch.tensor(w, device="cuda")).cpu().numpy()
    gref = oracle.grad(a.rowptr, a.colind, a.vals, p, w, sign=sign)
    assert np.linalg.norm(g - gref) / np.linalg.norm(gref) <= 1e-10
    assert np.abs(g - gref).max() <= 1e-10 * np.abs(gref).max()
    assert np.all(g[lo:lo + 33 * 33] == 0.0)


@pytest.mark.parametrize("kappa,bar", [(300.0, 1e-10), (1e5, 1e-5)])
def test_adjoint_wide_spectra(sm, kappa, bar):
    """A spectrum of the wide quadrature rule (two passes over the entries) and one beyond the
    engine (the Jacobi kernel).  f' ~ x^(-3/2) spans kappa^(3/2), so double-floats (2^-45)
    keep 300^1.5 * 60 * 2.8e-14 < 1e-8 of the smallest and 1e-10 of the largest part; at 1e5
    the divided differences themselves keep 1e-5."""
    rng = np.random.default_rng(3)
    q, _ = np.linalg.qr(rng.standard_normal((60, 60)))
    s = (q * np.geomspace(1.0 / kappa, 1.0, 60)) @ q.T
    a = wl.dense_to_csr(0.5 * (s + s.T), keep=np.ones((60, 60), bool))
    w = wl.random_on_pattern(a, seed=6)
    gref = oracle.grad(a.rowptr, a.colind, a.vals, 2, w)
    for det in (False, True):
        plan = sm.submat_plan(a.rowptr, a.colind, 2, precision="fp64", grad_deterministic=det)
        sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"))
        g = sm.submat_invroot_backward(plan, torch.tensor(w, device="cuda")).cpu().numpy()
        assert np.abs(g - gref).max() <= bar * np.abs(gref).max()


def test_first_backward_under_capture(sm):
    """The first backward of a plan inside a stream capture, where the Krylov adjoint's storage
    cannot be allocated: the Jacobi kernel takes every row, and the replay gives the gradient."""
    a = blocks([20, 50], seed=11)
    w = wl.random_on_pattern(a, seed=7)
    plan = sm.submat_plan(a.rowptr, a.colind, 2, use_graph=False)
    v, wd = torch.tensor(a.vals, device="cuda"), torch.tensor(w, device="cuda")
    out, grad = torch.empty_like(v), torch.empty_like(v)
    sm.submat_invroot(plan, v, out, sync=True)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sm.submat_invroot(plan, v, out)
        sm.submat_invroot_backward(plan, wd, grad)
    grad.zero_()
    graph.replay()
    torch.cuda.synchronize()
    gref = oracle.grad(a.rowptr, a.colind, a.vals, 2, w)
    assert np.abs(grad.cpu().numpy() - gref).max() <= 1e-10 * np.abs(gref).max()


@pytest.mark.parametrize("p,sign", [(1, -1), (2, -1), (3, -1), (2, 1), (3, 1)])
def test_rows_of_one_pattern(sm, p, sign):
    """Rows that share their submatrix run as one job of the tcgen05 engine: blocks of orders
    200..250 (every row of a block shares its pattern, so full jobs and a remainder), the mixed
    bar on every row, and the same rows one by one (mma.sync engine) within the two bars."""
    orders = [200, 224, 230, 250]
    a = blocks(orders, seed=30 + p)
    y, rep = forward(sm, a, p, precision="mixed", root_sign=sign)
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, p, sign=sign)
    assert row_err(a, y, ref, range(a.n)) <= 1e-6
    assert rep["n_fallback"] == 0 and rep["n_rows"] == a.n and rep["iters_sum"] >= a.n
    z, _ = forward(sm, a, p, precision="mixed_sync", root_sign=sign)
    assert row_err(a, y, z, range(a.n)) <= 2e-6


def test_rows_of_one_pattern_time_out_together(sm):
    """A pipeline wait that gives up leaves every row of its job NaN."""
    a = blocks([200, 210], seed=41)
    v = torch.tensor(a.vals, device="cuda")
    plan = sm.submat_plan(a.rowptr, a.colind, 2)
    ref = sm.submat_invroot(plan, v, sync=True).clone()
    plan.test_stall(True)
    out = torch.zeros_like(v)
    with pytest.raises(sm.SubmatError) as ei:
        sm.submat_invroot(plan, v, out, sync=True)
    assert ei.value.name == "SUBMAT_ETIMEOUT"
    assert torch.isnan(out).all()
    plan.test_stall(False)
    assert torch.equal(sm.submat_invroot(plan, v, out, sync=True), ref)


def test_rows_of_one_pattern_not_spd(sm):
    """A group whose submatrix is not positive definite: every member refused, others kept."""
    a = blocks([200, 210], seed=42)
    vals = a.vals.copy()
    r = 200 + 17
    d = a.rowptr[r] + int(np.nonzero(a.colind[a.rowptr[r]:a.rowptr[r + 1]] == r)[0][0])
    vals[d] = -5.0
    plan = sm.submat_plan(a.rowptr, a.colind, 2)
    out = torch.zeros(a.nnz, dtype=torch.float64, device="cuda")
    with pytest.raises(sm.SubmatError) as ei:
        sm.submat_invroot(plan, torch.tensor(vals, device="cuda"), out, sync=True)
    assert ei.value.name == "SUBMAT_ENOTSPD"
    y = out.cpu().numpy()
    assert np.isnan(y[200 * 200:]).all() and np.isfinite(y[:200 * 200]).all()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_many_short_rows(sm, precision):
    """More rows of order <= 32 than two waves (one warp per row in both roles), every fifth row
    and the gradient against the oracle, same bits twice."""
    a = wl.overlap_small(n=3000)
    assert (a.row_sizes() <= 32).all()
    plan = sm.submat_plan(a.rowptr, a.colind, 2, precision=precision)
    v = torch.tensor(a.vals, device="cuda")
    y = sm.submat_invroot(plan, v, sync=True)
    assert torch.equal(y, sm.submat_invroot(plan, v))
    rows = list(range(0, a.n, 5))
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, 2, rows=rows)
    # m kappa eps = 32 * 250 * 2.2e-16 and, in double-float, 32 * 250 * 2^-45
    assert row_err(a, y.cpu().numpy(), ref, rows) <= (2e-12 if precision == "fp64" else 3e-10)
    w = wl.random_on_pattern(a, seed=8)
    g = sm.submat_invroot_backward(plan, torch.tensor(w, device="cuda")).cpu().numpy()
    gref = oracle.grad(a.rowptr, a.colind, a.vals, 2, w)
    assert np.abs(g - gref).max() <= 1e-10 * np.abs(gref).max()


def test_long_row_forward_and_adjoint(sm):
    """A row of 700 entries (partial sums and most blocks in global scratch) among short ones:
    FP64 forward against the oracle (m kappa eps = 700 * 4 * 2.2e-16 < 2e-12) and the gradient."""
    n = 700
    rng = np.random.default_rng(12)
    dense = np.eye(n) * 2.0
    off = 0.15 * rng.uniform(0.5, 1.0, n - 1)
    dense += np.diag(off, 1) + np.diag(off, -1)
    dense[0, 1:] = dense[1:, 0] = 0.02 * rng.uniform(0.5, 1.0, n - 1)
    a = wl.dense_to_csr(dense)
    y, rep = forward(sm, a, 2, precision="fp64")
    rows = [0, 1, 2, 350, n - 1]
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, 2, rows=rows)
    assert row_err(a, y, ref, rows) <= 2e-12 and rep["n_fallback"] == 0
    w = wl.random_on_pattern(a, seed=13)
    for det in (False, True):
        plan = sm.submat_plan(a.rowptr, a.colind, 2, precision="fp64", grad_deterministic=det)
        sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"))
        g = sm.submat_invroot_backward(plan, torch.tensor(w, device="cuda")).cpu().numpy()
        gref = oracle.grad(a.rowptr, a.colind, a.vals, 2, w)
        assert np.linalg.norm(g - gref) / np.linalg.norm(gref) <= 1e-10
        assert np.abs(g - gref).max() <= 1e-10 * np.abs(gref).max()


@pytest.mark.parametrize("precision", ["fp64", "mixed_sync"])
def test_other_precisions_ignore_the_stall_flag(sm, precision):
    """Only the tcgen05 engine reads the flag: the other precisions write every row, with the same bits."""
    a = wl.overlap_small(n=300)
    v = torch.tensor(a.vals, device="cuda")
    plan = sm.submat_plan(a.rowptr, a.colind, 2, precision=precision)
    ref = sm.submat_invroot(plan, v, sync=True).clone()
    plan.test_stall(True)
    out = torch.full_like(v, 7.0)
    assert torch.equal(sm.submat_invroot(plan, v, out, sync=True), ref)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("p,sign", [(2, -1), (1, -1), (1, 1)])
@pytest.mark.parametrize("bad", [np.nan, -np.inf])
def test_non_finite_value_below_the_diagonal(sm, precision, p, sign, bad):
    """A non-finite value stored at (r, c), r > c, only: the rows whose submatrix holds it are NaN and reported,
    the others keep their bits."""
    a = blocks([20, 40, 70], seed=51)
    r, c = 20 + 33, 20 + 5
    e = a.rowptr[r] + int(np.nonzero(a.colind[a.rowptr[r]:a.rowptr[r + 1]] == c)[0][0])
    vals = a.vals.copy()
    vals[e] = bad
    plan = sm.submat_plan(a.rowptr, a.colind, p, precision=precision, root_sign=sign)
    ref = sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"), sync=True).cpu().numpy()
    out = torch.zeros(a.nnz, dtype=torch.float64, device="cuda")
    with pytest.raises(sm.SubmatError) as ei:
        sm.submat_invroot(plan, torch.tensor(vals, device="cuda"), out, sync=True)
    assert ei.value.name == "SUBMAT_ENOTSPD" and plan.report()["n_notspd"] == 40
    y = out.cpu().numpy()
    hit = np.zeros(a.nnz, bool)
    hit[a.rowptr[20]:a.rowptr[60]] = True
    assert np.isnan(y[hit]).all() and np.array_equal(y[~hit], ref[~hit])


@pytest.mark.parametrize("p,sign", [(2, -1), (3, -1), (2, 1)])
def test_group_not_converged_in_other_columns(sm, p, sign):
    """A diagonal submatrix of order 200 (full pattern) after one step only: the first row of each job of 13
    has a value that the step and the Taylor finish bring to the limit, the others the smallest one, which
    they do not.  Every row is right to the residual threshold 1e-3: those that are not converged take the fallback."""
    n = 200
    d = np.full(n, 0.02)
    d[::13] = np.linspace(0.2, 1.0, len(d[::13]))
    a = wl.dense_to_csr(np.diag(d), keep=np.ones((n, n), bool))
    y, rep = forward(sm, a, p, precision="mixed", root_sign=sign, k_max=1)
    got = y.reshape(n, n)
    ref = np.diag(d ** (sign / p))
    assert (np.linalg.norm(got - ref, axis=1) <= 2e-3 * np.diag(ref)).all()
    assert rep["n_fallback"] >= n - len(d[::13])


def test_inverse_column_residual_is_measured(sm):
    """p = 1 in FP64: the residual that resid_tol is compared with is that of the column itself, rounding included
    (about |y| eps; the recurrence alone always stops below 2e-16).  At resid_tol = 2e-16 rows of order 70 fail it
    and end in the fallback; at the default nothing does, and the report holds the residual of the rows written."""
    a = blocks([70], seed=61)
    y, rep = forward(sm, a, 1, precision="fp64")
    s = a.vals.reshape(70, 70).astype(np.longdouble)
    r = np.linalg.norm((np.eye(70) - y.reshape(70, 70).astype(np.longdouble) @ s).astype(float), axis=1).max()
    assert rep["n_fallback"] == 0 and 2e-16 < r < 1e-13 and r / 4 <= rep["max_resid"] <= 4 * r
    z, rep = forward(sm, a, 1, precision="fp64", resid_tol=2e-16)
    assert rep["n_fallback"] >= 1
    assert row_err(a, z, y, range(a.n)) <= 2e-12


@pytest.mark.parametrize("p,sign", [(1, -1), (2, -1), (2, 1)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_refused_rows_of_every_engine(sm, precision, p, sign):
    """Rows beyond the engine's condition limit (one eigenvalue 1/5000, the others 0.1 to 1) at orders around the
    small engine's: they come out of the coupled iteration or the fallback, short ones of the mixed mode out of
    the small engine (whose products are counted), and the accepted rows beside them keep their bits.
    Bars: the mixed one, and p m kappa eps = 2 * 64 * 2e4 * 2.2e-16 < 1e-9 in FP64."""
    rng = np.random.default_rng(71)
    orders, mats = [3, 31, 32, 33, 64], []
    for n in orders:
        q, _ = np.linalg.qr(rng.standard_normal((n, n)))
        s = (q * np.r_[1.0 / 5000.0, np.linspace(0.1, 1.0, n - 1)]) @ q.T
        mats += [0.5 * (s + s.T), np.eye(n) + 0.1 / n]
    a = wl.dense_to_csr(sl.block_diag(*mats), keep=sl.block_diag(*[np.ones(x.shape, bool) for x in mats]))
    ok = wl.dense_to_csr(sl.block_diag(*mats[1::2]), keep=sl.block_diag(*[np.ones(x.shape, bool) for x in mats[1::2]]))
    y, rep = forward(sm, a, p, precision=precision, root_sign=sign)
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, p, sign=sign)
    assert row_err(a, y, ref, range(a.n)) <= (1e-9 if precision == "fp64" else 1e-6)
    assert rep["n_notspd"] == 0 and (rep["flops_tensor"] > 0) == (precision == "mixed")
    z, _ = forward(sm, ok, p, precision=precision, root_sign=sign)
    good, at = [], 0
    for i, n in enumerate([n for n in orders for _ in range(2)]):
        if i % 2:
            good += range(a.rowptr[at], a.rowptr[at + n])
        at += n
    assert np.array_equal(y[good], z)


def low_block(n, kappa, rng):
    """One eigenvalue 1, the others 1/kappa to 2/kappa: the condition estimate sees it whole."""
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    s = (q * np.r_[np.linspace(1.0 / kappa, 2.0 / kappa, n - 1), 1.0]) @ q.T
    return 0.5 * (s + s.T)


@pytest.mark.parametrize("n", [30, 60, 120, 150])
@pytest.mark.parametrize("p,sign", [(2, -1), (3, -1), (2, 1)])
def test_wide_rows_of_the_mixed_mode_are_fp64(sm, n, p, sign):
    """Rows whose condition estimate exceeds kappa_max = 100: FP64 arithmetic (counted), m kappa eps of the
    column with kappa = 300; a narrow block beside them stays in double-float."""
    rng = np.random.default_rng(81)
    wide, narrow = low_block(n, 300.0, rng), np.eye(n) + 0.2 / n
    a = wl.dense_to_csr(sl.block_diag(wide, narrow), keep=sl.block_diag(np.ones((n, n), bool), np.ones((n, n), bool)))
    y, rep = forward(sm, a, p, precision="mixed", root_sign=sign)
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, p, sign=sign)
    assert row_err(a, y, ref, range(n)) <= n * 300 * 2.2e-16
    assert row_err(a, y, ref, range(n, 2 * n)) <= 1e-10
    assert rep["n_fallback"] == 0 and rep["n_notspd"] == 0
    # two flops a product, n^2 products a step, at least two steps a row, and not the narrow block's
    assert 2 * 2 * n ** 3 <= rep["flops_fp64"] <= 2 * 64 * n ** 3


@pytest.mark.parametrize("n", [30, 60, 120, 150, 200])
@pytest.mark.parametrize("p,sign", [(2, -1), (3, -1), (2, 1)])
def test_adjoint_of_wide_rows_is_fp64(sm, n, p, sign):
    """The gradient at kappa = 600 (two passes of the wide rule) to m kappa eps, as the Jacobi adjoint
    gave it (double-float: kappa 2^-45 times some tens)."""
    rng = np.random.default_rng(82)
    a = wl.dense_to_csr(low_block(n, 600.0, rng), keep=np.ones((n, n), bool))
    w = wl.random_on_pattern(a, seed=5)
    gref = oracle.grad(a.rowptr, a.colind, a.vals, p, w, sign=sign)
    for det in (False, True):
        plan = sm.submat_plan(a.rowptr, a.colind, p, root_sign=sign, grad_deterministic=det)
        sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"))
        g = sm.submat_invroot_backward(plan, torch.tensor(w, device="cuda")).cpu().numpy()
        assert np.abs(g - gref).max() <= n * 600 * 2.2e-16 * np.abs(gref).max()


def test_executed_work_is_counted(sm):
    """Products of the double-float rows: m^2 a step in the forward (two steps at least, 64 at most here), the same
    for an adjoint in one launch and in waves of a few rows; FP64 rows are counted as FP64 flops."""
    a = blocks([40, 150], seed=91)
    v, w = torch.tensor(a.vals, device="cuda"), torch.ones(a.nnz, dtype=torch.float64, device="cuda")
    m3 = float((a.row_sizes().astype(np.float64) ** 2).sum())
    done = []
    for kw in (dict(), dict(grad_deterministic=True, grad_wave_mib=1)):
        plan = sm.submat_plan(a.rowptr, a.colind, 2, **kw)
        sm.submat_invroot(plan, v, sync=True)
        assert 2 * m3 <= plan.work()["fwd_products_df"] <= 64 * m3 and plan.report()["flops_fp64"] == 0
        sm.submat_invroot_backward(plan, w)
        done.append(plan.work())
    assert done[0] == done[1] and done[0]["bwd_products_df"] >= 4 * m3 and done[0]["bwd_flops_fp64"] == 0


def test_mixed_inverse_is_refined_to_fp64(sm):
    """The mixed mode's inverse at every class and block edge to FP64 accuracy, m kappa eps with kappa = 9
    (its double-float recurrence alone stops at 1e-11)."""
    a = blocks(ORDERS, seed=101)
    y, rep = forward(sm, a, 1, precision="mixed")
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, 1)
    m = a.row_sizes()
    for n in ORDERS:
        assert row_err(a, y, ref, np.nonzero(m == n)[0]) <= max(n, 2) * 9 * 2.2e-16, n
    assert rep["n_fallback"] == 0 and rep["flops_tensor"] == 0
    z, _ = forward(sm, a, 1, precision="mixed", root_sign=1)          # A itself, once it is found definite
    assert np.array_equal(z, a.vals)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_inverse_of_long_rows(sm, precision):
    """The same in both modes for a row of 700 entries (four elements a thread, partial sums and most blocks in
    scratch; not a multiple of the block or of the threads) among short ones, kappa < 4."""
    n = 700
    rng = np.random.default_rng(102)
    off = 0.15 * rng.uniform(0.5, 1.0, n - 1)
    dense = np.eye(n) * 2.0 + np.diag(off, 1) + np.diag(off, -1)
    dense[0, 1:] = dense[1:, 0] = 0.02 * rng.uniform(0.5, 1.0, n - 1)
    a = wl.dense_to_csr(dense)
    y, rep = forward(sm, a, 1, precision=precision)
    rows = [0, 1, 2, 350, n - 1]
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, 1, rows=rows)
    assert row_err(a, y, ref, rows) <= n * 4 * 2.2e-16
    assert rep["n_fallback"] == 0 and rep["flops_tensor"] == 0 and rep["max_resid"] < 1e-9
    z, _ = forward(sm, a, 1, precision=precision, root_sign=1)
    assert np.array_equal(z, a.vals)


@pytest.mark.parametrize("deterministic", [False, True])
def test_captured_backward_after_an_eager_one(sm, deterministic):
    """A backward captured once the storage is there: the Krylov runs fork to the plan's streams and join again,
    rows repeated in FP64 included; the replay on other values of the cotangent gives its gradient."""
    a = blocks([20, 50, 150], seed=111)
    vals = a.vals.copy()
    vals[20 * 20:20 * 20 + 2500] = low_block(50, 300.0, np.random.default_rng(112)).ravel()
    w = wl.random_on_pattern(a, seed=7)
    plan = sm.submat_plan(a.rowptr, a.colind, 2, use_graph=False, grad_deterministic=deterministic)
    v, wd = torch.tensor(vals, device="cuda"), torch.ones(a.nnz, dtype=torch.float64, device="cuda")
    out, grad = torch.empty_like(v), torch.empty_like(v)
    sm.submat_invroot(plan, v, out, sync=True)
    sm.submat_invroot_backward(plan, wd, grad)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sm.submat_invroot(plan, v, out)
        sm.submat_invroot_backward(plan, wd, grad)
    wd.copy_(torch.tensor(w))
    grad.zero_()
    graph.replay()
    torch.cuda.synchronize()
    gref = oracle.grad(a.rowptr, a.colind, vals, 2, w)
    assert np.abs(grad.cpu().numpy() - gref).max() <= 1e-10 * np.abs(gref).max()


def test_wide_rows_of_one_warp(sm):
    """More rows of order 30 than two waves, all wide: the instance with one warp a row repeats them in FP64,
    forward and adjoint (bars as above, kappa = 300)."""
    rng = np.random.default_rng(121)
    mats = [low_block(30, 300.0, rng) for _ in range(90)]
    a = wl.dense_to_csr(sl.block_diag(*mats), keep=sl.block_diag(*[np.ones((30, 30), bool)] * 90))
    y, rep = forward(sm, a, 2, precision="mixed")
    rows = list(range(0, a.n, 13))
    ref = oracle.invroot(a.rowptr, a.colind, a.vals, 2, rows=rows)
    assert row_err(a, y, ref, rows) <= 30 * 300 * 2.2e-16 and rep["n_fallback"] == 0
    w = wl.random_on_pattern(a, seed=5)
    plan = sm.submat_plan(a.rowptr, a.colind, 2)
    sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"))
    g = sm.submat_invroot_backward(plan, torch.tensor(w, device="cuda")).cpu().numpy()
    gref = oracle.grad(a.rowptr, a.colind, a.vals, 2, w)
    assert np.abs(g - gref).max() <= 30 * 300 * 2.2e-16 * np.abs(gref).max()
    assert plan.work()["bwd_products_df"] == 0 and plan.work()["bwd_flops_fp64"] > 0


@pytest.mark.parametrize("n", [300, 520])
def test_adjoint_of_a_long_wide_row(sm, n):
    """A wide row with blocks (300) and with its partial sums and factors (520) in scratch, among rows of two
    entries: an arrow with one diagonal entry 1 and the others 1/300 to 2/300."""
    d = np.r_[1.0, np.linspace(1.0 / 300.0, 2.0 / 300.0, n - 1)]
    dense = np.diag(d)
    dense[0, 1:] = dense[1:, 0] = 1e-4 * np.random.default_rng(131).uniform(0.5, 1.0, n - 1)
    a = wl.dense_to_csr(dense)
    w = wl.random_on_pattern(a, seed=5)
    gref = oracle.grad(a.rowptr, a.colind, a.vals, 2, w)
    for det in (False, True):
        plan = sm.submat_plan(a.rowptr, a.colind, 2, grad_deterministic=det)
        sm.submat_invroot(plan, torch.tensor(a.vals, device="cuda"))
        g = sm.submat_invroot_backward(plan, torch.tensor(w, device="cuda")).cpu().numpy()
        assert np.abs(g - gref).max() <= n * 300 * 2.2e-16 * np.abs(gref).max()
        assert plan.work()["bwd_flops_fp64"] > 0
