"""Timing cases: the submatrix method's calls over the sizes, precisions and options in use.

The matrices are the Gaussian-overlap stand-ins of the repository's workloads (points in a
box, A_ij = exp(-r^2 / 0.01) inside the cutoff 0.12, a diagonal that sets the condition
number; atoms with 13 Gaussian functions each for the block-sparse one), built with torch on
the GPU.  A case's geometry, and with it the pattern, is fixed; the seed draws the norms of
the functions (A becomes D A D with D's entries in 0.9 .. 1.1), as a program meets new values
on the pattern it has planned.  A state holds what a program keeps between calls: the plan of
the pattern, the values, and for a training step the cotangent.
"""
import concurrent.futures
import math

import numpy as np
import torch

import paper_1710_10899_gb300 as sm

WIDTH = 0.01        # A_ij = exp(-r^2 / WIDTH)
CUTOFF = 0.12
FUNCS = 13          # functions per atom of the block-sparse matrix


def listed():
    return [
        # a few hundred points, a handful of entries per row: a call is launches and latency
        dict(name="tiny_mixed", kind="small", n=200, p=2, precision="mixed", sign=-1),
        # the plain method: n = 2000, FP64, rows of 1..27 entries
        dict(name="small_fp64", kind="small", n=2000, p=2, precision="fp64", sign=-1),
        # the FP64 path at ordinary row lengths (32..240): the accuracy reference in use
        dict(name="uniform_fp64", kind="uniform", n=2048, per_row=200, p=2, precision="fp64",
             sign=-1),
        # the headline: A^(-1/2), n = 32768, about 177 entries per row, mixed precision
        dict(name="uniform_p2", kind="uniform", n=32768, per_row=200, p=2, precision="mixed",
             sign=-1),
        # the inverse on the pattern
        dict(name="uniform_p1", kind="uniform", n=12288, per_row=200, p=1, precision="mixed",
             sign=-1),
        # inverse cube root, an odd number of rows, shorter rows
        dict(name="uniform_p3_odd", kind="uniform", n=9973, per_row=130, p=3, precision="mixed",
             sign=-1),
        # positive root A^(1/2), medium rows
        dict(name="uniform_sqrt", kind="uniform", n=8192, per_row=90, p=2, precision="mixed",
             sign=1),
        # uneven rows (clustered points): orders of about 10..500 in one call
        dict(name="clustered", kind="clustered", n=12000, p=2, precision="mixed", sign=-1),
        # block-sparse basis-function overlap: orders of about 550..1235, 13 rows per pattern
        dict(name="block", kind="block", atoms=400, p=2, precision="mixed", sign=-1),
        # a training step: forward and the gradient with respect to A's stored values
        dict(name="train_step", kind="train", n=6144, per_row=150, p=2, precision="mixed",
             sign=-1, deterministic=False),
        # the same in FP64, deterministic gradient, short rows
        dict(name="train_fp64_det", kind="train", n=2501, per_row=60, p=2, precision="fp64",
             sign=-1, deterministic=True),
        # conjugate gradients preconditioned with the method's A^(-1/2): a solve of an
        # anisotropic grid operator, forward for K included
        dict(name="pcg", kind="pcg", nx=64, p=2, precision="mixed", sign=-1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "small", "uniform", "uniform", "uniform", "uniform_fp64",
                       "clustered", "block", "train", "train", "pcg"])
    if kind == "small":
        return dict(kind="small", n=_log_int(rng, 100, 4000), p=rng.choice([1, 2, 2, 3]),
                    precision=rng.choice(["mixed", "fp64"]), sign=rng.choice([-1, -1, 1]))
    if kind == "uniform":
        return dict(kind="uniform", n=_log_int(rng, 1000, 20000), per_row=_log_int(rng, 50, 220),
                    p=rng.choice([1, 2, 2, 3]), precision="mixed", sign=rng.choice([-1, -1, 1]))
    if kind == "uniform_fp64":
        return dict(kind="uniform", n=_log_int(rng, 300, 2000), per_row=_log_int(rng, 50, 200),
                    p=rng.choice([1, 2, 3]), precision="fp64", sign=-1)
    if kind == "clustered":
        return dict(kind="clustered", n=_log_int(rng, 3000, 12000), p=rng.choice([1, 2, 2]),
                    precision="mixed", sign=-1)
    if kind == "block":
        return dict(kind="block", atoms=rng.randint(150, 400), p=2, precision="mixed", sign=-1)
    if kind == "train":
        return dict(kind="train", n=_log_int(rng, 500, 5000), per_row=_log_int(rng, 40, 160),
                    p=rng.choice([1, 2, 3]), precision=rng.choice(["mixed", "mixed", "fp64"]),
                    sign=rng.choice([-1, -1, 1]), deterministic=rng.choice([False, True]))
    return dict(kind="pcg", nx=rng.randint(24, 72), p=2, precision="mixed", sign=-1)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _points(n, side, seed, clusters=0):
    g = torch.Generator().manual_seed(seed)
    if not clusters:
        return torch.rand(n, 3, generator=g, dtype=torch.float64) * side
    nc = int(0.85 * n)
    centres = torch.rand(clusters, 3, generator=g, dtype=torch.float64) * side
    label = torch.randint(0, clusters, (nc,), generator=g)
    near = centres[label] + 0.05 * side * torch.randn(nc, 3, generator=g, dtype=torch.float64)
    rest = torch.rand(n - nc, 3, generator=g, dtype=torch.float64) * side
    return torch.cat([near, rest]) % side


def _pairs(x, cutoff, box):
    """Stored pairs (r, c), row by row with c ascending, both directions and the diagonal,
    and their squared distances."""
    n = x.shape[0]
    rs, cs, ds = [], [], []
    step = max(1, (1 << 27) // (8 * n))
    for b in range(0, n, step):
        d2 = torch.zeros(min(step, n - b), n, dtype=torch.float64, device=x.device)
        for k in range(3):
            d = x[b:b + step, k, None] - x[None, :, k]
            if box:
                d -= box * torch.round(d / box)
            d2 += d * d
        r, c = torch.nonzero(d2 < cutoff * cutoff, as_tuple=True)
        rs.append(r + b)
        cs.append(c)
        ds.append(d2[r, c])
    return torch.cat(rs), torch.cat(cs), torch.cat(ds)


def _rowptr(r, n):
    return torch.cat([torch.zeros(1, dtype=torch.int64, device=r.device),
                      torch.cumsum(torch.bincount(r, minlength=n), 0)])


def _extremes(r, c, v, n, seed, steps=60):
    """Estimates of the smallest and largest eigenvalue (Lanczos, rows padded to one length
    so that every sum has a fixed order)."""
    rp = _rowptr(r, n)
    at = torch.arange(r.numel(), device=r.device) - rp[r]
    width = int((rp[1:] - rp[:-1]).max())
    cols = torch.zeros(n, width, dtype=torch.int64, device=r.device)
    vals = torch.zeros(n, width, dtype=torch.float64, device=r.device)
    cols[r, at] = c
    vals[r, at] = v
    g = torch.Generator().manual_seed(seed + 77)
    q = torch.randn(n, generator=g, dtype=torch.float64).to(r.device)
    q /= q.norm()
    prev, beta = torch.zeros_like(q), torch.zeros((), dtype=torch.float64, device=r.device)
    al, be = [], []
    for _ in range(min(steps, n)):
        w = (vals * q[cols]).sum(1) - beta * prev
        a = torch.dot(w, q)
        w -= a * q
        beta = w.norm()
        prev, q = q, w / beta
        al.append(a)
        be.append(beta)
    al, be = torch.stack(al).cpu().numpy(), torch.stack(be).cpu().numpy()[:-1]
    e = np.linalg.eigvalsh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))
    return float(e[0]), float(e[-1])


def _shift(lo, hi, kappa):
    d = (hi - kappa * lo) / (kappa - 1.0)
    return float("%.4g" % d)     # the same number whatever the last bits of the estimates


def _matrix(case, seed):
    """(rowptr, colind, vals) on the GPU."""
    if case["kind"] == "pcg":
        return _grid(case["nx"], seed)
    rowptr, r, c, v = _overlap(case)
    g = torch.Generator().manual_seed(seed)
    d = (0.9 + 0.2 * torch.rand(rowptr.numel() - 1, generator=g, dtype=torch.float64)).to(v.device)
    return rowptr.int(), c.int(), v * (d[r] * d[c])


def _overlap(case, seed=0):
    """(rowptr, rows, columns, values) of the case's overlap matrix."""
    dev = "cuda"
    kind = case["kind"]
    if kind == "block":
        atoms = case["atoms"]
        rc = (64.0 / (20000 * 4.0 / 3.0 * math.pi)) ** (1.0 / 3.0)
        side = (atoms / 20000.0) ** (1.0 / 3.0)
        ra, ca, d2 = _pairs(_points(atoms, side, seed).to(dev), rc, side)
        n = atoms * FUNCS
        f = torch.arange(FUNCS, device=dev)
        alpha = 0.5 * 16.0 ** (f.double() / (FUNCS - 1)) / rc ** 2
        tot = alpha[:, None] + alpha[None, :]
        prod = alpha[:, None] * alpha[None, :]
        pref = (2.0 * torch.sqrt(prod) / tot) ** 1.5
        v = pref[None] * torch.exp(-(prod / tot)[None] * d2[:, None, None])
        r = (ra[:, None, None] * FUNCS + f[None, :, None]).expand(v.shape).reshape(-1)
        c = (ca[:, None, None] * FUNCS + f[None, None, :]).expand(v.shape).reshape(-1)
        key, order = torch.sort(r * n + c)
        r, c, v = key // n, key % n, v.reshape(-1)[order]
        lo, hi = _extremes(r, c, v, n, seed)
        v = torch.where(r == c, v + _shift(lo, hi, 1e4), v)
        return _rowptr(r, n), r, c, v
    n = case["n"]
    if kind == "small":
        pts, box = _points(n, (n / 2000.0) ** (1.0 / 3.0), seed), 0.0
    elif kind == "clustered":
        box = 2.0 * (n / 131072.0) ** (1.0 / 3.0)
        pts = _points(n, box, seed, clusters=64)
    else:
        box = 0.0
        pts = _points(n, (n * 4.0 / 3.0 * math.pi * CUTOFF ** 3 / case["per_row"]) ** (1.0 / 3.0),
                      seed)
    r, c, d2 = _pairs(pts.to(dev), CUTOFF, box)
    v = torch.exp(-d2 / WIDTH)
    if kind == "small":
        d = 1.5
    else:
        v = torch.where(r == c, torch.zeros_like(v), v)
        lo, hi = _extremes(r, c, v, n, seed)
        d = _shift(lo, hi, 1e3)
    v = torch.where(r == c, torch.full_like(v, d), v)
    return _rowptr(r, n), r, c, v


def _grid(nx, seed):
    """Five-point operator on an nx x nx grid: coupling 1 along x, about 0.01 along y."""
    n = nx * nx
    k = torch.arange(n)
    g = torch.Generator().manual_seed(seed)
    eps = 0.008 + 0.004 * float(torch.rand((), generator=g))
    x, y = k % nx, k // nx
    cols = torch.stack([k - nx, k - 1, k, k + 1, k + nx], 1)
    ok = torch.stack([y > 0, x > 0, k >= 0, x + 1 < nx, y + 1 < nx], 1)
    vals = torch.tensor([-eps, -1.0, 2.0 + 2.0 * eps, -1.0, -eps],
                        dtype=torch.float64).expand(n, 5)
    rowptr = torch.cat([torch.zeros(1, dtype=torch.int64), torch.cumsum(ok.sum(1), 0)])
    return rowptr.int().cuda(), cols[ok].int().cuda(), vals[ok].cuda()


def prepare(case, seed):
    rowptr, colind, vals = _matrix(case, seed)
    plan = sm.submat_plan(rowptr, colind, case["p"], precision=case["precision"],
                          root_sign=case["sign"],
                          grad_deterministic=bool(case.get("deterministic", False)))
    state = dict(kind=case["kind"], plan=plan, vals=vals)
    if case["kind"] == "train":
        g = torch.Generator().manual_seed(seed + 1)
        state["w"] = torch.randn(vals.numel(), generator=g, dtype=torch.float64).cuda()
    if case["kind"] == "pcg":
        state["b"] = torch.ones(plan.n, dtype=torch.float64, device="cuda")
    return state


def run(state):
    plan, vals = state["plan"], state["vals"]
    if state["kind"] == "train":
        x = vals.detach().requires_grad_(True)
        y = sm.SubmatInvRoot.apply(x, plan)
        y.backward(state["w"])
        return {"root": y.detach(), "grad": x.grad}
    if state["kind"] == "pcg":
        k = sm.submat_invroot(plan, vals)
        x, steps, resid = sm.submat_pcg(plan, vals, state["b"], vals_k=k)
        return {"k": k, "x": x, "steps": steps, "resid": resid}
    return sm.submat_invroot(plan, vals)


_sizes = {}


def work(case):
    """Bytes: the pattern and the values once, the results once.  Flops: a column of a root of
    a well-conditioned submatrix takes some tens of products with it (32 counted, 2 m^2 each);
    its gradient as many again for the cotangent and a rank-32 sum over the m^2 entries."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _sizes:
        rowptr = _matrix(case, 0)[0].long()
        m = (rowptr[1:] - rowptr[:-1]).double()
        _sizes[key] = (int(rowptr.numel() - 1), float(m.sum()), float((m * m).sum()))
    n, nnz, m2 = _sizes[key]
    out = dict(bytes=4.0 * (n + 1) + 20.0 * nnz, flops=64.0 * m2)
    if case["kind"] == "train":
        out["bytes"] += 16.0 * nnz
        out["flops"] += 128.0 * m2
    elif case["kind"] == "pcg":
        # of the order of 2 nx steps: A, K and K^T once each (12 bytes an entry), six vectors
        steps = 2.0 * case["nx"]
        out["bytes"] += steps * (36.0 * nnz + 48.0 * n)
        out["flops"] += steps * (6.0 * nnz + 12.0 * n)
    return out


# ---------------------------------------------------------------------------
# The same in 64 bits, from LAPACK eigendecompositions on the host
# ---------------------------------------------------------------------------

def _divided(lam, f, fprime):
    """First divided differences of f at the eigenvalues (f' on and near the diagonal)."""
    d = lam[:, None] - lam[None, :]
    close = np.abs(d) < 1e-5 * np.abs(lam).max()
    mid = 0.5 * (lam[:, None] + lam[None, :])
    q = (f(lam)[:, None] - f(lam)[None, :]) / np.where(close, 1.0, d)
    return np.where(close, fprime(mid), q)


def exact(case, seed):
    if case["kind"] == "pcg":
        return None                          # an iterative solve to 1e-6
    rowptr, colind, vals = _matrix(case, seed)
    rowptr, colind = rowptr.long(), colind.long()
    n = rowptr.numel() - 1
    m = rowptr[1:] - rowptr[:-1]
    r = torch.repeat_interleave(torch.arange(n, device=m.device), m)
    dense = torch.zeros(n, n, dtype=torch.float64, device=m.device)
    dense[r, colind] = vals
    train = case["kind"] == "train"
    w = gradient = None
    if train:
        g = torch.Generator().manual_seed(seed + 1)
        w = torch.randn(vals.numel(), generator=g, dtype=torch.float64)
        gradient = torch.zeros_like(dense)
    rp, ci = rowptr.cpu().numpy(), colind.cpu().numpy()
    # rows with the same pattern (the functions of one atom) have one submatrix
    groups = []
    for j in range(n):
        if groups and np.array_equal(ci[rp[j]:rp[j + 1]], ci[rp[j - 1]:rp[j]]):
            groups[-1].append(j)
        else:
            groups.append([j])
    if sum(float(rp[g[0] + 1] - rp[g[0]]) ** 3 for g in groups) > (8e10 if train else 3.5e11):
        return None                          # too many eigendecompositions
    s = case["sign"] / case["p"]
    out = torch.empty(vals.numel(), dtype=torch.float64)

    def one(job):
        group, S = job
        R = ci[rp[group[0]]:rp[group[0] + 1]]
        lam, V = torch.linalg.eigh(S)
        root, G = lam ** s, 0.0
        for j in group:
            at = slice(int(rp[j]), int(rp[j + 1]))
            pos = int(np.searchsorted(R, j))
            out[at] = torch.mv(V, root * V[pos])
            if train:
                ln = lam.numpy()
                phi = torch.from_numpy(_divided(ln, lambda x: x ** s,
                                                lambda x: s * x ** (s - 1.0)))
                sym = torch.outer(torch.mv(V.T, w[at]), V[pos])
                G = G + torch.mm(torch.mm(V, phi * (0.5 * (sym + sym.T))), V.T)
        return group, G

    # one LAPACK thread per worker: the submatrices are small
    with concurrent.futures.ThreadPoolExecutor(16, initializer=torch.set_num_threads,
                                               initargs=(1,)) as pool:
        for b in range(0, len(groups), 256):
            jobs = []
            for group in groups[b:b + 256]:
                R = colind[rp[group[0]]:rp[group[0] + 1]]
                jobs.append((group, dense[R[:, None], R[None, :]].cpu()))
            for group, G in pool.map(one, jobs):
                if train:
                    R = colind[rp[group[0]]:rp[group[0] + 1]]
                    gradient[R[:, None], R[None, :]] += G.to(gradient.device)
    if train:
        return {"root": out, "grad": gradient[r, colind].cpu()}
    return out
