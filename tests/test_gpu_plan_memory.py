"""Device memory of a plan: given back in full, and the Krylov engine's scratch optional."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1710_10899_gb300 as pkg
    pkg.load_library()
    return pkg


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def dense(n, seed=0):
    rng = np.random.default_rng(seed)
    q = rng.uniform(0.5, 1.0, (n, n)) * (0.2 / n)
    return wl.dense_to_csr(np.eye(n) + q + q.T)


@pytest.mark.parametrize("n,p,kw", [(150, 2, dict(precision="fp64")), (600, 1, dict(precision="mixed")),
                                    (150, 2, dict(precision="mixed"))])
def test_plans_give_their_memory_back(sm, n, p, kw):
    """Twenty plans made and dropped, the forward and (p > 1, which allocates for it) the backward run on each,
    leave the free memory where it was (tens to hundreds of MB a plan are at stake; the allocator's own
    granularity is 2 MB)."""
    a = dense(n)
    v, w = torch.tensor(a.vals, device="cuda"), torch.ones(a.nnz, dtype=torch.float64, device="cuda")
    y, g = torch.empty_like(v), torch.empty_like(v)

    def once():
        plan = sm.submat_plan(a.rowptr, a.colind, p, **kw)
        sm.submat_invroot(plan, v, y, sync=True)
        if p > 1:
            sm.submat_invroot_backward(plan, w, g)
        torch.cuda.synchronize()

    once()
    before = free_bytes()
    for _ in range(20):
        once()
    assert abs(before - free_bytes()) <= 8 << 20


def test_plan_without_room_for_the_krylov_scratch(sm):
    """With room for what the coupled iteration needs but not for the Krylov engine's scratch, the
    plan is made and gives the coupled iteration's bits (those of a plan whose k_max keeps it)."""
    a = dense(600, seed=1)
    v = torch.tensor(a.vals, device="cuda")

    def plan(**kw):
        before = free_bytes()
        p = sm.submat_plan(a.rowptr, a.colind, 2, precision="fp64", **kw)
        return p, before - free_bytes()

    plan()                                           # first use of the library on the device
    krylov, used_krylov = plan()
    coupled, used_coupled = plan(k_max=41)
    assert used_krylov > used_coupled + (100 << 20)
    ref, other = sm.submat_invroot(coupled, v, sync=True), sm.submat_invroot(krylov, v, sync=True)
    assert not torch.equal(ref, other)
    del krylov, coupled
    torch.cuda.empty_cache()
    hog = torch.empty(free_bytes() - (used_krylov + used_coupled) // 2, dtype=torch.uint8, device="cuda")
    try:
        small, _ = plan()
        y = sm.submat_invroot(small, v, sync=True)
        assert torch.equal(y, ref)
    finally:
        del hog
        torch.cuda.empty_cache()
