"""An allocation that fails anywhere in a plan or an apply, after the fork to the plan's
second stream too: the plan can be destroyed at once (its buffers go back to a pool that
the next plan draws from) or applied again, and the results are right."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ENOMEM = -4
CASES = [(2, 0, 0.0, 0), (2, 1, 12.0, 0), (2, 1, 12.0, 1), (3, 0, 0.0, 0), (3, 1, 2.0, 0)]


def graded(dim, n, seed):
    """Points thicker towards the origin: all four lists and several levels."""
    rng = np.random.default_rng(seed)
    re = rng.uniform(-1, 1, (n, dim)) ** 3
    return re, 0.2 * re, rng.standard_normal((2, 1, n)) + 1j * rng.standard_normal((2, 1, n))


@pytest.mark.parametrize("dim,ker,kap,prec", CASES)
def test_every_allocation_of_a_plan_and_an_apply(cuda, dim, ker, kap, prec):
    import torch

    import paper_2509_05458_gb300 as cf
    L = cf.lib()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    n = 3000 if dim == 2 else 1500
    a, b = [[t(x) for x in graded(dim, n, s)] for s in (1, 2)]

    def plan(g):
        return cf.plan(dim, ker | cf.SLP, kap, 1e-4, g[0], g[1], leaf_size=20, sep=1 if dim == 2 else 2, precision=prec,
                       top_level=0 if dim == 2 else cf.TOP_FIT)

    def other():
        p = plan(b)
        u = p.apply(b[2])
        torch.cuda.synchronize()
        return u

    ref_b, ref_a = other().clone(), [x.clone() for x in plan(a).apply_grad(a[2])]
    failures = [0, 0]
    try:
        for skip in range(400):                       # plan construction
            L.cfmm_debug_fail_allocs_after(skip, 1)
            try:
                plan(a)
                break
            except cf.CfmmError as e:
                assert e.status == ENOMEM
            failures[0] += 1
            assert torch.equal(other(), ref_b)
        for skip in range(100):                       # a plan's first apply
            L.cfmm_debug_fail_allocs(0)
            p = plan(a)
            L.cfmm_debug_fail_allocs_after(skip, 1)
            try:
                p.apply_grad(a[2])
                break
            except cf.CfmmError as e:
                assert e.status == ENOMEM
            failures[1] += 1
            if skip % 2:                              # applied again, or destroyed at once
                for x, y in zip(p.apply_grad(a[2]), ref_a):
                    assert torch.equal(x, y)
            p.destroy()
            assert torch.equal(other(), ref_b)
    finally:
        L.cfmm_debug_fail_allocs(0)
    assert failures[0] > 20 and failures[1] >= 4
