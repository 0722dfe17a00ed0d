"""3D M2L with the pairs on the lanes: tile remainders, flat and general shifts in
one list, several right-hand sides and lists that are split into ranges.

Against the direct sum the FMM meets eps; against itself (one right-hand side at a
time, another split of the same sums) it agrees to rounding: the M2L adds at most
a few thousand terms per coefficient in two orders, 1e-12 of the result's norm."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def two_layers(n, gap, seed):
    """A flat sheet and one above it: shifts with d3 = 0 and without."""
    rng = np.random.default_rng(seed)
    re = np.concatenate([rng.uniform(-4, 4, (n, 2)), gap * rng.integers(0, 2, (n, 1))], 1)
    im = 0.3 * np.concatenate([re[:, :2], np.zeros((n, 1))], 1)
    return re, im


@pytest.mark.parametrize("ker,kap,eps", [(0, 0.0, 1e-3), (0, 0.0, 1e-9), (1, 2.0, 1e-4), (1, 3.0, 1e-8)])
@pytest.mark.parametrize("n,gap,leaf", [(700, 0.0, 40), (900, 1.3, 30), (333, 2.7, 8)])
def test_layers(cuda, ker, kap, eps, n, gap, leaf):
    import torch

    import paper_2509_05458_gb300 as cf
    re, im = two_layers(n, gap, n)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    rng = np.random.default_rng(1)
    d = t(rng.standard_normal((3, 1, n)) + 1j * rng.standard_normal((3, 1, n)))
    p = cf.plan(3, ker | cf.SLP, kap, eps, t(re), t(im), leaf_size=leaf, sep=2, top_level=cf.TOP_FIT)
    assert p.info()["m2l_pairs"] > 0
    u = p.apply(d)
    ref = cf.direct(3, ker | cf.SLP, kap, t(re), t(im), t(re), t(im), d)
    err = torch.linalg.vector_norm(u - ref) / (torch.linalg.vector_norm(ref) + torch.linalg.vector_norm(d))
    assert float(err) <= eps
    for i in range(3):
        one = p.apply(d[i:i + 1])
        assert torch.equal(one[0], u[i])       # a pair's arithmetic does not depend on its neighbours


def test_ranges(cuda):
    """Enough right-hand sides that the pair vectors exceed one range's budget."""
    import torch

    import paper_2509_05458_gb300 as cf
    re, im = two_layers(2500, 0.0, 5)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    rng = np.random.default_rng(2)
    d = t(rng.standard_normal((96, 1, 2500)) + 1j * rng.standard_normal((96, 1, 2500)))
    p = cf.plan(3, cf.HELMHOLTZ | cf.SLP, 8.0, 1e-6, t(re), t(im), leaf_size=20, sep=2, top_level=cf.TOP_FIT)
    inf = p.info()
    per_level_bytes = 96 * 16 * (int(p.orders()[inf["l0"]]) + 1) ** 2 * inf["m2l_pairs"]
    assert per_level_bytes > 6 << 30
    u = p.apply(d)
    for i in (0, 50, 95):
        one = p.apply(d[i:i + 1])
        assert float(torch.linalg.vector_norm(one[0] - u[i]) / torch.linalg.vector_norm(one)) < 1e-12
