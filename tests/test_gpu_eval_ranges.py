"""3D M2P, L2P and gradients of a plan whose (List-3 entry, target) items exceed one range
of leaves: against direct sums at sampled targets within eps, potential the same from
apply and apply_grad."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SLOTS = 1 << 22        # of a range


@pytest.mark.parametrize("ker,kap", [(0, 0.0), (1, 1.0)])
def test_items_in_several_ranges(cuda, ker, kap):
    import torch

    import paper_2509_05458_gb300 as cf
    from oracle.direct import direct_grad
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    rng = np.random.default_rng(0)
    n, eps = 200_000, 1e-3
    re = rng.uniform(-1, 1, (n, 3))
    re[: 7 * n // 10] *= 0.25
    im = 0.05 * re
    p = cf.plan(3, ker | cf.SLP, kap, eps, t(re), t(im), leaf_size=100, sep=3, top_level=cf.TOP_FIT)
    tree, (off, _) = p.export_tree(), p.export_list(3)
    items = int((np.diff(off) * (tree["end"] - tree["start"])).sum())
    assert items > SLOTS + SLOTS // 4
    s = rng.standard_normal((2, 1, n)) + 1j * rng.standard_normal((2, 1, n))
    u, g = p.apply_grad(t(s))
    assert torch.equal(u, p.apply(t(s)))
    i = rng.choice(n, 1000, replace=False)
    ref = cf.direct(3, ker | cf.SLP, kap, t(re), t(im), t(re[i]), t(im[i]), t(s))
    size = torch.linalg.vector_norm(ref) + torch.linalg.vector_norm(t(s)) * (1000 / n) ** 0.5
    assert float(torch.linalg.vector_norm(u[:, i] - ref) / size) <= eps
    i = i[:12]
    pts = re + 1j * im
    gref = direct_grad(3, ker, kap, pts, pts[i], sigma=s[0, 0])
    err = np.linalg.norm(g[0][:, i].cpu().numpy() - gref) / np.linalg.norm(gref)
    assert err <= eps
