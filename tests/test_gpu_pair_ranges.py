"""3D M2L whose pairs of a level fall into several ranges: results are the same bits for two
plans of one geometry and for a right-hand side alone and among others (more of them than
a range's budget takes at once), and a captured apply survives one with fewer."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BUDGET, ROW, RHS = 6 << 30, 512, 4      # bytes of a range, of a row of a tile; right-hand sides it counts
KERNELS = [(0, 0.0), (1, 1.0)]


def setup(cuda, ker, kap, nrhs, stream=None):
    import torch

    import paper_2509_05458_gb300 as cf
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    rng = np.random.default_rng(1)
    n = 150_000
    re = t(rng.uniform(-1, 1, (n, 3)))
    im = 0.05 * re
    make = lambda: cf.plan(3, ker | cf.SLP, kap, 1e-3, re, im, leaf_size=48, sep=3, top_level=cf.TOP_FIT,
                           stream=stream)
    p = make()
    tree, (off, _), P = p.export_tree(), p.export_list(2), p.orders()
    for level in range(p.info()["l0"], p.info()["nlevels"]):
        at = tree["level"] == level
        tiles = int(np.diff(off)[at].sum()) // 64
        row = 2 * RHS * (P[level] + 1) ** 2 + ((P[level] + 1) * (P[level] + 2) * (P[level] + 3) // 6 if ker else 0)
        if tiles * int(row) * ROW > 2 * BUDGET:
            break
    else:
        raise AssertionError("no level of several ranges")
    d = t(rng.standard_normal((nrhs, 1, n)) + 1j * rng.standard_normal((nrhs, 1, n)))
    return p, make, d


@pytest.mark.parametrize("ker,kap", KERNELS)
def test_same_bits(cuda, ker, kap):
    import torch
    p, make, d = setup(cuda, ker, kap, 6)
    u = p.apply(d)
    for i in (0, 5):
        assert torch.equal(p.apply(d[i:i + 1])[0], u[i])
    q = make()
    for _ in range(2):
        assert torch.equal(q.apply(d), u)
    q.destroy()
    assert torch.equal(make().apply(d), u)


@pytest.mark.parametrize("ker,kap", KERNELS)
def test_replay_after_fewer_right_hand_sides(cuda, ker, kap):
    import torch
    s = torch.cuda.Stream(device=cuda)
    with torch.cuda.stream(s):
        p, make, d = setup(cuda, ker, kap, 6, stream=s)
        out = torch.empty((6, d.shape[2]), dtype=torch.complex128, device=cuda)
        p.capture(d, out)
        ref = out.clone()
        p.apply(d[:1])
        q = make()                        # takes whatever went back to the pool
        q.apply(d[:1])
        out.zero_()
        p.replay()
        s.synchronize()
        q.apply(d[:1])
        assert torch.equal(out, ref)
    s.synchronize()
