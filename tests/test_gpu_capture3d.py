"""A captured 3D apply replayed after other calls on its plan and on other plans: the graph
keeps the plan's workspaces, so no call that the interface allows in between may move them
(a gradient, fewer right-hand sides, mixed or repeated)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ker,kap", [(0, 0.0), (1, 3.0)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_replay_after_other_calls(cuda, ker, kap, nrhs):
    import torch

    import paper_2509_05458_gb300 as cf
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    rng = np.random.default_rng(6)
    n = 4000
    re = rng.uniform(-1, 1, (n, 3)) ** 3          # graded: List 3 is not empty
    s = torch.cuda.Stream(device=cuda)
    with torch.cuda.stream(s):
        mk = lambda m: cf.plan(3, ker | cf.SLP, kap, 1e-5, t(re[:m]), t(0.2 * re[:m]), leaf_size=24, sep=2,
                               top_level=cf.TOP_FIT, stream=s)
        p = mk(n)
        assert p.info()["list_len"][2] > 0
        d = t(rng.standard_normal((nrhs, 1, n)) + 1j * rng.standard_normal((nrhs, 1, n)))
        out = torch.empty((nrhs, n), dtype=torch.complex128, device=cuda)
        p.capture(d, out)
        ref = p.apply(d).clone()
        grad = p.apply_grad(d)[1].clone()
        one = p.apply(d[:1]).clone()
        others = [mk(n - 300 * i) for i in range(3)]   # takes whatever went back to the pool
        for q in others:
            q.apply_grad(d[:, :, : q.n].contiguous())
        for _ in range(2):
            out.zero_()
            p.replay()
            s.synchronize()
            assert torch.equal(out, ref)
            for q in others:
                q.apply(d[:, :, : q.n].contiguous())
        assert torch.equal(p.apply(d[:1]), one) and torch.equal(one[0], ref[0])
        assert torch.equal(p.apply_grad(d)[1], grad)
    s.synchronize()
