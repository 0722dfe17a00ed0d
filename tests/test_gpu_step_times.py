"""Per-step times of a 2D apply whose P2L (and, mixed, M2P) runs on the plan's second stream:
each shows in its own step, not in the near field's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
def test_side_work_is_timed_in_its_step(cuda, prec):
    import torch

    import paper_2509_05458_gb300 as cf
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    rng = np.random.default_rng(8)
    n = 4000
    re = rng.uniform(-1, 1, (n, 2)) ** 5            # graded: Lists 3 and 4
    p = cf.plan(2, cf.HELMHOLTZ | cf.SLP, 20.0, 1e-9, t(re), t(0.2 * re), leaf_size=32, precision=prec)
    inf = p.info()
    assert inf["list_len"][2] > 0 and inf["list_len"][3] > 0 and inf["p2p_pairs"] <= 1 << 21
    d = t(rng.standard_normal((1, n)) + 1j * rng.standard_normal((1, n)))
    ref = p.apply(d).clone()
    times = {}
    for mode in (1, 2):
        p.set_timing(mode)
        for _ in range(3):
            assert torch.equal(p.apply(d), ref)
        times[mode] = [min(x) for x in zip(*[(p.apply(d), p.timings())[1] for _ in range(8)])]
    both, alone = times[1], times[2]
    assert all(x >= 0 for x in both + alone)
    # beside other work a step's kernels take no less than alone, up to the events' own spread
    steps = (4, 6, 7) if prec else (4, 6)
    for i in steps:
        assert both[i] > 0.6 * alone[i], (i, both, alone)
    # and the near field's bracket holds the near field: P2L alone is longer than it here
    assert both[6] < alone[6] + 0.5 * alone[4] + 0.05, (both, alone)
