"""The admission estimate covers what a 3D request's plan and applies take on the device
(each in a process of its own, so that no cached block hides an allocation)."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import numpy as np, torch
import paper_2509_05458_gb300 as cf
from cfmm_inputs import surface3d, densities
from paper_2509_05458_gb300.serving import Request, estimate_bytes
n, ker, kap, eps, leaf, sep = {args}
g = surface3d(n, seed=3, half=20.0, random_shape=True)
d = densities(n, seed=4, nrhs=1, ncomp=1)
req = Request(0, 3, ker | cf.SLP, kap, eps, g.re, g.im, [d[0]], leaf_size=leaf, sep=sep)
t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to('cuda:0')
x = [t(g.re), t(g.im), t(d)]
u = torch.empty((1, n), dtype=torch.complex128, device='cuda:0')
s = g.re[:64]
cf.plan(3, ker | cf.SLP, kap, eps, t(s), t(s * 0), leaf_size=64).apply(t(d[:, :, :64]))    # context, modules
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
p = cf.plan(3, ker | cf.SLP, kap, eps, x[0], x[1], leaf_size=leaf, sep=sep, precision=cf.AUTO, top_level=cf.TOP_FIT)
p.apply(x[2], out=u)
torch.cuda.synchronize()
print('used', free - torch.cuda.mem_get_info()[0], 'estimate', estimate_bytes(req), p.orders().tolist())
"""


@pytest.mark.parametrize("args", [(200_000, 0, 0.0, 1e-9, 64, 1), (50_000, 0, 0.0, 1e-6, 64, 2),
                                  (200_000, 1, 5.0, 1e-6, 64, 2), (30_000, 1, 3.0, 1e-3, 32, 2)])
def test_estimate_covers_use(cuda, args):
    r = subprocess.run([sys.executable, "-c", CODE.format(args=args)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    w = r.stdout.split()
    used, estimate = int(w[w.index("used") + 1]), int(w[w.index("estimate") + 1])
    print(r.stdout)
    assert 0 < used <= estimate
