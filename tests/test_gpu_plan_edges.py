"""Plans at the sizes where the scan and the lists change their launch: key counts of
64 and 65 sort tiles (one block scans up to 16,384 counts), lists of more than 1,024
entries (not sorted in shared memory; the widest separation). A box's entries ascend; the potential
at some targets against direct sums, within eps."""
import numpy as np
import pytest

from cfmm_inputs import curve2d, surface3d, densities
from oracle.direct import direct, relerr_paper
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,leaf,sep", [(2, 131071, 40, 1), (2, 131072, 40, 1), (2, 131073, 40, 1),
                                            (2, 2049, 1, 1), (3, 1500, 2, 2), (3, 2500, 1, 3)])
def test_plan_sizes(cuda, dim, n, leaf, sep):
    import paper_2509_05458_gb300 as cf
    c = curve2d(n, seed=70, t_half=10.0, height=0.5) if dim == 2 else \
        surface3d(n, seed=71, half=4.0, amp=0.5, width=1.0, slope=0.3, rho0=1.0)
    dens = densities(n, seed=72, nrhs=1, ncomp=1)
    eps = 1e-6
    p = cf.plan(dim, cf.LAPLACE | cf.SLP, 0.0, eps, to_dev(c.re, cuda), to_dev(c.im, cuda), leaf_size=leaf, sep=sep)
    u = p.apply(to_dev(dens, cuda)).cpu().numpy()[0]
    pick = np.arange(5, n, n // 40)
    x = c.re + 1j * c.im
    u0 = direct(dim, 0, 0.0, x, x[pick], sigma=dens[0, 0])
    assert relerr_paper(u[pick], u0, dens[0].reshape(-1)) <= eps
    if n < 10000:
        for w in range(1, 5):
            off, ent = p.export_list(w)
            for b in range(len(off) - 1):
                assert np.all(np.diff(ent[off[b]:off[b + 1]]) > 0)
