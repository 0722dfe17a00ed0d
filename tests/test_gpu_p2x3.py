"""P2M and P2L of the 3D plans in FP64 for each layer, over the orders at which the
kernel holds its sums and source tables in shared memory differently (all sums with
two blocks an SM, with one, one product a pass, groups of 8 sources): the potential
against direct sums at some targets, within the plan's eps in the FMM's error measure.
Leaves of 1 to 70 points and a graded cloud (List-4 entries of a few sources)."""
import numpy as np
import pytest

from cfmm_inputs import surface3d, densities
from oracle.direct import direct, relerr_paper
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


def _cloud(n, graded):
    c = surface3d(n, seed=60, half=4.0, amp=0.5, width=1.0, slope=0.3, rho0=1.0)
    if graded:      # most points in a corner: leaves of many sizes beside one another
        c = surface3d(n, seed=61, half=4.0, amp=0.0, width=1.0, slope=0.0, rho0=1.0)
        rng = np.random.default_rng(62)
        c.re[: n // 2] = 0.3 * rng.standard_normal((n // 2, 3)) ** 3
    return c


@pytest.mark.parametrize("layers", ["s", "d", "sd"])
@pytest.mark.parametrize("ker,kap,eps,leaf,n,graded", [
    (0, 0.0, 1e-3, 7, 900, True), (0, 0.0, 1e-9, 70, 1500, True), (0, 0.0, 1e-13, 64, 1200, False),
    (1, 0.7, 1e-3, 7, 900, True), (1, 2.0, 1e-6, 33, 1500, True), (1, 6.0, 1e-6, 64, 1500, False),
    (1, 9.0, 1e-9, 64, 1500, False), (1, 6.0, 1e-6, 33, 1500, True), (1, 11.5, 1e-9, 300, 1500, False)])
def test_p2m_p2l_layers(cuda, ker, kap, eps, leaf, n, graded, layers):
    import paper_2509_05458_gb300 as cf
    c = _cloud(n, graded)
    dens = densities(n, seed=63, nrhs=1, ncomp=len(layers))
    flags = ker | (cf.SLP if "s" in layers else 0) | (cf.DLP if "d" in layers else 0)
    p = cf.plan(3, flags, kap, eps, *(to_dev(a, cuda) for a in (c.re, c.im, c.nrm_re, c.nrm_im)), leaf_size=leaf,
                sep=2)
    u = p.apply(to_dev(dens, cuda)).cpu().numpy()[0]
    pick = np.arange(0, n, 7)
    x = c.re + 1j * c.im
    u0 = direct(3, ker, kap, x, x[pick], sigma=dens[0, 0] if "s" in layers else None,
                tau=dens[0, -1] if "d" in layers else None, nrm=c.nrm_re + 1j * c.nrm_im)
    assert relerr_paper(u[pick], u0, dens[0].reshape(-1)) <= max(eps, 1e-12)
