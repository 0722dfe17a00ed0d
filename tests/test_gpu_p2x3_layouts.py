"""P2M and P2L of 3D plans in FP64 at the orders where the kernel's shared memory leaves room
for less: with the sums of a double layer one product a pass (Laplace above order 46, P2L 45;
Helmholtz above 38), with groups of 8 sources (Helmholtz from order 62). Orders are asserted,
so that each case runs the layout it is meant for. Real points (the truncation criterion
holds), against direct sums at some targets: within eps for Helmholtz, whose orders keep two
digits; within 10 eps for Laplace, one digit, of which the double layer's derivative takes up
to P/2 times the tail."""
import numpy as np
import pytest

from cfmm_inputs import densities, surface3d
from oracle.direct import direct, relerr_paper
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


def check(cuda, c, ker, kap, eps, leaf, sep, layers, orders, tol):
    import paper_2509_05458_gb300 as cf
    n = c.n
    dens = densities(n, seed=63, nrhs=1, ncomp=len(layers))
    flags = ker | (cf.SLP if "s" in layers else 0) | (cf.DLP if "d" in layers else 0)
    p = cf.plan(3, flags, kap, eps, *(to_dev(a, cuda) for a in (c.re, c.im, c.nrm_re, c.nrm_im)), leaf_size=leaf,
                sep=sep, top_level=cf.TOP_FIT)
    tree, P = p.export_tree(), p.orders()
    at = sorted(set(int(P[l]) for l in tree["level"][tree["leaf"] != 0]), reverse=True)
    assert orders[0] <= at[0] <= orders[1], at
    assert p.info()["list_len"][3] > 0                  # P2L runs too
    u = p.apply(to_dev(dens, cuda)).cpu().numpy()[0]
    pick = np.arange(0, n, 7)
    x = c.re + 1j * c.im
    u0 = direct(3, ker, kap, x, x[pick], sigma=dens[0, 0] if "s" in layers else None,
                tau=dens[0, -1] if "d" in layers else None, nrm=c.nrm_re + 1j * c.nrm_im)
    assert relerr_paper(u[pick], u0, dens[0].reshape(-1)) <= tol


@pytest.mark.parametrize("layers", ["s", "d", "sd"])
@pytest.mark.parametrize("eps,orders", [(1e-9, (40, 44)), (1e-10, (47, 49)), (1e-12, (53, 63))])
def test_laplace(cuda, eps, orders, layers):
    c = surface3d(1500, seed=61, half=4.0, amp=0.0, width=1.0, slope=0.0, rho0=1.0)
    c.re[:750] = 0.3 * np.random.default_rng(62).standard_normal((750, 3)) ** 3
    check(cuda, c, 0, 0.0, eps, 33, 1, layers, orders, 10 * eps)


@pytest.mark.parametrize("layers", ["s", "d", "sd"])
@pytest.mark.parametrize("kap,eps,orders", [(13.0, 1e-6, (33, 38)), (20.0, 1e-6, (48, 52)), (22.5, 1e-9, (62, 63))])
def test_helmholtz(cuda, kap, eps, orders, layers):
    c = surface3d(1500, seed=60, half=4.0, amp=0.5, width=1.0, slope=0.0, rho0=1.0)
    check(cuda, c, 1, kap, eps, 64, 2, layers, orders, eps)
