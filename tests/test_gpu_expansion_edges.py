"""Evaluations and translations at the edges of their launches: leaves of 1, 2, 17, 32
and 33 points (target groups of a warp and remainders, lanes on several columns),
orders from a few to where the 2D kernels take other shapes, each layer, graded trees
with List-3 and List-4 entries. Potential and gradient against direct sums at some
targets. The FMM's error measure is within eps for the potential; for a gradient, whose
terms carry a factor of up to the order, within 10 eps of its own norm and the
densities'."""
import numpy as np
import pytest

from cfmm_inputs import curve2d, surface3d, densities
from oracle.direct import direct, direct_grad, relerr_paper
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


def _graded(dim, n):
    c = curve2d(n, seed=80, t_half=10.0, height=0.5) if dim == 2 else \
        surface3d(n, seed=81, half=4.0, amp=0.0, width=1.0, slope=0.0, rho0=1.0)
    rng = np.random.default_rng(82)
    if dim == 3:
        c.re[: n // 2] = 0.3 * rng.standard_normal((n // 2, 3)) ** 3
    else:
        c.re[: n // 2] = 0.02 * rng.standard_normal((n // 2, 2)) ** 3
        c.im[: n // 2] = 0.0
    return c


@pytest.mark.parametrize("layers", ["s", "d", "sd"])
@pytest.mark.parametrize("dim,ker,kap,eps,leaf,n", [
    (3, 0, 0.0, 1e-6, 1, 150), (3, 0, 0.0, 1e-3, 2, 300), (3, 0, 0.0, 1e-6, 17, 700), (3, 0, 0.0, 1e-9, 33, 900),
    (3, 1, 1.0, 1e-3, 2, 300), (3, 1, 1.0, 1e-6, 17, 700), (3, 1, 1.5, 1e-6, 32, 700), (3, 1, 1.5, 1e-6, 33, 900),
    (2, 0, 0.0, 1e-3, 1, 300), (2, 0, 0.0, 1e-9, 2, 500), (2, 0, 0.0, 1e-12, 17, 900), (2, 0, 0.0, 1e-6, 33, 1500),
    (2, 1, 0.3, 1e-3, 1, 300), (2, 1, 5.0, 1e-9, 2, 500), (2, 1, 20.0, 1e-6, 17, 900), (2, 1, 60.0, 1e-9, 33, 1500)])
def test_potential_and_gradient(cuda, dim, ker, kap, eps, leaf, n, layers):
    import paper_2509_05458_gb300 as cf
    c = _graded(dim, n)
    dens = densities(n, seed=83, nrhs=1, ncomp=len(layers))
    flags = ker | (cf.SLP if "s" in layers else 0) | (cf.DLP if "d" in layers else 0)
    p = cf.plan(dim, flags, kap, eps, *(to_dev(a, cuda) for a in (c.re, c.im, c.nrm_re, c.nrm_im)), leaf_size=leaf,
                sep=1 if dim == 2 else 2)
    pick = np.arange(0, n, 5)
    x = c.re + 1j * c.im
    kw = dict(sigma=dens[0, 0] if "s" in layers else None, tau=dens[0, -1] if "d" in layers else None,
              nrm=c.nrm_re + 1j * c.nrm_im)
    u = p.apply(to_dev(dens, cuda)).cpu().numpy()[0]
    assert relerr_paper(u[pick], direct(dim, ker, kap, x, x[pick], **kw), dens[0].reshape(-1)) <= eps
    if layers == "s":
        ug, g = p.apply_grad(to_dev(dens, cuda))
        assert np.array_equal(ug.cpu().numpy()[0], u)
        g0 = direct_grad(dim, ker, kap, x, x[pick], **kw)
        assert relerr_paper(g.cpu().numpy()[0][:, pick].ravel(), np.asarray(g0).ravel(), dens[0].reshape(-1)) <= 10 * eps
