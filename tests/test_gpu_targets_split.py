"""plan_targets goes over the sources alone on the source side and over the targets
alone on the target side. Against the plan of sources and targets together (the
targets with zero density): the same tree and the same terms but for products with
zero, summed in another grouping, so the two agree to rounding -- 1e-12 relative l2
in FP64 (sums of up to some thousand terms of 1.1e-16), 1e-6 in mixed precision
(6e-8 a term). Sources and targets are interleaved, apart (boxes without sources,
boxes without targets), or one of them is a single point."""
import numpy as np
import pytest

from cfmm_inputs import curve2d, surface3d, densities
from oracle.direct import relerr_l2
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


def _split(dim, how):
    if dim == 2:
        c = curve2d(2400, seed=50, t_half=10.0, height=0.5)
    else:
        c = surface3d(1800, seed=51, half=4.0, amp=0.5, width=1.0, slope=0.3, rho0=1.0)
    rng = np.random.default_rng(52)
    src = {"mixed": rng.random(c.n) < 0.6, "apart": c.re[:, 0] < 0.0, "one target": np.arange(c.n) != 700,
           "one source": np.arange(c.n) == 700}[how]
    return c, src


@pytest.mark.parametrize("dim,ker,kap", [(2, 0, 0.0), (2, 1, 6.0), (3, 0, 0.0), (3, 1, 3.0)])
@pytest.mark.parametrize("how", ["mixed", "apart", "one target", "one source"])
def test_targets_against_union(cuda, dim, ker, kap, how):
    import paper_2509_05458_gb300 as cf
    c, src = _split(dim, how)
    eps, sep = (1e-6, 1) if dim == 2 else (1e-3, 2)
    order = np.concatenate([np.flatnonzero(src), np.flatnonzero(~src)])
    ns = int(src.sum())
    re, im, nre, nim = (np.ascontiguousarray(a[order]) for a in (c.re, c.im, c.nrm_re, c.nrm_im))
    dens = densities(c.n, seed=53, nrhs=2, ncomp=2)
    dens[..., ns:] = 0.0
    flags = ker | cf.SLP | cf.DLP
    for prec, tol in ((cf.FP64, 1e-12), (cf.MIXED, 1e-6)):
        kw = dict(leaf_size=20, sep=sep, precision=prec)
        p = cf.plan(dim, flags, kap, eps, *(to_dev(a, cuda) for a in (re, im, nre, nim)), **kw)
        ref = p.apply(to_dev(dens, cuda)).cpu().numpy()[:, ns:]
        q = cf.plan_targets(dim, flags, kap, eps, *(to_dev(a, cuda) for a in (re[:ns], im[:ns], re[ns:], im[ns:],
                                                                            nre[:ns], nim[:ns])), **kw)
        u = q.apply(to_dev(np.ascontiguousarray(dens[..., :ns]), cuda)).cpu().numpy()
        assert u.shape == ref.shape
        assert relerr_l2(u, ref) <= tol
