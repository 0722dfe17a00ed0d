"""2D Laplace expansions in boxes far below the root: more points than a leaf holds at one
place (or within 1e-8 of it) reach the deepest levels through a chain of single boxes with
no List-2 pair on the way, at orders whose powers of the unscaled shifts underflow.

Against the direct sum in FP64 (the paper's error measure). The truncation error is that of
the method on this geometry (separation 1: the criterion drops its prefactors): twice the oracle FMM's
on the coincident points in a unit domain, where the oracle's unscaled expansions are finite,
and 1e-12 for the rounding of sums of 300 terms of mixed size. Mixed precision within 1e-6."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def cloud(spread, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    re = np.concatenate([rng.uniform(0, 1, (230, 2)), np.array([0.3, 0.4]) + spread * rng.uniform(-1, 1, (70, 2))])
    return scale * re, scale * 0.2 * re[:, ::-1], rng


def truncation(layers, eps, scale, dens, nrm):
    """Error of the oracle FMM against the oracle's direct sum, unit domain, coincident points."""
    from oracle import fmm2d
    from oracle.direct import direct
    re, im, _ = cloud(0.0, 4)
    kw = {}
    if "s" in layers:
        kw["sigma"] = dens[0, 0]
    if "d" in layers:
        a, b = (x.cpu().numpy() / scale for x in nrm)
        kw["tau"] = dens[0, -1]
    pts = re + 1j * im
    u, _ = fmm2d.apply(re, im, 0, 0.0, eps, 64, **kw, **(dict(nrm_re=a, nrm_im=b) if "d" in layers else {}))
    ref = direct(2, 0, 0.0, pts, pts, **kw, **(dict(nrm=a + 1j * b) if "d" in layers else {}))
    err = np.linalg.norm(u - ref) / (np.linalg.norm(ref) + np.linalg.norm(dens))
    assert np.isfinite(err)
    return err


@pytest.mark.parametrize("layers", ["s", "d", "sd"])
@pytest.mark.parametrize("spread,eps,scale", [(0.0, 1e-12, 1.0), (0.0, 1e-14, 1.0), (1e-8, 1e-12, 1.0),
                                              (1e-8, 1e-14, 3e-5), (0.0, 1e-12, 7e4)])
def test_chain_of_single_boxes(cuda, layers, spread, eps, scale):
    import torch

    import paper_2509_05458_gb300 as cf
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    re, im, rng = cloud(spread, 4, scale)
    flags = cf.LAPLACE | (cf.SLP if "s" in layers else 0) | (cf.DLP if "d" in layers else 0)
    n, ncomp = len(re), len(layers)
    dens = rng.standard_normal((1, ncomp, n)) + 1j * rng.standard_normal((1, ncomp, n))
    d = t(dens)
    # normals of the points' size, so that both layers weigh alike
    nrm = [t(scale * rng.standard_normal((n, 2))) for _ in range(2)] if "d" in layers else [None, None]
    if "d" in layers and spread:
        for a in nrm:
            a[230:] = 0.0                 # a dipole next to its neighbours would outweigh all else
    geo = (t(re), t(im))
    p = cf.plan(2, flags, 0.0, eps, *geo, *nrm, leaf_size=64)
    assert p.info()["nlevels"] > 24
    ref = cf.direct(2, flags, 0.0, *geo, *geo, d, *nrm)
    size = torch.linalg.vector_norm(ref) + torch.linalg.vector_norm(d)
    u, g = p.apply_grad(d)
    assert torch.isfinite(torch.view_as_real(g)).all()
    assert float(torch.linalg.vector_norm(u - ref) / size) <= 2 * truncation(layers, eps, scale, dens, nrm) + 1e-12
    if scale < 1:
        return                            # r^4 of the mixed pairs leaves FP32's range there
    q = cf.plan(2, flags, 0.0, eps, *geo, *nrm, leaf_size=64, precision=cf.MIXED)
    assert float(torch.linalg.vector_norm(q.apply(d) - ref) / size) <= 1e-6


def test_gradient_of_a_chain(cuda):
    """The gradient's expansions over the same chain, against the oracle FMM's gradient (same
    tree and orders; parity as in tests/test_gpu_grad.py with a digit for 70 equal points)."""
    import torch

    import paper_2509_05458_gb300 as cf
    from oracle import fmm2d
    re, im, rng = cloud(0.0, 5)
    s = rng.standard_normal(len(re)) + 1j * rng.standard_normal(len(re))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    g = cf.plan(2, cf.LAPLACE | cf.SLP, 0.0, 1e-12, t(re), t(im), leaf_size=64).apply_grad(t(s))[1].cpu().numpy()[0]
    _, ref, _ = fmm2d.apply_grad(re, im, 0, 0.0, 1e-12, 64, sigma=s)
    assert np.linalg.norm(g.ravel() - ref.ravel()) <= 1e-11 * np.linalg.norm(ref.ravel())
