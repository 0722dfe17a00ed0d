"""FP64 pair evaluation and its block shapes against scipy in FP64.

The kernel values are compared pair by pair (one source) over the whole range of
|kappa r| with points on the limits of the evaluation's cases, inside and outside
the sector of its tables; AMOS and numpy are good to a few 1e-15 relative at
these arguments, r^2 rounds to 1e-16 relative in either, and the phase kappa r
magnifies that by |kappa r|: tolerance 4e-15 (1 + |kappa r|) relative to the
kernel (2D Laplace: absolute, as log r has a zero)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def kernel(dim, ker, kap, d, nrm):
    from scipy.special import hankel1
    r2 = (d * d).sum(1)
    r = np.sqrt(r2)
    nd = d @ nrm
    if dim == 2 and ker == 0:
        return np.log(r2) / 2, -nd / r2
    if dim == 2:
        return hankel1(0, kap * r), kap * hankel1(1, kap * r) / r * nd
    if ker == 0:
        return 1 / r, nd / (r2 * r)
    e = np.exp(1j * kap * r) / r
    return e, nd * (1 - 1j * kap * r) * e / r2


@pytest.mark.parametrize("dim,ker", [(2, 0), (2, 1), (3, 0), (3, 1)])
@pytest.mark.parametrize("slope", [0.0, 0.45, -0.45, 2.0])
def test_pair_values(cuda, dim, ker, slope):
    import torch

    import paper_2509_05458_gb300 as cf
    kap = 1.75
    z = np.concatenate([np.geomspace(1e-5, 300.0, 1500), [x * s for x in (0.5, 1.0, 2.0, 8.0)
                                                           for s in (1 - 1e-9, 1.0, 1 + 1e-9)]])
    rng = np.random.default_rng(7)
    u = rng.standard_normal((z.size, dim))
    u /= np.linalg.norm(u, axis=1)[:, None]
    re = u * (z / kap)[:, None]
    # slope 2: Im along one axis only, so that r^2 leaves the right half plane for some pairs
    im = slope * re if slope < 1 else slope * re * np.eye(dim)[0]
    nrm = rng.standard_normal(dim) + 1j * rng.standard_normal(dim)
    d = re + 1j * im
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    zero = torch.zeros((1, dim), dtype=torch.float64, device=cuda)
    one = torch.ones((1, 1, 1), dtype=torch.complex128, device=cuda)
    keep = np.abs((d * d).sum(1)) > 0.1 * (np.abs(d) ** 2).sum(1)     # r^2 not cancelled
    keep &= np.abs((kap * np.sqrt((d * d).sum(1))).imag) < 500.0
    slp, dlp = kernel(dim, ker, kap, d, nrm)
    for flag, ref in ((cf.SLP, slp), (cf.DLP, dlp)):
        got = cf.direct(dim, ker | flag, kap, zero, zero, t(re), t(im), one,
                        t(nrm.real[None]), t(nrm.imag[None])).cpu().numpy()[0]
        size = np.abs(ref) if flag == cf.DLP or (dim, ker) != (2, 0) else np.maximum(np.abs(ref), 1.0)
        if flag == cf.DLP:                                            # n.d cancels for some directions
            size = size * (np.abs(d) @ np.abs(nrm)) / np.abs(d @ nrm)
        err = np.abs(got - ref) / size / (1 + np.abs(kap * np.sqrt((d * d).sum(1))))
        assert err[keep].max() < 4e-15


@pytest.mark.parametrize("m,n", [(1, 1), (31, 33), (33, 31), (1, 129), (4097, 3), (127, 128), (128, 127), (700, 257)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_block_shapes(cuda, m, n, nrhs):
    """Every target gets every source once, whatever the remainders; 2D Laplace
    double layer plus single layer on points that coincide in part. Sums of at
    most 4,097 terms in two orders: 1e-12 of the sum of their moduli."""
    import torch

    import paper_2509_05458_gb300 as cf
    rng = np.random.default_rng(m * 1000 + n)
    src = rng.standard_normal((m, 2)) * (1 + 0.3j)
    trg = rng.standard_normal((n, 2)) * (1 + 0.3j)
    same = min(m, n) // 2
    trg[:same] = src[:same]
    nrm = rng.standard_normal((m, 2)) + 1j * rng.standard_normal((m, 2))
    dens = rng.standard_normal((nrhs, 2, m)) + 1j * rng.standard_normal((nrhs, 2, m))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    got = cf.direct(2, cf.LAPLACE | cf.SLP | cf.DLP, 0.0, t(src.real), t(src.imag), t(trg.real), t(trg.imag),
                    t(dens), t(nrm.real), t(nrm.imag)).cpu().numpy()
    d = trg[:, None, :] - src[None]
    r2 = (d * d).sum(2)
    skip = r2 == 0
    r2[skip] = 1.0
    ks, kd = np.log(r2) / 2, -(d * nrm[None]).sum(2) / r2
    ks[skip], kd[skip] = 0.0, 0.0
    ref = dens[:, 0] @ ks.T + dens[:, 1] @ kd.T
    size = np.abs(dens[:, 0]) @ np.abs(ks.T) + np.abs(dens[:, 1]) @ np.abs(kd.T) + 1e-300
    assert (np.abs(got - ref) / size).max() < 1e-12
