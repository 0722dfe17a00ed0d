"""Coincident points whose zero coordinates differ in sign (the difference of -0 and
+0 is -0): x == y all the same, so the pair is skipped in every FP64 kernel and layer.

The reference is the same call with every zero positive. The other pairs' differences
then change in the signs of zeros alone, which move no term of r^2 by more than its
rounding: 1e-13 of the result's norm."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KERNELS = [(2, 0, 0.0), (2, 1, 3.0), (3, 0, 0.0), (3, 1, 3.0)]


def points(dim, n, seed):
    """Points on the last axis' zero plane (in 3D a third of them on that of the first
    coordinate too), real in the last coordinate, and their negative-zero twins."""
    rng = np.random.default_rng(seed)
    re = rng.uniform(-1, 1, (n, dim))
    re[:, -1] = 0.0
    if dim == 3:
        re[: n // 3, 0] = 0.0
    im = 0.3 * re
    neg = lambda a: np.where(a == 0.0, -0.0, a)
    return re, im, neg(re), neg(im)


def close(a, b):
    import torch
    assert torch.isfinite(torch.view_as_real(a)).all()
    assert float(torch.linalg.vector_norm(a - b)) <= 1e-13 * float(torch.linalg.vector_norm(b))


@pytest.mark.parametrize("dim,ker,kap", KERNELS)
@pytest.mark.parametrize("layers", ["s", "d", "sd"])
def test_signed_zeros(cuda, dim, ker, kap, layers):
    import torch

    import paper_2509_05458_gb300 as cf
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    flags = ker | (cf.SLP if "s" in layers else 0) | (cf.DLP if "d" in layers else 0)
    n, ncomp = 150, len(layers)
    re, im, nre, nim = points(dim, n, 10 * dim + ker)
    rng = np.random.default_rng(3)
    dens = t(rng.standard_normal((1, ncomp, n)) + 1j * rng.standard_normal((1, ncomp, n)))
    nrm = [t(rng.standard_normal((n, dim))) for _ in range(2)] if "d" in layers else [None, None]
    src = (t(re), t(im))
    for x, y in (((nre, nim), src), (src, (nre, nim))):       # (-0) - (+0) and (+0) - (-0)
        x, y = [tuple(t(a) if isinstance(a, np.ndarray) else a for a in p) for p in (x, y)]
        ref = cf.direct(dim, flags, kap, *src, *src, dens, *nrm)
        close(cf.direct(dim, flags, kap, *y, *x, dens, *nrm), ref)
        out = torch.empty_like(ref)
        cf.direct_noalloc(dim, flags, kap, *y, *x, dens, out, *nrm)
        close(out, ref)
    # a plan over the points and their twins: potential and gradient
    both = [np.concatenate(p) for p in ((re, nre), (im, nim))]
    plus = [a + 0.0 for a in both]
    d2 = torch.cat([dens, dens], 2)
    n2 = [torch.cat([a, a]) if a is not None else None for a in nrm]
    got = cf.plan(dim, flags, kap, 1e-9, *map(t, both), *n2, leaf_size=24).apply_grad(d2)
    ref = cf.plan(dim, flags, kap, 1e-9, *map(t, plus), *n2, leaf_size=24).apply_grad(d2)
    for a, b in zip(got, ref):
        close(a, b)
