"""FP64 pairs next to the cut of the principal root and logarithm: r^2 < 0 with an
imaginary part that is zero or far below FP32's range. The direct sum takes such pairs
(a plan refuses them). Zero, of whatever products it is the sum, is the upper side.

Against the kernels on r = +-i s from scipy's functions of a real argument, |kappa r| <= 1
(beyond, H = J + i Y cancels on the imaginary axis). The pair evaluation is good to 4e-15
(1 + |kappa r|) relative (tests/test_gpu_near64.py): 2e-14 with the reference's rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def kernels(dim, ker, kap, s, up):
    """K and K'/r at r = i s (up) or -i s."""
    from scipy.special import i0, i1, k0, k1
    r = 1j * s if up else -1j * s
    if dim == 2 and ker == 0:
        return np.log(s) + (0.5j if up else -0.5j) * np.pi, 1 / r ** 2
    if dim == 2:
        # H_0(i x) = -(2i/pi) K_0(x), H_1(i x) = -(2/pi) K_1(x); H_nu(-i x) = 2 J_nu(-i x)
        # - conj(H_nu(i x)), J_0(-i x) = I_0(x), J_1(-i x) = -i I_1(x)
        x = kap * s
        h0, h1 = -2j / np.pi * k0(x), -2 / np.pi * k1(x)
        if not up:
            h0, h1 = 2 * i0(x) - np.conj(h0), -2j * i1(x) - np.conj(h1)
        return h0, -kap * h1 / r
    if ker == 0:
        return 1 / r, -1 / r ** 3
    e = np.exp(1j * kap * r) / r
    return e, (1j * kap - 1 / r) * e / r


@pytest.mark.parametrize("dim,ker,kap", [(2, 0, 0.0), (2, 1, 2.0), (3, 0, 0.0), (3, 1, 2.0)])
@pytest.mark.parametrize("tiny,sign", [(0.0, 1), (0.0, -1), (1e-60, 1), (1e-60, -1)])
def test_side_of_the_cut(cuda, dim, ker, kap, tiny, sign):
    import torch

    import paper_2509_05458_gb300 as cf
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    # d = x - y: imaginary but for `tiny`; with sign < 0 every product Re d Im d is -0
    s = np.geomspace(0.02, 0.5, 40)
    u = np.arange(1.0, dim + 1)
    u /= np.linalg.norm(u)
    im = sign * s[:, None] * u
    re = np.full_like(im, tiny)
    zero = torch.zeros((1, dim), dtype=torch.float64, device=cuda)
    one = torch.ones((1, 1, 1), dtype=torch.complex128, device=cuda)
    nrm = np.cos(np.arange(dim)) + 1j * np.sin(np.arange(dim))
    k, dk = kernels(dim, ker, kap, s, tiny == 0.0 or sign > 0)
    nd = (re + 1j * im) @ nrm
    size = np.abs(dk)
    if (dim, ker) == (3, 1):            # i kappa - 1/r vanishes at r = -i/kappa
        size = (kap + 1 / s) * np.exp(-kap * s * (1 if tiny == 0.0 or sign > 0 else -1)) / s ** 2
    for flag, ref, size in ((cf.SLP, k, np.abs(k)), (cf.DLP, -dk * nd, size * np.abs(nd))):
        got = cf.direct(dim, ker | flag, kap, zero, zero, t(re), t(im), one, t(nrm.real[None]),
                        t(nrm.imag[None])).cpu().numpy()[0]
        assert (np.abs(got - ref) / size).max() < 2e-14
