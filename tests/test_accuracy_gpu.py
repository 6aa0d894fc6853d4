"""Error of the FP32 transforms against 64 bits at lengths whose butterflies
hold rounded constants (16th and 32nd turns, thirds, fifths, sevenths, ninths):
no larger than what the transforms that stood here before them left on the
same inputs (self-sorting chains in scalar arithmetic, with other factors at
most lengths).

The bounds are those transforms' own errors, measured on a GB300: the root
mean square, over 8 maps with one long side, of the error over the map's
maximum.  The same inputs give the same bits on every run."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1907_02891_gb300 import lp  # noqa: E402

BOUNDS = {  # length: (along columns, along rows)
    384: (2.3329e-09, 2.5202e-09), 768: (2.2426e-09, 2.4037e-09), 1024: (2.2448e-09, 2.3800e-09),
    1344: (1.4475e-09, 1.5762e-09), 1792: (1.5132e-09, 1.6150e-09), 2520: (1.5467e-09, 1.7266e-09),
    4608: (1.3908e-09, 1.5283e-09), 4704: (1.3696e-09, 1.4873e-09), 5040: (1.1828e-09, 1.3073e-09),
    7168: (1.0438e-09, 1.1310e-09), 8640: (1.0241e-09, 1.1312e-09), 8820: (1.2047e-09, 1.3470e-09),
    9216: (9.2923e-10, 1.0084e-09), 10752: (1.0471e-09, 1.1303e-09), 12288: (9.8063e-10, 1.0739e-09),
    13440: (7.7942e-10, 8.6611e-10), 16384: (1.0219e-09, 1.1084e-09), 17280: (9.3999e-10, 1.0398e-09),
}

PSF = 31


def _psf():
    y = 0.742 * (np.arange(PSF) - PSF // 2)
    r = np.hypot(y[:, None], y[None, :])
    return (r * r + 0.1) ** -1.25 * np.exp(-r / 80.0)


def _radiance(rng, h, w):
    return (np.exp(1.5 * rng.standard_normal((h, w))) * (rng.random((h, w)) < 0.05)).astype(np.float32)


def error(ctx, n, columns):
    """Along columns of length n (rows of 96), or along rows."""
    ny, nx = (n, 96) if columns else (96, n)
    h, w = ny - PSF + 1, nx - PSF + 1
    K = torch.from_numpy(_psf()).cuda()
    spec = lp.lp_kernel_spectrum(ctx, K, pad_ny=ny, pad_nx=nx)
    P = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    P[:PSF, :PSF] = K
    S = torch.fft.rfft2(torch.roll(P, (-(PSF // 2), -(PSF // 2)), (0, 1)))
    rng, total = np.random.default_rng(n), 0.0
    for _ in range(8):
        L = torch.from_numpy(_radiance(rng, h, w)).cuda()
        out = torch.empty(h, w, device="cuda")
        lp.lp_map(ctx, L, [spec], [out])
        want = torch.fft.irfft2(torch.fft.rfft2(L.double(), s=(ny, nx)) * S, s=(ny, nx))[:h, :w]
        total += ((out.double() - want) / want.max()).pow(2).mean().item()
    lp.lp_sync_status(ctx)
    lp.lp_spectrum_release(ctx, spec)
    return (total / 8) ** 0.5


@pytest.mark.parametrize("n", sorted(BOUNDS))
def test_error_is_no_larger_than_before(n):
    ctx = lp.lp_create(0)
    try:
        got = [error(ctx, n, columns) for columns in (True, False)]
        assert got[0] <= BOUNDS[n][0] and got[1] <= BOUNDS[n][1], got
    finally:
        lp.lp_destroy(ctx)
