"""The in-place block transforms of the FP32 passes, for every supported
length as column length: the batched pass over several spectra and the
Eq. (4) pass over several classes against single-spectrum maps (themselves
held to the oracle in test_lp_gpu.py), for real and complex spectra, in both
output modes; the FULL crop starts on an odd row of the circular result.

Tolerance: every result is an FP32 transform pair of the same exact values.
Each of its at most seven stages rounds to within about 2 eps (eps = 6e-8)
of the stage's norm, so two results differ by at most about 2 * 7 * 2 * 6e-8
< 2e-6 of the map's maximum; three classes add up three such results."""

import numpy as np
import pytest

from paper_1907_02891_gb300 import build as B

pytestmark = pytest.mark.gpu

TOL = 2e-6


@pytest.fixture(scope="module")
def ctx():
    from paper_1907_02891_gb300 import lp
    c = lp.lp_create(0)
    yield c
    lp.lp_destroy(c)


def _psf(rng, hk, wk, symmetric):
    K = rng.random((hk, wk)) + 0.1
    return (K + K[::-1, ::-1]) / 2 if symmetric else K


@pytest.mark.parametrize("n", B.SIZES)
def test_batched_and_classes_match_single_maps(ctx, n):
    import torch
    from paper_1907_02891_gb300 import lp
    rng = np.random.default_rng(n)
    hk, wk, nx = 7, 5, 96
    h, w = n - hk + 1, 37
    for symmetric in (True, False):
        Ks = [torch.from_numpy(_psf(rng, hk, wk, symmetric)).cuda() for _ in range(3)]
        spectra = [lp.lp_kernel_spectrum(ctx, K, pad_ny=n, pad_nx=nx) for K in Ks]
        Ls = [torch.from_numpy(rng.random((h, w), dtype=np.float32)).cuda() for _ in range(3)]
        for mode in (lp.LP_OUT_SAME, lp.LP_OUT_FULL):
            shape = lp.output_shape(h, w, hk, wk, mode)
            single = [[torch.empty(shape, device="cuda") for _ in spectra] for _ in Ls]
            for L, outs in zip(Ls, single):
                for s, o in zip(spectra, outs):
                    lp.lp_map(ctx, L, [s], [o], mode=mode)
            batched = [torch.full(shape, float("nan"), device="cuda") for _ in spectra]
            lp.lp_map(ctx, Ls[0], spectra, batched, mode=mode)
            classes = torch.full(shape, float("nan"), device="cuda")
            lp.lp_map_multiclass(ctx, Ls, spectra, classes, mode=mode)
            lp.lp_sync_status(ctx)
            for a, b in zip(batched, single[0]):
                assert (a - b).abs().max().item() <= TOL * b.abs().max().item()
            total = sum(single[i][i].double() for i in range(3))
            assert (classes.double() - total).abs().max().item() <= 3 * TOL * total.abs().max().item()
        for s in spectra:
            lp.lp_spectrum_release(ctx, s)


def test_plans_name_block_geometries():
    for n, p in B.plan_table().items():
        r0, r1, r2 = p["geo"]["r"]
        assert r0 * r1 * r2 == n and 1 <= max(r1, r2) <= 32 and r0 <= B.R0_MAX
        for key in ("p1", "p2", "p3", "pm"):
            assert p["geo"][key][-2] % 32 == 0 and p["geo"][key][-2] <= B.MAX_THREADS


@pytest.mark.parametrize("kind", ["radial", "point", "none"])
@pytest.mark.parametrize("ny,nx,hk,wk", [(45, 64, 45, 63), (96, 45, 1, 1), (360, 1120, 101, 1119), (4704, 210, 541, 7),
                                         (1536, 128, 1535, 3), (17280, 45, 801, 5), (64, 8820, 5, 601)])
def test_spectrum_build_of_each_symmetry(ctx, kind, ny, nx, hk, wk):
    """The folded FP64 build against numpy's FP64 transform, for PSFs that are
    mirror-symmetric, point-symmetric only, and neither.  Tolerance: one
    rounding to FP32 of the largest value, 2^-24 < 6e-8 of it, doubled."""
    import torch
    from paper_1907_02891_gb300 import lp
    rng = np.random.default_rng(ny + 7 * nx)
    K = rng.random((hk, wk)) + 0.01
    if kind != "none":
        K = (K + K[::-1, ::-1]) / 2
    if kind == "radial":
        K = (K + K[::-1]) / 2
    spec = lp.lp_kernel_spectrum(ctx, torch.from_numpy(np.ascontiguousarray(K)).cuda(), pad_ny=ny, pad_nx=nx)
    real = lp.lp_spectrum_info(spec)["is_real"]
    assert real == bool((K == K[::-1, ::-1]).all())
    got = torch.empty(nx // 2 + 1, ny, 1 if real else 2, device="cuda")
    lp.lp_spectrum_copy(spec, got)
    lp.lp_sync_status(ctx)
    lp.lp_spectrum_release(ctx, spec)
    P = np.zeros((ny, nx))
    P[:hk, :wk] = K
    S = np.fft.rfft2(np.roll(P, (-(hk // 2), -(wk // 2)), (0, 1))).T / (2.0 * ny * nx)
    g = got.double().cpu().numpy()
    diff = np.abs(g[..., 0] - S.real) if real else np.hypot(g[..., 0] - S.real, g[..., 1] - S.imag)
    assert diff.max() <= 1.2e-7 * np.abs(S).max()


@pytest.mark.parametrize("offset", [0, 1])
def test_spectrum_copy_takes_any_float_address(ctx, offset):
    """A complex spectrum to a destination of 4-byte alignment: the same values
    as to an aligned one, nothing before or behind them."""
    import torch
    from paper_1907_02891_gb300 import lp
    K = torch.rand(5, 7, dtype=torch.float64, device="cuda") + 0.01
    spec = lp.lp_kernel_spectrum(ctx, K, pad_ny=96, pad_nx=64)
    n = 33 * 96 * 2
    aligned = torch.empty(n, device="cuda")
    buf = torch.full((n + 4,), -7.0, device="cuda")
    lp.lp_spectrum_copy(spec, aligned)
    lp.lp_spectrum_copy(spec, buf[offset:offset + n])
    lp.lp_sync_status(ctx)
    lp.lp_spectrum_release(ctx, spec)
    assert torch.equal(buf[offset:offset + n], aligned)
    assert (buf[:offset] == -7).all() and (buf[offset + n:] == -7).all()


@pytest.mark.parametrize("classes,h", [(1, 90), (2, 91), (32, 1)])
def test_row_pass_of_several_classes(ctx, classes, h):
    """One launch of the forward row pass for all classes' maps, the most that
    the entry takes among them, against the sum of single maps.  Tolerance: a
    class's two results differ by TOL of its maximum at most, and no class's
    maximum is above the total's (all values are positive)."""
    import torch
    from paper_1907_02891_gb300 import lp
    rng = np.random.default_rng(classes)
    spectra, maps = [], []
    total = torch.zeros(h, 88, dtype=torch.float64, device="cuda")
    out = torch.empty(h, 88, device="cuda")
    for i in range(classes):
        K = torch.from_numpy(np.ascontiguousarray(_psf(rng, 7, 5, True))).cuda()
        spectra.append(lp.lp_kernel_spectrum(ctx, K, pad_ny=120, pad_nx=96))
        maps.append(torch.from_numpy(rng.random((h, 88), dtype=np.float32)).cuda())
        lp.lp_map(ctx, maps[i], [spectra[i]], [out])
        lp.lp_sync_status(ctx)
        total += out.double()
    lp.lp_map_multiclass(ctx, maps, spectra, out)
    lp.lp_sync_status(ctx)
    for s in spectra:
        lp.lp_spectrum_release(ctx, s)
    assert (out.double() - total).abs().max().item() <= classes * TOL * total.abs().max().item()
