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
