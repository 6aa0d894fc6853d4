"""Columns parked in global memory, several side by side: the batched and the
Eq. (4) column passes of a plan that no stored one is (eight columns per
block), in the bounds-checked build, against maps of one spectrum each.  The
49 columns of the transform leave one in the last block, so the parked area
has to be whole blocks long.

Tolerance as in test_block_passes_gpu: two FP32 transform pairs of the same
values differ by less than 2e-6 of the map's maximum, a sum of three by three
times that."""

import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

from paper_1907_02891_gb300 import build  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N, SIZES = 2250, (96, 2250)

_CHILD = r"""
import sys
sys.path.insert(0, {root!r})
import numpy as np, torch
from paper_1907_02891_gb300 import lp
N, TOL = {n}, 2e-6
ctx = lp.lp_create(0)
rng = np.random.default_rng(1)
for sym in (True, False):
    Ks = [rng.random((7, 5)) + 0.1 for _ in range(3)]
    Ks = [torch.from_numpy(np.ascontiguousarray((K + K[::-1, ::-1]) / 2 if sym else K)).cuda() for K in Ks]
    sp = [lp.lp_kernel_spectrum(ctx, K, pad_ny=N, pad_nx=96) for K in Ks]
    h, w = N - 6, 92
    Ls = [torch.from_numpy(rng.random((h, w), dtype=np.float32)).cuda() for _ in range(3)]
    one = [[torch.empty(h, w, device="cuda") for _ in sp] for _ in Ls]
    for L, outs in zip(Ls, one):
        for s, o in zip(sp, outs):
            lp.lp_map(ctx, L, [s], [o])
    many = [torch.full((h, w), float("nan"), device="cuda") for _ in sp]
    lp.lp_map(ctx, Ls[0], sp, many)
    total = torch.full((h, w), float("nan"), device="cuda")
    lp.lp_map_multiclass(ctx, Ls, sp, total)
    lp.lp_sync_status(ctx)
    for a, b in zip(many, one[0]):
        assert (a - b).abs().max().item() <= TOL * b.abs().max().item()
    want = sum(one[i][i].double() for i in range(3))
    assert (total.double() - want).abs().max().item() <= 3 * TOL * want.abs().max().item()
print("parked bytes", lp.lp_map_workspace_bytes(h, w, N, 96, 7, 5, 3) - lp.lp_map_workspace_bytes(h, w, N, 96, 7, 5, 1))
lp.lp_destroy(ctx)
"""


def test_parked_in_global_memory_eight_columns_per_block(tmp_path, monkeypatch):
    plan = dict(build.plan_table()[N], batch=True)
    plan["geo"] = dict(plan["geo"], r=[10, 15, 15], pm=[8, 480, 1], grp=1)
    path = tmp_path / "plans.json"
    path.write_text(json.dumps({str(N): plan}))
    monkeypatch.setenv("LP_TUNE_CACHE", str(path))
    build.build(debug=True, sizes=SIZES)
    r = subprocess.run([sys.executable, "-c", _CHILD.format(root=ROOT, n=N)], capture_output=True, text=True,
                       env=dict(os.environ, LP_DEBUG="1"), timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    # two more U blocks (52 columns) and the parked set (56 columns), not in shared memory
    assert r.stdout.split()[-1] == str(8 * (2 * 52 * 2244 + 56 * N) + 256)
