"""Autotuner of the block transforms' geometry and launch shapes per length.

For each length N it builds small variant libraries that contain only N,
each with one candidate factorisation N = R0 R1 R2 and one launch shape of
the passes (transforms per block, threads, resident blocks per SM), times
the three passes of a map whose padded size is N x N on the GPU, and keeps,
for the factorisation whose best passes sum lowest, the best shape of each
pass.  With several spectra per map (--nspec) it times the shapes of the
batched column pass (and its groups per block), against one single-spectrum
pass per spectrum, at the two best factorisations, and weighs maps of one
spectrum and of several together.  The result is written to
``tuned_plans.json`` beside this file (or to the file $LP_TUNE_CACHE names)
as the entry's "geo"; ``build.py`` uses it for every length it lists.

    python -m paper_1907_02891_gb300.tune --sizes 4704 [--quick] \
        [--map-side 4096 --psf 541 --nspec 1]

The passes are timed one by one, with events between them, which stops the
launch overlap between passes of a real map; the last step times whole maps
with the trigger of the next pass at block start and at block exit.

Needs nvcc and one GPU.  Each variant is timed in a fresh subprocess (the
variant libraries export the same symbols).
"""

from __future__ import annotations

import argparse
import concurrent.futures as cf
import hashlib
import json
import os
import subprocess
import sys
import time
from typing import Dict, List, Sequence, Tuple

from . import build as B

TUNE_DIR = os.path.join(B.OUT, "tune")
COMMON_SRCS = ("api.cu", "spectrum.cu", "noalloc.cu", "serve.cpp")
PASSES = ("p1_rows", "p2_cols", "p3_rows")


def _prod(p) -> int:
    r = 1
    for x in p:
        r *= x
    return r


def candidate_shapes(r: Sequence[int], limit: int, parked: bool = False) -> List[List[int]]:
    """Launch shapes [transforms per block, threads, resident blocks] of a
    factorisation, by the share of idle threads in their rounds and the
    resident threads per SM; parked: with a parked column beside the working
    set (the batched column pass)."""
    r0, r1, r2 = r
    n, g = _prod(r), B.lanes_for(r1, r2)
    out = []
    for nt in ((4, 8, 16) if n <= 256 else (1, 2, 4, 8) if n <= 1024 else (1, 2, 4) if n <= 2600 else
               (1, 2) if n <= 6200 else (1,)):
        smem = B.pass_smem(r, nt) + (8 * nt * n if parked else 0)
        if smem > B.SMEM_LIMIT:
            continue
        for w in range(1, 33):
            t = 32 * w
            if r0 == 1:
                if t % g or nt % (t // g):
                    continue
                waste = 1.0
            else:
                if not 8 <= n * nt / t <= 48:
                    continue
                u1, ub, gr = r1 * r2 * nt, r0 * nt, w * (32 // g)
                waste = (-(-u1 // t) * t / u1 + 2.0 * (-(-ub // gr) * gr / ub)) / 3
            for regs in (2 * max(r) + 14, 2 * max(r) + 38):
                regs = (regs + 7) // 8 * 8
                mb = max(1, min((228 * 1024) // (smem + 1024), 65536 // (t * regs), 16))
                out.append((waste * (1 + 300.0 / min(mb * t, 2048)), [nt, t, mb]))
    out.sort(key=lambda x: x[0])
    res: List[List[int]] = []
    for _, s in out:
        if s not in res:
            res.append(s)
    return res[:limit]


def _compile_common(jobs: int) -> List[str]:
    os.makedirs(os.path.join(TUNE_DIR, "common"), exist_ok=True)
    os.makedirs(B.OBJ, exist_ok=True)
    deps = max(os.path.getmtime(h) for h in B._headers())
    srcs = [os.path.join(B.CSRC, f) for f in COMMON_SRCS]
    with cf.ThreadPoolExecutor(jobs) as ex:
        return list(ex.map(lambda s: B._compile(s, deps), srcs))


def _variant_lib(n: int, plan: dict, common: List[str]) -> str:
    vid = hashlib.sha1(json.dumps([n, plan], sort_keys=True).encode()).hexdigest()[:12]
    d = os.path.join(TUNE_DIR, vid)
    lib = os.path.join(d, "liblp.so")
    if os.path.exists(lib):
        return lib
    os.makedirs(d, exist_ok=True)
    src, reg = os.path.join(d, f"size_{n}.cu"), os.path.join(d, "registry.cu")
    with open(src, "w") as fh:
        fh.write(B.size_tu(n, plan))
    with open(reg, "w") as fh:
        fh.write(B._REGISTRY_TU.format(decls=f"extern const SizeKernels kSize_{n};",
                                       ptrs=f"&kSize_{n}", count=1))
    objs = []
    for s in (src, reg):
        o = s[:-3] + ".o"
        cmd = ["nvcc", *B.ARCH, *B.NVCC_FLAGS, "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"),
               "-c", s, "-o", o]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed for variant {vid}:\n{res.stderr}")
        objs.append(o)
    res = subprocess.run(["nvcc", *B.ARCH, "-shared", "-o", lib, *common, *objs, "-lcudart"],
                         capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed for variant {vid}:\n{res.stderr}")
    return lib


_RUNNER = r"""
import json, sys, time
import numpy as np
import torch
sys.path.insert(0, {root!r})
import paper_1907_02891_gb300.lp as lp
lp.load_library({lib!r})
n, reps, side, psf, nspec = {n}, {reps}, {side}, {psf}, {nspec}
hk = psf if psf > 0 else min(541, max(3, (n // 8) | 1))
h = w = side if side > 0 else n - hk + 1
dev = torch.device("cuda", 0)
ctx = lp.lp_create(0)
g = np.random.default_rng(1)
L = torch.from_numpy(g.random((h, w), dtype=np.float32)).to(dev)
r = np.hypot(*np.meshgrid(np.arange(hk) - hk // 2, np.arange(hk) - hk // 2, indexing="ij"))
specs = [lp.lp_kernel_spectrum(ctx, torch.from_numpy((r * r + 0.1) ** -(1.0 + 0.25 * i)).to(dev),
                               pad_ny=n, pad_nx=n) for i in range(nspec)]
outs = [torch.empty_like(L) for _ in specs]
flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
# a length below the linear-convolution padding (the SAME crop's own one)
# maps in one tile through lp_map_tiled
mapf = lp.lp_map if min(h, w) + hk - 1 <= n else (lambda c, L, s, o: lp.lp_map_tiled(c, L, s, o))
for _ in range(5):
    mapf(ctx, L, specs, outs)
lp.lp_sync_status(ctx)
if {whole}:
    # whole maps, CUDA events around each (the passes overlap as in use)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(reps)]
    for a, b in ev:
        flush.zero_()
        a.record()
        mapf(ctx, L, specs, outs)
        b.record()
    torch.cuda.synchronize()
    print(json.dumps({{"map": sum(a.elapsed_time(b) for a, b in ev) / len(ev)}}))
    lp.lp_destroy(ctx)
    sys.exit(0)
lp.lp_set_pass_timing(ctx, True)
lp.lp_get_pass_timing(ctx)
for _ in range(reps):
    flush.zero_()
    mapf(ctx, L, specs, outs)
lp.lp_sync_status(ctx)
t = lp.lp_get_pass_timing(ctx)
print(json.dumps({{k: v[0] / max(1, v[1]) for k, v in t.items()}}))
lp.lp_destroy(ctx)
"""


def time_variant(lib: str, n: int, reps: int, side: int = 0, psf: int = 0, nspec: int = 1,
                 whole: bool = False) -> Dict[str, float]:
    """Mean ms per launch of each pass (pass events), or with whole the mean
    ms of whole maps ({"map": ms}), whose passes overlap as in use."""
    code = _RUNNER.format(root=B.ROOT, lib=lib, n=n, reps=reps, side=side, psf=psf, nspec=nspec,
                          whole="True" if whole else "False")
    res = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600)
    if res.returncode != 0:
        raise RuntimeError(f"timing failed for {lib}:\n{res.stderr[-2000:]}")
    return json.loads(res.stdout.strip().splitlines()[-1])


def tune_size(n: int, quick: bool, jobs: int, common: List[str], log, side: int = 0, psf: int = 0,
              nspec: int = 1) -> dict:
    base = B.plan_table()[n]
    reps = 100 if n <= 5200 else 20

    def run(plans, whole=False, ns=1):
        """[(plan, timing)] of the plans that build and launch."""
        def lib_or_error(p):
            try:
                return _variant_lib(n, p, common)
            except RuntimeError as e:
                return e
        t0 = time.time()
        with cf.ThreadPoolExecutor(jobs) as ex:
            libs = list(ex.map(lib_or_error, plans))
        log(f"N={n}: built {sum(isinstance(l, str) for l in libs)} of {len(libs)} variants in {time.time() - t0:.0f} s")
        got = []
        for p, lib in zip(plans, libs):
            try:
                if not isinstance(lib, str):
                    raise lib
                t = time_variant(lib, n, reps, side, psf, ns, whole)
            except Exception as e:  # a variant that does not build or launch (resources) is skipped
                log(f"  skip {p['geo']}: {str(e).strip().splitlines()[-1][:120]}")
                continue
            got.append((p, t))
            log(f"  {p['geo']['r']} {p['geo']['p1']} pm={p['geo']['pm']}x{p['geo']['grp']} packed={int(p['packed'])} "
                f"late={p.get('late')}: " + " ".join(f"{k}={v * 1e3:.1f}us" for k, v in t.items()))
        return got

    plans = []
    for r in B.candidate_geos(n)[:2 if quick else 5]:
        for s in candidate_shapes(r, 4 if quick else 8):
            plans.append(dict(base, packed=True, geo=dict(B.geo_plan(r), p1=s, p2=s, p3=s)))
    got = run(plans)
    if not got:
        raise RuntimeError(f"no variant of {n} ran")
    geos = []
    for r in {tuple(p["geo"]["r"]) for p, _ in got}:
        rs = [(p, t) for p, t in got if tuple(p["geo"]["r"]) == r]
        pick = [min(rs, key=lambda x, k=k: x[1][k]) for k in PASSES]
        total = sum(t[k] for k, (_, t) in zip(PASSES, pick))
        shapes = [p["geo"][k] for k, (p, _) in zip(("p1", "p2", "p3"), pick)]
        geos.append((total, dict(base, packed=True, geo=dict(B.geo_plan(r), p1=shapes[0], p2=shapes[1], p3=shapes[2]))))
    geos.sort(key=lambda x: x[0])
    scored = []
    # with several spectra: the two best factorisations (the second where it is
    # within 4 %), by the passes of a map of one spectrum plus 2 / nspec of
    # those of a map of nspec
    for total, out in geos[:2] if nspec > 1 else geos[:1]:
        if total > 1.04 * geos[0][0]:
            break
        score = total
        if nspec > 1:
            multi = [dict(out, batch=False)]
            for s in candidate_shapes(out["geo"]["r"], 4 if quick else 8, parked=True):
                for grp in (1, 2, 3):
                    if s[1] * grp <= 1024:
                        multi.append(dict(out, batch=True, geo=dict(out["geo"], pm=s, grp=grp)))
            out, t = min(run(multi, ns=nspec), key=lambda x: x[1]["p2_cols"])
            score = total + 2.0 / nspec * sum(t[k] for k in PASSES)
        scored.append((score, total, out))
    _, total, out = min(scored, key=lambda x: x[0])
    # packed FP32x2 arithmetic, and the trigger of the next pass: whole maps
    late = list(base.get("late", B.DEFAULT_LATE))
    whole = run([dict(out, packed=pk, late=l) for pk in (True, False) for l in (late, [0, 0, 0])], whole=True)
    pick = min(whole, key=lambda x: x[1]["map"])
    out = dict(pick[0], tuned_total_us=total * 1e3, tuned_map_us=pick[1]["map"] * 1e3)
    log(f"N={n}: chose {out['geo']} packed={out['packed']} late={out.get('late')} batch={out.get('batch')} "
        f"(passes {out['tuned_total_us']:.1f} us, map {out['tuned_map_us']:.1f} us)")
    return out


def main() -> None:
    ap = argparse.ArgumentParser()
    ap.add_argument("--sizes", type=int, nargs="+", required=True)
    ap.add_argument("--quick", action="store_true")
    ap.add_argument("--jobs", type=int, default=0)
    ap.add_argument("--out", default=B.tuned_json_path(),
                    help="plan file to update (default: $LP_TUNE_CACHE, else tuned_plans.json)")
    ap.add_argument("--log", default=None)
    ap.add_argument("--psf", type=int, default=0, help="PSF side of the timed maps (default min(541, N/8))")
    ap.add_argument("--nspec", type=int, default=1, help="spectra per timed map (one forward transform)")
    ap.add_argument("--map-side", type=int, default=0,
                    help="time maps of this side instead of N - PSF + 1, to compare "
                         "padded lengths for one workload")
    args = ap.parse_args()
    jobs = args.jobs or (os.cpu_count() or 1)
    logf = open(args.log, "a") if args.log else None

    def log(msg):
        print(msg, flush=True)
        if logf:
            logf.write(msg + "\n")
            logf.flush()

    for n in args.sizes:
        if n not in B.SIZES:
            raise SystemExit(f"{n} is not in the supported size list")
    common = _compile_common(jobs)
    table = {}
    if os.path.exists(args.out):
        with open(args.out) as fh:
            table = json.load(fh)
    for n in args.sizes:
        table[str(n)] = tune_size(n, args.quick, jobs, common, log, args.map_side, args.psf, args.nspec)
        table[str(n)]["tuned_on"] = {"map_side": args.map_side, "psf": args.psf, "nspec": args.nspec}
        with open(args.out, "w") as fh:
            json.dump(table, fh, indent=1, sort_keys=True)
    log(f"wrote {args.out}")


if __name__ == "__main__":
    main()
