"""Build liblp.so (sm_103a) in-tree.

The FP32 FFT kernels are templates over the radix sequence of each supported
transform length.  This script picks one radix sequence per length (the
plan table below), writes one small translation unit per length into
``_build/gen``, and compiles everything with nvcc in parallel:

    python -m paper_1907_02891_gb300.build          # or build() from Python

Output: ``paper_1907_02891_gb300/_build/liblp.so``.
"""

from __future__ import annotations

import concurrent.futures as cf
import hashlib
import json
import os
import shutil
import subprocess
import sys
from typing import Dict, List, Sequence, Tuple

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
GEN = os.path.join(OUT, "gen")
OBJ = os.path.join(OUT, "obj")
LIB = os.path.join(OUT, "liblp.so")
# debug build (LP_DEBUG=1: the passes check every work unit's extents in
# every buffer first and report a miss in the device status word); a
# library of its own, loaded by lp.py when $LP_DEBUG is set
DEBUG_OBJ = os.path.join(OUT, "debug", "obj")
DEBUG_LIB = os.path.join(OUT, "debug", "liblp.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "--expt-relaxed-constexpr", "-lineinfo",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-O2"]

# radices the in-register DFTs are instantiated for (7-smooth, <= 32)
RADICES = (2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 15, 16, 18, 20, 21, 24, 25, 27, 28, 30, 32)
MAX_THREADS = 1024
# trigger of the next pass at block exit for the forward row pass and the
# one-spectrum column pass; the inverse row pass triggers at block start.
# Whole maps, against all three at block start: 15.3 / 18.3 us at 1260, 127.1 /
# 130.9 at 4704, 555 / 558 at 8820, 2378 / 2387 at 17280; 480 equal
DEFAULT_LATE = [1, 1, 0]
SMEM_LIMIT = 227 * 1024

# Supported transform lengths.  Every length is 7-smooth; the list covers
# the workload sizes (360, 480, 720, 1260, 2250, 4320, 4704, 8400, 8820,
# 17280; 4608 = 4096 + 512 for the 4096^2 map's SAME crop with a 541^2 PSF
# in one tile), powers of two, and a ladder in between.
SIZES = (
    45, 64, 96, 100, 120, 128, 160, 192, 210, 240, 256, 288, 320, 360, 384, 420, 480, 512,
    560, 640, 720, 768, 840, 960, 1024, 1120, 1260, 1344, 1536, 1680, 1792, 2048, 2250, 2520,
    2688, 3072, 3360, 3584, 4096, 4320, 4608, 4704, 4800, 4860, 5040, 5120, 5376, 6144, 6720, 7168,
    8192, 8400, 8640, 8820, 9000, 9216,
    10080, 10752, 12288, 13440, 15360, 16384, 17280,
)


def factorizations(n: int, max_stages: int = 4) -> List[Tuple[int, ...]]:
    out: List[Tuple[int, ...]] = []

    def rec(rem: int, start: int, cur: List[int]) -> None:
        if rem == 1:
            out.append(tuple(cur))
            return
        if len(cur) == max_stages:
            return
        for i in range(start, len(RADICES)):
            r = RADICES[i]
            if rem % r == 0:
                rec(rem // r, i, cur + [r])

    rec(n, 0, [])
    return out


def threads_for(n: int, radices: Sequence[int]) -> int:
    return (n // min(radices) + 31) // 32 * 32


def choose_plan(n: int) -> Tuple[int, ...]:
    """Radices of the tensor-core column pass: fewest stages; then the
    smallest largest radix (register pressure); then the largest smallest
    radix (fewer threads); descending."""
    best = None
    for f in factorizations(n):
        if threads_for(n, f) > MAX_THREADS:
            continue
        key = (len(f), max(f), -min(f))
        if best is None or key < best[0]:
            best = (key, f)
    if best is None:
        raise ValueError(f"no radix plan for {n}")
    return tuple(sorted(best[1], reverse=True))


# ---------------------------------------------------------------------------
# Geometry of the FP32 passes: N = R0 R1 R2, the R1 R2-point sub-transforms on
# groups of 8, 16 or 32 lanes, R0 of them per transform (R0 = 1 for the lengths
# one group holds).
# ---------------------------------------------------------------------------
_FACTOR_COST = {2: 2.0, 3: 5.0, 5: 7.0, 7: 10.0}   # operations per point of one prime factor
R0_MAX = 42


def _dft_cost(r: int) -> float:
    c = 7.0   # the exchange around the butterfly
    for p in (2, 3, 5, 7):
        while r % p == 0:
            c += _FACTOR_COST[p]
            r //= p
    return c


def lanes_for(r1: int, r2: int) -> int:
    m = max(r1, r2)
    return 8 if m <= 8 else 16 if m <= 16 else 32


def candidate_geos(n: int) -> List[Tuple[int, int, int]]:
    """Factors (R0, R1, R2) by estimated cost: operations per point of each
    stage, over the share of the lanes it keeps busy (stage 2 runs on R2 of
    the group's lanes, stage 3 on R1)."""
    out = []
    for r1 in range(2, 33):
        for r2 in range(2, 33):
            if n % (r1 * r2):
                continue
            r0 = n // (r1 * r2)
            if r0 > R0_MAX or (r0 == 1 and n > 1024) or (r0 > 1 and n <= 1024):
                continue
            g = lanes_for(r1, r2)
            cost = _dft_cost(r1) * g / r2 + _dft_cost(r2) * g / r1
            if r0 > 1:
                cost += _dft_cost(r0) + (0 if r0 <= 21 else 3 if r0 <= 32 else 8)
            cost += 1.0 * (max(r1, r2) > 24) + 0.5 * (r2 % 2)
            out.append((round(cost, 6), abs(r1 - r2), r2, (r0, r1, r2)))
    if not out:
        raise ValueError(f"no block geometry for {n}")
    return [x[-1] for x in sorted(out)]


def choose_geo(n: int) -> Tuple[int, int, int]:
    return candidate_geos(n)[0]


def layout_elems(r: Sequence[int]) -> int:
    """Complex elements of shared memory of one transform (Lay in fft_core.cuh)."""
    r0, r1, r2 = r
    vec = r2 % 2 == 0
    s1 = r2 if not vec or (r2 // 2) % 2 else r2 + 2
    s0 = r1 * s1
    s0 = (s0 | 1) if not vec else s0 if (s0 // 2) % 2 else s0 + 2
    return (r0 * s0 + 7) // 16 * 16 + 8


def pass_smem(r: Sequence[int], nt: int) -> int:
    """Shared-memory bytes of a pass with nt transforms per block (PassCfg)."""
    r0, r1, _ = r
    w1 = (r0 * ((r1 + 1) // 2 * 2) + 7) // 8 * 8 if r0 > 1 else 0
    return 8 * (w1 + nt * layout_elems(r))


def pass_shape(r: Sequence[int], nt: int, extra: int = 0) -> List[int]:
    """[transforms per block, threads, resident blocks per SM] of one pass:
    the thread count whose rounds waste least among those with 12 to 40
    points per thread; resident blocks by shared memory (extra: bytes beside
    the working set) and by the registers the largest radix needs."""
    r0, r1, r2 = r
    n, g = r0 * r1 * r2, lanes_for(r1, r2)
    if r0 == 1:
        th = max(32, min(128, nt * g))
        nt = th // g
    else:
        best = None
        for w in range(1, 25):
            t = 32 * w
            if not 12 <= n * nt / t <= 36:
                continue
            u1, ub, gr = r1 * r2 * nt, r0 * nt, w * (32 // g)
            waste = -(-u1 // t) * t / u1 + 2.0 * (-(-ub // gr) * gr / ub)
            key = (round(waste, 3) + (0.4 if t > 512 else 0.0), -w)
            if best is None or key < best[0]:
                best = (key, t)
        th = best[1]
    smem = pass_smem(r, nt) + extra
    regs = max(64, 2 * max(r) + 32)
    by_smem = (228 * 1024) // (smem + 1024)
    by_regs = 65536 // (th * (regs + 7) // 8 * 8)
    return [nt, th, max(1, min(by_smem, by_regs, 16))]


def geo_plan(r: Sequence[int]) -> dict:
    """Pass shapes of a geometry before any measurement."""
    n = r[0] * r[1] * r[2]
    two = 8 if r[0] == 1 else 2 if n <= 5120 else 1
    pm_nt = 4 if r[0] == 1 else 2 if n <= 2560 else 1
    return dict(r=list(r), p1=pass_shape(r, two), p2=pass_shape(r, two), p3=pass_shape(r, two),
                pm=pass_shape(r, pm_nt, 8 * pm_nt * n), grp=2 if n > 5120 else 1)


TUNED_JSON = os.path.join(HERE, "tuned_plans.json")


def tuned_json_path() -> str:
    """The measured plans: the file named by $LP_TUNE_CACHE when set (same
    form, e.g. plans re-measured on another GPU), else tuned_plans.json
    beside this file."""
    return os.environ.get("LP_TUNE_CACHE") or TUNED_JSON


def plan_table_entry(n: int) -> dict:
    """Heuristic plan of one length (used when the autotuner has not
    measured it).  `radices` and `threads` are the tensor-core column pass's;
    `geo` is the FP32 passes'.  upb, minb, pf and db are fields of the plan
    files' form that no kernel reads."""
    r = choose_plan(n)
    return dict(radices=list(r), threads=threads_for(n, r), upb=[1] * 3, minb=[1] * 3, pf=[1] * 3, db=[0] * 3,
                batch=True, geo=geo_plan(choose_geo(n)))


def plan_table() -> Dict[int, dict]:
    """Plan of every supported length: the autotuner's measured choice from
    tuned_plans.json where there is one, the heuristic otherwise (a plan
    without a geometry gets the heuristic one)."""
    tuned = {}
    path = tuned_json_path()
    if os.path.exists(path):
        with open(path) as fh:
            tuned = json.load(fh)
    table = {}
    for n in SIZES:
        e = plan_table_entry(n)
        t = tuned.get(str(n))
        if t:
            e.update(radices=list(t["radices"]), threads=threads_for(n, t["radices"]),
                     upb=list(t["upb"]), minb=list(t["minb"]), pf=list(t.get("pf", [1, 1, 1])),
                     db=list(t.get("db", [0, 0, 0])), batch=bool(t.get("batch", True)),
                     packed=bool(t.get("packed", False)), late=list(t.get("late", DEFAULT_LATE)))
            if "geo" in t:
                e["geo"] = dict(t["geo"])
        table[n] = e
    return table


_SIZE_TU = """// generated by paper_1907_02891_gb300/build.py -- one supported FFT length
// packed FP32x2 complex arithmetic in this length's DFTs
#define LP_PACKED_FP32 {packed}
#include "conv_kernels.cuh"
#include "lp_internal.h"
#include "tc_kernels.cuh"

namespace lpk {{
namespace {{
constexpr int kN = {n};
using Ge = Geo<kN, {geo}>;
// shape of each pass: transforms per block, threads, resident blocks
using C1 = PassCfg<Ge, {p1}, {late1}>;
using C2 = PassCfg<Ge, {p2}, {late2}>;
using C3 = PassCfg<Ge, {p3}, {late3}>;
using CM = PassCfg<Ge, {pm}, {late2}>;   // several spectra or classes
// the passes over several spectra or classes keep one parked column (set)
// beside their working sets: in shared memory where that fits, else in
// global memory; kGrp groups share the parked column
constexpr int kMaxSmem = 227 * 1024;
constexpr int kParkB = 8 * CM::NT * kN;
constexpr bool kParkG = kParkB + CM::SMEM > kMaxSmem;
constexpr int kSmemG = kParkB + CM::SMEM + ({grp} - 1) * 8 * CM::WORK;
constexpr int kGrp = !kParkG && kSmemG <= kMaxSmem && CM::TH * {grp} <= 1024 ? {grp} : 1;
constexpr int kSmemM = kGrp > 1 ? kSmemG : (kParkG ? 0 : kParkB) + CM::SMEM;
constexpr int kSmemC = (kParkG ? 0 : kParkB) + CM::SMEM;
// several spectra: the batched column kernel (one forward transform, one
// product + inverse per spectrum) or one single-spectrum pass per spectrum
constexpr bool kBatch = {batch};
// split-precision tensor-core column pass (0 shared bytes: not available)
using P = Plan<kN, Seq<{seq}>>;
using TP = TcPlan<P, kN>;
constexpr bool kTC = TP::FITS;
constexpr int kTcSmem = kTC ? TP::SMEM_BYTES : 0;

template <class K>
cudaError_t attr(K k, int bytes)
{{
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}}

cudaError_t set_attrs()
{{
    cudaError_t e;
    if ((e = attr(p1_rows<C1>, C1::SMEM)) != cudaSuccess) return e;
    if ((e = attr(p2_cols<C2, true>, C2::SMEM)) != cudaSuccess) return e;
    if ((e = attr(p2_cols<C2, false>, C2::SMEM)) != cudaSuccess) return e;
    if ((e = attr(p2_cols_multi<CM, kGrp, kParkG, true>, kSmemM)) != cudaSuccess) return e;
    if ((e = attr(p2_cols_multi<CM, kGrp, kParkG, false>, kSmemM)) != cudaSuccess) return e;
    if ((e = attr(p2_multiclass<CM, kParkG, true>, kSmemC)) != cudaSuccess) return e;
    if ((e = attr(p2_multiclass<CM, kParkG, false>, kSmemC)) != cudaSuccess) return e;
    if constexpr (kTC) {{
        if ((e = attr(p2_cols_tc<P, kN, true>, kTcSmem)) != cudaSuccess) return e;
        if ((e = attr(p2_cols_tc<P, kN, false>, kTcSmem)) != cudaSuccess) return e;
    }}
    return attr(p3_rows<C3>, C3::SMEM);
}}

cudaError_t p1(const P1Args& a, cudaStream_t s)
{{
    return launch_pdl(p1_rows<C1>, dim3((a.npairs - a.pair0 + C1::NT - 1) / C1::NT, a.nmaps), dim3(C1::TH), C1::SMEM, s, a);
}}

cudaError_t p2(const P2Args& a, bool kreal, cudaStream_t s)
{{
    if (a.nspec == 1) {{
        const dim3 g((a.ncols + C2::NT - 1) / C2::NT);
        return kreal ? launch_pdl(p2_cols<C2, true>, g, dim3(C2::TH), C2::SMEM, s, a)
                     : launch_pdl(p2_cols<C2, false>, g, dim3(C2::TH), C2::SMEM, s, a);
    }}
    if (kBatch && (!kParkG || a.park)) {{
        const dim3 g((a.ncols + CM::NT - 1) / CM::NT);
        return kreal ? launch_pdl(p2_cols_multi<CM, kGrp, kParkG, true>, g, dim3(CM::TH * kGrp), kSmemM, s, a)
                     : launch_pdl(p2_cols_multi<CM, kGrp, kParkG, false>, g, dim3(CM::TH * kGrp), kSmemM, s, a);
    }}
    // one single-spectrum pass per spectrum (the plan measured this faster)
    for (int i = 0; i < a.nspec; ++i) {{
        P2Args b = a;
        b.K[0] = a.K[i];
        b.nspec = 1;
        b.U = a.U + (long long)i * a.specU;
        b.u_elems = a.u_elems - (long long)i * a.specU;
        cudaError_t e = p2(b, kreal, s);
        if (e != cudaSuccess) return e;
    }}
    return cudaSuccess;
}}

cudaError_t p2m(const P2MArgs& a, bool kreal, cudaStream_t s)
{{
    const dim3 g((a.a.ncols + CM::NT - 1) / CM::NT);
    return kreal ? launch_pdl(p2_multiclass<CM, kParkG, true>, g, dim3(CM::TH), kSmemC, s, a)
                 : launch_pdl(p2_multiclass<CM, kParkG, false>, g, dim3(CM::TH), kSmemC, s, a);
}}

// persistent grid of the tensor-core column pass: resident blocks per SM
// (registers, shared memory, threads, TMEM columns) times the SMs, computed
// once, for the device of the first launch (a different GPU model in the
// same process would only get a less fitting grid, never a wrong result)
template <bool KREAL>
int tc_grid(int ncols)
{{
    static int cap = 0;
    if (cap == 0) {{
        int dev = 0, sms = 0, smem_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
        cudaFuncAttributes fa{{}};
        cudaFuncGetAttributes(&fa, p2_cols_tc<P, kN, KREAL>);
        const int warps = TP::THREADS / 32;
        const int regs_warp = (fa.numRegs * 32 + 255) / 256 * 256;
        int occ = regs_warp > 0 ? 65536 / (regs_warp * warps) : 1;
        const int by_smem = smem_sm / (kTcSmem + 1024);
        const int by_thr = 2048 / TP::THREADS;
        const int by_tmem = 512 / TP::TMEM_COLS;
        occ = occ < by_smem ? occ : by_smem;
        occ = occ < by_thr ? occ : by_thr;
        occ = occ < by_tmem ? occ : by_tmem;
        cap = (occ < 1 ? 1 : occ) * sms;
    }}
    return ncols < cap ? ncols : cap;
}}

cudaError_t p2tc(const P2TcArgs& a, bool kreal, cudaStream_t s)
{{
    if constexpr (kTC) {{
        return kreal ? launch_pdl(p2_cols_tc<P, kN, true>, dim3(tc_grid<true>(a.a.ncols)), dim3(TP::THREADS), kTcSmem, s, a)
                     : launch_pdl(p2_cols_tc<P, kN, false>, dim3(tc_grid<false>(a.a.ncols)), dim3(TP::THREADS), kTcSmem, s, a);
    }} else {{
        return cudaErrorNotSupported;
    }}
}}

cudaError_t p3(const P3Args& a, int nspec, cudaStream_t s)
{{
    return launch_pdl(p3_rows<C3>, dim3((a.npairs - a.pair0 + C3::NT - 1) / C3::NT, nspec), dim3(C3::TH), C3::SMEM, s, a);
}}
}}  // namespace

extern const SizeKernels kSize_{n} = {{kN, {{{geo}}}, Ge::VK, {ns}, {{{rad6}}}, kBatch ? 1 : 0, kParkG ? 1 : 0, kParkG ? 1 : 0, CM::NT,
                                       set_attrs, p1, p2, p2m, p3,
                                       kTC ? TP::THREADS : 0, kTcSmem, p2tc}};
}}  // namespace lpk
"""

_REGISTRY_TU = """// generated by paper_1907_02891_gb300/build.py -- table of supported lengths
#include "lp_internal.h"

namespace lpk {{
{decls}
const SizeKernels* const kAllSizes[] = {{{ptrs}}};
const int kNumSizes = {count};
}}  // namespace lpk
"""


def _b(x) -> str:
    return "true" if x else "false"


def _write_if_changed(path: str, text: str) -> None:
    if os.path.exists(path):
        with open(path) as fh:
            if fh.read() == text:
                return
    with open(path, "w") as fh:
        fh.write(text)


def size_tu(n: int, p: dict) -> str:
    """Translation unit of one length with plan p."""
    r, g = list(p["radices"]), p["geo"]
    late = p.get("late", DEFAULT_LATE)
    return _SIZE_TU.format(n=n, seq=", ".join(map(str, r)), ns=len(r), rad6=", ".join(map(str, r + [0] * (6 - len(r)))),
                           geo=", ".join(map(str, g["r"])), grp=g["grp"],
                           **{k: ", ".join(map(str, g[k])) for k in ("p1", "p2", "p3", "pm")},
                           batch=_b(p.get("batch", True)), packed=int(bool(p.get("packed", False))),
                           late1=_b(late[0]), late2=_b(late[1]), late3=_b(late[2]))


def generate(sizes: Sequence[int] = ()) -> List[str]:
    """Write one translation unit per supported length (all, or `sizes`)
    and the registry of the lengths written; returns their paths.  A
    subset goes to its own directory, so that it never replaces the
    registry of the full build."""
    table = plan_table()
    gen = GEN
    if sizes:
        table = {n: table[n] for n in sorted(set(sizes))}
        gen = os.path.join(OUT, "gen_" + "_".join(map(str, table)))
    os.makedirs(gen, exist_ok=True)
    files = []
    for n, p in table.items():
        text = size_tu(n, p)
        path = os.path.join(gen, f"size_{n}.cu")
        _write_if_changed(path, text)
        files.append(path)
    decls = "\n".join(f"extern const SizeKernels kSize_{n};" for n in table)
    ptrs = ", ".join(f"&kSize_{n}" for n in table)
    path = os.path.join(gen, "registry.cu")
    _write_if_changed(path, _REGISTRY_TU.format(decls=decls, ptrs=ptrs, count=len(table)))
    files.append(path)
    return files


def _headers() -> List[str]:
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    hs.append(os.path.join(ROOT, "include", "lp.h"))
    return hs


def _compile(src: str, deps_mtime: float, debug: bool = False) -> str:
    name = os.path.splitext(os.path.basename(src))[0]
    digest = hashlib.sha1(src.encode()).hexdigest()[:8]
    obj = os.path.join(DEBUG_OBJ if debug else OBJ, f"{name}_{digest}.o")
    if os.path.exists(obj) and os.path.getmtime(obj) >= max(os.path.getmtime(src), deps_mtime):
        return obj
    cmd = ["nvcc", *ARCH, *NVCC_FLAGS, *(["-DLP_DEBUG=1"] if debug else []), "-I", CSRC,
           "-I", os.path.join(ROOT, "include"), "-c", src, "-o", obj + ".tmp"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    os.replace(obj + ".tmp", obj)
    return obj


def build(jobs: int = 0, verbose: bool = False, debug: bool = False, sizes: Sequence[int] = ()) -> str:
    """Compile every CUDA/C++ source of the library for sm_103a and link
    liblp.so (with debug, the bounds-checked library DEBUG_LIB, optionally
    with only the FFT lengths `sizes`).  Returns the library path."""
    if sizes and not debug:
        raise ValueError("a subset of lengths is for the debug build only")
    if shutil.which("nvcc") is None:
        raise RuntimeError("nvcc not found on PATH")
    obj_dir, lib = (DEBUG_OBJ, DEBUG_LIB) if debug else (OBJ, LIB)
    os.makedirs(obj_dir, exist_ok=True)
    gen = generate(sizes)
    srcs = [os.path.join(CSRC, f) for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cpp"))]
    srcs += gen
    deps = max(os.path.getmtime(h) for h in _headers() + [os.path.abspath(__file__)])
    jobs = jobs or max(1, os.cpu_count() or 1)
    with cf.ThreadPoolExecutor(jobs) as ex:
        objs = list(ex.map(lambda s: _compile(s, deps, debug), srcs))
    # relink when an object is newer or the set of objects differs (a debug
    # build of another subset of lengths)
    manifest = lib + ".objs"
    listed = open(manifest).read() if os.path.exists(manifest) else ""
    if (not os.path.exists(lib) or listed != "\n".join(objs) or
            os.path.getmtime(lib) < max(os.path.getmtime(o) for o in objs)):
        tmp = lib + f".tmp{os.getpid()}"
        cmd = ["nvcc", *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
        os.replace(tmp, lib)
        with open(manifest, "w") as fh:
            fh.write("\n".join(objs))
    if verbose:
        print(lib)
    return lib


if __name__ == "__main__":
    build(verbose=True, debug="--debug" in sys.argv[1:])
    sys.exit(0)
