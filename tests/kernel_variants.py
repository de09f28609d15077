"""Kernel variants: the library built beside itself with other compile-time
choices of the simulation kernel and timed against it on the same workload, each
required to give bit-identical results (GPU only).

    python -m tests.kernel_variants FAMILY [--traces 64] [--reps 3] [--out FILE]

Family `occupancy`: 8, 7 or 6 resident 4-warp blocks per SM (the
register budget follows).  A variant is a list of nvcc flags for
hx_kernels.cu, each setting a macro that the source leaves to the build.
"""
from __future__ import annotations

import argparse
import json
import os
import shutil
import subprocess
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

CSRC = os.path.join(ROOT, "paper_2505_05286_gb300", "csrc")
OUT = os.path.join(ROOT, "paper_2505_05286_gb300", "_variants")
NVCC = ["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-lineinfo", "-std=c++17", "-Xcompiler",
        "-fPIC", "-I", os.path.join(ROOT, "include")]

VARIANTS = {
    "occupancy": {f"blocks{n}": [f"-DHX_SIM_MIN_BLOCKS(J)={n}"] for n in (8, 7, 6)},
}


def make_variant(name, flags):
    """Build the library into a .so of its own (extra nvcc flags for hx_kernels.cu)."""
    d = os.path.join(OUT, name)
    shutil.rmtree(d, ignore_errors=True)
    os.makedirs(d)
    objs = []
    for src in ("hx_kernels.cu", "hx_api.cu"):
        o = os.path.join(d, src.replace(".cu", ".o"))
        extra = list(flags) if src == "hx_kernels.cu" else []
        subprocess.check_call(NVCC + ["-I", CSRC, *extra, "-c", os.path.join(CSRC, src), "-o", o])
        objs.append(o)
    lib = os.path.join(d, "libhxsim.so")
    subprocess.check_call(NVCC[:3] + ["-shared", "-o", lib] + objs)
    return lib


def time_lib(lib_path, wl, reps, **sim_options):
    """Median simulation-kernel milliseconds over `reps` runs after one
    warm-up, and the results, with the library at lib_path (Sim options
    passed through)."""
    from paper_2505_05286_gb300 import hxsim as H
    saved = H._lib
    H._lib = H.load(lib_path)
    try:
        sim = H.Sim(wl.traces, wl.cluster, wl.grid, timing=True, **sim_options)
        sim.run()
        ms = []
        for _ in range(reps):
            sim.run()
            ms.append(sim.timings()[1])
        r = sim.results()
        sim.close()
    finally:
        H._lib = saved
    return float(np.median(ms)), ms, r


def main(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("family", choices=sorted(VARIANTS))
    ap.add_argument("--traces", type=int, default=64)
    ap.add_argument("--reps", type=int, default=3)
    ap.add_argument("--out", default=None)
    args = ap.parse_args(argv)
    import torch

    from paper_2505_05286_gb300 import build as B
    from paper_2505_05286_gb300 import hxsim as H
    from paper_2505_05286_gb300 import workloads as W
    B.build()
    torch.cuda.set_device(0)
    wl = W.make_workload(4, n_traces=args.traces)
    fields = ("p95_us", "makespan_us", "events", "digest", "slo_met", "n_done", "status")
    base_ms, base_all, base = time_lib(H.LIB_PATH, wl, args.reps)
    out = {"workload": f"{wl.name} cut to {args.traces} traces", "sims": wl.n_sims, "library_ms": base_ms,
           "library_all_ms": base_all, "variants": {}}
    print("library", base_ms, base_all, flush=True)
    for name, flags in VARIANTS[args.family].items():
        ms, all_ms, r = time_lib(make_variant(name, flags), wl, args.reps)
        same = all(np.array_equal(r[f], base[f]) for f in fields)
        out["variants"][name] = {"ms": ms, "all_ms": all_ms, "same_results": same, "speedup": base_ms / ms}
        print(name, ms, all_ms, same, round(base_ms / ms, 4), flush=True)
    again, again_all, _ = time_lib(H.LIB_PATH, wl, args.reps)
    out["library_again_ms"] = again
    print("library again", again, again_all, flush=True)
    if args.out:
        with open(args.out, "w") as f:
            json.dump(out, f, indent=1)
    return 0 if all(v["same_results"] for v in out["variants"].values()) else 1


if __name__ == "__main__":
    sys.exit(main())
