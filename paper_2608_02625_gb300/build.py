"""Builds libdlmrefine.so, libdlmsynth.so and the binding's native marshalling
(_marshal.so) in-tree for sm_103a (GB300).

    python -m paper_2608_02625_gb300.build [--force] [--verbose] [--check-bounds --out DIR]

Each .cu is compiled to an object in parallel (nvcc, one -gencode), then the
objects are linked into position-independent shared libraries with the CUDA
runtime linked statically, so loading the library needs no libcudart on the
library path. The driver API entry used for TMA descriptors is resolved at
run time through the runtime (no -lcuda).

--check-bounds compiles with DLM_CHECK_BOUNDS, which makes the kernels check
their inputs' value contracts and report violations in the device error word
(DLM_DEVERR_INPUT); such a build goes to its own object directory and, with
--out, to another directory than the package's.
"""
from __future__ import annotations

import argparse
import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]

LIBS = {
    "libdlmrefine.so": ["dlm_api.cu", "attn_tc.cu", "attn_f32.cu", "vocab.cu", "update.cu", "loop.cu", "lmhead.cu",
                        "selftest.cu"],
    "libdlmsynth.so": ["synth.cu"],
}
# The Python binding's marshalling: host code against torch's headers, beside the library it calls.
MARSHAL, MARSHAL_SRC = "_marshal.so", "marshal.cpp"
HEADERS = ["dlm_common.cuh", "dlm_internal.h", "update_impl.cuh"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _flags(verbose: bool, check_bounds: bool = False):
    f = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-O2", "-I", INCLUDE,
                "--expt-relaxed-constexpr"]
    if check_bounds:
        f += ["-DDLM_CHECK_BOUNDS"]
    if verbose:
        f += ["-Xptxas", "-v"]
    return f


def _newest_input(srcs):
    paths = [os.path.join(CSRC, s) for s in srcs] + [os.path.join(CSRC, h) for h in HEADERS]
    paths += [os.path.join(INCLUDE, h) for h in os.listdir(INCLUDE)]
    return max(os.path.getmtime(p) for p in paths)


def _compile(src: str, verbose: bool, check_bounds: bool = False) -> tuple[str, str]:
    obj = os.path.join(BUILD + ("_checked" if check_bounds else ""), src.replace(".cu", ".o"))
    cmd = [nvcc()] + _flags(verbose, check_bounds) + ["-c", os.path.join(CSRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    return obj, r.stdout + r.stderr


def _marshal_built_for() -> str:
    """What _marshal.so is compiled against besides its sources."""
    import torch
    return f"python {sys.version_info[:3]} torch {torch.__version__} cxx11 {int(torch._C._GLIBCXX_USE_CXX11_ABI)}\n"


def _marshal_stamp() -> str:
    return os.path.join(BUILD, "marshal.built_for")


def _marshal_stale(force: bool) -> bool:
    src, out = os.path.join(CSRC, MARSHAL_SRC), os.path.join(PKG, MARSHAL)
    newest = max(os.path.getmtime(p) for p in (src, os.path.join(INCLUDE, "dlmrefine.h")))
    if force or not os.path.exists(out) or os.path.getmtime(out) < newest or not os.path.exists(_marshal_stamp()):
        return True
    with open(_marshal_stamp()) as f:
        return f.read() != _marshal_built_for()


def _host_cxx(args: list[str]) -> None:
    r = subprocess.run([os.environ.get("CXX", "g++")] + args, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"{MARSHAL_SRC} failed to build:\n{r.stdout}\n{r.stderr}")


def _compile_marshal() -> str:
    import sysconfig

    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    obj = os.path.join(BUILD, MARSHAL_SRC.replace(".cpp", ".o"))
    dirs = [INCLUDE, inc, os.path.join(inc, "torch", "csrc", "api", "include"),
            os.path.join(os.path.dirname(os.path.dirname(nvcc())), "include"), sysconfig.get_paths()["include"]]
    _host_cxx(["-O2", "-fPIC", "-std=c++17", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] +
              [f"-I{d}" for d in dirs] + ["-c", os.path.join(CSRC, MARSHAL_SRC), "-o", obj])
    return obj


def _link_marshal(obj: str) -> None:
    import torch
    tlib = os.path.join(os.path.dirname(torch.__file__), "lib")
    out = os.path.join(PKG, MARSHAL)
    _host_cxx(["-shared", obj, "-o", out + ".tmp", "-L" + PKG, "-ldlmrefine", "-Wl,-rpath,$ORIGIN", "-L" + tlib,
               "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath," + tlib])
    os.replace(out + ".tmp", out)
    with open(_marshal_stamp(), "w") as f:
        f.write(_marshal_built_for())


def build(force: bool = False, verbose: bool = False, check_bounds: bool = False, out_dir: str | None = None) -> dict:
    out_dir = out_dir or PKG
    if check_bounds and os.path.abspath(out_dir) == PKG:
        raise ValueError("a --check-bounds build goes to its own directory (--out)")
    os.makedirs(BUILD + ("_checked" if check_bounds else ""), exist_ok=True)
    os.makedirs(out_dir, exist_ok=True)
    todo = {}
    for lib, srcs in LIBS.items():
        out = os.path.join(out_dir, lib)
        if force or not os.path.exists(out) or os.path.getmtime(out) < _newest_input(srcs):
            todo[lib] = srcs
    logs = {}
    marshal = out_dir == PKG and not check_bounds and _marshal_stale(force)
    if not todo and not marshal:
        return logs
    srcs = sorted({s for v in todo.values() for s in v})
    with cf.ThreadPoolExecutor(max_workers=8) as ex:
        marshal_obj = ex.submit(_compile_marshal) if marshal else None
        futs = {s: ex.submit(_compile, s, verbose, check_bounds) for s in srcs}
        objs = {s: f.result() for s, f in futs.items()}
    for s, (_, log) in objs.items():
        logs[s] = log
    for lib, lsrcs in todo.items():
        out = os.path.join(out_dir, lib)
        tmp = out + ".tmp"
        cmd = [nvcc()] + ARCH + ["-shared", "-cudart", "static", "-o", tmp] + [objs[s][0] for s in lsrcs]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed for {lib}:\n{r.stdout}\n{r.stderr}")
        os.replace(tmp, out)
    if marshal:
        _link_marshal(marshal_obj.result())
    return logs


def main(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--force", action="store_true")
    ap.add_argument("--verbose", action="store_true", help="print ptxas register/smem usage")
    ap.add_argument("--check-bounds", action="store_true", help="compile the input-contract checks in")
    ap.add_argument("--out", default=None, help="directory of the libraries (required with --check-bounds)")
    args = ap.parse_args(argv)
    logs = build(force=args.force, verbose=args.verbose, check_bounds=args.check_bounds, out_dir=args.out)
    if args.verbose:
        for s, log in sorted(logs.items()):
            print(f"==== {s}\n{log}")
    print("built:", ", ".join(sorted(LIBS)) if logs or args.force else "up to date")


if __name__ == "__main__":
    sys.exit(main())
