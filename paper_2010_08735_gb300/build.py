"""Build libbh.so in-tree with nvcc for sm_103a (GB300).

Each .cu file compiles in its own nvcc process (in parallel), then one link
step makes ``paper_2010_08735_gb300/libbh.so``.  The cube-map builder is
compiled without multiply-add contraction (its FP64 binning arithmetic must
round exactly as written); the FP32 renderer uses the approximate (2 ulp)
division and square root, and is also compiled without contraction: every
fused multiply-add in it is written out (fmaf), so that the single-camera and
batched instantiations of the pixel code round identically.  It flushes
denormals: every reciprocal, root and logarithm otherwise carries the scaling
of an operand below 1.2e-38 (80.2 -> 76.4 M warp instructions per 1080p frame,
90.5 -> 87.3 us, frames equal bit for bit).  No visible quantity of a pixel gets
there: radiances are relative to the disc's peak and to the exposures (the
disc's own luminance, 4e-50 at 256 K, is only ever handled as a logarithm).
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

HERE = Path(__file__).resolve().parent
CSRC = HERE / "csrc"
OUT = HERE / "libbh.so"
BUILD = HERE.parent / "_build"
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
COMMON = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
          "--expt-relaxed-constexpr", "-I", str(HERE.parent / "include")]
SOURCES = {"bh_core.cu": [], "bh_cubemap.cu": ["-fmad=false"],
           "bh_render.cu": ["-ftz=true", "-prec-div=false", "-prec-sqrt=false", "-fmad=false"], "bh_serve.cu": [], "bh_io.cu": [], "bh_peaks.cu": [], "bh_bloom.cu": []}


def nvcc() -> str:
    for c in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and Path(c).exists():
            return c
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libbh")


def _stale() -> bool:
    if not OUT.exists():
        return True
    t = OUT.stat().st_mtime
    deps = list(CSRC.glob("*")) + [HERE.parent / "include" / "bh.h", Path(__file__)]
    return any(p.stat().st_mtime > t for p in deps)


def build(force: bool = False, verbose: bool = False, extra: list[str] | None = None) -> Path:
    if not force and not _stale():
        return OUT
    BUILD.mkdir(exist_ok=True)
    cc = nvcc()
    extra = extra or []

    def compile_one(item):
        name, flags = item
        obj = BUILD / (name + ".o")
        cmd = [cc, *ARCH, *COMMON, *flags, *extra, "-c", str(CSRC / name), "-o", str(obj)]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {name}:\n{r.stderr}")
        if verbose and r.stderr:
            print(r.stderr, file=sys.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES.items()))
    tmp = OUT.with_suffix(f".so.tmp{os.getpid()}")
    cmd = [cc, *ARCH, "-shared", "-Xlinker", "--no-undefined", "-o", str(tmp), *map(str, objs), "-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, OUT)
    return OUT


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv,
          extra=["-Xptxas", "-v"] if "--ptxas" in sys.argv else None)
    print(OUT)
