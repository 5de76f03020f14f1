"""Build of the CUDA library libgvegas.so for sm_103a (in-tree).

Each csrc/*.cu translation unit is compiled by its own nvcc process (in
parallel), then linked into paper_1010_2107_gb300/_build/libgvegas.so with the
CUDA runtime linked statically.  Rebuilds only when a source is newer than the
library."""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libgvegas.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "--expt-relaxed-constexpr", "-I", OUT]
# Headers the run-time compiled kernels (rtc.cu) are built from, embedded in
# the library as text under the names their #include lines use.
RTC_HEADERS = [("col_hist.cuh", os.path.join(CSRC, "col_hist.cuh")),
               ("common.cuh", os.path.join(CSRC, "common.cuh")),
               ("integrands.cuh", os.path.join(CSRC, "integrands.cuh")),
               ("kernels.h", os.path.join(CSRC, "kernels.h")),
               ("sample_kernel.cuh", os.path.join(CSRC, "sample_kernel.cuh")),
               ("../../include/gvegas.h", os.path.join(ROOT, "include", "gvegas.h"))]
RTC_INC = os.path.join(OUT, "rtc_sources.inc")


def nvcc() -> str:
    for c in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libgvegas")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return _sources() + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + \
        sorted(glob.glob(os.path.join(CSRC, "*.h"))) + [os.path.join(ROOT, "include", "gvegas.h")]


def stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(p) > t for p in _deps())


def _write_rtc_sources() -> None:
    """Write _build/rtc_sources.inc: kRtcHeaders[i] = {include name, text}."""
    parts = ["// generated by _build.py from the kernel headers; do not edit\n",
             "static const char* const kRtcHeaders[][2] = {\n"]
    for name, path in RTC_HEADERS:
        with open(path) as f:
            text = f.read()
        # raw literals in pieces (compilers cap one literal's length)
        pieces = [text[i:i + 8000] for i in range(0, len(text), 8000)] or [""]
        for p in pieces:
            if ")gvrtc\"" in p:
                raise RuntimeError(f"{path} contains the raw-string delimiter")
        body = "\n".join('R"gvrtc(' + p + ')gvrtc"' for p in pieces)
        parts.append('    {"' + name + '",\n' + body + '},\n')
    parts.append("};\n")
    new = "".join(parts)
    old = open(RTC_INC).read() if os.path.exists(RTC_INC) else None
    if new != old:
        with open(RTC_INC + ".tmp", "w") as f:
            f.write(new)
        os.replace(RTC_INC + ".tmp", RTC_INC)
    else:  # current: only its time (a header touched without a change)
        os.utime(RTC_INC)


def _compile(src: str) -> str:
    obj = os.path.join(OUT, os.path.basename(src)[:-3] + ".o")
    if os.path.exists(obj) and os.path.getmtime(obj) >= max(
            os.path.getmtime(p) for p in [src] + _deps()[len(_sources()):]):
        return obj
    cmd = [nvcc()] + ARCH + FLAGS + ["-c", src, "-o", obj + ".tmp"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stderr}")
    os.replace(obj + ".tmp", obj)
    return obj


def build(force: bool = False, jobs: int | None = None) -> str:
    """Compile every CUDA source for sm_103a and link libgvegas.so."""
    os.makedirs(OUT, exist_ok=True)
    _write_rtc_sources()  # rewritten when a header changed, else only touched
    if not force and not stale():
        return LIB
    if force:
        for o in glob.glob(os.path.join(OUT, "*.o")):
            os.remove(o)
    srcs = _sources()
    jobs = jobs or min(len(srcs), os.cpu_count() or 4)
    with cf.ThreadPoolExecutor(max_workers=jobs) as ex:
        objs = list(ex.map(_compile, srcs))
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc()] + ARCH + ["-shared", "-o", tmp] + objs + ["-cudart", "static", "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build())
