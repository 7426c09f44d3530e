"""Builds libsar.so (the C-ABI library of include/sar.h) in-tree with nvcc for sm_100a, and _sar_torch.so (the native
side of api.py: allocation with torch's allocator and the calls into libsar) with g++.

    python -m paper_2111_06483_b200.build [--force] [--verbose]

nvcc cross-compiles, so this works on a machine without a GPU.  Sources are compiled in
parallel into csrc/build/*.o and linked into paper_2111_06483_b200/libsar.so.
"""
from __future__ import annotations

import hashlib
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(CSRC, "build")
LIB = os.path.join(PKG, "libsar.so")
TORCH_EXT = os.path.join(PKG, "_sar_torch.so")
ROW_PASSES = ["fwd", "fwd_part", "dst", "dst_part", "src", "sum"]   # one translation unit per pass and storage type
SOURCES = ["sar_linear.cu"] + [f"sar_lean_{p}_{t}.cu" for p in ("fwd", "bwd_dst", "bwd_src") for t in ("f32", "bf16")] + [f"sar_rows_{p}_{t}.cu" for p in ROW_PASSES for t in ("f32", "bf16")] + [
    "sar_gat.cu", "sar_span.cu", "sar_rows_merge.cu", "sar_graph.cu", "sar_host.cu", "sar_noalloc.cu", "sar_storing.cu",
    "sar_glue.cu", "sar_norm.cu", "sar_rgcn.cu"]
NVCC_FLAGS = [
    "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--expt-relaxed-constexpr",
    "-DSAR_BUILT_FOR_SM=100", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _cutlass_includes() -> list:
    """Include paths of a CUTLASS / CuTe header tree with sm100 support (sar_linear.cu instantiates its
    collective templates).  The image vendors one inside the flashinfer package."""
    import site
    roots = list(site.getsitepackages()) + [os.environ.get("CUTLASS_PATH", "")]
    for root in roots:
        for sub in ("flashinfer/data/cutlass", "tilelang/3rdparty/cutlass", ""):
            base = os.path.join(root, sub) if root else ""
            if base and os.path.exists(os.path.join(base, "include", "cute", "arch", "mma_sm100_umma.hpp")):
                return ["-I", os.path.join(base, "include"), "-I", os.path.join(base, "tools", "util", "include")]
    raise RuntimeError("sar_linear.cu needs a CUTLASS / CuTe header tree with sm100 support (cute/arch/mma_sm100_umma.hpp): "
                       "none found in this Python environment's flashinfer or tilelang packages; set CUTLASS_PATH to the "
                       "root of a CUTLASS checkout (the directory that holds include/ and tools/util/include/)")


def _deps(path: str, seen=None) -> list:
    """The file and every header of this library it includes, directly or not (quoted includes only)."""
    import re
    seen = seen if seen is not None else []
    if path in seen or not os.path.exists(path):
        return seen
    seen.append(path)
    for inc in re.findall(r'^\s*#\s*include\s+"([^"]+)"', open(path).read(), flags=re.M):
        for base in (os.path.dirname(path), CSRC, os.path.join(ROOT, "include")):
            cand = os.path.join(base, inc)
            if os.path.exists(cand):
                _deps(cand, seen)
                break
    return seen


def _fingerprint(src: str) -> str:
    """Hash of one source file, the headers it reaches and the compiler flags."""
    h = hashlib.sha256()
    for path in sorted(_deps(os.path.join(CSRC, src))):
        h.update(os.path.basename(path).encode())
        h.update(open(path, "rb").read())
    h.update(" ".join(NVCC_FLAGS).encode())
    return h.hexdigest()


def build_torch_ext(force: bool = False) -> str:
    """_sar_torch.so, when its source, sar.h or torch changed.  It links against nothing of libsar: the entry points are
    looked up in the library that the process has loaded."""
    import sysconfig
    import torch
    from torch.utils.cpp_extension import include_paths
    src, stamp = os.path.join(CSRC, "sar_torch.cpp"), os.path.join(OBJ, "sar_torch.fingerprint")
    fp = hashlib.sha256((_fingerprint("sar_torch.cpp") + torch.__version__ + sys.version).encode()).hexdigest()
    if not force and os.path.exists(TORCH_EXT) and os.path.exists(stamp) and open(stamp).read() == fp:
        return TORCH_EXT
    inc = [f"-I{p}" for p in include_paths() + [sysconfig.get_paths()["include"], os.path.join(ROOT, "include"),
                                                os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include")]]
    libdir = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = TORCH_EXT + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *inc, src, "-o", tmp, f"-L{libdir}",
           f"-Wl,-rpath,{libdir}", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch", "-ltorch_python", "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed on sar_torch.cpp:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, TORCH_EXT)
    open(stamp, "w").write(fp)
    return TORCH_EXT


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles the sources whose contents (or headers, or flags) changed since their object was built, in
    parallel, and links libsar.so when any object is new."""
    os.makedirs(OBJ, exist_ok=True)
    nvcc = _nvcc()
    extra = ["-Xptxas", "-v"] if verbose else []

    def compile_one(src):
        obj = os.path.join(OBJ, src.replace(".cu", ".o"))
        stamp = obj + ".fingerprint"
        fp = _fingerprint(src)
        if not force and os.path.exists(obj) and os.path.exists(stamp) and open(stamp).read() == fp:
            return obj, False
        inc = _cutlass_includes() if src == "sar_linear.cu" else []
        cmd = [nvcc, *NVCC_FLAGS, *inc, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stderr.write(r.stderr)
        open(stamp, "w").write(fp)
        return obj, True

    with ThreadPoolExecutor(min(len(SOURCES), os.cpu_count() or 4)) as ex:
        ext = ex.submit(build_torch_ext, force)
        results = list(ex.map(compile_one, SOURCES))
        ext.result()
    objs = [o for o, _ in results]
    if not force and os.path.exists(LIB) and not any(new for _, new in results):
        return LIB
    tmp = LIB + f".tmp{os.getpid()}"
    r = subprocess.run([nvcc, "-shared", "-o", tmp, *objs, "-Xcompiler", "-fPIC"], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
