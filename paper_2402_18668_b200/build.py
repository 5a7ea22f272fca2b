"""Builds libbased.so (CUDA, sm_100a only) in-tree with nvcc, and the binding's extension with g++.

``python -m paper_2402_18668_b200.build`` or ``build()``; objects are rebuilt only
when their source (or a header) is newer.  nvcc cross-compiles without a GPU.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
INCLUDE = PKG.parent / "include"
OBJ = PKG / "build"
LIB = PKG / "libbased.so"
NATIVE_SRC = PKG / "csrc_host" / "native.cpp"
NATIVE = PKG / "_native.so"

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xptxas=-v",
    "-I", str(INCLUDE), "-I", str(CSRC),
] + (os.environ.get("BASED_NVCC_EXTRA", "").split())


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or Path(cand).exists()):
            return cand
    raise RuntimeError("nvcc not found")


def _cuda_include() -> str:
    """The headers of the toolkit that the compiler belongs to: beside its bin folder, links followed."""
    nvcc = Path(shutil.which(_nvcc()) or _nvcc())
    for root in (nvcc.parent.parent, nvcc.resolve().parent.parent, Path("/usr/local/cuda")):
        for inc in (root / "include", root / "targets" / "x86_64-linux" / "include"):
            if (inc / "cuda_runtime_api.h").exists():
                return str(inc)
    raise RuntimeError(f"no CUDA headers beside {nvcc}")


def sources():
    return sorted(CSRC.glob("*.cu"))


def _native_is_stale() -> bool:
    """Also after a change of the interpreter or of torch, whose C++ headers the extension is compiled against."""
    stamp = OBJ / "native.stamp"
    return (not NATIVE.exists() or not stamp.exists() or stamp.read_text() != _native_versions() or
            NATIVE.stat().st_mtime < max(p.stat().st_mtime for p in (NATIVE_SRC, INCLUDE / "based.h")))


def _native_versions() -> str:
    import torch
    return f"{sys.version_info[:3]} {torch.__version__}"


def build_native() -> Path:
    """_native.so: compiled against torch's headers; libbased.so is found beside it when it is loaded."""
    import sysconfig

    import torch
    t = Path(torch.__file__).resolve().parent
    stub = OBJ / "libbased.so"             # stands in for the library at link time: its symbols are resolved at load time
    r = subprocess.run(["g++", "-shared", "-Wl,-soname,libbased.so", "-o", str(stub), "-x", "c", os.devnull],
                       capture_output=True, text=True)
    tmp = NATIVE.with_suffix(f".so.tmp{os.getpid()}")
    if r.returncode == 0:
        r = subprocess.run(
            ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
             "-isystem", str(t / "include"), "-isystem", str(t / "include" / "torch" / "csrc" / "api" / "include"),
             "-isystem", sysconfig.get_paths()["include"], "-isystem", _cuda_include(), "-I", str(INCLUDE),
             str(NATIVE_SRC), "-o", str(tmp), "-L", str(t / "lib"), "-Wl,--no-as-needed", "-lc10", "-lc10_cuda", "-ltorch_cpu",
             "-ltorch", "-ltorch_python", "-L", str(OBJ), "-l:libbased.so", "-Wl,-rpath,$ORIGIN"],
            capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"{NATIVE_SRC.name} failed to build:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, NATIVE)
    (OBJ / "native.stamp").write_text(_native_versions())
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> Path:
    OBJ.mkdir(exist_ok=True)
    srcs = sources()
    hdr_mtime = max(p.stat().st_mtime for p in list(CSRC.glob("*.cuh")) + list(INCLUDE.glob("*.h")))
    nvcc = _nvcc()
    jobs = []
    for src in srcs:
        obj = OBJ / (src.stem + ".o")
        if force or not obj.exists() or obj.stat().st_mtime < max(src.stat().st_mtime, hdr_mtime):
            jobs.append((src, obj))

    def compile_one(job):
        src, obj = job
        r = subprocess.run([nvcc, *NVCC_FLAGS, "-c", str(src), "-o", str(obj)], capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src.name}:\n{r.stdout}\n{r.stderr}")
        (OBJ / (src.stem + ".ptxas.log")).write_text(r.stderr)
        if verbose:
            sys.stderr.write(r.stderr)

    native_jobs = [build_native] if force or _native_is_stale() else []
    with ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs) + len(native_jobs)))) as ex:
        running = [ex.submit(j) for j in native_jobs] + [ex.submit(compile_one, j) for j in jobs]
        for r in running:
            r.result()
    objs = [OBJ / (s.stem + ".o") for s in srcs]
    if jobs or not LIB.exists() or force:
        tmp = LIB.with_suffix(f".so.tmp{os.getpid()}")
        r = subprocess.run([nvcc, "-shared", "-cudart", "static", "-gencode", "arch=compute_100a,code=sm_100a",
                            "-o", str(tmp), *map(str, objs)], capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
