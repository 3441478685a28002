"""Build liblords.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
INCLUDE = PKG.parent / "include"
LIB = PKG / "liblords.so"
# the CPython module over it; the tag (cpython-312-x86_64-linux-gnu) keeps an interpreter from loading another's
NATIVE = PKG / f"_native.{sysconfig.get_config_var('SOABI')}.so"

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    # no fast-math: IEEE arithmetic, parity is judged against an fp64 oracle
    "-Xcompiler", "-fPIC",
]


def sources():
    return sorted(CSRC.glob("*.cu"))


def _headers():
    return [*CSRC.glob("*.h"), *CSRC.glob("*.cuh"), *INCLUDE.glob("*.h"), Path(__file__)]


def _older(target: Path, deps) -> bool:
    return not target.exists() or any(d.stat().st_mtime > target.stat().st_mtime for d in deps)


def needs_build() -> bool:
    deps = [*CSRC.glob("*"), *_headers()]
    return _older(LIB, deps) or _older(NATIVE, deps)


def build(force: bool = False, verbose: bool = False) -> Path:
    """Compile every .cu under csrc/ into paper_2601_22716_b200/liblords.so, and the CPython module over it.

    One nvcc process per translation unit; objects that are newer than their source and every header are kept."""
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    objdir = PKG / "_build"
    objdir.mkdir(exist_ok=True)

    def compile_one(src: Path):
        obj = objdir / (src.stem + ".o")
        if force or verbose or _older(obj, [src, *_headers()]):
            tmp = obj.with_name(f"{src.stem}.tmp{os.getpid()}.o")
            _run([nvcc, *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), f"-I{INCLUDE}", f"-I{CSRC}", "-c", str(src), "-o", str(tmp)], verbose)
            os.replace(tmp, obj)
        return obj

    with ThreadPoolExecutor() as pool:
        objs = list(pool.map(compile_one, sources()))
    tmp = LIB.with_name(f"liblords.tmp{os.getpid()}.so")
    _run([nvcc, *NVCC_FLAGS, "-shared", "-cudart", "static", *map(str, objs), "-o", str(tmp)])
    os.replace(tmp, LIB)
    build_module()
    return LIB


def _run(cmd, verbose: bool = False):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"{cmd[0]} failed")


def build_module() -> Path:
    tmp = NATIVE.with_name(f"_native_tmp{os.getpid()}.so")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-I{INCLUDE}", f"-I{sysconfig.get_paths()['include']}",
           str(CSRC / "lords_module.cc"), f"-L{PKG}", "-l:liblords.so", "-Wl,-rpath,$ORIGIN", "-o", str(tmp)]
    _run(cmd)
    os.replace(tmp, NATIVE)
    return NATIVE


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
