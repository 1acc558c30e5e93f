"""Compile libsjq.so (hand-written sm_100a CUDA kernels + C ABI) in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
LIB = os.path.join(HERE, "libsjq.so")
OBJ = os.path.join(HERE, "csrc", "obj")  # one object per translation unit, so that an edit recompiles only its own
# CPython extension: the binding's argument marshalling, linked to LIB.  The name carries the interpreter's tag: another
# version of Python does not load it and builds its own.
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC"]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(HERE, "csrc", "*.cu")))


def _headers() -> list[str]:
    return glob.glob(os.path.join(HERE, "csrc", "*.h")) + glob.glob(os.path.join(HERE, "csrc", "*.cuh")) + glob.glob(
        os.path.join(ROOT, "include", "*.h"))


def _object(src: str) -> str:
    return os.path.join(OBJ, os.path.splitext(os.path.basename(src))[0] + ".o")


def _stale(target: str, deps: list[str]) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile the translation units that changed (all of them with force) in parallel, then link."""
    extra = os.environ.get("SJQ_NVCC_EXTRA", "").split()  # e.g. -D switches for kernel experiments
    headers = _headers()
    if not force and not extra and not _stale(LIB, sources() + headers):  # whatever became of the objects
        _build_marshal(False)
        return LIB
    todo = [s for s in sources() if force or extra or _stale(_object(s), [s] + headers)]
    if not todo and not _stale(LIB, [_object(s) for s in sources()]):
        _build_marshal(force)
        return LIB
    os.makedirs(OBJ, exist_ok=True)

    def compile_one(src: str) -> None:
        cmd = ["nvcc", *NVCC_FLAGS, *extra, "-I" + os.path.join(ROOT, "include"), "-c", src, "-o", _object(src)]
        if verbose:
            cmd[1:1] = ["-Xptxas", "-v"]
        subprocess.check_call(cmd, cwd=HERE)

    with ThreadPoolExecutor(max_workers=max(1, min(len(todo), os.cpu_count() or 1))) as pool:
        list(pool.map(compile_one, todo))
    subprocess.check_call(["nvcc", "-shared", *NVCC_FLAGS[:2], "-Xlinker", "-soname=libsjq.so", "-o", LIB, *[_object(s) for s in sources()]], cwd=HERE)
    _build_marshal(force)
    return LIB


def _build_marshal(force: bool) -> None:
    src = os.path.join(HERE, "csrc", "sjq_py.cpp")
    untagged = os.path.join(HERE, "_marshal.so")  # as it was named before: any version of Python would load it
    if os.path.exists(untagged):
        os.remove(untagged)
    if force or _stale(MARSHAL, [src, os.path.join(ROOT, "include", "sjq.h")]):
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-fPIC", "-shared", "-fvisibility=hidden",
                               "-I" + os.path.join(ROOT, "include"), "-I" + sysconfig.get_paths()["include"], src, LIB,
                               "-Wl,-rpath,$ORIGIN", "-o", MARSHAL], cwd=HERE)


if __name__ == "__main__":
    print(build(force=True, verbose=True))
