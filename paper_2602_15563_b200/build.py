"""Build libkmq.so and its Python extension module in-tree with nvcc for sm_100a (no JIT cache involved)."""
from __future__ import annotations

import glob
import importlib.util
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libkmq.so")
NATIVE_SRC = os.path.join(CSRC, "kmq_python.cpp")
NATIVE_PATH = os.path.join(PKG_DIR, "_kmq_native" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]
OBJ_DIR = os.path.join(PKG_DIR, "_build")


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: libkmq cannot be built")


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _torch_include() -> list[str]:
    """torch's header folder as an include option (the extension module uses its DLPack header where it has the exchange
    table), found without importing torch; nothing where torch is not installed."""
    spec = importlib.util.find_spec("torch")
    return ["-I", os.path.join(os.path.dirname(spec.origin), "include")] if spec and spec.origin else []


def native_command(out: str, torch_include: list[str]) -> list[str]:
    """How the extension module is compiled and linked: host code only; it finds libkmq.so beside itself at run time."""
    return [_nvcc(), "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I",
            sysconfig.get_paths()["include"], *torch_include, NATIVE_SRC, "-L", PKG_DIR, "-l:libkmq.so", "-Xlinker",
            "-rpath=$ORIGIN", "-o", out]


def needs_build() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(NATIVE_PATH):
        return True
    t = min(os.path.getmtime(LIB_PATH), os.path.getmtime(NATIVE_PATH))
    deps = sources() + [NATIVE_SRC] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into libkmq.so and the extension module beside it; returns the library's path."""
    if not force and not needs_build():
        return LIB_PATH
    os.makedirs(OBJ_DIR, exist_ok=True)
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    newest_header = max(os.path.getmtime(h) for h in headers)
    base = [_nvcc(), *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        base += ["-Xptxas", "-v"]

    def compile_one(src: str) -> str:
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        if not force and os.path.exists(obj) and os.path.getmtime(obj) > max(os.path.getmtime(src), newest_header):
            return obj
        res = subprocess.run(base + ["-c", src, "-o", obj], capture_output=True, text=True)
        if res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
            raise RuntimeError(f"nvcc failed on {os.path.basename(src)}")
        if verbose:
            sys.stderr.write(res.stderr)
        return obj

    # one translation unit per kernel file, compiled side by side, then linked into the shared library
    with ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as pool:
        objs = list(pool.map(compile_one, sources()))
    res = subprocess.run([_nvcc(), "-shared", "-gencode", "arch=compute_100a,code=sm_100a", *objs, "-o",
                          LIB_PATH + ".tmp"], capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc failed linking libkmq.so")
    os.replace(LIB_PATH + ".tmp", LIB_PATH)

    res = subprocess.run(native_command(NATIVE_PATH + ".tmp", _torch_include()), capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("building the extension module failed")
    os.replace(NATIVE_PATH + ".tmp", NATIVE_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
