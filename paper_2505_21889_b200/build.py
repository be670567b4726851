"""Compile the CUDA sources into libefim.so (sm_100a only) and the argument marshalling of the
Python package into _calls.so, in-tree."""
import glob
import os
import shutil
import subprocess
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
LIB_PATH = os.path.join(PKG_DIR, "libefim.so")
EXT_PATH = os.path.join(PKG_DIR, "_calls.so")


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found; the EFIM library needs the CUDA toolkit to build")
    return exe


def sources():
    return sorted(glob.glob(os.path.join(PKG_DIR, "csrc", "*.cu")))


def needs_build() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(EXT_PATH):
        return True
    t = min(os.path.getmtime(LIB_PATH), os.path.getmtime(EXT_PATH))
    deps = sources() + glob.glob(os.path.join(PKG_DIR, "csrc", "*.cuh")) + \
        glob.glob(os.path.join(PKG_DIR, "csrc", "*.c")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """nvcc -> paper_2505_21889_b200/libefim.so.  Returns the library path."""
    if not force and not needs_build():
        return LIB_PATH
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-Xlinker", "-soname=libefim.so", "-I" + os.path.join(ROOT, "include"),
           "-o", LIB_PATH] + sources()
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stderr)
    # the extension finds the library beside it
    cmd = ["gcc", "-O2", "-shared", "-fPIC", "-I" + os.path.join(ROOT, "include"),
           "-I" + sysconfig.get_paths()["include"], "-o", EXT_PATH, os.path.join(PKG_DIR, "csrc", "calls.c"), LIB_PATH,
           "-Wl,-rpath,$ORIGIN"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("gcc failed:\n" + res.stdout + res.stderr)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
