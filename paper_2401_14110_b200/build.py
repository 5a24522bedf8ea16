"""Build ``liblba.so`` (the CUDA library behind the C ABI) in-tree for sm_100a, and ``lba_torch.so`` (its calls from PyTorch tensors).

Objects go to ``_build/`` at the repository root (ignored by git); the shared library is written
next to this file so that it travels with the source tree.  nvcc cross-compiles without a GPU.
"""
import glob
import os
import subprocess
import sys
import sysconfig
import warnings
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ_DIR = os.path.join(ROOT, "_build", "liblba")
LIB = os.path.join(HERE, "liblba.so")
TORCH_SRC = os.path.join(CSRC, "lba_torch.cpp")
TORCH_LIB = os.path.join(HERE, "lba_torch.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC",
         "-I", os.path.join(ROOT, "include")]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.inc")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h"))


def _stale(target, sources):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(s) > t for s in sources)


def _compile(src, verbose):
    obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
    if _stale(obj, [src] + _deps()):
        cmd = [NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stderr.write(r.stderr)
    return obj


def torch_tag() -> str:
    """What lba_torch.so is built for; it carries this text (``built_for``) and runs with no other torch or interpreter."""
    import torch
    return f"lba_torch for torch {torch.__version__} {sys.implementation.cache_tag}"


def _carries(path, text) -> bool:
    with open(path, "rb") as f:
        return text.encode() in f.read()


def build_torch(force: bool = False) -> str:
    """The Python module over the library, linked to the liblba.so beside it."""
    tag = torch_tag()
    if force or _stale(TORCH_LIB, [TORCH_SRC] + glob.glob(os.path.join(ROOT, "include", "*.h"))) or not _carries(TORCH_LIB, tag):
        import torch
        top = os.path.dirname(torch.__file__)
        cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", TORCH_SRC, "-o", TORCH_LIB + ".tmp",
               f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DLBA_TORCH_TAG="{tag}"']
        for inc in (os.path.join(ROOT, "include"), os.path.join(top, "include"),
                    os.path.join(top, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
                    os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")):
            cmd += ["-I", inc]
        cmd += ["-L", os.path.join(top, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
                "-L", HERE, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"g++ failed on {TORCH_SRC}:\n{r.stdout}\n{r.stderr}")
        os.replace(TORCH_LIB + ".tmp", TORCH_LIB)
    return TORCH_LIB


def build(force: bool = False, verbose: bool = False, jobs: int = 0) -> str:
    os.makedirs(OBJ_DIR, exist_ok=True)
    srcs = _sources()
    if force:
        for o in glob.glob(os.path.join(OBJ_DIR, "*.o")):
            os.remove(o)
    jobs = jobs or max(1, min(len(srcs), len(os.sched_getaffinity(0))))
    with ThreadPoolExecutor(jobs) as ex:
        objs = list(ex.map(lambda s: _compile(s, verbose), srcs))
    if force or _stale(LIB, objs):
        cmd = [NVCC, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB + ".tmp"] + objs
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
        os.replace(LIB + ".tmp", LIB)
    try:
        build_torch(force)
    except (OSError, RuntimeError) as e:  # no g++, or a torch without CUDA: the library is complete without the module
        warnings.warn(f"lba_torch.so was not built, calls will go through ctypes: {e}")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
