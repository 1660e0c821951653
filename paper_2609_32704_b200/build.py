"""Builds libcowa.so (all CUDA translation units, sm_100a) in-tree with nvcc, and the binding's argument path with g++."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
OBJ_DIR = os.path.join(HERE, "build")
LIB_PATH = os.path.join(HERE, "libcowa.so")
CALL_SRC = os.path.join(HERE, "csrc_py", "cowa_call.cpp")
CALL_PATH = os.path.join(HERE, "_cowa_call" + sysconfig.get_config_var("EXT_SUFFIX"))  # (another Python does not load it)

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-I", INCLUDE,
]


def _nvcc():
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _headers_mtime():
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    paths += [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return max(os.path.getmtime(p) for p in paths)


def _compile(src, verbose):
    obj = os.path.join(OBJ_DIR, src[:-3] + ".o")
    spath = os.path.join(CSRC, src)
    if os.path.exists(obj) and os.path.getmtime(obj) >= max(os.path.getmtime(spath), _headers_mtime()):
        return obj, False
    cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", spath, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}")
    return obj, True


def _call_stamp():
    """What the argument path's module was built against, kept beside the objects: PyTorch's headers do not get newer than
    the module when another version is installed."""
    return os.path.join(OBJ_DIR, "cowa_call.torch")


def _read(path):
    try:
        with open(path) as f:
            return f.read()
    except OSError:
        return None


def _build_call_module(verbose):
    """The binding's native argument path: a Python extension over torch's headers (no CUDA code)."""
    import torch
    if (os.path.exists(CALL_PATH) and os.path.getmtime(CALL_PATH) >= max(os.path.getmtime(CALL_SRC), _headers_mtime())
            and _read(_call_stamp()) == torch.__version__):
        return
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc())) or "/usr/local/cuda"
    inc = [INCLUDE, os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    cmd += [f"-I{d}" for d in inc] + [CALL_SRC, "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu",
                                      "-ltorch_python", "-o", CALL_PATH]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError("g++ failed on cowa_call.cpp")
    with open(_call_stamp(), "w") as f:
        f.write(torch.__version__)


def build_library(verbose=False, force=False):
    """Compiles every .cu under csrc/ and links libcowa.so.  Returns its path.  The binding's argument path is built beside it
    where that can be done (PyTorch, g++, Python headers); without it every call takes the Python path."""
    os.makedirs(OBJ_DIR, exist_ok=True)
    if force:
        for f in os.listdir(OBJ_DIR):
            if f.endswith(".o"):
                os.remove(os.path.join(OBJ_DIR, f))
        if os.path.exists(CALL_PATH):
            os.remove(CALL_PATH)
    with ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as ex:
        call = ex.submit(_build_call_module, verbose)
        res = list(ex.map(lambda s: _compile(s, verbose), _sources()))
    objs = [o for o, _ in res]
    rebuilt = any(ch for _, ch in res)
    if rebuilt or not os.path.exists(LIB_PATH):
        cmd = [_nvcc(), "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB_PATH] + objs
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    try:
        call.result()
    except (ImportError, OSError, RuntimeError) as e:
        sys.stderr.write(f"{os.path.basename(CALL_SRC)} not built, calls take the Python path: {e}\n")
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(verbose="-v" in sys.argv, force="-f" in sys.argv))
