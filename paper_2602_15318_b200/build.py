"""Builds libsparrow_attn.so (C ABI, sm_100a only; nvcc) and _pycall.so (the Python binding's argument
marshalling; g++) in-tree."""
import importlib.metadata
import importlib.util
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsparrow_attn.so")
PYCALL = os.path.join(HERE, "_pycall.so")
PYCALL_VERSIONS = os.path.join(HERE, "_pycall.versions")
PYCALL_SOURCES = [os.path.join(CSRC, "pycall.c"), os.path.join(CSRC, "pycall_torch.cpp")]
SOURCES = [os.path.join(CSRC, "api.cu")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC"]


def _newest_source() -> float:
    t = 0.0
    for d in (CSRC, os.path.join(ROOT, "include")):
        for f in os.listdir(d):
            t = max(t, os.path.getmtime(os.path.join(d, f)))
    return t


def nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.isabs(c) and os.path.exists(c) or not os.path.isabs(c)):
            return c
    return "nvcc"


def pycall_versions() -> str:
    """What _pycall.so is only good for: this interpreter and this torch, whose C++ symbols it is linked to."""
    return f"{sys.implementation.cache_tag} torch {importlib.metadata.version('torch')}"


def pycall_is_current() -> bool:
    """Built from the present sources for the present interpreter and torch (recorded beside it at the build)."""
    if not os.path.exists(PYCALL) or os.path.getmtime(PYCALL) < max(os.path.getmtime(s) for s in PYCALL_SOURCES):
        return False
    try:
        with open(PYCALL_VERSIONS) as f:
            return f.read() == pycall_versions()
    except OSError:
        return False


def build_pycall(force: bool = False) -> str:
    if force or not pycall_is_current():
        torch_dir = importlib.util.find_spec("torch").submodule_search_locations[0]
        torch_lib = os.path.join(torch_dir, "lib")
        include = [os.path.join(torch_dir, "include"), os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
                   os.path.join(os.path.dirname(os.path.dirname(nvcc())), "include"), sysconfig.get_paths()["include"]]
        subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-shared", "-fPIC", *["-I" + i for i in include], "-o", PYCALL,
                        "-x", "c", PYCALL_SOURCES[0], "-x", "c++", PYCALL_SOURCES[1], "-x", "none",
                        "-L" + torch_lib, "-Wl,-rpath," + torch_lib, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"],
                       check=True)
        with open(PYCALL_VERSIONS, "w") as f:
            f.write(pycall_versions())
    return PYCALL


def build(force: bool = False, verbose: bool = False) -> str:
    build_pycall(force)
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source():
        return LIB
    cmd = [nvcc()] + NVCC_FLAGS + ["-I" + os.path.join(ROOT, "include"), "-I" + CSRC, "-o", LIB] + SOURCES
    if verbose:
        cmd.insert(1, "-Xptxas"); cmd.insert(2, "-v")
    subprocess.run(cmd, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
