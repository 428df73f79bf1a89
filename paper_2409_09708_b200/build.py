"""Builds ``libelsa.so`` (nvcc for sm_100a; cross-compiles without a GPU) and the native half of the binding in-tree."""
from __future__ import annotations

import importlib.metadata
import importlib.util
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libelsa.so")
HOST_SOURCE = os.path.join(CSRC, "elsa_host.cpp")
# The module holds for one Python and one torch: its name has the one's tag, the file beside it the other's version.
HOST_LIB = os.path.join(HERE, "_elsa_host" + sysconfig.get_config_var("EXT_SUFFIX"))
HOST_STAMP = os.path.join(HERE, "_build", "elsa_host_torch_version")
SOURCES = ["elsa_api.cu", "elsa_attention.cu", "elsa_attention_rows.cu", "elsa_attention_window.cu", "elsa_backward.cu", "elsa_block.cu", "elsa_compress.cu", "elsa_int8.cu", "elsa_linear_simt.cu", "elsa_linear_small.cu", "elsa_linear_tc.cu", "elsa_linear_tc2.cu",
           "elsa_no_alloc.cu", "elsa_search.cu", "elsa_selftest.cu", "elsa_sparse24.cu", "elsa_sparse24_pair.cu", "elsa_sparse24_st.cu", "elsa_sparse24_ws.cu", "elsa_weight_images.cu"]


def nvcc_path() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def cuda_include() -> str:
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc_path()))), "include")


def sources() -> list[str]:
    return [os.path.join(CSRC, s) for s in SOURCES]


def is_stale() -> bool:
    header = os.path.join(ROOT, "include", "elsa.h")
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    return _older(LIB, [d for d in deps if d != HOST_SOURCE] + [header])


def _older(built: str, deps: list[str]) -> bool:
    return not os.path.exists(built) or any(os.path.getmtime(d) > os.path.getmtime(built) for d in deps)


def _stamp() -> str:
    return open(HOST_STAMP).read() if os.path.exists(HOST_STAMP) else ""


def host_is_stale() -> bool:
    return _stamp() != importlib.metadata.version("torch") or _older(HOST_LIB, [HOST_SOURCE, os.path.join(ROOT, "include", "elsa.h")])


def build_host(force: bool = False) -> str:
    """The extension module behind binding.py: C++ against torch's headers, the entry points handed to it by address."""
    if not force and not host_is_stale():
        return HOST_LIB
    version = importlib.metadata.version("torch")
    torch = importlib.util.find_spec("torch").submodule_search_locations[0]
    include = os.path.join(torch, "include")
    cmd = [os.environ.get("CXX") or "g++", "-O2", "-std=c++17", "-shared", "-fPIC", '-DELSA_TORCH_VERSION="%s"' % version,
           "-I", os.path.join(ROOT, "include"), "-isystem", include, "-isystem", os.path.join(include, "torch", "csrc", "api", "include"),
           "-isystem", sysconfig.get_paths()["include"], "-isystem", cuda_include(), HOST_SOURCE,
           "-L", os.path.join(torch, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-o", HOST_LIB + ".tmp"]
    subprocess.run(cmd, check=True)
    os.replace(HOST_LIB + ".tmp", HOST_LIB)
    os.makedirs(os.path.dirname(HOST_STAMP), exist_ok=True)
    with open(HOST_STAMP, "w") as f:
        f.write(version)
    untagged = os.path.join(HERE, "_elsa_host.so")          # what earlier builds left: any Python would try it
    if untagged != HOST_LIB and os.path.exists(untagged):
        os.remove(untagged)
    return HOST_LIB


def build(force: bool = False, verbose: bool = False) -> str:
    build_host(force)
    if not force and not is_stale():
        return LIB
    cmd = [nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "-shared", "-Xcompiler", "-fPIC", "-cudart", "static",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += sources() + ["-o", LIB + ".tmp"]
    subprocess.run(cmd, check=True)
    os.replace(LIB + ".tmp", LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
