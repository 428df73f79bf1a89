"""Where the native half of the binding takes its outputs from."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

ALLOCATOR = r"""
#include <cuda_runtime_api.h>
#include <mutex>
#include <set>
#include <sys/types.h>
static std::mutex lock;
static std::set<void*> live;
extern "C" void* take(ssize_t size, int, cudaStream_t)
{
    void* p = nullptr;
    if (cudaMalloc(&p, size) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> held(lock);
    live.insert(p);
    return p;
}
extern "C" void give(void* p, ssize_t, int, cudaStream_t)
{
    std::lock_guard<std::mutex> held(lock);
    live.erase(p);
    cudaFree(p);
}
extern "C" int owns(void* p)
{
    std::lock_guard<std::mutex> held(lock);
    return live.count(p) != 0;
}
"""

PROGRAM = r"""
import ctypes, sys, torch
path = sys.argv[1]
torch.cuda.memory.change_current_allocator(torch.cuda.memory.CUDAPluggableAllocator(path, "take", "give"))
owns = lambda t: bool(ctypes.CDLL(path).owns(ctypes.c_void_p(t.data_ptr())))
from paper_2409_09708_b200 import binding as lib
X = torch.randn(8, 64, device="cuda", dtype=torch.float16)
W = torch.randn(16, 64, device="cuda", dtype=torch.float16)
assert owns(X) and owns(W)
vals, idx = lib.elsa_nm_compress(W, 2, 8)
out = [vals, idx, lib.elsa_nm_linear(X, vals, idx, None, 16, 64, 2, 8), lib.elsa_nm_linear_masked(X, W, None, 2, 8)]
out += [t for pair in lib.elsa_nm_compress_levels(W, [1, 4], 8) for t in pair]
out += lib.elsa_nm_linear_backward(out[2], X, vals, idx, 16, 64, 2, 8)
torch.cuda.synchronize()
assert all(owns(t) for t in out), [owns(t) for t in out]
print("ok", len(out))
"""


@pytest.mark.gpu
def test_outputs_come_from_the_allocator_in_place(tmp_path):
    """A program with an allocator of its own (a pool that has the whole device, say) gets the outputs from there as well."""
    from paper_2409_09708_b200 import build
    source, built = tmp_path / "allocator.cpp", tmp_path / "allocator.so"
    source.write_text(ALLOCATOR)
    include = build.cuda_include()
    subprocess.run(["g++", "-shared", "-fPIC", "-I", include, str(source), "-L", os.path.join(os.path.dirname(include), "lib64"), "-lcudart",
                    "-o", str(built)], check=True)
    run = subprocess.run([sys.executable, "-c", PROGRAM, str(built)], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert run.returncode == 0 and "ok 11" in run.stdout, run.stdout + run.stderr


@pytest.mark.gpu
def test_transforms_reach_the_outputs():
    """Inside a transform torch.empty's result belongs to the transform and has no memory to hand to the library: the call is refused,
    with outputs from the allocator it would leave the transform without a word."""
    import torch
    from paper_2409_09708_b200 import binding as lib
    W = torch.randn(16, 64, device="cuda", dtype=torch.float16)

    def f(s):
        with pytest.raises(RuntimeError, match="storage"):
            lib.elsa_nm_compress(W, 2, 8)
        return 2 * s

    assert float(torch.func.grad(f)(torch.tensor(1.0))) == 2.0
    lib.elsa_nm_compress(W, 2, 8)
    torch.cuda.synchronize()
