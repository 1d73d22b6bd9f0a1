"""Other Python threads go on while the native way allocates: an allocator that takes its time, and a thread that counts meanwhile."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

ALLOCATOR = r"""
#include <cuda_runtime_api.h>
#include <unistd.h>
static volatile int slow = 0;
extern "C" void set_slow(int on) { slow = on; }
extern "C" void* slow_malloc(ssize_t size, int, cudaStream_t) {
    if (slow) usleep(200000);
    void* p = nullptr;
    return cudaMalloc(&p, size) == cudaSuccess ? p : nullptr;
}
extern "C" void slow_free(void* p, ssize_t, int, cudaStream_t) { cudaFree(p); }
"""

PROGRAM = r"""
import ctypes, sys, threading, time
import numpy as np
import torch
torch.cuda.memory.change_current_allocator(torch.cuda.memory.CUDAPluggableAllocator(sys.argv[1], "slow_malloc", "slow_free"))
import paper_2502_08141_b200 as lw

N, K, M, r = 256, 256, 4, 16
layout = lw.Layout(np.full(N, 2, np.uint8), K)
z = lambda *shape: torch.zeros(*shape, dtype=torch.bfloat16, device="cuda")
packed = torch.zeros(layout.packed_bytes, dtype=torch.uint8, device="cuda")
absmax, maps = torch.zeros(N, K // 64, device="cuda"), torch.zeros(N, 16, device="cuda")
args = (layout.address, layout.device_index, packed, absmax, maps, z(M, K), z(K, r), z(r, N), 1.0, None, None)
assert lw._py_calls.forward(*args) is not None
torch.cuda.synchronize()
count, done = 0, False


def counting():
    global count
    while not done:
        count += 1
        time.sleep(0.002)


thread = threading.Thread(target=counting)
thread.start()
slow = ctypes.CDLL(sys.argv[1])
slow.set_slow(1)
before = count
out = lw._py_calls.forward(*args)      # the output and the scratch: two allocations of 0.2 s
counted = count - before
slow.set_slow(0)
done = True
thread.join()
torch.cuda.synchronize()
assert out is not None and not out.any()
assert counted >= 20, counted
"""


def test_threads_go_on_during_allocations(tmp_path):
    import torch
    from torch.utils import cpp_extension

    source, library, program = tmp_path / "allocator.cpp", tmp_path / "allocator.so", tmp_path / "program.py"
    source.write_text(ALLOCATOR)
    program.write_text(PROGRAM)
    includes = ["-I" + i for i in cpp_extension.include_paths(device_type="cuda")]
    subprocess.run(["g++", "-shared", "-fPIC", "-w", *includes, str(source), "-o", str(library), "-L/usr/local/cuda/lib64", "-lcudart"], check=True)
    subprocess.run([sys.executable, str(program), str(library)], cwd=ROOT, env={**os.environ, "PYTHONPATH": ROOT}, check=True, timeout=300)
