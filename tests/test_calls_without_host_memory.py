"""Calls on plans without generated kernels neither allocate host memory nor throw: an exception may not leave the C
interface.  A child process runs them with an operator new that fails, and without a device: all they can do is
report that the kernel could not be launched."""
import os
import subprocess
import sys

NEW = r"""
#include <cstdlib>
#include <new>
static bool failing = false;
extern "C" void fail_allocations(int on) { failing = on != 0; }
void* operator new(std::size_t n) { if (failing) throw std::bad_alloc(); return std::malloc(n ? n : 1); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""

CHILD = r"""
import ctypes, os
import paper_2609_35099_b200 as e3j
lib, new = e3j._load(), ctypes.CDLL(os.environ["LD_PRELOAD"])
plan = e3j.e3j_plan_create("8x0e+8x1o+8x2e", 2, "0e+1o+1e")
p = 1 << 20   # never read: there is no device
big = 1 << 40
calls = [
    lambda: lib.e3j_conv_fwd(plan.handle, 5, 9, *[p] * 8, big, None),
    lambda: lib.e3j_conv_bwd(plan.handle, 5, 9, *[p] * 13, big, None),
    lambda: lib.e3j_tp_fwd(plan.handle, 5, *[p] * 4, None),
    lambda: lib.e3j_tp_bwd(plan.handle, 5, *[p] * 7, None),
    lambda: lib.e3j_conv_fwd_f64(plan.handle, 5, 9, *[p] * 8, big, None),
    lambda: lib.e3j_conv_bwd_f64(plan.handle, 5, 9, *[p] * 12, big, None),
]
for call in calls:
    call()        # the CUDA runtime's own first steps
for call in calls:
    new.fail_allocations(1)
    status = call()
    new.fail_allocations(0)
    assert status == e3j.E3J_ERR_CUDA, status
print("all calls returned")
"""


def test_calls_return_a_status_when_host_memory_is_exhausted(tmp_path, repo_root):
    src, lib = tmp_path / "new.cpp", tmp_path / "new.so"
    src.write_text(NEW)
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", str(src), "-o", str(lib)], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), CUDA_VISIBLE_DEVICES="", PYTHONPATH=repo_root)
    run = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=repo_root, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0 and "all calls returned" in run.stdout, run.stdout + run.stderr
