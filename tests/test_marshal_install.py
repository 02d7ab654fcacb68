"""How the binding takes up its native marshalling (csrc/host/marshal.cpp): no device."""
import subprocess
import sys

import pytest

pytest.importorskip("torch")


def _run(code, cwd):
    return subprocess.run([sys.executable, "-c", code], cwd=cwd, capture_output=True, text=True, timeout=300)


def test_two_threads_in_their_first_call(repo_root):
    """Whoever comes second must not make the native functions their own fall-back."""
    done = _run("""
import threading
import torch
import paper_2609_35099_b200 as e3j
gate = threading.Barrier(2)
def first_call():
    gate.wait()
    e3j._torch()
threads = [threading.Thread(target=first_call) for _ in range(2)]
for t in threads: t.start()
for t in threads: t.join()
for _ in range(2):   # (again with everything in place: the order that a preempted thread gives)
    try:
        e3j._dev_ptr(torch.zeros(3), torch.float32, (3,), "x")
    except TypeError as error:
        print(error)
    e3j._torch_module = None
    e3j._torch()
""", repo_root)
    assert done.stdout.splitlines() == ["x must be a CUDA tensor"] * 2, done.stderr[-2000:]
