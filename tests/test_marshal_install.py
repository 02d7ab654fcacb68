"""How the binding takes up its native marshalling (csrc/host/marshal.cpp): no device."""
import ctypes
import pathlib
import shutil
import subprocess
import sys
import sysconfig

import pytest

torch = pytest.importorskip("torch")


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


def test_a_module_built_for_another_torch_is_not_used(repo_root):
    """Its functions would read tensors with the wrong layouts."""
    done = _run("""
import sys, types, warnings
import paper_2609_35099_b200 as e3j
def never(*args): raise SystemExit("called")
other = types.SimpleNamespace(set_slow=never, dev_ptr=never, empty=never, call=never, call_size=never, built_for="torch 1.0")
sys.modules[e3j.__name__ + "._marshal"] = other
with warnings.catch_warnings(record=True) as seen:
    warnings.simplefilter("always")
    e3j._torch()
print(e3j._native, "torch 1.0" in str(seen[0].message))
""", repo_root)
    assert done.stdout.split() == ["None", "True"], done.stderr[-2000:]


def test_it_is_there_where_it_can_be_built(repo_root):
    from torch.utils import cpp_extension
    if not shutil.which("g++") or not any((pathlib.Path(d) / "torch" / "csrc" / "Dtype.h").exists() for d in cpp_extension.include_paths()):
        pytest.skip("no g++, or no headers of torch")
    done = _run("import paper_2609_35099_b200 as e3j; t = e3j._torch(); print(e3j._native.built_for == e3j._marshal_abi(t))", repo_root)
    assert done.stdout.split() == ["True"], done.stderr[-2000:]


@pytest.mark.parametrize("missing", ["torch", "g++"])
def test_the_library_is_linked_without_it(missing, tmp_path, monkeypatch, capsys):
    """The C library needs neither torch nor a host compiler of that name; what an earlier build left is taken away."""
    from paper_2609_35099_b200 import build
    stale = tmp_path / f"_marshal{sysconfig.get_config_var('EXT_SUFFIX')}"
    stale.write_bytes(b"")
    obj = tmp_path / "one.o"
    obj.write_bytes(b"")
    for name, value in dict(PKG=tmp_path, BUILD=tmp_path, OUT=tmp_path / "libe3j.so", sources=lambda: ["one.cu"],
                            _deps_digest=lambda: "", _compile=lambda *args: obj, _link=lambda objs, out: out.write_text("linked")).items():
        monkeypatch.setattr(build, name, value)
    if missing == "torch":
        monkeypatch.setitem(sys.modules, "torch", None)
    else:
        monkeypatch.setenv("PATH", str(tmp_path))
    assert build.build().read_text() == "linked"
    assert not stale.exists() and "the binding converts its arguments in Python" in capsys.readouterr().err


def test_an_integer_parameter_is_not_null():
    """A size query without the list's length is refused with the native call as it is without; a plan that is gone has size 0."""
    import paper_2609_35099_b200 as e3j
    e3j._torch()
    plan = e3j.e3j_plan_create("8x0e", 1)
    for query in (lambda *a: e3j.e3j_conv_bwd_workspace_bytes(plan, *a), lambda *a: e3j.e3j_conv_fwd_workspace_bytes(plan, *a),
                  lambda *a: e3j.e3j_conv_radial_fwd_workspace_bytes(plan, 10, *a)):
        for args in ((None, 20), (10, None)):
            with pytest.raises((TypeError, ctypes.ArgumentError)):
                query(*args)
    assert e3j.e3j_conv_bwd_workspace_bytes(plan, 10, 20) > 0
    e3j.e3j_plan_destroy(plan)
    assert e3j.e3j_conv_bwd_workspace_bytes(plan, 10, 20) == 0
