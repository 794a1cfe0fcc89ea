"""The native marshalling of the decode calls, away from the arithmetic: what it does with tensors that torch refuses
to give an address for."""
import ctypes
import subprocess
import sys
import threading
import time

import pytest
import torch
from torch._subclasses.fake_tensor import FakeTensorMode

import paper_2607_11897_b200 as sfda

ROOT = __file__.rsplit("/tests/", 1)[0]


def decode_tensors(B=1, H=2, d_k=64, d_v=64, device="cuda"):
    f = lambda *shape: torch.empty(*shape, device=device)  # noqa: E731
    return (f(B, H, d_k), f(B, H, d_k), f(B, H, d_v), f(B, H, d_k // 2), f(B, H, d_k // 2), f(B, H)), f(B, H, d_k, d_v), f(B, H, d_v)


def call_with_fake_tensors(fused):
    with FakeTensorMode():
        x, S, o = decode_tensors()
        if fused:
            sfda.sfda_step_fused(*x, 0.0, 1.0, 3.0, 1e-6, S, o, None)
        else:
            sfda.sfda_step(*x, S, o, None)


@pytest.mark.parametrize("fused", [False, True])
def test_tensors_without_storage_raise_a_python_exception(fused):
    """In a process of its own: a C++ exception that leaves the extension would end it."""
    code = ("import tests.test_decode_binding as t\n"
            "try:\n    t.call_with_fake_tensors(%r)\nexcept RuntimeError as e:\n    print('raised')\n" % fused)
    p = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert p.returncode == 0 and "raised" in p.stdout, (p.returncode, p.stdout, p.stderr[-2000:])


SLOW_STEP = """#include <unistd.h>
extern "C" int slow_step(...) { usleep(400000); return 0; }
"""


@pytest.mark.gpu
def test_other_python_threads_run_while_a_call_blocks(tmp_path):
    """A stand-in for a launch that waits for room in the queue: the other thread must not stop meanwhile."""
    from paper_2607_11897_b200 import binding
    (tmp_path / "slow.cpp").write_text(SLOW_STEP)
    subprocess.run(["g++", "-shared", "-fPIC", "-o", str(tmp_path / "slow.so"), str(tmp_path / "slow.cpp")], check=True)
    slow = ctypes.cast(ctypes.CDLL(str(tmp_path / "slow.so")).slow_step, ctypes.c_void_p).value
    x, S, o = decode_tensors()
    sfda.sfda_step(*x, S, o, None)
    ticks, stop = [], threading.Event()

    def count():
        while not stop.wait(0.01):
            ticks.append(time.monotonic())
    thread = threading.Thread(target=count)
    thread.start()
    binding._host.bind(slow, slow)
    try:
        t0 = time.monotonic()
        sfda.sfda_step(*x, S, o, None)
        t1 = time.monotonic()
    finally:
        binding._bind_decode()
        stop.set()
        thread.join()
    assert t1 - t0 >= 0.4
    assert sum(t0 + 0.05 < t < t1 - 0.05 for t in ticks) >= 10, "the other thread stood still during the call"


def in_a_new_process(body):
    code = "import threading\nimport tests.test_decode_binding as t\nfrom paper_2607_11897_b200 import binding\n" + body
    p = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert p.returncode == 0 and "done" in p.stdout, (p.returncode, p.stdout, p.stderr[-2000:])


def test_an_unbound_extension_raises():
    """The extension by itself, before anybody gave it the library's addresses."""
    in_a_new_process("""
host = binding._load_host() if hasattr(binding, "_load_host") else binding._host
x, S, o = t.decode_tensors(device="cpu")
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
class Stream:
    cuda_stream = 0
with FakeTensorMode():
    x, S, o = t.decode_tensors()
    try:
        host.step(*x, S, o, None, Stream())
    except RuntimeError as e:
        assert "bind" in str(e), e
        print("done")
""")


def test_the_first_calls_of_two_threads_both_find_the_library_bound():
    """The second thread calls while the first is still loading the extension."""
    in_a_new_process("""
import time
held, slow = [], threading.Event()
real = binding._load_host
def load_host():
    slow.set()
    time.sleep(0.5)
    return real()
binding._load_host = load_host
def call():
    try:
        t.call_with_fake_tensors(False)
    except RuntimeError as e:
        held.append("bind" not in str(e))
a = threading.Thread(target=call)
a.start()
slow.wait()
b = threading.Thread(target=call)
b.start()
a.join(); b.join()
assert held == [True, True], held
print("done")
""")


def test_a_call_after_a_failed_load_of_the_extension_tries_again():
    in_a_new_process("""
real = binding._load_host
def missing():
    raise ImportError("not there yet")
binding._load_host = missing
for fused in (False, True):
    try:
        t.call_with_fake_tensors(fused)
    except ImportError:
        pass
    else:
        raise AssertionError("no error")
binding._load_host = real
try:
    t.call_with_fake_tensors(True)
except RuntimeError as e:
    assert "bind" not in str(e), e
print("done")
""")


def test_only_the_decode_calls_need_the_extension():
    in_a_new_process("""
from paper_2607_11897_b200 import build
build.HOST = binding.__dict__["_HERE"] + "/no_such_host.so"
binding._load_host = lambda: (_ for _ in ()).throw(ImportError("missing"))
import paper_2607_11897_b200 as sfda
assert sfda.sfda_plan(256, 64) and not build.is_stale() and build.host_is_stale()
print("done")
""")


def test_an_extension_for_another_torch_or_interpreter_is_stale(monkeypatch):
    import torch

    from paper_2607_11897_b200 import build
    build.build()
    assert not build.host_is_stale()
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", "0.0.1")
        assert build.host_is_stale()
    with monkeypatch.context() as m:
        m.setattr(sys, "version", "2.0")
        assert build.host_is_stale()
    assert not build.host_is_stale()
