"""The binding's native argument path, on the CPU: what it does not take is raised by the Python path behind it."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Each case ends in an error of torch's, the binding's or the library's.  They run in a child process: a C++ exception that leaves a C
# function ends the interpreter.
ODD_TENSORS = """
import sys, torch, paper_2608_30310_b200 as gdn
gdn.load_library()
T, H, D = 8, 2, 64
q, k, v = (torch.zeros(T, H, D) for _ in range(3))
g, beta = torch.zeros(T, H), torch.zeros(T, H)
cu = torch.tensor([0, T], dtype=torch.int32)

def static(q=q, k=k, v=v, g=g, beta=beta, cu=cu, o=None):
    gdn.gdn_tail_replay_static_scratch(q, k, v, g, beta, cu, 64, o, None)

def nested():
    n = torch.nested.nested_tensor([torch.zeros(3, D), torch.zeros(5, D)])
    gdn.gdn_tail_replay(n, k, v, g, beta, cu, 64, None, None)

def sparse():
    static(q=q.to_sparse(), k=k.to_sparse(), v=v.to_sparse())

def fake():
    from torch._subclasses.fake_tensor import FakeTensorMode
    with FakeTensorMode():
        x = torch.empty(T, H, D)
        static(x, x, x, torch.empty(T, H), torch.empty(T, H), torch.empty(2, dtype=torch.int32))

def fake_decode():
    from torch._subclasses.fake_tensor import FakeTensorMode
    with FakeTensorMode():
        x, s = torch.empty(T, H, D, device="cuda"), torch.empty(T, H, D, D, device="cuda")
        y = torch.empty(T, H, device="cuda")
        gdn.gdn_decode_step(x, x, x, y, y, s, x, s)

def vmap():
    torch.func.vmap(lambda x: static(x, x, x) or x)(torch.zeros(3, T, H, D))

def host_memory():
    static()                                   # no driver: no current stream; with one: the entry takes device memory only

try:
    {case}()
except (RuntimeError, ValueError):
    print("raised")
"""


@pytest.mark.parametrize("case", ["nested", "sparse", "fake", "fake_decode", "vmap", "host_memory"])
def test_tensors_without_sizes_or_storage_raise(case):
    r = subprocess.run([sys.executable, "-c", ODD_TENSORS.replace("{case}", case)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.strip() == "raised", r.stdout + r.stderr[-2000:]


# PyGILState_Check stands in for the library's entry points: it answers whether its thread holds the interpreter lock (1) or not (0,
# which is also GDN_OK).
LOCK = """
import ctypes, torch, paper_2608_30310_b200 as gdn
from paper_2608_30310_b200 import _binding as B
gdn.load_library()
check = ctypes.cast(ctypes.pythonapi.PyGILState_Check, ctypes.c_void_p).value
size = ctypes.cast(gdn.load_library().gdn_workspace_size, ctypes.c_void_p).value
B._native.bind(check, check, check, check, size, gdn.Workspace)
class Stream: cuda_stream = 0
x, y = torch.zeros(8, 2, 64), torch.zeros(8, 2)
cu = torch.tensor([0, 8], dtype=torch.int32)
print(B._native.forward(2, x, x, x, y, y, cu, 64, x, None, None, None, None, 0, Stream(), False))
if torch.cuda.is_available():
    x, y, s = x.cuda(), y.cuda(), torch.zeros(8, 2, 64, 64, device="cuda")
    print(B._native.decode(x, x, x, y, y, s, x, s, Stream()))
"""


def test_the_library_is_called_without_the_interpreter_lock():
    r = subprocess.run([sys.executable, "-c", LOCK], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert set(r.stdout.split()) == {"0"}, r.stdout


@pytest.mark.parametrize("name,value", [("init_state", "torch.zeros(1, 2, 64, 63)"), ("init_state", "torch.zeros(1, 2, 64, 64).double()"),
                                        ("status_word", "torch.zeros(1, dtype=torch.int16)"), ("status_word", "torch.zeros(1, dtype=torch.int32)")])
def test_start_state_and_status_word_are_checked(name, value):
    """Too short, of another type, or not for the device to write (host memory that is not pinned)."""
    import torch
    import paper_2608_30310_b200 as gdn
    x, y, cu = torch.zeros(8, 2, 64), torch.zeros(8, 2), torch.tensor([0, 8], dtype=torch.int32)
    with pytest.raises(ValueError, match=name):
        gdn.gdn_tail_replay_static_scratch(x, x, x, y, y, cu, 64, None, None, **{name: eval(value)})


class _Stream:
    def __init__(self, handle):
        self.cuda_stream = handle


def test_every_stream_has_a_buffer_of_its_own(monkeypatch):
    import contextlib
    import paper_2608_30310_b200 as gdn
    from paper_2608_30310_b200 import _binding as B
    entered = []
    monkeypatch.setattr(B, "_on_stream", lambda s: entered.append(s.cuda_stream) or contextlib.nullcontext())
    ws = gdn.Workspace(device="cpu")
    a = ws.reserve(512, _Stream(0))
    b = ws.reserve(512, _Stream(7))
    assert entered == [0, 7] and a.data_ptr() != b.data_ptr()                  # allocated for the stream that uses it
    assert ws.reserve(500, _Stream(7)) is b and ws.buf is a and len(entered) == 2
    ring = ws.reserve(9 << 20, _Stream(7))
    assert ring.numel() >= 12 << 20 and ws.by_stream == {0: a, 7: ring}
    assert any(x is b for x in ws.outgrown)                                    # (a captured call may have its address)
    big = ws.reserve(30 << 20, _Stream(7))
    assert any(x is ring for x in ws.outgrown) and ws.reserve(1 << 20, _Stream(7)) is big
    ws.reserve(60 << 20, _Stream(7))
    assert not any(x is big for x in ws.outgrown)                              # staging of host-memory calls is given back
    base, size = ws.ensure(512, _Stream(0))
    assert base % 256 == 0 and a.data_ptr() <= base and base + size == a.data_ptr() + a.numel()


OTHER_TORCH = """
import sys, types, warnings, torch, paper_2608_30310_b200 as gdn
from paper_2608_30310_b200 import _binding as B
ext = {ext}
sys.modules["paper_2608_30310_b200._native"] = ext
if ext is not None: gdn._native = ext
with warnings.catch_warnings(record=True) as seen:
    warnings.simplefilter("always")
    assert gdn.tail_select(100, 0.07) == 7
assert any("native argument path" in str(w.message) for w in seen)
x, y = torch.zeros(8, 2, 64), torch.zeros(8, 2)
class Stream: cuda_stream = 0
try:
    gdn.gdn_tail_replay_static_scratch(x, x, x, y, y, torch.tensor([0, 8], dtype=torch.int32), 64, None, None, stream=Stream())
except gdn.GdnError as e:
    print(e.status)
try:
    gdn.gdn_decode_step(x, x, x, y, y, x, None, x)
except ValueError:
    print("checked")
"""


@pytest.mark.parametrize("ext", ["types.SimpleNamespace(built_for_torch='1.0')", "types.SimpleNamespace()", "None"])
def test_an_extension_for_another_torch_is_not_used(ext):
    """The library still loads and the Python path takes the calls (host memory: unsupported by that entry, -2)."""
    r = subprocess.run([sys.executable, "-c", OTHER_TORCH.replace("{ext}", ext)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["-2", "checked"], r.stdout + r.stderr[-2000:]
