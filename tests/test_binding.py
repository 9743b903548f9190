"""The Python binding's argument conversion, on tensors without storage (no GPU needed)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Fake CUDA tensors: they have a device, sizes and a type, and nothing behind them.
PRELUDE = """
import ctypes, sys, torch
import paper_1603_05279_b200 as X
from paper_1603_05279_b200 import binding as B
from torch._subclasses.fake_tensor import FakeTensorMode
X.load()
real = torch.zeros(4, 4, 3, 3)
fake = lambda *s, dtype=torch.float32: torch.empty(s, device="cuda", dtype=dtype)
w, wp, al = (4, 4, 3, 3), (9, 4, 2), (4,)
def args():
    return fake(*w), fake(*wp, dtype=torch.int32), fake(*al)
def raises(kind, call):
    try:
        call()
    except kind:
        return
    raise SystemExit("no " + str(kind))
"""


# xnor_binarize_weights_transposed replaced by a function that records what the native module passes.
RECORD = """
seen = []
vp, ci = ctypes.c_void_p, ctypes.c_int
entry = ctypes.CFUNCTYPE(ci, vp, ci, ci, ci, ci, vp, vp)(lambda *a: seen.append(a) or 0)
addresses = [ctypes.cast(getattr(X.load(), "xnor_" + n), vp).value for n in B._MARSHALLED]
addresses[B._MARSHALLED.index("binarize_weights_transposed")] = ctypes.cast(entry, vp).value
B._m.bind(addresses, X.xnor_conv_desc, B._address)
"""


def run_child(body, prelude=PRELUDE):
    """In a process of its own: what is tested for is that the interpreter survives."""
    code = prelude + "with FakeTensorMode(allow_non_fake_inputs=True):\n" + \
        "".join("    %s\n" % line for line in body.strip().splitlines())
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout[-500:], r.stderr[-2000:])


@pytest.mark.parametrize("body", [
    # no data pointer: under vmap, under vjp
    """
a, p, al = args()
f = lambda x, y: (X.xnor_maxpool2d(x, 2, 2, 0, False, y, stream=0), x)[1]
raises(RuntimeError, lambda: torch.vmap(f)(fake(5, 2, 3, 8, 8), fake(5, 2, 3, 4, 4)))
raises(RuntimeError, lambda: torch.func.vjp(lambda x: (X.xnor_binarize_weights(x, p, al, stream=0), x)[1], a))
""",
    # the size read beside the pointers
    """
f = lambda y: (X.xnor_shortcut_conv1x1(fake(2, 3, 8, 8), y, 2, fake(2, 4, 4, 4), stream=0), y)[1]
raises(RuntimeError, lambda: torch.vmap(f)(fake(5, 4, 3)))
""",
], ids=["pointer", "size"])
def test_torch_exceptions_reach_python(body):
    run_child(body)


def test_stream_arguments():
    """A torch stream or what int() takes (cuda-python's handles, numpy's integers); an attribute that
    fails for another reason than being absent is reported as it is."""
    run_child("""
import numpy
class Torch: cuda_stream = 0x7000
class Handle:
    def __int__(self): return 0x8000
class Broken:
    @property
    def cuda_stream(self): raise RuntimeError("lost")
a, p, al = args()
for s in (Torch(), Handle(), numpy.int64(0x9000), 0xA000, 0): X.xnor_binarize_weights_transposed(a, p, stream=s)
assert [x[-1] for x in seen] == [0x7000, 0x8000, 0x9000, 0xA000, None], seen
raises(RuntimeError, lambda: X.xnor_binarize_weights_transposed(a, p, stream=Broken()))
raises(TypeError, lambda: X.xnor_binarize_weights_transposed(a, p, stream=object()))
assert len(seen) == 5
""", PRELUDE + RECORD)


def test_descriptor_arguments():
    """An xnor_conv_desc (or a subclass): not another structure, or bytes, of its size."""
    run_child("""
class Other(ctypes.Structure): _fields_ = X.xnor_conv_desc._fields_
class Derived(X.xnor_conv_desc): pass
d = X.make_desc(1, 8, 5, 5, 4, 3, 3, 1, 1)
call = lambda d: X.xnor_binactiv(fake(1, 8, 5, 5), None, None, d, fake(25, dtype=torch.int32), fake(25), fake(25), stream=0)
for bad in (bytes(d), bytearray(bytes(d)), Other(), None, 3): raises(TypeError, lambda: call(bad))
raises(X.XnorError, lambda: call(Derived()))                 # converted; the library refuses its zeros
""")


def test_tensor_subclasses_and_lookalikes():
    """What a subclass, or an object with a tensor's attributes, says of itself counts."""
    run_child("""
class Sub(torch.Tensor):
    is_cuda = True
    def data_ptr(self): return 0x1000
class Like:
    is_cuda, dtype, device, shape = True, torch.int32, "cuda", (9, 4, 2)
    def is_contiguous(self): return True
    def data_ptr(self): return 0x2000
sub = real.as_subclass(Sub)
X.xnor_binarize_weights_transposed(sub, Like(), stream=0)
assert seen == [(0x1000, 4, 4, 3, 3, 0x2000, None)], seen
raises(ValueError, lambda: X.xnor_binarize_weights_transposed(Like(), sub, stream=0))       # three dimensions
raises(ValueError, lambda: X.xnor_binarize_weights_transposed(sub, sub, stream=0))          # not int32
raises(AttributeError, lambda: X.xnor_binarize_weights_transposed(sub, 3, stream=0))
raises(AttributeError, lambda: X.xnor_binarize_weights_transposed(None, Like(), stream=0))
""", PRELUDE + RECORD)


def test_load_order():
    """After any instruction of load(), a thread that finds the library loaded finds the native module too."""
    run_child("""
B._lib, B._m = None, B._Unloaded()
states = set()
def watch(frame, event, arg):
    if frame.f_code is not B.load.__code__: return None
    if event == "call":
        frame.f_trace_opcodes = True
        sys.settrace(watch)                  # Python 3.12 instruments the instructions from here on
    states.add((B._lib is not None, not isinstance(B._m, B._Unloaded)))
    return watch
sys.settrace(watch)
X.load()
sys.settrace(None)
assert (True, True) in states and (False, False) in states and (True, False) not in states, states
""")
