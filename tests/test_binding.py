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


def run_child(body):
    """In a process of its own: what is tested for is that the interpreter survives."""
    code = PRELUDE + "with FakeTensorMode(allow_non_fake_inputs=True):\n" + \
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
