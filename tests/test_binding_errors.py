"""Errors on the tensor side of the binding, without a GPU: library functions stand in that return success, so that what
torch raises around them shows.  In a child process: a mistake here ends the interpreter."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = r"""
import ctypes as C, sys
sys.path.insert(0, %r)
import torch
from paper_2609_36601_b200 import binding as B
lib = B.load_library()
ran = []
@C.CFUNCTYPE(C.c_int, C.c_void_p, C.c_int, C.c_int, *[C.c_void_p] * 5, C.c_float, C.c_void_p, C.c_void_p, C.c_int, C.c_void_p)
def stage(*a):
    ran.append(a[2])
    return 0
def bind(**functions):
    at = {f: C.cast(functions.get(f, getattr(lib, f)), C.c_void_p).value for f in B._BOUND}
    B._fast.bind(B.SakiError, *(at[f] for f in B._BOUND))
""" % ROOT


def _child(text):
    r = subprocess.run([sys.executable, "-c", HEAD + text], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, (r.returncode, r.stdout[-500:], r.stderr[-2000:])


def test_an_error_while_the_interpreter_lock_is_released():
    """Reading the counters of the sharded stages may raise (here: a tensor without data; in earnest a CUDA error or an
    allocation that fails) while the interpreter lock is released: it has to be taken again before the error is reported."""
    _child(r"""
bind(saki_vshard_stage=stage)
s = torch.zeros(3, 8, dtype=torch.bfloat16, device="meta")
x = torch.zeros(3, dtype=torch.int32, device="meta")
for _ in range(3):
    try:
        B._fast.vshard_local([(s, s, 0)], 8, x, 0.1, 1.0, 0, 0, None, 1.0, False, 1234, 2, 5)
        raise SystemExit("no error")
    except RuntimeError as e:
        assert "meta" in str(e), e
assert ran == [0, 1, 1] * 3, ran
print("done")
""")


def test_torch_errors_keep_their_types():
    """An index error, an allocation that fails and a tensor without data are the exceptions that torch makes of them."""
    _child(r"""
def raises(kind, f, *a):
    try:
        f(*a)
    except Exception as e:
        assert type(e) is kind, (type(e), e)
        assert "frame #" not in str(e), e          # no C++ stack in the text
    else:
        raise SystemExit("no error")
u8 = torch.zeros(3, dtype=torch.uint8)
raises(IndexError, B.select_tm, torch.tensor(3), u8, None, 0)
raises(IndexError, B._fast.propose, torch.zeros(3), 1.0, 0, 0, 1234)           # one dimension of two
bind(saki_vshard_stage=stage)
s = torch.zeros(3, 8, dtype=torch.bfloat16, device="meta")
raises(NotImplementedError, B._fast.vshard_local, [(s, s, 0)], 8, s, 0.1, 1.0, 0, 0, None, 1.0, False, 1234, 2, 5)
raises(B.SakiError, B.route_fwd, torch.zeros(2, 3), torch.zeros(2, 4), u8, 0.1)
raises(TypeError, B.route_fwd, [1], torch.zeros(2, 4), u8, 0.1)
print("done")
""")


@pytest.mark.gpu
def test_out_of_memory_keeps_its_type():
    import torch
    import paper_2609_36601_b200 as P
    with pytest.raises(torch.OutOfMemoryError):
        P.alloc_outputs(1 << 42, "cuda:0")             # 16 TB
    P.alloc_outputs(16, "cuda:0")
