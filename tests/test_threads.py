"""Other Python threads run while a device entry point is under way: the C function behind it may wait (a full
launch queue, or the stream in checked mode).

No GPU is needed: the marshalling module is bound to ``sem_wait`` in place of the library, which blocks on its
first argument -- the descriptor, here the memory of a semaphore -- until another thread posts it.  Child process:
the binding is process-wide, and a call that kept the interpreter lock would never come back."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, sys, threading, time
import torch
from paper_1905_10138_b200 import _sqnn_python as mod, sqnn

libc = ctypes.CDLL(None)
mod.bind(*[ctypes.cast(libc.sem_wait, ctypes.c_void_p).value] * 3)


class Stream:
    cuda_stream = 0


x, y = torch.zeros((16, 8), dtype=torch.bfloat16), torch.zeros((16, 4))
desc = sqnn.Desc()
calls = {
    "decode": lambda: mod.decode(desc, None, None, None, sqnn.OUT_BITS, None, None, Stream()),
    "matmul": lambda: mod.matmul(desc, None, None, None, x, y, None, None, Stream()),
    "matmul_static": lambda: mod.matmul_static(desc, None, None, None, x, y, None, Stream()),
}
libc.sem_init(ctypes.byref(desc), 0, 0)
results = []
t = threading.Thread(target=lambda: results.append(calls[sys.argv[1]]()))
t.start()
time.sleep(0.3)                                  # the thread is inside sem_wait by now
assert t.is_alive() and not results
libc.sem_post(ctypes.byref(desc))
t.join(10)
assert results == [0], results
print("other threads ran")
"""


@pytest.mark.parametrize("entry", ["decode", "matmul", "matmul_static"])
def test_a_call_that_waits_leaves_the_interpreter_to_other_threads(entry):
    env = dict(os.environ, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD, entry], env=env, cwd=ROOT, capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "other threads ran" in r.stdout
