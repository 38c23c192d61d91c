"""The native half of the binding: what torch throws while arguments are read becomes a Python error.

The calls are made in a child process, because an exception that leaves through the interpreter's C frames ends the
process.  No context and no GPU: the arguments are read, and refused, before anything is called.
"""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import torch
from paper_2410_20046_b200.binding import load_native

native = load_native()

def host_step(grad=None, lr=0.1, stream=None):
    # train_step_host(ctx, tables, h_indices, h_offsets, h_grad_out, scales, bits, h_out, lr, B, L, ws, bytes, stream)
    return native.train_step_host(0, None, None, None, grad, None, None, None, lr, 1, 1, 0, 0, stream)

def raises(call, kinds=RuntimeError):
    try:
        call()
    except kinds as e:
        print("raised", type(e).__name__, flush=True)
        return
    raise SystemExit("no error")

class Stream:
    cuda_stream = 0
"""

CASES = {
    # a tensor inside vmap has no data pointer
    "vmap": "raises(lambda: torch.vmap(lambda x: (host_step(x, stream=Stream()), x)[1])(torch.zeros(3, 4)))",
    # a sparse tensor has no strides to ask about
    "sparse": "raises(lambda: host_step(torch.eye(3).to_sparse(), stream=Stream()), (RuntimeError, AssertionError))",
    # the current stream where there is no device
    "stream": "raises(host_step) if not torch.cuda.is_available() else print('raised nothing: a device is there')",
    # what Python's own float() takes, the rate may be (the C ABI then refuses the null context)
    "rate": "assert host_step(lr='0.25', stream=Stream()) == -1 and host_step(lr=torch.tensor(0.5), stream=Stream()) == -1; print('raised')",
    "no_rate": "raises(lambda: host_step(lr=None, stream=Stream()), TypeError)",
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_native_calls_raise_and_do_not_abort(case):
    r = subprocess.run([sys.executable, "-c", PRELUDE + CASES[case]], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "raised" in r.stdout, (r.returncode, r.stdout, r.stderr[-2000:])


def test_native_module_is_rebuilt_for_another_torch_or_python(monkeypatch):
    """Dates alone say nothing of a module that another torch was installed under."""
    from paper_2410_20046_b200 import build

    build.build()
    assert not build._native_stale()
    monkeypatch.setattr(build, "_native_for", lambda: "python cpython-399 torch 9.9\n")
    assert build._native_stale()
