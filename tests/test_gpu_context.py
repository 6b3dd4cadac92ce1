"""The library goes on after the process resets its own device context, as a
caller does between two independent parts of a program: what it keeps between
calls (its memory pool, page-locked result buffers) belongs to the context
that was current then. In a process of its own; nothing runs on the device
while the context is reset."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import ctypes
import numpy as np
import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth
p = synth.covtype_like(n=700, n_test=50, seed=1)
a = np.full(700, 0.5)

def calls():
    r = pkg.svm_train(p.X, p.y, p.C, p.gamma, p.tau)
    return [r["alpha"]] + [pkg.svm_decision(p.X, p.y, a, 0.1, p.gamma, p.Z, precision=q)
                           for q in (pkg.SVM_FP64, pkg.SVM_MIXED_BF16)]

first = calls()
assert ctypes.CDLL("libcuda.so.1").cuDevicePrimaryCtxReset_v2(0) == 0
again = calls()
assert all(np.array_equal(x, y) for x, y in zip(first, again))
print("same")
"""


def test_calls_after_a_context_reset():
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "same", (r.returncode, r.stdout, r.stderr[-2000:])
