"""The device memory that the library keeps between calls, on a device whose
other memory is taken: what it keeps is there for all of its own allocations
(a served job's among them), and a repeated call gets the kernel-row cache
that the first one got."""
import numpy as np
import pytest

import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

MiB = 1 << 20


def _keep_some():
    """An FP64 batch whose kernel rows (2.4 GB) the pool keeps when it ends."""
    p = synth.small_dense(5500, 8, seed=1, sep=0.5)
    pkg.svm_train_batch(p.X, [{"y": p.y, "C": 1.0, "gamma": 0.1, "max_iter": 60}] * 10, cluster_size=8, lanes_per_row=1)


class _Filled:
    """All of the device's free memory but `leave` bytes is taken."""

    def __init__(self, leave):
        self.leave = leave

    def __enter__(self):
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        self.t = torch.empty(max(0, free - self.leave), dtype=torch.uint8, device="cuda")

    def __exit__(self, *exc):
        self.t = None
        torch.cuda.empty_cache()


def test_served_job_takes_the_memory_that_is_kept():
    n, d = 30000, 1500
    rng = np.random.default_rng(2)
    X = synth.CSR(n, d, np.arange(0, n * d + 1, d, dtype=np.int64), np.tile(np.arange(d, dtype=np.int32), n),
                  rng.random(n * d, dtype=np.float32))
    y = np.where(np.arange(n) % 2 == 0, 1, -1).astype(np.int8)
    with pkg.Server(budget_bytes=4 << 30, max_d=1504) as srv:
        small = synth.small_dense(200, 8, seed=1)
        assert srv.wait(srv.submit(small.X, small.y, 1.0, 0.1))["status"] == pkg.SVM_OK
        _keep_some()
        with _Filled(400 * MiB):   # the job needs 640 MB
            out = srv.wait(srv.submit(X, y, 1.0, 1e-3, max_iter=5), timeout=30.0)
    assert out is not None and out["status"] == pkg.SVM_NOT_CONVERGED


def test_repeated_call_gets_the_same_cache():
    p = synth.small_dense(20000, 8, seed=3, sep=0.5)
    X, y = pkg.to_device(p.X), torch.as_tensor(p.y, device="cuda")
    with _Filled(6 << 30):
        slots = [pkg.svm_train(X, y, 1.0, 0.1, 1e-3, max_iter=100)["stats"]["cache_slots"] for _ in range(3)]
    assert slots[0] > 0 and slots == [slots[0]] * 3, slots


def test_trim_gives_the_kept_memory_back():
    _keep_some()
    torch.cuda.synchronize()
    before, _ = torch.cuda.mem_get_info()
    pkg.svm_trim_memory()
    after, _ = torch.cuda.mem_get_info()
    assert after - before >= 2 << 30, (before, after)
    p = synth.small_dense(300, 8, seed=1)   # and the library goes on
    assert pkg.svm_train(p.X, p.y, 1.0, 0.1, 1e-3)["status"] == pkg.SVM_OK
