"""Calls from threads that come and go while a server's engine kernel runs: no
call waits for the engine (it runs for as long as its jobs do), and values are
those of the main thread."""
import threading
import time

import numpy as np
import pytest

import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)


def test_new_threads_do_not_wait_for_the_engine():
    p = synth.covtype_like(n=2000, n_test=8, seed=3)
    X, y, Z = pkg.to_device(p.X), torch.as_tensor(p.y, device="cuda"), pkg.to_device(p.Z)
    a = torch.full((2000,), 0.5, dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()

    def call():
        t0 = time.perf_counter()
        v = pkg.svm_decision(X, y, a, 0.1, 0.1, Z, stream=side, precision=pkg.SVM_MIXED_BF16_SIMT)
        return time.perf_counter() - t0, v

    call()
    want = call()[1]
    # a job of some seconds, ended by its step limit
    q = synth.small_dense(30000, 200, seed=1, sep=0.05, gamma=0.005, C=10.0)
    with pkg.Server(budget_bytes=2 << 30, max_d=208, cluster_size=8) as srv:
        ticket = srv.submit(q.X, q.y, q.C, q.gamma, 1e-3, max_iter=60000)
        while srv.stats()["running"] == 0:
            time.sleep(0.01)
        done = []   # (compared after the job: other libraries' first launches do wait)
        for group in (1, 1, 1, 3):   # one after another, then three at once
            out = []
            threads = [threading.Thread(target=lambda: out.append((call(), call()))) for _ in range(group)]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            done += [v for pair in out for v in pair]
        still = srv.stats()["running"]
        res = srv.wait(ticket)
    took = [v[0] for v in done]
    assert still == 1 and len(took) == 12 and max(took) < 0.5, (still, took)
    assert all(torch.equal(v[1], want) for v in done)
    assert res["status"] == pkg.SVM_NOT_CONVERGED and np.isfinite(res["alpha"]).all()
