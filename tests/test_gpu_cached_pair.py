"""The pair step's K(up, low) read from the kernel-row cache on one cluster,
where another CTA stored it, often in the step before: the solve is that of
the same call without a cache bit for bit, in every repetition. Both
directories (a slot per row, and sets of four) and the row passes that store:
a lane pair per row, and a lane per row for segments of more than 240."""
import numpy as np
import pytest

import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("n", [512, 600, 1500, 4000])
@pytest.mark.parametrize("cache_mb", [0, 2])
def test_cached_pair_value_is_the_computed_one(n, cache_mb):
    p = synth.gaussian_mixture(n=n, n_test=0, seed=n)
    X, y = pkg.to_device(p.X), torch.as_tensor(p.y, device="cuda")
    kw = dict(trace_len=4000, max_iter=20000)
    off = pkg.svm_train(X, y, 8.0, p.gamma, p.tau, cache_mb=-1, **kw)
    assert off["stats"]["cluster_size"] == off["stats"]["ctas"]   # one cluster
    for _ in range(4):
        on = pkg.svm_train(X, y, 8.0, p.gamma, p.tau, cache_mb=cache_mb, **kw)
        assert on["stats"]["cache_hits"] > 0
        assert on["iters"] == off["iters"] and np.array_equal(on["trace"], off["trace"])
        assert torch.equal(on["alpha"], off["alpha"]) and on["b"] == off["b"]
