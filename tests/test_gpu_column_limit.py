"""The largest number of columns that the solvers accept (their target rows
fill shared memory): a solve there runs and has the multipliers of the same
rows in few columns, and one column more is refused with an error. Sparse
rows whose columns are moved to the far end, so nothing else changes; the
results are compared bit for bit."""
import numpy as np
import pytest

import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)


def _rows(kind, d):
    rng = np.random.default_rng(1)
    n, k = 48, 4
    cols = np.sort(np.stack([rng.choice(12, k, replace=False) for _ in range(n)]), 1).astype(np.int32) + d - 12
    vals = None if kind == "binary" else rng.uniform(0.5, 1.5, n * k).astype(np.float32)
    y = np.where(rng.random(n) < 0.5, 1, -1).astype(np.int8)
    return synth.CSR(n, d, np.arange(0, n * k + 1, k, dtype=np.int64), cols.reshape(-1), vals), y


def _solve(entry, kind, d):
    X, y = _rows(kind, d)
    prec = pkg.SVM_MIXED_BF16_SIMT if kind == "mixed" else pkg.SVM_FP64
    if entry == "train":
        r = pkg.svm_train(X, y, 2.0, 0.1, 1e-3, precision=prec)
    else:
        r = pkg.svm_train_batch(X, [{"y": y, "C": 2.0, "gamma": 0.1}], precision=prec, cluster_size=2, lanes_per_row=1)["results"][0]
    return r["iters"], r["alpha"]


# the limits of the first library that had these entry points
LIMITS = {("train", "fp64"): 6743, ("train", "mixed"): 13358, ("train", "binary"): 54400,
          ("batch", "fp64"): 6878, ("batch", "mixed"): 9404, ("batch", "binary"): 54968}


@pytest.mark.parametrize("entry,kind", sorted(LIMITS))
def test_solves_at_the_largest_column_count(entry, kind):
    d = LIMITS[entry, kind]
    it, a = _solve(entry, kind, d)
    it0, a0 = _solve(entry, kind, 64)
    assert it == it0 and np.array_equal(a, a0)
    with pytest.raises(pkg.SvmError):
        _solve(entry, kind, d + 1)
