"""The one-cluster solve against the same solve with streamed rows (which takes
the several-cluster exchange, target rows from global memory and one lane per
row): the same steps and multipliers bit for bit, at the sizes where the
one-cluster row pass changes its shape (16 segments of at most 240 rows take a
lane pair per row) and with the kernel-row cache on and off."""
import numpy as np
import pytest

import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("n", [512, 513, 3825, 3840, 3841, 3857, 6000])
@pytest.mark.parametrize("precision,cache_mb", [("FP64", 0), ("FP64", -1), ("MIXED_BF16", 0), ("MIXED_BF16", 64)])
def test_one_cluster_equals_streamed(n, precision, cache_mb):
    p = synth.covtype_like(n=n, n_test=0, seed=n)
    prec = getattr(pkg, "SVM_" + precision)
    kw = dict(precision=prec, shrink=pkg.POLICIES["Multi500"], cache_mb=cache_mb, trace_len=400, max_iter=6000)
    a = pkg.svm_train(p.X, p.y, p.C, p.gamma, p.tau, **kw)
    b = pkg.svm_train(p.X, p.y, p.C, p.gamma, p.tau, flags=pkg.SVM_FLAG_STREAM_ROWS, **kw)
    assert a["stats"]["resident"] == 1 and b["stats"]["resident"] == 0
    assert a["iters"] == b["iters"] and np.array_equal(a["trace"], b["trace"])
    assert np.array_equal(a["alpha"], b["alpha"]) and a["b"] == b["b"]
    assert a["stats"]["row_visits"] == b["stats"]["row_visits"]


@pytest.mark.parametrize("n", [512, 3841])
def test_ragged_rows_with_empty_ones(n):
    p = synth.random_sparse(n=n, d=90, density=0.08, seed=n)
    a = pkg.svm_train(p.X, p.y, p.C, p.gamma, p.tau, trace_len=300)
    b = pkg.svm_train(p.X, p.y, p.C, p.gamma, p.tau, trace_len=300, flags=pkg.SVM_FLAG_STREAM_ROWS)
    assert np.array_equal(a["trace"], b["trace"]) and np.array_equal(a["alpha"], b["alpha"])


@pytest.mark.parametrize("d", [32, 64, 100, 200])
@pytest.mark.parametrize("n", [530, 3840, 4100])
def test_row_tiles_on_chip_equal_streamed_ones(n, d):
    # one and two tiles per warp, rows on chip, on chip without their dense
    # copy (d = 200, the larger sizes) and from L2
    p = synth.small_dense(n, d, seed=n + d, sep=0.15, C=2.0, gamma=1.0 / d)
    kw = dict(precision=pkg.SVM_MIXED_BF16, shrink=pkg.POLICIES["Multi500"], trace_len=300, max_iter=3000)
    a = pkg.svm_train(p.X, p.y, p.C, p.gamma, p.tau, flags=pkg.SVM_FLAG_TENSOR_ROWS, **kw)
    b = pkg.svm_train(p.X, p.y, p.C, p.gamma, p.tau, flags=pkg.SVM_FLAG_TENSOR_ROWS | pkg.SVM_FLAG_STREAM_ROWS, **kw)
    assert a["stats"]["row_tiles"] == b["stats"]["row_tiles"] == 1 and b["stats"]["resident"] == 0
    assert a["iters"] == b["iters"] and np.array_equal(a["trace"], b["trace"])
    assert np.array_equal(a["alpha"], b["alpha"]) and a["b"] == b["b"]
