"""A model on the device against svm_decision on the same rows, where the
queries alone do not tell the arithmetic's format: few FP64 queries whose
values span fewer binades than the support vectors', and binary support
vectors (with and without stored ones) with queries that are not, and the
other way round. svm_decision's values bit for bit, and the oracle's within
the sum's rounding (FP64: nsv 2^-50 sum |alpha|; mixed: the BF16 rounding of
the values, gamma 2^-6 (|x|^2 + |z|^2) per term)."""
import numpy as np
import pytest

import oracle
import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)


def _alpha(n, C):
    rng = np.random.default_rng(n)
    a = np.where(rng.random(n) < 0.5, C, rng.uniform(0.0, C, n))
    a[rng.random(n) < 0.3] = 0.0
    return a


@pytest.mark.parametrize("m", [1, 3, 8])
def test_few_fp64_queries(m):
    p = synth.covtype_like(n=3000, n_test=m, seed=5)
    a = _alpha(3000, p.C)
    want = pkg.svm_decision(p.X, p.y, a, 0.25, p.gamma, p.Z)
    ref = oracle.decision(p.X, p.y, a, 0.25, p.gamma, p.Z)
    with pkg.Model(p.X, p.y, a, 0.25, p.gamma) as mod:
        got = mod.decision(p.Z)
    assert np.array_equal(got, want)
    assert np.abs(got - ref).max() <= 3000 * 2.0 ** -50 * a.sum()


@pytest.mark.parametrize("precision", [pkg.SVM_FP64, pkg.SVM_MIXED_BF16, pkg.SVM_MIXED_BF16_SIMT])
@pytest.mark.parametrize("binary_side", ["x", "x-no-values", "z"])
def test_one_side_binary(precision, binary_side):
    n, m, d = 700, 40, 60
    b = synth.random_sparse(n=n + m, d=d, density=0.2, seed=1, binary=True)
    v = synth.random_sparse(n=n + m, d=d, density=0.2, seed=2)
    bx = binary_side != "z"
    X = (b if bx else v).X.take(np.arange(n))
    Z = (v if bx else b).X.take(np.arange(n, n + m))
    y, gamma = b.y[:n], 0.1
    a = _alpha(n, 1.0)
    Xc = synth.CSR(X.n, X.d, X.indptr, X.indices, None) if binary_side == "x-no-values" else X
    want = pkg.svm_decision(Xc, y, a, 0.25, gamma, Z, precision=precision)
    with pkg.Model(Xc, y, a, 0.25, gamma, precision=precision) as mod:
        got = mod.decision(Z)
        assert np.array_equal(mod.decision(Z), got)
    assert np.array_equal(got, want)
    ref = oracle.decision(X, y, a, 0.25, gamma, Z)
    if precision == pkg.SVM_FP64:
        bound = n * 2.0 ** -50 * a.sum()
    else:
        sq = lambda M: np.array([float((M.values[s:e].astype(np.float64) ** 2).sum())  # noqa: E731
                                 for s, e in zip(M.indptr[:-1], M.indptr[1:])])
        bound = (a[None, :] * gamma * 2.0 ** -6 * (sq(Z)[:, None] + sq(X)[None, :])).sum(1)
    assert np.all(np.abs(got - ref) <= bound)
