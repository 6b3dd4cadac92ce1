"""The decision contraction at the sizes where its work is cut differently: a
few queries (two to a tile, support vectors split over many CTAs), sizes around
the tiles (2, 8, 16, 128 queries) and around the split's smallest share, more
queries than the split needs; FP64, binary, mixed on CUDA cores and on the
tensor cores. Reference: the FP64 oracle.

Bounds: FP64 and binary, sums of nsv terms of at most C with kernel values
within one unit in the last place, (nsv + 4) 2^-53 sum |coef|; mixed, BF16
rounding of the values (2^-8 relative each, so at most 2^-7 of |x||z| in the
inner product): |dK| <= gamma (4 2^-8 (|x|^2 + |z|^2)) on every term."""
import numpy as np
import pytest

import oracle
import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

CASES = [(1, 5), (2, 255), (3, 257), (7, 1024), (8, 1025), (9, 3000), (17, 600), (127, 1300), (129, 1000), (400, 2500)]


def _alpha(n, C):
    rng = np.random.default_rng(n)
    a = np.where(rng.random(n) < 0.7, C, rng.uniform(0.0, C, n))
    a[rng.random(n) < 0.3] = 0.0
    a[:2] = C
    return a


@pytest.mark.parametrize("m,n", CASES)
@pytest.mark.parametrize("kind", ["fp64", "binary", "binary200", "simt", "mixed"])
def test_decision_against_the_oracle(m, n, kind):
    if kind == "binary200":   # masks of eight words, ragged rows
        p = synth.random_sparse(n=n + m, d=200, density=0.08, seed=n, binary=True)
        p.Z, p.X, p.y = p.X.take(np.arange(n, n + m)), p.X.take(np.arange(n)), p.y[:n]
    else:
        p = synth.onehot_sparse(n=n, n_test=m, seed=n) if kind == "binary" else synth.covtype_like(n=n, n_test=m, seed=n)
    a = _alpha(n, p.C)
    prec = {"fp64": pkg.SVM_FP64, "binary": pkg.SVM_FP64, "binary200": pkg.SVM_FP64, "simt": pkg.SVM_MIXED_BF16_SIMT, "mixed": pkg.SVM_MIXED_BF16}[kind]
    ref = oracle.decision(p.X, p.y, a, 0.25, p.gamma, p.Z)
    got = pkg.svm_decision(p.X, p.y, a, 0.25, p.gamma, p.Z, precision=prec)
    if kind in ("fp64", "binary", "binary200"):
        bound = (n + 4) * 2.0 ** -53 * a.sum() + 1e-15
    else:
        sq = lambda M: np.add.reduceat(M.values.astype(np.float64) ** 2, M.indptr[:-1])  # noqa: E731
        bound = (a[None, :] * p.gamma * 4 * 2.0 ** -8 * (sq(p.Z)[:, None] + sq(p.X)[None, :])).sum(1)
    assert np.all(np.abs(got - ref) <= bound), np.abs(got - ref).max()
    # the same values through a model held on the device
    with pkg.Model(p.X, p.y, a, 0.25, p.gamma, precision=prec) as mod:
        if kind != "fp64":
            assert np.array_equal(mod.decision(p.Z), got)


def test_two_query_tiles_per_cta():
    # enough queries that a CTA of the tensor-core contraction takes two tiles
    # (a last one half empty): the rows' values in small calls, whose sums of
    # the same 128-vector partial sums are added in another order
    n, m = 300, 38785
    p = synth.covtype_like(n=n, n_test=m, seed=3)
    a = _alpha(n, p.C)
    got = pkg.svm_decision(p.X, p.y, a, 0.25, p.gamma, p.Z, precision=pkg.SVM_MIXED_BF16)
    bound = (n / 128 + 4) * 2.0 ** -52 * a.sum()
    for lo, hi in ((0, 700), (19000, 19300), (m - 500, m)):
        part = pkg.svm_decision(p.X, p.y, a, 0.25, p.gamma, p.Z.take(np.arange(lo, hi)), precision=pkg.SVM_MIXED_BF16)
        assert np.abs(part - got[lo:hi]).max() <= bound


@pytest.mark.parametrize("gamma", [0.03, 1.0])
def test_binary_decision_keeps_small_kernel_values(gamma):
    # one class and b = 0, so nothing cancels and the bound is relative to the
    # decision itself: K and its exponent's rounding, a term each, and the sum
    # of n terms. At gamma = 1 the largest K of a query is near e^-20.
    n, m = 400, 40
    p = synth.random_sparse(n=n + m, d=200, density=0.08, seed=11, binary=True)
    Z, X = p.X.take(np.arange(n, n + m)), p.X.take(np.arange(n))
    y, a = np.ones(n, p.y.dtype), np.full(n, 1.0)
    got = pkg.svm_decision(X, y, a, 0.0, gamma, Z, precision=pkg.SVM_FP64)
    D = lambda M: np.array([np.bincount(M.indices[M.indptr[i]:M.indptr[i + 1]], minlength=200) for i in range(M.n)])  # noqa: E731
    dx, dz = D(X), D(Z)
    dist = dz.sum(1)[:, None] + dx.sum(1)[None, :] - 2 * (dz @ dx.T)
    ref = np.exp(-gamma * dist.astype(np.float64)).sum(1)
    rel = (n + 4 + gamma * dist.max()) * 2.0 ** -52
    assert np.all(np.abs(got - ref) <= rel * ref), (np.abs(got - ref) / ref).max()
