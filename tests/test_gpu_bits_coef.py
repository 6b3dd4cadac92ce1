"""Binary decisions (bit masks, fixed-point sums) with multipliers at the ends
of the double range: infinite ones give the infinity or NaN that sums of
positive kernel values have, and subnormal ones count by their value. Wide
exponent ranges keep the sum's rounding. Reference: FP64 sums on the host."""
import numpy as np
import pytest

import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)

N, M, GAMMA = 300, 20, 0.1


def _problem():
    p = synth.random_sparse(n=N + M, d=60, density=0.2, seed=4, binary=True)
    X, Z = p.X.take(np.arange(N)), p.X.take(np.arange(N, N + M))
    dense = lambda A: np.array([np.bincount(A.indices[A.indptr[i]:A.indptr[i + 1]], minlength=60) for i in range(A.n)])  # noqa: E731
    x, z = dense(X), dense(Z)
    K = np.exp(-GAMMA * (z.sum(1)[:, None] + x.sum(1)[None, :] - 2.0 * (z @ x.T)))
    return X, np.where(np.arange(N) % 3 == 0, -1, 1).astype(np.int8), Z, K


@pytest.mark.parametrize("infinite", [(1,), (0,), (0, 1), (1, 2, 4)])   # rows 0, 3, .. have label -1
def test_infinite_multipliers(infinite):
    X, y, Z, K = _problem()
    a = np.full(N, 0.5)
    a[list(infinite)] = np.inf
    with np.errstate(invalid="ignore"):
        want = (K * (a * y)).sum(1) - 0.25
    got = pkg.svm_decision(X, y, a, 0.25, GAMMA, Z)
    assert np.array_equal(got, want, equal_nan=True)


@pytest.mark.parametrize("scale", [1e-310, 2.0 ** -1022, 1e-300, 1e300])
def test_multipliers_at_the_ends_of_the_range(scale):
    X, y, Z, K = _problem()
    a = scale * np.random.default_rng(1).uniform(0.5, 1.5, N)
    got = pkg.svm_decision(X, y, a, 0.0, GAMMA, Z)
    want = (K * (a * y)).sum(1)
    # a rounding of every term and of the sum on both sides, in units of the
    # last place or of the smallest subnormal
    bound = 2 * N * (2.0 ** -52 * scale * 1.5 * N + 5e-324)
    assert np.all(np.abs(got - want) <= bound), np.abs(got - want).max()


def test_one_large_multiplier_among_small_ones():
    X, y, Z, K = _problem()
    a = np.full(N, 1e-9)
    a[7] = 1e9
    got = pkg.svm_decision(X, y, a, 0.0, GAMMA, Z)
    want = (K * (a * y)).sum(1)
    assert np.all(np.abs(got - want) <= (N + 4) * 2.0 ** -53 * (K * a).sum(1))
