"""The tensor-core contraction with two query tiles per CTA where the last
CTA has one tile only (its second lies outside the queries) or two, for d <=
64 and for 64 < d <= 128, which differ in stages and shared memory. The number
of queries follows the device: two tiles a CTA begin at one CTA per SM. The
same rows in small calls (one tile a CTA) are the reference: the same FP32
partial sums of 128 vectors, added in another order."""
import numpy as np
import pytest

import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("d", [54, 100])
@pytest.mark.parametrize("extra", [1, 128, 129])   # beyond 2 SMs tiles: a CTA of one row, of one full tile, of two
def test_last_pair_of_tiles(d, extra):
    m = 128 * 2 * torch.cuda.get_device_properties(0).multi_processor_count + extra
    n = 700
    if d == 54:
        p = synth.covtype_like(n=n, n_test=m, seed=3)
        X, y, Z, gamma = p.X, p.y, p.Z, p.gamma
    else:
        p = synth.small_dense(n + m, d, seed=d, sep=0.1)
        X, y, Z, gamma = p.X.take(np.arange(n)), p.y[:n], p.X.take(np.arange(n, n + m)), 1.0 / d
    rng = np.random.default_rng(n)
    a = np.where(rng.random(n) < 0.7, 4.0, rng.uniform(0.0, 4.0, n))
    got = pkg.svm_decision(X, y, a, 0.25, gamma, Z, precision=pkg.SVM_MIXED_BF16)
    bound = (n / 128 + 4) * 2.0 ** -52 * a.sum()
    for lo, hi in ((0, 300), (m - 700, m)):
        part = pkg.svm_decision(X, y, a, 0.25, gamma, Z.take(np.arange(lo, hi)), precision=pkg.SVM_MIXED_BF16)
        assert np.abs(part - got[lo:hi]).max() <= bound
