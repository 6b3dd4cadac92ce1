"""Batched solves over the sizes where their row pass changes its shape. Dense
mixed rows with 16 lanes (tensor-core units of 32 rows, staged in shared
memory): every row's FP32 inner products keep their order whatever the number
of CTAs, so the multipliers are the same bits for each cluster size. FP64 rows
(exact inner products, kernel-row cache): the multipliers of svm_train alone."""
import numpy as np
import pytest

import paper_1406_5161_gb300 as pkg
from paper_1406_5161_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("d", [32, 96, 256])
def test_units_do_not_depend_on_the_cluster_size(d):
    p = synth.small_dense(1100, d, seed=d, sep=0.2, gamma=1.0 / d)
    rng = np.random.default_rng(d)
    jobs = []
    for n in (31, 64, 65, 400, 1025):
        rows = np.sort(rng.choice(1100, n, replace=False)).astype(np.int32)
        jobs.append({"rows": rows, "y": p.y[rows], "C": 2.0, "gamma": p.gamma})
    ref = None
    for cs in (1, 2, 4, 8):
        out = pkg.svm_train_batch(p.X, jobs, precision=pkg.SVM_MIXED_BF16, cluster_size=cs, lanes_per_row=16)
        got = [(r["iters"], r["alpha"]) for r in out["results"]]
        ref = ref or got
        for (i0, a0), (i1, a1) in zip(ref, got):
            assert i0 == i1 and np.array_equal(a0, a1)


@pytest.mark.parametrize("n,cs", [(40, 1), (300, 2), (961, 2), (1500, 4)])
def test_fp64_jobs_are_the_single_solve(n, cs):
    p = synth.gaussian_mixture(n=n, n_test=0, seed=n)
    jobs = [{"y": p.y, "C": C, "gamma": g} for C in (0.5, 4.0) for g in (0.03, 0.2)]
    out = pkg.svm_train_batch(p.X, jobs, cluster_size=cs, lanes_per_row=1)
    for j, r in zip(jobs, out["results"]):
        one = pkg.svm_train(p.X, p.y, j["C"], j["gamma"], 1e-3)
        assert r["iters"] == one["iters"] and np.array_equal(r["alpha"], one["alpha"])
