"""K > 12 (FP32: > 16) of a few rows: the exhaustive scan up to the line where the contraction's launches pay, the
contraction's lists past it, both exact."""
import numpy as np
import pytest

from tests.parity_util import compare_knn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "fp32", "fp8"])
@pytest.mark.parametrize("n,d,K,scan", [
    (19, 3, 17, True), (40, 130, 20, True), (152, 64, 50, True), (160, 16, 16, True), (130, 512, 20, True),
    (152, 64, 51, False), (153, 33, 17, False), (153, 64, 50, False), (200, 20, 17, False),
])
def test_few_rows(prec, n, d, K, scan):
    from paper_2408_05459_gb300 import ancka
    if prec == "fp32" and K <= 16:
        pytest.skip("certified by the FP32 lists")
    rng = np.random.default_rng(n + K)
    X = rng.standard_normal((n, d)).astype(np.float32)
    X[5] = X[n - 1]
    idx, sim, info = ancka.knn(torch.as_tensor(X, device="cuda"), K, prec)
    torch.cuda.synchronize()
    compare_knn(X, K, np.arange(n), idx.cpu().numpy(), sim.cpu().numpy())
    assert info["knn_fallback_rows"] == n
    assert (info["knn_exhaustive_rows"] == n) == scan


def test_few_zero_rows():
    """Zero rows and all-equal rows by either route: the lowest other indices."""
    from paper_2408_05459_gb300 import ancka
    for n, K in ((60, 30), (153, 20)):
        for X in (torch.zeros(n, 7, device="cuda"), torch.ones(n, 7, device="cuda")):
            idx, sim, _ = ancka.knn(X, K, "bf16")
            assert idx.tolist() == [[j for j in range(n) if j != i][:K] for i in range(n)]
            assert (sim - X[0, 0]).abs().max() <= 1e-6
