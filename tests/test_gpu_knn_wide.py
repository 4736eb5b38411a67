"""KNN lists of K beyond what two 16-entry lists certify (13 to 64): the shared sweep, threshold, collect pass and
exact selection against the oracle's exact lists."""
import numpy as np
import pytest

from paper_2408_05459_gb300 import synth
from tests.parity_util import compare_knn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "fp32", "fp8"])
@pytest.mark.parametrize("n,d,K", [
    (66, 9, 64),        # K = n - 2 and fewer candidates than K: every key collected
    (300, 512, 13),     # one share, the widest row
    (1025, 64, 31),     # two shares, one row past a tile
    (1100, 65, 32),     # four shares
    (2900, 100, 64),    # blocks whole and split
    (600, 600, 20),     # too wide for the contraction: the exhaustive scan
])
def test_wide_lists(prec, n, d, K):
    from paper_2408_05459_gb300 import ancka
    rng = np.random.default_rng(n + d + K)
    X = synth.gaussian_mixture(rng, rng.integers(0, 4, n), 4, d, 1.5)
    X[5] = X[11] = X[n - 1]   # ties by index
    X[17] = 2.0 * X[18]       # scaled copy
    idx, sim, info = ancka.knn(torch.as_tensor(X, device="cuda"), K, prec)
    torch.cuda.synchronize()
    compare_knn(X, K, np.arange(n), idx.cpu().numpy(), sim.cpu().numpy())


def test_wide_lists_overflow():
    """Zero rows tie with every key and overflow their buffers (2048 keys): the exhaustive scan takes them."""
    from paper_2408_05459_gb300 import ancka
    n, d, K = 2500, 40, 50
    X = np.random.default_rng(3).standard_normal((n, d)).astype(np.float32)
    X[[4, 1300, n - 1]] = 0.0
    idx, sim, info = ancka.knn(torch.as_tensor(X, device="cuda"), K, "bf16")
    torch.cuda.synchronize()
    for z in (4, 1300, n - 1):
        assert idx[z].tolist() == [j for j in range(n) if j != z][:K]
        assert not sim[z].any()
    rows = np.array([0, 3, 5, 255, 256, 1299, 1301, n - 2])
    compare_knn(X, K, rows, idx.cpu().numpy(), sim.cpu().numpy())
    assert 3 <= info["knn_exhaustive_rows"] < n // 10
