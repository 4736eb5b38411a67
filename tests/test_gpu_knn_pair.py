"""The full sweep by CTA pairs (bf16 and fp8 lists): the edges of its 256-row blocks, 256-key tiles, 128-byte
feature blocks and stream-K runs, against the oracle's exact lists."""
import numpy as np
import pytest

from tests.parity_util import compare_knn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("n,d,K", [
    (2, 1, 1),          # one block, one tile, almost all of both padding
    (128, 64, 12),      # the second CTA's rows and keys all padding
    (257, 65, 10),      # one row past a block; one feature past a 64-feature block
    (385, 512, 10),     # the largest resident query block (eight feature blocks)
    (2305, 129, 7),     # every block split between several pairs
    (20011, 20, 10),    # blocks whole and split, one per pair
    (40001, 16, 12),    # several whole blocks per pair
])
def test_pair_sweep_edges(prec, n, d, K):
    from paper_2408_05459_gb300 import ancka
    rng = np.random.default_rng(n + d)
    X = rng.standard_normal((n, d)).astype(np.float32)
    if n > 300:
        X[7] = 0.0
        X[n - 1] = X[3]  # an exact duplicate across the whole key range
    rows = np.arange(n) if n <= 400 else np.unique(np.r_[0:8, 120:136, 250:262, n - 40:n, rng.choice(n, 40)])
    idx, sim, info = ancka.knn(torch.as_tensor(X, device="cuda"), K, prec)
    torch.cuda.synchronize()
    if K < n - 1:
        compare_knn(X, K, rows, idx.cpu().numpy(), sim.cpu().numpy())
    else:
        assert idx.cpu().numpy().ravel().tolist() == [1, 0]
    if n > 300:
        assert idx[7].tolist() == [j for j in range(n) if j != 7][:K]  # a zero row: the lowest indices
