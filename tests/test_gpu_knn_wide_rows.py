"""K > 12 with more rows than the sliced exhaustive kernels take: lists of equal cosines that overflow every row's
buffer, and more rows than one pass of the collected keys."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,K", [(5001, 24, 13), (4200, 500, 64)])
def test_every_row_overflows(n, d, K):
    """Two distinct rows, each more often than a buffer holds keys: a row's list is the lowest other indices of its
    own copies."""
    from paper_2408_05459_gb300 import ancka
    rng = np.random.default_rng(n)
    rows = rng.standard_normal((2, d)).astype(np.float32)
    kind = np.arange(n) % 2
    idx, sim, info = ancka.knn(torch.as_tensor(rows[kind], device="cuda"), K, "bf16")
    torch.cuda.synchronize()
    assert info["knn_exhaustive_rows"] == n  # n / 2 - 1 > 2048 keys
    idx, sim = idx.cpu().numpy(), sim.cpu().numpy()
    for k in (0, 1):
        first = np.flatnonzero(kind == k)[:K + 1]
        later = kind == k
        later[first] = False
        assert (idx[later] == first[:K]).all()
        for i in first:
            assert idx[i].tolist() == [j for j in first if j != i][:K]
    assert np.abs(sim - 1.0).max() <= 1e-6


def test_overflowing_rows_cost_the_scan_they_end_in():
    """Near-parallel rows (every key within the margin of every row): the passes before the exhaustive scan add about
    1% at this size.  The same rows padded past the contraction's width go to the scan at once; 6% between the two
    times leaves the rest for noise (304 CTAs and an atomic per key took 13%)."""
    import time

    from paper_2408_05459_gb300 import ancka
    n, d, K = 8000, 512, 13
    X = torch.ones(n, d, device="cuda")
    X += 1e-4 * torch.randn(n, d, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    wider = torch.zeros(n, d + 1, device="cuda")
    wider[:, :d] = X

    def best(x):
        times = []
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            ancka.knn(x, K, "bf16", with_info=False)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t)
        return min(times)

    assert best(X) <= 1.06 * best(wider)
    _, _, info = ancka.knn(X, K, "bf16")
    assert info["knn_exhaustive_rows"] == n


def test_more_rows_than_one_collect_pass():
    """The collected keys are taken 2^18 rows at a time: rows on both sides of the second pass's first one and the
    last rows, with copies across it."""
    from tests.parity_util import compare_knn

    from paper_2408_05459_gb300 import ancka
    step = 1 << 18
    n, d, K = step + 131, 16, 13
    X = np.random.default_rng(2).standard_normal((n, d)).astype(np.float32)
    X[step] = X[step - 1]
    X[n - 1] = X[3]
    X[step + 5] = 0.0
    idx, sim, info = ancka.knn(torch.as_tensor(X, device="cuda"), K, "bf16")
    torch.cuda.synchronize()
    rows = np.r_[0:6, step // 2:step // 2 + 3, step - 4:step + 5, step + 6:step + 10, step + 120:n]
    compare_knn(X, K, rows, idx.cpu().numpy(), sim.cpu().numpy())
    assert idx[step + 5].tolist() == list(range(K))  # a zero row: the lowest indices
    assert info["knn_exhaustive_rows"] >= 1
