"""The inverted lists' counting sort at its edges (few and many cells: both chunk lengths; a last partial chunk and
round): every row lands in a list, lists are valid, exact and the same on every call."""
import numpy as np
import pytest

from tests.test_gpu_ivf import _check_lists

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,nlist,nprobe", [
    (33, 5, 1, 1), (1025, 64, 3, 3), (4097, 30, 1024, 16), (9001, 129, 1025, 32), (8192, 512, 40, 8),
])
def test_ivf_sort_edges(n, d, nlist, nprobe):
    from paper_2408_05459_gb300 import ancka
    rng = np.random.default_rng(n)
    X = (rng.standard_normal((8, d))[rng.integers(0, 8, n)] + 0.5 * rng.standard_normal((n, d))).astype(np.float32)
    Xd = torch.as_tensor(X, device="cuda")
    idx, sim, _ = ancka.knn_ivf(Xd, 5, nlist=nlist, nprobe=nprobe)
    again, sim2, _ = ancka.knn_ivf(Xd, 5, nlist=nlist, nprobe=nprobe)
    torch.cuda.synchronize()
    assert torch.equal(idx, again) and torch.equal(sim, sim2)
    recall = _check_lists(X, idx.cpu().numpy(), sim.cpu().numpy(), np.arange(0, n, max(1, n // 200)), 5)
    assert recall == 1.0 or nprobe < nlist
