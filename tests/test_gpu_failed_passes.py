"""Calls whose tensor-core pass fails (its bounded wait expired): a stand-in for the pass sets the error word and
leaves its outputs unwritten (failing_pass.cu).  Nothing reads those outputs as indices, and the context stays usable.

Lists and keys that were never written must not be followed, so this runs on code that checks the error words first."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from tests.parity_util import compare_knn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    """The library with tests/failing_pass.cu in the place of knn_tc.o, and its signatures."""
    from paper_2408_05459_gb300 import ancka, build
    objs = [os.path.join(build.BUILD_DIR, os.path.splitext(f)[0] + ".o") for f in build.SOURCES if f != "knn_tc.cu"]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    out = str(tmp_path_factory.mktemp("failing") / "libfailing.so")
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I",
                    os.path.join(build.ROOT, "include"), os.path.join(HERE, "failing_pass.cu"), *objs, "-o", out,
                    "-lcudart", "-L/usr/local/cuda/lib64", "-Xlinker", "-rpath=/usr/local/cuda/lib64"], check=True)
    L = ctypes.CDLL(out)
    real = ancka.load()
    for fn in ("ancka_knn", "ancka_knn_ivf"):
        getattr(L, fn).argtypes = getattr(real, fn).argtypes
    return L


def _knn(lib, X, K, nth, info=None):
    from paper_2408_05459_gb300 import ancka
    n, d = X.shape
    idx = torch.full((n, K), -7, dtype=torch.int32, device="cuda")
    sim = torch.zeros((n, K), device="cuda")
    lib.set_failing_pass(nth)
    st = lib.ancka_knn(ancka._ptr(X), n, d, K, ancka.PREC["bf16"], ancka._ptr(idx), ancka._ptr(sim),
                       ctypes.byref(info) if info is not None else None, ancka._stream())
    lib.set_failing_pass(0)
    torch.cuda.synchronize()
    return st, idx, sim


@pytest.mark.parametrize("nth", [1, 2])  # the list pass, the collect pass
@pytest.mark.parametrize("n,d,K", [(700, 40, 20), (1500, 100, 64)])
def test_wide_lists_without_their_pass(lib, n, d, K, nth):
    """K > 12, nothing read back: the exhaustive scan gives the same exact lists."""
    X = np.random.default_rng(n + nth).standard_normal((n, d)).astype(np.float32)
    st, idx, sim = _knn(lib, torch.as_tensor(X, device="cuda"), K, nth)
    assert st == 0
    compare_knn(X, K, np.arange(0, n, 7), idx.cpu().numpy(), sim.cpu().numpy())


@pytest.mark.parametrize("nth", [1, 2])
def test_wide_lists_report_their_pass(lib, nth):
    """K > 12 with info, which the call reads back: the status says so, and the next call works."""
    from paper_2408_05459_gb300 import ancka
    X = np.random.default_rng(nth).standard_normal((700, 40)).astype(np.float32)
    Xd = torch.as_tensor(X, device="cuda")
    assert _knn(lib, Xd, 20, nth, ancka.Info())[0] == 5  # ANCKA_ERR_TIMEOUT
    info = ancka.Info()
    st, idx, sim = _knn(lib, Xd, 20, 0, info)
    assert st == 0 and info.knn_exhaustive_rows == 0
    compare_knn(X, 20, np.arange(0, 700, 7), idx.cpu().numpy(), sim.cpu().numpy())


def test_narrow_lists_without_their_pass(lib):
    """K <= 12: the status says so, and the next call works."""
    X = np.random.default_rng(5).standard_normal((900, 64)).astype(np.float32)
    Xd = torch.as_tensor(X, device="cuda")
    assert _knn(lib, Xd, 10, 1)[0] == 5  # ANCKA_ERR_TIMEOUT
    st, idx, sim = _knn(lib, Xd, 10, 0)
    assert st == 0
    compare_knn(X, 10, np.arange(0, 900, 7), idx.cpu().numpy(), sim.cpu().numpy())


@pytest.mark.parametrize("n,d,nlist,nprobe", [(1500, 40, 7, 3), (9000, 20, 1025, 16)])
@pytest.mark.parametrize("nth", [1, 8, 9, 10])  # the first and last round of the cells, the probes, the tile lists
def test_inverted_lists_without_their_pass(lib, n, d, nlist, nprobe, nth):
    """The status says so, every index on the way stays in range, and the next call is right."""
    from paper_2408_05459_gb300 import ancka
    K = 6
    X = torch.as_tensor(np.random.default_rng(n).standard_normal((n, d)).astype(np.float32), device="cuda")
    ref, ref_sim, _ = ancka.knn_ivf(X, K, nlist, nprobe)
    idx = torch.empty((n, K), dtype=torch.int32, device="cuda")
    sim = torch.empty((n, K), device="cuda")
    for fail, status in ((nth, 5), (0, 0)):
        lib.set_failing_pass(fail)
        assert lib.ancka_knn_ivf(ancka._ptr(X), n, d, K, nlist, nprobe, ancka._ptr(idx), ancka._ptr(sim), None,
                                 ancka._stream()) == status
        lib.set_failing_pass(0)
        torch.cuda.synchronize()
    assert torch.equal(idx, ref) and torch.equal(sim, ref_sim)
