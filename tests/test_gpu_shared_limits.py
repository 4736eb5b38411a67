"""A kernel's shared memory limit belongs to the process, so a call may not set it to its own size: a thread with a
larger call would find it too low at its launch.  After any call the limits are the same."""
import ctypes
import os
import subprocess
import threading

import numpy as np
import pytest

from paper_2408_05459_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    """The package on a library whose limits can be read (shared_limits.cu in place of knn_tc.o and warm.o)."""
    from paper_2408_05459_gb300 import ancka, build
    objs = [os.path.join(build.BUILD_DIR, os.path.splitext(f)[0] + ".o") for f in build.SOURCES
            if f not in ("knn_tc.cu", "warm.cu")]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    tmp = tmp_path_factory.mktemp("limits")
    flags = [build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I",
             os.path.join(build.ROOT, "include")]
    for part, define in (("knn.o", ["-DKNN"]), ("warm.o", [])):
        subprocess.run([*flags, *define, "-c", os.path.join(HERE, "shared_limits.cu"), "-o", str(tmp / part)],
                       check=True)
    out = str(tmp / "liblimits.so")
    subprocess.run([*flags, "-shared", str(tmp / "knn.o"), str(tmp / "warm.o"), *objs, "-o", out, "-lcudart",
                    "-L/usr/local/cuda/lib64", "-Xlinker", "-rpath=/usr/local/cuda/lib64"], check=True)
    before, ancka._lib = ancka._lib, None
    try:
        yield ancka.load(out)
    finally:
        ancka._lib = before


def _limits(lib, fn, count):
    torch.cuda.synchronize()
    a = (ctypes.c_int * count)()
    getattr(lib, fn)(a)
    return list(a)


def test_knn_limits(lib):
    from paper_2408_05459_gb300 import ancka

    def calls(d):
        X = torch.randn(400, d, device="cuda", generator=torch.Generator(device="cuda").manual_seed(d))
        X[:200] = 1.0 + 1e-4 * X[:200]  # rows for the collect pass
        for K, prec in ((10, "bf16"), (20, "bf16"), (10, "fp8")):
            ancka.knn(X, K, prec)
        ancka.knn_ivf(X, 10, 4, 2)
        ancka.set_symmetric_knn_min_rows(1)
        ancka.knn(X, 10, "bf16")
        ancka.set_symmetric_knn_min_rows(2**63 - 1)
        return _limits(lib, "knn_limits", 6)

    wide = calls(512)
    assert min(wide) >= 200 * 1024  # every kernel ran with a block of A of 128 KB and its stages
    assert calls(40) == wide
    assert calls(100) == wide


def test_warm_limits(lib):
    from paper_2408_05459_gb300 import ancka
    g = synth.sbm_graph(700, 3, 0.03, 0.003, 30, 1.0, seed=0)
    topo, X = ancka.topology_to_device(g), torch.as_tensor(g["X"], device="cuda")

    def calls(k):
        w = {q: torch.as_tensor(np.ascontiguousarray(v, np.float32), device="cuda")
             for q, v in synth.warm_init(1, 60, 256, k).items()}
        Qt = torch.linalg.qr(torch.randn(700, k, device="cuda")).Q.contiguous()
        ancka.warm_gradients(topo, X, Qt, w)
        return _limits(lib, "warm_limits", 2)

    wide = calls(64)
    assert wide[0] >= 256 * 64 * 4 and wide[1] >= 5 * 64 * 64 * 8
    assert calls(3) == wide


def test_threads_with_calls_of_different_widths(lib):
    """Four threads, a stream each, d = 60 to 500: every call returns its own lists."""
    from paper_2408_05459_gb300 import ancka
    inputs, expected, wrong = [], [], []
    for t, d in enumerate((60, 120, 60, 500)):
        X = torch.randn(300, d, device="cuda", generator=torch.Generator(device="cuda").manual_seed(t))
        inputs.append(X)
        expected.append(ancka.knn(X, 10, "bf16")[0])
    torch.cuda.synchronize()

    def work(t):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            try:
                for _ in range(100):
                    idx = ancka.knn(inputs[t], 10, "bf16", with_info=False)[0]
                s.synchronize()
                if not torch.equal(idx, expected[t]):
                    wrong.append(t)
            except Exception as e:
                wrong.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
