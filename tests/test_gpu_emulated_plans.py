"""Emulated float64 products: K at whole exact chunks, CTAs that walk several
tiles of several chunks for every slice count (ring slots, phases and barrier
parities carried over), and first calls from several threads at once.  Sums
are exact integers, so a part of a product has the bits of that part alone,
whatever N tile and K split either takes."""
import subprocess
import sys

import numpy as np
import pytest

from tests.libutil import ROOT, ensure_library
from tests.test_gpu_emulated import operands, scale

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()


def product(A, B, slices):
    import torch
    from paper_1005_5340_gb300 import tddft
    return tddft.gemm_f64_emulated(torch.from_numpy(np.ascontiguousarray(A)).cuda(),
                                   torch.from_numpy(np.ascontiguousarray(B)).cuda(),
                                   slices).cpu().numpy()


def chunk(slices):
    """Entries of K whose group sums stay below 2^24, in whole 64-entry blocks."""
    return 4096 // (slices + 2) // 64 * 64


@pytest.mark.parametrize("slices", [3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("M,N,chunks,more", [(130, 70, 1, 0), (130, 70, 2, 0), (64, 64, 1, 1),
                                             (2100, 1500, 3, 40)])
def test_chunks_and_tiles(slices, M, N, chunks, more):
    K = chunks * chunk(slices) + more
    A, B = operands(M, N, K, slices + K)
    C = product(A, B, slices)
    bound = (1.0 + (slices + 1) / 4.0) * 2.0 ** (-7 * slices) + 2.0 ** -52
    assert np.all(np.abs(C - A @ B) <= bound * scale(A, B))
    m, n = M // 3, N // 2
    assert np.array_equal(product(A[m:m + 40], B[:, n:n + 30], slices), C[m:m + 40, n:n + 30])


THREADS = """
import sys, threading
sys.path.insert(0, sys.argv[1])
import torch
from paper_1005_5340_gb300 import tddft
g = torch.Generator("cuda").manual_seed(1)
rand = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=torch.float64)
work = [(rand(100 + 90 * i, 700 * (i + 1)), rand(700 * (i + 1), 60 + 50 * i), 3 + i % 6)
        for i in range(8)]
torch.cuda.synchronize()
got, gate = [None] * 8, threading.Barrier(8)
def run(i):
    with torch.cuda.stream(torch.cuda.Stream()):
        gate.wait()
        got[i] = tddft.gemm_f64_emulated(*work[i])
ts = [threading.Thread(target=run, args=(i,)) for i in range(8)]
[t.start() for t in ts]
[t.join() for t in ts]
torch.cuda.synchronize()
assert all(torch.equal(got[i], tddft.gemm_f64_emulated(*work[i])) for i in range(8))
print("same bits")
"""


def test_first_calls_from_several_threads():
    out = subprocess.run([sys.executable, "-c", THREADS, ROOT], capture_output=True, text=True,
                         timeout=300)
    assert out.returncode == 0 and "same bits" in out.stdout, out.stderr[-2000:]
