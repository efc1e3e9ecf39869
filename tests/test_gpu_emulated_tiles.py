"""Emulated float64 products over the choices of their launch: row slicing by
a warp, a CTA or chunks, column slicing in one or two passes, both N tiles,
and K split over clusters of CTAs.  Each product is held to its stated bound
(plus the float64 reference's own rounding), rows and columns of zeros
included; strides are odd."""
import numpy as np
import pytest

from tests.libutil import ensure_library
from tests.test_gpu_emulated import operands, scale

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()


def padded(x, pad):
    import torch
    buf = torch.full((x.shape[0], x.shape[1] + pad), float("nan"), dtype=torch.float64,
                     device="cuda")
    buf[:, :x.shape[1]] = torch.from_numpy(x)
    return buf[:, :x.shape[1]]


@pytest.mark.parametrize("shape,slices", [
    ((1, 1, 1), 6),              # one entry
    ((129, 65, 63), 5),          # one past a tile, short K
    ((128, 96, 512), 5),         # the wide tile, one exact chunk of K blocks
    ((130, 81, 520), 6),         # one past the 80-wide tile, long columns
    ((257, 193, 2049), 3),       # one past two wide tiles, one CTA per row
    ((64, 31, 8129), 4),         # long rows, K split
    ((300, 129, 9080), 6),       # long rows, K split, ragged N
    ((140, 64, 3000), 7),        # K split in the 64-wide tile
    ((2500, 700, 700), 5),       # many tiles, unsplit
    ((40, 200, 4160), 8),        # eight slices
])
def test_product_within_its_bound(shape, slices):
    from paper_1005_5340_gb300 import tddft
    M, N, K = shape
    A, B = operands(M, N, K, sum(shape))
    if M > 2 and N > 2:
        A[M // 2] = 0.0
        B[:, N // 2] = 0.0
    C = tddft.gemm_f64_emulated(padded(A, 3), padded(B, 1), slices,
                                out=padded(np.zeros((M, N)), 1)).cpu().numpy()
    bound = (1.0 + (slices + 1) / 4.0) * 2.0 ** (-7 * slices) + 2.0 ** -52
    assert np.all(np.abs(C - A @ B) <= bound * scale(A, B))
    if M > 2 and N > 2:
        assert not C[M // 2].any() and not C[:, N // 2].any()
