"""The guess network over the range of float32: values that the bf16 planes of
its tensor-core kernels cannot hold (infinities, NaN, the largest finite ones)
take part as float32 arithmetic has it, and gradients far below 1 keep their
bits.  The sums of a positive network have no cancelling infinities, so the
oracle's pattern of infinities is the float32 one; elsewhere the bounds are
those of the kernels in their ordinary range (3e-6 forward, 6e-6 gradient)."""
import numpy as np
import pytest

import oracle.mlp_oracle as MO
from tests.libutil import ensure_library

pytestmark = pytest.mark.gpu

DIMS = (10, 100, 2)
MAXF = float(np.finfo(np.float32).max)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()


def network(rows, p):
    from paper_1005_5340_gb300 import tddft
    net = tddft.Mlp(*DIMS, max_rows=rows, seed=1)
    net.set_params(p)
    return net


def params(rng, lo=-0.1, w3=1.0):
    ni, w, no = DIMS
    n1 = w * ni + w
    return np.concatenate([rng.uniform(lo, 0.1, n1 + w * w + w),
                           w3 * rng.uniform(10 * lo, 1.0, no * w + no)]).astype(np.float32)


def cuda(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def same(a, b, tol):
    """Equal non-finite entries, and the others within tol of their norm."""
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    odd = ~np.isfinite(b)
    assert np.array_equal(a[odd], b[odd], equal_nan=True) and np.isfinite(a[~odd]).all()
    return np.linalg.norm(a[~odd] - b[~odd]) <= tol * np.linalg.norm(b[~odd])


@pytest.mark.parametrize("rows", [300, 20000])
@pytest.mark.parametrize("value", [float("inf"), -float("inf"), float("nan"), MAXF, 1e30])
def test_gradients_without_planes(rows, value):
    rng = np.random.default_rng(rows)
    p = params(rng, lo=0.01)
    f = rng.uniform(0.1, 1.0, (rows, DIMS[0])).astype(np.float32)
    dy = rng.uniform(0.1, 1.0, (rows, DIMS[2])).astype(np.float32)
    dy[rows // 3, 1] = value
    if abs(value) == MAXF:
        dy[:, 0] = 0.0     # the sum with W3 stays a float32
    with np.errstate(invalid="ignore"):
        ref = MO.backward(p, f.astype(np.float64), dy.astype(np.float64), DIMS)
    assert same(network(rows, p).backward(cuda(f), cuda(dy)), ref, 6e-6)


@pytest.mark.parametrize("scale", [3e-37, 1e-30, 1e25])
def test_gradients_far_from_one(scale):
    rows = 20000
    rng = np.random.default_rng(7)
    p = params(rng)
    f = rng.normal(size=(rows, DIMS[0])).astype(np.float32)
    dy = (scale * rng.normal(size=(rows, DIMS[2]))).astype(np.float32)
    ref = MO.backward(p, f.astype(np.float64), dy.astype(np.float64), DIMS)
    g = network(rows, p).backward(cuda(f), cuda(dy)).astype(np.float64)
    # layer by layer: one scale would hide the smaller ones
    ni, w, no = DIMS
    for a, b in zip(np.split(g, np.cumsum([w * ni, w, w * w, w, no * w])),
                    np.split(ref, np.cumsum([w * ni, w, w * w, w, no * w]))):
        assert np.linalg.norm(a - b) <= 6e-6 * np.linalg.norm(b)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("value", [float("inf"), -float("inf"), MAXF, 1e33])
def test_weights_without_planes(bf16, value):
    import torch
    rows = 300
    rng = np.random.default_rng(8)
    p = params(rng)
    ni, w, no = DIMS
    p[w * ni + w + 3 * w + 5] = value      # W2[3][5]
    f = rng.normal(size=(rows, ni)).astype(np.float32)
    q = p.copy()
    if bf16:
        for a, b in ((0, w * ni), (w * ni + w, w * ni + w + w * w), (p.size - no * w - no, p.size - no)):
            q[a:b] = torch.from_numpy(p[a:b]).to(torch.bfloat16).float().numpy()
    ref = MO.forward(q, f.astype(np.float64), DIMS)[0]
    net = network(rows, p)
    y = net.forward(cuda(f), bf16=bf16).double().cpu().numpy()
    assert np.isfinite(ref).all() and same(y, ref, 3e-6)
    if not bf16:
        # unit 3 is saturated: 1 - h^2 = 0, and 0 * inf is NaN in dH1
        dy = rng.normal(size=(rows, no)).astype(np.float32)
        with np.errstate(invalid="ignore"):
            g = MO.backward(p, f.astype(np.float64), dy.astype(np.float64), DIMS)
        assert same(net.backward(cuda(f), cuda(dy)), g, 6e-6)


@pytest.mark.parametrize("rows", [300, 20000])
@pytest.mark.parametrize("value", [1e20, 1e25, 1e30])
def test_large_output_weights(rows, value):
    # no row overflows, and zero gradients stay zero (also those of the last
    # tile's rows past the end)
    rng = np.random.default_rng(rows)
    ni, w, no = DIMS
    p = params(rng)
    p[-(no * w + no) + 7] = value          # W3[0][7]
    f = rng.normal(size=(rows, ni)).astype(np.float32)
    dy = rng.normal(size=(rows, no)).astype(np.float32)
    dy[::5] = 0.0
    ref = MO.backward(p, f.astype(np.float64), dy.astype(np.float64), DIMS)
    g = network(rows, p).backward(cuda(f), cuda(dy)).astype(np.float64)
    assert np.isfinite(g).all()
    parts = np.cumsum([w * ni, w, w * w, w, no * w])
    for a, b in zip(np.split(g, parts), np.split(ref, parts)):
        assert np.linalg.norm(a - b) <= 6e-6 * np.linalg.norm(b)
    # dW2 and db2 unit by unit: unit 7 would hide the others
    unit = lambda x: np.linalg.norm(x.reshape(w, -1), axis=1)
    for i, j in ((parts[1], parts[2]), (parts[2], parts[3])):
        assert np.all(unit(g[i:j] - ref[i:j]) <= 6e-5 * unit(ref[i:j]))


@pytest.mark.parametrize("rows", [300, 304, 20001])
@pytest.mark.parametrize("value", [float("inf"), -float("inf")])
def test_infinite_output_weight(rows, value):
    # every infinity of a sum has the weight's sign; rows past the end have no share
    rng = np.random.default_rng(rows)
    ni, w, no = DIMS
    p = params(rng, lo=0.01)
    p[-(no * w + no) + 7] = value          # W3[0][7]
    f = rng.uniform(0.1, 1.0, (rows, ni)).astype(np.float32)
    dy = rng.uniform(0.1, 1.0, (rows, no)).astype(np.float32)
    ref = MO.backward(p, f.astype(np.float64), dy.astype(np.float64), DIMS)
    assert not np.isnan(ref).any() and np.isinf(ref).any()
    assert same(network(rows, p).backward(cuda(f), cuda(dy)), ref, 6e-6)
