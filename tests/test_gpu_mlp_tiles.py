"""The guess network's tensor-core kernels at the edges of their tiles: row
counts around one and several 128-row tiles, widths that are no multiple of a
64-unit chunk, the smallest and largest numbers of inputs and outputs, and the
shapes beyond them that stay on the CUDA cores.  Forward and gradient are held
to float64: a leading-product accumulator truncates 16 times (forward) or up
to 24 times between drains (dW2) at 2^-23 of its partial sums, so 3e-6 and
6e-6 of the result's norm bound them with the rounding of tanh and of the
smaller products."""
import numpy as np
import pytest

import oracle.mlp_oracle as MO
from tests.libutil import ensure_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()


def rounded(p, dims):
    """The parameters as inference takes them: weights in bf16, biases as they are."""
    import torch
    ni, w, no = dims
    parts = np.split(p, np.cumsum([w * ni, w, w * w, w, no * w]))
    for i in (0, 2, 4):
        parts[i] = torch.from_numpy(parts[i]).to(torch.bfloat16).float().numpy()
    return np.concatenate(parts)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("shape", [(10, 256, 2), (1, 1, 1), (12, 192, 4), (10, 100, 2),
                                   (7, 255, 3), (13, 64, 2), (10, 260, 2)])
@pytest.mark.parametrize("rows", [1, 127, 128, 129, 20000])
def test_network_at_tile_edges(shape, rows):
    import torch
    from paper_1005_5340_gb300 import tddft
    ni, w, no = shape
    rng = np.random.default_rng(rows + w)
    net = tddft.Mlp(ni, w, no, max_rows=rows, seed=1)
    p = np.concatenate([rng.uniform(-s, s, n) for n, s in
                        ((w * ni, ni ** -0.5), (w, 0.1), (w * w, w ** -0.5), (w, 0.1),
                         (no * w, w ** -0.5), (no, 0.1))]).astype(np.float32)
    net.set_params(p)
    f = rng.normal(size=(rows, ni)).astype(np.float32)
    dy = (rng.normal(size=(rows, no)) / rows).astype(np.float32)
    ft, dt = torch.from_numpy(f).cuda(), torch.from_numpy(dy).cuda()
    f64 = f.astype(np.float64)
    assert rel(net.forward(ft).double().cpu().numpy(), MO.forward(p, f64, shape)[0]) < 3e-6
    assert rel(net.backward(ft, dt), MO.backward(p, f64, dy.astype(np.float64), shape)) < 6e-6
    y16 = MO.forward(rounded(p, shape), f64, shape)[0]
    assert rel(net.forward(ft, bf16=True).double().cpu().numpy(), y16) < 3e-6


def test_infinite_and_nan_features_stay_in_their_row():
    import torch
    from paper_1005_5340_gb300 import tddft
    net = tddft.Mlp(10, 100, 2, max_rows=300, seed=4)
    p = np.random.default_rng(5).uniform(0.01, 0.1, size=net.n_params).astype(np.float32)
    net.set_params(p)
    f = torch.randn((300, 10), device="cuda", generator=torch.Generator("cuda").manual_seed(6))
    clean = net.forward(f)
    f[7, 3] = float("inf")      # saturates every unit (positive weights): a finite output
    f[130, 0] = float("nan")
    y = net.forward(f)
    keep = [i for i in range(300) if i not in (7, 130)]
    assert torch.equal(y[keep], clean[keep])
    assert torch.isfinite(y[7]).all() and torch.isnan(y[130]).all()
