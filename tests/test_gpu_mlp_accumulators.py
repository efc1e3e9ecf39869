"""The guess network's second layer with every product positive, where the
tensor core's truncations all go one way.  The leading products' accumulator
truncates once per 16 units, at most half a unit in the last place of its
partial sum on average: 16 times at k/16 of the sum s, 4.3 x 2^-23 s.  The
small products' accumulator adds a 2^-8th of its 80 truncations, the two tanhf
and the sum of both accumulators less than 2 x 2^-23 on average: 8 x 2^-23 in
all.  (All products in one accumulator: 12.8 x 2^-23 in a model of it.)"""
import numpy as np
import pytest

import oracle.mlp_oracle as MO
from tests.libutil import ensure_library

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [5000, 20000])
def test_truncations_stay_few(rows):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()
    from paper_1005_5340_gb300 import tddft
    ni, w, no = 10, 256, 4
    rng = np.random.default_rng(rows)
    # hidden values of 0.3 to 0.8, sums s of about 0.5; output o is unit 60 o
    w3 = np.zeros((no, w))
    w3[np.arange(no), 60 * np.arange(no)] = 1.0
    p = np.concatenate([rng.uniform(0.05, 0.1, w * ni), rng.uniform(0.0, 0.2, w),
                        rng.uniform(0.5, 1.0, w * w) / 200, np.zeros(w), w3.ravel(),
                        np.zeros(no)]).astype(np.float32)
    f = rng.uniform(0.5, 1.0, (rows, ni)).astype(np.float32)
    net = tddft.Mlp(ni, w, no, max_rows=rows, seed=1)
    net.set_params(p)
    y = net.forward(torch.from_numpy(f).cuda()).double().cpu().numpy()
    y64 = MO.forward(p, f.astype(np.float64), (ni, w, no))[0]
    assert y64.min() > 0.2 and y64.max() < 0.8
    assert np.mean(np.abs(y / y64 - 1.0)) < 8 * 2.0 ** -23
