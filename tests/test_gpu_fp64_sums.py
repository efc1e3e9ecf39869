"""Length of the summation chains of the float64 K product: at most 2048
entries for any number of products and vectors.

Every term is p = 1 + 1023 2^-52.  While a partial sum is below 2048 its unit
in the last place is at most 2^-42 = 1024 2^-52 and adding p is off by one
2^-52; from 2048 on it is twice that, p rounds to 1 and every addition loses
1023 2^-52, 222 times in a chain of 9080 / 4.  Chains of 2048 at most leave
9080 2^-52 and seven additions of partial sums with half a unit in the last
place of a result below 2^14, 2^-40 each."""
import dataclasses

import numpy as np
import pytest

from paper_1005_5340_gb300 import synth
from tests.libutil import ensure_library

pytestmark = pytest.mark.gpu


def test_kernel_product_of_9080_products_sums_in_short_chains():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()
    from paper_1005_5340_gb300 import tddft
    w = synth.WORKLOADS["medium64"]
    s = synth.make_system(w["n_atoms"], w["seed"], density=w["density"], with_K=False)
    n = s.n_prod
    assert n > 8192 and n // 4 > 2048
    s = dataclasses.replace(s, K=np.ones((n, n)))
    p = 1.0 + 1023 * 2.0 ** -52
    bound = n * 2.0 ** -52 + 7 * 2.0 ** -40
    with tddft.Context(s, batch=60, restart=4) as ctx:
        for rhs in (1, 8, 60):   # 4- to 32-wide tiles
            out = ctx.kernel_apply(np.full((rhs, n), p * (1 - 1j)))
            for part in (out.real, -out.imag):
                # n p is exact as n + n 1023 2^-52 with both parts exact
                err = (part - n) - n * 1023 * 2.0 ** -52
                assert np.max(np.abs(err)) <= bound
