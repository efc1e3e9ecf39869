"""The split-bf16 K product in clusters of 3 and 4 CTAs with two K halves, at a
size where the launch takes the clusters (2760 products: 22 M row blocks in two
halves are 44 clusters, one or two waves of the 46 and 36 that fit on 152 SMs,
and as many waves as of single CTAs).  At 9080 products three N tiles run as
single CTAs in the same order instead (four waves of clusters against three).
apply_A in split bf16 (relative error about 1e-5) is held to 1e-4 of the
float64 form for every vector, in TF32 (10 operands rounded by 2^-11) to 1e-2."""
import numpy as np
import pytest

from paper_1005_5340_gb300 import synth
from tests.libutil import ensure_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def reference():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()
    from paper_1005_5340_gb300 import tddft
    s = synth.make_system(24, 31, density=0.0094)
    z = synth.random_complex_vectors(128, s.n_prod, 78)
    om = np.linspace(0.0, 1.5, 128)
    with tddft.Context(s, batch=128) as ctx:
        return s, z, om, ctx.apply_A(z, om, 0.005)


# 192, 130 (tiles that end past the last column) and 256 real columns
@pytest.mark.parametrize("n_rhs,ncl", [(96, 3), (65, 3), (128, 4)])
@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
def test_clusters_of_three_and_four(reference, n_rhs, ncl, prec):
    from paper_1005_5340_gb300 import tddft
    s, z, om, ref = reference
    tol = 1e-4 if prec == "bf16x3" else 1e-2
    with tddft.Context(s, batch=n_rhs, prec=prec, n_tile=64) as ctx:
        assert ctx.kproduct_plan(n_rhs) == (ncl, 2)
        out = ctx.apply_A(z[:n_rhs], om[:n_rhs], 0.005)
    a, b = out - z[:n_rhs], ref[:n_rhs] - z[:n_rhs]
    assert np.all(np.max(np.abs(a - b), axis=-1) < tol * np.max(np.abs(b), axis=-1))
