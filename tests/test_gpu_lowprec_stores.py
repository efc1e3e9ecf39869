"""Reduced-precision products at the sizes their stores and tile orders change:
n_occ a multiple of 16 (transform 2 writes 16 states at a time; n_occ 32 and 64
columns put the pieces at both parities), and a kernel product of three N tiles
with and without clusters (30 and 27 atoms).  A vector's summation order does not
depend on the batch below 2048 products, so its bits do not either; above, the
products are held to the float64 form at 1e-4, the tolerance of split bf16."""
import pytest

import oracle.tddft_oracle as O
from paper_1005_5340_gb300 import synth
from tests.libutil import ensure_library
from tests.test_gpu_parity import rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()


@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
@pytest.mark.parametrize("atoms", [8, 16])
def test_states_by_sixteen(atoms, prec):
    import torch
    from paper_1005_5340_gb300 import tddft
    s = synth.make_system(atoms, 30 + atoms, density=0.0094)
    assert s.n_occ % 16 == 0 and s.n_prod < 2048
    n = 100
    z = torch.from_numpy(synth.random_complex_vectors(n, s.n_prod, 5)).cuda()
    omega = torch.linspace(0.0, 1.5, n, dtype=torch.float64, device="cuda")
    V = O.transition_vertex(s)
    with tddft.Context(s, batch=n, restart=4, prec=prec) as ctx:
        full = ctx.apply_A(z, omega, 0.005)
        for r in (0, 31, 99):
            zr = z[r].cpu().numpy()
            ref = zr - O.chi0_explicit(s, float(omega[r]), 0.005, V) @ (s.K @ zr)
            assert rel(full[r].cpu().numpy(), ref) < (1e-4 if prec == "bf16x3" else 2e-3)
        for k in (1, 3, 33, 64, 97):
            assert torch.equal(ctx.apply_A(z[:k], omega[:k], 0.005), full[:k])


@pytest.mark.parametrize("atoms", [27, 30])
@pytest.mark.parametrize("n", [129, 192])
def test_kernel_product_of_three_tiles(atoms, n):
    import torch
    from paper_1005_5340_gb300 import tddft
    s = synth.make_system(atoms, 40 + atoms, density=0.0094)
    z = torch.from_numpy(synth.random_complex_vectors(n, s.n_prod, 6)).cuda()
    omega = torch.linspace(0.0, 1.5, n, dtype=torch.float64, device="cuda")
    with tddft.Context(s, batch=n, restart=2, prec="bf16x3") as ctx:
        got = ctx.apply_A(z, omega, 0.005)
    with tddft.Context(s, batch=n, restart=2, prec="fp64") as ctx:
        want = ctx.apply_A(z, omega, 0.005)
    err = torch.linalg.vector_norm(got - want, dim=1) / torch.linalg.vector_norm(want, dim=1)
    assert float(err.max()) < 1e-4
