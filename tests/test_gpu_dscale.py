"""D(omega) of consecutive columns: equal frequencies share one, so the result of
a column must not depend on where its neighbours' frequencies change.  Columns in
runs of one to seven equal frequencies, and the same columns shuffled, agree to
1e-12 (the products' rounding, about 1e-15 times the root of 300 terms, and
slack); small systems take three columns a thread, the large one six."""
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


@pytest.mark.parametrize("prec", ["fp64", "fp64emu"])
@pytest.mark.parametrize("atoms,n", [(4, 1), (4, 2), (4, 7), (10, 13), (24, 80)])
def test_runs_of_frequencies(atoms, n, prec):
    import torch
    from paper_1005_5340_gb300 import tddft
    s = synth.make_system(atoms, 50 + atoms, density=0.0094)
    z = torch.from_numpy(synth.random_complex_vectors(n, s.n_prod, 8)).cuda()
    run = torch.tensor([k for k in range(n) for _ in range(1 + k % 7)][:n])   # 0 11 222 ...
    omega = (0.03 + 0.05 * run.double()).cuda()
    order = torch.randperm(n, generator=torch.Generator().manual_seed(3)).cuda()
    with tddft.Context(s, batch=n, restart=2, prec=prec) as ctx:
        a = ctx.chi0_apply(z, omega, 0.005)
        b = ctx.chi0_apply(z[order].contiguous(), omega[order].contiguous(), 0.005)
    err = torch.linalg.vector_norm(a[order] - b, dim=1) / torch.linalg.vector_norm(b, dim=1)
    assert float(err.max()) < 1e-12
    if atoms <= 10:
        V = O.transition_vertex(s)
        for r in (0, n - 1):
            ref = O.chi0_explicit(s, float(omega[r]), 0.005, V) @ z[r].cpu().numpy()
            assert rel(a[r].cpu().numpy(), ref) < 1e-9
