"""Float64 operator over the tile choices of its kernels: the GEMM tile (4x8
to 32x32) and the columns per CTA of the vertex contraction and the block
dots depend on the molecule and the number of vectors, the result of a vector
does not.  Each application is held to the oracle's explicit chi0 at 1e-12
(a few hundred ulps over sums of up to 10^3 terms), and every vector of a
batch has the bits it has alone."""
import numpy as np
import pytest

import oracle.tddft_oracle as O
from paper_1005_5340_gb300 import synth
from tests.libutil import ensure_library
from tests.test_gpu_parity import ragged_system, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()


SYSTEMS = {
    "tiny2": lambda: synth.tiny_system(3),                       # 3 orbitals, 1 occupied per atom
    "ragged5": ragged_system,                                    # 5 to 16 orbitals per atom
    "ten": lambda: synth.make_system(10, 21, density=0.0094),    # 13 orbitals, over 500 products
}


@pytest.mark.parametrize("name", SYSTEMS)
def test_operator_over_its_tiles(name):
    from paper_1005_5340_gb300 import tddft
    s = SYSTEMS[name]()
    V = O.transition_vertex(s)
    counts = [1, 3, 17, 96]
    z = synth.random_complex_vectors(counts[-1], s.n_prod, 9)
    omega = np.linspace(0.0, 1.5, counts[-1])
    with tddft.Context(s, batch=counts[-1], restart=4) as ctx:
        full = ctx.apply_A(z, omega, 0.005)
        for n in counts:
            part = ctx.apply_A(z[:n], omega[:n], 0.005)
            assert np.array_equal(part, full[:n]), f"{n} vectors differ from {counts[-1]}"
    for r in (0, 1, 16, 50, 95):
        ref = z[r] - O.chi0_explicit(s, omega[r], 0.005, V) @ (s.K @ z[r])
        assert rel(full[r], ref) < 1e-12
