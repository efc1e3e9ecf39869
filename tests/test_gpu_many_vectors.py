"""The tensor-core operator on more vectors than one grid dimension holds groups
of: 1 048 600 of them (2 097 200 columns: the gather's groups of 8 and the
combination's of 32 both exceed 65535) on one atom.  A few vectors repeat, so
every repeat must have the first one's bits, and those are held to the
oracle's at 1e-4, the tolerance of split bf16."""
import numpy as np
import pytest

import oracle.tddft_oracle as O
from paper_1005_5340_gb300 import synth
from tests.libutil import ensure_library
from tests.test_gpu_parity import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["A", "chi0"])
def test_over_a_million_vectors(op):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()
    from paper_1005_5340_gb300 import tddft
    s = synth.make_system(1, 5, orb_per_atom=4, occ_per_atom=1, n_local=3)
    few, n = 200, 1048600
    z = torch.from_numpy(synth.random_complex_vectors(few, s.n_prod, 3)).cuda()
    omega = torch.linspace(0.0, 1.5, few, dtype=torch.float64, device="cuda")
    with tddft.Context(s, batch=n, restart=1, prec="bf16x3") as ctx:
        fn = ctx.apply_A if op == "A" else ctx.chi0_apply
        out = fn(z.repeat(n // few, 1), omega.repeat(n // few), 0.005)
        out = out.view(n // few, few, s.n_prod)
        assert bool((out == out[0]).all())
    V = O.transition_vertex(s)
    for r in (0, 77, few - 1):
        zr = z[r].cpu().numpy()
        c = O.chi0_explicit(s, float(omega[r]), 0.005, V)
        ref = zr - c @ (s.K @ zr) if op == "A" else c @ zr
        assert rel(out[0, r].cpu().numpy(), ref) < 1e-4
