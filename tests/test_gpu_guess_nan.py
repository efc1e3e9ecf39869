"""An initial guess whose residual is no number is dropped like one that is
worse than zero: the solve of that right-hand side is the one from zero, and
its neighbours keep their guesses."""
import numpy as np
import pytest

from paper_1005_5340_gb300 import synth
from tests.libutil import ensure_library

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "bf16x3", "bf16x3emu"])
@pytest.mark.parametrize("stop", ["residual", "eps_px"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_guess_that_is_no_number_is_dropped(prec, stop, bad):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()
    from paper_1005_5340_gb300 import tddft
    s, w = synth.workload("tiny4")
    om = w["omega"][5:8]
    with tddft.Context(s, batch=9, restart=w["restart"], tol=1e-6, prec=prec, stop=stop) as ctx:
        P0, X, st0 = ctx.polarizability_guess(om, w["eps"])
        x0 = 0.999 * X
        x0[2, 17] = bad
        P, _, st = ctx.polarizability_guess(om, w["eps"], x0)
    assert st["converged"].all()
    rejected = st["guess_rejected"].reshape(-1)
    assert rejected[2] and rejected.sum() == 1
    # the solve from zero after one product for the residual of the guess; the
    # float32 sums of the refinement form depend on the columns solved with it
    exact = prec == "fp64"
    extra = st["matvecs"].reshape(-1)[2] - st0["matvecs"].reshape(-1)[2] - 1
    assert abs(extra) <= (0 if exact else 2)
    a, b = P[0, :, 2].cpu().numpy(), P0[0, :, 2].cpu().numpy()
    assert np.max(np.abs(a - b)) <= (1e-12 if exact else 1e-4) * np.max(np.abs(b))
