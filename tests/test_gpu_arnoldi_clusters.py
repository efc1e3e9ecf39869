"""The Arnoldi step on clusters of 2 and 4 CTAs (2048 to 8191 products) under
the residual rule, whose scalar work one CTA does for the cluster, and under
the error estimates, where every CTA does it: columns of one and of two warps'
length, restarts, and product counts that are no multiple of 4 (scalar loads).

The float64 form runs on the oracle's Krylov path, so it stops after the same
number of products up to a decision that sits on the tolerance, with the same P
to 1e-9 where the numbers agree; the refinement form's P is held to 100 times
the tolerance (residuals of that size, amplified by the system's condition)."""
import functools

import numpy as np
import pytest

import oracle.tddft_oracle as O
from paper_1005_5340_gb300 import synth
from tests.libutil import ensure_library

pytestmark = pytest.mark.gpu

OMEGA = np.array([0.9])
EPS = 0.005


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()


@functools.cache
def molecule(n_atoms, n_local):
    return synth.make_system(n_atoms, 31, density=0.0094, n_local=n_local)


@functools.cache
def oracle(n_atoms, n_local, restart, tol, stop):
    P, infos = O.polarizability_gmres(molecule(n_atoms, n_local), OMEGA, EPS, restart, tol,
                                      stop=stop)
    return P, np.array([i["matvecs"] for i in infos]).reshape(1, 3)


# (atoms, local products per atom, cluster):
# 2760, 2059 and 4460 products
@pytest.mark.parametrize("n_atoms,n_local,cluster", [(24, 40, 2), (19, 41, 2), (36, 40, 4)])
@pytest.mark.parametrize("restart,tol,stop", [(40, 1e-6, "residual"), (12, 1e-6, "residual"),
                                              (40, 1e-3, "eps_p"), (40, 1e-3, "eps_px")])
def test_cluster_steps_follow_the_oracle(n_atoms, n_local, cluster, restart, tol, stop):
    from paper_1005_5340_gb300 import tddft
    s = molecule(n_atoms, n_local)
    assert (s.n_prod >= 4096) == (cluster == 4) and 2048 <= s.n_prod < 8192
    assert (s.n_prod % 4 == 0) == (n_local == 40)
    P_o, mv_o = oracle(n_atoms, n_local, restart, tol, stop)
    with tddft.Context(s, batch=3, restart=restart, tol=tol, stop=stop) as ctx:
        P, info = ctx.polarizability(OMEGA, EPS)
    assert info["converged"].all()
    assert np.all(np.abs(info["matvecs"] - mv_o) <= 2)
    for k in np.flatnonzero(info["matvecs"][0] == mv_o[0]):
        assert abs(P[0, k, k] - P_o[0, k, k]) <= 1e-9 * abs(P_o[0, k, k])
    with tddft.Context(s, batch=3, restart=restart, tol=tol, stop=stop, prec="bf16x3") as ctx:
        P, info = ctx.polarizability(OMEGA, EPS)
    assert info["converged"].all()
    for k in range(3):
        assert abs(P[0, k, k] - P_o[0, k, k]) <= 100 * tol * abs(P_o[0, k, k])
