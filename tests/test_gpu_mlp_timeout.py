"""The bounded waits of the guess network's tensor-core kernels: with a limit
of 1 ns they give up, no partial result passes for a whole one, the next call
that synchronises returns TIMEOUT once, and afterwards the network gives the
bits of one that never timed out."""
import numpy as np
import pytest

from paper_1005_5340_gb300 import synth
from tests.libutil import ensure_library

pytestmark = pytest.mark.gpu

ROWS = 20000


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()


def T():
    from paper_1005_5340_gb300 import tddft
    return tddft


def network():
    net = T().Mlp(10, 256, 2, max_rows=ROWS, seed=3)
    net.set_params((np.random.default_rng(4).normal(size=net.n_params) * 0.1).astype(np.float32))
    return net


def reported_once(net):
    with pytest.raises(T().TddftError) as e:
        net.get_params()
    assert e.value.status == T().ERR_TIMEOUT and "gave up" in str(e.value)
    return net.get_params()


def rows(seed, *shape, dtype=None):
    import torch
    return torch.randn(shape, device="cuda", dtype=dtype or torch.float32,
                       generator=torch.Generator("cuda").manual_seed(seed))


@pytest.mark.parametrize("bf16", [False, True])
def test_forward_marks_the_rows_it_lost(bf16):
    import torch
    net, f = network(), rows(1, ROWS, 10)
    ref = net.forward(f, bf16=bf16)
    net.set_wait_timeout(1)
    y = net.forward(f, bf16=bf16)
    lost = torch.isnan(y).any(dim=1)
    assert lost.any()
    assert torch.isnan(y[lost]).all() and torch.equal(y[~lost], ref[~lost])
    reported_once(net)
    net.set_wait_timeout(0)
    assert torch.equal(net.forward(f, bf16=bf16), ref)
    net.get_params()


def test_backward_reports_and_recovers():
    net, f, dy = network(), rows(1, ROWS, 10), rows(2, ROWS, 2)
    ref = net.backward(f, dy)
    net.set_wait_timeout(1)
    with pytest.raises(T().TddftError) as e:
        net.backward(f, dy)
    assert e.value.status == T().ERR_TIMEOUT
    net.set_wait_timeout(0)
    assert np.array_equal(net.backward(f, dy), ref)


def test_training_steps_leave_the_parameters_alone():
    import torch
    nt, n_prod = 10, ROWS // 10
    f = rows(1, ROWS, 10)
    lin, xs = (rows(s, nt, n_prod, dtype=torch.complex128) for s in (2, 3))
    scale = torch.ones(nt, dtype=torch.float64, device="cuda")
    net, twin = network(), network()
    step = lambda n: n.train_step(f, lin, xs, scale, 1e-3)
    step(net), step(twin)
    before = net.get_params()
    net.set_wait_timeout(1)
    step(net), step(net)
    assert np.array_equal(reported_once(net), before)
    net.set_wait_timeout(0)
    step(net), step(twin)
    assert np.array_equal(net.get_params(), twin.get_params())


def test_learned_sweep_returns_timeout_and_recovers(tmp_path):
    s, w = synth.workload("tiny4")
    om = np.linspace(0.40, 0.47, 9)
    net = network()
    net.save(tmp_path / "guess.net")
    with T().Context(s, batch=27, restart=w["restart"], tol=1e-8) as ctx:
        P_zero, _ = ctx.polarizability(om, w["eps"])
        ctx.guess_load(tmp_path / "guess.net")
        ctx.set_guess("learned")
        ctx.set_wait_timeout(1)
        with pytest.raises(T().TddftError) as e:
            ctx.polarizability(om, w["eps"])
        assert e.value.status == T().ERR_TIMEOUT and "network" in str(e.value)
        ctx.set_wait_timeout(0)
        P, info = ctx.polarizability(om, w["eps"])
        assert info["converged"].all()
        assert np.max(np.abs(P - P_zero)) <= 1e-5 * np.max(np.abs(P_zero))
        # a network loaded later takes the context's limit
        ctx.set_wait_timeout(1)
        ctx.guess_load(tmp_path / "guess.net")
        with pytest.raises(T().TddftError) as e:
            ctx.polarizability(om, w["eps"])
        assert e.value.status == T().ERR_TIMEOUT
