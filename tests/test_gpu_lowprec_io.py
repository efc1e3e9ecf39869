"""Reduced-precision operator: how its vectors come and go, and its tiles.
Aligned complex vectors are read and written as they are, others through
planar copies: both give the same bits, in place and over each other too.
The tiles and epilogues depend on the molecule (n_occ odd, even, a multiple of
8) and on the number of vectors, an output's summation order does not, so a
vector has the same bits alone and in a batch (molecules below 2048 products,
whose K product is never split).  Each product is held to the oracle's at
1e-4 (split bf16) and 2e-3 (tf32), the tolerances of these forms."""
import ctypes

import numpy as np
import pytest

import oracle.tddft_oracle as O
from paper_1005_5340_gb300 import synth
from tests.libutil import ensure_library
from tests.test_gpu_parity import ragged_system, rel

pytestmark = pytest.mark.gpu

SYSTEMS = {
    "ragged5": ragged_system,                                     # n_occ 11
    "ten": lambda: synth.make_system(10, 21, density=0.0094),     # n_occ 20
    "twelve": lambda: synth.make_system(12, 22, density=0.0094),  # n_occ 24
}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()


def raw_apply(ctx, fn, z_ptr, out_ptr, omega, n):
    ctx._check(fn(ctx.h, n, omega.data_ptr(), 0.005, ctypes.c_void_p(z_ptr),
                  ctypes.c_void_p(out_ptr), 1))


@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
@pytest.mark.parametrize("name", SYSTEMS)
def test_vectors_and_tiles(name, prec):
    import torch
    from paper_1005_5340_gb300 import tddft
    s = SYSTEMS[name]()
    n_max, n, np_ = 100, 7, s.n_prod
    z = torch.from_numpy(synth.random_complex_vectors(n_max, np_, 3)).cuda()
    omega = torch.linspace(0.0, 1.5, n_max, dtype=torch.float64, device="cuda")
    V = O.transition_vertex(s)
    tol = 1e-4 if prec == "bf16x3" else 2e-3
    with tddft.Context(s, batch=n_max, restart=4, prec=prec) as ctx:
        for op, fn in (("A", ctx._lib.tddft_apply_A), ("chi0", ctx._lib.tddft_chi0_apply)):
            full = (ctx.apply_A if op == "A" else ctx.chi0_apply)(z, omega, 0.005)
            for r in (0, 6, 63, 64, 99):
                zr = z[r].cpu().numpy()
                c = O.chi0_explicit(s, float(omega[r]), 0.005, V)
                ref = zr - c @ (s.K @ zr) if op == "A" else c @ zr
                assert rel(full[r].cpu().numpy(), ref) < tol
            for k in (1, 2, 33, 65):
                part = (ctx.apply_A if op == "A" else ctx.chi0_apply)(z[:k], omega[:k], 0.005)
                assert torch.equal(part, full[:k])
            # 8-byte aligned vectors (planar route), in place, and shifted by one vector
            buf = torch.empty(2 * n * np_ + 1, dtype=torch.float64, device="cuda")
            buf[1:] = torch.view_as_real(z[:n]).reshape(-1)
            res = torch.empty_like(buf)
            raw_apply(ctx, fn, buf.data_ptr() + 8, res.data_ptr() + 8, omega, n)
            want = torch.view_as_real(full[:n]).reshape(-1)
            assert torch.equal(res[1:], want)
            place = z[:n].clone()
            raw_apply(ctx, fn, place.data_ptr(), place.data_ptr(), omega, n)
            assert torch.equal(place, full[:n])
            both = torch.cat([z[:n], z[:1]])
            raw_apply(ctx, fn, both.data_ptr(), both.data_ptr() + 16 * np_, omega, n)
            assert torch.equal(both[1:], full[:n])
