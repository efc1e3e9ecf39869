"""The work that users of this library have it do, as measurable cases.

Each case is a dict of plain values.  Its "kind" selects the entry point:

  operator      Context.apply_A / Context.chi0_apply: one batched application
                of A(omega) z = z - chi0(omega) K z (or of chi0 alone), the
                unit every solve is made of
  gemm          gemm_f64_emulated: one emulated float64 product
  mlp_forward   Mlp.forward: inference of the guess network over the rows
                (right-hand side, product) of a sweep chunk
  mlp_backward  Mlp.backward: one gradient of the guess network (training)
  spectrum      Context.polarizability: a whole spectrum of one molecule
  batch         Batch.polarizability: several molecules of uneven size

Molecules are the seeded synthetic ones of the package's own workloads (13
orbitals and 2 occupied states per atom); a molecule is what a program loads
once, so it depends on the atom count alone, and the seed of a case draws the
vectors, frequencies, matrices and network rows.  Every right-hand side of an
operator case is one GMRES basis vector (unit norm, three field directions
per frequency).
"""
import functools
import math

import numpy as np
import torch

from paper_1005_5340_gb300 import synth, tddft

EPS = 0.005          # broadening of the workloads (Hartree)
W_HI = 1.5           # upper end of their frequency grids (Hartree)
NET = (10, 256, 2)   # the guess network: features, width, outputs


# -- cases ------------------------------------------------------------------

def listed():
    """The fixed cases."""
    return [
        # three field directions at one frequency on the 4-atom workload: the
        # smallest call there is, all launches and latency
        dict(name="chi0 fp64 4at x3", kind="operator", op="chi0", prec="fp64", atoms=4, rhs=3),
        # the default precision on an ordinary small molecule: a group of 16
        # frequencies
        dict(name="A fp64 24at x48", kind="operator", op="A", prec="fp64", atoms=24, rhs=48),
        # the refinement form on a small molecule with an uneven group (the
        # live count of a solve shrinks as right-hand sides converge): no size
        # is a multiple of a tile
        dict(name="A bf16x3emu 23at x45", kind="operator", op="A", prec="bf16x3emu", atoms=23,
             rhs=45),
        # the inner product of the 64-atom workload at its full group of 64
        # frequencies: where a spectrum spends most of its time
        dict(name="A bf16x3emu 64at x192", kind="operator", op="A", prec="bf16x3emu", atoms=64,
             rhs=192),
        # the same product of a large molecule: the largest call
        dict(name="A bf16x3emu 128at x192", kind="operator", op="A", prec="bf16x3emu", atoms=128,
             rhs=192),
        # the emulated float64 operator: the residual that closes every
        # refinement cycle, in groups of 64 right-hand sides
        dict(name="A fp64emu 64at x64", kind="operator", op="A", prec="fp64emu", atoms=64, rhs=64),
        # one emulated float64 product, tall and ragged (the shape of a kernel
        # product with few vectors)
        dict(name="gemm 1000x129x9080 s6", kind="gemm", m=1000, n=129, k=9080, slices=6),
        # guess inference for a chunk of 64 frequencies of the 64-atom molecule
        dict(name="mlp forward 1.74M", kind="mlp_forward", rows=192 * 9080, bf16=True),
        # one training gradient: 64 targets of a 32-atom molecule
        dict(name="mlp backward 218k", kind="mlp_backward", rows=64 * 3400),
        # the 4-atom workload end to end: 64 frequencies, device loop
        dict(name="spectrum fp64 4at 64w", kind="spectrum", prec="fp64", atoms=4, omegas=64,
             graph=2, restart=30, tol=1e-8),
        # the 64-atom workload end to end: one group of 64 frequencies
        dict(name="spectrum bf16x3emu 64at 64w", kind="spectrum", prec="bf16x3emu", atoms=64,
             omegas=64, graph=0, restart=40, tol=1e-6),
        # screening: eight molecules of 8 to 24 atoms together
        dict(name="batch bf16x3emu 8mol 16w", kind="batch", prec="bf16x3emu", molecules=8, lo=8,
             hi=24, omegas=16, restart=40, tol=1e-6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    kind = rng.choice(["operator", "operator", "operator", "operator", "gemm", "mlp_forward",
                       "mlp_backward", "spectrum", "spectrum", "batch"])
    if kind == "operator":
        prec = rng.choice(["fp64", "fp64emu", "bf16x3", "bf16x3emu", "bf16x3emu", "tf32emu"])
        # native float64 runs at 1/30 of the other forms' rate
        atoms = _log_int(rng, 4, 32 if prec == "fp64" else 96)
        rhs = _log_int(rng, 1, 64 if prec == "fp64" else 192)
        return dict(kind=kind, op=rng.choice(["A", "A", "chi0"]), prec=prec, atoms=atoms, rhs=rhs)
    if kind == "gemm":
        return dict(kind=kind, m=_log_int(rng, 33, 2100), n=_log_int(rng, 9, 2100),
                    k=_log_int(rng, 40, 9080), slices=rng.choice([5, 6, 6, 7]))
    if kind == "mlp_forward":
        return dict(kind=kind, rows=_log_int(rng, 2000, 192 * 9080),
                    bf16=rng.choice([True, True, False]))
    if kind == "mlp_backward":
        return dict(kind=kind, rows=_log_int(rng, 2000, 64 * 3400))
    if kind == "spectrum":
        if rng.random() < 0.5:
            return dict(kind=kind, prec="fp64", atoms=_log_int(rng, 4, 10),
                        omegas=_log_int(rng, 4, 64), graph=rng.choice([0, 1, 2]), restart=30,
                        tol=1e-8)
        return dict(kind=kind, prec=rng.choice(["bf16x3emu", "bf16x3emu", "fp64emu"]),
                    atoms=_log_int(rng, 12, 64), omegas=_log_int(rng, 5, 64),
                    graph=rng.choice([0, 2]), restart=40, tol=1e-6)
    return dict(kind=kind, prec=rng.choice(["bf16x3emu", "fp64"]), molecules=rng.randint(2, 8),
                lo=rng.randint(4, 8), hi=rng.randint(9, 20), omegas=rng.randint(4, 16), restart=40,
                tol=1e-6)


# -- inputs -----------------------------------------------------------------

@functools.lru_cache(maxsize=12)
def _molecule(atoms):
    """The molecule of an atom count (the workloads' own where there is one)."""
    for w in ("tiny4", "medium64"):
        if synth.WORKLOADS[w]["n_atoms"] == atoms:
            return synth.workload(w)[0]
    return synth.make_system(atoms, 4000 + atoms, density=0.0094)


@functools.lru_cache(maxsize=16)
def _batch_molecules(n_mol, lo, hi):
    return tuple(_molecule(n) for n in synth.batch_sizes(n_mol, lo, hi))


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _vectors(case, seed):
    """Unit basis vectors [rhs, n_prod] and their frequencies [rhs]."""
    g = _generator(seed)
    n_prod = _molecule(case["atoms"]).n_prod
    z = torch.randn((case["rhs"], n_prod), dtype=torch.complex128, device="cuda", generator=g)
    z /= torch.linalg.vector_norm(z, dim=1, keepdim=True)
    w = W_HI * torch.rand((case["rhs"] + 2) // 3, dtype=torch.float64, device="cuda", generator=g)
    return z, torch.sort(w).values.repeat_interleave(3)[:case["rhs"]].contiguous()


def _grid(case, seed):
    """A uniform grid on [0, 1.5] with every point moved within its cell."""
    n = case["omegas"]
    return (np.arange(n) + np.random.default_rng(seed).uniform(size=n)) * (W_HI / n)


def _matrices(case, seed):
    """Operands whose rows and columns differ in scale, as basis vectors and
    kernel rows do."""
    g = _generator(seed)
    a = torch.randn((case["m"], case["k"]), dtype=torch.float64, device="cuda", generator=g)
    b = torch.randn((case["k"], case["n"]), dtype=torch.float64, device="cuda", generator=g)
    a *= torch.exp(torch.randn((case["m"], 1), dtype=torch.float64, device="cuda", generator=g))
    b *= torch.exp(torch.randn((1, case["n"]), dtype=torch.float64, device="cuda", generator=g))
    return a, b


def _features(rows, seed):
    """Feature rows in the order of the guess network's inputs."""
    g = _generator(seed)
    f = torch.randn((rows, 10), dtype=torch.float32, device="cuda", generator=g)
    u = torch.rand((rows, 4), dtype=torch.float32, device="cuda", generator=g)
    f[:, 4] = 0.5                               # interpolation weight on a uniform grid
    f[:, 5] = W_HI * u[:, 0]                    # omega
    f[:, 6] = 1.0 + u[:, 1]                     # neighbour spacing over the broadening
    f[:, 7] = (u[:, 2] < 0.7).to(torch.float32)   # bilocal flag
    f[:, 9] = 0.2 + 1.6 * u[:, 3]               # vertex norm over its mean
    return f


def _parameters(seed):
    """Parameters as training leaves them: hidden layers of the usual scale,
    small biases and output weights."""
    n_in, width, n_out = NET
    rng = np.random.default_rng(seed)
    u = lambda n, s: rng.uniform(-s, s, size=n)
    return np.concatenate([u(width * n_in, n_in ** -0.5), u(width, 0.1),
                           u(width * width, width ** -0.5), u(width, 0.1),
                           u(n_out * width, width ** -0.5), u(n_out, 0.1)]).astype(np.float32)


def prepare(case, seed):
    """What a program holds before the call."""
    kind = case["kind"]
    if kind == "operator":
        z, w = _vectors(case, seed)
        ctx = tddft.Context(_molecule(case["atoms"]), batch=case["rhs"], prec=case["prec"],
                            restart=8)
        return dict(call=ctx.apply_A if case["op"] == "A" else ctx.chi0_apply, kind=kind, ctx=ctx,
                    z=z, omega=w)
    if kind == "gemm":
        a, b = _matrices(case, seed)
        return dict(kind=kind, a=a, b=b, slices=case["slices"])
    if kind in ("mlp_forward", "mlp_backward"):
        net = tddft.Mlp(*NET, max_rows=case["rows"], seed=seed)
        net.set_params(_parameters(seed))
        state = dict(kind=kind, net=net, features=_features(case["rows"], seed))
        if kind == "mlp_forward":
            state["bf16"] = case["bf16"]
        else:
            state["dy"] = torch.randn((case["rows"], NET[2]), dtype=torch.float32, device="cuda",
                                      generator=_generator(seed + 1)) / case["rows"]
        return state
    if kind == "spectrum":
        ctx = tddft.Context(_molecule(case["atoms"]), batch=3 * case["omegas"], prec=case["prec"],
                            restart=case["restart"], tol=case["tol"], graph=case["graph"])
        return dict(kind=kind, ctx=ctx, omega=_grid(case, seed))
    mols = _batch_molecules(case["molecules"], case["lo"], case["hi"])
    batch = tddft.Batch(mols, batch=3 * case["omegas"], prec=case["prec"],
                        restart=case["restart"], tol=case["tol"])
    return dict(kind=kind, ctx=batch, omega=_grid(case, seed))


# -- one pass ---------------------------------------------------------------

def run(state):
    """One pass through the public entry point; its outputs whole."""
    kind = state["kind"]
    if kind == "operator":
        return state["call"](state["z"], state["omega"], EPS)
    if kind == "gemm":
        return tddft.gemm_f64_emulated(state["a"], state["b"], state["slices"])
    if kind == "mlp_forward":
        return state["net"].forward(state["features"], bf16=state["bf16"])
    if kind == "mlp_backward":
        return state["net"].backward(state["features"], state["dy"])
    p, stats = state["ctx"].polarizability(state["omega"], EPS)
    return dict(P=p, converged=stats["converged"])


# -- what a pass cannot do without ------------------------------------------

@functools.lru_cache(maxsize=256)
def _sizes(atoms):
    """(n_orb, n_occ, n_virt, n_prod, pairs of neighbouring atoms) from the
    geometry alone."""
    for w in ("tiny4", "medium64"):
        if synth.WORKLOADS[w]["n_atoms"] == atoms:
            seed, density = synth.WORKLOADS[w]["seed"], synth.WORKLOADS[w]["density"]
            break
    else:
        seed, density = 4000 + atoms, 0.0094
    x = synth.atom_positions(atoms, seed, density, 2.5)
    r = np.linalg.norm(x[:, None, :] - x[None, :, :], axis=2)
    pairs = int(np.count_nonzero(np.triu(r < 8.0, 1)))
    return 13 * atoms, 2 * atoms, 11 * atoms, 40 * atoms + 20 * pairs, pairs


def _operator_work(atoms, rhs, with_k, kernel_bytes):
    """Constants (K, V, X) read once, vectors read and written once; the
    flops of the re-associated vertex route."""
    n_orb, n_occ, n_virt, n_prod, pairs = _sizes(atoms)
    column = (4 * 169 * n_prod                                # vertex, in and out
              + 4 * 169 * n_occ * (atoms + 2 * pairs)         # times X_occ, in and out
              + 4 * n_virt * n_orb * n_occ)                   # the two transforms
    if with_k:
        column += 2 * n_prod * n_prod
    constants = 8 * 169 * n_prod + 8 * n_orb * n_orb + (kernel_bytes * n_prod ** 2 if with_k else 0)
    return constants, 32 * n_prod * rhs, 2 * rhs * column


def _products(atoms):
    """GMRES products per right-hand side (about 10 on 4 atoms, 30 on 64)."""
    return 10.0 * (atoms / 4.0) ** 0.4


def work(case):
    """Bytes and flops of one pass."""
    kind = case["kind"]
    kernel_bytes = 8 if case.get("prec", "").startswith("fp64") else 4   # split or tf32: 4
    if kind == "operator":
        constants, vectors, flops = _operator_work(case["atoms"], case["rhs"], case["op"] == "A",
                                                   kernel_bytes)
        return dict(bytes=constants + vectors, flops=flops)
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=8 * (m * k + k * n + m * n), flops=2 * m * n * k)
    if kind in ("mlp_forward", "mlp_backward"):
        n_in, width, n_out = NET
        rows, hidden = case["rows"], width * width + n_out * width
        params = n_in * width + hidden + 2 * width + n_out
        if kind == "mlp_forward":
            return dict(bytes=4 * rows * (n_in + n_out) + 4 * params,
                        flops=2 * rows * (n_in * width + hidden))
        return dict(bytes=4 * rows * (n_in + n_out) + 8 * params,
                    flops=2 * rows * (2 * n_in * width + 3 * hidden))
    if kind == "spectrum":
        sizes = [case["atoms"]]
    else:
        sizes = synth.batch_sizes(case["molecules"], case["lo"], case["hi"])
    total = dict(bytes=8 * 19 * case["omegas"] * len(sizes), flops=0)
    for atoms in sizes:
        constants, _, flops = _operator_work(atoms, 3 * case["omegas"], True, kernel_bytes)
        total["bytes"] += constants
        total["flops"] += flops * _products(atoms)
    return total


# -- 64-bit values ----------------------------------------------------------

class _Exact:
    """chi0(omega) and K of one molecule in float64 with plain torch."""

    def __init__(self, s):
        dev = dict(dtype=torch.float64, device="cuda")
        self.n_orb, self.n_occ, self.n_prod = s.n_orb, s.n_occ, s.n_prod
        x = torch.as_tensor(np.ascontiguousarray(s.X), **dev)
        self.xo, self.xv = x[:, :s.n_occ].contiguous(), x[:, s.n_occ:].contiguous()
        e = torch.as_tensor(s.eigenvalues, **dev)
        self.delta = e[s.n_occ:, None] - e[None, :s.n_occ]
        self.occ = float(s.occupations[0])
        self.k = torch.as_tensor(s.K, **dev)
        self.d = torch.as_tensor(s.dipole, **dev)
        # every vertex entry as (orbital a, orbital b, product, value), the
        # mirrored entries of bilocal products included
        off, row, col, prod, val = s.atom_orb_offset, [], [], [], []
        for mu in range(s.n_prod):
            A, B = (int(i) for i in s.prod_atoms[mu])
            v = s.vertex_block(mu)
            a, b = np.meshgrid(np.arange(off[A], off[A + 1]), np.arange(off[B], off[B + 1]),
                               indexing="ij")
            for p, q in ((a, b), (b, a)) if A != B else ((a, b),):
                row.append(p.ravel())
                col.append(q.ravel())
                val.append(v.ravel())
                prod.append(np.full(v.size, mu))
        self.at = torch.as_tensor(np.concatenate(row) * s.n_orb + np.concatenate(col),
                                  device="cuda")
        self.prod = torch.as_tensor(np.concatenate(prod), device="cuda")
        self.val = torch.as_tensor(np.concatenate(val), **dev)

    def denominators(self, w):
        z = w + 1j * EPS
        return self.occ * (1.0 / (z - self.delta) - 1.0 / (z + self.delta))

    def chi0(self, w, y):
        """chi0(w) y for one complex vector."""
        a = []
        for part in (y.real, y.imag):
            m = torch.zeros(self.n_orb * self.n_orb, dtype=torch.float64, device="cuda")
            m.index_add_(0, self.at, self.val * part[self.prod])
            a.append(self.xv.T @ (m.view(self.n_orb, self.n_orb) @ self.xo))
        a = torch.complex(*a) * self.denominators(w)
        n = []
        for part in (a.real, a.imag):
            g = ((self.xv @ part) @ self.xo.T).reshape(-1)
            n.append(torch.zeros(self.n_prod, dtype=torch.float64,
                                 device="cuda").index_add_(0, self.prod, self.val * g[self.at]))
        return torch.complex(*n)

    def kernel(self, z):
        return torch.complex(z.real @ self.k, z.imag @ self.k)   # K is symmetric

    def pairs(self):
        """M[mu, F E] = sum_ab V_mu^ab X_a^F X_b^E."""
        m = torch.empty((self.n_prod, self.delta.numel()), dtype=torch.float64, device="cuda")
        order = torch.argsort(self.prod, stable=True)
        at, val = self.at[order], self.val[order]
        ends = torch.cumsum(torch.bincount(self.prod, minlength=self.n_prod), 0).cpu().tolist()
        for lo in range(0, self.n_prod, 64):
            hi = min(self.n_prod, lo + 64)
            i0, i1 = (ends[lo - 1] if lo else 0), ends[hi - 1]
            block = torch.zeros((hi - lo, self.n_orb * self.n_orb), dtype=torch.float64,
                                device="cuda")
            which = self.prod[order][i0:i1] - lo
            block.view(-1).index_add_(0, which * self.n_orb * self.n_orb + at[i0:i1], val[i0:i1])
            v = block.view(hi - lo, self.n_orb, self.n_orb)
            m[lo:hi] = (self.xv.T @ (v @ self.xo)).reshape(hi - lo, -1)
        return m

    def polarizability(self, omega):
        """P[w, i, k] by dense complex solves."""
        m, out = self.pairs(), []
        eye = torch.eye(self.n_prod, dtype=torch.complex128, device="cuda")
        d = self.d.to(torch.complex128)
        for w in omega:
            f = self.denominators(float(w)).reshape(-1)
            chi = torch.complex((m * f.real) @ m.T, (m * f.imag) @ m.T)
            a = eye - torch.complex(chi.real @ self.k, chi.imag @ self.k)
            out.append(d @ torch.linalg.solve(a, chi @ d.T))
        return torch.stack(out).cpu().numpy()


def _exact_forward(case, seed, f):
    n_in, width, n_out = NET
    p, parts, at = torch.as_tensor(_parameters(seed), device="cuda"), [], 0
    for n in (width * n_in, width, width * width, width, n_out * width, n_out):
        q = p[at:at + n]
        if case.get("bf16") and n not in (width, n_out):
            q = q.to(torch.bfloat16)   # inference rounds the weights, not the biases
        parts.append(q.double())
        at += n
    w1, b1, w2, b2, w3, b3 = parts
    w1, w2, w3 = w1.view(width, n_in), w2.view(width, width), w3.view(n_out, width)
    h1 = torch.tanh(f @ w1.T + b1)
    h2 = torch.tanh(h1 @ w2.T + b2)
    return h1, h2, h2 @ w3.T + b3, w2, w3


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits; None where that takes
    too long (a whole spectrum of a molecule too large for dense solves)."""
    kind = case["kind"]
    if kind == "operator":
        ref = _Exact(_molecule(case["atoms"]))
        z, omega = _vectors(case, seed)
        y = ref.kernel(z) if case["op"] == "A" else z
        out = torch.stack([ref.chi0(float(w), y[i]) for i, w in enumerate(omega)])
        return z - out if case["op"] == "A" else out
    if kind == "gemm":
        a, b = _matrices(case, seed)
        return a @ b
    if kind == "mlp_forward":
        f = _features(case["rows"], seed)
        return torch.cat([_exact_forward(case, seed, c.double())[2] for c in f.split(1 << 18)])
    if kind == "mlp_backward":
        f = _features(case["rows"], seed).double()
        dy = (torch.randn((case["rows"], NET[2]), dtype=torch.float32, device="cuda",
                          generator=_generator(seed + 1)) / case["rows"]).double()
        h1, h2, _, w2, w3 = _exact_forward(case, seed, f)
        d2 = (dy @ w3) * (1.0 - h2 * h2)
        d1 = (d2 @ w2) * (1.0 - h1 * h1)
        return torch.cat([(d1.T @ f).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0),
                          (dy.T @ h2).reshape(-1), dy.sum(0)]).cpu().numpy()
    if kind == "spectrum":
        _, n_occ, n_virt, n_prod, _ = _sizes(case["atoms"])
        if case["omegas"] * 4.0 * n_prod ** 2 * (n_occ * n_virt + 2 * n_prod) > 1.2e13:
            return None
        return dict(P=_Exact(_molecule(case["atoms"])).polarizability(_grid(case, seed)),
                    converged=None)
    mols = _batch_molecules(case["molecules"], case["lo"], case["hi"])
    return dict(P=np.stack([_Exact(s).polarizability(_grid(case, seed)) for s in mols]),
                converged=None)
