"""The batched filter's captured graph belongs to one mesh, enrichment, set of k-points and split of the
stored matrices: after any of them changes on the same context, a filter of the same tensor with the same
bounds follows the new operator, against the oracle."""
import numpy as np
import pytest
import torch

import workloads as W
from cases import oracle_problem, uniform_xb
from gpu_cases import to_gpu
from oracle import solver

pytestmark = pytest.mark.gpu

A, P, N, QUAD, R0, RC = 6.0, 3, 2, (4, 5, 2), 1.5, 2.5
POS, Z = np.array([[0.0, 0.0, 0.0], [3.0, 3.0, 3.0]]), np.array([3, 4])
DEG, BOUNDS, NV = 5, (5.0, 2500.0, -10.0), 20


def _graded():
    x = A * np.array([0.0, 0.42, 1.0])
    return np.stack([x] * 3)


FIRST = dict(xb=uniform_xb(A, N), k=(0.25, -0.4, 0.1), pos=POS)
CHANGES = {
    "kpoints": dict(FIRST, k=(-0.1, 0.3, 0.2)),
    "enrichment": dict(FIRST, pos=POS + np.array([0.6, 0.0, 0.3])),
    "mesh": dict(FIRST, xb=_graded()),
}


def _problem(s):
    pr = oracle_problem(A, s["xb"], P, s["pos"], Z, k=s["k"], quad=QUAD, r0=R0, rc=RC)
    V = W.veff(pr.quad.points, A, s["pos"], Z, sigma=0.3)
    pr.build(V)
    return pr, to_gpu(V)


def _filter(ctx, pr, X, buf, tol):
    from paper_2010_09701_gb300 import FILTER_BF16X3
    ref = solver.chebyshev_filter(pr.apply_A, X, DEG, *BOUNDS)
    for rep in range(2):   # captured, then replayed
        buf.copy_(to_gpu(X))
        ctx.filter_batched([buf], DEG, *BOUNDS, FILTER_BF16X3)
        out = buf.cpu().numpy().astype(ref.dtype)
        assert np.max(np.linalg.norm(out - ref, axis=0) / np.linalg.norm(ref, axis=0)) < tol, rep


@pytest.mark.parametrize("change", sorted(CHANGES))
def test_filter_after_a_new_setup(change):
    from paper_2010_09701_gb300 import Context, STORE_BF16X6
    R, dR = W.radial_tables(Z, W.ORBITALS_1S_2P, rc=RC, ngrid=2000)
    lm = W.orbital_lm_codes(W.ORBITALS_1S_2P)
    ctx = Context(0)
    buf = None
    for s in (FIRST, CHANGES[change]):
        if buf is None or change == "mesh":
            ctx.mesh(A, s["xb"], P)
        if buf is None or change != "kpoints":
            ctx.enrichment(s["pos"], lm, R, dR, R0, RC)
            ctx.quadrature(*QUAD)
        ctx.kpoints(np.array([s["k"]]), [1.0])
        pr, Vd = _problem(s)
        ctx.build_hamiltonian(Vd, STORE_BF16X6)
        X = W.random_vectors(pr.n, NV, complex_=True, seed=81)
        if buf is None:
            buf = torch.empty(X.shape, dtype=torch.complex64, device="cuda")
        _filter(ctx, pr, X, buf, 5e-5)


@pytest.mark.parametrize("shape", [0, 3])   # matrices read through plain pointers, through tensor maps
def test_filter_after_another_split(shape):
    from paper_2010_09701_gb300 import Context, STORE_BF16X3, STORE_F64
    R, dR = W.radial_tables(Z, W.ORBITALS_1S_2P, rc=RC, ngrid=2000)
    ctx = Context(0)
    ctx.mesh(A, FIRST["xb"], P)
    ctx.enrichment(POS, W.orbital_lm_codes(W.ORBITALS_1S_2P), R, dR, R0, RC)
    ctx.quadrature(*QUAD)
    ctx.kpoints(np.array([FIRST["k"]]), [1.0])
    ctx.set_filter_shape(shape)
    pr, Vd = _problem(FIRST)
    X = W.random_vectors(pr.n, NV, complex_=True, seed=82)
    buf = torch.empty(X.shape, dtype=torch.complex64, device="cuda")
    ctx.build_hamiltonian(Vd, STORE_BF16X3)
    _filter(ctx, pr, X, buf, 2e-4)
    held = [torch.empty(1 << 22, dtype=torch.uint8, device="cuda") for _ in range(4)]
    ctx.build_hamiltonian(Vd, STORE_F64)   # the split goes
    held += [torch.empty(1 << 22, dtype=torch.uint8, device="cuda") for _ in range(4)]
    ctx.build_hamiltonian(Vd, STORE_BF16X3)
    _filter(ctx, pr, X, buf, 2e-4)
