"""A setup that is refused leaves no trace in later calls: after an enrichment overlap that is not positive
definite, the same context set up again computes fields and filters as a new one does."""
import numpy as np
import pytest
import torch

import workloads as W
from cases import oracle_problem, uniform_xb
from gpu_cases import rel, to_gpu
from oracle import solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["fields", "filter"])
def test_after_a_singular_enrichment(call):
    from paper_2010_09701_gb300 import (Context, F64_PAIRS, FILTER_BF16X3, STORE_BF16X6, STORE_F64, STORE_F64PAIR,
                                        OefeError, binding)
    a, n, p, quad, r0, rc = 6.0, 2, 3, (4, 6, 1), 1.5, 2.5
    pos, Z = np.array([[3.0, 3.0, 3.0]]), np.array([3])
    R, dR = W.radial_tables(Z, W.ORBITALS_1S_2P, rc=rc, ngrid=2000)
    ctx = Context(0)
    ctx.set_f64_products(F64_PAIRS)
    ctx.mesh(a, uniform_xb(a, n), p)
    ctx.enrichment(pos, W.orbital_lm_codes(W.ORBITALS_1S_2P), 0.0 * R, 0.0 * dR, r0, rc)   # functions that vanish
    ctx.quadrature(*quad)
    with pytest.raises(OefeError) as e:
        ctx.kpoints(np.zeros((1, 3)), [1.0])
    assert e.value.code == binding.ERR_NOTPD_MOO
    # the mesh alone: nothing to factor
    ctx.enrichment(np.zeros((0, 3)), np.zeros(0, np.int32), np.zeros(0), np.zeros(0), r0, rc)
    ctx.quadrature(*quad)
    ctx.kpoints(np.zeros((1, 3)), [1.0])
    pr = oracle_problem(a, uniform_xb(a, n), p, pos, Z, quad=quad, r0=r0, rc=rc, enrich=False)
    V = W.veff(pr.quad.points, a, pos, Z, sigma=0.3)
    pr.build(V)
    ctx.build_hamiltonian(to_gpu(V), STORE_F64 | STORE_F64PAIR | STORE_BF16X6)
    X = W.random_vectors(pr.n, 9, seed=99)
    if call == "fields":
        occ = np.linspace(2.0, 0.0, 9)
        rho = torch.empty(pr.quad.nq, dtype=torch.float64, device="cuda")
        ctx.density([to_gpu(X)], [occ], rho)
        assert rel(rho.cpu().numpy(), solver.density([pr], [X], [occ])) < 3.2e-12
    else:
        ref = solver.chebyshev_filter(pr.apply_A, X, 4, 5.0, 2500.0, -10.0)
        Xd = to_gpu(X, torch.float32)
        ctx.filter_batched([Xd], 4, 5.0, 2500.0, -10.0, FILTER_BF16X3)
        out = Xd.cpu().numpy().astype(np.float64)
        assert np.max(np.linalg.norm(out - ref, axis=0) / np.linalg.norm(ref, axis=0)) < 5e-5
