"""Rayleigh-Ritz at the largest projected problems that one CTA's shared memory holds, and just above."""
import numpy as np
import pytest

import workloads as W
from gpu_cases import paired, to_gpu
from oracle import solver

pytestmark = pytest.mark.gpu

KS = [(0.0, 0.0, 0.0), (0.25, -0.4, 0.1)]


@pytest.mark.parametrize("products", ["native", "pairs"])
@pytest.mark.parametrize("k", KS)
@pytest.mark.parametrize("nv", [78, 79, 80, 81])
def test_rayleigh_ritz_at_the_limit(k, nv, products):
    # tolerances of the same quantities at other widths (FP64; 32 times that for pairs)
    from paper_2010_09701_gb300 import F64_NATIVE, F64_PAIRS, STORE_F64, STORE_F64PAIR
    prs, ctx, V, _ = paired(ks=[k], n=4, a=8.0, store=STORE_F64 | STORE_F64PAIR)
    pr = prs[0]
    ctx.set_f64_products(F64_PAIRS if products == "pairs" else F64_NATIVE)
    f = 32.0 if products == "pairs" else 1.0
    Q = to_gpu(W.random_vectors(pr.n, nv, complex_=pr.complex, seed=93))
    ctx.orthonormalize(0, Q)
    Qh = Q.cpu().numpy()
    eps_o, X_o = solver.rayleigh_ritz(Qh, pr.apply_H, pr.apply_M)
    s = max(1.0, np.max(np.abs(eps_o)))
    eps, res = ctx.rayleigh_ritz(0, Q, resid=True)
    assert np.max(np.abs(eps - eps_o)) < 1e-10 * f * s
    assert np.allclose(res, solver.residual_norms(pr, X_o, eps_o), rtol=1e-8 * f, atol=1e-12 * f * s)
    Xh = Q.cpu().numpy()
    assert np.allclose(Xh.conj().T @ pr.apply_M(Xh), np.eye(nv), atol=1e-11 * f)
