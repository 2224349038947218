"""Cholesky-QR and Rayleigh-Ritz in pair mode on blocks of more than 512 real columns: the rotation then
accumulates over several chunks of the small matrix's rows."""
import numpy as np
import pytest

import workloads as W
from gpu_cases import paired, to_gpu
from oracle import solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,nv", [((0.0, 0.0, 0.0), 530), ((0.25, -0.4, 0.1), 270)])
def test_more_than_512_real_columns(k, nv):
    # 32 times the FP64 tolerances of the same quantities
    from paper_2010_09701_gb300 import F64_PAIRS, STORE_F64, STORE_F64PAIR
    prs, ctx, V, _ = paired(ks=[k], n=4, a=8.0, store=STORE_F64 | STORE_F64PAIR)
    pr = prs[0]
    ctx.set_f64_products(F64_PAIRS)
    Q = to_gpu(W.random_vectors(pr.n, nv, complex_=pr.complex, seed=98))
    ctx.orthonormalize(0, Q)
    Qh = Q.cpu().numpy()
    assert np.allclose(Qh.conj().T @ pr.apply_M(Qh), np.eye(nv), atol=3.2e-11)
    eps_o, X_o = solver.rayleigh_ritz(Qh, pr.apply_H, pr.apply_M)
    s = max(1.0, np.max(np.abs(eps_o)))
    eps, res = ctx.rayleigh_ritz(0, Q, resid=True)
    assert np.max(np.abs(eps - eps_o)) < 3.2e-9 * s
    assert np.allclose(res, solver.residual_norms(pr, X_o, eps_o), rtol=3.2e-7, atol=3.2e-11 * s)
    Xh = Q.cpu().numpy()
    assert np.allclose(Xh.conj().T @ pr.apply_M(Xh), np.eye(nv), atol=3.2e-10)
