"""Edges of the kernels that take a block's width, the polynomial degree or the projected problem's size
into their tiling: the FP64-class products, Gram matrices, rotations, fields, small solvers and the
low-precision filter at widths on both sides of every tile, against the oracle. Tolerances are those of
the same quantities elsewhere in this suite: FP64 1e-12 to 1e-13 of the natural scale, 32 times that
for FP32 pairs (u = 2^-48, 2^5 FP64 units)."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_cases import paired, rel, to_gpu
from oracle import solver

pytestmark = pytest.mark.gpu

KS = [(0.0, 0.0, 0.0), (0.25, -0.4, 0.1)]


def _factor(ctx, products):
    from paper_2010_09701_gb300 import F64_NATIVE, F64_PAIRS
    ctx.set_f64_products(F64_PAIRS if products == "pairs" else F64_NATIVE)
    return 32.0 if products == "pairs" else 1.0


@pytest.mark.parametrize("k", KS)
@pytest.mark.parametrize("p,n,quad", [(3, 4, (4, 6, 1)), (4, 3, (5, 7, 1)), (5, 3, (6, 8, 1)), (6, 3, (7, 9, 1)),
                                      (2, 4, (3, 5, 1)), (3, 4, (5, 5, 1))])
def test_products_and_fields(p, n, quad, k):
    # the register-tiled kernels (P = nq = 4..7) and the general ones that the last two cases keep; one
    # column, an odd count, both sides of 32 real columns and of one pass of 64
    from paper_2010_09701_gb300 import STORE_COMPACT, STORE_F64, STORE_F64PAIR
    prs, ctx, V, _ = paired(ks=[k], p=p, n=n, a=8.0, quad=quad, store=STORE_F64 | STORE_F64PAIR | STORE_COMPACT)
    pr = prs[0]
    X = W.random_vectors(pr.n, 67, complex_=pr.complex, seed=71)
    HX = pr.apply_H(X)
    scale = abs(pr.assemble_H()) @ np.abs(X)
    occ = np.linspace(2.0, 0.0, 67)
    for products in ("native", "pairs"):
        f = _factor(ctx, products)
        for nv in (1, 5, 16, 33, 67):
            Xd = to_gpu(np.ascontiguousarray(X[:, :nv]))
            Y = torch.empty_like(Xd)
            ctx.apply_h(0, Xd, Y)
            assert np.max(np.abs(Y.cpu().numpy() - HX[:, :nv]) / scale[:, :nv]) < 1e-13 * f, (products, nv)
            g = torch.zeros(pr.quad.nq, dtype=torch.float64, device="cuda")
            rho = torch.zeros_like(g)
            ctx.density_grad([Xd], [occ[:nv]], rho, 0, g)
            tol = 3.2e-12 if products == "pairs" else 1e-12
            assert rel(rho.cpu().numpy(), solver.density([pr], [X[:, :nv]], [occ[:nv]])) < tol, (products, nv)
            assert rel(g.cpu().numpy(), solver.band_trace_grad_V(pr, X[:, :nv])) < tol, (products, nv)


@pytest.mark.parametrize("products", ["native", "pairs"])
@pytest.mark.parametrize("k", KS)
def test_subspace_sizes(k, products):
    # Gram tiles of 64 and 128 real rows, Cholesky panels of 16, the one-CTA eigensolver up to 24 and the
    # pair blocks of the cooperative one (odd sizes and a last pair without a partner)
    from paper_2010_09701_gb300 import STORE_F64, STORE_F64PAIR
    prs, ctx, V, _ = paired(ks=[k], n=4, a=8.0, store=STORE_F64 | STORE_F64PAIR)
    f = _factor(ctx, products)
    pr = prs[0]
    Y = W.random_vectors(pr.n, 129, complex_=pr.complex, seed=72)
    for nv in (1, 2, 15, 16, 17, 24, 25, 31, 33, 63, 65, 129):
        Q = to_gpu(np.ascontiguousarray(Y[:, :nv]))
        ctx.orthonormalize(0, Q)
        Qh = Q.cpu().numpy()
        assert np.allclose(Qh.conj().T @ pr.apply_M(Qh), np.eye(nv), atol=1e-12 * f), nv
        eps_o, X_o = solver.rayleigh_ritz(Qh, pr.apply_H, pr.apply_M)
        s = max(1.0, np.max(np.abs(eps_o)))
        eps, res = ctx.rayleigh_ritz(0, Q, resid=True)
        assert np.max(np.abs(eps - eps_o)) < 1e-10 * f * s, nv
        res_o = solver.residual_norms(pr, X_o, eps_o)
        assert np.allclose(res, res_o, rtol=1e-8 * f, atol=1e-12 * f * s), nv
        Xh = Q.cpu().numpy()
        assert np.allclose(Xh.conj().T @ pr.apply_M(Xh), np.eye(nv), atol=1e-11 * f), nv


@pytest.mark.parametrize("k", KS)
def test_filter_widths(k):
    # the batched filter's column groups and the ragged rows of its node update and tile stores: odd
    # widths, both sides of the column tiles, two blocks of unequal width in one call
    from paper_2010_09701_gb300 import FILTER_BF16X3, STORE_BF16X6, STORE_COMPACT, STORE_F64
    prs, ctx, V, _ = paired(ks=[k, k], n=4, a=8.0, store=STORE_F64 | STORE_BF16X6 | STORE_COMPACT)
    a, b, a0, deg = 5.0, 2500.0, -10.0, 4
    dt = torch.complex64 if prs[0].complex else torch.float32
    pr = prs[0]
    X = W.random_vectors(pr.n, 203, complex_=pr.complex, seed=73)
    ref = solver.chebyshev_filter(pr.apply_A, X, deg, a, b, a0)
    err = lambda out, r: np.max(np.linalg.norm(out - r, axis=0) / np.linalg.norm(r, axis=0))
    for nvs in ((1, 7), (32, 33), (64, 65), (97, 203)):
        Xl = [to_gpu(np.ascontiguousarray(X[:, :nv])).to(dt) for nv in nvs]
        ctx.filter_batched(Xl, deg, a, b, a0, FILTER_BF16X3)
        for nv, out in zip(nvs, Xl):
            assert err(out.cpu().numpy(), ref[:, :nv]) < 5e-5, nvs
