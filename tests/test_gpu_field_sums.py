"""The density and the band-trace gradient in pair mode sum the vectors without losing bits as their number
grows: against the native FP64 sums of the same fields."""
import numpy as np
import pytest
import torch

from gpu_cases import paired

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [(0.0, 0.0, 0.0), (0.25, -0.4, 0.1)])
def test_sum_over_many_vectors(k):
    # An accumulator takes every fourth real column. A sum of m positive terms, each addition rounded at u = 2^-48,
    # carries an error of about sqrt(m) u for independent roundings (m u at worst): 4 sqrt(m) u over all points, and
    # 16 u for the terms, whose own errors average out over the columns
    from paper_2010_09701_gb300 import F64_NATIVE, F64_PAIRS, STORE_F64, STORE_F64PAIR
    nv = 8192 if any(k) else 16384
    m = nv * (2 if any(k) else 1) // 4
    tol = (16 + 4 * np.sqrt(m)) * 2.0 ** -48
    prs, ctx, V, _ = paired(ks=[k], n=2, a=6.0, p=3, quad=(4, 6, 1), store=STORE_F64 | STORE_F64PAIR)
    gen = torch.Generator(device="cuda").manual_seed(17)
    X = 2 * torch.rand(prs[0].n, nv * (2 if any(k) else 1), dtype=torch.float64, device="cuda", generator=gen) - 1
    if any(k):
        X = torch.view_as_complex(X.view(prs[0].n, nv, 2))
    occ = np.linspace(2.0, 0.5, nv)
    out = {}
    for mode in (F64_NATIVE, F64_PAIRS):
        ctx.set_f64_products(mode)
        rho, g, g1 = (torch.empty(prs[0].quad.nq, dtype=torch.float64, device="cuda") for _ in range(3))
        ctx.density_grad([X], [occ], rho, 0, g)
        ctx.band_trace_grad(0, X, g1)
        out[mode] = (rho, g, g1)
    for a, b in zip(out[F64_NATIVE], out[F64_PAIRS]):
        assert float(((a - b).abs() / a.abs()).max()) < tol
