"""Cholesky-QR of a block that is not positive definite, at sizes whose trailing blocks take several waves of
CTAs: the failing column is reported and the context keeps working."""
import numpy as np
import pytest

import workloads as W
from gpu_cases import paired, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("products", ["native", "pairs"])
@pytest.mark.parametrize("nv,col", [(1100, 20), (1100, 700), (40, 0), (33, 32)])
def test_failing_column(nv, col, products):
    from paper_2010_09701_gb300 import F64_NATIVE, F64_PAIRS, STORE_F64, STORE_F64PAIR, OefeError, binding
    prs, ctx, V, _ = paired(n=4, a=8.0, store=STORE_F64 | STORE_F64PAIR)
    pr = prs[0]
    ctx.set_f64_products(F64_PAIRS if products == "pairs" else F64_NATIVE)
    X = W.random_vectors(pr.n, nv, seed=91)
    bad = X.copy()
    bad[5, col] = np.nan
    for _ in range(3):
        with pytest.raises(OefeError) as e:
            ctx.orthonormalize(0, to_gpu(bad))
        assert e.value.code == binding.ERR_CHOLESKY
        assert "column %d" % (col + 1) in str(e.value)
    Q = to_gpu(X)
    ctx.orthonormalize(0, Q)
    Qh = Q.cpu().numpy()
    tol = 1e-12 * (32.0 if products == "pairs" else 1.0)   # as for the same quantity at other widths
    assert np.allclose(Qh.T @ pr.apply_M(Qh), np.eye(nv), atol=tol)
