"""Fields in pair mode on meshes whose cells have no, few and many active enrichment functions: cells out of
every ball's reach, and more functions than one pass of the tensor-core product holds (32 complex, 64 real)."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_cases import paired, rel, to_gpu
from oracle import solver

pytestmark = pytest.mark.gpu

K = (0.25, -0.4, 0.1)
# five functions an atom, the atoms of a face-centred and of a finer cubic arrangement
FCC = 0.25 * np.array([[0, 0, 0], [0, 2, 2], [2, 0, 2], [2, 2, 0], [1, 1, 1], [1, 3, 3], [3, 1, 3], [3, 3, 1], [2, 2, 2]])
CUBIC = 0.5 * np.array([[i, j, l] for i in range(2) for j in range(2) for l in range(2)])
CASES = {
    "none_real": dict(a=12.0, n=6, Zs=(3,), k=(0.0, 0.0, 0.0), pos=None, r0=1.5, rc=2.5),
    "none_complex": dict(a=12.0, n=6, Zs=(3,), k=K, pos=None, r0=1.5, rc=2.5),
    "many_complex": dict(a=10.0, n=3, Zs=(3,) * 9, k=K, pos=10.0 * FCC, r0=2.0, rc=3.0),
    "many_real": dict(a=12.0, n=3, Zs=(3,) * 16, k=(0.0, 0.0, 0.0), pos=12.0 * np.concatenate([CUBIC, CUBIC + 0.25]),
                      r0=2.0, rc=3.0),
}


def _check(name, nvs):
    from paper_2010_09701_gb300 import F64_PAIRS, STORE_F64, STORE_F64PAIR
    c = dict(CASES[name])
    k = c.pop("k")
    prs, ctx, V, _ = paired(ks=[k], p=3, quad=(4, 6, 1), store=STORE_F64 | STORE_F64PAIR, **c)
    pr = prs[0]
    ne = np.array([len(pr.index(e)) - 64 for e in range(pr.mesh.ncells)])
    if name.startswith("none"):
        assert np.any(ne == 0) and np.any(ne > 0)
    else:
        assert np.max(ne) > (32 if pr.complex else 64)
    ctx.set_f64_products(F64_PAIRS)
    X = W.random_vectors(pr.n, max(nvs), complex_=pr.complex, seed=97)
    occ = np.linspace(2.0, 0.0, max(nvs))
    g = torch.empty(pr.quad.nq, dtype=torch.float64, device="cuda")
    rho, g2 = torch.empty_like(g), torch.empty_like(g)
    for nv in nvs:
        Xd = to_gpu(np.ascontiguousarray(X[:, :nv]))
        ctx.density_grad([Xd], [occ[:nv]], rho, 0, g)
        ctx.band_trace_grad(0, Xd, g2)
        rho_o = solver.density([pr], [X[:, :nv]], [occ[:nv]])
        g_o = solver.band_trace_grad_V(pr, X[:, :nv])
        for out, ref in ((rho, rho_o), (g, g_o), (g2, g_o)):   # (as for the fields in pairs elsewhere)
            assert rel(out.cpu().numpy(), ref) < 3.2e-12, nv


@pytest.mark.parametrize("name", ["none_real", "none_complex"])
def test_cells_without_functions(name):
    _check(name, (1, 33, 70))


@pytest.mark.parametrize("name", ["many_complex", "many_real"])
def test_more_functions_than_one_pass(name):
    # the operand halves are used again and the table's digits are cut anew for every column block
    _check(name, (1, 33, 131))
