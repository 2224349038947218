"""Calls that take a large workspace when there is room for it, with little device memory left: they run in
smaller passes instead of failing, and return the same."""
import contextlib

import numpy as np
import pytest
import torch

import workloads as W
from gpu_cases import paired, rel, to_gpu
from oracle import solver

pytestmark = pytest.mark.gpu

MB = 1 << 20


@contextlib.contextmanager
def device_memory_left(nbytes):
    """Holds the device's free memory but for about nbytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    while torch.cuda.mem_get_info()[0] >= nbytes + 2048 * MB:
        held.append(torch.empty(1024 * MB, dtype=torch.uint8, device="cuda"))
    held.append(torch.empty(torch.cuda.mem_get_info()[0] - nbytes - 2 * MB, dtype=torch.uint8, device="cuda"))
    try:
        yield
    finally:
        held.clear()
        torch.cuda.empty_cache()


def colerr(out, ref):
    return np.max(np.linalg.norm(out - ref, axis=0) / np.linalg.norm(ref, axis=0))


def test_batched_filter_takes_column_groups():
    # 300 and 260 complex vectors need 60 MB in one pass (the defect form 91 MB): with 64 MB left that is more than it
    # leaves, so three groups of at most 100 columns run, each from its own captured graph
    from paper_2010_09701_gb300 import FILTER_BF16X3, STORE_BF16X6, STORE_COMPACT, STORE_F64, launch_count
    prs, ctx, V, Vd = paired(ks=[(0.3, 0.0, 0.0), (-0.3, 0.1, 0.0)], n=4, a=8.0,
                             store=STORE_F64 | STORE_BF16X6 | STORE_COMPACT)
    nvs = [300, 260]
    a, b, a0, deg = 5.0, 2500.0, -10.0, 5
    Xs = [W.random_vectors(pr.n, nv, complex_=True, seed=50 + i) for i, (pr, nv) in enumerate(zip(prs, nvs))]
    refs = [solver.chebyshev_filter(pr.apply_A, Xk, deg, a, b, a0) for pr, Xk in zip(prs, Xs)]
    th = [np.random.default_rng(7).uniform(a0, a, nv) for nv in nvs]
    src = [to_gpu(Xk) for Xk in Xs]
    Xd = [torch.empty_like(x) for x in src]
    Xl = [torch.empty_like(x, dtype=torch.complex64) for x in src]

    def both():
        counts = []
        for rep in range(2):   # captured (a launch of no tiles before each capture), then replayed
            for x, s in zip(Xl, src):
                x.copy_(s)
            n0 = launch_count()
            ctx.filter_batched(Xl, deg, a, b, a0, FILTER_BF16X3)
            counts.append(launch_count() - n0)
            for out, ref in zip(Xl, refs):
                assert colerr(out.cpu().numpy().astype(np.complex128), ref) < 5e-5, rep
        for rep in range(2):
            for x, s in zip(Xd, src):
                x.copy_(s)
            ctx.filter_batched_defect(Xd, deg, a, b, a0, th, FILTER_BF16X3)
            for out, ref in zip(Xd, refs):
                assert colerr(out.cpu().numpy(), ref) < 5e-5, rep
        return counts

    one = both()
    ctx.release_workspace()
    with device_memory_left(64 * MB):
        groups = both()
    assert groups == [3 * n for n in one]


@pytest.mark.parametrize("k", [(0.0, 0.0, 0.0), (0.25, -0.4, 0.1)])
def test_fields_in_batches_of_leaves(k):
    # pair mode, 328 leaves of 4^3 and 6^3 points; room for all of them, for a part, for too few to be worth it
    # (the general kernel). Tolerance of the fields in pairs elsewhere in this suite.
    from paper_2010_09701_gb300 import F64_PAIRS, STORE_F64, STORE_F64PAIR, launch_count
    nv = 67 if any(k) else 131
    prs, ctx, V, Vd = paired(ks=[k], n=6, a=12.0, p=3, quad=(4, 6, 1), store=STORE_F64 | STORE_F64PAIR)
    pr = prs[0]
    ctx.set_f64_products(F64_PAIRS)
    X = W.random_vectors(pr.n, nv, complex_=pr.complex, seed=95)
    occ = np.linspace(2.0, 0.0, nv)
    Xd = to_gpu(X)
    rho = torch.empty(pr.quad.nq, dtype=torch.float64, device="cuda")
    g, g2 = torch.empty_like(rho), torch.empty_like(rho)
    rho_o, g_o = solver.density([pr], [X], [occ]), solver.band_trace_grad_V(pr, X)
    ncp = nv if pr.complex else (nv + 1) // 2
    full = pr.quad.nq * ncp * 16

    def fields():
        n0 = launch_count()
        ctx.density_grad([Xd], [occ], rho, 0, g)
        n1 = launch_count()
        ctx.band_trace_grad(0, Xd, g2)
        n2 = launch_count()
        for out, ref in ((rho, rho_o), (g, g_o), (g2, g_o)):
            assert rel(out.cpu().numpy(), ref) < 3.2e-12
        return n1 - n0, n2 - n1

    fields()                           # (the first call forms the pair copy of the enrichment table)
    assert fields() == (3, 3)          # the enrichment part, the two rules
    ctx.release_workspace()
    with device_memory_left(full):     # half of it: two or three batches
        assert fields() in ((6, 6), (9, 9))
    ctx.release_workspace()
    with device_memory_left(full // 8):
        assert fields()[1] == 1        # the general kernel
    ctx.release_workspace()
    assert fields() == (3, 3)
