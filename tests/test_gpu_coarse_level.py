"""Coarse multigrid levels: the one-CTA smoother at the edges of its range, h-transfers, new tissue.

It takes a Q_1 level of at most 1024 nodes whose metric fits in shared memory: levels of a few
nodes, of one element, near 1024 nodes (taken), above (the launch-per-step path), thin ones, and
degrees 1 and 2.  Against the oracle's FP64 V-cycle with the bounds of the other low-precision
V-cycle tests: FP32 5e-7, bf16 metric 5e-3.
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import mesh as Mh
from oracle import multigrid as MG

pytestmark = pytest.mark.gpu

gb = pytest.importorskip("paper_2205_05136_gb300")
capi = gb.capi

ALPHA = 1.5 / 0.05


@pytest.mark.parametrize("quad", ["LGL", "LG"])
@pytest.mark.parametrize("dims,coarse_degree", [((1, 1, 1), 5), ((3, 2, 1), 1), ((9, 9, 9), 2), ((10, 10, 8), 3),
                                                ((40, 4, 4), 4), ((60, 1, 1), 3)])
def test_vcycle_small_coarsest_level(dims, coarse_degree, quad):
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    tissue = (np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), W.transmural_fiber_angles(s))
    g = gb.Slab(s.flat_vertices(), *dims, 2, quad)
    g.set_tissue(*tissue)
    coarse = (dims[0] + 1) * (dims[1] + 1) * (dims[2] + 1)  # stop at the Q_1 level of the mesh
    o = Mh.SlabSpace(s.flat_vertices(), *dims, 2, quad)
    H = MG.Hierarchy(o, tissue, ALPHA, degree=2, coarse_degree=coarse_degree, min_coarse_dofs=coarse)
    assert H.nlevels == 2
    r = W.uniform_vector(o.ndofs, -1.0, 1.0, seed=3)
    ref = H.vcycle(r)
    z = torch.empty(o.ndofs, dtype=torch.float64, device="cuda")
    for prec, tol in ((capi.SEM_PREC_FP32, 5e-7), (capi.SEM_PREC_FP32_BF16, 5e-3)):
        capi.sem_set_gmg(g.ctx, 2, coarse_degree, coarse, prec)
        capi.sem_vcycle(g.ctx, ALPHA, torch.tensor(r, device="cuda"), z)
        e = np.linalg.norm(z.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert e < tol, (prec, e)
    g.close()


@pytest.mark.parametrize("dims", [(7, 5, 3), (8, 6, 4), (5, 1, 2), (1, 9, 1)])
def test_h_transfers_odd_and_even(dims):
    """h-levels of odd, even and single element counts, FP64 V-cycle against the oracle."""
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    tissue = (np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), W.transmural_fiber_angles(s))
    g = gb.Slab(s.flat_vertices(), *dims, 1, "LGL")
    g.set_tissue(*tissue)
    capi.sem_set_gmg(g.ctx, 2, 4, 4, capi.SEM_PREC_FP64)
    o = Mh.SlabSpace(s.flat_vertices(), *dims, 1, "LGL")
    H = MG.Hierarchy(o, tissue, ALPHA, degree=2, coarse_degree=4, min_coarse_dofs=4)
    assert H.nlevels >= 2
    r = W.uniform_vector(o.ndofs, -1.0, 1.0, seed=3)
    z = torch.empty(o.ndofs, dtype=torch.float64, device="cuda")
    capi.sem_vcycle(g.ctx, ALPHA, torch.tensor(r, device="cuda"), z)
    ref = H.vcycle(r)
    assert np.linalg.norm(z.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-10
    g.close()


@pytest.mark.parametrize("precision,tol", [(capi.SEM_PREC_FP64, 1e-12), (capi.SEM_PREC_FP32, 1e-6),
                                           (capi.SEM_PREC_FP32_BF16, 1e-6), (capi.SEM_PREC_BF16_TC, 2e-6)])
def test_hierarchy_follows_new_tissue(precision, tol):
    """A standing hierarchy (p- and h-levels, captured solves) after sem_set_tissue is that of a context made
    with the new tissue: the same V-cycle up to the order of the atomic sums, and the same solution."""
    dims, p = (9, 5, 4), 4
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    ne = s.n_elements
    rng = np.random.default_rng(5)
    old = (np.full(ne, 0.12), np.full(ne, 0.03), W.transmural_fiber_angles(s))
    new = (0.2 * rng.uniform(0.8, 1.2, ne), 0.05 * rng.uniform(0.8, 1.2, ne), -W.transmural_fiber_angles(s))
    out = []
    for first in (old, new):
        g = gb.Slab(s.flat_vertices(), *dims, p, "LGL")
        g.set_tissue(*first)
        capi.sem_set_gmg(g.ctx, 3, 6, 60, precision)
        r = torch.tensor(W.uniform_vector(g.ndofs, -1.0, 1.0, seed=3), device="cuda")
        x = torch.zeros_like(r)
        if first is old:
            for _ in range(4):  # captures the set-up, an iteration, and both as one graph
                x.zero_()
                g.cg_solve(ALPHA, r, x, rtol=1e-12, precond=capi.SEM_PC_GMG)
            g.set_tissue(*new)
        z = torch.empty_like(r)
        capi.sem_vcycle(g.ctx, ALPHA, r, z)
        x.zero_()
        it, _ = g.cg_solve(ALPHA, r, x, rtol=1e-12, precond=capi.SEM_PC_GMG)
        out.append((z, x.clone(), it, capi.sem_gmg_info(g.ctx, ALPHA)["lambda_max"]))
        g.close()
    (z0, x0, it0, l0), (z1, x1, it1, l1) = out
    assert np.allclose(l0, l1, rtol=1e-12, atol=0)
    assert float(torch.linalg.norm(z0 - z1) / torch.linalg.norm(z1)) < tol
    assert float(torch.linalg.norm(x0 - x1) / torch.linalg.norm(x1)) < 1e-10
    assert abs(it0 - it1) <= 1
