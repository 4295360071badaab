"""Chebyshev smoother: the iterate takes its corrections two at a time, so every parity and the shortest degrees.

Degrees 1 to 5 on the fine level and 1 to 4 on a coarsest level that is smoothed launch by
launch (FP64), on a node count that is no multiple of the vector width.  Against the oracle's
V-cycle with the bounds of the other V-cycle tests: FP64 1e-10, FP32 5e-7.
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


@pytest.mark.parametrize("degree,coarse_degree", [(1, 1), (2, 2), (3, 1), (4, 3), (5, 4)])
def test_vcycle_degrees(degree, coarse_degree):
    dims, p = (5, 4, 2), 3
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    tissue = (np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), W.transmural_fiber_angles(s))
    g = gb.Slab(s.flat_vertices(), *dims, p, "LGL")
    g.set_tissue(*tissue)
    o = Mh.SlabSpace(s.flat_vertices(), *dims, p, "LGL")
    H = MG.Hierarchy(o, tissue, ALPHA, degree=degree, coarse_degree=coarse_degree, min_coarse_dofs=30)
    r = W.uniform_vector(o.ndofs, -1.0, 1.0, seed=3)
    ref = H.vcycle(r)
    z = torch.empty(o.ndofs, dtype=torch.float64, device="cuda")
    for prec, tol in ((capi.SEM_PREC_FP64, 1e-10), (capi.SEM_PREC_FP32, 5e-7)):
        capi.sem_set_gmg(g.ctx, degree, coarse_degree, 30, prec)
        capi.sem_vcycle(g.ctx, ALPHA, torch.tensor(r, device="cuda"), z)
        e = np.linalg.norm(z.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert e < tol, (prec, e)
    g.close()
