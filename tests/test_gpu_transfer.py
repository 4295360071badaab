"""The p-transfer kernels at the edges of their bricks, through the FP64 V-cycle.

A CTA transfers a brick of elements (15 x 4 x 8, 9 x 3 x 4, 7 x 2 x 4, 5 x 1 x 2, 4 x 1 x 2 for
p = 2..6): meshes of several bricks with a partial one at the end of each axis, of exactly two
bricks, and of one element.  Degrees 1 and 2 take the smoother's first and last steps, which
leave out a vector.  Against the oracle's V-cycle with the bound of the other FP64 V-cycle
tests, 1e-10.
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


@pytest.mark.parametrize("p,dims", [(2, (17, 5, 9)), (2, (15, 4, 8)), (3, (10, 4, 5)), (4, (8, 3, 5)), (4, (14, 2, 4)),
                                    (4, (1, 1, 1)), (5, (6, 2, 3)), (6, (5, 2, 3))])
@pytest.mark.parametrize("degree,coarse_degree", [(1, 1), (2, 3)])
def test_vcycle_at_brick_edges(p, dims, degree, coarse_degree):
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    tissue = (np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), W.transmural_fiber_angles(s))
    g = gb.Slab(s.flat_vertices(), *dims, p, "LGL")
    g.set_tissue(*tissue)
    pc = max(1, p // 2)
    coarse = (pc * dims[0] + 1) * (pc * dims[1] + 1) * (pc * dims[2] + 1)  # stop at the first p-level
    capi.sem_set_gmg(g.ctx, degree, coarse_degree, coarse, capi.SEM_PREC_FP64)
    o = Mh.SlabSpace(s.flat_vertices(), *dims, p, "LGL")
    H = MG.Hierarchy(o, tissue, ALPHA, degree=degree, coarse_degree=coarse_degree, min_coarse_dofs=coarse)
    assert H.nlevels == 2
    r = W.uniform_vector(o.ndofs, -1.0, 1.0, seed=3)
    z = torch.empty(o.ndofs, dtype=torch.float64, device="cuda")
    capi.sem_vcycle(g.ctx, ALPHA, torch.tensor(r, device="cuda"), z)
    ref = H.vcycle(r)
    assert np.linalg.norm(z.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-10
    g.close()
