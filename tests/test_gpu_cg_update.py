"""The one-kernel CG vector update at the edges of its range.

It takes 100,000 to 622,592 nodes with x on a 16-byte boundary; up to 155,648 and 311,296 nodes a
thread holds one and two pairs.  Node counts at and beside these limits (odd ones end in half a
pair), with and without the Jacobi preconditioner, FP64 and double-float operators.  The reference
is the same solve with x 8 bytes off the boundary, which takes the kernel-per-update path: the same
recurrences, sums in another order.  Both end below |r| <= rtol |b| and lambda_min(alpha M + K) >=
alpha lambda_min(M), so the bound on their difference is 2 rtol |b| / (alpha min(diag M / 8)) for
the consistent mass too; the true residuals are checked at twice rtol.
"""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

gb = pytest.importorskip("paper_2205_05136_gb300")
capi = gb.capi

ALPHA, RTOL = 30.0, 1e-10


@pytest.mark.parametrize("p,quad,dims", [(1, "LGL", (99, 39, 24)), (1, "LG", (98, 39, 24)), (1, "LGL", (63, 63, 37)),
                                         (2, "LG", (25, 25, 30)), (1, "LGL", (63, 63, 75)), (2, "LGL", (23, 30, 54)),
                                         (1, "LGL", (127, 63, 75)), (1, "LGL", (127, 63, 76))])
@pytest.mark.parametrize("df64", [False, True])
def test_cg_update_edges(p, quad, dims, df64):
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    g = gb.Slab(s.flat_vertices(), *dims, p, quad)
    g.set_tissue(np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), W.transmural_fiber_angles(s))
    if df64:
        capi.sem_set_operator_precision(g.ctx, capi.SEM_PREC_DF64)
    n = g.ndofs
    mass = g.apply(torch.ones(n, dtype=torch.float64, device="cuda"), 1.0, 0.0)  # row sums of M
    b = mass * torch.tensor(W.uniform_vector(n, -1.0, 1.0, seed=4), device="cuda")
    nb = float(torch.linalg.norm(b))
    buf = torch.zeros(n + 2, dtype=torch.float64, device="cuda")
    for pc in (gb.SEM_PC_JACOBI, gb.SEM_PC_NONE):
        got = []
        for off in (0, 1):
            x = buf[off:off + n]
            x.zero_()
            iters = g.cg_solve(ALPHA, b, x, rtol=RTOL, precond=pc)[0]
            assert float(torch.linalg.norm(b - g.apply(x, ALPHA, 1.0))) < 2 * RTOL * nb
            got.append((x.clone(), iters))
        assert abs(got[0][1] - got[1][1]) <= 1
        bound = 2 * RTOL * nb / (ALPHA * float(mass.min()) / 8)
        assert float(torch.linalg.norm(got[0][0] - got[1][0])) < bound
    g.close()
