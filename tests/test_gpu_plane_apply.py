"""The plane kernel of the FP32 operator at the edges of its units, and the kernel for few elements.

A unit is G = 32 // (p + 1) consecutive elements of one warp: meshes of one element, of
one unit exactly, of one element more or less, of rows that end inside a unit, of more
elements than one CTA of the metric's conversion takes, and vectors
that start 4 bytes past a 16-byte boundary (the gather copies single words).  From p = 3 the
meshes of up to some 3,000 elements take the kernel of one line per thread; 4,067 and 4,320
elements (no multiple and a multiple of every unit) take the plane kernel.  The reference
is the FP64 apply, which the other tests hold to the oracle.  Bounds as in test_gpu_apply:
FP32 arithmetic with an FP32 metric 6e-7, the bf16 metric 5e-3 (relative, 2-norm).
"""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

gb = pytest.importorskip("paper_2205_05136_gb300")


def _dims(p):
    g = 32 // (p + 1)
    large = [(83, 7, 7), (60, 8, 9)] if p >= 3 else []  # above the sizes of the kernel for few elements
    return large + [(1, 1, 1), (g, 1, 1), (g - 1, 1, 1), (g + 1, 1, 1), (3, 2, 2), (g + 2, 3, 2), (8 * g + 1, 1, 1)]


@pytest.mark.parametrize("quad", ["LGL", "LG"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
def test_plane_kernel_unit_edges(p, quad):
    for dims in _dims(p):
        s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
        g = gb.Slab(s.flat_vertices(), *dims, p, quad)
        g.set_tissue(np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), W.transmural_fiber_angles(s))
        buf = torch.tensor(W.uniform_vector(g.ndofs + 1, -1.0, 1.0, seed=2), device="cuda").float()
        out = torch.empty_like(buf)
        for off in (0, 1):
            u = buf[off:off + g.ndofs]
            y = out[off:off + g.ndofs]
            for alpha, beta in ((30.0, 1.0), (2.5, -0.7)):
                ref = g.apply(u.double(), alpha, beta)
                for prec, tol in ((gb.SEM_PREC_FP32, 6e-7), (gb.SEM_PREC_FP32_BF16, 5e-3)):
                    g.apply(u, alpha, beta, prec, out=y)
                    err = float(torch.linalg.norm(y.double() - ref) / torch.linalg.norm(ref))
                    assert err < tol, (p, quad, dims, off, alpha, prec, err)
        g.close()


@pytest.mark.parametrize("quad", ["LGL", "LG"])
@pytest.mark.parametrize("p,dims", [(1, (20, 12, 9)), (2, (12, 8, 5)), (3, (83, 7, 7)), (4, (83, 7, 7)), (5, (60, 8, 9)),
                                    (6, (60, 8, 9)), (3, (9, 5, 3)), (5, (6, 4, 3))])
def test_deterministic_element_results(p, quad, dims):
    """Deterministic mode of the plane kernel at every degree (from p = 3 on 4,067 and 4,320 elements) and of
    the kernel for few elements at odd degrees: bitwise repeat, and the FP64 operator within the bounds above."""
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    g = gb.Slab(s.flat_vertices(), *dims, p, quad)
    g.set_tissue(np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), W.transmural_fiber_angles(s))
    gb.capi.sem_set_deterministic(g.ctx, True)
    u = torch.tensor(W.uniform_vector(g.ndofs, -1.0, 1.0, seed=2), device="cuda").float()
    for alpha, beta in ((30.0, 1.0), (2.5, -0.7)):
        ref = g.apply(u.double(), alpha, beta)
        for prec, tol in ((gb.SEM_PREC_FP32, 6e-7), (gb.SEM_PREC_FP32_BF16, 5e-3)):
            y = g.apply(u, alpha, beta, prec)
            assert torch.equal(y, g.apply(u, alpha, beta, prec))
            err = float(torch.linalg.norm(y.double() - ref) / torch.linalg.norm(ref))
            assert err < tol, (p, quad, dims, alpha, prec, err)
    g.close()
