"""The FP32 mass operator with Gauss quadrature (beta = 0), float and bf16 weights.

It reads the weights behind the metric's copy, written with the first conversion whoever asks for
it: this apply, an alpha M + K apply or the multigrid hierarchy.  They do not depend on the tissue,
so a tissue update, which converts the metric again, leaves them.  Meshes of one element, of one
element beyond a CTA of the conversion, and of rows that end inside one.  Reference: the FP64 mass
operator, which the other tests hold to the oracle; bounds as there, 6e-7 and 5e-3 (2-norm).
"""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

gb = pytest.importorskip("paper_2205_05136_gb300")
capi = gb.capi


def _dims(p):
    e = max(1, 1024 // (p + 1) ** 3)  # elements of a CTA of the conversion
    return [(1, 1, 1), (e + 1, 1, 1), (7, 5, 3)]


def _tissue(s, scale):
    return np.full(s.n_elements, 0.12 * scale), np.full(s.n_elements, 0.03 * scale), W.transmural_fiber_angles(s)


@pytest.mark.parametrize("prec,tol", [(capi.SEM_PREC_FP32, 6e-7), (capi.SEM_PREC_FP32_BF16, 5e-3)])
@pytest.mark.parametrize("first", ["mass", "stiffness", "vcycle"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
def test_mass_weights(p, first, prec, tol):
    for dims in _dims(p):
        s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
        g = gb.Slab(s.flat_vertices(), *dims, p, "LG")
        g.set_tissue(*_tissue(s, 1.0))
        u = torch.tensor(W.uniform_vector(g.ndofs, -1.0, 1.0, seed=2), device="cuda").float()
        ref = g.apply(u.double(), 2.5, 0.0)
        if first == "stiffness":
            g.apply(u, 30.0, 1.0, prec)
        elif first == "vcycle":
            capi.sem_set_gmg(g.ctx, 3, 5, 20, prec)
            capi.sem_vcycle(g.ctx, 30.0, u.double(), torch.empty_like(u.double()))
        got = [g.apply(u, 2.5, 0.0, prec)]
        g.set_tissue(*_tissue(s, 1.5))
        if first != "mass":
            g.apply(u, 30.0, 1.0, prec)
        got.append(g.apply(u, 2.5, 0.0, prec))
        for y in got:
            err = float(torch.linalg.norm(y.double() - ref) / torch.linalg.norm(ref))
            assert err < tol, (p, dims, first, prec, err)
        g.close()
