"""The parameter-gradient kernel for every degree and quadrature (one instantiation each).

The adjoint gradient on a perturbed mesh against the oracle's, with the bound of the other
adjoint tests (relative 1e-8: both solve to 1e-13 and the misfit cancels digits).
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import adjoint as AD
from oracle import mesh as Mh

pytestmark = pytest.mark.gpu

gb = pytest.importorskip("paper_2205_05136_gb300")

# No face of the box passes through a node: at z = 1 the last bit of a coordinate would decide on which
# side of the face the node lies, and the two sides may round it differently.
BOX = (-0.1, -0.1, -0.1, 1.1, 1.1, 1.1)


@pytest.mark.parametrize("quad", ["LGL", "LG"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
def test_param_grad_degrees(p, quad):
    dims, dt, steps = (2, 2, 1), 0.05, 3
    s = W.slab(*dims, (3.0, 2.0, 1.0), perturb=0.1, seed=1)
    sp = Mh.SlabSpace(s.flat_vertices(), *dims, p, quad)
    rng = np.random.default_rng(3)
    ne = s.n_elements
    tissue = (0.12 * rng.uniform(0.8, 1.2, ne), 0.03 * rng.uniform(0.8, 1.2, ne), rng.uniform(-1.0, 1.0, ne))
    sensors = W.seeded_indices(sp.ndofs, 5, seed=W.SEED_SENSORS)
    model = AD.AdjointModel(sp, dt, steps, sensors, region=("box", BOX), amplitude=50.0, t_on=0.0, t_off=0.2)
    u0 = W.uniform_vector(sp.ndofs, -85.0, -40.0, seed=2)
    h0 = np.full(sp.ndofs, 0.9)
    tl, tt = W.perturbed_conductivities(tissue[0], tissue[1])
    target = model.forward((tl, tt, tissue[2]), u0, h0)[2]
    _, tbar = AD.misfit(model.forward(tissue, u0, h0)[2], target, dt)
    ref = np.concatenate(model.gradient(tissue, u0, h0, tbar))
    g = gb.Slab(s.flat_vertices(), *dims, p, quad)
    g.set_ionic()
    g.set_stimulus("box", BOX, 50.0, 0.0, 0.2)
    leaves = [torch.tensor(t, device="cuda", requires_grad=True) for t in tissue]
    T = gb.traces(g, *leaves, torch.tensor(u0, device="cuda"), torch.tensor(h0, device="cuda"), dt, steps,
                  torch.tensor(sensors, dtype=torch.int32), checkpoint_every=2, rtol=1e-13, precond=gb.SEM_PC_JACOBI)
    (0.5 * dt * torch.sum((T - torch.tensor(target, device="cuda")) ** 2)).backward()
    got = np.concatenate([t.grad.cpu().numpy() for t in leaves])
    assert np.linalg.norm(got - ref) < 1e-8 * np.linalg.norm(ref)
    g.close()
