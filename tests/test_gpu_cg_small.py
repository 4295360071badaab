"""The one-kernel CG of small meshes against a sparse direct solve.

Meshes of one element (most CTAs of the cluster without work), of a few nodes a CTA, with more
elements a CTA than one batch, on both sides of the change from 8 to 16 CTAs, and past its range
(the launch-per-step path); Jacobi and no preconditioner, whose solves take more iterations than
one launch runs; an iteration limit in the middle; a carried initial residual (time steps).  The
bound is that of the other CG tests, 1e-11 at rtol 1e-13.
"""
import numpy as np
import pytest
import scipy.sparse.linalg as spla
import torch

import workloads as W
from oracle import mesh as Mh

pytestmark = pytest.mark.gpu

gb = pytest.importorskip("paper_2205_05136_gb300")
capi = gb.capi

ALPHA = 1.5 / 0.05


def _problem(dims, p, quad):
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    tissue = (np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), W.transmural_fiber_angles(s))
    g = gb.Slab(s.flat_vertices(), *dims, p, quad)
    g.set_tissue(*tissue)
    return s, tissue, g


@pytest.mark.parametrize("quad", ["LGL", "LG"])
@pytest.mark.parametrize("p,dims", [(1, (1, 1, 1)), (1, (19, 9, 7)), (2, (3, 1, 1)), (2, (9, 5, 4)), (2, (13, 7, 5)),
                                    (3, (5, 4, 3)), (4, (6, 3, 2)), (4, (10, 6, 4)), (5, (4, 2, 2)), (6, (2, 2, 1))])
def test_small_cg_matches_direct_solve(p, dims, quad):
    s, tissue, g = _problem(dims, p, quad)
    o = Mh.SlabSpace(s.flat_vertices(), *dims, p, quad)
    A = Mh.assemble(o, tissue, ALPHA, 1.0).tocsc()
    b = W.uniform_vector(o.ndofs, -1.0, 1.0, seed=5)
    ref = spla.spsolve(A, b)
    bt = torch.tensor(b, device="cuda")
    for precond in (capi.SEM_PC_JACOBI, capi.SEM_PC_NONE):
        x = torch.zeros_like(bt)
        it, res = g.cg_solve(ALPHA, bt, x, rtol=1e-13, maxit=5000, precond=precond)
        assert np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-11, (precond, it)
        true = float(np.linalg.norm(b - A @ x.cpu().numpy()))
        assert abs(res - true) < 1e-12 * np.linalg.norm(b)
        if it > 3:  # stopped in the middle, then continued from that iterate
            y = torch.zeros_like(bt)
            rc, half, _ = capi.sem_cg_solve(g.ctx, ALPHA, bt, y, 1e-13, 0.0, it // 2, precond, raise_on_error=False)
            assert rc == capi.SEM_ERR_NOT_CONVERGED and half == it // 2
            g.cg_solve(ALPHA, bt, y, rtol=1e-13, maxit=5000, precond=precond)
            assert np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-11
    bad = bt.clone()
    bad[-1] = float("nan")
    with pytest.raises(capi.SemError) as e:
        g.cg_solve(ALPHA, bad, torch.zeros_like(bt))
    assert e.value.code == capi.SEM_ERR_NONFINITE
    g.close()


@pytest.mark.parametrize("quad", ["LGL", "LG"])
def test_small_steps_match_launched_steps(quad):
    """Time steps (with the carried residual) of the one-kernel solve and of the deterministic mode, which
    takes the launch-per-step path: the same fields up to the solver's tolerance, the same iteration count."""
    out = []
    for det in (False, True):
        s, tissue, g = _problem((9, 5, 4), 2, quad)
        capi.sem_set_deterministic(g.ctx, det)
        g.set_ionic()
        g.set_stimulus("box", (0.0, 0.0, 0.0, 3.0, 3.0, 3.0), 50.0, 0.0, 1.0)
        st = g.new_state(-85.0, 1.0)
        r = st.step(0.05, 30, rtol=1e-12)
        out.append((*st.get()[:2], r.cg_iters))
        st.close()
        g.close()
    (u0, h0, i0), (u1, h1, i1) = out
    assert float(torch.linalg.norm(u0 - u1) / torch.linalg.norm(u1)) < 1e-10
    assert float(torch.linalg.norm(h0 - h1) / torch.linalg.norm(h1)) < 1e-11
    assert abs(i0 - i1) <= 2, (i0, i1)


def test_timing_changes_the_timed_solve_only():
    """With timing on, one solve in ten runs a kernel per step to bracket its apply; the nine after it
    launch what they launch with timing off (three kernels a time step)."""
    s, tissue, g = _problem((9, 5, 4), 2, "LGL")
    g.set_ionic()
    g.set_stimulus("box", (0.0, 0.0, 0.0, 3.0, 3.0, 3.0), 50.0, 0.0, 1.0)
    st = g.new_state(-85.0, 1.0)
    st.step(0.05, 2, rtol=1e-12)  # both alphas' diagonals
    assert st.step(0.05, 9, rtol=1e-12).kernel_launches == 3 * 9
    capi.sem_set_timing(g.ctx, True)
    timed = st.step(0.05, 1, rtol=1e-12)
    assert timed.n_apply == 1 and timed.apply_ms > 0.0 and timed.kernel_launches > 3
    rest = st.step(0.05, 9, rtol=1e-12)
    assert rest.n_apply == 0 and rest.kernel_launches == 3 * 9
    assert st.step(0.05, 1, rtol=1e-12).n_apply == 1
    st.close()
    g.close()
