"""Which kernels a CG solve runs, and the one-kernel vector update's endings.

A time step's launch count tells its path: ionic update, residual and solve, the solve being one
launch of the small-mesh kernel per 64 iterations, or the initial residual and, an iteration, two
launches (apply, one-kernel update: 100,000 to 622,592 nodes) or four (apply, sum, two updates) in
chunks of 4, 8, 16, 16, ...  Meshes on both sides of every limit; the other tests compare results.

The update's endings: a non-finite value that first appears in an iteration (zero tissue and alpha 0:
p . A p = 0), an iteration limit inside and at the edge of a chunk, and the deterministic mode (bitwise
repeat).  Bound on the solution as in the kernel's other tests, 2 rtol |b| / (alpha min(diag M / 8)).
"""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

gb = pytest.importorskip("paper_2205_05136_gb300")
capi = gb.capi

ALPHA, RTOL = 30.0, 1e-10


def _slab(p, quad, dims):
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    g = gb.Slab(s.flat_vertices(), *dims, p, quad)
    g.set_tissue(np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), W.transmural_fiber_angles(s))
    return s, g


def _launched(iters):
    """Iterations launched for a solve that takes `iters`."""
    total, chunk = 4, 8
    while total < iters:
        total, chunk = total + chunk, min(16, 2 * chunk)
    return total


def _step(g, precond=gb.SEM_PC_JACOBI):
    """Statistics of a time step that carries its initial residual."""
    g.set_ionic()
    g.set_stimulus("box", (0.0, 0.0, 0.0, 3.0, 3.0, 3.0), 50.0, 0.0, 1.0)
    st = g.new_state(-85.0, 1.0)
    st.step(0.05, 3, rtol=RTOL, maxit=5000, precond=precond)
    r = st.step(0.05, 1, rtol=RTOL, maxit=5000, precond=precond)
    st.close()
    return r


@pytest.mark.parametrize("p,quad,dims,one", [
    (1, "LGL", (20, 14, 13), True), (1, "LGL", (20, 14, 14), False),     # 4,410 and 4,725 nodes
    (1, "LG", (15, 11, 11), True), (1, "LG", (20, 14, 7), False),        # 2,304 and 2,520
    (2, "LGL", (14, 8, 7), True), (2, "LGL", (14, 8, 8), False),         # 7,395 and 8,381
    (2, "LG", (14, 8, 5), True), (2, "LG", (14, 8, 6), False),           # 5,423 and 6,409
    (3, "LGL", (12, 6, 4), True), (3, "LGL", (12, 6, 5), False),         # 9,139 and 11,248
    (4, "LG", (7, 5, 4), True), (4, "LG", (7, 5, 5), False),             # 10,353 and 12,789
    (6, "LGL", (7, 4, 2), True), (6, "LGL", (8, 4, 2), False)])          # 13,975 and 15,925
def test_small_mesh_limits(p, quad, dims, one):
    s, g = _slab(p, quad, dims)
    r = _step(g)
    mass = 1 if quad == "LG" else 0  # the consistent mass of the right-hand side
    if one:
        assert r.kernel_launches == 3 + mass + (max(r.cg_iters, 1) - 1) // 64, (g.ndofs, r.cg_iters)
    else:
        assert r.kernel_launches == 3 + mass + 4 * _launched(r.cg_iters), (g.ndofs, r.cg_iters)
    g.close()


def test_small_mesh_solve_continues_past_64_iterations():
    s, g = _slab(6, "LG", (3, 2, 1))
    r = _step(g, gb.SEM_PC_NONE)
    assert r.cg_iters > 64 and r.kernel_launches == 4 + (r.cg_iters - 1) // 64, (r.cg_iters, r.kernel_launches)
    g.close()


@pytest.mark.parametrize("df64", [False, True])
@pytest.mark.parametrize("p,dims,one", [(1, (99, 39, 23), False), (1, (99, 39, 24), True),      # 96,000 and 100,000 nodes
                                        (1, (127, 63, 75), True), (1, (127, 63, 76), False)])   # 622,592 and 630,784
def test_one_kernel_update_limits(p, dims, one, df64):
    s, g = _slab(p, "LGL", dims)
    if df64:
        capi.sem_set_operator_precision(g.ctx, capi.SEM_PREC_DF64)
    r = _step(g)
    assert r.kernel_launches == 3 + (2 if one else 4) * _launched(r.cg_iters), (g.ndofs, r.cg_iters)
    g.close()


DIMS = (63, 39, 49)  # p = 1: 128,000 nodes


@pytest.mark.parametrize("p,dims", [(1, DIMS), (2, (4, 3, 2)), (1, (127, 63, 76))])  # update, small mesh, four launches
def test_value_that_turns_non_finite_in_an_iteration(p, dims):
    s, g = _slab(p, "LGL", dims)
    zero = np.zeros(s.n_elements)
    g.set_tissue(zero, zero, zero)
    b = torch.ones(g.ndofs, dtype=torch.float64, device="cuda")
    rc, it, _ = capi.sem_cg_solve(g.ctx, 0.0, b, torch.zeros_like(b), RTOL, 0.0, 100, capi.SEM_PC_NONE, raise_on_error=False)
    assert rc == capi.SEM_ERR_NONFINITE and it == 1
    g.set_tissue(np.full(s.n_elements, 0.12), np.full(s.n_elements, 0.03), zero)
    x = torch.zeros_like(b)
    g.cg_solve(ALPHA, b, x, rtol=RTOL)  # the context solves as before
    assert float(torch.linalg.norm(b - g.apply(x, ALPHA, 1.0))) < 2 * RTOL * float(torch.linalg.norm(b))
    g.close()


@pytest.mark.parametrize("df64", [False, True])
def test_update_iteration_limit_and_deterministic_mode(df64):
    s, g = _slab(1, "LGL", DIMS)
    if df64:
        capi.sem_set_operator_precision(g.ctx, capi.SEM_PREC_DF64)
    n = g.ndofs
    mass = g.apply(torch.ones(n, dtype=torch.float64, device="cuda"), 1.0, 0.0)
    b = mass * torch.tensor(W.uniform_vector(n, -1.0, 1.0, seed=4), device="cuda")
    nb = float(torch.linalg.norm(b))
    bound = 2 * RTOL * nb / (ALPHA * float(mass.min()) / 8)

    def solve(maxit, x=None):
        x = torch.zeros_like(b) if x is None else x
        rc, it, _ = capi.sem_cg_solve(g.ctx, ALPHA, b, x, RTOL, 0.0, maxit, capi.SEM_PC_JACOBI, raise_on_error=False)
        return rc, it, x

    rc, full, ref = solve(1000)
    assert rc == capi.SEM_OK and full > 5
    for maxit in (1, 4, 5, full - 1):
        rc, it, x = solve(maxit)
        assert rc == capi.SEM_ERR_NOT_CONVERGED and it == maxit
        rc, it, x = solve(1000, x)  # continued from that iterate
        assert rc == capi.SEM_OK and float(torch.linalg.norm(x - ref)) < bound
    capi.sem_set_deterministic(g.ctx, True)
    runs = [solve(1000) for _ in range(2)]
    assert torch.equal(runs[0][2], runs[1][2]) and runs[0][1] == runs[1][1]
    assert float(torch.linalg.norm(runs[0][2] - ref)) < bound
    g.close()
