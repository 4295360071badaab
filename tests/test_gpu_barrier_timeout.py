"""The one-kernel CG vector update whose grid barrier does not open.

In the SEM_DEBUG build sem_debug_hold_update keeps one CTA (the first, one in the middle, the last)
from arriving at the barrier: the others' bounded wait runs out, the kernel returns, the solve gives
SEM_ERR_TIMEOUT, and the next solve is right, although arrivals were left behind: solves run on a
stream that does not synchronise with the legacy default stream.  The bound on the solution is that
of the kernel's other tests, 2 rtol |b| / (alpha min(diag M / 8)).
"""
import os
import subprocess
import sys

import pytest

import workloads as W

pytestmark = pytest.mark.gpu

gb = pytest.importorskip("paper_2205_05136_gb300")
capi = gb.capi

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path.insert(0, {root!r})
import torch
import workloads as W
from paper_2205_05136_gb300 import capi
import paper_2205_05136_gb300 as gb
assert "SEM_DEBUG" in capi.sem_version(), capi.sem_version()
ALPHA, RTOL = 30.0, 1e-10
s = W.slab(63, 39, 49, (20.0, 7.0, 3.0), perturb=0.1, seed=1)   # 128,000 nodes: 143 CTAs
g = gb.Slab(s.flat_vertices(), s.nx, s.ny, s.nz, 1, "LGL")
mass = g.apply(torch.ones(g.ndofs, dtype=torch.float64, device="cuda"), 1.0, 0.0)
b = mass * torch.tensor(W.uniform_vector(g.ndofs, -1.0, 1.0, seed=4), device="cuda")
bound = 2 * RTOL * float(torch.linalg.norm(b)) / (ALPHA * float(mass.min()) / 8)
torch.cuda.synchronize()
with torch.cuda.stream(torch.cuda.Stream()):
    ref = torch.zeros_like(b)
    n0 = g.cg_solve(ALPHA, b, ref, rtol=RTOL)[0]
    for cta in (0, 60, 142):
        capi.sem_debug_hold_update(g.ctx, cta)
        rc, _, _ = capi.sem_cg_solve(g.ctx, ALPHA, b, torch.zeros_like(b), RTOL, 0.0, 100, raise_on_error=False)
        assert rc == capi.SEM_ERR_TIMEOUT, (cta, rc)
        capi.sem_debug_hold_update(g.ctx, -1)
        x = torch.zeros_like(b)
        n1 = g.cg_solve(ALPHA, b, x, rtol=RTOL)[0]
        assert abs(n1 - n0) <= 1, (cta, n0, n1)
        assert float(torch.linalg.norm(x - ref)) < bound, cta
g.close()
print("barrier timeout ok")
"""


def test_update_barrier_timeout_is_reported_and_recovered():
    from paper_2205_05136_gb300 import build
    env = dict(os.environ)
    env["SEM_LIBRARY"] = build.build(debug=True)
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "barrier timeout ok" in r.stdout


def test_normal_build_has_no_held_barrier():
    s = W.slab(2, 2, 1, (2.0, 2.0, 1.0))
    g = gb.Slab(s.flat_vertices(), 2, 2, 1, 2, "LGL")
    with pytest.raises(capi.SemError) as e:
        capi.sem_debug_hold_update(g.ctx, 0)
    assert e.value.code == capi.SEM_ERR_UNSUPPORTED
    g.close()
