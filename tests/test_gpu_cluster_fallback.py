"""CG of a small mesh on a device that cannot place the one-kernel solve's cluster.

That kernel needs a cluster of 8 CTAs (up to 1,500 nodes from p = 2 on) or of 16.  In the SEM_DEBUG
build sem_debug_limit_cluster makes the context take the device for a smaller one: the solves then
run a kernel per step, told by their launch count (three a time step otherwise: ionic update, solve,
residual; and the inverse diagonals of the first step's alpha and of the others'), and give the same fields up to the solver's tolerance.
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
for p, dims, need in ((2, (8, 4, 2), 8), (3, (9, 5, 4), 16), (1, (9, 5, 4), 16)):
    s = W.slab(*dims, (20.0, 7.0, 3.0), perturb=0.1, seed=1)
    g = gb.Slab(s.flat_vertices(), *dims, p, "LGL")
    g.set_ionic()
    g.set_stimulus("box", (0.0, 0.0, 0.0, 3.0, 3.0, 3.0), 50.0, 0.0, 1.0)
    ref = None
    for limit in (16, 15, 8, 7, 0):
        capi.sem_debug_limit_cluster(g.ctx, limit)
        st = g.new_state(-85.0, 1.0)
        r = st.step(0.05, 6, rtol=1e-12)
        assert (r.kernel_launches == 3 * 6 + 2) == (limit >= need), (p, dims, limit, r.kernel_launches)
        u = st.get()[0].clone()
        ref = u if ref is None else ref
        assert float(torch.linalg.norm(u - ref) / torch.linalg.norm(ref)) < 1e-10, (p, dims, limit)
        st.close()
    g.close()
print("cluster fallback ok")
"""


def test_small_cg_without_its_cluster():
    from paper_2205_05136_gb300 import build
    env = dict(os.environ)
    env["SEM_LIBRARY"] = build.build(debug=True)
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "cluster fallback ok" in r.stdout


def test_normal_build_has_no_cluster_limit():
    s = W.slab(2, 2, 1, (2.0, 2.0, 1.0))
    g = gb.Slab(s.flat_vertices(), 2, 2, 1, 2, "LGL")
    with pytest.raises(capi.SemError) as e:
        capi.sem_debug_limit_cluster(g.ctx, 0)
    assert e.value.code == capi.SEM_ERR_UNSUPPORTED
    g.close()
