"""Error paths of the engines: what a call leaves behind when a bounded device
wait expires.  Child processes, since the handle is unusable afterwards."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _child(script, env=None, timeout=300):
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True, timeout=timeout,
                       env=dict(os.environ, **(env or {})))
    assert r.returncode == 0, r.stderr[-3000:]
    return r


_BATCH_EXPIRY = r"""
import os, sys
sys.path.insert(0, os.getcwd())
sys.path.insert(0, os.path.join(os.getcwd(), "tests"))
os.environ["HJ_TEST_SKIP_BARRIER_CTA"] = "0"
os.environ["HJ_TEST_BARRIER_TIMEOUT_NS"] = "50000000"
import torch
import paper_2006_16465_gb300 as hj
import workloads as W
pipeline, prec, nprob, field = int(sys.argv[1]), sys.argv[2], int(sys.argv[3]), int(sys.argv[4])
probs = [W.poisson2d_uniform(70 + 13 * i, 45 + 9 * i, seed=i) for i in range(nprob)]
s = hj.Solver(probs[0].st, tile_x=32, tile_y=32, k=4, precision=prec, tol=1e-8, pipeline=pipeline)
fs = [hj.grid_from(p.f, 2, torch.float64) for p in probs]
us = [hj.grid_from(p.u0, 2, torch.float64) for p in probs]
for u in us:
    u[1:-1, 1:-1] += 0.25
keep = [u.clone() for u in us]
sg = [torch.full_like(f, 3.0) if field else None for f in fs]
descs = [hj.make_desc(2, p.st.nx, p.st.ny, f.shape[1], p.st.cW, p.st.cE, p.st.cS, p.st.cN, p.st.cD, p.st.sigma_const, g)
         for p, f, g in zip(probs, fs, sg)]
code = hj.hj_solve_batched(s.h, descs, [f.data_ptr() for f in fs], [u.data_ptr() for u in us], 0)
print("RESULT", code, all(torch.equal(a, b) for a, b in zip(us, keep)))
s.close()
"""


@pytest.mark.parametrize("pipeline,prec,nprob,field", [(-1, "f32_ir", 1, 0), (-1, "f32_ir", 5, 0), (-1, "f32_ir", 3, 1),
                                                        (-1, "bf16corr_ir", 3, 0), (0, "f32_ir", 3, 0)])
def test_batched_expiry_leaves_the_iterates(pipeline, prec, nprob, field):
    """One CTA of the inner launch leaves before the grid barrier (test hook); the
    others give up after 50 ms.  No problem has a correction then (its cycle index
    is still -1): the call returns HJ_ERR_TIMEOUT and the iterates are the caller's."""
    import paper_2006_16465_gb300 as hj
    script = f"import sys; sys.argv[1:] = {[str(pipeline), prec, str(nprob), str(field)]!r}\n" + _BATCH_EXPIRY
    line = [ln for ln in _child(script).stdout.splitlines() if ln.startswith("RESULT")][0].split()
    assert int(line[1]) == hj.HJ_ERR_TIMEOUT and line[2] == "True", line
