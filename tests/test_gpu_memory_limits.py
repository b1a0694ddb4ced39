"""What runs when the third iterate (correction) buffers cannot be had: the grid
reduction and the two-barrier batched engine, with the same iterates, and without
asking again.  A child process on the debug library, which refuses allocations
above a limit."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_SCRIPT = r"""
import os, sys
sys.path.insert(0, os.getcwd())
sys.path.insert(0, os.path.join(os.getcwd(), "tests"))
import torch
import paper_2006_16465_gb300 as hj
import workloads as W
from helpers import gpu_solver, to_dev
assert hj.LIB_PATH.name == "libhj_debug.so"
kind = sys.argv[1]

def limit(n):
    if n is None:
        os.environ.pop("HJ_TEST_ALLOC_LIMIT", None)
    else:
        os.environ["HJ_TEST_ALLOC_LIMIT"] = str(n)

def single(prec, dim, nx, ny, **kw):
    p = W.random_bc_problem(dim, nx, ny, seed=4, sigma_kind="const")
    out = []
    for refuse in (False, True):
        s = gpu_solver(p, precision=prec, check_every=8, **kw)
        dt = torch.float32 if prec == "f32" else torch.float64
        f, u = to_dev(p.f, dim, dt), to_dev(p.u0, dim, dt)
        limit(1024 if refuse else None)
        o = s.solve(f, u)
        u2 = to_dev(p.u0, dim, dt)
        o2 = s.solve(f, u2)          # a second call asks for nothing
        limit(None)
        assert o["status"] == 0 and o2["cycles"] == o["cycles"] and torch.equal(u, u2)
        out.append((o["cycles"], u))
        s.close()
    assert out[0][0] == out[1][0] and torch.equal(out[0][1], out[1][1]), [o[0] for o in out]

if kind == "f64":
    single("f64", 2, 96, 80, tile_x=32, tile_y=32, k=8, tol=1e-3)      # clusters
elif kind == "1d":
    single("f64", 1, 300, 3, tile_x=128, k=16, tol=1e-3)
elif kind == "ir":
    single("f32_ir", 2, 200, 150, tile_x=32, tile_y=32, k=16, tol=1e-9, inner_tol=1e-2)   # several inner solves
else:
    probs = [W.poisson2d_uniform(70 + 13 * i, 45 + 9 * i, seed=i) for i in range(4)]
    fs = [to_dev(p.f, 2, torch.float64) for p in probs]
    descs = [hj.make_desc(2, p.st.nx, p.st.ny, f.shape[1], p.st.cW, p.st.cE, p.st.cS, p.st.cN, p.st.cD, p.st.sigma_const)
             for p, f in zip(probs, fs)]
    ref = None
    for refuse in (False, True):
        s = gpu_solver(probs[0], precision=kind, tile_x=32, tile_y=32, k=8, tol=1e-6)
        for call in range(3):
            us = [torch.zeros_like(f) for f in fs]
            cyc = (hj.C.c_longlong * 4)()
            # two binary64, one binary32 and the corrections: room for all but the third ones
            dsz = 2 if kind == "bf16corr_ir" else 4
            need = sum(((p.st.ny + 2) * f.shape[1] * 8 + 255) // 256 * 256
                       + ((p.st.ny + 2) * ((p.st.nx + 33) // 32 * 32) * 4 + 255) // 256 * 256
                       + 2 * (((p.st.ny + 2) * ((p.st.nx + 33) // 32 * 32) * dsz + 255) // 256 * 256)
                       for p, f in zip(probs, fs))
            limit(need if refuse else None)
            code = hj.hj_solve_batched(s.h, descs, [f.data_ptr() for f in fs], [u.data_ptr() for u in us], 0, None, cyc)
            limit(None)
            assert code == 0, hj.hj_last_error()
            got = (list(cyc), us)
            if ref is None:
                ref = got
            assert got[0] == ref[0] and all(torch.equal(a, b) for a, b in zip(got[1], ref[1]))
        s.close()
code, site, index = hj.hj_debug_check()
print("CHECK", code, site, index)
"""


@pytest.mark.parametrize("kind", ["f64", "1d", "ir", "f32_ir", "bf16corr_ir"])
def test_runs_without_the_third_buffer(kind):
    sys.path.insert(0, ROOT)
    from paper_2006_16465_gb300 import _build
    _build.build(debug=True)
    r = subprocess.run([sys.executable, "-c", f"import sys; sys.argv[1:] = [{kind!r}]\n" + _SCRIPT], cwd=ROOT,
                       env=dict(os.environ, HJ_LIBRARY="debug"), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    assert [ln for ln in r.stdout.splitlines() if ln.startswith("CHECK")][0].split()[1] == "0"
    refused = [ln for ln in r.stderr.splitlines() if ln.startswith("HJ_TEST_ALLOC_LIMIT")]
    assert len(refused) == 1, refused   # asked for once, not in every call or refinement step
