"""The one-barrier batched kernel (decisions one cycle late, checks as queue
entries, CTAs leaving as the queue shrinks) against the plain-staging kernel
(pipeline = 0, two barriers a cycle): same cycle counts and iterates bit for bit,
for one problem, for more problems than CTAs can hold at once, for problems of
very different lengths, and where the inner cycle cap ends the solves."""
import numpy as np
import pytest

import workloads as W
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _run(probs, pipeline, prec, **kw):
    import torch
    import paper_2006_16465_gb300 as hj
    params = dict(tile_x=32, tile_y=32, k=8, precision=prec, tol=1e-7, max_outer=60)
    params.update(kw)
    s = hj.Solver(probs[0].st, pipeline=pipeline, **params)
    fs = [to_dev(q.f, 2, torch.float64) for q in probs]
    us = [to_dev(q.u0, 2, torch.float64) for q in probs]
    descs = [hj.make_desc(2, q.st.nx, q.st.ny, f.shape[1], q.st.cW, q.st.cE, q.st.cS, q.st.cN, q.st.cD, q.st.sigma_const)
             for q, f in zip(probs, fs)]
    cyc = (hj.C.c_longlong * len(probs))()
    code = hj.hj_solve_batched(s.h, descs, [f.data_ptr() for f in fs], [u.data_ptr() for u in us], 0, None, cyc)
    s.close()
    return code, list(cyc), us


def _problem(nx, ny, sigma, seed):
    st = W.poisson_stencil(2, nx, ny, sigma_const=sigma)
    f = W.zeros_grid(st)
    f[1:-1, 1:-1] = W.uniform(seed, nx * ny, -1, 1).reshape(ny, nx)
    return W.Problem(st, f, W.zeros_grid(st))


CASES = {
    "one": [(70, 45)],
    "one_tile": [(1, 1)],
    "uneven": [(200, 130), (3, 2), (33, 32), (64, 1), (32, 97)],
    "many": [(5 + i % 36, 40 - i % 33) for i in range(2200)],
}


@pytest.mark.parametrize("name,prec,kw", [("one", "f32_ir", {}), ("one_tile", "f32_ir", {}), ("uneven", "f32_ir", {}),
                                           ("uneven", "bf16corr_ir", {}), ("many", "f32_ir", {}),
                                           ("uneven", "f32_ir", dict(inner_max_cycles=1, max_outer=4)),
                                           ("uneven", "f32_ir", dict(inner_max_cycles=2, max_outer=4)),
                                           ("uneven", "f32_ir", dict(inner_max_cycles=3, max_outer=5))])
def test_late_decisions_equal_two_barrier_kernel(name, prec, kw):
    import torch
    probs = [_problem(nx, ny, 5.0 + (7 * i) % 90, 50 + i) for i, (nx, ny) in enumerate(CASES[name])]
    a, ca, ua = _run(probs, -1, prec, **kw)
    b, cb, ub = _run(probs, 0, prec, **kw)
    assert a == b and ca == cb
    assert all(torch.equal(x, y) for x, y in zip(ua, ub))
    assert np.isfinite(ua[0].sum().item())
