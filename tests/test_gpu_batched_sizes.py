"""The one-barrier batched engine against the plain-staging one (pipeline = 0) where
its box sizes and CTA counts differ: one-warp 32 x 8 and 32 x 16 subdomains, wider
ones, and per-point sigma fields.  Same cycle counts and iterates bit for bit."""
import pytest

import workloads as W
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


SIZES = {"uneven": [(200, 130), (3, 2), (33, 32), (64, 1), (32, 97)], "one": [(129, 65)],
         "many": [(20 + i % 90, 100 - i % 77) for i in range(600)]}


@pytest.mark.parametrize("sizes,tile,prec,field", [("uneven", (32, 8), "f32_ir", False), ("many", (32, 8), "f32_ir", False),
                                                    ("uneven", (32, 16), "bf16corr_ir", False), ("many", (32, 16), "f32_ir", False),
                                                    ("uneven", (64, 32), "f32_ir", False), ("one", (64, 64), "f32_ir", True),
                                                    ("uneven", (32, 32), "f32_ir", True), ("uneven", (32, 8), "bf16corr_ir", True),
                                                    ("many", (32, 32), "f32_ir", True)])
def test_one_barrier_engine_equals_plain_engine(sizes, tile, prec, field):
    import torch
    import paper_2006_16465_gb300 as hj
    probs = []
    for i, (nx, ny) in enumerate(SIZES[sizes]):
        st = W.poisson_stencil(2, nx, ny, sigma_const=5.0 + (7 * i) % 90)
        f = W.zeros_grid(st)
        f[1:-1, 1:-1] = W.uniform(90 + i, nx * ny, -1, 1).reshape(ny, nx)
        probs.append(W.Problem(st, f, W.zeros_grid(st)))
    fs = [to_dev(q.f, 2, torch.float64) for q in probs]
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    sg = [torch.rand(f.shape, generator=g, device="cuda", dtype=torch.float64) * 50 if field and i % 2 == 0 else None
          for i, f in enumerate(fs)]
    descs = [hj.make_desc(2, q.st.nx, q.st.ny, f.shape[1], q.st.cW, q.st.cE, q.st.cS, q.st.cN, q.st.cD, q.st.sigma_const, s)
             for q, f, s in zip(probs, fs, sg)]
    runs = []
    for pipeline in (-1, 0):
        h = hj.Solver(probs[0].st, tile_x=tile[0], tile_y=tile[1], k=8, precision=prec, tol=1e-7, pipeline=pipeline)
        us = [torch.zeros_like(f) for f in fs]
        cyc = (hj.C.c_longlong * len(probs))()
        code = hj.hj_solve_batched(h.h, descs, [f.data_ptr() for f in fs], [u.data_ptr() for u in us], 0, None, cyc)
        h.close()
        runs.append((code, list(cyc), us))
    assert runs[0][:2] == runs[1][:2] and runs[0][0] == 0
    assert all(torch.equal(a, b) for a, b in zip(runs[0][2], runs[1][2]))
