"""Both sides of the rules by which a call takes one kernel or another, at the sizes
around their lines: the same iterates and cycle counts, or the oracle's."""
import numpy as np
import pytest

import oracle
import workloads as W
from helpers import gpu_solver, rel_max, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _dt(prec):
    import torch
    return torch.float32 if prec == "f32" else torch.float64


def _solve(p, dim, history=0, **kw):
    s = gpu_solver(p, **kw)
    u = to_dev(p.u0, dim, _dt(kw["precision"]))
    out = s.solve(to_dev(p.f, dim, _dt(kw["precision"])), u, history=history, check=False)
    s.close()
    return out, to_host(u, p.st.nx)


@pytest.mark.parametrize("prec,tile,n", [("f64", (32, 32), (96, 80)), ("f64", (32, 8), (70, 45)), ("f32", (32, 32), (200, 130)),
                                          ("f32", (32, 16), (64, 64)), ("f64", (128, 1), (300, 3))])
def test_short_solves_equal_the_persistent_engine(prec, tile, n):
    """Small grids run their first 48 launches singly, checked in short runs, then
    graphs: every cycle cap around those lengths, and tolerances met within them."""
    dim = 1 if tile[1] == 1 else 2
    p = W.random_bc_problem(dim, *n, seed=17, sigma_kind="const")
    base = dict(precision=prec, tile_x=tile[0], tile_y=tile[1], k=3)
    runs = [dict(tol=0.0, max_cycles=m) for m in (1, 2, 3, 4, 5, 6, 7, 11, 12, 13, 46, 47, 48, 49, 66, 113, 114, 115, 200)]
    runs += [dict(tol=t, max_cycles=100000) for t in (1.0, 0.9, 0.5, 0.2, 0.1, 0.05, 0.02, 0.01)]
    for kw in runs:
        a, ua = _solve(p, dim, history=300, persistent=-1, **base, **kw)
        b, ub = _solve(p, dim, history=300, persistent=1, pipeline=0, **base, **kw)
        assert (a["persistent"], b["persistent"]) == (0, 1)
        assert (a["status"], a["cycles"]) == (b["status"], b["cycles"]), kw
        assert np.array_equal(ua, ub), kw
        assert a["history_len"] == b["history_len"] and np.allclose(a["history"], b["history"], rtol=1e-6, atol=0), kw
        assert a["rel_final"] == pytest.approx(b["rel_final"], rel=1e-6), kw


@pytest.mark.parametrize("prec,tile,n", [("f32", (32, 32), (2200, 2080)), ("f32", (32, 16), (1500, 2600)), ("f32", (32, 8), (1100, 1000)),
                                          ("f64", (32, 8), (1100, 1000)), ("f32", (32, 16), (3000, 1500))])
def test_folds_of_many_ctas_equal_the_pipelined_kernel(prec, tile, n):
    """One partial per CTA, 4,000 to 9,000 of them, folded in the next launch or (the
    last case and 32 x 8) reduced at the launch's end."""
    p = W.random_bc_problem(2, *n, seed=8, sigma_kind="const")
    res = [_solve(p, 2, precision=prec, tile_x=tile[0], tile_y=tile[1], k=2, tol=2e-2, check_every=6, pipeline=pl, persistent=0)
           for pl in (0, 1)]
    (a, ua), (b, ub) = res
    assert a["status"] == 0 and a["cycles"] == b["cycles"] and np.array_equal(ua, ub)


@pytest.mark.parametrize("shape,tile,k", [((64, 224, 224), (16, 8, 8), 1), ((60, 230, 222), (16, 8, 8), 4), ((250, 130, 110), (16, 8, 8), 4),
                                           ((33, 300, 230), (16, 8, 4), 2), ((240, 120, 120), (16, 8, 8), 1), ((64, 224, 120), (16, 8, 4), 8)])
def test_3d_pairs_and_single_subdomains_equal_the_one_warp_kernel(shape, tile, k):
    """Even and odd numbers of 16-wide subdomains, with and without the residual."""
    import torch
    nx, ny, nz = shape
    import paper_2006_16465_gb300 as hj
    st = W.poisson3d_uniform(nx, ny, nz, seed=1).st
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    f = hj.alloc_grid(3, nx, ny, torch.float32, nz=nz)
    f[1:-1, 1:-1, 1:nx + 1] = torch.rand((nz, ny, nx), generator=g, device="cuda") - 0.5
    u0 = hj.alloc_grid(3, nx, ny, torch.float32, nz=nz)
    u0[..., :nx + 2] = torch.rand((nz + 2, ny + 2, nx + 2), generator=g, device="cuda") - 0.5
    for kw in (dict(fixed_cycles=3), dict(tol=0.0, max_cycles=5)):
        us = []
        for pipeline in (-1, 0):
            s = hj.Solver(st, precision="f32", tile_x=tile[0], tile_y=tile[1], tile_z=tile[2], k=k, pipeline=pipeline, **kw)
            u = u0.clone()
            out = s.solve(f, u, check=False)
            assert out["pipeline_stages"] == (1 if pipeline == -1 else 0)
            s.close()
            us.append(u[..., :nx + 2])
        assert torch.equal(us[0], us[1])


@pytest.mark.parametrize("tile", [(32, 4), (32, 12), (32, 24), (32, 32)])
@pytest.mark.parametrize("n,threads_per_point", [((457, 313), False), ((130, 70), True)])
def test_varcoef_rows_and_points_match_oracle(tile, n, threads_per_point):
    """Four rows a warp from 900 points per SM on, a thread per point below."""
    p = W.variable_coef_problem(2, *n, seed=6, contrast=8.0, screening=20.0)
    out, u = _solve(p, 2, precision="f32", tile_x=tile[0], tile_y=tile[1], k=3, fixed_cycles=4)
    rows = not threads_per_point or tile[1] >= 28
    assert out["tile_threads"] == (8 if rows else 32) * tile[1]
    assert rel_max(u, oracle.run_fixed(p.st, p.f, p.u0, 4, tile[0], tile[1], 3)) <= 1e-5
    out, u = _solve(p, 2, precision="f32", tile_x=tile[0], tile_y=tile[1], k=3, tol=0.0, max_cycles=9)
    assert rel_max(u, oracle.run_fixed(p.st, p.f, p.u0, 9, tile[0], tile[1], 3)) <= 1e-5


@pytest.mark.parametrize("n", [(300, 200), (700, 500), (1300, 1000)])
@pytest.mark.parametrize("prec,sigma", [("f64", "field"), ("f64", "none"), ("f32", "field"), ("f32", "none")])
def test_residual_forms_match_oracle(n, prec, sigma):
    """A point a thread, rows (between), and a point a thread again: ||f - A u|| to
    rounding (binary64 arithmetic on the same inputs)."""
    import torch
    p = W.random_bc_problem(2, *n, seed=9, sigma_kind=sigma)
    if prec == "f32":
        p.f = p.f.astype(np.float32).astype(np.float64)
        p.u0 = p.u0.astype(np.float32).astype(np.float64)
    s = gpu_solver(p, precision=prec)
    a, _ = s.residual(to_dev(p.f, 2, _dt(prec)), to_dev(p.u0, 2, _dt(prec)))
    s.close()
    assert a == pytest.approx(oracle.residual(p.st, p.f, p.u0), rel=1e-12)


@pytest.mark.parametrize("n", [(45, 37), (560, 540)])
def test_bf16_ragged_subdomains_equal_padded_ones(n):
    """Guarded 16-bit loads at the ragged edge: the engines that stage by copies
    (zero fill) and by guarded loads give the same corrections."""
    p = W.random_bc_problem(2, *n, seed=12, sigma_kind="const")
    kw = dict(precision="bf16corr_ir", tile_x=32, tile_y=32, k=4, tol=1e-6, inner_tol=1e-2, max_outer=6)
    (a, ua), (b, ub) = _solve(p, 2, persistent=-1, **kw), _solve(p, 2, persistent=1, **kw)
    assert a["cycles"] == b["cycles"] and np.array_equal(ua, ub)
