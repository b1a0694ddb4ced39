"""In-place runs: which engine the library picks by itself, and what they give
where the halo never changes (one subdomain)."""
import pytest

import oracle
import workloads as W
from helpers import gpu_solver, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("prec,nx,ny,threads", [("f64", 96, 80, 128), ("f64", 320, 310, 128), ("f64", 780, 700, (128, 64)),
                                                 ("f32", 96, 80, 32), ("f32", 500, 450, 32), ("f32_ir", 96, 80, 32),
                                                 ("f32_ir", 500, 450, 32)])
def test_automatic_in_place_runs_take_the_persistent_engine(prec, nx, ny, threads):
    """9, 100 and 550 binary64 subdomains (clusters and eight warps are for runs in
    two arrays), one warp each in binary32: the persistent engine, whose array is one
    cycle past the checked one, and threads that can be set again."""
    import torch
    dt = torch.float32 if prec == "f32" else torch.float64
    p = W.random_bc_problem(2, nx, ny, seed=7, sigma_kind="const")
    tol = 1e-2
    s = gpu_solver(p, precision=prec, tile_x=32, tile_y=32, k=8, tol=tol, in_place=1)
    u = to_dev(p.u0, 2, dt)
    out = s.solve(to_dev(p.f, 2, dt), u)
    s.close()
    assert out["status"] == 0 and out["persistent"] == 1
    assert out["tile_threads"] in (threads if isinstance(threads, tuple) else (threads,))
    r0 = oracle.residual(p.st, p.f, p.u0)
    assert oracle.residual(p.st, p.f, to_host(u, nx)) <= tol * r0 * 1.01
    gpu_solver(p, precision=prec, tile_x=32, tile_y=32, k=8, tol=tol, in_place=1, tile_threads=out["tile_threads"]).close()


@pytest.mark.parametrize("prec,tile,threads,coef", [("f32", (32, 32), 64, False), ("f32", (32, 32), 256, False),
                                                     ("f64", (32, 32), 0, False), ("f64", (32, 32), 256, False),
                                                     ("f64", (64, 64), 0, False), ("f32", (32, 32), 0, True),
                                                     ("f32", (32, 28), 0, True), ("f64", (16, 16), 0, True)])
@pytest.mark.parametrize("k,cycles", [(1, 25), (1, 1), (3, 7)])
def test_one_subdomain_in_place_equals_two_arrays(prec, tile, threads, coef, k, cycles):
    """A grid of one subdomain has no neighbour whose writes it could see: in place
    it gives what two arrays give, bit for bit (all warps stage before any writes)."""
    import torch
    nx, ny = tile
    dt = torch.float32 if prec == "f32" else torch.float64
    p = (W.variable_coef_problem(2, nx, ny, seed=3) if coef
         else W.random_bc_problem(2, nx, ny, seed=3, sigma_kind="const", asym=True))
    us = []
    for in_place in (0, 1):
        s = gpu_solver(p, precision=prec, tile_x=nx, tile_y=ny, tile_threads=threads, k=k, fixed_cycles=cycles,
                       pipeline=0, in_place=in_place)
        u = to_dev(p.u0, 2, dt)
        s.solve(to_dev(p.f, 2, dt), u)
        s.close()
        us.append(u[:, :nx + 2])
    assert torch.equal(us[0], us[1])
