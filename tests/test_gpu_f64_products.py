"""Binary64 kernels share a neighbour's product c u between the points that read
it where coefficients are equal: none shared (general stencil), opposite pairs
equal (rectangular grid), all equal (square grid, cube).  Every rounding stays
where the general path has it, so the cycles equal the oracle's bit for bit in
each mode, on ragged grids and with a screening field."""
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


def _cycles(p, dim, **kw):
    import torch
    s = gpu_solver(p, precision="f64", **kw)
    u = to_dev(p.u0, dim, torch.float64)
    s.solve(to_dev(p.f, dim, torch.float64), u)
    s.close()
    return to_host(u, p.st.nx)


@pytest.mark.parametrize("engine", [dict(pipeline=0), dict(pipeline=1), dict(pipeline=0, overlap_x=4, overlap_y=6)])
@pytest.mark.parametrize("shape,sigma,asym", [((71, 71), "field", False), ((71, 71), "none", False),
                                               ((71, 38), "field", False), ((71, 71), "none", True)])
def test_2d_modes(shape, sigma, asym, engine):
    import paper_2006_16465_gb300 as hj
    p = W.random_bc_problem(2, *shape, seed=shape[1], sigma_kind=sigma, asym=asym)
    ovl = (engine.get("overlap_x", 0), engine.get("overlap_y", 0))
    for tx, ty, th in hj.hj_tile_variants(2, hj.PRECISIONS["f64"]):
        if engine["pipeline"]:
            th = 0   # the pipelined kernel is not built for every number of warps
        if max(ovl) and (ty <= max(ovl) or tx <= max(ovl)):
            continue
        got = _cycles(p, 2, tile_x=tx, tile_y=ty, tile_threads=th, k=3, fixed_cycles=3, **engine)
        ref = oracle.run_fixed(p.st, p.f, p.u0, 3, tx, ty, 3, overlap=ovl)
        assert np.array_equal(got, ref), (tx, ty, th, rel_max(got, ref))


@pytest.mark.parametrize("shape,asym", [((19, 19, 19), False), ((33, 33, 20), False), ((33, 20, 9), True)])
def test_3d_modes(shape, asym):
    import paper_2006_16465_gb300 as hj
    p = W.random_bc_problem3d(*shape, seed=sum(shape), sigma_kind="const", asym=asym)
    for tx, ty, tz in hj.hj_tile_shapes3d(hj.PRECISIONS["f64"]):
        got = _cycles(p, 3, tile_x=tx, tile_y=ty, tile_z=tz, k=3, fixed_cycles=2)
        ref = oracle.run_fixed(p.st, p.f, p.u0, 2, tx, ty, 3, tz=tz)
        assert np.array_equal(got, ref), (tx, ty, tz, rel_max(got, ref))


@pytest.mark.parametrize("shape,tile", [((63, 63), (32, 8)), ((63, 63), (16, 2)), ((95, 95), (8, 3)), ((63, 31), (32, 8))])
def test_multigrid_modes(shape, tile):
    p = W.random_bc_problem(2, *shape, seed=9, sigma_kind="const")
    L = oracle.mg_max_levels(*shape)
    got = _cycles(p, 2, method="mg", tile_x=tile[0], tile_y=tile[1], k=3, fixed_cycles=2)
    ref = p.u0
    for _ in range(2):
        ref = oracle.mg_vcycle(p.st, p.f, ref, L, 1, 1, tile[0], tile[1], 3, 0.8)
    assert np.array_equal(got, ref), rel_max(got, ref)


@pytest.mark.parametrize("scale,zeros", [(1e-303, False), (1e-306, True), (1e-311, False), (1e295, True), (1.0, True)])
@pytest.mark.parametrize("shape,asym", [((64, 64), False), ((71, 38), False)])
def test_products_at_the_edges_of_the_range(shape, asym, scale, zeros):
    """Products formed on the integer pipes cover normal numbers; zeros, subnormal
    values and products near the limits take the FP64 pipe, per subiteration."""
    import paper_2006_16465_gb300 as hj
    p = W.random_bc_problem(2, *shape, seed=77, sigma_kind="none", asym=asym)
    p.f *= scale
    p.u0 *= scale
    if zeros:   # half the grid exactly zero, its front moving one row a subiteration
        p.f[: shape[1] // 2] = 0.0
        p.u0[: shape[1] // 2] = 0.0
    for tx, ty, th in hj.hj_tile_variants(2, hj.PRECISIONS["f64"]):
        got = _cycles(p, 2, tile_x=tx, tile_y=ty, tile_threads=th, k=5, fixed_cycles=3, pipeline=0)
        ref = oracle.run_fixed(p.st, p.f, p.u0, 3, tx, ty, 5)
        assert np.array_equal(got, ref), (tx, ty, th, rel_max(got, ref))


@pytest.mark.parametrize("shape,tile,prec", [((191, 127), (32, 8), "f32"), ((191, 127), (32, 32), "f32"),
                                              ((255, 31), (32, 4), "f32"), ((191, 95), (32, 32), "f64"),
                                              ((127, 127), (1, 8), "f64")])
def test_multigrid_transfer_and_smoothing_edges(shape, tile, prec):
    """Ragged last subdomains of every level, levels of one CTA, and coarse levels
    of one row: binary64 bitwise, binary32 within 1e-5 of the oracle's V-cycles."""
    import torch
    p = W.random_bc_problem(2, *shape, seed=21, sigma_kind="const", asym=True)
    L = oracle.mg_max_levels(*shape)
    dt = torch.float32 if prec == "f32" else torch.float64
    s = gpu_solver(p, method="mg", precision=prec, tile_x=tile[0], tile_y=tile[1], k=3, mg_pre=2, mg_post=1, fixed_cycles=2)
    u = to_dev(p.u0, 2, dt)
    s.solve(to_dev(p.f, 2, dt), u)
    s.close()
    ref = p.u0
    for _ in range(2):
        ref = oracle.mg_vcycle(p.st, p.f, ref, L, 2, 1, tile[0], tile[1], 3, 0.8)
    got = to_host(u, shape[0])
    if prec == "f64":
        assert np.array_equal(got, ref), rel_max(got, ref)
    else:
        assert rel_max(got, ref) <= 1e-5


@pytest.mark.parametrize("shape,sigma,asym,ovl,k", [((96, 70), "field", True, 0, 4), ((64, 64), "none", False, 0, 1),
                                                     ((200, 150), "const", False, 0, 3), ((200, 150), "field", False, 6, 5),
                                                     ((33, 250), "none", True, 0, 16), ((7, 5), "none", False, 0, 2)])
def test_clusters_match_oracle(shape, sigma, asym, ovl, k):
    """Few 32 x 32 subdomains: each runs on a cluster of CTAs (fixed cycles, and a
    converging solve with the deferred fold); same iterates and stopping cycle."""
    import torch
    p = W.random_bc_problem(2, *shape, seed=13, sigma_kind=sigma, asym=asym)
    kw = dict(tile_x=32, tile_y=32, k=k, overlap_x=min(ovl, 31), overlap_y=min(ovl, 31))
    got = _cycles(p, 2, fixed_cycles=5, **kw)
    assert np.array_equal(got, oracle.run_fixed(p.st, p.f, p.u0, 5, 32, 32, k, overlap=(ovl, ovl)))
    s = gpu_solver(p, precision="f64", tol=1e-2, max_cycles=2000, check_every=8, **kw)
    u = to_dev(p.u0, 2, torch.float64)
    out = s.solve(to_dev(p.f, 2, torch.float64), u, check=False)
    assert out["tile_threads"] == 512
    s.close()
    uo, c, status, _ = oracle.solve(p.st, p.f, p.u0, 1e-2, 2000, 32, 32, k, overlap=(ovl, ovl))
    assert out["cycles"] == c and np.array_equal(to_host(u, shape[0]), uo)
