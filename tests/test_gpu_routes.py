"""Routes that the library picks by itself: a configuration that a call reports can
be set again, and a pick kept in a file is not read under another meaning."""
import os
import subprocess
import sys

import pytest

import workloads as W
from helpers import gpu_solver, to_dev

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nx,ny,overlap", [(96, 80, 0), (256, 256, 0), (100, 100, 4)])
def test_reported_cluster_threads_can_be_set(nx, ny, overlap):
    """Binary64 on clusters of four and two CTAs: 512 threads a subdomain are
    reported, and asking for them gives the same run."""
    import torch
    p = W.random_bc_problem(2, nx, ny, seed=5, sigma_kind="const")
    kw = dict(precision="f64", tile_x=32, tile_y=32, k=5, overlap_x=overlap, overlap_y=overlap, fixed_cycles=6)
    us = []
    for threads in (0, 512):
        s = gpu_solver(p, tile_threads=threads, **kw)
        u = to_dev(p.u0, 2, torch.float64)
        assert s.solve(to_dev(p.f, 2, torch.float64), u)["tile_threads"] == 512
        s.close()
        us.append(u)
    assert torch.equal(us[0], us[1])


@pytest.mark.parametrize("kw", [dict(nx=600, ny=600), dict(in_place=1), dict(pipeline=1), dict(persistent=1),
                                dict(tile_y=16), dict(precision="f32")])
def test_cluster_threads_are_refused_elsewhere(kw):
    import paper_2006_16465_gb300 as hj
    kw = dict(kw)
    p = W.poisson2d_uniform(kw.pop("nx", 96), kw.pop("ny", 80), seed=1)
    params = dict(precision="f64", tile_x=32, tile_y=32, tile_threads=512)
    params.update(kw)
    with pytest.raises(hj.HJError) as e:
        gpu_solver(p, **params)
    assert e.value.code == hj.HJ_ERR_UNSUPPORTED


_TUNE = r"""
import os, sys
sys.path.insert(0, os.getcwd())
import torch
import paper_2006_16465_gb300 as hj
import workloads as W
p = W.poisson2d_uniform(1400, 1300, seed=1)
s = hj.Solver(p.st, tile_x=32, tile_y=32, k=4, precision="f32", tol=0.0, max_cycles=4, autotune=3)
f = hj.grid_from(p.f, 2, torch.float32)
print("PICK", s.solve(f, hj.grid_from(p.u0, 2, torch.float32), check=False)["ctas_per_sm"])
s.close()
"""


def test_cached_pick_of_an_older_version_is_measured_again(tmp_path):
    """Lines of the earlier key version kept ctas_per_sm = 0 with another meaning."""
    cache = tmp_path / "cache.txt"

    def run():
        r = subprocess.run([sys.executable, "-c", _TUNE], cwd=ROOT, capture_output=True, text=True, timeout=300,
                           env=dict(os.environ, HJ_AUTOTUNE_CACHE=str(cache)))
        assert r.returncode == 0, r.stderr[-2000:]
        return int([ln for ln in r.stdout.splitlines() if ln.startswith("PICK")][0].split()[1])

    assert run() > 0
    line = cache.read_text().splitlines()[0].split()
    key, picks = line[0], line[1:]
    assert run() == int(picks[2]) and len(cache.read_text().splitlines()) == 1   # the kept pick is used
    picks[2] = "0"
    cache.write_text(" ".join(["v2_" + key.split("_", 1)[1]] + picks) + "\n")
    assert run() > 0


def test_autotune_measures_the_cluster_variant():
    """The pick for a binary64 plane of few 32 x 32 subdomains is no slower than the
    default (on clusters): with the shape given, it is the cluster variant; a pick for
    an in-place run stays one that in-place runs take."""
    import torch
    p = W.poisson2d_uniform(128, 128, seed=1)
    f = to_dev(p.f, 2, torch.float64)
    for in_place, threads in ((0, (512,)), (1, (64, 128, 256))):
        s = gpu_solver(p, precision="f64", tile_x=32, tile_y=32, tol=1e-3, autotune=2, in_place=in_place)
        out = s.solve(f, to_dev(p.u0, 2, torch.float64))
        s.close()
        assert out["status"] == 0 and out["tile_threads"] in threads
