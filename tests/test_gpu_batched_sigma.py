"""Batched solves judge diagonal dominance by the sigma values of this call: an
array changed in place, or seen with another size, is read again."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("side_stream", [False, True])
def test_sigma_is_read_in_every_call(side_stream):
    import torch
    import paper_2006_16465_gb300 as hj
    nx, ny = 60, 41
    p = W.poisson2d_uniform(nx, ny, seed=2)
    s = hj.Solver(p.st, tile_x=32, tile_y=32, k=8, precision="f32_ir", tol=1e-6)
    f = hj.grid_from(p.f, 2, torch.float64)
    u = hj.grid_from(p.u0, 2, torch.float64)
    sg = torch.full_like(f, 2.0)

    def call(rows=ny):
        u.zero_()
        d = hj.make_desc(2, nx, rows, f.shape[1], p.st.cW, p.st.cE, p.st.cS, p.st.cN, p.st.cD, 0.0, sg)
        return hj.hj_solve_batched(s.h, [d, d], [f.data_ptr()] * 2, [u.data_ptr(), u2.data_ptr()],
                                   torch.cuda.current_stream().cuda_stream)

    u2 = torch.zeros_like(u)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if side_stream else torch.cuda.current_stream()):
        assert call() == hj.HJ_OK
        sg[ny, nx] = -1.0                       # the last interior point: no longer dominant
        assert call() == hj.HJ_ERR_NOT_DIAG_DOMINANT
        assert call(ny - 1) == hj.HJ_OK         # the same array, a grid that ends before it
        assert call() == hj.HJ_ERR_NOT_DIAG_DOMINANT
        sg[ny, nx] = 0.0
        assert call() == hj.HJ_OK
    torch.cuda.synchronize()
    s.close()
