"""Performance cases: the solves a user of this package runs, through its public
entry points (``Solver.solve``, ``hj_solve_batched``, ``autograd.solve_screened``).

Families (the "family" of a case):

  plane   2D five-point hierarchical cycles, a fixed number of them or up to a
          cycle cap with the fused residual on (smoothing, throughput runs)
  solve   1D / 2D solves to a relative residual (binary64, binary32, refined)
  batch   many independent screened 2D problems in one call
  grad    a differentiable screened solve: forward and adjoint
  cube    3D seven-point cycles
  mg      multigrid V-cycles with the hierarchical smoother
  varcoef 2D cycles with per-point neighbour coefficients

Sizes and options come from the package's own tests and benchmark: 512-point
lines and 512 x 512 planes to 1e-6 / 1e-8, 8192 x 8192 binary32 at k = 4, batches
of screened problems with sides 64 to 512, screening fields between 10 and 1000,
512^3 cubes, multigrid on 2^m - 1 sides, heterogeneous diffusion with contrast 10.
"""
from __future__ import annotations

import math

import torch

import paper_2006_16465_gb300 as hj
from paper_2006_16465_gb300 import autograd as hj_autograd

DEV = "cuda"


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------

def _plane(nx, ny, precision, k, cycles, tile_x=32, tile_y=32, check=False, sigma=0.0):
    return {"family": "plane", "nx": nx, "ny": ny, "precision": precision, "k": k, "cycles": cycles,
            "tile_x": tile_x, "tile_y": tile_y, "check": check, "sigma": sigma}


def _solve(dim, nx, ny, precision, k, tol, tile_x=32, tile_y=32, overlap=0, sigma=0.0):
    return {"family": "solve", "dim": dim, "nx": nx, "ny": ny, "precision": precision, "k": k, "tol": tol,
            "tile_x": tile_x, "tile_y": tile_y, "overlap": overlap, "sigma": sigma}


def listed():
    cases = [
        # smallest call: a few smoothing cycles on a small ragged grid, as inside a
        # time step or another solver's loop; launches and host work count
        dict(_plane(96, 70, "f64", 4, 8, sigma=37.5), name="plane_f64_96x70_k4"),
        # 1D line to 1e-6 with 128-point subdomains, the package's 1D configuration
        dict(_solve(1, 512, 1, "f64", 32, 1e-6, tile_x=128, tile_y=1), name="line_f64_512"),
        # ordinary all-binary64 solve of a plane with the default subdomains and k
        dict(_solve(2, 256, 256, "f64", 16, 1e-6), name="plane_f64_256_to_1e-6"),
        # the package's headline solve: binary32 inner cycles, binary64 refinement, to 1e-8
        dict(_solve(2, 512, 512, "f32_ir", 32, 1e-8), name="plane_f32ir_512_to_1e-8"),
        # the same with overlapping subdomains, the setting its tuner picks
        dict(_solve(2, 512, 512, "f32_ir", 64, 1e-8, overlap=8), name="plane_f32ir_512_overlap"),
        # large odd rectangle in binary64 (ragged subdomains on two sides)
        dict(_plane(3001, 2003, "f64", 16, 10), name="plane_f64_3001x2003_k16"),
        # the throughput run: 8192 x 8192 binary32, k = 4, fused residual on
        dict(_plane(8192, 8192, "f32", 4, 200, check=True), name="plane_f32_8192_k4"),
        # batch of uneven screened problems to 1e-8 (one persistent launch per refinement step)
        {"name": "batch_f32ir_64", "family": "batch", "nprob": 64, "lo": 64, "hi": 512, "k": 32, "tol": 1e-8,
         "tile_x": 32, "tile_y": 32, "precision": "f32_ir", "shape_seed": 3},
        # training-style use: forward solve and adjoint for a batch of right-hand sides
        {"name": "grad_256x8", "family": "grad", "n": 256, "nrhs": 8, "k": 32, "tol": 1e-10, "tile_x": 32, "tile_y": 32},
        # 3D throughput in binary32, default 3D subdomain
        {"name": "cube_f32_512_k4", "family": "cube", "nx": 512, "ny": 512, "nz": 512, "precision": "f32", "k": 4,
         "cycles": 20, "tile_x": 16, "tile_y": 8, "tile_z": 8},
        # multigrid solve in binary64 to 1e-8
        {"name": "mg_f64_1023_to_1e-8", "family": "mg", "nx": 1023, "ny": 1023, "precision": "f64", "k": 2, "tol": 1e-8,
         "cycles": 0, "tile_x": 32, "tile_y": 8},
        # heterogeneous diffusion with per-point coefficients, default subdomain
        {"name": "varcoef_f32_4096_k4", "family": "varcoef", "nx": 4096, "ny": 4096, "precision": "f32", "k": 4,
         "cycles": 20, "tile_x": 32, "tile_y": 32},
    ]
    return cases


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["plane", "plane", "solve", "solve", "batch", "grad", "cube", "mg", "varcoef"])
    if family == "plane":
        precision = rng.choice(["f32", "f64"])
        cap = 8192 * 8192 if precision == "f32" else 2500 * 2500
        nx = _log_int(rng, 40, 8192 if precision == "f32" else 4500)
        ny = min(_log_int(rng, 40, 8192 if precision == "f32" else 4500), max(40, cap // nx))
        tx, ty = rng.choice([(32, 32), (32, 32), (32, 16), (32, 8), (64, 32), (64, 64)])
        return _plane(nx, ny, precision, rng.choice([1, 4, 8, 16]), rng.randint(4, 40), tx, ty,
                      check=rng.random() < 0.5, sigma=rng.choice([0.0, 37.5]))
    if family == "solve":
        kind = rng.choice(["line", "f64", "f32", "f32_ir", "f32_ir", "bf16corr_ir"])
        if kind == "line":
            return _solve(1, _log_int(rng, 100, 512), rng.choice([1, 1, 7, 64]), "f64", rng.choice([16, 32, 64]), 1e-6,
                          tile_x=rng.choice([64, 128, 256]), tile_y=1, overlap=rng.choice([0, 0, 4]))
        hi = {"f64": 256, "f32": 512, "f32_ir": 512, "bf16corr_ir": 300}[kind]
        tol = {"f64": 1e-6, "f32": 1e-4, "f32_ir": 1e-8, "bf16corr_ir": 1e-8}[kind]
        return _solve(2, _log_int(rng, 64, hi), _log_int(rng, 64, hi), kind, rng.choice([16, 32, 64]), tol,
                      overlap=rng.choice([0, 0, 4, 8]), sigma=rng.choice([0.0, rng.uniform(1.0, 100.0)]))
    if family == "batch":
        return {"family": "batch", "nprob": rng.randint(3, 64), "lo": 64, "hi": rng.choice([256, 384, 512]),
                "k": rng.choice([16, 32]), "tol": 1e-8, "tile_x": 32, "tile_y": 32,
                "precision": rng.choice(["f32_ir", "f32_ir", "bf16corr_ir"]),
                "shape_seed": rng.randint(1, 10 ** 6)}
    if family == "grad":
        t = rng.choice([32, 64])
        return {"family": "grad", "n": _log_int(rng, 64, 256), "nrhs": rng.randint(1, 8), "k": rng.choice([16, 32]),
                "tol": rng.choice([1e-8, 1e-10]), "tile_x": t, "tile_y": t}
    if family == "cube":
        precision = rng.choice(["f32", "f64"])
        hi = 512 if precision == "f32" else 256
        tx, ty, tz = rng.choice([(16, 8, 8), (32, 4, 8), (8, 8, 8), (16, 8, 4)] if precision == "f32" else
                                [(16, 4, 8), (8, 8, 8), (32, 2, 8), (16, 8, 4)])
        return {"family": "cube", "nx": _log_int(rng, 24, hi), "ny": _log_int(rng, 24, hi), "nz": _log_int(rng, 24, hi),
                "precision": precision, "k": rng.choice([1, 4, 8]), "cycles": rng.randint(2, 20), "tile_x": tx,
                "tile_y": ty, "tile_z": tz}
    if family == "mg":
        precision = rng.choice(["f32", "f64"])
        side = [63, 127, 255, 511, 1023, 2047, 191, 383, 767]
        nx = rng.choice(side)
        ny = rng.choice([s for s in side if (s & (s + 1) == 0) == (nx & (nx + 1) == 0)])
        ty = rng.choice([8, 32])
        if precision == "f32":   # a fixed number of V-cycles, as a preconditioner runs them
            return {"family": "mg", "nx": nx, "ny": nx if max(nx, ny) > 4 * min(nx, ny) else ny, "precision": "f32",
                    "k": 2, "tol": 0.0, "cycles": rng.randint(1, 10), "tile_x": 32, "tile_y": ty}
        return {"family": "mg", "nx": nx, "ny": nx, "precision": "f64", "k": 2, "tol": 1e-8, "cycles": 0,
                "tile_x": 32, "tile_y": ty}
    precision = rng.choice(["f32", "f64"])
    hi = 4096 if precision == "f32" else 2000
    tx, ty = rng.choice([(32, 32), (32, 8), (16, 16)])
    return {"family": "varcoef", "nx": _log_int(rng, 40, hi), "ny": _log_int(rng, 40, hi), "precision": precision,
            "k": rng.choice([1, 4, 16]), "cycles": rng.randint(4, 20), "tile_x": tx, "tile_y": ty}


# ---------------------------------------------------------------------------
# Problem data (all of it from the seed)
# ---------------------------------------------------------------------------

class _Stencil:
    """Coefficients of -Lap u + s u on the unit interval / square / cube."""

    def __init__(self, dim, nx, ny=1, nz=1, sigma=0.0):
        self.dim, self.nx, self.ny, self.nz = dim, nx, ny, nz
        ix2 = float(nx + 1) ** 2
        iy2 = float(ny + 1) ** 2 if dim >= 2 else 0.0
        iz2 = float(nz + 1) ** 2 if dim == 3 else 0.0
        self.cW = self.cE = -ix2
        self.cS = self.cN = -iy2
        self.cB = self.cT = -iz2
        self.cD = 2.0 * ix2 + 2.0 * iy2 + 2.0 * iz2
        self.sigma_const = sigma


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + 17)
    return g


def _uniform(g, shape, lo, hi, dtype=torch.float64):
    return torch.rand(shape, generator=g, device=DEV, dtype=dtype) * (hi - lo) + lo


def _dtype(case):
    return torch.float32 if case["precision"] == "f32" else torch.float64


def _rhs2d(g, st, dtype):
    """f ~ U[-1, 1] on interior points (1D: per row), zero elsewhere."""
    f = hj.alloc_grid(st.dim, st.nx, st.ny, dtype, DEV)
    r = slice(1, st.ny + 1) if st.dim == 2 else slice(0, st.ny)
    f[r, 1:st.nx + 1] = _uniform(g, (st.ny, st.nx), -1.0, 1.0).to(dtype)
    return f


def _plane_data(case, seed):
    st = _Stencil(2, case["nx"], case["ny"], sigma=case["sigma"])
    g = _gen(seed)
    dt = _dtype(case)
    f = _rhs2d(g, st, dt)
    u0 = hj.alloc_grid(2, st.nx, st.ny, dt, DEV)
    # random Dirichlet ring and a small random initial guess
    u0[:, :st.nx + 2] = _uniform(g, (st.ny + 2, st.nx + 2), -0.5, 0.5, torch.float32).to(dt)
    return st, f, u0


def _solve_data(case, seed):
    st = _Stencil(case["dim"], case["nx"], case["ny"], sigma=case["sigma"])
    g = _gen(seed)
    dt = _dtype(case)
    if case["dim"] == 1:
        # -u'' = f, f a sum of eight sine modes with normal amplitudes per row
        f = hj.alloc_grid(1, st.nx, st.ny, dt, DEV)
        a = torch.randn((st.ny, 8), generator=g, device=DEV, dtype=torch.float64)
        x = torch.arange(1, st.nx + 1, device=DEV, dtype=torch.float64) / (st.nx + 1)
        m = torch.arange(1, 9, device=DEV, dtype=torch.float64)
        f[:, 1:st.nx + 1] = (a[:, :, None] * torch.sin(math.pi * m[:, None] * x[None, :])[None]).sum(1).to(dt)
    else:
        f = _rhs2d(g, st, dt)
    return st, f


def _batch_data(case, seed):
    import random
    rs = random.Random(case["shape_seed"])   # the shapes belong to the case, the values to the seed
    g = _gen(seed)
    sides = list(range(case["lo"], case["hi"] + 1, 32))
    out = []
    for _ in range(case["nprob"]):
        st = _Stencil(2, rs.choice(sides), rs.choice(sides), sigma=rs.uniform(1.0, 100.0))
        out.append((st, _rhs2d(g, st, torch.float64)))
    return out


def _grad_data(case, seed):
    n = case["n"]
    st = _Stencil(2, n, n)
    g = _gen(seed)
    # screening field 10 exp(sum of 16 random Fourier modes), clipped to [10, 1000]
    x = torch.arange(1, n + 1, device=DEV, dtype=torch.float64) / (n + 1)
    kx = torch.randint(-5, 6, (16,), generator=g, device=DEV).double()
    ky = torch.randint(-5, 6, (16,), generator=g, device=DEV).double()
    amp = 0.5 * torch.randn((16,), generator=g, device=DEV, dtype=torch.float64)
    phi = _uniform(g, (16,), 0.0, 2.0 * math.pi)
    arg = 2.0 * math.pi * (kx[:, None, None] * x[None, None, :] + ky[:, None, None] * x[None, :, None])
    field = (amp[:, None, None] * torch.cos(arg + phi[:, None, None])).sum(0)
    sigma = hj.alloc_grid(2, n, n, torch.float64, DEV)
    sigma[1:n + 1, 1:n + 1] = (10.0 * torch.exp(field)).clamp(10.0, 1000.0)
    f = torch.stack([_rhs2d(g, st, torch.float64) for _ in range(case["nrhs"])])
    target = torch.stack([_rhs2d(g, st, torch.float64) for _ in range(case["nrhs"])])
    return st, f, sigma, target


def _cube_data(case, seed):
    st = _Stencil(3, case["nx"], case["ny"], case["nz"])
    g = _gen(seed)
    dt = _dtype(case)
    f = hj.alloc_grid(3, st.nx, st.ny, dt, DEV, nz=st.nz)
    f[1:-1, 1:-1, 1:st.nx + 1] = _uniform(g, (st.nz, st.ny, st.nx), -1.0, 1.0, torch.float32).to(dt)
    u0 = hj.alloc_grid(3, st.nx, st.ny, dt, DEV, nz=st.nz)
    u0[:, :, :st.nx + 2] = _uniform(g, (st.nz + 2, st.ny + 2, st.nx + 2), -0.5, 0.5, torch.float32).to(dt)
    return st, f, u0


def _mg_data(case, seed):
    st = _Stencil(2, case["nx"], case["ny"])
    g = _gen(seed)
    return st, _rhs2d(g, st, _dtype(case))


def _varcoef_data(case, seed):
    """Flux-form diffusion with a smooth conductivity between 1 and 10."""
    nx, ny = case["nx"], case["ny"]
    g = _gen(seed)
    dt = _dtype(case)
    ph = _uniform(g, (3,), 0.0, 2.0 * math.pi)
    x = torch.arange(nx + 2, device=DEV, dtype=torch.float64) / (nx + 1)
    y = torch.arange(ny + 2, device=DEV, dtype=torch.float64) / (ny + 1)
    w = torch.sin(2 * math.pi * x[None, :] + ph[0]) * torch.cos(2 * math.pi * y[:, None] + ph[1]) \
        + 0.5 * torch.sin(6 * math.pi * x[None, :] + ph[2])
    kappa = torch.exp(math.log(10.0) * 0.5 * (w / 1.5 + 1.0))
    ld = hj.padded_ld(nx, dt)
    coef = torch.zeros((4, ny + 2, ld), device=DEV, dtype=torch.float64)
    ix2, iy2 = float(nx + 1) ** 2, float(ny + 1) ** 2
    mid = kappa[1:-1, 1:-1]
    coef[0, 1:-1, 1:nx + 1] = -0.5 * (mid + kappa[1:-1, :-2]) * ix2
    coef[1, 1:-1, 1:nx + 1] = -0.5 * (mid + kappa[1:-1, 2:]) * ix2
    coef[2, 1:-1, 1:nx + 1] = -0.5 * (mid + kappa[:-2, 1:-1]) * iy2
    coef[3, 1:-1, 1:nx + 1] = -0.5 * (mid + kappa[2:, 1:-1]) * iy2
    # the diagonal in the screening plane; the ghost and padding entries are not used
    a = coef.abs()
    sigma = a[0] + a[1] + a[2] + a[3]
    st = _Stencil(2, nx, ny)
    st.cD = 0.0
    f = _rhs2d(g, st, dt)
    u0 = hj.alloc_grid(2, nx, ny, dt, DEV)
    u0[:, :nx + 2] = _uniform(g, (ny + 2, nx + 2), -0.5, 0.5, torch.float32).to(dt)
    return st, f, u0, coef, sigma


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    fam = case["family"]
    if fam == "plane":
        st, f, u0 = _plane_data(case, seed)
        kw = dict(tol=0.0, max_cycles=case["cycles"]) if case["check"] else dict(fixed_cycles=case["cycles"])
        s = hj.Solver(st, tile_x=case["tile_x"], tile_y=case["tile_y"], k=case["k"], precision=case["precision"], **kw)
        return {"family": fam, "solver": s, "f": f, "u0": u0, "u": torch.empty_like(u0)}
    if fam == "solve":
        st, f = _solve_data(case, seed)
        s = hj.Solver(st, tile_x=case["tile_x"], tile_y=case["tile_y"], k=case["k"], precision=case["precision"],
                      tol=case["tol"], overlap_x=case["overlap"], overlap_y=case["overlap"] if case["dim"] == 2 else 0)
        return {"family": fam, "solver": s, "f": f, "u0": torch.zeros_like(f), "u": torch.empty_like(f)}
    if fam == "batch":
        probs = _batch_data(case, seed)
        params = hj.make_params(precision=case["precision"], tile_x=case["tile_x"], tile_y=case["tile_y"], k=case["k"],
                                tol=case["tol"], inner_tol=1e-4)
        solver = hj.Solver(probs[0][0], params)
        descs = [hj.make_desc(2, st.nx, st.ny, f.shape[-1], st.cW, st.cE, st.cS, st.cN, st.cD, st.sigma_const)
                 for st, f in probs]
        return {"family": fam, "solver": solver, "descs": descs, "f": [f for _, f in probs],
                "u": [torch.empty_like(f) for _, f in probs]}
    if fam == "grad":
        st, f, sigma, target = _grad_data(case, seed)
        return {"family": fam, "st": st, "f": f.requires_grad_(True), "sigma": sigma.requires_grad_(True),
                "target": target,
                "params": dict(precision="f32_ir", tile_x=case["tile_x"], tile_y=case["tile_y"], k=case["k"],
                               tol=case["tol"])}
    if fam == "cube":
        st, f, u0 = _cube_data(case, seed)
        s = hj.Solver(st, tile_x=case["tile_x"], tile_y=case["tile_y"], tile_z=case["tile_z"], k=case["k"],
                      precision=case["precision"], fixed_cycles=case["cycles"])
        return {"family": fam, "solver": s, "f": f, "u0": u0, "u": torch.empty_like(u0)}
    if fam == "mg":
        st, f = _mg_data(case, seed)
        kw = dict(fixed_cycles=case["cycles"]) if case["cycles"] else dict(tol=case["tol"])
        s = hj.Solver(st, method="mg", tile_x=case["tile_x"], tile_y=case["tile_y"], k=case["k"],
                      precision=case["precision"], **kw)
        return {"family": fam, "solver": s, "f": f, "u0": torch.zeros_like(f), "u": torch.empty_like(f)}
    st, f, u0, coef, sigma = _varcoef_data(case, seed)
    s = hj.Solver(st, sigma=sigma, coef=coef, tile_x=case["tile_x"], tile_y=case["tile_y"], k=case["k"],
                  precision=case["precision"], fixed_cycles=case["cycles"])
    return {"family": fam, "solver": s, "f": f, "u0": u0, "u": torch.empty_like(u0)}


def run(state):
    if state["family"] == "batch":
        for u in state["u"]:
            u.zero_()
        code = hj.hj_solve_batched(state["solver"].h, state["descs"], [f.data_ptr() for f in state["f"]],
                                   [u.data_ptr() for u in state["u"]], torch.cuda.current_stream().cuda_stream)
        if code != hj.HJ_OK:
            raise hj.HJError(code, "hj_solve_batched")
        return state["u"]
    if state["family"] == "grad":
        f, sigma = state["f"], state["sigma"]
        f.grad = sigma.grad = None
        u = hj_autograd.solve_screened(f, sigma, state["st"], **state["params"])
        loss = 0.5 * ((u - state["target"]) ** 2).sum()
        loss.backward()
        return {"u": u.detach(), "df": f.grad, "dsigma": sigma.grad}
    u = state["u"]
    u.copy_(state["u0"])
    state["solver"].solve(state["f"], u)
    return u


# ---------------------------------------------------------------------------
# Work one pass cannot do without
# ---------------------------------------------------------------------------

def _sweeps_needed(st, tol, sigma=0.0):
    """Jacobi sweeps that take the slowest mode's share of a random residual
    (about 1 / sqrt(points) of it) to the tolerance: hierarchical cycles need
    at least as many inner sweeps."""
    d = -2.0 * (st.cW + (st.cS if st.dim == 2 else 0.0))
    rho = 2.0 * abs(st.cW) * math.cos(math.pi / (st.nx + 1))
    if st.dim == 2:
        rho += 2.0 * abs(st.cS) * math.cos(math.pi / (st.ny + 1))
    rho /= d + sigma
    share = math.sqrt(st.nx * st.ny) if st.dim == 2 else 1.0
    return max(1.0, math.log(1.0 / (tol * share)) / -math.log(rho))


def work(case):
    fam = case["family"]
    esz = 4 if case.get("precision") == "f32" else 8
    if fam == "plane":
        pts = case["nx"] * case["ny"]
        return {"bytes": 3 * esz * pts, "flops": 8.0 * pts * case["k"] * case["cycles"]}
    if fam == "solve":
        st = _Stencil(case["dim"], case["nx"], case["ny"])
        pts = case["nx"] * case["ny"]
        return {"bytes": 3 * esz * pts,
                "flops": (8.0 if case["dim"] == 2 else 5.0) * pts * _sweeps_needed(st, case["tol"], case["sigma"])}
    if fam == "batch":
        import random
        rs = random.Random(case["shape_seed"])
        sides = list(range(case["lo"], case["hi"] + 1, 32))
        pts, flops = 0, 0.0
        for _ in range(case["nprob"]):
            st = _Stencil(2, rs.choice(sides), rs.choice(sides), sigma=rs.uniform(1.0, 100.0))
            pts += st.nx * st.ny
            flops += 8.0 * st.nx * st.ny * _sweeps_needed(st, case["tol"], st.sigma_const)
        return {"bytes": 24 * pts, "flops": flops}
    if fam == "grad":
        st = _Stencil(2, case["n"], case["n"])
        pts = case["n"] ** 2
        sweeps = _sweeps_needed(st, case["tol"], 30.0)
        # read f, sigma, target; write u, dL/df, dL/dsigma
        return {"bytes": 8 * pts * (4 * case["nrhs"] + 2), "flops": 2 * 8.0 * pts * case["nrhs"] * sweeps}
    if fam == "cube":
        pts = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 3 * esz * pts, "flops": 12.0 * pts * case["k"] * case["cycles"]}
    if fam == "mg":
        pts = case["nx"] * case["ny"]
        cycles = case["cycles"] or 8   # a V-cycle contracts the residual about tenfold
        return {"bytes": 3 * esz * pts, "flops": (4.0 / 3.0) * pts * cycles * (2 * case["k"] * 10.0 + 24.0)}
    pts = case["nx"] * case["ny"]
    return {"bytes": pts * (3 * esz + 5 * 8), "flops": 8.0 * pts * case["k"] * case["cycles"]}


# ---------------------------------------------------------------------------
# The same in 64 bits, without the package
# ---------------------------------------------------------------------------

def _tiled_cycles(u, f, inv, cw, ce, cs, cn, tile_x, tile_y, k, cycles):
    """Hierarchical cycles on a (ny + 2, nx + 2) grid in float64: every
    tile_x x tile_y subdomain runs k Jacobi sweeps with its halo frozen.  inv
    (1 / diagonal) and the neighbour coefficients are scalars or (ny, nx)."""
    ny, nx = u.shape[0] - 2, u.shape[1] - 2
    nby, nbx = -(-ny // tile_y), -(-nx // tile_x)
    py, px = nby * tile_y, nbx * tile_x

    def tiles(a):   # (ny, nx) -> (nby, tile_y, nbx, tile_x) -> blocks first
        if not torch.is_tensor(a):
            return a
        b = torch.zeros((py, px), device=u.device, dtype=torch.float64)
        b[:ny, :nx] = a
        return b.view(nby, tile_y, nbx, tile_x).transpose(1, 2).contiguous()

    act = tiles(torch.ones((ny, nx), device=u.device, dtype=torch.float64)).bool()
    ragged = py != ny or px != nx
    F, I, W, E, S, N = tiles(f), tiles(inv), tiles(cw), tiles(ce), tiles(cs), tiles(cn)
    full = torch.zeros((py + 2, px + 2), device=u.device, dtype=torch.float64)
    full[:ny + 2, :nx + 2] = u
    for _ in range(cycles):
        t = full.unfold(0, tile_y + 2, tile_y).unfold(1, tile_x + 2, tile_x).contiguous()
        for _ in range(k):
            nv = (F - W * t[..., 1:-1, :-2] - E * t[..., 1:-1, 2:] - S * t[..., :-2, 1:-1] - N * t[..., 2:, 1:-1]) * I
            if ragged:
                nv = torch.where(act, nv, t[..., 1:-1, 1:-1])
            t[..., 1:-1, 1:-1] = nv
        inner = t[..., 1:-1, 1:-1].transpose(1, 2).reshape(py, px)
        full[1:ny + 1, 1:nx + 1] = inner[:ny, :nx]
    return full[:ny + 2, :nx + 2]


def _tiled_cycles3(u, f, st, tx, ty, tz, k, cycles):
    nz, ny, nx = (s - 2 for s in u.shape)
    bz, by, bx = -(-nz // tz), -(-ny // ty), -(-nx // tx)
    pz, py, px = bz * tz, by * ty, bx * tx

    def tiles(a):
        b = torch.zeros((pz, py, px), device=u.device, dtype=torch.float64)
        b[:nz, :ny, :nx] = a
        return b.view(bz, tz, by, ty, bx, tx).permute(0, 2, 4, 1, 3, 5).contiguous()

    act = tiles(torch.ones((nz, ny, nx), device=u.device, dtype=torch.float64)).bool()
    ragged = (pz, py, px) != (nz, ny, nx)
    F = tiles(f)
    inv = 1.0 / st.cD
    full = torch.zeros((pz + 2, py + 2, px + 2), device=u.device, dtype=torch.float64)
    full[:nz + 2, :ny + 2, :nx + 2] = u
    c = slice(1, -1)
    for _ in range(cycles):
        t = full.unfold(0, tz + 2, tz).unfold(1, ty + 2, ty).unfold(2, tx + 2, tx).contiguous()
        for _ in range(k):
            acc = (t[..., c, c, :-2] + t[..., c, c, 2:]).mul_(st.cW)
            acc.add_(t[..., c, :-2, c] + t[..., c, 2:, c], alpha=st.cS)
            acc.add_(t[..., :-2, c, c] + t[..., 2:, c, c], alpha=st.cB)
            nv = (F - acc).mul_(inv)
            if ragged:
                nv = torch.where(act, nv, t[..., c, c, c])
            t[..., c, c, c] = nv
        inner = t[..., c, c, c].permute(0, 3, 1, 4, 2, 5).reshape(pz, py, px)
        full[1:nz + 1, 1:ny + 1, 1:nx + 1] = inner[:nz, :ny, :nx]
    return full[:nz + 2, :ny + 2, :nx + 2]


def _dst1(a):
    """Sine transform along the last axis: sum_j a_j sin(pi (j+1)(m+1)/(n+1))."""
    n = a.shape[-1]
    z = torch.zeros(a.shape[:-1] + (2 * n + 2,), device=a.device, dtype=torch.float64)
    z[..., 1:n + 1] = a
    z[..., n + 2:] = -a.flip(-1)
    return -0.5 * torch.fft.fft(z)[..., 1:n + 1].imag


def _direct(st, f_int, sigma):
    """Exact solution of the constant-coefficient Dirichlet problem with a zero
    ring: f_int (ny, nx) (1D: independent rows)."""
    nx = st.nx
    lx = 2.0 * abs(st.cW) * (1.0 - torch.cos(math.pi * torch.arange(1, nx + 1, device=DEV, dtype=torch.float64) / (nx + 1)))
    if st.dim == 1:
        return _dst1(_dst1(f_int) / (lx + sigma)) * (2.0 / (nx + 1))
    ny = st.ny
    ly = 2.0 * abs(st.cS) * (1.0 - torch.cos(math.pi * torch.arange(1, ny + 1, device=DEV, dtype=torch.float64) / (ny + 1)))
    h = _dst1(_dst1(f_int).transpose(0, 1).contiguous())
    h = h / (lx[:, None] + ly[None, :] + sigma)
    h = _dst1(h).transpose(0, 1).contiguous()
    return _dst1(h) * (4.0 / ((nx + 1) * (ny + 1)))


def _apply(st, u, sig):
    """A u on interiors (B, n, n) with a zero ring."""
    p = torch.nn.functional.pad(u, (1, 1, 1, 1))
    return (st.cD + sig) * u + st.cW * (p[:, 1:-1, :-2] + p[:, 1:-1, 2:]) + st.cS * (p[:, :-2, 1:-1] + p[:, 2:, 1:-1])


def _cg(st, sig, b):
    x = torch.zeros_like(b)
    r = b.clone()
    p = r.clone()
    rr = (r * r).sum((1, 2), keepdim=True)
    stop = 1e-30 * rr.max()
    for it in range(6000):
        ap = _apply(st, p, sig)
        alpha = rr / (p * ap).sum((1, 2), keepdim=True)
        x = x + alpha * p
        r = r - alpha * ap
        new = (r * r).sum((1, 2), keepdim=True)
        if it % 50 == 49 and bool((new.max() <= stop).item()):
            break
        p = r + (new / rr) * p
        rr = new
    return x


def _place(st, shape, dtype, inner):
    out = torch.zeros(shape, device=DEV, dtype=torch.float64)
    r = slice(1, st.ny + 1) if st.dim == 2 else slice(0, st.ny)
    out[..., r, 1:st.nx + 1] = inner
    return out


def exact(case, seed):
    fam = case["family"]
    if fam == "plane":
        st, f, u0 = _plane_data(case, seed)
        out = u0.double()
        d = st.cD + st.sigma_const
        out[:, :st.nx + 2] = _tiled_cycles(out[:, :st.nx + 2].contiguous(), f[1:-1, 1:st.nx + 1].double(), 1.0 / d, st.cW,
                                           st.cE, st.cS, st.cN, case["tile_x"], case["tile_y"], case["k"], case["cycles"])
        return out
    if fam == "solve":
        st, f = _solve_data(case, seed)
        r = slice(1, st.ny + 1) if st.dim == 2 else slice(0, st.ny)
        return _place(st, f.shape, f.dtype, _direct(st, f[r, 1:st.nx + 1].double(), case["sigma"]))
    if fam == "batch":
        return [_place(st, f.shape, f.dtype, _direct(st, f[1:-1, 1:st.nx + 1], st.sigma_const))
                for st, f in _batch_data(case, seed)]
    if fam == "grad":
        st, f, sigma, target = _grad_data(case, seed)
        n = case["n"]
        sig = sigma[1:n + 1, 1:n + 1]
        u = _cg(st, sig, f[:, 1:n + 1, 1:n + 1])
        lam = _cg(st, sig, u - target[:, 1:n + 1, 1:n + 1])
        return {"u": _place(st, f.shape, f.dtype, u), "df": _place(st, f.shape, f.dtype, lam),
                "dsigma": _place(st, sigma.shape, f.dtype, -(lam * u).sum(0))}
    if fam == "cube":
        st, f, u0 = _cube_data(case, seed)
        out = u0.double()
        out[:, :, :st.nx + 2] = _tiled_cycles3(out[:, :, :st.nx + 2].contiguous(), f[1:-1, 1:-1, 1:st.nx + 1].double(), st,
                                               case["tile_x"], case["tile_y"], case["tile_z"], case["k"], case["cycles"])
        return out
    if fam == "mg":
        if case["cycles"]:
            return None   # a few V-cycles: not the solution, and no short 64-bit restatement
        st, f = _mg_data(case, seed)
        return _place(st, f.shape, f.dtype, _direct(st, f[1:-1, 1:st.nx + 1].double(), 0.0))
    st, f, u0, coef, sigma = _varcoef_data(case, seed)
    out = u0.double()
    nx = st.nx
    c = [coef[m, 1:-1, 1:nx + 1] for m in range(4)]
    out[:, :nx + 2] = _tiled_cycles(out[:, :nx + 2].contiguous(), f[1:-1, 1:nx + 1].double(), 1.0 / sigma[1:-1, 1:nx + 1],
                                    c[0], c[1], c[2], c[3], case["tile_x"], case["tile_y"], case["k"], case["cycles"])
    return out
