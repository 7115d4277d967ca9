"""Large prime radices (19, 23, 29, 31) in both of their forms: by the roots'
symmetry in the operators, projection and pressure solve (FP32 pairs; the FP64
operators are in test_gpu_large_radix), and summed in order in the time step (FP64
and pairs), as a radix of the length itself and of the convolutions of 47 and 59."""
import numpy as np
import pytest

from gpu_common import binding, grid_lengths, oracle_problem, parity_tol, rel_l2, to_dev, torch_cuda, ulp_floor
from oracle import fc as ofc
from oracle import ops as oops
from oracle import ppe as oppe
from oracle import step as ostep
from paper_2606_06247_gb300 import inputs

NY = [13, 21, 22, 32, 33, 34, 37, 68, 127]  # extended lengths 38, 46, 47, 57, 58, 59, 62, 93, 152


def _pair_error(f, E, xw):
    """Norm of the rounding of one extended field and its transform in FP32 pairs (unit roundoff 2^-48): the
    continuation sums carry 2^-47 of the sum of their terms' magnitudes, the transforms 8 units a factor of two."""
    F = ofc.extend2d(f, E, E if xw else None)
    A = ofc.extend2d(np.abs(f), np.abs(E), np.abs(E) if xw else None)
    return 2.0 ** -47 * np.linalg.norm(A) + 2.0 ** -48 * 8 * np.log2(F.size) * np.linalg.norm(F)


@pytest.mark.gpu
@pytest.mark.parametrize("ny", NY)
@pytest.mark.parametrize("xw", [False, True])
def test_operators_and_projection_in_pairs(ny, xw):
    torch = torch_cuda()
    b = binding()
    nx, batch = (ny if xw else 19), 3
    lx, ly = grid_lengths(nx, ny, xw)
    ctx = b.Context(nx, ny, lx, ly, x_walls=xw, batch=batch, family="G8", h_over_dx=1.3, prec="f32x2")
    p = oracle_problem(nx, ny, xw, "G8", 1.3)
    f = np.stack([inputs.smooth_field(nx, ny, seed=5 + k) for k in range(batch)])
    g = np.stack([inputs.smooth_field(nx, ny, seed=50 + k) for k in range(batch)])
    names = ["DX", "DY", "LAP"]
    outs = [torch.zeros((batch, nx, ny), dtype=torch.float64, device="cuda") for _ in range(5)]
    ctx.spectral_op(to_dev(f), names, outs[:3])
    ctx.spectral_project(to_dev(f), to_dev(g), outs[3], outs[4])
    ctx.sync()
    Ex = p.E_dir if xw else None
    for k in range(batch):
        ef, eg = _pair_error(f[k], p.E_dir, xw), _pair_error(g[k], p.E_dir, xw)
        for n, o, r in zip(names, outs, oops.apply_symbols(f[k], [p.sym[n] for n in names], p.E_dir, Ex)):
            err = np.linalg.norm(o[k].cpu().numpy() - r)
            assert err < np.abs(p.sym[n]).max() * ef, (n, k, err)
        # each component of the projection takes at most the whole of its own field and half of the other
        refs = oppe.extended_projection(f[k], g[k], p.sym["DX"], p.sym["DY"], p.E_dir, Ex)
        for o, r, bar in zip(outs[3:], refs, (ef + eg / 2, eg + ef / 2)):
            assert np.linalg.norm(o[k].cpu().numpy() - r) < bar


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(19, 20), (23, 24), (38, 30), (31, 32), (47, 24), (59, 20)])
@pytest.mark.parametrize("xw", [False, True])
@pytest.mark.parametrize("prec", ["f64", "f32x2"])
def test_pressure_solves(nx, ny, xw, prec):
    torch = torch_cuda()
    b = binding()
    lx, ly = grid_lengths(nx, ny, xw)
    ctx = b.Context(nx, ny, lx, ly, x_walls=xw, batch=2, prec=prec)
    rhs = np.random.default_rng(nx).standard_normal((2, nx, ny))
    phi = torch.zeros((2, nx, ny), dtype=torch.float64, device="cuda")
    ctx.ppe_solve(to_dev(rhs), phi)
    ctx.sync()
    for k in range(2):  # the bar of the other pressure solves of these sizes, 32 units for pairs
        assert rel_l2(phi[k].cpu().numpy(), oppe.ppe_solve(rhs[k], lx, ly, xw)) < 1e-12 * (1 if prec == "f64" else 32)


@pytest.mark.gpu
@pytest.mark.parametrize("ny", NY[:7])
@pytest.mark.parametrize("xw", [False, True])
@pytest.mark.parametrize("prec", ["f64", "f32x2"])
def test_one_step(ny, xw, prec):
    torch = torch_cuda()
    b = binding()
    nx = ny if xw else 19
    lx, ly = grid_lengths(nx, ny, xw)
    kw = dict(nu=1e-2, rho=1.0, dt=1e-3, u_top=1.0 if xw else 0.0, force=(0.0, 0.0) if xw else (0.8, 0.0), scheme="fop")
    init = inputs.cavity_initial if xw else inputs.channel_initial
    u0, v0 = init(nx, ny, seed=ny, sigma=1e-2)
    ctx = b.Context(nx, ny, lx, ly, x_walls=xw, batch=2, family="G8", h_over_dx=1.3, prec=prec)
    u, v = (to_dev(np.stack([a, a])) for a in (u0, v0))
    ph, fu, fv = (torch.zeros_like(u) for _ in range(3))
    ctx.isph_step(u, v, ph, fu, fv, 1, **kw)
    ctx.sync()
    p = oracle_problem(nx, ny, xw, "G8", 1.3, **kw)
    fn = lambda a, c: ostep.isph_steps(p, a, c, 1)
    for got, ref, fl in zip((u, v, ph), fn(u0, v0), ulp_floor(fn, u0, v0, scale=1.0)):
        for k in range(2):
            err = rel_l2(got[k].cpu().numpy(), ref)
            assert err < parity_tol(fl) * (1 if prec == "f64" else 32), (k, err, fl)
