"""Launches that leave SMs idle run FP64 stages by pairs of outputs and split the
step's column passes by velocity component: one instance alone must equal the
same instance in a batch that fills the GPU, bit for bit, at lengths with every
butterfly.  And the pressure solve without its FP64 copies: solved in place, and
refined with the constant mode removed by weighted sums."""
import numpy as np
import pytest

from gpu_common import binding, grid_lengths, to_dev, torch_cuda


def _fields(nx, ny, batch, seed):
    rng = np.random.default_rng(seed)
    x = np.arange(nx)[:, None] / nx
    y = np.linspace(0.0, 1.0, ny)[None, :]
    f = np.cos(2 * np.pi * x + 1.0) * (0.3 + y - 2 * y ** 3) + 0.1 * np.sin(6 * y)
    return np.stack([f * (1 + 0.1 * b) + 1e-3 * rng.standard_normal((nx, ny)) for b in range(batch)])


# extended lengths: 64, 65 = 5 13, 66 = 2 3 11, 68 = 4 17, 70 = 2 5 7, 89 (Rader 8 11), 94 = 2 47 (chirp-z), 96
@pytest.mark.gpu
@pytest.mark.parametrize("ny", [39, 40, 41, 43, 45, 64, 69, 71])
@pytest.mark.parametrize("xw", [False, True])
def test_alone_equals_in_a_full_batch(ny, xw):
    torch = torch_cuda()
    b = binding()
    nx, full = 28, 24
    lx, ly = grid_lengths(nx, ny, xw)
    f = _fields(nx, ny, full, ny)
    got = []
    for batch in (1, full):
        ctx = b.Context(nx, ny, lx, ly, x_walls=xw, batch=batch, family="G8")
        fd = to_dev(f[:batch])
        outs = [torch.zeros_like(fd) for _ in range(3)]
        ctx.spectral_op(fd, ["DX", "DY", "LAP"], outs)
        lines = [torch.zeros_like(fd) for _ in range(2)]
        ctx.line_op(fd, ["DY", "LAP"], lines)
        phi = torch.zeros_like(fd)
        ctx.ppe_solve(fd, phi)
        u, v = (0.01 * fd).clone(), (0.02 * fd).clone()
        p, fu, fv = torch.zeros_like(fd), torch.zeros_like(fd), torch.zeros_like(fd)
        ctx.isph_step(u, v, p, fu, fv, 2, nu=1e-2, dt=1e-4, u_top=0.1, scheme="rk3")
        ctx.sync()
        got.append([x[0].cpu().numpy() for x in outs + lines + [phi, u, v, p, fu, fv]])
    for a, r in zip(*got):
        np.testing.assert_array_equal(a, r)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32x2", "f32"])
@pytest.mark.parametrize("xw", [False, True])
def test_pressure_solve_in_place(prec, xw):
    torch = torch_cuda()
    b = binding()
    nx, ny = 30, 37
    lx, ly = grid_lengths(nx, ny, xw)
    ctx = b.Context(nx, ny, lx, ly, x_walls=xw, batch=2, prec=prec)
    f = to_dev(_fields(nx, ny, 2, 3), "f32" if prec == "f32" else "f64")
    phi = torch.zeros_like(f)
    ctx.ppe_solve(f, phi)
    g = f.clone()
    ctx.ppe_solve(g, g)
    h = torch.zeros_like(f)
    ctx.ppe_solve(f, h, want_resid=True)
    ctx.sync()
    np.testing.assert_array_equal(phi.cpu().numpy(), g.cpu().numpy())
    np.testing.assert_array_equal(phi.cpu().numpy(), h.cpu().numpy())


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,xw", [(8, 12, False), (70, 65, True), (129, 40, False), (33, 257, True)])
def test_refined_solve_ignores_the_constant_mode(nx, ny, xw):
    """A constant added to the right-hand side (1e3 times its size) is removed in FP64 before the FP32 sweeps: the
    refined solution stays at the plain FP64 one, to FP32 rounding of the result."""
    torch = torch_cuda()
    b = binding()
    lx, ly = grid_lengths(nx, ny, xw)
    f = _fields(nx, ny, 3, 5)
    ref = b.Context(nx, ny, lx, ly, x_walls=xw, batch=3)
    fd = to_dev(f.astype(np.float32).astype(np.float64))
    exact = torch.zeros_like(fd)
    ref.ppe_solve(fd, exact)
    ctx = b.Context(nx, ny, lx, ly, x_walls=xw, batch=3, prec="f32", refine=2)
    phi = torch.zeros_like(fd, dtype=torch.float32)
    ctx.ppe_solve(fd.float(), phi)
    ctx.sync()
    e, p = exact.cpu().numpy(), phi.cpu().numpy().astype(np.float64)
    # one FP32 rounding of the result (6e-8) and two sweeps of FP32 corrections
    assert np.linalg.norm(p - e) / np.linalg.norm(e) < 2e-7
