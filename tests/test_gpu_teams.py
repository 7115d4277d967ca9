"""Packed teams of the FP32 register column passes: column counts around whole
groups of pairs (1 .. 9 pairs a CTA), with and without bulk-copy staging, against
the FP64 operators."""
import numpy as np
import pytest

from gpu_common import binding, grid_lengths, rel_l2, to_dev, torch_cuda


@pytest.mark.gpu
@pytest.mark.parametrize("ny,cont", [(512, 28), (1024, 26), (512, 25), (1024, 25)])
@pytest.mark.parametrize("nx", [4, 6, 7, 14, 15, 22])
def test_column_counts(nx, ny, cont):
    torch = torch_cuda()
    b = binding()
    lx, ly = grid_lengths(nx, ny, False)
    rng = np.random.default_rng(nx)
    y = np.linspace(0.0, 1.0, ny)
    f = np.cos(2 * np.pi * (3 * y[None, None, :] + rng.uniform(size=(2, nx, 1)))) + y ** 3
    ops = ["W", "DY"]
    ref = b.Context(nx, ny, lx, ly, batch=2, n_cont=cont)
    fd = to_dev(f.astype(np.float32).astype(np.float64))
    exact, lines = ([torch.zeros_like(fd) for _ in ops] for _ in range(2))
    ref.spectral_op(fd, ops, exact)
    ref.line_op(fd, ops, lines)
    ctx = b.Context(nx, ny, lx, ly, batch=2, n_cont=cont, prec="f32")
    ff = fd.float()
    got = []
    for tma in (True, False):
        ctx.set_tma(tma)
        outs = [torch.full_like(ff, float("nan")) for _ in ops]
        ctx.spectral_op(ff, ops, outs)
        got.append(outs)
    lout = [torch.full_like(ff, float("nan")) for _ in ops]
    ctx.line_op(ff, ops, lout)
    ctx.sync()
    for a, c in zip(*got):
        np.testing.assert_array_equal(a.cpu().numpy(), c.cpu().numpy())
    # FP32 transforms: unit roundoff 6e-8 times log2 of the convolution length, and (DY) the largest wavenumber
    # pi ny over the field's own 6 pi
    for o, a, e, l, le in zip(ops, got[0], exact, lout, lines):
        tol = 6e-8 * 12 * (1 if o == "W" else ny / 6) * 2
        assert rel_l2(a.cpu().numpy(), e.cpu().numpy()) < tol
        assert rel_l2(l.cpu().numpy(), le.cpu().numpy()) < tol
