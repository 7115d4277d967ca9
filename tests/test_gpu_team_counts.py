"""The FP32 register column passes take one column pair per CTA where few columns
would leave SMs idle and packed pairs otherwise: a few instances alone must equal
the same instances in a batch that packs them, bit for bit, with ragged groups."""
import numpy as np
import pytest

from gpu_common import binding, grid_lengths, to_dev, torch_cuda


@pytest.mark.gpu
@pytest.mark.parametrize("ny,cont", [(512, 28), (1024, 26), (512, 25), (1024, 25)])
@pytest.mark.parametrize("nx,full", [(9, 150), (13, 152), (20, 152), (20, 76)])
def test_alone_equals_packed(nx, full, ny, cont):
    torch = torch_cuda()
    b = binding()
    lx, ly = grid_lengths(nx, ny, False)
    rng = np.random.default_rng(nx)
    y = np.linspace(0.0, 1.0, ny)
    f = np.cos(2 * np.pi * (3 * y[None, None, :] + rng.uniform(size=(full, nx, 1)))) + y ** 3
    got = []
    for part in (f[:2], f):
        ctx = b.Context(nx, ny, lx, ly, batch=len(part), n_cont=cont, prec="f32")
        fd = to_dev(part, "f32")
        outs = []
        for tma in (True, False):
            ctx.set_tma(tma)
            o = [torch.full_like(fd, float("nan")) for _ in range(2)]
            ctx.spectral_op(fd, ["DX", "LAP"], o)
            outs += o
        if nx % 2 == 0:  # lines are paired across instances
            o = [torch.full_like(fd, float("nan")) for _ in range(2)]
            ctx.line_op(fd, ["W", "DY"], o)
            outs += o
        ctx.sync()
        assert all(bool(torch.isfinite(o).all()) for o in outs)
        got.append([o[:2].cpu().numpy() for o in outs])
    for a, r in zip(*got):
        np.testing.assert_array_equal(a, r)
