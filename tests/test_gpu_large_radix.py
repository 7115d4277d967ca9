"""FP64 operators at extended lengths with a large prime radix (19, 23, 29, 31), as a
radix of the length itself and of the convolutions of 47 and 59 (46 = 2 23, 58 =
2 29), against the oracle: one line pair up to several and a ragged last one."""
import numpy as np
import pytest

from gpu_common import binding, grid_lengths, oracle_problem, parity_tol, rel_l2, to_dev, torch_cuda, ulp_floor
from oracle import ops as oops
from paper_2606_06247_gb300 import inputs


# extended lengths: 38, 46, 47, 57, 58, 59, 62, 93, 152
@pytest.mark.gpu
@pytest.mark.parametrize("ny", [13, 21, 22, 32, 33, 34, 37, 68, 127])
@pytest.mark.parametrize("xw", [False, True])
def test_large_prime_radices(ny, xw):
    torch = torch_cuda()
    b = binding()
    nx, batch = (ny if xw else 19), 3
    lx, ly = grid_lengths(nx, ny, xw)
    ctx = b.Context(nx, ny, lx, ly, x_walls=xw, batch=batch, family="G8", h_over_dx=1.3)
    p = oracle_problem(nx, ny, xw, "G8", 1.3)
    f = np.stack([inputs.smooth_field(nx, ny, seed=5 + k) for k in range(batch)])
    names = ["DX", "DY", "LAP"]
    outs = [torch.zeros((batch, nx, ny), dtype=torch.float64, device="cuda") for _ in names]
    ctx.spectral_op(to_dev(f), names, outs)
    ctx.sync()
    fn = lambda x: oops.apply_symbols(x, [p.sym[n] for n in names], p.E_dir, p.E_dir if xw else None)
    for k in range(batch):
        for n, o, r, fl in zip(names, outs, fn(f[k]), ulp_floor(fn, f[k])):
            err = rel_l2(o[k].cpu().numpy(), r)
            assert err < parity_tol(fl), (n, k, err, fl)
