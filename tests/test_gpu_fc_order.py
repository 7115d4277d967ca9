"""The FC continuation sums of small FP64 launches (two threads a sum) and of full
ones must round alike: one instance alone equals the same instance in a batch that
fills the GPU, bit for bit, on walls whose sums are nearly halfway between two
doubles, where any other order of the compensated sum shows."""
import os

import numpy as np
import pytest

from gpu_common import binding, to_dev, torch_cuda
from tables import gram_golden

WALLS = np.loadtxt(os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fc_halfway_walls.txt"))[:32, 1:]


@pytest.mark.gpu
@pytest.mark.parametrize("ny", [10, 39, 64])
def test_halfway_sums_alone_and_in_a_full_batch(ny):
    torch = torch_cuda()
    b = binding()
    nx, full = len(WALLS), 24  # 16 column pairs alone, 384 in the batch: 152 SMs
    f = np.zeros((full, nx, ny))
    f[:, :, :5], f[:, :, ny - 5:] = WALLS[:, :5], WALLS[:, 5:]
    E = gram_golden(5, 25)
    got = []
    for batch in (1, full):
        ctx = b.Context(nx, ny, nx / (ny - 1.0), 1.0, batch=batch, table_dir=E, table_neu=E)
        fd = to_dev(f[:batch])
        outs = [torch.zeros_like(fd) for _ in range(3)]
        ctx.line_op(fd, ["W", "DY", "LAP"], outs)
        plane = [torch.zeros_like(fd)]
        ctx.spectral_op(fd, ["LAP"], plane)
        ctx.sync()
        got.append([o[0].cpu().numpy() for o in outs + plane])
    for a, r in zip(*got):
        np.testing.assert_array_equal(a, r)
