"""The in-place engine at the lengths where its places can go wrong: large prime
radices (19, 23, 29, 31: one scratch line), Rader lengths whose p - 1 ends in
one, lengths around whole 128-byte blocks, and line counts from one to a ragged
last CTA, against numpy's FFT."""
import numpy as np
import pytest

from gpu_common import binding, torch_cuda


@pytest.mark.gpu
@pytest.mark.parametrize("n", [6, 15, 17, 19, 23, 38, 47, 59, 73, 127, 179, 186, 311, 361, 363, 899, 1919])
@pytest.mark.parametrize("prec", ["f64", "f32", "f32x2"])
@pytest.mark.parametrize("nl", [1, 19])
def test_lines_match_numpy(n, prec, nl):
    torch = torch_cuda()
    b = binding()
    rng = np.random.default_rng(n)
    x = rng.standard_normal((nl, n)) + 1j * rng.standard_normal((nl, n))
    xd = torch.tensor(x, dtype=torch.complex64 if prec == "f32" else torch.complex128).cuda()
    for direction in (-1, 1):
        y = b.fcsph_dft(xd, direction, double_float=prec == "f32x2").cpu().numpy()
        ref = np.fft.fft(x, axis=-1) if direction < 0 else np.fft.ifft(x, axis=-1) * n
        # unit roundoff per pass (FP64 2^-53, FP32 pairs 32x that, FP32 2^-24) times log2 n passes, twice for
        # the two transforms of a convolution, and the 31 terms summed in order by a large radix
        u = {"f64": 2e-15, "f32x2": 32 * 2e-15, "f32": 3e-7}[prec]
        err = np.linalg.norm(y - ref) / np.linalg.norm(ref)
        assert err < u * np.log2(n) * 4, (n, prec, direction, err)
