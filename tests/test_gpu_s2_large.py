"""s2_fft on both sides of the line between the transforms mod p (extents whose
transforms hold up to 4096 values, 2^22 in all) and the double-precision FFTs,
against the correlation counts from NumPy's FFT, rounded to whole numbers.
Bound of the FFTs: half an ulp of float32 plus their rounding (a few 1e-16
times log2(WH) relative to the largest value, which is at most 1)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _counts(img, phase):
    f = np.fft.rfft2((img == phase).astype(np.float64))
    return np.rint(np.fft.irfft2(f * f.conj(), img.shape))


@pytest.mark.parametrize("H,W,exact", [(1024, 4096, True), (4096, 1024, True), (2048, 2048, True), (1024, 1025, True),
                                       (1, 4097, False), (5000, 1, False), (2049, 3, False), (3, 2050, False),
                                       (1025, 1025, False), (4096, 2048, False), (8192, 16, False)])
def test_both_sides_of_the_line(gpu_lib, H, W, exact):
    img = synth.random_binary(H, W, 0.4, seed=H + W)
    d = torch.from_numpy(img).cuda()
    for phase in (0, 1):
        got, ref = gpu_lib.s2_fft(d, phase).cpu().numpy(), _counts(img, phase) / img.size
        if exact:
            np.testing.assert_array_equal(got, ref.astype(np.float32))
        else:
            assert (np.abs(got - ref) <= 2.0 ** -24 * ref + 1e-12 * (1 + np.log2(H * W))).all()
