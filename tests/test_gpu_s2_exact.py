"""s2_fft's transforms mod p against the correlation counts from NumPy's FFT,
rounded to whole numbers (they are): equal to the last bit, on extents that
are and are not powers of two, thin images, both phases, and in a stream of
the caller's."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _expected(img, phase):
    chi = (img == phase).astype(np.float64)
    f = np.fft.fft2(chi)
    return (np.rint(np.fft.ifft2(f * f.conj()).real) / img.size).astype(np.float32)


@pytest.mark.parametrize("H,W", [(1, 1), (1, 2), (2, 3), (3, 1), (5, 7), (8, 8), (31, 64), (100, 33), (256, 5), (129, 512),
                                 (500, 375), (1, 4096), (2048, 3), (1023, 1024)])
def test_whole_counts_over_the_area(gpu_lib, H, W):
    img = synth.random_binary(H, W, 0.4, seed=H + W)
    s = torch.cuda.Stream()
    for phase in (0, 1):
        d = torch.from_numpy(img).cuda()
        torch.cuda.synchronize()
        got = gpu_lib.s2_fft(d, phase, stream=s)
        s.synchronize()
        np.testing.assert_array_equal(got.cpu().numpy(), _expected(img, phase))



def test_recorded_into_a_graph(gpu_lib):
    a, b = (synth.random_binary(96, 130, 0.4, seed=k) for k in (3, 4))
    d = torch.from_numpy(a).cuda()
    out = torch.empty((96, 130), dtype=torch.float32, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gpu_lib.s2_fft(d, 1, out)
    for img in (b, a):
        d.copy_(torch.from_numpy(img))
        g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy(), _expected(img, 1))
