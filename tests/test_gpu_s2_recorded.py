"""s2_fft recorded into CUDA graphs: recorded calls of one size have areas of
their own, so they may run side by side -- two graphs on two streams, two
branches of one graph -- and the areas go when the graphs do."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _expected(img, phase):
    chi = (img == phase).astype(np.float64)
    f = np.fft.fft2(chi)
    return (np.rint(np.fft.ifft2(f * f.conj()).real) / img.size).astype(np.float32)


@pytest.mark.parametrize("H,W", [(512, 512), (300, 1024), (1, 9)])
def test_two_graphs_on_two_streams(gpu_lib, H, W):
    imgs = [synth.random_binary(H, W, 0.2 + 0.4 * k, seed=k) for k in range(2)]
    d = [torch.from_numpy(i).cuda() for i in imgs]
    outs = [torch.empty((H, W), dtype=torch.float32, device="cuda") for _ in imgs]
    streams, graphs = [torch.cuda.Stream() for _ in imgs], []
    for x, out in zip(d, outs):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            gpu_lib.s2_fft(x, 1, out)
        graphs.append(g)
    for _ in range(20):
        for out in outs:
            out.zero_()
        torch.cuda.synchronize()
        for _ in range(10):
            for g, s in zip(graphs, streams):
                with torch.cuda.stream(s):
                    g.replay()
        torch.cuda.synchronize()
        for out, i in zip(outs, imgs):
            np.testing.assert_array_equal(out.cpu().numpy(), _expected(i, 1))


def test_two_branches_of_one_graph(gpu_lib):
    img = synth.random_binary(300, 500, 0.3, seed=5)
    d = torch.from_numpy(img).cuda()
    outs = [torch.empty(img.shape, dtype=torch.float32, device="cuda") for _ in range(2)]
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g):
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        gpu_lib.s2_fft(d, 0, outs[0], stream=side)
        gpu_lib.s2_fft(d, 1, outs[1], stream=main)
        main.wait_stream(side)
    for _ in range(50):
        g.replay()
        torch.cuda.synchronize()
        for phase in (0, 1):
            np.testing.assert_array_equal(outs[phase].cpu().numpy(), _expected(img, phase))


def test_areas_go_with_their_graphs(gpu_lib):
    img = synth.random_binary(4096, 1024, 0.3, seed=6)  # 25 MB each
    d, out = torch.from_numpy(img).cuda(), torch.empty(img.shape, dtype=torch.float32, device="cuda")
    gpu_lib.s2_fft(d, 1, out)
    ref = out.clone()
    torch.cuda.synchronize()
    free = None
    for k in range(40):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            gpu_lib.s2_fft(d, 1, out)
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
        if k == 4:
            free = torch.cuda.mem_get_info()[0]
        del g
    assert free - torch.cuda.mem_get_info()[0] < 200 << 20  # (40 areas: 1 GB)
