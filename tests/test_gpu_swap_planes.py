"""Swap deltas from bit planes against the oracle's recount: word and row
edges, segments up to the longest the byte sums take, windows of the full
domain (displacements that wrap), both ways of evaluating candidates (sums
for every pixel, lookups per candidate) and sampled translations."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

# H, W, rx, ry, exchanges checked
SIZES = [(8, 5, 4, 7, 12), (31, 32, 16, 15, 12), (33, 31, 30, 9, 8), (20, 33, 7, 19, 12), (64, 65, 20, 21, 6),
         (40, 96, 48, 11, 6), (97, 64, 12, 33, 4), (12, 256, 254, 2, 2), (256, 9, 2, 254, 2), (150, 130, 3, 4, 6)]


@pytest.mark.parametrize("copies", [1, 400], ids=["few", "many"])
@pytest.mark.parametrize("H,W,rx,ry,k", SIZES)
def test_exchanges_match_a_recount(gpu_lib, H, W, rx, ry, k, copies):
    cell = synth.clustered_disks(H, W, 0.4, seed=H + W, R=2.5) if min(H, W) > 8 else synth.random_binary(H, W, 0.4, 3)
    rng = np.random.default_rng(1)
    ones, zeros = np.flatnonzero(cell), np.flatnonzero(cell.reshape(-1) == 0)
    pairs = np.stack([rng.choice(ones, k), rng.choice(zeros, k)], 1).astype(np.int32)
    pairs[1] = pairs[0][::-1]              # reversed
    pairs[-1] = (ones[0], ones[-1])        # same phase: no change
    # neighbours, so that many segments hold both pixels
    y, x = np.argwhere((cell == 1) & (np.roll(cell, -1, 1) == 0))[0]
    pairs[0] = (y * W + x, y * W + (x + 1) % W)
    ref = oracle.delta_swap(cell, rx, ry, pairs)
    p = gpu_lib.lpf_build_paths(rx, ry)
    d = torch.from_numpy(cell).cuda()
    counts = gpu_lib.lpf_full(d, p)
    target = (counts.double() / cell.size * 0.9).float()
    dc, de = gpu_lib.lpf_delta_swap(d, p, torch.from_numpy(np.tile(pairs, (copies, 1))).cuda(), target=target,
                                    counts=counts, want_de=True)
    assert gpu_lib.lpf_paths_status(p) == 0
    dc, de = dc.cpu().numpy().reshape(copies, k, 2, -1), de.cpu().numpy().reshape(copies, k)
    assert all(np.array_equal(c, ref) for c in dc)
    assert all(np.array_equal(e, de[0]) for e in de)  # the same sums for every copy
    # float32 terms of about n_canon vectors, summed sequentially per chunk
    # and then over the chunks: one rounding per addition
    ref_de = oracle.delta_objective(target.cpu().numpy(), counts.cpu().numpy(), ref, rx, ry, H, W)
    _, n_canon, base = oracle.window_sizes(rx, ry)
    dd = target.cpu().numpy()[:, base:] - counts.cpu().numpy()[:, base:] / cell.size
    mag = np.abs(ref / cell.size * (ref / cell.size - 2 * dd[None])).sum(axis=(1, 2))
    assert (np.abs(de[0] - ref_de) <= (2 * n_canon + 8) * 2.0 ** -24 * mag + 1e-12).all()


@pytest.mark.parametrize("copies", [1, 400], ids=["few", "many"])
@pytest.mark.parametrize("H,W,rx,ry", [(31, 33, 15, 14), (20, 64, 30, 5)])
def test_sampled_translations(gpu_lib, H, W, rx, ry, copies):
    cell = synth.clustered_disks(H, W, 0.4, seed=7, R=2.5)
    sel = (np.random.default_rng(2).random((H, W)) < 0.3).astype(np.uint8)
    pairs = synth.swap_candidates(cell, 5, seed=3)
    before = oracle.lpf_full_selected(cell, rx, ry, sel)
    ref = []
    for a, b in pairs:
        c = cell.copy()
        c.reshape(-1)[[a, b]] = c.reshape(-1)[[b, a]]
        n_full = before.shape[1]
        ref.append((oracle.lpf_full_selected(c, rx, ry, sel) - before)[:, (n_full - 1) // 2:])
    p = gpu_lib.lpf_build_paths(rx, ry)
    dc, _ = gpu_lib.lpf_delta_swap_mc(torch.from_numpy(cell).cuda(), p, torch.from_numpy(sel).cuda(),
                                      torch.from_numpy(np.tile(pairs, (copies, 1))).cuda())
    assert gpu_lib.lpf_paths_status(p) == 0
    assert all(np.array_equal(c, np.stack(ref)) for c in dc.cpu().numpy().reshape(copies, 5, 2, -1))


def test_rounds_of_candidates(gpu_lib):
    """More candidates than the sums of one round hold: every copy has the sums
    and count changes of a short call."""
    H = W = 128
    r, k, copies = 64, 100, 1500
    cell = synth.clustered_disks(H, W, 0.4, seed=5)
    pairs = synth.swap_candidates(cell, k, seed=6).astype(np.int32)
    p = gpu_lib.lpf_build_paths(r, r)
    d, tp = torch.from_numpy(cell).cuda(), torch.from_numpy(pairs).cuda()
    counts = gpu_lib.lpf_full(d, p)
    target = (counts.double() / cell.size * 0.9).float()
    dc, one = gpu_lib.lpf_delta_swap(d, p, tp, target=target, counts=counts, want_de=True)
    assert np.array_equal(dc[:2].cpu().numpy(), oracle.delta_swap(cell, r, r, pairs[:2]))
    _, de = gpu_lib.lpf_delta_swap(d, p, tp.repeat(copies, 1), target=target, counts=counts, want_de=True,
                                   want_dcounts=False)
    assert (de.reshape(copies, k) == one).all()
