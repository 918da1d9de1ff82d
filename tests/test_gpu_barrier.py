"""The grid barrier of the annealer's larger batches (more than three
candidates; smaller ones exchange messages) is made to run out, in every block
and in one: reported, the run left consistent, and its result still that of the
sequential annealer."""
import time

import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import sa as osa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [-1, 0, 1])
def test_timeout_leaves_a_consistent_run(gpu_lib, block):
    H = W = 24
    r = 6
    orig = synth.clustered_disks(2 * H, 2 * W, 0.3, seed=9)
    target = (oracle.lpf_full(orig, r, r) / float(orig.size)).astype(np.float32)
    cell = synth.exact_fraction_shuffle(H, W, int(round(0.3 * H * W)), seed=4)
    n_step, c_max, s_max, t_max = 400, 40, 4, 2e-4
    p = gpu_lib.lpf_build_paths(r, r)
    d_cell = torch.from_numpy(cell).cuda()
    counts = torch.empty((2, p.n_full), dtype=torch.int64, device="cuda")
    ann = gpu_lib.lpf_sa_create(d_cell, p, torch.from_numpy(target).cuda(), counts, n_step=n_step, c_max=c_max,
                                s_max=s_max, t_max=t_max, k_min=4, k_max=64, seed=3)
    gpu_lib.lpf_sa_run(ann, 5)
    st1 = gpu_lib.lpf_sa_read(ann)
    assert st1["n_batches"] == 5 and st1["n_candidates"] >= 20  # four candidates or more in each batch
    t0 = time.time()
    rc = gpu_lib.lpf_sa_selftest_timeout(ann, block)
    assert rc == 0, gpu_lib.lpf_strerror(rc)
    assert time.time() - t0 < 60
    st2 = gpu_lib.lpf_sa_read(ann)  # status cleared: no LpfError
    assert st2["n_batches"] == st1["n_batches"] + (1 if block == 1 else 0)
    cell2 = d_cell.cpu().numpy()
    np.testing.assert_array_equal(counts.cpu().numpy(), oracle.lpf_full(cell2, r, r))
    e_ref = oracle.objective(target, oracle.lpf_full(cell2, r, r), r, r, H, W)
    assert abs(st2["error"] - e_ref) <= 1e-9 * max(1.0, abs(e_ref))
    while not gpu_lib.lpf_sa_read(ann)["done"]:
        gpu_lib.lpf_sa_run(ann, 16)
    ref_cell, ref_acc, _ = osa.anneal(cell, target, oracle.lpf_full(cell, r, r), r, r, n_step, c_max, s_max, t_max,
                                      0.01, seed=3)
    np.testing.assert_array_equal(d_cell.cpu().numpy(), ref_cell)
    assert gpu_lib.lpf_sa_read(ann)["n_accept"] == ref_acc
