"""What the speed of this framework is measured on: the calls its users make, over the sizes they make them at.

A case names one public entry point and the sizes of one call.  ``prepare``
makes what a program holds before the call (images on the device, segment
tables, a network, an annealing run); ``run`` is one call; ``exact`` restates
the result in plain NumPy / PyTorch where that takes seconds.

Media: Boolean models of disks, ellipses, squares and balls on the torus, and
clustered disks (parents uniform, Poisson children displaced normally), the
kinds of microstructure the paper evaluates.
"""
import math

import numpy as np
import torch

import paper_1601_04359_gb300 as lpf

CHANNELS = (2, 32, 64, 48, 32, 2)  # of the proposal network


def listed():
    return [
        # The smallest descriptor anyone computes: a 64x64 cell, window 32.
        # Launches and latency decide; annealing start-ups and tests do this.
        {"name": "full_64", "path": "full", "H": 64, "W": 64, "rx": 32, "ry": 32, "medium": "disks",
         "fraction": 0.4, "tuned": False},
        # The headline workload: the descriptor of a 512x512 original, window
        # 256, with the launch shape tuned once as for a fixed image size.
        {"name": "full_512", "path": "full", "H": 512, "W": 512, "rx": 256, "ry": 256, "medium": "ellipses",
         "fraction": 0.35, "tuned": True},
        # The whole domain of a non-square image of odd extents, as in the
        # timing table over full domains; sparse squares, long dead segments.
        {"name": "domain_175x201", "path": "full", "H": 175, "W": 201, "rx": 200, "ry": 174, "medium": "squares",
         "fraction": 0.2, "tuned": False},
        # Average over the parallel cuts of a volume: many small images, one sum.
        {"name": "ensemble_64", "path": "ensemble", "n": 64, "H": 100, "W": 128, "rx": 40, "ry": 32,
         "medium": "disks", "fraction": 0.3},
        # Independent images of uneven sizes in one graph launch.
        {"name": "batch_32", "path": "batch", "n": 32, "lo": 48, "hi": 256, "sizes": 4},
        # A periodic volume, 3D segments (the 3D extension's benchmark).
        {"name": "volume_128", "path": "volume", "D": 128, "H": 128, "W": 128, "r": 16, "fraction": 0.3},
        # A large batch of candidate exchanges, error changes only: what a
        # user who searches for swaps or logs training data evaluates.
        {"name": "delta_4096", "path": "delta", "H": 128, "W": 128, "rx": 64, "ry": 64, "K": 4096,
         "fraction": 0.3, "counts": False},
        # A snapshot's 64 candidates on a 50x50 cell with its full domain,
        # count changes and error changes.
        {"name": "delta_64", "path": "delta", "H": 50, "W": 50, "rx": 49, "ry": 49, "K": 64, "fraction": 0.3,
         "counts": True},
        # Simulated annealing of a 128x128 cell against a 512x512 original:
        # 256 batches between two looks at the progress.
        {"name": "anneal_128", "path": "anneal", "H": 128, "W": 128, "rx": 64, "ry": 64, "batches": 256,
         "fraction": 0.3},
        # The proposal network scoring one cell (between annealing batches).
        {"name": "scores_128", "path": "scores", "H": 128, "W": 128, "fraction": 0.3},
        # One training step of the network on 8 snapshots, then its weights.
        {"name": "train_128", "path": "train", "H": 128, "W": 128, "B": 8, "n": 64, "fraction": 0.3},
        # The two-point probability of a 512x512 image (the other descriptor).
        {"name": "s2_512", "path": "s2", "H": 512, "W": 512, "medium": "ellipses", "fraction": 0.35, "phase": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["full", "full", "full", "ensemble", "batch", "volume", "delta", "delta", "anneal", "scores",
                       "train", "s2"])
    fraction = round(rng.uniform(0.2, 0.6), 3)
    medium = rng.choice(["disks", "ellipses", "squares", "clustered"])
    if path == "full":
        H, W = _log(rng, 24, 400), _log(rng, 24, 400)
        share = rng.choice([0.25, 0.5, 0.5, 1.0 if H * W < 40000 else 0.5])
        return {"path": path, "H": H, "W": W, "rx": min(W - 1, max(1, int(share * W))),
                "ry": min(H - 1, max(1, int(share * H))), "medium": medium, "fraction": fraction,
                "tuned": rng.random() < 0.3}
    if path == "ensemble":
        H, W = _log(rng, 40, 128), _log(rng, 40, 128)
        return {"path": path, "n": _log(rng, 4, 64), "H": H, "W": W, "rx": W // 4 + rng.randint(0, 6),
                "ry": H // 4 + rng.randint(0, 6), "medium": medium, "fraction": fraction}
    if path == "batch":
        lo = rng.choice([32, 48, 64])
        return {"path": path, "n": rng.randint(8, 32), "lo": lo, "hi": rng.randint(2 * lo, 240),
                "sizes": rng.randint(0, 1 << 20)}
    if path == "volume":
        D, H, W = (_log(rng, 32, 128) for _ in range(3))
        return {"path": path, "D": D, "H": H, "W": W, "r": rng.randint(6, 15), "fraction": fraction}
    if path == "delta":
        H, W = _log(rng, 20, 128), _log(rng, 20, 128)
        share = rng.choice([0.25, 0.5])
        return {"path": path, "H": H, "W": W, "rx": max(1, int(share * W)), "ry": max(1, int(share * H)),
                "K": _log(rng, 1, 4000), "fraction": fraction, "counts": rng.random() < 0.4}
    if path == "anneal":
        H, W = rng.randint(48, 128), rng.randint(48, 128)
        return {"path": path, "H": H, "W": W, "rx": W // 4 + rng.randint(0, W // 4), "ry": H // 4 + rng.randint(0, H // 4),
                "batches": rng.randint(32, 256), "fraction": fraction}
    if path == "scores":
        return {"path": path, "H": _log(rng, 20, 160), "W": _log(rng, 20, 160), "fraction": fraction}
    if path == "train":
        return {"path": path, "H": _log(rng, 20, 128), "W": _log(rng, 20, 128), "B": rng.randint(1, 8),
                "n": rng.randint(16, 64), "fraction": fraction}
    return {"path": path, "H": _log(rng, 50, 512), "W": _log(rng, 50, 512), "medium": medium, "fraction": fraction,
            "phase": rng.randint(0, 1)}


# ---- media ------------------------------------------------------------------

def _stamp(img, rows, cols, dy, dx, hit):
    """Set img where hit [n][m] at rows [n] + dy [m], cols [n] + dx [m], on the torus."""
    H, W = img.shape
    y = (rows[:, None] + dy[None, :]) % H
    x = (cols[:, None] + dx[None, :]) % W
    img[y[hit], x[hit]] = 1


def _medium(rng, H, W, medium, fraction):
    """A two-phase image (uint8 0/1) whose expected phase-1 fraction is about `fraction`."""
    img = np.zeros((H, W), np.uint8)
    load = -math.log(1.0 - fraction) * H * W  # area of all particles, overlaps counted
    small = min(H, W)
    if medium == "squares":
        s = 4
        n = max(1, int(round(load / s ** 2)))
        dy, dx = (a.reshape(-1) for a in np.mgrid[0:s, 0:s])
        _stamp(img, rng.integers(0, H, n), rng.integers(0, W, n), dy, dx, np.ones((n, s * s), bool))
        return img
    lo, hi = (6.0, 20.0) if medium == "ellipses" else (5.0, 5.0)
    lo, hi = min(lo, small / 6), min(hi, small / 4)
    n = max(1, int(round(load / (math.pi * (0.5 * (lo + hi)) ** 2))))
    if medium == "clustered":
        parents = rng.uniform(0, 1, (max(1, n // 8), 2)) * (H, W)
        c = parents[rng.integers(0, len(parents), n)] + rng.normal(0, 12.0, (n, 2))
    else:
        c = rng.uniform(0, 1, (n, 2)) * (H, W)
    a, b = rng.uniform(lo, hi, n), rng.uniform(lo, hi, n)
    t = rng.uniform(0, math.pi, n)
    rows, cols = np.floor(c[:, 0]).astype(int), np.floor(c[:, 1]).astype(int)
    m = int(math.ceil(hi)) + 1
    dy, dx = (q.reshape(-1) for q in np.mgrid[-m:m + 1, -m:m + 1])
    py = rows[:, None] + dy + 0.5 - c[:, 0:1]
    px = cols[:, None] + dx + 0.5 - c[:, 1:2]
    u = np.cos(t)[:, None] * px + np.sin(t)[:, None] * py
    v = -np.sin(t)[:, None] * px + np.cos(t)[:, None] * py
    _stamp(img, rows, cols, dy, dx, (u / a[:, None]) ** 2 + (v / b[:, None]) ** 2 <= 1.0)
    return img


def _balls(rng, D, H, W, fraction):
    """A periodic volume of overlapping balls of radius 5 (or a sixth of its shortest side)."""
    R = min(5.0, min(D, H, W) / 6)
    n = max(1, int(round(-math.log(1.0 - fraction) * D * H * W / (4.0 / 3.0 * math.pi * R ** 3))))
    c = rng.uniform(0, 1, (n, 3)) * (D, H, W)
    m = int(math.ceil(R)) + 1
    o = np.stack([q.reshape(-1) for q in np.mgrid[-m:m + 1, -m:m + 1, -m:m + 1]], axis=1)
    vol = np.zeros((D, H, W), np.uint8)
    p = np.floor(c).astype(int)[:, None, :] + o[None]
    hit = ((p + 0.5 - c[:, None, :]) ** 2).sum(-1) <= R * R
    p = p[hit] % (D, H, W)
    vol[p[:, 0], p[:, 1], p[:, 2]] = 1
    return vol


def _two_phases(img):
    """At least a few pixels of each phase (a cell of one phase has no exchanges)."""
    if img.min() == img.max():
        img[: max(1, img.shape[0] // 2)] ^= 1
    return img


def _exchanges(rng, cell, K):
    """int32 [K][2]: a phase-1 pixel and a phase-0 pixel of the cell each, uniform."""
    flat = cell.reshape(-1)
    return np.stack([rng.choice(np.flatnonzero(flat == 1), K), rng.choice(np.flatnonzero(flat == 0), K)],
                    axis=1).astype(np.int32)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _network(rng):
    """He-normal weights and small biases, in the network's parameter order."""
    parts = []
    for ci, co in zip(CHANNELS[:-1], CHANNELS[1:]):
        parts += [rng.normal(0, math.sqrt(2.0 / (9 * ci)), 9 * ci * co), rng.normal(0, 0.01, co)]
    return np.concatenate(parts).astype(np.float32)


# ---- one call -----------------------------------------------------------------

def _cell(case, rng):
    return _two_phases(_medium(rng, case["H"], case["W"], "clustered", case["fraction"]))


def _delta_inputs(case, seed):
    rng = np.random.default_rng(seed)
    cell = _cell(case, rng)
    return cell, _exchanges(rng, cell, case["K"]), rng.uniform(0.8, 1.0)


def _score_inputs(case, seed):
    rng = np.random.default_rng(seed)
    return _cell(case, rng), _network(rng)


def _train_inputs(case, seed):
    rng = np.random.default_rng(seed)
    cells = np.stack([_cell(case, rng) for _ in range(case["B"])])
    pairs = np.stack([_exchanges(rng, c, case["n"]) for c in cells])
    y = np.clip(rng.normal(size=(case["B"], case["n"])), -3, 3).astype(np.float32)
    return cells, pairs, y, _network(rng)


LEARNING_RATE = 1e-3


def prepare(case, seed):
    path = case["path"]
    rng = np.random.default_rng(seed)
    if path == "full":
        img = _gpu(_medium(rng, case["H"], case["W"], case["medium"], case["fraction"]))
        paths = lpf.lpf_build_paths(case["rx"], case["ry"])
        counts = torch.empty((2, paths.n_full), dtype=torch.int64, device="cuda")
        if case["tuned"]:
            lpf.lpf_autotune_full(img, paths, counts)
        return {"case": case, "img": img, "paths": paths, "counts": counts}
    if path == "ensemble":
        imgs = _gpu(np.stack([_medium(rng, case["H"], case["W"], case["medium"], case["fraction"])
                              for _ in range(case["n"])]))
        paths = lpf.lpf_build_paths(case["rx"], case["ry"])
        counts = torch.empty((2, paths.n_full), dtype=torch.int64, device="cuda")
        return {"case": case, "imgs": imgs, "paths": paths, "counts": counts}
    if path == "batch":
        kinds = ("disks", "ellipses", "clustered")
        sizes = np.random.default_rng(case["sizes"]).integers(case["lo"], case["hi"] + 1, (case["n"], 2))
        imgs = [_medium(rng, int(H), int(W), kinds[i % 3], float(rng.uniform(0.2, 0.6)))
                for i, (H, W) in enumerate(sizes)]
        paths = [lpf.lpf_build_paths(i.shape[1] // 2, i.shape[0] // 2) for i in imgs]
        batch = lpf.lpf_batch_create([_gpu(i) for i in imgs], paths)
        return {"case": case, "batch": batch}
    if path == "volume":
        vol = _gpu(_balls(rng, case["D"], case["H"], case["W"], case["fraction"]))
        paths = lpf.lpf_build_paths_3d(case["r"], case["r"], case["r"])
        counts = torch.empty((2, paths.n_full), dtype=torch.int64, device="cuda")
        return {"case": case, "vol": vol, "paths": paths, "counts": counts}
    if path == "delta":
        cell, pairs, scale = _delta_inputs(case, seed)
        paths = lpf.lpf_build_paths(case["rx"], case["ry"])
        d = _gpu(cell)
        counts = lpf.lpf_full(d, paths)
        target = (counts.double() * (scale / cell.size)).float()
        return {"case": case, "cell": d, "paths": paths, "counts": counts, "target": target, "pairs": _gpu(pairs)}
    if path == "anneal":
        # the target is the descriptor of an original four times as wide and
        # high; the cell starts as a shuffle with the original's fraction
        orig = _two_phases(_medium(rng, 4 * case["H"], 4 * case["W"], "clustered", case["fraction"]))
        paths = lpf.lpf_build_paths(case["rx"], case["ry"])
        target = (lpf.lpf_full(_gpu(orig), paths).double() / float(orig.size)).float()
        flat = np.zeros(case["H"] * case["W"], np.uint8)
        ones = min(flat.size - 1, max(1, int(round(float(orig.mean()) * flat.size))))
        flat[rng.choice(flat.size, ones, replace=False)] = 1
        cell = _gpu(flat.reshape(case["H"], case["W"]))
        run_ = lpf.lpf_sa_create(cell, paths, target, n_step=1_000_000, seed=int(rng.integers(1, 1 << 30)))
        return {"case": case, "anneal": run_}
    if path == "scores":
        cell, params = _score_inputs(case, seed)
        net = lpf.lpf_cnn_create(case["H"], case["W"])
        lpf.lpf_cnn_set_params(net, params)
        return {"case": case, "net": net, "cell": _gpu(cell)}
    if path == "train":
        cells, pairs, y, params = _train_inputs(case, seed)
        net = lpf.lpf_cnn_create(case["H"], case["W"])
        lpf.lpf_cnn_set_params(net, params)
        return {"case": case, "net": net, "cells": _gpu(cells), "pairs": _gpu(pairs), "y": _gpu(y)}
    img = _gpu(_medium(rng, case["H"], case["W"], case["medium"], case["fraction"]))
    return {"case": case, "img": img, "out": torch.empty((case["H"], case["W"]), dtype=torch.float32, device="cuda")}


def run(state):
    case = state["case"]
    path = case["path"]
    if path == "full":
        return lpf.lpf_full(state["img"], state["paths"], state["counts"])
    if path == "ensemble":
        return lpf.lpf_full_ensemble(state["imgs"], state["paths"], state["counts"])
    if path == "batch":
        return lpf.lpf_batch_run(state["batch"], use_graph=True)
    if path == "volume":
        return lpf.lpf_full_3d(state["vol"], state["paths"], state["counts"])
    if path == "delta":
        dcounts, de = lpf.lpf_delta_swap(state["cell"], state["paths"], state["pairs"], target=state["target"],
                                         counts=state["counts"], want_dcounts=case["counts"], want_de=True)
        return {"dcounts": dcounts, "de": de} if case["counts"] else {"de": de}
    if path == "anneal":
        lpf.lpf_sa_run(state["anneal"], case["batches"])
        st = lpf.lpf_sa_read(state["anneal"])  # the look at the progress
        return {"cell": state["anneal"].cell, "counts": state["anneal"].counts, "n_eval": st["n_eval"],
                "n_accept": st["n_accept"]}
    if path == "scores":
        return lpf.lpf_cnn_forward(state["net"], state["cell"])
    if path == "train":
        loss = lpf.lpf_cnn_train_step(state["net"], state["cells"], state["pairs"], state["y"], LEARNING_RATE)
        return {"loss": loss, "params": lpf.lpf_cnn_get_params(state["net"])}
    return lpf.s2_fft(state["img"], case["phase"], state["out"])


# ---- what a pass cannot do without ----------------------------------------------

def _window(rx, ry):
    """Vectors of the window and of its canonical half."""
    n = (2 * rx + 1) * (2 * ry + 1)
    return n, (n + 1) // 2


def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: for counts,
    one AND and one shift per canonical vector, 32 translations and phase (a
    segment is at least one pixel longer than what it shares); for
    exchanges, four per candidate and vector; for the network, its
    multiply-adds; for the two-point probability, two real transforms."""
    path = case["path"]
    if path in ("full", "ensemble"):
        n_full, n_canon = _window(case["rx"], case["ry"])
        n = case.get("n", 1)
        return {"bytes": n * case["H"] * case["W"] + 16 * n_full,
                "flops": 4 * n * n_canon * case["H"] * -(-case["W"] // 32)}
    if path == "batch":
        side = 0.5 * (case["lo"] + case["hi"])
        n_full = (side + 1) ** 2
        return {"bytes": int(case["n"] * (side * side + 16 * n_full)),
                "flops": int(case["n"] * 2 * n_full * side * side / 32)}
    if path == "volume":
        n_full = (2 * case["r"] + 1) ** 3
        cells = case["D"] * case["H"] * case["W"]
        return {"bytes": cells + 16 * n_full, "flops": 2 * n_full * cells // 32}
    if path == "delta":
        n_full, n_canon = _window(case["rx"], case["ry"])
        out = 4 + (8 * n_canon if case["counts"] else 0)
        return {"bytes": case["H"] * case["W"] + 24 * n_canon + case["K"] * (8 + out),
                "flops": 4 * case["K"] * n_canon}
    if path == "anneal":
        n_full, n_canon = _window(case["rx"], case["ry"])
        return {"bytes": 2 * case["H"] * case["W"] + 24 * n_full, "flops": 4 * case["batches"] * n_canon}
    if path in ("scores", "train"):
        pix = case["H"] * case["W"]
        macs = 9 * sum(a * b for a, b in zip(CHANNELS[:-1], CHANNELS[1:]))
        if path == "scores":
            return {"bytes": pix * 9 + 2 * macs, "flops": 2 * pix * macs}
        return {"bytes": case["B"] * (pix + 12 * case["n"]) + 24 * macs, "flops": 6 * case["B"] * pix * macs}
    pix = case["H"] * case["W"]
    return {"bytes": 5 * pix, "flops": int(2 * 2.5 * pix * math.log2(max(2, pix)))}


# ---- the results in 64 bits --------------------------------------------------------

def _segments(rx, ry):
    """Canonical vectors (dx, dy) in window order and their pixels: step i of
    a = max(|dx|, |dy|) moves i along the longer axis and round(i b / a)
    along the other, halves away from the start."""
    for dy in range(0, ry + 1):
        for dx in range(-rx if dy else 0, rx + 1):
            a, b = max(abs(dx), dy), min(abs(dx), dy)
            i = np.arange(a + 1)
            o = (2 * i * b + a) // (2 * a) if a else i
            s = -1 if dx < 0 else 1
            yield (s * i, o) if abs(dx) >= dy else (s * o, i)


def _phase0_pixels(flat, pos, H, W, sx, sy):
    """Phase-0 pixels of the segment placed at every translation."""
    y, x = pos
    q = ((y[None] + sy[:, None]) % H) * W + (x[None] + sx[:, None]) % W
    return (flat[q] == 0).sum(0)


def _exact_counts(img, rx, ry):
    H, W = img.shape
    flat = _gpu(img.reshape(-1))
    i = torch.arange(H * W, device="cuda")
    half = []
    for sx, sy in _segments(rx, ry):
        z = _phase0_pixels(flat, (i // W, i % W), H, W, _gpu(sx), _gpu(sy))
        half.append(torch.stack([(z == len(sx)).sum(), (z == 0).sum()]))
    half = torch.stack(half, dim=1)
    return torch.cat([half[:, 1:].flip(1), half], dim=1)


def _exact_delta(case, seed):
    cell, pairs, scale = _delta_inputs(case, seed)
    H, W = cell.shape
    rx, ry = case["rx"], case["ry"]
    N = H * W
    flat = _gpu(cell.reshape(-1))
    i = torch.arange(N, device="cuda")
    pos = (i // W, i % W)
    pairs = _gpu(pairs).long()
    ay, ax, by, bx = pairs[:, 0] // W, pairs[:, 0] % W, pairs[:, 1] // W, pairs[:, 1] % W
    de = torch.zeros(len(pairs), dtype=torch.float64, device="cuda")
    d0s, d1s = [], []
    for sx, sy in _segments(rx, ry):
        L = len(sx)
        tx, ty = _gpu(sx), _gpu(sy)
        z = _phase0_pixels(flat, pos, H, W, tx, ty)
        c0, c1 = (z == L).sum().double(), (z == 0).sum().double()
        xa, xb = ((py[:, None] - ty) % H * W + (px[:, None] - tx) % W for py, px in ((ay, ax), (by, bx)))
        both_a = (xa[:, :, None] == xb[:, None, :]).any(2) if L * L * len(pairs) < 5e7 else _in_rows(xa, xb, N)
        both_b = (xb[:, :, None] == xa[:, None, :]).any(2) if L * L * len(pairs) < 5e7 else _in_rows(xb, xa, N)
        za, zb = z[xa], z[xb]
        d0 = ((za == L - 1) & ~both_a).sum(1) - ((zb == L) & ~both_b).sum(1)
        d1 = ((zb == 1) & ~both_b).sum(1) - ((za == 0) & ~both_a).sum(1)
        for c, d in ((c0, d0), (c1, d1)):
            t = (c * (scale / N)).float().double()
            de += (t - (c + d) / N) ** 2 - (t - c / N) ** 2
        d0s.append(d0)
        d1s.append(d1)
    if not case["counts"]:
        return {"de": de}
    return {"dcounts": torch.stack([torch.stack(d0s, 1), torch.stack(d1s, 1)], dim=1), "de": de}


def _in_rows(a, b, N):
    """Whether a[k][i] is among b[k] (values in [0, N))."""
    mark = torch.zeros((len(b), N), dtype=torch.bool, device=b.device).scatter_(1, b, True)
    return mark.gather(1, a)


def _features(cells):
    """[B][2][H][W] float64: the cell and its interfacial mask (4-neighbourhood on the torus)."""
    c = _gpu(cells).double()
    m = torch.zeros_like(c)
    for axis in (1, 2):
        for s in (1, -1):
            m = torch.maximum(m, (c != c.roll(s, axis)).double())
    return torch.stack([c, m], dim=1)


def _split(params):
    out, at = [], 0
    for ci, co in zip(CHANNELS[:-1], CHANNELS[1:]):
        w = params[at:at + 9 * ci * co].reshape(3, 3, ci, co).permute(3, 2, 0, 1)
        at += 9 * ci * co
        out.append((w, params[at:at + co]))
        at += co
    return out


def _scores(params, cells):
    """[B][H][W][2] scores in 64 bits."""
    x = _features(cells)
    layers = _split(params)
    for k, (w, b) in enumerate(layers):
        x = torch.nn.functional.conv2d(torch.nn.functional.pad(x, (1, 1, 1, 1), mode="circular"), w, b)
        if k + 1 < len(layers):
            x = torch.relu(x)
    return x.permute(0, 2, 3, 1)


def _exact_train(case, seed):
    cells, pairs, y, params = _train_inputs(case, seed)
    p = _gpu(params).double().requires_grad_(True)
    s = _scores(p, cells).reshape(case["B"], -1, 2)
    q, t = _gpu(pairs).long(), _gpu(y).double()
    k = torch.arange(case["B"], device="cuda")[:, None]
    r = s[k, q[:, :, 0], 1] + s[k, q[:, :, 1], 0] - t
    loss = 0.5 * (r * r).mean()
    (g,) = torch.autograd.grad(loss, p)
    new = p.detach() - LEARNING_RATE * g / (g.abs() + 1e-8)  # the first Adam step
    return {"loss": loss.detach().reshape(1), "params": new.cpu().numpy()}


def exact(case, seed):
    path = case["path"]
    if path == "full":
        if (case["rx"] + 1) * (case["ry"] + 1) * case["H"] * case["W"] > 5e6:
            return None  # minutes
        img = _medium(np.random.default_rng(seed), case["H"], case["W"], case["medium"], case["fraction"])
        return _exact_counts(img, case["rx"], case["ry"])
    if path == "delta":
        return _exact_delta(case, seed)
    if path == "scores":
        cell, params = _score_inputs(case, seed)
        with torch.no_grad():
            return _scores(_gpu(params).double(), cell[None])[0]
    if path == "train":
        return _exact_train(case, seed)
    if path == "s2":
        img = _medium(np.random.default_rng(seed), case["H"], case["W"], case["medium"], case["fraction"])
        f = torch.fft.fft2((_gpu(img) == case["phase"]).double())
        return torch.fft.ifft2(f * f.conj()).real / img.size
    return None  # whole numbers, and no short way to them
