"""What the framework is timed on: reconstruction of single tiles from a
nucleus-sized patch to a 4096 x 4096 slide tile, batches of tiles (many small
ragged patches, slide tiles of uneven sizes under the learned schedule, tiles
in host buffers), the distance transform, and the cost model's training.

Inputs follow the recipe of the repository's generator (noise in [20, 60] plus
Gaussian blobs; h-dome and border-seeded markers), drawn on the GPU from the
seed. Every case goes through the calls a user's program makes; a marker is
reconstructed in place, so a pass starts by copying the marker it was given.
"""
import math
import random

import numpy as np
import torch

import paper_1311_0378_gb300 as rc
from paper_1311_0378_gb300 import cost_model

OPS = {"dilate": rc.RECON_OP_DILATE, "erode": rc.RECON_OP_ERODE, "fill_holes": rc.RECON_OP_FILL_HOLES}
NFEAT, HIDDEN, NOUT = 20, 64, 2
NPARAMS = HIDDEN * NFEAT + HIDDEN + HIDDEN * HIDDEN + HIDDEN + NOUT * HIDDEN + NOUT


def listed():
    return [
        # one nucleus-sized patch cut out of a slide: a single small call, all latency
        dict(name="patch64", kind="tile", H=64, W=64, conn=8, op="dilate", marker="hdome"),
        # the small tile of the benchmark (h-domes of a 512 x 512 field of view)
        dict(name="tile512_hdome", kind="tile", H=512, W=512, conn=8, op="dilate", marker="hdome"),
        # the slide tile of the study, h-dome marker: propagation is local
        dict(name="tile4096_hdome", kind="tile", H=4096, W=4096, conn=8, op="dilate", marker="hdome"),
        # the same tile seeded from its border: values travel across the whole tile
        dict(name="tile4096_border", kind="tile", H=4096, W=4096, conn=4, op="dilate", marker="border"),
        # a region of interest of any size (odd row length), the dual operation
        dict(name="roi_erode", kind="tile", H=2999, W=3001, conn=8, op="erode", marker="border"),
        # hole filling of one mask
        dict(name="holes", kind="tile", H=1536, W=2560, conn=4, op="fill_holes", marker="none"),
        # patches of a segmentation's bounding boxes, any sizes, in one call
        dict(name="patches", kind="batch", tiles=256, lo=24, hi=320, step=1, conn=8, op="dilate", marker="hdome",
             learned=False),
        # slide tiles of uneven sizes and both markers, learned schedule (the benchmark's law)
        dict(name="uneven_learned", kind="batch", tiles=200, lo=256, hi=4096, step=256, conn=8, op="dilate",
             marker="both", learned=True),
        # masks in pinned host buffers, holes filled and copied back: the whole call
        dict(name="host_holes", kind="host", tiles=24, lo=512, hi=3072, step=64, conn=8, op="fill_holes",
             marker="none"),
        # distance transform of the objects, and of the space between them
        dict(name="dt_objects", kind="dt", H=2048, W=3000, mask="objects"),
        dict(name="dt_space", kind="dt", H=4096, W=4096, mask="space"),
        # a short training run of the cost model (forward, backward and Adam steps)
        dict(name="train", kind="train", samples=4096, batch=256, epochs=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tile"] * 5 + ["batch"] * 2 + ["host", "dt", "train"])
    conn = rng.choice([4, 8])
    if kind == "tile":
        op = rng.choice(["dilate", "dilate", "erode", "fill_holes"])
        return dict(kind=kind, H=_log(rng, 40, 4096), W=_log(rng, 40, 4096), conn=conn, op=op,
                    marker="none" if op == "fill_holes" else rng.choice(["hdome", "border"]))
    if kind == "batch":
        op = rng.choice(["dilate", "dilate", "erode", "fill_holes"])
        hi = _log(rng, 100, 3000)
        return dict(kind=kind, tiles=_log(rng, 2, 120), lo=max(16, hi // 12), hi=hi, step=rng.choice([1, 1, 16]),
                    conn=conn, op=op, marker="none" if op == "fill_holes" else rng.choice(["hdome", "border", "both"]),
                    learned=rng.random() < 0.5)
    if kind == "host":
        hi = _log(rng, 200, 2600)
        return dict(kind=kind, tiles=_log(rng, 1, 24), lo=max(16, hi // 8), hi=hi, step=1, conn=conn, op="fill_holes",
                    marker="none")
    if kind == "dt":
        return dict(kind=kind, H=_log(rng, 64, 4096), W=_log(rng, 64, 4096), mask=rng.choice(["objects", "space"]))
    return dict(kind=kind, samples=_log(rng, 300, 4096), batch=rng.choice([64, 100, 256]), epochs=1)


# --- inputs -----------------------------------------------------------------

def _mask(g, r, H, W, density=1.0 / 2500, rmin=4, rmax=12):
    """Noise in [20, 60] plus Gaussian blobs (sigma = radius / 2, peak 120..230),
    in 1/256 gray levels; g draws on the GPU, r (NumPy) the blobs' numbers."""
    dev = "cuda"
    acc = 256 * torch.randint(20, 61, (H, W), generator=g, device=dev, dtype=torch.int32)
    flat = acc.view(-1)
    n = int(round(density * H * W))
    radii = r.randint(rmin, rmax + 1, size=n)
    for rad in range(rmin, rmax + 1):
        k = int((radii == rad).sum())
        if not k:
            continue
        cy = torch.from_numpy(r.randint(0, H, size=(k, 1))).to(dev)
        cx = torch.from_numpy(r.randint(0, W, size=(k, 1))).to(dev)
        peak = torch.from_numpy(r.randint(120, 231, size=(k, 1))).to(dev)
        dy, dx = (a.reshape(-1) for a in np.mgrid[-rad:rad + 1, -rad:rad + 1])
        inside = dy * dy + dx * dx <= rad * rad
        dy, dx = dy[inside], dx[inside]
        prof = np.floor(65536.0 * np.exp(-2.0 * (dy * dy + dx * dx) / float(rad * rad)) + 0.5).astype(np.int64)
        y = cy + torch.from_numpy(dy).to(dev)
        x = cx + torch.from_numpy(dx).to(dev)
        v = (peak * torch.from_numpy(prof).to(dev) + 128) >> 8
        ok = (y >= 0) & (y < H) & (x >= 0) & (x < W)
        at = torch.where(ok, y * W + x, torch.zeros_like(y))
        flat.scatter_add_(0, at.reshape(-1), torch.where(ok, v, torch.zeros_like(v)).reshape(-1).to(torch.int32))
    return ((acc + 128) >> 8).clamp_(max=255).to(torch.uint8)


def _marker(I, marker):
    if marker == "hdome":
        return torch.where(I > 10, I - 10, torch.zeros_like(I))
    J = torch.zeros_like(I)
    J[0], J[-1], J[:, 0], J[:, -1] = I[0], I[-1], I[:, 0], I[:, -1]
    return J


def _pair(g, r, H, W, op, marker, **blobs):
    I = _mask(g, r, H, W, **blobs)
    J = torch.zeros_like(I) if marker == "none" else _marker(I, marker)
    return (255 - I, 255 - J) if op == "erode" else (I, J)


def _sizes(case, r):
    q = case["step"]
    lo, hi = -(-case["lo"] // q), case["hi"] // q
    return [(q * int(r.randint(lo, hi + 1)), q * int(r.randint(lo, hi + 1))) for _ in range(case["tiles"])]


def _case_sizes(case):
    """A batch's tile sizes belong to the case, so that every seed has the same work."""
    return _sizes(case, np.random.RandomState(case["tiles"] * 1009 + case["hi"]))


def _rngs(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed)), np.random.RandomState(int(seed) % (1 << 32))


def _train_data(case, seed):
    r = np.random.RandomState(int(seed) % (1 << 32))
    X = r.uniform(0, 1, size=(case["samples"], NFEAT)).astype(np.float32)
    T = np.stack([X[:, :5].sum(1) - 2.5, 2 * X[:, 5] - X[:, 6]], axis=1) + 0.05 * r.normal(size=(case["samples"], 2))
    parts = []
    for o, i in ((HIDDEN, NFEAT), (HIDDEN, HIDDEN), (NOUT, HIDDEN)):
        b = math.sqrt(6.0 / i)
        parts += [r.uniform(-b, b, size=o * i), np.zeros(o)]
    return np.concatenate(parts).astype(np.float32), X, T.astype(np.float32)


LR = 1e-3


def prepare(case, seed):
    g, r = _rngs(seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind == "tile":
        s["I"], s["J0"] = _pair(g, r, case["H"], case["W"], case["op"], case["marker"])
        s["J"] = torch.empty_like(s["I"])
    elif kind == "batch":
        sizes = _case_sizes(case)
        off, n = [], 0
        for H, W in sizes:
            off.append(n)
            n += -(-H * W // 512) * 512          # tiles 512-byte aligned, as separate tensors would be
        s["J0"] = torch.zeros(n, dtype=torch.uint8, device="cuda")
        s["J"] = torch.zeros_like(s["J0"])
        s["pairs"] = []
        for (H, W), o in zip(sizes, off):
            marker = case["marker"] if case["marker"] != "both" else ("hdome", "border")[r.randint(2)]
            I, J = _pair(g, r, H, W, case["op"], marker, density=r.uniform(0, 1e-3), rmin=3, rmax=20)
            s["J0"][o:o + H * W].view(H, W).copy_(J)
            s["pairs"].append((I, s["J"][o:o + H * W].view(H, W)))
        flags = rc.RECON_FLAG_SYNC | (rc.RECON_FLAG_LEARNED if case["learned"] else 0)
        s["ctx"] = rc.context_for("cuda", flags=flags)
        if case["learned"]:
            cost_model.install(s["ctx"])
    elif kind == "host":
        s["I"] = [_mask(g, r, H, W, density=r.uniform(0, 1e-3), rmin=3, rmax=20).cpu().pin_memory()
                  for H, W in _case_sizes(case)]
        s["out"] = [torch.zeros_like(I).pin_memory() for I in s["I"]]
        s["ctx"] = rc.context_for("cuda")
        s["tiles"] = [(I.data_ptr(), o.data_ptr(), I.shape[0], I.shape[1], I.shape[1], case["conn"], OPS[case["op"]])
                      for I, o in zip(s["I"], s["out"])]
    elif kind == "dt":
        I = _mask(g, r, case["H"], case["W"])
        s["B"] = ((I >= 100) if case["mask"] == "objects" else (I < 100)).to(torch.uint8)
        s["d2"] = torch.empty((case["H"], case["W"]), dtype=torch.int32, device="cuda")
        s["ctx"] = rc.context_for("cuda")
    else:
        theta0, X, T = _train_data(case, seed)
        s["theta0"], s["X"], s["T"] = (torch.from_numpy(a).cuda() for a in (theta0, X, T))
        s["theta"] = torch.empty_like(s["theta0"])
        s["ctx"] = rc.context_for("cuda")
    return s


# --- one pass ---------------------------------------------------------------

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "tile":
        if case["op"] != "fill_holes":
            s["J"].copy_(s["J0"])
        return rc.run(s["I"], s["J"], case["conn"], OPS[case["op"]])
    if kind == "batch":
        if case["op"] != "fill_holes":
            s["J"].copy_(s["J0"])
        rc.batch(s["pairs"], case["conn"], OPS[case["op"]], ctx=s["ctx"])
        return s["J"]
    if kind == "host":
        rc.check(rc.recon_batch_host(s["ctx"], s["tiles"]), "recon_batch_host")
        return s["out"]
    if kind == "dt":
        rc.check(rc.recon_dt(s["ctx"], s["B"].data_ptr(), s["d2"].data_ptr(), 0, case["H"], case["W"]), "recon_dt")
        return s["d2"]
    s["theta"].copy_(s["theta0"])
    st, losses = rc.recon_mlp_train(s["ctx"], s["theta"].data_ptr(), s["X"].data_ptr(), s["T"].data_ptr(),
                                    case["samples"], case["epochs"], case["batch"], LR, 1)
    rc.check(st, "recon_mlp_train")
    return [s["theta"], losses]


def work(case):
    """Bytes: masks and markers read once, results written once (1 byte a pixel
    each; 4 for a distance). Flops: 2 per weight forward, 4 backward."""
    kind = case["kind"]
    if kind == "train":
        w = HIDDEN * NFEAT + HIDDEN * HIDDEN + NOUT * HIDDEN
        n = case["samples"] * case["epochs"]
        return {"bytes": 4 * n * (NFEAT + NOUT) + 8 * NPARAMS, "flops": 6 * w * n}
    if kind == "dt":
        return {"bytes": 5 * case["H"] * case["W"], "flops": 0}
    px = case["H"] * case["W"] if kind == "tile" else sum(H * W for H, W in _case_sizes(case))
    return {"bytes": (2 if case["op"] == "fill_holes" else 3) * px, "flops": 0}


# --- what run() returns, in plain torch / NumPy -----------------------------

def _dilate_to_stability(I, J, conn):
    """R = the limit of J <- min(I, max of J over the neighbourhood)."""
    H, W = I.shape
    P = torch.zeros((H + 2, W + 2), dtype=torch.uint8, device=I.device)
    P[1:-1, 1:-1] = J
    c = P[1:-1, 1:-1]
    while True:
        before = c.clone()
        for _ in range(64):
            m = torch.maximum(c, torch.maximum(P[1:-1, :-2], P[1:-1, 2:]))
            if conn == 8:
                Q = torch.zeros_like(P)
                Q[1:-1, 1:-1] = m
                m = torch.maximum(m, torch.maximum(Q[:-2, 1:-1], Q[2:, 1:-1]))
            else:
                m = torch.maximum(m, torch.maximum(P[:-2, 1:-1], P[2:, 1:-1]))
            c.copy_(torch.minimum(m, I))
        if torch.equal(before, c):
            return c.clone()


def _mix(z):
    M = (1 << 64) - 1
    z = (z + 0x9E3779B97F4A7C15) & M
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M
    return z ^ (z >> 31)


def _train64(case, seed):
    theta, X, T = (a.astype(np.float64) for a in _train_data(case, seed))
    n, batch = case["samples"], case["batch"]
    cut = np.cumsum([HIDDEN * NFEAT, HIDDEN, HIDDEN * HIDDEN, HIDDEN, NOUT * HIDDEN])
    lr, b1, b2, eps = (float(np.float32(v)) for v in (LR, 0.9, 0.999, 1e-8))
    m, v, step, losses = np.zeros(NPARAMS), np.zeros(NPARAMS), 0, []
    for e in range(case["epochs"]):
        perm, st = list(range(n)), _mix(1 ^ _mix(e + 1))
        for i in range(n - 1, 0, -1):
            st = _mix(st)
            j = st % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        total, count = 0.0, 0
        for o in range(0, n, batch):
            x, t = X[perm[o:o + batch]], T[perm[o:o + batch]]
            W1, c1, W2, c2, W3, c3 = np.split(theta, cut)
            W1, W2, W3 = W1.reshape(HIDDEN, NFEAT), W2.reshape(HIDDEN, HIDDEN), W3.reshape(NOUT, HIDDEN)
            z1 = x @ W1.T + c1
            a1 = np.maximum(z1, 0)
            z2 = a1 @ W2.T + c2
            a2 = np.maximum(z2, 0)
            d = (a2 @ W3.T + c3 - t) / len(x)
            total, count = total + 0.5 * len(x) * float((d * d).sum()), count + 1
            d2 = (d @ W3) * (z2 > 0)
            d1 = (d2 @ W2) * (z1 > 0)
            g = np.concatenate([(d1.T @ x).ravel(), d1.sum(0), (d2.T @ a1).ravel(), d2.sum(0), (d.T @ a2).ravel(),
                                d.sum(0)])
            step += 1
            m = b1 * m + (1 - b1) * g
            v = b2 * v + (1 - b2) * g * g
            theta = theta - lr * (m / (1 - b1 ** step)) / (np.sqrt(v / (1 - b2 ** step)) + eps)
        losses.append(total / count)
    return [theta, losses]


def exact(case, seed):
    """Single tiles by repeated dilation and the training run in float64. None
    for the batches and host tiles (repeated dilation takes too long there)
    and for the distance transform (its result depends on the order in which
    sites meet)."""
    if case["kind"] == "train":
        return _train64(case, seed)
    if case["kind"] != "tile":
        return None
    g, r = _rngs(seed)
    I, J = _pair(g, r, case["H"], case["W"], case["op"], case["marker"])
    if case["op"] == "dilate":
        return _dilate_to_stability(I, J, case["conn"])
    if case["op"] == "erode":
        return 255 - _dilate_to_stability(255 - I, 255 - J, case["conn"])
    return 255 - _dilate_to_stability(255 - I, _marker(255 - I, "border"), case["conn"])
