"""The work that users have this library do, as timed cases.

A case is one call (or one round of calls) through the public Python entry points on windows of synthetic ultrasound
frames: a single plan solve, a batch of windows in one launch, a round of requests to the server, or the frame
pre-filter.  Window contents follow the recipe of paper_2506_10257_gb300/synth.py (rank-2 Rayleigh speckle with a slow
gain drift, static and moving Gaussian blobs, N(0, 0.1^2) noise, a random phase per pixel and blob in IQ windows), drawn
here on the GPU.  Windows are written as "ny x nx x frames" texts joined by ";".

BF16X3 is left out: at every size it is both slower than another precision and less accurate, and warm starts are left
out because they are off unless asked for and end at another point than a cold solve.
"""
import math
import random

import numpy as np
import torch

from paper_2506_10257_gb300 import rpca

THETA = 2.5  # bound-bubble threshold on the temporal mean of |L|: half the level of a blob on top of the speckle
ITERS = 32   # iterations of a solve at the default schedule and tolerance (they vary by one or two with the window)


def listed():
    uneven = np.random.Generator(np.random.PCG64(3000))  # the uneven workload of the benchmark: its first 16 windows
    grids = ("64x64", "128x256", "256x256", "512x512")
    uneven = ";".join("%sx%d" % (grids[int(uneven.integers(0, 4))], int(uneven.integers(10, 201))) for _ in range(16))
    return [
        # the smallest window in use, with the bound-bubble mask: latency of the eigen-steps and launches
        {"name": "plan 64x64x20 mask", "kind": "plan", "windows": "64x64x20", "precision": "fp32", "iq": False, "mask": True},
        # the paper's execution-time image at its shortest window
        {"name": "plan 338x260x20", "kind": "plan", "windows": "338x260x20", "precision": "fp32", "iq": False, "mask": False},
        # an odd crop of an image (a region of interest) and a frame count that no tile divides
        {"name": "plan 333x257x29", "kind": "plan", "windows": "333x257x29", "precision": "fp32", "iq": False, "mask": False},
        # the headline window, solved alone
        {"name": "plan 512x512x20", "kind": "plan", "windows": "512x512x20", "precision": "fp32", "iq": False, "mask": False},
        # a longer window at full size: the tiled path
        {"name": "plan 512x512x50", "kind": "plan", "windows": "512x512x50", "precision": "fp32", "iq": False, "mask": False},
        # the longest window at full size in the reduced precision that is the faster one there
        {"name": "plan 512x512x100 tf32x3", "kind": "plan", "windows": "512x512x100", "precision": "tf32x3", "iq": False, "mask": False},
        # the paper's in vivo reference: its execution-time image over 132 frames
        {"name": "plan 338x260x132", "kind": "plan", "windows": "338x260x132", "precision": "fp32", "iq": False, "mask": False},
        # beamformed IQ data (complex64)
        {"name": "plan 256x256x50 iq", "kind": "plan", "windows": "256x256x50", "precision": "fp32", "iq": True, "mask": False},
        # throughput: many headline windows in one launch (offline processing of a recording)
        {"name": "batch 16x 512x512x20", "kind": "batch", "windows": ";".join(["512x512x20"] * 16), "precision": "fp32", "iq": False, "mask": False},
        # windows of several studies in one launch
        {"name": "batch uneven 16", "kind": "batch", "windows": uneven, "precision": "fp32", "iq": False, "mask": False},
        # eight probes' newest sliding windows, queued at once and waited for
        {"name": "serve 8 probes", "kind": "serve", "windows": "128x128x20;256x256x20;256x512x20;384x384x20;512x512x20;512x640x20;640x512x20;768x512x20",
         "precision": "fp32", "iq": False, "mask": False},
        # the frame exclusion and moving average that the paper's in vivo reference runs before its solve
        {"name": "prefilter 338x260x132", "kind": "prefilter", "windows": "338x260x132", "precision": "fp32", "iq": False, "mask": False},
    ]


def _size(rng, lo, hi):
    """A whole number spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    iq, precision, mask = False, "fp32", False
    u = rng.random()
    if u < 0.55:
        kind = "plan"
        ny, nx = _size(rng, 48, 512), _size(rng, 48, 512)
        iq = rng.random() < 0.2
        top = min(56 if iq else 140, ny * nx // 24)  # windows are tall: many more pixels than frames
        T = _size(rng, 5, top)
        if not iq and 33 <= T <= 128 and rng.random() < 0.4:
            precision = "tf32x3"
        mask = not iq and ny * nx <= 16384 and rng.random() < 0.5
        windows = "%dx%dx%d" % (ny, nx, T)
    elif u < 0.75:
        kind = "batch"
        n, top = rng.randint(3, 12), rng.choice((20, 32, 90))
        windows = ";".join("%dx%dx%d" % (_size(rng, 48, 256), _size(rng, 48, 256), _size(rng, 5, top)) for _ in range(n))
    elif u < 0.88:
        kind = "serve"
        T = _size(rng, 10, 32)
        windows = ";".join("%dx%dx%d" % (_size(rng, 64, 512), _size(rng, 64, 512), T) for _ in range(rng.randint(2, 8)))
    else:
        kind = "prefilter"
        windows = "%dx%dx%d" % (_size(rng, 64, 512), _size(rng, 64, 512), _size(rng, 24, 140))
    return {"kind": kind, "windows": windows, "precision": precision, "iq": iq, "mask": mask}


def _shapes(case):
    return [tuple(int(v) for v in w.split("x")) for w in case["windows"].split(";")]


# ---- inputs ----

def _window(ny, nx, T, seed, iq=False, speed=(0.5, 5.0), bad_frames=0):
    """One window of frames, (T, ny * nx) float32 or complex64 on the GPU; speed of the free blobs in pixels a frame."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    h = random.Random(seed)
    m = ny * nx
    n_bound = max(4, round(15 * (m / 4096) ** 0.79))  # 15 on 64x64, 400 on 512x512 pixels
    n_free = 2 * n_bound

    def uniform(lo, hi, *shape):
        return torch.rand(*shape, generator=g, device=dev) * (hi - lo) + lo

    def rayleigh(n):
        return torch.sqrt(-2 * torch.log1p(-torch.rand(n, generator=g, device=dev).clamp(max=1 - 1e-7)))

    ys, xs = torch.arange(ny, device=dev, dtype=torch.float32), torch.arange(nx, device=dev, dtype=torch.float32)

    def blobs(cy, cx, a):  # sum of the Gaussian blobs (sigma 1.5 pixels)
        gy = torch.exp((ys[None, :] - cy[:, None]) ** 2 / -4.5) * a[:, None]
        gx = torch.exp((xs[None, :] - cx[:, None]) ** 2 / -4.5)
        return gy.t() @ gx

    def image(cy, cx, a, ph):  # its real part, and in IQ windows its imaginary part
        return torch.stack([blobs(cy, cx, a * torch.cos(ph)), blobs(cy, cx, a * torch.sin(ph))]) if iq else blobs(cy, cx, a)[None]

    t = torch.linspace(0, 1, T, device=dev) if T > 1 else torch.zeros(1, device=dev)
    bg = rayleigh(m)[None] * (1 + 0.02 * t[:, None]) + 0.01 * rayleigh(m)[None] * torch.cos(math.pi * t)[:, None]
    if iq:
        ph = uniform(-math.pi, math.pi, m)
        frames = torch.stack([bg * torch.cos(ph), bg * torch.sin(ph)])
    else:
        frames = bg[None]
    parts = frames.shape[0]
    ph = uniform(-math.pi, math.pi, n_bound) if iq else None
    frames = frames + image(uniform(0, ny, n_bound), uniform(0, nx, n_bound), uniform(3, 6, n_bound), ph).reshape(parts, 1, m)
    cy, cx, a = uniform(0, ny, n_free), uniform(0, nx, n_free), uniform(3, 6, n_free)
    v, th = uniform(*speed, n_free), uniform(-math.pi, math.pi, n_free)
    ph = uniform(-math.pi, math.pi, n_free) if iq else None
    for k in range(T):
        py, px = cy + v * torch.sin(th) * k, cx + v * torch.cos(th) * k
        inside = (py >= 0) & (py < ny) & (px >= 0) & (px < nx)  # straight tracks: one that left does not come back
        frames[:, k] += image(py, px, a * inside, ph).reshape(parts, m)
    frames += 0.1 * torch.randn(frames.shape, generator=g, device=dev)
    for k in sorted(h.sample(range((T - 2) // 3), bad_frames)):  # frames of another place (the probe or the animal moved),
        frames[:, 3 * k + 2] = rayleigh(m)  # two good ones or more between them and at the ends: each is excluded alone
    return torch.complex(frames[0], frames[1]) if iq else frames[0].contiguous()


def _inputs(case, seed):
    # the pre-filter's frames are those of a slow reference acquisition (neighbours correlate well above its limit of
    # 0.8) with one frame in twenty lost to motion
    more = (lambda T: {"speed": (0.1, 1.0), "bad_frames": max(1, T // 20)}) if case["kind"] == "prefilter" else lambda T: {}
    return [_window(ny, nx, T, 1000 * seed + i, case["iq"], **more(T)) for i, (ny, nx, T) in enumerate(_shapes(case))]


def prepare(case, seed):
    precision = {"fp32": rpca.PREC_FP32, "tf32x3": rpca.PREC_TF32X3}[case["precision"]]
    X = _inputs(case, seed)
    shapes = [(ny * nx, T) for ny, nx, T in _shapes(case)]
    kw = {"precision": precision}
    if case["iq"]:
        kw["dtype"] = rpca.C64
    state = {"case": case, "X": X, "L": [torch.empty_like(x) for x in X], "S": [torch.empty_like(x) for x in X]}
    if case["kind"] == "plan":
        state["plan"] = rpca.Plan(*shapes[0], **kw)
        state["mask"] = torch.empty(shapes[0][0], dtype=torch.uint8, device="cuda") if case["mask"] else None
    elif case["kind"] == "batch":
        state["batch"] = rpca.Batch(shapes, **kw)
    elif case["kind"] == "serve":
        state["server"] = rpca.Server(max_slots=8)
        state["kw"] = kw
    else:
        state["out"] = rpca.prefilter_buffers(X[0])
        del state["L"], state["S"]
    return state


def run(state):
    kind, X = state["case"]["kind"], state["X"]
    if kind == "plan":
        L, S, _ = state["plan"].solve(X[0], L=state["L"][0], S=state["S"][0], mask=state["mask"], theta=THETA)
        return {"L": L, "S": S} if state["mask"] is None else {"L": L, "S": S, "mask": state["mask"]}
    if kind == "batch":
        Ls, Ss, _ = state["batch"].solve(X, Ls=state["L"], Ss=state["S"])
        return {"L": Ls, "S": Ss}
    if kind == "serve":
        server = state["server"]
        ids = [server.submit(x, key=i, L=state["L"][i], S=state["S"][i], **state["kw"]) for i, x in enumerate(X)]
        for r in ids:
            server.wait(r)
        return {"L": state["L"], "S": state["S"]}
    Y, kept, corr = rpca.prefilter(X[0], out=state["out"])
    return {"Y": Y, "kept": kept, "corr": corr}


def work(case):
    """X read once and L, S (the mask) written once; the three contractions of every iteration (Z Wbar, the Gram of the
    next Z and its eigenvectors' product Z' V) and a dozen operations an element.  The pre-filter: the frames read
    once and the averages written once, three moments and the average of every element."""
    nbytes = flops = 0
    for ny, nx, T in _shapes(case):
        m, esz = ny * nx, 8 if case["iq"] else 4
        if case["kind"] == "prefilter":
            nbytes += (2 * T - 19) * m * 4 if T > 19 else T * m * 4
            flops += 10 * T * m
        else:
            nbytes += 3 * m * T * esz + (m if case["mask"] else 0)
            flops += ITERS * m * T * (5 * T * (4 if case["iq"] else 1) + 12 * (2 if case["iq"] else 1))
    return {"bytes": nbytes, "flops": flops}


# ---- the same in 64 bits ----

def _pcp(X):
    """Principal component pursuit by the inexact augmented-Lagrangian iteration in 64 bits, X (frames, pixels): L, S."""
    A = X.t().to(torch.complex128 if X.is_complex() else torch.float64)
    m, T = A.shape
    lam = 1 / math.sqrt(max(m, T))
    norm = float(torch.linalg.norm(A))

    def gram_vectors(Z):
        """Eigenvalues and vectors of Z^H Z; formed twice, the second time in the first's basis, for the small ones."""
        _, V = torch.linalg.eigh(Z.mH @ Z)
        U = Z @ V
        w, Q = torch.linalg.eigh(U.mH @ U)
        return w.clamp(min=0), V @ Q

    w, V = gram_vectors(A)
    mu = 1.25 / math.sqrt(float(w[-1]))
    mu_max = 1e7 * mu
    S, Y = torch.zeros_like(A), torch.zeros_like(A)
    for k in range(500):
        Z = A - S + Y / mu
        if k:
            w, V = gram_vectors(Z)
        sig = w.sqrt()
        keep = sig > 1 / mu
        g = torch.where(keep, 1 - 1 / (mu * torch.where(keep, sig, torch.ones_like(sig))), torch.zeros_like(sig))
        L = (Z @ V) @ (g[:, None] * V.mH)
        del Z
        R = A - L + Y / mu
        gamma = lam / mu
        mag = R.abs()
        S = R * ((mag - gamma).clamp(min=0) / mag.clamp(min=1e-300))
        del R, mag
        E = A - L - S
        Y = Y + mu * E
        if float(torch.linalg.norm(E)) <= 1e-7 * norm:
            break
        del E
        mu = min(1.5 * mu, mu_max)
    return L.t().contiguous(), S.t().contiguous()


def exact(case, seed):
    X = _inputs(case, seed)
    if case["kind"] != "prefilter":
        LS = [_pcp(x) for x in X]
        Ls, Ss = [a for a, _ in LS], [b for _, b in LS]
        if case["kind"] == "plan":
            return {"L": Ls[0], "S": Ss[0], "mask": None}
        return {"L": Ls, "S": Ss}
    F = X[0].double()
    D = F - F.mean(1, keepdim=True)
    s = (D * D).sum(1)
    corr = (D[1:] * D[:-1]).sum(1) / torch.sqrt(s[1:] * s[:-1])
    ok = corr >= 0.8
    no = torch.zeros(1, dtype=torch.bool, device=ok.device)
    kept = torch.nonzero(torch.cat([no, ok]) | torch.cat([ok, no])).flatten()
    F = F[kept]
    n = max(len(kept) - 19, 0)
    Y = torch.stack([F[j:j + 20].mean(0) for j in range(n)]) if n else F[:0]
    return {"Y": Y, "kept": None, "corr": corr}
