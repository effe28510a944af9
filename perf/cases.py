"""The work that users of this library have it do, as cases that can be timed.

A case is one call of a public entry point on one image, one sequence or one
batch. Images are nested-ellipse phantoms (background and 2 to 7 tissue
classes) with noise, drawn on the GPU from the seed alone; sizes come from the
benchmark, the tests and the paper's table (about 1 KB to 16 MB), with odd and
ragged ones among them.

The listed sequence and the warm-started batch run until the stopping test
holds (``eps`` 1e-5). Every other case runs a fixed number of iterations
(``eps`` 0, ``max_iter`` k), so that the work of a pass does not depend on which
side of ``eps`` a rounded quantity falls, and two correct runs return the same
iterate. The counts are those that ``eps`` 1e-5 takes on such images, or a
little above.

Starts are the two that the entry points have: memberships U0 or centers V0.
The random (Dirichlet) U0 of the paper is used for the single images; the
batches start from the memberships of a rough earlier segmentation, and
centers are rough guesses of the class means.
"""
import math
import random

import numpy as np
import torch

from paper_1601_00072_gb300.fcm import FCM, Batch, Slice

DEVICE = "cuda"
MEANS4 = (0.0, 40.0, 110.0, 150.0)  # background, CSF, GM, WM
_handles = {}


def listed():
    return [
        # one small slice (the paper's 40 KB row): the smallest call, all latency
        {"name": "slice_200x200", "call": "run", "shape": "200x200", "C": 4, "m": 2.0, "k": 60, "start": "random", "pixels": "u8"},
        # a slice cropped to its bounding box: an odd number of pixels, so rows of U are unaligned
        {"name": "slice_199x201", "call": "run", "shape": "199x201", "C": 4, "m": 2.0, "k": 60, "start": "random", "pixels": "u8"},
        # the paper's largest image, 1 MB
        {"name": "slice_1024x1024", "call": "run", "shape": "1024x1024", "C": 4, "m": 2.0, "k": 60, "start": "random", "pixels": "u8"},
        # one whole volume: the largest single image
        {"name": "volume_256", "call": "run", "shape": "256x256x256", "C": 4, "m": 2.0, "k": 60, "start": "random", "pixels": "u8"},
        # a cropped volume after bias correction: real-valued intensities, odd size, a sharp fuzzifier, started from centers
        {"name": "volume_cropped_m1.5", "call": "run", "shape": "191x193x193", "C": 3, "m": 1.5, "k": 24, "start": "centers", "pixels": "real"},
        # a large image without memberships kept between iterations, more classes, a general fuzzifier, intensities in [0, 1]
        {"name": "ufree_2048_m2.5", "call": "recompute", "shape": "2048x2048", "C": 6, "m": 2.5, "k": 30, "start": "centers", "pixels": "unit"},
        # a volume of grey levels through its histogram
        {"name": "hist_volume_256", "call": "hist", "shape": "256x256x256", "C": 4, "m": 2.0, "k": 60, "start": "random", "pixels": "u8"},
        # three co-registered channels
        {"name": "channels3_2048", "call": "multi", "shape": "2048x2048", "D": 3, "C": 4, "m": 2.0, "k": 30, "start": "centers", "pixels": "u8"},
        # slices read from and written to pinned host memory, one after the other, each run to convergence (at most k iterations)
        {"name": "stream_8x1024", "call": "stream", "count": 8, "shape": "1024x1024", "C": 4, "m": 2.0, "k": 60, "eps": 1e-5, "start": "random", "pixels": "u8"},
        # 512 slices of uneven sizes and iteration counts in one launch
        {"name": "batch_512", "call": "batch", "count": 512, "layout": 4, "m": 2.0},
        # the same batch, each slice through its histogram
        {"name": "batch_hist_512", "call": "batch_hist", "count": 512, "layout": 4, "m": 2.0},
        # the same batch, started from the learned centers and judged against the cold start, run to eps
        {"name": "batch_warm_512", "call": "batch_warm", "count": 512, "layout": 4, "m": 2.0},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(("run", "run", "run", "run", "recompute", "hist", "multi", "stream", "batch", "batch_hist"))
    m = rng.choice((2.0, 2.0, 1.5, 3.0, 2.5))
    if call.startswith("batch"):
        return {"call": call, "count": int(_log_uniform(rng, 4, 512)), "layout": rng.randrange(1 << 20), "m": m}
    C = rng.randint(2, 8)
    case = {"call": call, "C": C, "m": m}
    hi = {"run": 1 << 24, "recompute": 1 << 24, "hist": 1 << 24, "multi": 1 << 22, "stream": 1 << 20}[call]
    n = _log_uniform(rng, 1024, hi)
    k = rng.randint(20, 60)
    # no dearer than the largest listed case (general powers cost the most)
    n = min(n, (1 << 24) * 4.0 / C * min(1.0, 30.0 / k) * (1.0 if m == 2.0 else 0.25))
    h = max(16, int(math.sqrt(n * rng.uniform(0.6, 1.0))))
    w = max(16, int(n / h))
    if call in ("recompute", "stream"):
        w += -w % 4  # these two entries need n % 4 == 0
    case.update(shape="%dx%d" % (h, w), k=k, start="centers", pixels="u8" if call == "hist" else rng.choice(("u8", "u8", "real", "unit")))
    if call == "stream":
        case["count"] = rng.randint(2, 6)
        case["start"] = "rough"
    elif rng.random() < 0.5:
        case["start"] = "rough"
    if call == "multi":
        case["D"] = rng.randint(1, 4)
    return case


# ---- inputs ----------------------------------------------------------------

def _gen(*key):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(np.random.SeedSequence([int(v) for v in key]).generate_state(1, np.uint64)[0] >> 1))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEVICE)


def _shape(case):
    return tuple(int(v) for v in case["shape"].split("x"))


def _means(C, r):
    """Class means of a phantom: the four tissues, or C levels in [0, 235] at least 20 apart."""
    if C == 4 and r is None:
        return MEANS4
    r = r or random.Random(C)
    free = 235.0 - 20.0 * (C - 1)
    cuts = sorted(r.uniform(0.0, free) for _ in range(C))
    return tuple(c + 20.0 * j for j, c in enumerate(cuts))


def _labels(shape, C, r):
    """Nested ellipses (ellipsoids): the label map of C classes."""
    axes = [torch.linspace(-1.0, 1.0, s, device=DEVICE) for s in shape]
    grid = torch.meshgrid(*axes, indexing="ij")
    lab = torch.zeros(shape, dtype=torch.long, device=DEVICE)
    c = [r.uniform(-0.05, 0.05) for _ in shape]
    a = [r.uniform(0.85, 0.97) for _ in shape]
    for level in range(1, C):
        q = sum(((g - ci) / ai) ** 2 for g, ci, ai in zip(grid, c, a))
        lab[q <= 1.0] = level
        c = [ci + r.uniform(-0.05, 0.05) * ai for ci, ai in zip(c, a)]
        a = [ai * r.uniform(0.78, 0.9) for ai in a]
    return lab


def _image(shape, C, sigma, pixels, g, r, means=None):
    """One image, flat: grey levels as floats ("u8"), real-valued intensities
    of the same range ("real"), or those scaled to [0, 1] ("unit")."""
    mu = torch.tensor(means or _means(C, None), device=DEVICE)
    v = mu[_labels(shape, C, r)]
    if len(shape) == 3 and pixels == "u8":
        # a smooth bias field and Rician noise
        for d, s in enumerate(shape):
            t = torch.linspace(-1.0, 1.0, s, device=DEVICE)
            v *= (1.0 + r.uniform(-0.06, 0.06) * t * t).view([-1 if i == d else 1 for i in range(3)])
        v += sigma * torch.randn(shape, generator=g, device=DEVICE)
        v = torch.hypot(v, sigma * torch.randn(shape, generator=g, device=DEVICE))
    else:
        v = v + sigma * torch.randn(shape, generator=g, device=DEVICE)
    v.clamp_(0.0, 255.0)
    if pixels == "u8":
        v.round_()
    elif pixels == "unit":
        v /= 255.0
    return v.reshape(-1)


def _guess(means, r, scale):
    """Rough centers: the class means, each off by a few grey levels."""
    return [scale * min(254.3, max(0.7, mu + r.uniform(-8.0, 8.0))) for mu in means]


def _random_u0(C, n, g):
    u = (-torch.log(1.0 - _rand(g, C, n))).clamp_(min=1e-7)
    return (u / u.sum(0)).contiguous()


def _rough_u0(x, V0, g):
    """Memberships of a rough earlier segmentation: soft assignments to rough centers, with noise."""
    V = torch.tensor(V0, device=DEVICE, dtype=torch.float32)[:, None]
    w = 1.0 / (1.0 + ((x[None] - V) / (0.1 * (max(V0) - min(V0)) + 1e-6)) ** 2)
    w = w * (0.5 + _rand(g, *w.shape))
    return (w / w.sum(0)).contiguous()


def _layout(case):
    """Sizes, cluster counts and iteration budgets of a batch: sides log-uniform
    in 64..512, C in 3..5, budgets spread as convergence spreads them (mean
    about 33, at most 167)."""
    r = random.Random(case["layout"])
    out, x_at, u_at, v_at = [], 0, 0, 0
    for _ in range(case["count"]):
        h, w, C = int(_log_uniform(r, 64, 512.99)), int(_log_uniform(r, 64, 512.99)), r.choice((3, 4, 5))
        k = min(167, max(12, round(math.exp(r.gauss(math.log(29.0), 0.5)))))
        n = h * w
        out.append({"shape": (h, w), "n": n, "C": C, "k": k, "x": x_at, "u": u_at, "v": v_at})
        x_at += n + -n % 4  # every slice on a 16-byte boundary
        u_at += C * n + -(C * n) % 4
        v_at += C
    return out, x_at, u_at, v_at


def _batch_inputs(case, seed):
    layout, nx, nu, nv = _layout(case)
    r = random.Random(seed * 1000003 + case["layout"])
    g = _gen(7, seed, case["layout"])
    x, U0 = torch.zeros(nx, device=DEVICE), torch.zeros(nu, device=DEVICE)
    for s in layout:
        means = _means(s["C"], r)
        img = _image(s["shape"], s["C"], r.uniform(4.0, 7.0), "u8", g, r, means)
        x[s["x"]:s["x"] + s["n"]] = img
        U0[s["u"]:s["u"] + s["C"] * s["n"]] = _rough_u0(img, _guess(means, r, 1.0), g).reshape(-1)
    return layout, x, U0, nu, nv


def _inputs(case, seed):
    """x [n] or [D, n], then (U0, None) or (None, V0)."""
    shape, C, D = _shape(case), case["C"], case.get("D", 1)
    r = random.Random(seed * 1000003 + 17 * C + D)
    g = _gen(5, seed, C, D)
    scale = 1.0 / 255.0 if case["pixels"] == "unit" else 1.0
    sigma = 8.0 if C <= 4 else 4.0
    orders = [list(range(C))] + [r.sample(range(C), C) for _ in range(1, D)]
    base = _means(C, None)
    form = r.random()  # the channels of one image share their layout
    xs, V0 = [], []
    for order in orders:
        means = tuple(base[j] for j in order)
        xs.append(_image(shape, C, sigma, case["pixels"], g, random.Random(form), means))
        V0.append(_guess(means, r, scale))
    x = torch.stack(xs) if case["call"] == "multi" else xs[0]
    if case["start"] == "random":
        return x, _random_u0(C, x.shape[-1], g), None
    if case["start"] == "rough":
        return x, _rough_u0(xs[0], V0[0], g), None
    v = torch.tensor(V0, dtype=torch.float32, device=DEVICE).T.contiguous()  # [C, D]
    return x, None, v if case["call"] == "multi" else v.reshape(-1)


# ---- the cases ---------------------------------------------------------------

def _fcm():
    """The handle that a program keeps (with the shipped warm-start weights)."""
    if "fcm" not in _handles:
        from paper_1601_00072_gb300 import warmstart
        h = FCM()
        h.model_load(str(warmstart.MODEL_PATH))
        _handles["fcm"] = h
    return _handles["fcm"]


def prepare(case, seed):
    h = _fcm()
    if case["call"].startswith("batch"):
        layout, x, U0, nu, nv = _batch_inputs(case, seed)
        U, V = torch.zeros(nu, device=DEVICE), torch.zeros(nv, device=DEVICE)
        warm = case["call"] == "batch_warm"
        slices = [Slice(x=x[s["x"]:s["x"] + s["n"]], C=s["C"], m=case["m"], eps=1e-5 if warm else 0.0,
                        max_iter=300 if warm else s["k"],
                        U0=U0[s["u"]:s["u"] + s["C"] * s["n"]].view(s["C"], s["n"]),
                        U=U[s["u"]:s["u"] + s["C"] * s["n"]].view(s["C"], s["n"]), V=V[s["v"]:s["v"] + s["C"]])
                  for s in layout]
        return {"case": case, "fcm": h, "batch": Batch(slices), "U": U, "V": V}
    if case["call"] == "stream":
        xs, u0s, us = [], [], []
        for i in range(case["count"]):
            x, U0, _ = _inputs(case, seed * 64 + i)
            xs.append(x.cpu().pin_memory())
            u0s.append(U0.cpu().pin_memory())
            us.append(torch.empty_like(u0s[-1]).pin_memory())
        return {"case": case, "fcm": h, "xs": xs, "U0s": u0s, "Us": us, "V": np.empty((len(xs), case["C"]), np.float32)}
    x, U0, V0 = _inputs(case, seed)
    C, n, D = case["C"], x.shape[-1], case.get("D", 1)
    return {"case": case, "fcm": h, "x": x, "U0": U0, "V0": V0, "U": torch.empty((C, n), device=DEVICE),
            "V": torch.empty((C, D) if case["call"] == "multi" else (C,), device=DEVICE)}


def run(state):
    case, h = state["case"], state["fcm"]
    call = case["call"]
    if call.startswith("batch"):
        b = state["batch"]
        if call == "batch":
            h.run_batched(b)
        elif call == "batch_hist":
            h.run_batched_hist(b)
        else:
            h.run_batched_warm(b)
        return {"U": state["U"], "V": state["V"], "J": b.arr["J"].astype(np.float32)}
    if call == "stream":
        rs = h.run_stream(state["xs"], case["C"], case["m"], case.get("eps", 0.0), case["k"], U0s=state["U0s"], Us=state["Us"], V=state["V"])
        return {"U": state["Us"], "V": state["V"], "J": np.array([r.J for r in rs], np.float32)}
    kw = {"U0": state["U0"]} if state["U0"] is not None else {"V0": state["V0"]}
    f = {"hist": h.run_hist, "multi": h.run_multi}.get(call, h.run)
    if call == "recompute":
        kw["recompute"] = True
    r = f(state["x"], case["C"], case["m"], 0.0, case["k"], U=state["U"], V=state["V"], **kw)
    return {"U": r.U, "V": r.V, "J": r.J, "iters": r.iters}


def work(case):
    """Inputs read once (x, and U0 when the start is from memberships), U
    written once; per pixel and iteration the arithmetic of Eq. 4 and Eq. 3
    (about 9 operations per cluster and channel pair), or for the histogram
    calls that of the 256 bins."""
    if case["call"].startswith("batch"):
        layout = _layout(case)[0]
        nbytes = sum(4 * s["n"] * (1 + 2 * s["C"]) for s in layout)
        hist = case["call"] == "batch_hist"
        return {"bytes": nbytes, "flops": sum((256 if hist else s["n"]) * s["k"] * 9 * s["C"] + s["n"] * 3 * s["C"] for s in layout)}
    n, C, D, count = math.prod(_shape(case)), case["C"], case.get("D", 1), case.get("count", 1)
    rows = D + C * (1 if case["start"] == "centers" else 2)
    px = 256 if case["call"] == "hist" else n
    return {"bytes": 4 * n * rows * count, "flops": count * (px * case["k"] * C * (4 * D + 5) + n * 3 * C)}


# ---- the same in 64 bits -------------------------------------------------------

def _memberships64(x, V, m):
    """Eq. 4 for x [D, n] and V [C, D]: (U, sum over pixels of the J term's parts d2)."""
    d2 = ((x[None] - V[:, :, None]) ** 2).sum(1)
    if bool((d2 == 0).any()):
        z = (d2 == 0).double()
        w = torch.where(z.sum(0) > 0, z, (d2.min(0).values / d2.clamp(min=1e-300)) ** (1.0 / (m - 1.0)))
    else:
        w = d2.min(0).values / d2
        if m != 2.0:
            w = w ** (1.0 / (m - 1.0))
    return w / w.sum(0), d2


def _powm(U, m):
    return U * U if m == 2.0 else U ** m


def _fcm64(x, C, m, k, U0=None, V0=None):
    """Algorithm 1, k iterations, in 64 bits: x [D, n]."""
    x = x.double()
    U = U0.double() if U0 is not None else _memberships64(x, V0.double(), m)[0]
    for _ in range(k):
        um = _powm(U, m)
        V = (um @ x.T) / um.sum(1, keepdim=True)
        U, d2 = _memberships64(x, V, m)
    return U, V, float((_powm(U, m) * d2).sum())


def exact(case, seed):
    if case["call"] == "batch_warm" or case.get("eps"):
        # the stopping test is a threshold on a rounded quantity: a run that
        # stops one iteration to either side of it is as right
        return None
    if case["call"].startswith("batch"):
        layout, x, U0, nu, nv = _batch_inputs(case, seed)
        U, V, J = torch.zeros(nu, dtype=torch.float64, device=DEVICE), torch.zeros(nv, dtype=torch.float64, device=DEVICE), []
        for s in layout:
            at = slice(s["u"], s["u"] + s["C"] * s["n"])
            u, v, j = _fcm64(x[None, s["x"]:s["x"] + s["n"]], s["C"], case["m"], s["k"], U0=U0[at].view(s["C"], s["n"]))
            U[at] = u.reshape(-1)
            V[s["v"]:s["v"] + s["C"]] = v[:, 0]
            J.append(j)
        return {"U": U, "V": V, "J": np.array(J)}
    if case["call"] == "stream":
        got = []
        for i in range(case["count"]):
            x, U0, _ = _inputs(case, seed * 64 + i)
            got.append(_fcm64(x[None], case["C"], case["m"], case["k"], U0=U0))
        return {"U": [u for u, _, _ in got], "V": np.stack([v[:, 0].cpu().numpy() for _, v, _ in got]), "J": np.array([j for _, _, j in got])}
    x, U0, V0 = _inputs(case, seed)
    multi = case["call"] == "multi"
    U, V, J = _fcm64(x if multi else x[None], case["C"], case["m"], case["k"], U0=U0,
                     V0=None if V0 is None else V0 if multi else V0[:, None])
    return {"U": U, "V": V if multi else V[:, 0], "J": J, "iters": case["k"]}
