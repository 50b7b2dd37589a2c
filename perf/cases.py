"""The work that users of this package have it do, as cases for timing.

A case is one call (or one short sequence of calls) of the public entry
points on synthetic event windows of a camera descending onto a plane: scene
points move radially about the focus of expansion, x(t) = FOE + (x0 - FOE) /
(1 - D t), each giving about 35 events at random times, plus uniform noise.

Kinds of case (`kind`):
    solve     one exact search of one window (Context.solve)
    batch     many windows of uneven size in one call (Context.solve_batch)
    stream    a continuous stream cut into overlapping windows (Context.stream_solve)
    serve     windows handed to the continuous-batching server (Server)
    contrast  the contrast curve over a list of hypotheses (Context.contrast,
              dd_contrast_noalloc)
    bound     upper bounds over a list of intervals (Context.bound)
    fast      the fast mode: coordinates resized, events resampled, then solved
    train     forward and backward of the warm-start network on a batch

Every output but the network's gradient is decided by binary32 operations in a
stated order followed by exact integer sums, so another correct implementation
returns the same bits.
"""
import math
import os

import numpy as np
import torch

import paper_2209_13168_gb300 as dd

PARAMS = (-1.0, 1.0, 1e-4, 0.0)      # D range, leaf width and stopping gap of the benchmark's searches
MODEL = os.path.join(os.path.dirname(os.path.abspath(dd.__file__)), "warm_start_640x480.bin")
PER_POINT = 35                       # events per scene point


def listed():
    return [
        # The smallest search: a DAVIS346 frame with few events, where the
        # latency of a round counts.
        {"name": "solve_346x260_4k", "kind": "solve", "W": 346, "H": 260, "n": 4000, "D": 0.2, "tau": 0.5,
         "noise": 0.25, "knobs": "tuned"},
        # The benchmark's window: one estimate from a 640x480 camera.
        {"name": "solve_640x480_100k", "kind": "solve", "W": 640, "H": 480, "n": 100000, "D": 0.35, "tau": 0.3,
         "noise": 0.3, "knobs": "tuned"},
        # A first-time user: no knobs (Algorithm 1 as printed, one interval a
        # round), events in numpy arrays, an odd number of them, FOE off centre.
        {"name": "solve_default_30k_host", "kind": "solve", "W": 640, "H": 480, "n": 30011, "D": 0.5, "tau": 0.2,
         "noise": 0.2, "knobs": "default", "host": True, "foe_x": 301.3, "foe_y": 262.7},
        # The last seconds of a descent seen by a 1280x720 camera, from host arrays.
        {"name": "solve_1280x720_600k_host", "kind": "solve", "W": 1280, "H": 720, "n": 600000, "D": 0.62,
         "tau": 0.2, "noise": 0.15, "knobs": "tuned", "host": True},
        # The objective with one image per polarity.
        {"name": "solve_polarity_77k", "kind": "solve", "W": 640, "H": 480, "n": 77773, "D": 0.3, "tau": 0.25,
         "noise": 0.25, "knobs": "tuned", "polarity": True},
        # Offline processing: 256 uneven windows in one call, warm-started by the shipped model.
        {"name": "batch_256_warm", "kind": "batch", "W": 640, "H": 480, "windows": 256, "n_lo": 5000,
         "n_hi": 200000, "warm": True},
        # Stream-wise estimation: 0.2 s windows every 0.1 s of a 1280x720 descent.
        {"name": "stream_1280x720", "kind": "stream", "W": 1280, "H": 720, "windows": 96, "rate": 400000},
        # Serving: windows of a descent waiting for sixteen slots.
        {"name": "serve_1280x720", "kind": "serve", "W": 1280, "H": 720, "windows": 40, "slots": 16, "n_lo": 50000,
         "n_hi": 400000},
        # The contrast curve of one window on a grid of hypotheses.
        {"name": "contrast_640x480_129", "kind": "contrast", "W": 640, "H": 480, "n": 100000, "hyp": 129},
        # Bounds over a grid of intervals covering the search range.
        {"name": "bound_640x480_64", "kind": "bound", "W": 640, "H": 480, "n": 100000, "intervals": 64,
         "span": 2.0},
        # The fast mode: 1280x720 resized to 160x90 with a quarter of the events.
        {"name": "fast_160x90", "kind": "fast", "W": 1280, "H": 720, "W2": 160, "H2": 90, "n": 200000, "keep": 0.25},
        # One backward pass of the warm-start network's training.
        {"name": "train_256", "kind": "train", "samples": 256},
    ]


FRAMES = ((346, 260), (640, 480), (1280, 720), (160, 90), (333, 251), (511, 389))


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "solve", "batch", "stream", "serve", "contrast", "bound", "fast",
                       "train"))
    W, H = rng.choice(FRAMES)
    c = {"kind": kind, "W": W, "H": H}
    most = min(400000, W * H // 2)       # events of a window: far more per pixel and the bounds say little
    if kind == "solve":
        c["n"] = _log_int(rng, min(2000, most // 4), most)
        c["D"] = round(rng.uniform(0.05, 0.8), 4)
        c["tau"] = round(rng.uniform(0.1, 0.5), 4)
        c["noise"] = round(rng.uniform(0.1, 0.4), 3)
        c["knobs"] = "default" if rng.random() < 0.25 else "tuned"
        for option, share in (("host", 0.3), ("polarity", 0.2), ("to_start", 0.2)):
            if rng.random() < share:
                c[option] = True
        if rng.random() < 0.3:
            c["foe_x"] = round(rng.uniform(0.2, 0.8) * W, 2)
            c["foe_y"] = round(rng.uniform(0.2, 0.8) * H, 2)
    elif kind == "batch":
        c["windows"] = _log_int(rng, 2, 128)
        c["n_lo"] = _log_int(rng, 1000, 8000)
        c["n_hi"] = _log_int(rng, c["n_lo"] + 1, min(150000, max(most, 2 * c["n_lo"])))
        c["warm"] = rng.random() < 0.3
    elif kind == "stream":
        c["windows"] = _log_int(rng, 4, 64)
        c["rate"] = _log_int(rng, 20000, max(40000, min(600000, 2 * most)))
    elif kind == "serve":
        c["windows"] = _log_int(rng, 2, 40)
        c["slots"] = rng.choice((4, 8, 16))
        c["n_lo"] = _log_int(rng, 1000, 8000)
        c["n_hi"] = _log_int(rng, c["n_lo"] + 1, min(200000, max(most, 2 * c["n_lo"])))
    elif kind == "contrast":
        c["n"] = _log_int(rng, 1000, 600000)
        c["hyp"] = _log_int(rng, 1, 300)
        c["noalloc"] = rng.random() < 0.4
        if not c["noalloc"] and rng.random() < 0.3:
            c["hyp"] = _log_int(rng, 1, 8)
            c["image"] = True
    elif kind == "bound":
        c["n"] = _log_int(rng, 1000, 300000)
        c["intervals"] = _log_int(rng, 1, 128)
        c["span"] = round(math.exp(rng.uniform(math.log(0.002), math.log(2.0))), 4)
    elif kind == "fast":
        c["W"], c["H"] = rng.choice(((640, 480), (1280, 720)))
        c["W2"], c["H2"] = rng.choice(((160, 90), (320, 240), (173, 131)))
        c["n"] = _log_int(rng, 20000, 200000)
        c["keep"] = round(rng.uniform(0.1, 0.4), 3)
    else:
        c = {"kind": "train", "samples": _log_int(rng, 16, 2048)}
    return c


# ------------------------------------------------------------------- inputs

def _descent(gen, W, H, fx, fy, n, D, tau, noise, t_from=0.0):
    """(x, y, t, p) device tensors of one window, sorted by time; D is the
    divergence at t = 0 and the window covers [t_from, t_from + tau]."""
    dev = "cuda"
    n_noise = int(round(noise * n))
    points = max(1, (n - n_noise) // PER_POINT)
    pos = torch.rand(2, points, generator=gen, device=dev, dtype=torch.float64)
    pol = torch.rand(points, generator=gen, device=dev) < 0.5
    u = torch.rand(4, n, generator=gen, device=dev, dtype=torch.float64)
    t = u[0] * tau
    t, order = torch.sort(t)
    u = u[1:, order]
    who = torch.randint(points, (n,), generator=gen, device=dev)
    g = 1.0 / (1.0 - D * t)
    x = torch.floor(fx + (pos[0, who] * W - fx) * g + 0.5)
    y = torch.floor(fy + (pos[1, who] * H - fy) * g + 0.5)
    # noise, and whatever has left the frame, is uniform
    away = (u[2] * n < n_noise) | (x < 0) | (x >= W) | (y < 0) | (y >= H)
    x = torch.where(away, torch.floor(u[0] * W), x).clamp_(0, W - 1)
    y = torch.where(away, torch.floor(u[1] * H), y).clamp_(0, H - 1)
    p = torch.where(pol[who], 1, -1).to(torch.int8)
    tau32 = float(np.float32(tau))
    return x.to(torch.int16), y.to(torch.int16), (t + t_from).float().clamp_(t_from, t_from + tau32), p


def _uneven(case, seed, k):
    """(n, D, tau, noise) of window k of an uneven set of windows."""
    r = np.random.default_rng([seed, k])
    a, b = math.log(case["n_lo"]), math.log(max(case["n_hi"], case["n_lo"] + 1))
    return int(math.exp(r.uniform(a, b))), r.uniform(0.05, 0.8), r.uniform(0.1, 0.5), r.uniform(0.1, 0.4)


class State:
    """What a user's program keeps between calls."""

    server = None

    def __del__(self):
        if self.server is not None:
            self.server.stop()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = State()
    s.case = case
    kind = case["kind"]
    if kind == "train":
        B = case["samples"]
        s.X = -torch.log(1.0 - torch.rand(B, dd.DD_MLP_FEATURES, generator=gen, device="cuda"))
        s.u = 0.35 * torch.rand(B, generator=gen, device="cuda")
        s.mlp = dd.Mlp()
        s.mlp.set_params(_weights(seed))
        return s
    W, H = case["W"], case["H"]
    fx, fy = case.get("foe_x", W / 2.0), case.get("foe_y", H / 2.0)
    if kind in ("batch", "serve"):
        s.events = []
        for k in range(case["windows"]):
            n, D, tau, noise = _uneven(case, seed, k)
            x, y, t, _ = _descent(gen, W, H, fx, fy, n, D, tau, noise)
            s.events.append(dd.Events(x, y, t, 0.0, tau))
        s.ctx = dd.Context.tuned(W, H, fx, fy, (case["n_lo"] + case["n_hi"]) // 2, mode="batch", pop_k=16)
        s.params = [PARAMS] * case["windows"]
        if case.get("warm"):
            s.mlp = dd.Mlp(path=MODEL)
            s.ctx.set_warm_model(s.mlp)
            s.params = [PARAMS + ("model",)] * case["windows"]
        if kind == "serve":
            s.server = dd.Server(s.ctx, max_slots=case["slots"], max_events=case["n_hi"] + 1)
        torch.cuda.synchronize()
        return s
    if kind == "stream":
        # slots of 0.1 s of one descent, divergence rising towards contact
        parts = []
        for k in range(case["windows"] + 1):
            D = 1.0 / (12.0 - 0.1 * k)
            n = int(0.1 * case["rate"] * (0.5 + k / (case["windows"] + 1.0)))
            parts.append(_descent(gen, W, H, fx, fy, n, D, 0.1, 0.15, t_from=0.1 * k)[:3])
        x, y, t = (torch.cat(v) for v in zip(*parts))
        t, order = torch.sort(t)
        s.events = dd.Events(x[order].contiguous(), y[order].contiguous(), t.contiguous(), 0.0, 1.0)
        s.ctx = dd.Context.tuned(W, H, fx, fy, int(0.2 * case["rate"]), mode="batch", pop_k=16)
        torch.cuda.synchronize()
        return s
    n = case["n"]
    D, tau, noise = case.get("D", 0.35), case.get("tau", 0.3), case.get("noise", 0.3)
    x, y, t, p = _descent(gen, W, H, fx, fy, n, D, tau, noise)
    if not case.get("polarity"):
        p = None
    if case.get("host"):
        x, y, t = (a.cpu().numpy() for a in (x, y, t))
        p = None if p is None else p.cpu().numpy()
    s.events = dd.Events(x, y, t, 0.0, tau, p)
    s.foe = (fx, fy)
    options = {}
    if case.get("polarity"):
        options["polarity"] = 1
    if case.get("to_start"):
        options["warp_to_start"] = 1
    if kind == "fast":
        W2, H2 = case["W2"], case["H2"]
        fx2, fy2 = dd.dd_resample_foe(W, H, fx, fy, W2, H2)
        s.ctx = dd.Context.tuned(W2, H2, fx2, fy2, int(n * case["keep"]))
        s.seed = seed
    elif not case.get("noalloc"):
        if case.get("knobs") == "default":
            s.ctx = dd.Context(W, H, fx, fy, **options)
        else:
            s.ctx = dd.Context.tuned(W, H, fx, fy, n, **options)
    if kind == "contrast":
        s.D = np.linspace(-1.0, 1.0, case["hyp"] + 2)[1:-1].astype(np.float32) + np.float32(1e-3 * (seed % 97) / 97)
    if kind == "bound":
        lo = 0.35 - 0.5 * case["span"] if case["span"] < 1.0 else -1.0
        edges = np.linspace(lo, lo + case["span"], case["intervals"] + 1).astype(np.float32)
        s.lo, s.hi = edges[:-1], edges[1:]
    torch.cuda.synchronize()
    return s


def _weights(seed):
    """Network parameters (W1 b1 W2 b2 W3 b3, matrices [out][in])."""
    r = np.random.default_rng([seed, 7])
    a = math.sqrt(6.0 / 128.0)
    parts = []
    for out in (128, 128, 2):
        parts += [r.uniform(-a, a, out * 128), r.uniform(-0.05, 0.05, out)]
    p = np.concatenate(parts).astype(np.float32)
    p[-1] = math.log(0.05)
    return p


# --------------------------------------------------------------------- runs

def _wide(v):
    """128-bit integers as [n][2] int64 words, low word first."""
    m = (1 << 64) - 1
    return np.array([[k & m, (k >> 64) & m] for k in v], np.uint64).view(np.int64)


FLOATS = ("D_star", "D_end", "contrast", "bound_gap", "D_warm", "w_warm")
INTS = ("nodes_expanded", "point_evals", "bound_evals", "event_warps", "cell_increments", "bound_increments",
        "rounds", "max_queue", "status")


def _results(rs):
    return {"floats": np.array([[r[k] for k in FLOATS] for r in rs], np.float64),
            "ints": np.array([[r[k] for k in INTS] for r in rs], np.int64),
            "K_hat": _wide([r["K_hat"] for r in rs]), "gap_K": _wide([r["gap_K"] for r in rs])}


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "solve":
        return _results([s.ctx.solve(s.events, *PARAMS)])
    if kind == "batch":
        return _results(s.ctx.solve_batch(s.events, s.params)[1])
    if kind == "stream":
        _, res, ttc, first = s.ctx.stream_solve(s.events, 0.0, 0.2, 0.1, case["windows"], PARAMS)
        return dict(_results(res), ttc=ttc, first=first)
    if kind == "serve":
        tickets = [s.server.submit(e, p) for e, p in zip(s.events, s.params)]
        return _results([s.server.wait(k) for k in tickets])
    if kind == "contrast":
        if case.get("noalloc"):
            return {"K": _wide(dd.dd_contrast_noalloc(case["W"], case["H"], s.foe[0], s.foe[1], s.events, s.D))}
        K, S, N, images = s.ctx.contrast(s.events, s.D, want_iwe=bool(case.get("image")))
        return {"K": _wide(K), "S": S.view(np.int64), "N": N,
                "images": None if images is None else images.view(np.int32)}
    if kind == "bound":
        K, S, N, _ = s.ctx.bound(s.events, s.lo, s.hi)
        return {"K": _wide(K), "S": S.view(np.int64), "N": N}
    if kind == "fast":
        return _results([s.ctx.solve(s.ctx.resample(s.events, case["W"], case["H"], case["keep"], s.seed), *PARAMS)])
    grad, loss = s.mlp.grad(s.X, s.u)
    return {"grad": grad, "loss": loss}


# ------------------------------------------------------------ work and truth

# What a search cannot do without, in lane operations per event: at these
# ranges about 300 centres (8 each), 500 bounds (20 each) and 1,000 cells of
# the bounds' images (4 each).
SEARCH_OPS = 300 * 8 + 500 * 20 + 1000 * 4


def work(case):
    kind = case["kind"]
    if kind == "train":
        B, P = case["samples"], dd.DD_MLP_PARAMS
        return {"bytes": 4 * B * 129 + 2 * P + 4 * P, "flops": 6 * B * P}
    per = 9 if case.get("polarity") else 8
    if kind in ("batch", "serve"):
        a, b = math.log(case["n_lo"]), math.log(max(case["n_hi"], case["n_lo"] + 1))
        n = case["windows"] * (math.exp(b) - math.exp(a)) / (b - a)
        return {"bytes": per * n, "flops": SEARCH_OPS * n}
    if kind == "stream":
        n = 0.2 * case["rate"] * case["windows"]
        return {"bytes": per * n / 2, "flops": SEARCH_OPS * n}
    n = case["n"]
    if kind == "contrast":
        image = 4 * case["W"] * case["H"] * case["hyp"] if case.get("image") else 0
        return {"bytes": per * n + 36 * case["hyp"] + image, "flops": 8 * n * case["hyp"]}
    if kind == "bound":
        cells = 1 + 0.3 * case["span"] / case["intervals"] * 0.25 * (case["W"] + case["H"])
        return {"bytes": per * n + 40 * case["intervals"], "flops": n * case["intervals"] * (20 + 4 * cells)}
    if kind == "fast":
        return {"bytes": per * n + 16 * n * case["keep"], "flops": SEARCH_OPS * n * case["keep"]}
    return {"bytes": per * n, "flops": SEARCH_OPS * n}


def tolerance(case):
    # The gradient is a binary32 sum over the samples (2e-7 to 1e-6 off its
    # binary64 value); everything else is decided exactly.
    return {"rel": 1e-5, "max": 1e-3} if case["kind"] == "train" else "exact"


def exact(case, seed):
    # The estimator's outputs are integers (and the hypotheses they select)
    # that its binary32 warp defines: there is no nearer value in 64 bits.
    if case["kind"] != "train":
        return None
    s = prepare(case, seed)
    X, u = s.X.double(), s.u.double()
    p = torch.from_numpy(_weights(seed)).cuda()
    at, layers = 0, []
    for out in (128, 128, 2):
        w = p[at:at + out * 128].reshape(out, 128).bfloat16().double().requires_grad_()
        b = p[at + out * 128:at + out * 129].double().requires_grad_()
        layers.append((w, b))
        at += out * 129
    h = torch.relu(X @ layers[0][0].T + layers[0][1])
    h = torch.relu(h @ layers[1][0].T + layers[1][1])
    o = h @ layers[2][0].T + layers[2][1]
    loss = (4.5 * (u - o[:, 0]) ** 2 * torch.exp(-2.0 * o[:, 1]) + o[:, 1]).mean()
    grads = torch.autograd.grad(loss, [v for layer in layers for v in layer])
    return {"grad": torch.cat([g.reshape(-1) for g in grads]), "loss": loss.detach().reshape(1)}
