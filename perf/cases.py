"""Performance cases of the interpolator: what users of the library have it do.

A user has an edge-cost map and a list of sparse matches per frame pair and
wants the dense flow: one pair at a time (latency), a batch (throughput), or
batches of host buffers; with or without consistency pruning, as affine (LA)
or Nadaraya-Watson (NW) estimate.  Around that path stand the cost map from an
image, the assignment map alone, the exact per-pixel variant and the
variational refinement.  Every case goes through the public entry points of
``paper_1501_02565_gb300.native``.

Inputs are drawn on the GPU from the seed alone and follow the distributions
of ``paper_1501_02565_gb300.synth``: convex regions and thin strips with edge
strengths on their borders, cost 1e-3 + max(edge + N(0, 0.02), 0), a match on
about every hundredth pixel with 0.5 px noise and 10 % outliers, one affine
motion per region.

``exact`` gives 64-bit values for the cost map, the assignment distances, the
Euclidean exact variant and the refinement.  It gives none for interpolated
flows: geodesic distances of synthetic maps tie often, the side of a tie that
a pixel falls on is a convention of the fixed-point distances, and the match
graph (hence the flow of whole cells) depends on it.
"""

from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1501_02565_gb300 import native

# frame sizes (H, W) of the mixed batches and of the serving stream
BATCH_SIZES = ((480, 640), (436, 1024), (375, 1242), (1080, 1920))
SERVE_SIZES = ((480, 640), (436, 1024), (375, 1242), (1024, 2048))


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest frame, one at a time: latency and launches
        {"name": "pair_256x128", "kind": "pair", "H": 128, "W": 256, "N": 500, "K": 32,
         "regions": 6, "graph": False, "estimator": 0},
        # a film frame with the paper's match count, one at a time
        {"name": "pair_1024x436", "kind": "pair", "H": 436, "W": 1024, "N": 5000, "K": 100,
         "regions": 40, "graph": False, "estimator": 0},
        # a driving frame (odd width and height, denser matches) from a
        # program that replays captured launches
        {"name": "pair_1242x375_graph", "kind": "pair", "H": 375, "W": 1242, "N": 8000, "K": 100,
         "regions": 22, "graph": True, "estimator": 0},
        # the largest frame of the serving stream
        {"name": "pair_2048x1024", "kind": "pair", "H": 1024, "W": 2048, "N": 20972, "K": 100,
         "regions": 60, "graph": False, "estimator": 0},
        # throughput: 64 pairs of mixed sizes and neighbourhoods in one run
        {"name": "batch_64_mixed", "kind": "batch", "pairs": 64, "sizes": "batch",
         "regions": 40, "prune": False, "estimator": 0, "graph": True},
        # a batch whose outliers are pruned first (two passes)
        {"name": "batch_8_pruned", "kind": "batch", "pairs": 8, "sizes": "sintel",
         "regions": 40, "prune": True, "estimator": 0, "graph": False},
        # a client that holds everything in pinned host memory
        {"name": "host_16_serving", "kind": "host", "pairs": 16, "sizes": "serve", "regions": 40},
        # the assignment map alone, for hosts that own all device memory
        {"name": "labels_1024x436", "kind": "labels", "H": 436, "W": 1024, "N": 5000,
         "regions": 40},
        # the exact per-pixel variant, both metrics
        {"name": "exact_geodesic_1024x436", "kind": "exact", "metric": "geodesic", "H": 436,
         "W": 1024, "N": 5000, "K": 100, "regions": 40, "lists": False},
        {"name": "exact_euclidean_1024x436", "kind": "exact", "metric": "euclidean", "H": 436,
         "W": 1024, "N": 5000, "K": 100, "regions": 40, "lists": False},
        # refinement of an interpolated flow between two colour frames
        {"name": "refine_1024x436", "kind": "refine", "H": 436, "W": 1024, "channels": 3,
         "regions": 40},
        # cost maps of a stack of colour frames
        {"name": "cost_32x1024x436", "kind": "cost", "frames": 32, "H": 436, "W": 1024,
         "channels": 3, "regions": 12},
    ]


def _between(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _frame(rng, lo, hi):
    """(H, W) with lo to hi pixels and an aspect ratio from 1:1 to 3.3:1."""
    P = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    r = rng.uniform(1.0, 3.3)
    return max(16, int(math.sqrt(P / r))), max(16, int(math.sqrt(P * r)))


def draw(rng):
    kind = rng.choice(("pair", "pair", "pair", "batch", "batch", "host", "labels", "exact",
                       "exact", "refine", "cost"))
    if kind == "pair":
        H, W = _frame(rng, 16000, 2097152)
        return {"kind": kind, "H": H, "W": W,
                "N": max(64, min(30000, int(H * W / math.exp(rng.uniform(math.log(55), math.log(250)))))),
                "K": rng.choice((16, 25, 32, 64, 100, 128)), "regions": rng.randint(4, 80),
                "graph": rng.random() < 0.4, "estimator": int(rng.random() < 0.2)}
    if kind == "batch":
        return {"kind": kind, "pairs": _between(rng, 2, 40),
                "sizes": rng.choice(("batch", "serve", "sintel", "small", "any")),
                "regions": rng.randint(10, 80), "prune": rng.random() < 0.25,
                "estimator": int(rng.random() < 0.2), "graph": rng.random() < 0.5}
    if kind == "host":
        return {"kind": kind, "pairs": _between(rng, 1, 24),
                "sizes": rng.choice(("batch", "serve", "small", "any")),
                "regions": rng.randint(10, 80)}
    if kind == "labels":
        H, W = _frame(rng, 16000, 500000)
        return {"kind": kind, "H": H, "W": W, "N": max(64, int(H * W / rng.uniform(55, 250))),
                "regions": rng.randint(4, 60)}
    if kind == "exact":
        H, W = _frame(rng, 10000, 440000)
        return {"kind": kind, "metric": rng.choice(("geodesic", "euclidean")), "H": H, "W": W,
                "N": max(40, min(5000, int(H * W / rng.uniform(80, 250)))),
                "K": rng.choice((8, 25, 32, 64, 100)), "regions": rng.randint(4, 40),
                "lists": rng.random() < 0.3}
    if kind == "refine":
        H, W = _frame(rng, 16000, 2097152)
        return {"kind": kind, "H": H, "W": W, "channels": rng.choice((1, 3)),
                "regions": rng.randint(4, 60)}
    H, W = _frame(rng, 16000, 2097152)
    return {"kind": "cost", "frames": max(1, min(64, _between(rng, 16000, 14000000) // (H * W))),
            "H": H, "W": W, "channels": rng.choice((1, 3, 4)), "regions": rng.randint(4, 12)}


def _batch_shapes(case):
    """(H, W, N, K) of every pair of a batch: a fixed mix per case, so that
    only the contents depend on the seed."""
    import random
    rng = random.Random("%s/%d" % (case["sizes"], case["pairs"]))
    out = []
    for i in range(case["pairs"]):
        if case["sizes"] == "batch":
            H, W = BATCH_SIZES[i % 4]
            N = min(20000, max(2000, round(H * W / 100)))
            K = (64, 100, 128)[(i // 4) % 3]
        elif case["sizes"] == "serve":
            H, W = SERVE_SIZES[i % 4]
            N, K = int(min(H * W / 100 * rng.uniform(0.7, 1.4), 30000)), 100
        elif case["sizes"] == "sintel":
            H, W, N, K = 436, 1024, 5000, 100
        elif case["sizes"] == "small":
            H, W, N, K = 128, 256, 500, 32
        else:
            H, W = _frame(rng, 16000, 1000000)
            N, K = max(64, int(H * W / rng.uniform(60, 200))), rng.choice((32, 64, 100))
        out.append((H, W, N, K))
    return out


# ---------------------------------------------------------------------------
# inputs, drawn on the GPU
# ---------------------------------------------------------------------------

def _device():
    return torch.device("cuda", 0)


def _generators(seed, stream=0):
    s = (int(seed) * 1000003 + stream) % (1 << 62)
    g = torch.Generator(device=_device())
    g.manual_seed(s)
    return np.random.Generator(np.random.PCG64(s)), g


def _regions(rng, H, W, n):
    """Region map int64 [H, W]: n convex regions painted over a background,
    a quarter of them thin strips of 8 to 30 px."""
    dev = _device()
    R = torch.zeros((H, W), dtype=torch.int64, device=dev)
    for rid in range(1, n + 1):
        if rid > n - n // 4:
            # a rotated thin rectangle
            half = np.array([0.5 * rng.uniform(0.2, 0.6) * max(H, W), 0.5 * rng.uniform(8.0, 30.0)])
            c = np.array([rng.uniform(0, W), rng.uniform(0, H)])
            t = rng.uniform(0, math.pi)
            d = np.array([math.cos(t), math.sin(t)])
            e = np.array([-d[1], d[0]])
            V = np.array([c + half[0] * d + half[1] * e, c - half[0] * d + half[1] * e,
                          c - half[0] * d - half[1] * e, c + half[0] * d - half[1] * e])
        else:
            # a polygon inscribed in an ellipse
            k = int(rng.integers(5, 9))
            t = np.sort(rng.uniform(0, 2 * math.pi, size=k))
            rx, ry = 0.5 * rng.uniform(0.15, 0.5) * W, 0.5 * rng.uniform(0.15, 0.5) * H
            V = np.stack([rng.uniform(0, W) + rx * np.cos(t), rng.uniform(0, H) + ry * np.sin(t)], 1)
        x0, x1 = max(0, math.floor(V[:, 0].min())), min(W, math.ceil(V[:, 0].max()) + 1)
        y0, y1 = max(0, math.floor(V[:, 1].min())), min(H, math.ceil(V[:, 1].max()) + 1)
        if x1 <= x0 or y1 <= y0:
            continue
        xs = torch.arange(x0, x1, dtype=torch.float32, device=dev)[None, :]
        ys = torch.arange(y0, y1, dtype=torch.float32, device=dev)[:, None]
        inside = None
        for i in range(len(V)):
            a, b = V[i], V[(i + 1) % len(V)]
            m = (float(b[0] - a[0]) * (ys - float(a[1]))) >= (float(b[1] - a[1]) * (xs - float(a[0])))
            inside = m if inside is None else inside & m
        R[y0:y1, x0:x1].masked_fill_(inside, rid)
    return R


def _scene(seed, H, W, n_regions, stream=0):
    """(regions, cost map, true flow, numpy rng, torch generator)."""
    rng, g = _generators(seed, stream)
    dev = _device()
    R = _regions(rng, H, W, n_regions)
    strength = torch.from_numpy(rng.uniform(0.2, 1.0, size=n_regions + 1).astype(np.float32)).to(dev)
    S = strength[R]
    E = torch.zeros((H, W), dtype=torch.float32, device=dev)
    for A, B in (((slice(None), slice(0, W - 1)), (slice(None), slice(1, W))),
                 ((slice(0, H - 1), slice(None)), (slice(1, H), slice(None)))):
        s = torch.maximum(S[A], S[B]) * (R[A] != R[B])
        E[A] = torch.maximum(E[A], s)
        E[B] = torch.maximum(E[B], s)
    noise = torch.randn((H, W), generator=g, device=dev) * 0.02
    C = (1e-3 + (E + noise).clamp_(min=0)).contiguous()
    # one affine motion per region, about a point of the frame
    A = torch.from_numpy(rng.uniform(-0.05, 0.05, size=(n_regions + 1, 4)).astype(np.float32)).to(dev)
    t = torch.from_numpy(rng.uniform(-60.0, 60.0, size=(n_regions + 1, 2)).astype(np.float32)).to(dev)
    c = torch.from_numpy((rng.uniform(0, 1, size=(n_regions + 1, 2)) * [W, H]).astype(np.float32)).to(dev)
    dx = torch.arange(W, dtype=torch.float32, device=dev)[None, :] - c[R, 0]
    dy = torch.arange(H, dtype=torch.float32, device=dev)[:, None] - c[R, 1]
    flow = torch.stack([A[R, 0] * dx + A[R, 1] * dy + t[R, 0],
                        A[R, 2] * dx + A[R, 3] * dy + t[R, 1]], -1).contiguous()
    return R, C, flow, rng, g


def _matches(flow, N, g):
    """N matches [N, 4] on distinct pixels: jittered grid cells where the
    frame has enough of them, else any pixels."""
    H, W = flow.shape[:2]
    dev = flow.device
    gx, gy = (W + 3) // 8, (H + 3) // 8
    if gx * gy >= N:
        pick = torch.randperm(gx * gy, generator=g, device=dev)[:N]
        jx = torch.randint(-3, 4, (N,), generator=g, device=dev)
        jy = torch.randint(-3, 4, (N,), generator=g, device=dev)
        x = ((pick % gx) * 8 + 4 + jx).clamp_(0, W - 1)
        y = ((pick // gx) * 8 + 4 + jy).clamp_(0, H - 1)
    else:
        pick = torch.randperm(H * W, generator=g, device=dev)[:N]
        x, y = pick % W, pick // W
    uv = flow[y, x] + 0.5 * torch.randn((N, 2), generator=g, device=dev)
    out = torch.rand((N,), generator=g, device=dev) < 0.1
    wild = (torch.rand((N, 2), generator=g, device=dev) - 0.5) * 300.0
    uv = torch.where(out[:, None], wild, uv)
    xy = torch.stack([x, y], 1).to(torch.float32)
    return torch.cat([xy, xy + uv], 1).contiguous()


def _image(R, n_regions, channels, rng, g):
    """An image [H, W, channels] in [0, 1]: a colour and a texture of plane
    waves per region, and pixel noise."""
    H, W = R.shape
    dev = R.device
    n = n_regions + 1

    def per_region(lo, hi, *shape):
        return torch.from_numpy(rng.uniform(lo, hi, size=(n,) + shape).astype(np.float32)).to(dev)[R]

    xs = torch.arange(W, dtype=torch.float32, device=dev)[None, :]
    ys = torch.arange(H, dtype=torch.float32, device=dev)[:, None]
    img = per_region(0.15, 0.85, channels)
    for _ in range(3):
        ang, freq = per_region(0, math.pi), per_region(0.1, 0.5)
        wave = per_region(0.03, 0.08) * torch.sin(
            freq * (torch.cos(ang) * xs + torch.sin(ang) * ys) + per_region(0, 2 * math.pi))
        img = img + wave[..., None]
    img = img + 0.005 * torch.randn((H, W, channels), generator=g, device=dev)
    return img.clamp_(0, 1).contiguous()


def _sample(img, X, Y):
    """img [H, W, C] at (X, Y), bilinear, coordinates clamped to the frame."""
    H, W = img.shape[:2]
    X = X.clamp(0, W - 1)
    Y = Y.clamp(0, H - 1)
    x0 = X.floor().long().clamp_(max=max(W - 2, 0))
    y0 = Y.floor().long().clamp_(max=max(H - 2, 0))
    x1, y1 = (x0 + 1).clamp_(max=W - 1), (y0 + 1).clamp_(max=H - 1)
    ax, ay = (X - x0)[..., None], (Y - y0)[..., None]
    return ((1 - ay) * ((1 - ax) * img[y0, x0] + ax * img[y0, x1]) +
            ay * ((1 - ax) * img[y1, x0] + ax * img[y1, x1]))


def _frames(seed, H, W, channels, n_regions):
    """Two frames under a smooth-per-region motion and a flow to refine (the
    true flow disturbed by a smooth field of about 1 px)."""
    R, _, flow, rng, g = _scene(seed, H, W, n_regions)
    I1 = _image(R, n_regions, channels, rng, g)
    xs = torch.arange(W, dtype=torch.float32, device=I1.device)[None, :]
    ys = torch.arange(H, dtype=torch.float32, device=I1.device)[:, None]
    back = flow
    for _ in range(4):
        back = _sample(flow, xs - back[..., 0], ys - back[..., 1])
    I2 = _sample(I1, xs - back[..., 0], ys - back[..., 1]).contiguous()
    coarse = torch.randn((H // 32 + 2, W // 32 + 2, 2), generator=g, device=I1.device)
    smooth = _sample(coarse, (xs / 32).expand(H, W), (ys / 32).expand(H, W))
    return I1, I2, (flow + smooth).contiguous()


_side_stream = None


def _stream():
    """The one stream that a program with captured launches runs them on."""
    global _side_stream
    if _side_stream is None:
        _side_stream = torch.cuda.Stream()
    return _side_stream


def _engine(shapes, **cfg):
    return native.EpicInterp(0, max_pairs=len(shapes), max_H=max(s[0] for s in shapes),
                             max_W=max(s[1] for s in shapes), max_N=max(s[2] for s in shapes),
                             max_K=max(s[3] for s in shapes), **cfg)


def _batch_inputs(case, seed):
    shapes = _batch_shapes(case)
    items = []
    for i, (H, W, N, K) in enumerate(shapes):
        _, C, flow, _, g = _scene(seed, H, W, case["regions"], 1 + i)
        items.append((C, _matches(flow, N, g), K, 1.0))
    return shapes, items


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pair":
        _, C, flow, _, g = _scene(seed, case["H"], case["W"], case["regions"])
        M = _matches(flow, case["N"], g)
        eng = _engine([(case["H"], case["W"], case["N"], case["K"])],
                      use_graphs=int(case["graph"]), estimator=case["estimator"])
        return {"case": case, "eng": eng, "C": C, "M": M, "out": torch.empty_like(flow),
                "stream": _stream() if case["graph"] else None}
    if kind == "batch":
        shapes, items = _batch_inputs(case, seed)
        items = [(C, M, K, a, torch.empty(C.shape + (2,), device=C.device)) for C, M, K, a in items]
        eng = _engine(shapes, use_graphs=int(case["graph"]), estimator=case["estimator"],
                      prune=int(case["prune"]))
        return {"case": case, "eng": eng, "items": items,
                "stream": _stream() if case["graph"] else None}
    if kind == "host":
        shapes, items = _batch_inputs(case, seed)
        items = [(C.cpu().pin_memory(), M.cpu().pin_memory(), K, a,
                  torch.empty(C.shape + (2,)).pin_memory()) for C, M, K, a in items]
        return {"case": case, "eng": _engine(shapes), "items": items}
    if kind == "labels":
        _, C, flow, _, g = _scene(seed, case["H"], case["W"], case["regions"])
        return {"case": case, "lib": native.load(), "C": C, "M": _matches(flow, case["N"], g),
                "L": torch.empty(C.shape, dtype=torch.int32, device=C.device),
                "D": torch.empty_like(C)}
    if kind == "exact":
        _, C, flow, _, g = _scene(seed, case["H"], case["W"], case["regions"])
        eng = _engine([(case["H"], case["W"], case["N"], case["K"])])
        return {"case": case, "eng": eng, "C": C, "M": _matches(flow, case["N"], g)}
    if kind == "refine":
        I1, I2, start = _frames(seed, case["H"], case["W"], case["channels"], case["regions"])
        return {"case": case, "eng": native.EpicInterp(0), "I1": I1, "I2": I2, "start": start,
                "flow": start.clone()}
    if kind == "cost":
        frames = []
        for i in range(case["frames"]):
            rng, g = _generators(seed, i)
            R = _regions(rng, case["H"], case["W"], case["regions"])
            frames.append(_image(R, case["regions"], case["channels"], rng, g))
        imgs = torch.stack(frames)
        return {"case": case, "imgs": imgs, "out": torch.empty(imgs.shape[:3], device=imgs.device)}
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "pair":
        return state["eng"].run(state["C"], state["M"], case["K"], 1.0, flow=state["out"],
                                stream=state["stream"])
    if kind == "batch":
        state["eng"].run_batch(state["items"], stream=state["stream"])
        return [it[4] for it in state["items"]]
    if kind == "host":
        state["eng"].run_batch_host(state["items"])
        return [it[4] for it in state["items"]]
    if kind == "labels":
        ptr = ctypes.c_void_p
        rc = state["lib"].epic_geodesic_labels_noalloc(
            ptr(state["C"].data_ptr()), ptr(state["M"].data_ptr()), case["H"], case["W"],
            case["N"], ptr(state["L"].data_ptr()), ptr(state["D"].data_ptr()),
            ptr(torch.cuda.current_stream().cuda_stream))
        if rc != native.EPIC_OK:
            raise native.EpicError(rc, "epic_geodesic_labels_noalloc")
        return state["L"], state["D"]
    if kind == "exact":
        return state["eng"].exact(state["C"], state["M"], case["K"], 1.0, metric=case["metric"],
                                  with_knn=case["lists"])
    if kind == "refine":
        # the interpolated flow arrives anew for every frame
        state["flow"].copy_(state["start"])
        return state["eng"].refine(state["I1"], state["I2"], state["flow"])
    if kind == "cost":
        return native.gradient_cost(state["imgs"], 1e-3, out=state["out"])
    raise ValueError(kind)


def work(case):
    """Bytes and operations that a pass cannot do without: inputs and outputs
    once; per pixel the eight neighbour steps of its distance and the model's
    value, per fit its weighted sums, per refinement the linear systems and
    their red-black updates."""
    kind = case["kind"]
    if kind in ("pair", "batch", "host"):
        shapes = ([(case["H"], case["W"], case["N"], case["K"])] if kind == "pair"
                  else _batch_shapes(case))
        P = sum(s[0] * s[1] for s in shapes)
        N = sum(s[2] for s in shapes)
        fits = sum(s[2] * s[3] for s in shapes) + (25 * N if case.get("prune") else 0)
        return {"bytes": 12 * P + 16 * N, "flops": (24 + 10) * P + 45 * fits}
    if kind == "cost":
        n = case["frames"] * case["H"] * case["W"]
        return {"bytes": 4 * n * (case["channels"] + 1), "flops": n * (8 * case["channels"] + 2)}
    P = case["H"] * case["W"]
    if kind == "labels":
        return {"bytes": 12 * P + 16 * case["N"], "flops": 24 * P}
    if kind == "exact":
        K = min(case["K"], case["N"])
        read = 4 * P if case["metric"] == "geodesic" else 0
        steps = 24 * P * K if case["metric"] == "geodesic" else 6 * P * K
        return {"bytes": read + 16 * case["N"] + 8 * P + (8 * P * K if case["lists"] else 0),
                "flops": steps + 45 * P * K}
    if kind == "refine":
        return {"bytes": 8 * P * case["channels"] + 16 * P,
                "flops": 5 * P * (120 * case["channels"] + 30 * 50)}
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------

def _grad(a, axis):
    """Central difference on the edge-replicated array."""
    n = a.shape[axis]
    i = torch.arange(n, device=a.device)
    return 0.5 * (a.index_select(axis, (i + 1).clamp(max=n - 1)) -
                  a.index_select(axis, (i - 1).clamp(min=0)))


def _exact_cost(case, seed):
    imgs = prepare(case, seed)["imgs"]
    out = []
    for f in imgs:
        f = f.double()
        out.append(float(np.float32(1e-3)) +
                   (_grad(f, 1) ** 2 + _grad(f, 0) ** 2).sum(-1).sqrt())
    return torch.stack(out)


def _exact_distance(case, seed):
    """Shortest-path distance of every pixel to its nearest match: steps of
    |p - q| (C(p) + C(q)) / 2 on the 8-connected grid, to the fixed point."""
    s = prepare(case, seed)
    C, M = s["C"].double(), s["M"]
    H, W = C.shape
    D = torch.full((H + 2, W + 2), math.inf, dtype=torch.float64, device=C.device)
    Cp = torch.zeros_like(D)
    Cp[1:-1, 1:-1] = C
    D[(M[:, 1] + 0.5).floor().long() + 1, (M[:, 0] + 0.5).floor().long() + 1] = 0.0
    steps = []
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            if dx or dy:
                w = math.hypot(dx, dy) * 0.5 * (C + Cp[1 + dy:H + 1 + dy, 1 + dx:W + 1 + dx])
                steps.append((dy, dx, w))
    for it in range(H * W):
        old = D[1:-1, 1:-1].clone()
        new = old
        for dy, dx, w in steps:
            new = torch.minimum(new, D[1 + dy:H + 1 + dy, 1 + dx:W + 1 + dx] + w)
        D[1:-1, 1:-1] = new
        if it % 16 == 15 and bool((new == old).all()):
            break
    return [None, D[1:-1, 1:-1].contiguous()]


def _exact_euclidean(case, seed):
    s = prepare(case, seed)
    M = s["M"].double()
    H, W, N = case["H"], case["W"], case["N"]
    K = min(case["K"], N)
    P = H * W
    mx, my = (M[:, 0] + 0.5).floor().long(), (M[:, 1] + 0.5).floor().long()
    flow, idx, dist = [], [], []
    step = max(1, (1 << 27) // N)
    for p0 in range(0, P, step):
        p = torch.arange(p0, min(P, p0 + step), device=M.device)
        px, py = p % W, p // W
        d2 = (px[:, None] - mx[None, :]) ** 2 + (py[:, None] - my[None, :]) ** 2
        # the K smallest (distance, index)
        key = d2 * N + torch.arange(N, device=M.device)[None, :]
        key = key.topk(K, dim=1, largest=False, sorted=True).values
        n, d = key % N, (key // N).double().sqrt()
        k = torch.exp(-d)
        w = k * k
        q = M[n]
        xt, yt = q[..., 0] - px[:, None], q[..., 1] - py[:, None]
        uv = q[..., 2:] - q[..., :2]
        X = torch.stack([xt, yt, torch.ones_like(xt)], -1)
        A = torch.einsum("pk,pki,pkj->pij", w, X, X)
        b = torch.einsum("pk,pki,pkc->pic", w, X, uv)
        det = torch.linalg.det(A)
        tr3 = A.diagonal(dim1=1, dim2=2).sum(-1) / 3
        ok = (det > float(np.float32(1e-10)) * tr3 ** 3) & (K >= 3)
        eye = torch.eye(3, dtype=A.dtype, device=A.device)
        sol = torch.linalg.solve(torch.where(ok[:, None, None], A, eye), b)[:, 2]
        nw = (k[..., None] * uv).sum(1) / k.sum(1, keepdim=True)
        flow.append(torch.where(ok[:, None], sol, nw))
        idx.append(n.to(torch.int32))
        dist.append(d)
    flow = torch.cat(flow).reshape(H, W, 2)
    return (flow, torch.cat(idx), torch.cat(dist)) if case["lists"] else flow


def _exact_refine(case, seed):
    s = prepare(case, seed)
    I1, I2 = s["I1"].double(), s["I2"].double()
    u, v = s["start"][..., 0].double(), s["start"][..., 1].double()
    H, W = u.shape
    dev = u.device
    f32 = lambda x: float(np.float32(x))  # noqa: E731  (the parameters are 32-bit)
    gamma, kappa, eps, zeta, omega = f32(0.7), 5.0, f32(1e-3), f32(0.1), f32(1.6)
    xs = torch.arange(W, dtype=torch.float64, device=dev)[None, :]
    ys = torch.arange(H, dtype=torch.float64, device=dev)[:, None]
    red = ((xs + ys) % 2) == 0

    def dx(a):
        return _grad(a, 1)

    def dy(a):
        return _grad(a, 0)

    def dpsi(s2):
        return 0.5 / torch.sqrt(s2 + eps * eps)

    for _ in range(5):
        Iw = _sample(I2, xs + u, ys + v)
        Ix, Iy, Iz = 0.5 * (dx(I1) + dx(Iw)), 0.5 * (dy(I1) + dy(Iw)), Iw - I1
        t0 = 1 / (Ix * Ix + Iy * Iy + zeta ** 2)
        g1x, g1y, g2x, g2y = dx(I1), dy(I1), dx(Iw), dy(Iw)
        Ixx, Ixy = 0.5 * (dx(g1x) + dx(g2x)), 0.5 * (dy(g1x) + dy(g2x))
        Iyx, Iyy = 0.5 * (dx(g1y) + dx(g2y)), 0.5 * (dy(g1y) + dy(g2y))
        Ixz, Iyz = g2x - g1x, g2y - g1y
        tx, ty = 1 / (Ixx ** 2 + Ixy ** 2 + zeta ** 2), 1 / (Iyx ** 2 + Iyy ** 2 + zeta ** 2)
        pc = dpsi((t0 * Iz * Iz).sum(-1))
        pg = gamma * dpsi((tx * Ixz ** 2 + ty * Iyz ** 2).sum(-1))
        A11 = pc * (t0 * Ix * Ix).sum(-1) + pg * (tx * Ixx ** 2 + ty * Iyx ** 2).sum(-1)
        A12 = pc * (t0 * Ix * Iy).sum(-1) + pg * (tx * Ixx * Ixy + ty * Iyx * Iyy).sum(-1)
        A22 = pc * (t0 * Iy * Iy).sum(-1) + pg * (tx * Ixy ** 2 + ty * Iyy ** 2).sum(-1)
        b1 = pc * (t0 * Ix * Iz).sum(-1) + pg * (tx * Ixx * Ixz + ty * Iyx * Iyz).sum(-1)
        b2 = pc * (t0 * Iy * Iz).sum(-1) + pg * (tx * Ixy * Ixz + ty * Iyy * Iyz).sum(-1)
        alpha = torch.exp(-kappa * (g1x ** 2 + g1y ** 2).sum(-1).sqrt())
        phi = alpha * dpsi(dx(u) ** 2 + dy(u) ** 2 + dx(v) ** 2 + dy(v) ** 2)
        # edge weights to the right, left, lower and upper neighbour
        sr, sd = torch.zeros_like(phi), torch.zeros_like(phi)
        sr[:, :-1] = 0.5 * (phi[:, :-1] + phi[:, 1:])
        sd[:-1] = 0.5 * (phi[:-1] + phi[1:])
        sl, su = torch.roll(sr, 1, 1), torch.roll(sd, 1, 0)
        S = sr + sl + sd + su
        a, d = A11 + S, A22 + S
        det = a * d - A12 * A12

        def around(f):
            return (sr * torch.roll(f, -1, 1) + sl * torch.roll(f, 1, 1) +
                    sd * torch.roll(f, -1, 0) + su * torch.roll(f, 1, 0))

        du, dv = torch.zeros_like(u), torch.zeros_like(v)
        for _ in range(30):
            for colour in (red, ~red):
                r1 = around(u + du) - S * u - b1
                r2 = around(v + dv) - S * v - b2
                m = colour & (det > 0)
                nu, nv = (d * r1 - A12 * r2) / det, (a * r2 - A12 * r1) / det
                du = torch.where(m, (1 - omega) * du + omega * nu, du)
                dv = torch.where(m, (1 - omega) * dv + omega * nv, dv)
        u, v = u + du, v + dv
    return torch.stack([u, v], -1)


def exact(case, seed):
    if case["kind"] == "cost":
        return _exact_cost(case, seed)
    if case["kind"] == "labels":
        return _exact_distance(case, seed)
    if case["kind"] == "exact" and case["metric"] == "euclidean":
        return _exact_euclidean(case, seed)
    if case["kind"] == "refine":
        return _exact_refine(case, seed)
    return None
