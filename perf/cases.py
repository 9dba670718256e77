"""The cases this library's speed is measured on, through its public entry points.

A case is one call, or one chain of calls, that a program quantizing a network (or running a
quantized one) makes:

  layer         pipeline.LayerPlan.run_device: greedy points, output error, allocation and
                multipoint weights of one layer (centred first where ``center`` says so)
  network       pipeline.CapturedNetwork.replay: every layer of a network in one step
  greedy        mpq_quantize_layer alone, linear grid or the caller's own
  output_error  mpq_output_error alone, on the points of the greedy search
  adaptive      mpq_quantize_layer_adaptive
  clip          mpq_clip_search
  infer         mpq_multipoint_linear on a packed layer

Sizes are those of the repository's workloads (ResNet-18/-50- and MobileNetV2-shaped layers, the
large linear layers) and generic ones around them.  ``exact`` restates every path in plain torch,
sums and contractions in 64 bits.
"""
import math

import torch

from paper_2002_09049_gb300 import binding, pipeline

ETA = 2.0 ** -10          # largest step of the adaptive grid (the experiments' value)


# ---------------------------------------------------------------------------------------------
# The cases


def _layer(C, d, N, bits, G, k_max, beta, wdist, xdist="relu", depthwise=False, center=-1):
    return dict(kind="layer", C=C, d=d, N=N, bits=bits, G=G, k_max=k_max, beta=beta, wdist=wdist,
                xdist=xdist, depthwise=depthwise, center=center)


def _greedy(C, d, bits, G, k_max, wdist, grid="linear"):
    return dict(kind="greedy", C=C, d=d, bits=bits, G=G, k_max=k_max, wdist=wdist, grid=grid)


def _output_error(C, d, N, bits, G, k_max, wdist, xdist):
    return dict(kind="output_error", C=C, d=d, N=N, bits=bits, G=G, k_max=k_max, wdist=wdist,
                xdist=xdist)


def _adaptive(C, d, bits, k_max, wdist):
    return dict(kind="adaptive", C=C, d=d, bits=bits, k_max=k_max, wdist=wdist)


def _clip(C, d, N, bits, n_cand, per_layer, wdist, xdist="relu"):
    return dict(kind="clip", C=C, d=d, N=N, bits=bits, n_cand=n_cand, per_layer=per_layer,
                wdist=wdist, xdist=xdist)


def _infer(C, d, T, bits, k_max, beta, p, centered, wdist):
    return dict(kind="infer", C=C, d=d, T=T, bits=bits, k_max=k_max, beta=beta, p=p,
                centered=centered, wdist=wdist)


def _network(layers, N, bits, G, k_max, beta, wdist):
    return dict(kind="network", layers=layers, N=N, bits=bits, G=G, k_max=k_max, beta=beta,
                wdist=wdist)


# The ResNet-18-shaped set with one block per stage: first convolution, every stage's
# convolutions and downsampling, classifier.
RESNET_LAYERS = ("64x147,64x576,64x576,128x576,128x1152,128x64,256x1152,256x2304,256x128,"
                 "512x2304,512x4608,512x256,1000x512")


def listed():
    return [
        # one small convolution on its own, where launches and latency count
        dict(_layer(64, 576, 512, 4, 64, 4, 2.0, "normal"), name="layer_conv_64x576"),
        # an image network's first convolution: 3x7x7 weights, an odd row length
        dict(_layer(64, 147, 1024, 4, 128, 4, 1.3, "normal"), name="layer_first_conv_64x147"),
        # a depthwise 3x3 convolution: thousands of 9-element channels, each its own inputs
        dict(_layer(960, 9, 1024, 4, 64, 8, 1.5, "laplace", depthwise=True),
             name="layer_depthwise_960x9"),
        # a pointwise (1x1) convolution
        dict(_layer(1280, 320, 1024, 4, 64, 8, 1.5, "laplace"), name="layer_pointwise_1280x320"),
        # a last-stage 3x3 convolution, heavy-tailed weights, 3 bits, asymmetric sets
        dict(_layer(512, 4608, 2048, 3, 128, 6, 1.5, "student", center=0),
             name="layer_conv_512x4608_3bit"),
        # a whole network in one captured step
        dict(_network(RESNET_LAYERS, 1024, 4, 128, 4, 1.3, "normal"), name="network_13_layers"),
        # a large linear layer with outlier weights: the greedy search and the output error alone
        dict(_greedy(11008, 4096, 4, 256, 8, "outliers"), name="greedy_linear_11008x4096"),
        dict(_output_error(11008, 4096, 2048, 4, 256, 8, "outliers", "hot"),
             name="output_error_linear_11008x4096"),
        # the experiments' adaptive grid on a convolution
        dict(_adaptive(64, 576, 4, 4, "normal"), name="adaptive_conv_64x576"),
        # the experiments' clipping factors, a classifier layer
        dict(_clip(1000, 2048, 2048, 4, 20, False, "student"), name="clip_fc_1000x2048"),
        # integer inference with the allocated points: a handful of inputs, and a large batch
        dict(_infer(4096, 4096, 8, 4, 4, 1.25, 16, False, "outliers"),
             name="infer_4096x4096_8_inputs"),
        dict(_infer(4096, 4096, 2048, 4, 4, 1.25, 16, False, "outliers"),
             name="infer_4096x4096_2048_inputs"),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _row(rng, lo, hi):
    """A row length: any whole number, or (two times in three, as most layers have) a multiple
    of 16."""
    d = _log(rng, lo, hi)
    return d if rng.random() < 1 / 3 else max(16, d // 16 * 16)


def draw(rng):
    kind = rng.choice(("layer", "layer", "depthwise", "network", "greedy", "output_error",
                       "output_error", "adaptive", "clip", "infer", "infer"))
    wdist = rng.choice(("normal", "student", "laplace", "outliers"))
    bits = rng.choice((3, 4, 4, 4, 5, 8))
    if kind == "layer":
        G = rng.choice((32, 64, 100, 128, 256))
        return _layer(_log(rng, 16, 2048), _row(rng, 16, 4608), _log(rng, 100, 2048), bits, G,
                      rng.randint(1, 8), round(rng.uniform(1.0, 2.5), 2), wdist,
                      rng.choice(("relu", "hot")), False, rng.choice((-1, -1, 0, 1)))
    if kind == "depthwise":
        return _layer(_log(rng, 32, 1536), rng.choice((9, 9, 25)), _log(rng, 100, 1024), bits,
                      rng.choice((32, 64, 128)), rng.randint(2, 8),
                      round(rng.uniform(1.0, 2.5), 2), wdist, "relu", True)
    if kind == "network":
        shapes = ["%dx%d" % (_log(rng, 16, 1024), _row(rng, 27, 4608))
                  for _ in range(rng.randint(4, 12))]
        return _network(",".join(shapes), _log(rng, 256, 1024), 4, rng.choice((64, 128)),
                        rng.randint(2, 6), round(rng.uniform(1.0, 2.0), 2), wdist)
    if kind == "greedy":
        return _greedy(_log(rng, 64, 8192), _row(rng, 64, 4096), bits,
                       rng.choice((32, 64, 100, 128, 256)), rng.randint(1, 8), wdist,
                       rng.choice(("linear", "linear", "geometric")))
    if kind == "output_error":
        return _output_error(_log(rng, 64, 8192), _row(rng, 64, 4096), _log(rng, 100, 2048), bits,
                             32, rng.randint(1, 8), wdist, rng.choice(("relu", "hot")))
    if kind == "adaptive":
        return _adaptive(_log(rng, 8, 160), _log(rng, 9, 576), rng.choice((3, 4)),
                         rng.randint(1, 4), rng.choice(("normal", "laplace")))
    if kind == "clip":
        return _clip(_log(rng, 64, 2048), _row(rng, 64, 2048), _log(rng, 100, 2048), bits,
                     rng.choice((10, 20, 32)), rng.random() < 0.3, wdist,
                     rng.choice(("relu", "hot")))
    d = _row(rng, 64, 4608)
    bits = bits if bits < 8 or d <= 1024 else 4
    return _infer(_log(rng, 64, 4096), d, _log(rng, 1, 2048), bits, rng.randint(2, 6),
                  round(rng.uniform(1.0, 2.0), 2), rng.choice((8, 16)), rng.random() < 0.3, wdist)


# ---------------------------------------------------------------------------------------------
# Inputs (plain torch, from the seed alone)


def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _weights(C, d, wdist, g):
    n = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    if wdist == "normal":                              # Kaiming fan-in
        return n(C, d) * math.sqrt(2.0 / d)
    if wdist == "student":                             # Student-t(4) rows of lognormal scale
        chi = sum(n(C, d).square_() for _ in range(4))
        return n(C, d) / (chi / 4).sqrt_() * math.sqrt(1.0 / d) * (0.5 * n(C, 1)).exp_()
    if wdist == "laplace":
        u = torch.rand(C, d, device="cuda", generator=g) - 0.5
        return -0.05 * u.sign() * torch.log1p(-2 * u.abs().clamp_max_(0.4999999))
    W = n(C, d) * 0.02                                 # 0.1 % of entries 20 times as large
    return torch.where(torch.rand(C, d, device="cuda", generator=g) < 0.001, W * 20, W)


def _calibration(shape, xdist, g):
    X = torch.randn(*shape, device="cuda", generator=g)
    if xdist == "relu":
        return X.relu_()
    hot = torch.randperm(shape[-1], device="cuda", generator=g)[:8]   # 8 large input columns
    X[..., hot] *= 10.0
    return X


def _inputs(c, seed):
    """W and X (None where the case has none) of a case of one layer."""
    W = _weights(c["C"], c["d"], c["wdist"], _gen(seed, 1))
    X = None
    if "N" in c:
        shape = (c["C"], c["N"], c["d"]) if c.get("depthwise") else (c["N"], c["d"])
        X = _calibration(shape, c["xdist"], _gen(seed, 2))
    return W, X


def _shapes(c):
    return [tuple(int(v) for v in s.split("x")) for s in c["layers"].split(",")]


def _network_inputs(c, seed):
    Ws, Xs = [], []
    for i, (C, d) in enumerate(_shapes(c)):
        Ws.append(_weights(C, d, c["wdist"], _gen(seed, 10 + i)))
        Xs.append(_calibration((c["N"], d), "relu", _gen(seed, 1000 + i)))
    return Ws, Xs


def _fractions(c):
    """The caller's own grid of the greedy search: geometric from 1/16 to 1, or None."""
    if c.get("grid", "linear") == "linear":
        return None
    G = c["G"]
    f = [16.0 ** ((g + 1 - G) / G) for g in range(G)]
    return torch.tensor(f, dtype=torch.float32).tolist()


def _int8_inputs(c, seed):
    return torch.randint(-128, 128, (c["T"], c["d"]), device="cuda", generator=_gen(seed, 3),
                         dtype=torch.int8)


def _spec(c, C, d):
    return pipeline.LayerSpec(C=C, d=d, N=c["N"], groups=C if c.get("depthwise") else 1,
                              bits=c["bits"], G=c["G"], k_max=c["k_max"],
                              budget_or_eps=c["beta"], center=c.get("center", -1))


def prepare(case, seed):
    c = case
    s = {"case": c}
    if c["kind"] == "network":
        s["Ws"], s["Xs"] = _network_inputs(c, seed)
        net = pipeline.NetworkPlan([_spec(c, C, d) for C, d in _shapes(c)], "cuda", n_streams=12)
        s["net"] = pipeline.CapturedNetwork(net, s["Ws"], s["Xs"])
        return s
    W, X = _inputs(c, seed)
    C, d = W.shape
    s.update(W=W, X=X)
    if c["kind"] == "layer":
        s["plan"] = pipeline.LayerPlan(_spec(c, C, d), "cuda")
    elif c["kind"] == "greedy":
        s["grid"] = _fractions(c)
        s["rmax"] = torch.empty((C, c["k_max"] + 1), device="cuda")
    elif c["kind"] == "output_error":
        s["rmax"] = torch.empty((C, c["k_max"] + 1), device="cuda")
        s["codes"], s["scales"], _, _ = binding.mpq_quantize_layer(W, c["bits"], c["G"],
                                                                   c["k_max"], rmax=s["rmax"])
    elif c["kind"] == "infer":
        center = None
        if c["centered"]:
            center, W = binding.mpq_center_weights(W)
        codes, scales, _, _ = binding.mpq_quantize_layer(W, c["bits"], 64, c["k_max"])
        s["npoints"] = _point_counts(c, seed)
        s["layout"] = binding.mpq_pack_layout(s["npoints"], d, c["k_max"], c["bits"], c["p"],
                                              centered=c["centered"])
        s["packed"] = binding.mpq_pack_points(codes, scales, s["npoints"], s["layout"],
                                              center=center)
        s["X"] = _int8_inputs(c, seed)
        del s["W"]
    return s


def _point_counts(c, seed):
    """Point counts on the host that add up to the budget: one point a channel, the others where
    the output errors had asked for them (here: at random)."""
    g = torch.Generator()
    g.manual_seed(int(seed) % (1 << 62))
    n = torch.ones(c["C"], dtype=torch.int32)
    extra = min(int(c["beta"] * c["C"] + 0.5) - c["C"], c["C"] * (c["k_max"] - 1))
    at = torch.randperm(c["C"] * (c["k_max"] - 1), generator=g)[:max(0, extra)] % c["C"]
    return n.index_add_(0, at, torch.ones_like(at, dtype=torch.int32))


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "layer":
        p = s["plan"].run_device(s["W"], s["X"])
        out = dict(codes=p.codes, scales=p.scales, resid_sq=p.resid_sq, err=p.err,
                   npoints=p.npoints, points_used=p.points_used, W_hat=p.W_hat)
        if p.center is not None:
            out["center"] = p.center
        return out
    if kind == "network":
        net = s["net"].replay()
        return dict(codes=[p.codes for p in net.plans], scales=[p.scales for p in net.plans],
                    err=[p.err for p in net.plans], W_hat=[p.W_hat for p in net.plans],
                    counts=net.counts)
    if kind == "greedy":
        codes, scales, resid_sq, _ = binding.mpq_quantize_layer(
            s["W"], c["bits"], c["G"], c["k_max"], grid_frac=s["grid"], rmax=s["rmax"])
        return dict(codes=codes, scales=scales, resid_sq=resid_sq, rmax=s["rmax"])
    if kind == "output_error":
        return binding.mpq_output_error(s["X"], s["W"], s["codes"], s["scales"], c["k_max"],
                                        rmax=s["rmax"])
    if kind == "adaptive":
        codes, scales, resid_sq, ncand = binding.mpq_quantize_layer_adaptive(
            s["W"], c["bits"], c["k_max"], eta=ETA, max_cand=1 << 62)
        return dict(codes=codes, scales=scales, resid_sq=resid_sq, ncand=ncand)
    if kind == "clip":
        clip, err, best = binding.mpq_clip_search(
            s["X"], s["W"], c["bits"], n_cand=c["n_cand"],
            mode=binding.MPQ_CLIP_PER_LAYER if c["per_layer"] else binding.MPQ_CLIP_PER_CHANNEL)
        return dict(clip=clip, err=err, best=best)
    return binding.mpq_multipoint_linear(s["X"], s["layout"], s["packed"])


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without


def _greedy_bytes(C, d, k):
    return C * (4 * d + k * d + 4 * k + 4 * (k + 1))


def _layer_work(C, d, N, k, depthwise=False, center=-1):
    b = _greedy_bytes(C, d, k) + 4 * N * d * (C if depthwise else 1)
    b += C * (4 * (k + 1) + 4 + 4 * d) + (4 * C if center >= 0 else 0)
    return b, 2 * N * d * C * (k + 1)


def work(case):
    c = case
    if c["kind"] == "network":
        b = [_layer_work(C, d, c["N"], c["k_max"]) for C, d in _shapes(c)]
        return {"bytes": sum(x for x, _ in b), "flops": sum(y for _, y in b)}
    C, d = c["C"], c["d"]
    if c["kind"] == "layer":
        b, f = _layer_work(C, d, c["N"], c["k_max"], c["depthwise"], c["center"])
        return {"bytes": b, "flops": f}
    if c["kind"] == "greedy":
        return {"bytes": _greedy_bytes(C, d, c["k_max"]) + 4 * C * (c["k_max"] + 1), "flops": 0}
    if c["kind"] == "output_error":
        k = c["k_max"]
        return {"bytes": 4 * c["N"] * d + C * (4 * d + k * d + 4 * k + 8 * (k + 1)),
                "flops": 2 * c["N"] * d * C * (k + 1)}
    if c["kind"] == "adaptive":
        return {"bytes": _greedy_bytes(C, d, c["k_max"]) + 8 * C * c["k_max"], "flops": 0}
    if c["kind"] == "clip":
        return {"bytes": 4 * c["N"] * d + 4 * C * d + C * (8 * c["n_cand"] + 4),
                "flops": 2 * c["N"] * d * C * c["n_cand"]}
    points = int(_point_counts(c, 0).sum())
    return {"bytes": c["T"] * d + points * d + 4 * C * c["T"], "flops": 2 * points * d * c["T"]}


def tolerance(case):
    """Codes, scales and counts are decisions on exact quantities and the same for any correct
    implementation; sums are not.  Output errors are means of squared 22-bit dot products with
    32-bit sums: 3e-6 off their 64-bit values where measured; squared norms are 32-bit sums."""
    if case["kind"] == "infer":
        return "exact"
    if case["kind"] in ("greedy", "adaptive"):
        return {"rel": 1e-6, "max": 1e-5}
    return {"rel": 1.2e-5, "max": 5e-5}


# ---------------------------------------------------------------------------------------------
# The same results in plain torch, 64-bit sums


def _div(a, b):
    """One correctly rounded fp32 division (a Python divisor would become a reciprocal)."""
    return a / torch.full_like(a, b)


def _codes_at(r, s, qmax):
    q = (r / s).round_().clamp_(-qmax, qmax)           # correctly rounded fp32 division, ties even
    return torch.where(s > 0, q, torch.zeros_like(q))


def _update(r, s, q):
    """fmaf(-s, q, r): the product is exact in 64 bits."""
    return (r.double() - s.double() * q.double()).float()


def _sq(r):
    return r.double().square().sum(1)


def _exact_greedy(W, bits, G, k_max, frac=None):
    """codes [k][C][d], scales [C][k], resid_sq [C][k+1], the last residuals' list [k+1][C][d]."""
    qmax = 2 ** (bits - 1) - 1
    f = _div(torch.arange(1, G + 1, device="cuda", dtype=torch.float32), G) if frac is None \
        else torch.tensor(frac, device="cuda", dtype=torch.float32)
    C, d = W.shape
    codes = torch.empty((k_max, C, d), dtype=torch.int8, device="cuda")
    scales = torch.empty((C, k_max), device="cuda")
    sq = torch.empty((C, k_max + 1), dtype=torch.float64, device="cuda")
    rmax = torch.empty((C, k_max + 1), device="cuda")
    step = max(1, (1 << 23) // d)                      # rows at a time: in L2 for all candidates
    for c0 in range(0, C, step):
        r = W[c0:c0 + step].clone()
        at = slice(c0, c0 + r.shape[0])
        sq[at, 0], rmax[at, 0] = _sq(r), r.abs().amax(1)
        for i in range(k_max):
            smax = _div(rmax[at, i], qmax)
            best = torch.full_like(sq[at, 0], math.inf)
            s_best = torch.zeros_like(smax)
            for g in range(G):
                s = f[g] * smax
                q = _codes_at(r, s[:, None], qmax)
                e = torch.addcmul(r.double(), s.double()[:, None], q.double(), value=-1)
                e = e.square_().sum(1)
                less = e < best
                best, s_best = torch.where(less, e, best), torch.where(less, s, s_best)
            q = _codes_at(r, s_best[:, None], qmax)
            r = _update(r, s_best[:, None], q)
            codes[i, at], scales[at, i] = q.to(torch.int8), s_best
            sq[at, i + 1], rmax[at, i + 1] = _sq(r), r.abs().amax(1)
    return codes, scales, sq, rmax


def _exact_error(X, W, codes, scales):
    """Eq. 11 for n = 0..k_max; X [N][d], or [C][N][d] with a block per channel."""
    k_max, C, d = codes.shape
    Xd = X.double()
    r, err = W, []
    for n in range(k_max + 1):
        if n:
            r = _update(r, scales[:, n - 1:n], codes[n - 1])
        if X.dim() == 3:
            y = torch.einsum("cnd,cd->cn", Xd, r.double())
        else:
            y = r.double() @ Xd.t()
        err.append(y.square().mean(1))
    return torch.stack(err, 1)


def _exact_counts(err, k_max, beta):
    """Budget mode of Algorithm 2 on an fp32 error table (C [k_max+1])."""
    e = err.float().cpu()
    C = e.shape[0]
    gain = (e[:, 1:-1] - e[:, 2:]).tolist()
    n = [1] * C
    extra = max(0, min(int(math.floor(beta * C + 0.5)) - C, C * (k_max - 1)))
    import heapq
    heap = [(-gain[c][0], c) for c in range(C)] if k_max > 1 else []
    heapq.heapify(heap)
    while extra and heap and heap[0][0] < 0:
        _, c = heapq.heappop(heap)
        n[c] += 1
        extra -= 1
        if n[c] < k_max:
            heapq.heappush(heap, (-gain[c][n[c] - 1], c))
    return torch.tensor(n, dtype=torch.int32, device="cuda")


def _exact_weights(codes, scales, n, center):
    acc = torch.zeros_like(codes[0], dtype=torch.float64)
    if center is not None:
        acc += center.double()[:, None]
    for i in range(codes.shape[0]):
        term = scales[:, i:i + 1].double() * codes[i].double()
        acc += torch.where((n > i)[:, None], term, torch.zeros_like(term))
    return acc


def _exact_center(W, mode):
    lo, hi = W.amin(1).double(), W.amax(1).double()
    if mode == 1:
        lo, hi = lo.amin().expand_as(lo), hi.amax().expand_as(hi)
    B = ((lo + hi) / 2).float()
    return B, W - B[:, None]


def _exact_layer(c, W, X):
    center = None
    if c.get("center", -1) >= 0:
        center, W = _exact_center(W, c["center"])
    codes, scales, sq, _ = _exact_greedy(W, c["bits"], c["G"], c["k_max"])
    err = _exact_error(X, W, codes, scales)
    n = _exact_counts(err, c["k_max"], c["beta"])
    out = dict(codes=codes, scales=scales, resid_sq=sq, err=err, npoints=n,
               points_used=n.sum(dtype=torch.int32).reshape(1),
               W_hat=_exact_weights(codes, scales, n, center))
    if center is not None:
        out["center"] = center
    return out


def _exact_adaptive(W, bits, k_max):
    """Each step's minimiser over the grid s_m = fl32(m gamma / Qmax), m = 1..M: the objective is
    a quadratic between the scales where a code changes, so the best grid points lie next to the
    pieces' minimisers.  The pieces come from 64-bit sums, the winner is evaluated directly."""
    qmax = 2 ** (bits - 1) - 1
    C, d = W.shape
    codes = torch.zeros((k_max, C, d), dtype=torch.int8, device="cuda")
    scales = torch.zeros((C, k_max), device="cuda")
    sq = torch.zeros((C, k_max + 1), dtype=torch.float64, device="cuda")
    ncand = torch.zeros((C, k_max), dtype=torch.int64, device="cuda")
    levels = torch.arange(1, qmax + 1, device="cuda", dtype=torch.float64)
    for k in range(C):
        r = W[k].clone()
        sq[k, 0] = r.double().square().sum()
        for i in range(k_max):
            a = r.double().abs()
            norm2 = float(a.square().sum())
            if not norm2:
                break
            distinct = torch.unique(a)
            gap = float((distinct[1:] - distinct[:-1]).min()) / 2 if distinct.numel() > 1 \
                else math.inf
            gamma = min(gap / qmax, ETA)
            M = int(math.floor(2 * qmax * math.sqrt(norm2) / gamma))
            ncand[k, i] = M
            # thresholds in decreasing order: below the t-th, the first t codes have risen
            tau = (a[:, None] / (levels - 0.5)).reshape(-1)
            tau, order = tau.sort(descending=True)
            P = a[:, None].expand(d, qmax).reshape(-1)[order].cumsum(0)
            N = (2 * levels - 1).expand(d, qmax).reshape(-1)[order].cumsum(0)
            low = torch.cat((tau[1:], tau.new_zeros(1)))
            s = torch.minimum(torch.maximum(P / N, low), tau)
            obj = s * (s * N - 2 * P)
            top = torch.topk(-obj, min(16, obj.numel())).indices
            m = (s[top] * (qmax / gamma)).floor()
            spread = max(1.0, float(s[top[0]]) * 2.0 ** -24 * qmax / gamma)
            m = m[:, None] + spread * torch.arange(-3, 5, device="cuda", dtype=torch.float64)
            m = m.floor().clamp(1, M).reshape(-1).unique()
            cand = (m * gamma / qmax).float()
            q = (r[None] / cand[:, None]).round_().clamp_(-qmax, qmax)
            e = (r.double()[None] - cand.double()[:, None] * q.double()).square().sum(1)
            best = int(torch.argmin(e))
            codes[i, k], scales[k, i] = q[best].to(torch.int8), cand[best]
            r = _update(r, cand[best], q[best])
            sq[k, i + 1] = r.double().square().sum()
    return dict(codes=codes, scales=scales, resid_sq=sq, ncand=ncand)


def _exact_clip(c, W, X):
    qmax = 2 ** (c["bits"] - 1) - 1
    n = c["n_cand"]
    f = _div(torch.arange(1, n + 1, device="cuda", dtype=torch.float32), n)
    m = W.abs().amax(1)
    if c["per_layer"]:
        m = m.amax().expand_as(m)
    K = f[None] * m[:, None]
    Xd = X.double().t()
    err = torch.empty((W.shape[0], n), dtype=torch.float64, device="cuda")
    for j in range(n):
        s = _div(K[:, j], qmax)[:, None]
        r = _update(W, s, _codes_at(W, s, qmax))
        err[:, j] = (r.double() @ Xd).square().mean(1)
    best = (err.float().double().sum(0).argmin().expand(W.shape[0]) if c["per_layer"]
            else err.argmin(1)).to(torch.int32)
    return dict(clip=K, err=err, best=best)


def _exact_infer(c, seed):
    W = _weights(c["C"], c["d"], c["wdist"], _gen(seed, 1))
    center = None
    if c["centered"]:
        center, W = _exact_center(W, 0)
    codes, scales, _, _ = _exact_greedy(W, c["bits"], 64, c["k_max"])
    n = _point_counts(c, seed).cuda()
    X = _int8_inputs(c, seed).double()
    y = torch.zeros((c["C"], c["T"]), dtype=torch.float64, device="cuda")
    for i in range(c["k_max"]):                        # whole numbers far below 2^53: exact
        A = (scales[:, i].double() * 2.0 ** c["p"]).round()
        A = torch.where(n > i, A, torch.zeros_like(A))
        y += A[:, None] * (codes[i].double() @ X.t())
    if center is not None:
        y += (center.double() * 2.0 ** c["p"]).round()[:, None] * X.sum(1)[None]
    y = (y / 2.0 ** c["p"]).floor()
    return y.clamp(-2.0 ** 31, 2.0 ** 31 - 1).to(torch.int32)


def exact(case, seed):
    c = case
    if c["kind"] == "infer":
        return _exact_infer(c, seed)
    if c["kind"] == "network":
        Ws, Xs = _network_inputs(c, seed)
        o = [_exact_layer(c, W, X) for W, X in zip(Ws, Xs)]
        counts = torch.cat([x["npoints"] for x in o] + [x["points_used"] for x in o])
        return dict(codes=[x["codes"] for x in o], scales=[x["scales"] for x in o],
                    err=[x["err"] for x in o], W_hat=[x["W_hat"] for x in o], counts=counts)
    W, X = _inputs(c, seed)
    if c["kind"] == "layer":
        return _exact_layer(c, W, X)
    if c["kind"] == "adaptive":
        return _exact_adaptive(W, c["bits"], c["k_max"])
    if c["kind"] == "clip":
        return _exact_clip(c, W, X)
    codes, scales, sq, rmax = _exact_greedy(W, c["bits"], c["G"], c["k_max"], _fractions(c))
    if c["kind"] == "greedy":
        return dict(codes=codes, scales=scales, resid_sq=sq, rmax=rmax)
    return _exact_error(X, W, codes, scales)
