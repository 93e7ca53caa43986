"""The calls this package is measured on: error-feedback compression steps and
their exchange, through the public functions of the package.

A case is what one worker, or n workers simulated on one GPU, do in an
iteration of distributed EF-SGD:

  ht          ef_hard_threshold on each worker's gradient
  topk        ef_topk on each worker's gradient
  layerwise   ef_topk_layerwise on each worker's gradient
  round       ef_scaled_round on each worker's gradient, then int_aggregate
  exchange    no compression: the n workers' messages are there already

followed, for "then" = "sum" or "update" (not for round), by
sparse_aggregate or sparse_aggregate_apply (momentum form) of the messages.

Inputs. Gradients are seeded noise shaped like the workloads of this package:
per-tensor scales, the workload's distribution, the embedding's zero rows. A
training loop gives the step another gradient at every iteration, so each pass
takes a window of the gradient buffer that is a few thousand coordinates
further on: the residual then does the random walk it does in training, and
the share of coordinates sent stays where it is however often a state is run.
The error memory starts in that walk's stationary distribution: a walk of
step variance v from 0, reset to 0 where it leaves (-lambda, lambda), is
triangular on (-lambda, lambda), and leaves at the rate
v / (lambda^2 + 2 lambda o + v) with o its mean overshoot (Wald's identity;
exact for Laplace steps).
"""
import math

import numpy as np
import torch

import paper_2108_00951_gb300 as efs
from paper_2108_00951_gb300 import workloads

DEV = "cuda"
GAMMA = float(np.float32(0.1))
MU, LR = float(np.float32(0.9)), float(np.float32(0.01))
SHIFTS = 4096                 # windows of the gradient buffer, 8 coordinates apart
PAD = 8 * SHIFTS
EMB = 650                     # width of the LSTM workload's embedding rows

# step variance and mean overshoot, at scale 1
VARIANCE = {"gauss": 1.0, "laplace": 2.0, "student": 3.0, "outlier": 2.0}
OVERSHOOT = {"gauss": 0.58, "laplace": 1.0, "student": 1.3, "outlier": 0.7}


# ------------------------------------------------------------------- cases
def _case(name, kind, d, **more):
    c = {"name": name, "kind": kind, "d": d, "n": 1, "dtype": "f32", "dist": "laplace",
         "shape": "", "segments": 1, "decades": 0.0, "scale": 1e-3, "lam": 0.0, "density": 0.0,
         "rows": False, "norm": False, "tiles": False, "then": ""}
    c.update(more)
    return c


def listed():
    by = workloads.BY_NAME
    return [
        # the smallest calls: a logistic-regression-sized model, one whole
        # iteration of 4 workers and the model update; everything is latency
        _case("lr_step", "ht", by["lr"].d, n=4, dist="gauss", scale=0.01, lam=2e-3,
              then="update"),
        # the same size under Top-k (1 %), with the error norm that the
        # convex experiments record at every step
        _case("lr_topk", "topk", by["lr"].d, dist="gauss", scale=0.01, density=0.01, norm=True),
        # CIFAR-10 training of a ResNet-18: an iteration of 8 workers with
        # tile indexes, and the momentum update
        _case("resnet18_step", "ht", by["resnet18"].d, n=8, shape="resnet18", decades=3.0,
              scale=1e-2, lam=2.7e-3, tiles=True, then="update"),
        # the same model compressed layer by layer (0.1 % of each of its 62 tensors)
        _case("resnet18_layerwise", "layerwise", by["resnet18"].d, shape="resnet18",
              decades=3.0, scale=1e-2, density=1e-3),
        # the LSTM language model: Top-k at 1 % of 28.9 M, embedding rows
        # mostly zero
        _case("lstm_topk", "topk", by["lstm"].d, shape="lstm", dist="student", density=1e-2),
        # the LSTM workers' gradients and error memories kept as rows of one
        # [n, d] matrix (as this package's EF-SGD loop keeps them): d is odd,
        # so rows start at any multiple of 4 bytes; then the exchange
        _case("lstm_rows_ht", "ht", by["lstm"].d, n=4, shape="lstm", dist="student",
              lam=4.1e-4, rows=True, then="sum"),
        # ResNet-50 at the smallest threshold of its sweep: the densest messages
        _case("resnet50_ht", "ht", by["resnet50"].d, shape="resnet50", dist="outlier",
              decades=4.0, scale=1e-2, lam=1e-4),
        # the exchange of 16 workers' Top-k messages (1 %) without tile indexes
        _case("resnet50_exchange", "exchange", by["resnet50"].d, n=16, shape="resnet50",
              decades=4.0, scale=1e-2, density=1e-2, then="sum"),
        # the largest vector: one worker's step, fp32 and bf16 gradients
        _case("vgg16_ht", "ht", by["vgg16"].d, shape="vgg16", decades=0.6, scale=2e-4,
              lam=1.584e-4),
        _case("vgg16_ht_bf16", "ht", by["vgg16"].d, shape="vgg16", decades=0.6, scale=2e-4,
              lam=1.584e-4, dtype="bf16"),
        # the exchange of 8 workers' hard-threshold messages on it
        _case("vgg16_exchange", "exchange", by["vgg16"].d, n=8, shape="vgg16", decades=0.6,
              scale=2e-4, density=0.05, tiles=True, then="sum"),
        # scaled integer rounding of 8 workers on ResNet-18, and its exact exchange
        _case("resnet18_round", "round", by["resnet18"].d, n=8, shape="resnet18", decades=3.0,
              scale=1e-2),
    ]


def draw(rng):
    """A call of the same kinds anywhere in their ranges: vectors from 500
    coordinates (the smallest convex problem) to VGG-16's, mostly not
    multiples of anything, 1 to 16 workers, densities from 1e-4 to 0.25."""
    kind = rng.choice(["ht", "ht", "ht", "topk", "topk", "layerwise", "exchange", "round"])
    n = rng.choice([1, 1, 2, 3, 4, 8, 16]) if kind != "exchange" else rng.choice([2, 4, 5, 8, 16])
    d = int(math.exp(rng.uniform(math.log(500), math.log(138_357_544 // n))))
    if rng.random() < 0.25:
        d = max(8, d // 8 * 8)
    low, high = {"ht": (1e-4, 0.25), "exchange": (1e-4, 0.1)}.get(kind, (1e-4, 1e-2))
    c = _case("", kind, d, n=n,
              dtype=rng.choice(["f32", "f32", "bf16"]),
              dist=rng.choice(["gauss", "laplace", "student"]),
              segments=min(d, int(math.exp(rng.uniform(0.0, math.log(200))))),
              decades=round(rng.uniform(0.0, 3.0), 2), scale=1e-2,
              density=float("%.3g" % math.exp(rng.uniform(math.log(low), math.log(high)))),
              rows=n > 1 and kind != "exchange" and rng.random() < 0.4,
              norm=kind in ("ht", "topk") and rng.random() < 0.2,
              then=rng.choice(["", "sum", "update"]) if n > 1 else "")
    if kind == "exchange":
        c["then"] = rng.choice(["sum", "update"])
    if kind == "round":
        c["then"], c["density"] = "", 0.0
    c["tiles"] = kind in ("ht", "exchange") and c["then"] != "" and rng.random() < 0.5
    while work(c)["bytes"] > 1.8e9:   # no more than the largest listed case
        c["d"] = c["d"] * 3 // 4
    del c["name"]
    return c


# ------------------------------------------------------------------- model
def _sizes(case):
    """The tensors of the vector, in order."""
    if case["shape"]:
        return list(workloads.BY_NAME[case["shape"]].segments)
    n, d = case["segments"], case["d"]
    if n == 1:
        return [d]
    # lengths spread over four decades, as a model's tensors are
    w = np.random.RandomState(d % 2**31).uniform(0.0, 4.0, n)
    cut = np.floor(np.cumsum(10.0**w) / np.sum(10.0**w) * (d - n)).astype(np.int64)
    ends = cut + np.arange(1, n + 1)
    ends[-1] = d
    return np.diff(np.concatenate([[0], ends])).tolist()


def _scales(case):
    """One scale per tensor, log-uniform over the case's decades below
    `scale`, a property of the model and not of the seed."""
    if case["shape"]:
        seed = workloads.BY_NAME[case["shape"]].seed
    else:
        seed = case["d"]
    u = torch.rand(len(_sizes(case)), generator=torch.Generator().manual_seed(seed),
                   dtype=torch.float64).numpy()
    return case["scale"] * 10.0 ** ((u - 1.0) * case["decades"])


def _variances(case):
    v = np.full(len(_sizes(case)), VARIANCE[case["dist"]])
    if case["shape"] == "lstm":
        v[0] *= 0.05   # the embedding: 95 % of its rows are zero at each step
    return v


def _rate(lam, scale, v, o):
    """Share sent per step by coordinates of step scale gamma * scale."""
    x = lam / (GAMMA * scale)
    return v / (x * x + 2.0 * x * o + v)


def _thresholds(case):
    """Per tensor: the magnitude at which coordinates are sent in the
    stationary state, and the share sent per step."""
    size = np.asarray(_sizes(case), dtype=np.float64)
    s, v, o = _scales(case), _variances(case), OVERSHOOT[case["dist"]]
    if case["kind"] == "round":
        return np.zeros_like(size), np.ones_like(size)
    if case["kind"] == "layerwise":
        lam = np.empty_like(s)
        for i in range(len(s)):
            want = min(1.0, max(case["density"], 1.0 / size[i]))
            lam[i] = _solve(lambda x: _rate(x, s[i], v[i], o), want, s[i])
        return lam, _rate(lam, s, v, o)
    lam = case["lam"]
    if lam == 0.0:
        lam = _solve(lambda x: float(np.sum(size * _rate(x, s, v, o)) / np.sum(size)),
                     case["density"], float(s.max()))
    lam = float(np.float32(lam))
    return np.full_like(s, lam), _rate(lam, s, v, o)


def _solve(f, want, scale):
    lo, hi = 1e-9 * scale, 1e3 * scale   # f falls from 1 to 0
    for _ in range(80):
        mid = math.sqrt(lo * hi)
        lo, hi = (mid, hi) if f(mid) > want else (lo, mid)
    return math.sqrt(lo * hi)


def _budget(case):
    """Top-k: k; layer-wise: (segment ends, k per segment)."""
    if case["kind"] == "topk":
        return max(1, int(case["density"] * case["d"]))
    size = _sizes(case)
    return (np.cumsum(size).astype(np.uint64),
            np.array([max(1, int(case["density"] * m)) for m in size], dtype=np.uint64))


def _spread(values, case):
    """Per-tensor values as a per-coordinate tensor."""
    v = torch.as_tensor(np.asarray(values), dtype=torch.float32, device=DEV)
    if v.numel() == 1:
        return v
    return torch.repeat_interleave(v, torch.as_tensor(_sizes(case), device=DEV),
                                   output_size=case["d"])


def _noise(case, gen):
    d = case["d"]
    if case["dist"] == "laplace":
        x = torch.empty(d, device=DEV).exponential_(generator=gen)
        x = torch.where(torch.rand(d, device=DEV, generator=gen) < 0.5, -x, x)
    elif case["dist"] == "student":
        x = torch.randn(d, device=DEV, generator=gen)
        chi = torch.randn(d, device=DEV, generator=gen).square_()
        for _ in range(2):
            chi += torch.randn(d, device=DEV, generator=gen).square_()
        x /= torch.sqrt_(chi / 3.0)
    else:
        x = torch.randn(d, device=DEV, generator=gen)
        if case["dist"] == "outlier":
            far = torch.rand(d, device=DEV, generator=gen) < 1e-4
            x = torch.where(far, 100.0 * torch.randn(d, device=DEV, generator=gen), x)
    if case["shape"] == "lstm":
        rows = _sizes(case)[0] // EMB
        zero = torch.rand(rows, device=DEV, generator=gen) < 0.95
        x[:rows * EMB].view(rows, EMB).masked_fill_(zero[:, None], 0.0)
    return x


def _generator(seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    return gen


# ----------------------------------------------------------------- prepare
def prepare(case, seed):
    gen = _generator(seed)
    return _messages(case, gen) if case["kind"] == "exchange" else _workers(case, gen)


def _workers(case, gen):
    d, n, kind = case["d"], case["n"], case["kind"]
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    scale = _spread(_scales(case), case)
    lam, rate = _thresholds(case)
    lam_j = _spread(lam, case)
    rate_j = _spread(rate, case)
    if case["rows"]:
        gbuf = torch.empty(n * d + PAD, dtype=dtype, device=DEV)
        emat = torch.empty(n, d, device=DEV)
        gbufs, e = [gbuf[w * d:(w + 1) * d] for w in range(n)], list(emat.unbind(0))
    else:
        gbufs = [torch.empty(d + PAD, dtype=dtype, device=DEV) for _ in range(n)]
        e = [torch.empty(d, device=DEV) for _ in range(n)]
    for w in range(n):
        gbufs[w][:d] = _noise(case, gen).mul_(scale)
        if not case["rows"]:
            gbufs[w][d:] = gbufs[w][:PAD] if d >= PAD else gbufs[w][:d].repeat(
                -(-PAD // d))[:PAD]
        if kind == "round":   # residuals of rounding to the grid
            e[w].uniform_(-2.0**-21, 2.0**-21, generator=gen)
        else:                 # just sent, or somewhere on the triangle
            tri = torch.rand(d, device=DEV, generator=gen)
            tri -= torch.rand(d, device=DEV, generator=gen)
            tri *= lam_j
            sent = torch.rand(d, device=DEV, generator=gen) < rate_j
            e[w].copy_(tri.masked_fill_(sent, 0.0))
    if case["rows"]:
        m = n * d
        gbuf[m:] = gbuf[:PAD] if m >= PAD else gbuf[:m].repeat(-(-PAD // m))[:PAD]
    s = {"case": case, "t": 0, "e": e, "gbufs": [gbuf] if case["rows"] else gbufs}
    if kind == "round":
        s["q"] = [torch.zeros(d, dtype=torch.int32, device=DEV) for _ in range(n)]
        s["unsent"] = torch.zeros(n, dtype=torch.int32, device=DEV)
        s["dense"] = torch.zeros(d, device=DEV)
        return s
    room = d
    if kind == "topk":
        s["k"] = room = _budget(case)
    elif kind == "layerwise":
        s["ends"], s["ks"] = _budget(case)
        room = int(s["ks"].sum())
    else:
        s["lam"] = float(lam[0])
    s["idx"] = [torch.zeros(room, dtype=torch.int32, device=DEV) for _ in range(n)]
    s["val"] = [torch.zeros(room, device=DEV) for _ in range(n)]
    s["counts"] = torch.zeros(n, dtype=torch.int32, device=DEV)
    s["count"] = [s["counts"][w:w + 1] for w in range(n)]
    s["tiles"] = [torch.zeros(efs.tiles_for(d), dtype=torch.int32, device=DEV)
                  for _ in range(n)] if case["tiles"] else None
    s["err"] = torch.zeros(n, dtype=torch.float64, device=DEV) if case["norm"] else None
    _model(s, gen)
    return s


def _model(s, gen):
    case = s["case"]
    if case["then"] == "sum":
        s["dense"] = torch.zeros(case["d"], device=DEV)
    elif case["then"] == "update":
        s["x"] = torch.randn(case["d"], device=DEV, generator=gen)
        s["m"] = torch.randn(case["d"], device=DEV, generator=gen) * 1e-4


def _messages(case, gen):
    """Messages as the compression leaves them: each tensor's coordinates sent
    at its stationary rate, the values just beyond the threshold."""
    d, n = case["d"], case["n"]
    lam, rate = _thresholds(case)
    rate_j = _spread(rate, case)
    s = {"case": case, "idx": [], "val": [], "tiles": [] if case["tiles"] else None}
    edges = torch.arange(efs.tiles_for(d) - 1, device=DEV) * efs.TILE
    for _ in range(n):
        j = torch.nonzero(torch.rand(d, device=DEV, generator=gen) < rate_j).flatten()
        if j.numel() == 0:
            j = torch.zeros(1, dtype=torch.int64, device=DEV)
        v = torch.empty(j.numel(), device=DEV).exponential_(generator=gen)
        v = (v * 0.1 + 1.0) * float(lam[0])
        v = torch.where(torch.rand(v.numel(), device=DEV, generator=gen) < 0.5, -v, v)
        s["idx"].append(j.to(torch.int32))
        s["val"].append(v)
        if case["tiles"]:
            first = torch.searchsorted(j, edges)
            s["tiles"].append(torch.cat([first, first.new_tensor([j.numel()])]).to(torch.int32))
    s["counts"] = torch.tensor([j.numel() for j in s["idx"]], dtype=torch.int32, device=DEV)
    _model(s, gen)
    return s


# --------------------------------------------------------------------- run
def _gradients(s, t):
    """The iteration's gradients, one per worker."""
    case, o = s["case"], 8 * (t * 2531 % SHIFTS)
    d, n = case["d"], case["n"]
    if case["rows"]:
        return s["gbufs"][0][o:o + n * d].view(n, d).unbind(0)
    return [g[o:o + d] for g in s["gbufs"]]


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    d, n = case["d"], case["n"]
    if kind != "exchange":
        g, e = _gradients(s, s["t"]), s["e"]
        s["t"] += 1
    if kind == "round":
        for w in range(n):
            efs.ef_scaled_round(g[w], e[w], GAMMA, 20, s["q"][w], s["unsent"][w:w + 1])
        efs.int_aggregate(s["q"], d, 20, s["dense"])
        return {"q": s["q"], "unsent": s["unsent"], "e": e, "dense": s["dense"]}
    out = {}
    if kind != "exchange":
        for w in range(n):
            err = None if s["err"] is None else s["err"][w:w + 1]
            to = (s["idx"][w], s["val"][w], s["count"][w])
            if kind == "ht":
                efs.ef_hard_threshold(g[w], e[w], GAMMA, s["lam"], *to, err_sq_out=err,
                                      tiles_out=s["tiles"][w] if s["tiles"] else None)
            elif kind == "topk":
                efs.ef_topk(g[w], e[w], GAMMA, s["k"], *to, err_sq_out=err)
            else:
                efs.ef_topk_layerwise(g[w], e[w], GAMMA, s["ends"], s["ks"], *to,
                                      err_sq_out=err)
        out = {"idx": s["idx"], "val": s["val"], "counts": s["counts"], "e": e}
        if s["tiles"]:
            out["tiles"] = s["tiles"]
        if s["err"] is not None:
            out["err"] = s["err"]
    if case["then"] == "sum":
        efs.sparse_aggregate(s["idx"], s["val"], s["counts"], d, s["dense"], tiles=s["tiles"])
        out["dense"] = s["dense"]
    elif case["then"] == "update":
        efs.sparse_aggregate_apply(s["idx"], s["val"], s["counts"], d, 1.0 / n, s["x"],
                                   m=s["m"], momentum=MU, lr=LR, tiles=s["tiles"])
        out["x"], out["m"] = s["x"], s["m"]
    return out


# -------------------------------------------------------------------- work
def _sent(case):
    """Pairs in one worker's message."""
    if case["kind"] == "topk":
        return _budget(case)
    if case["kind"] == "layerwise":
        return int(_budget(case)[1].sum())
    return int(np.sum(np.asarray(_sizes(case)) * _thresholds(case)[1]))


def work(case):
    d, n, kind = case["d"], case["n"], case["kind"]
    wide = 2 if case["dtype"] == "bf16" else 4
    if kind == "round":   # read g, e; write e, q; then read n q, write the sum
        return {"bytes": n * d * (wide + 12) + (4 * n + 4) * d, "flops": 5 * n * d}
    sent, size, flops = _sent(case), 0, 0
    if kind != "exchange":
        size += n * (d * (wide + 8) + 8 * sent)
        flops += 2 * n * d
    if case["then"]:
        size += 8 * n * sent + d * (4 if case["then"] == "sum" else 16)
        flops += n * sent + (0 if case["then"] == "sum" else 6 * d)
    return {"bytes": size, "flops": flops}


def tolerance(case):
    # every output is defined to the bit (one fused multiply-add per
    # coordinate, the sums in worker order) but the error norm, an fp32-based
    # sum that is within 1e-6 of the exact one
    return {"rel": 1e-6, "max": 4e-6} if case["norm"] else "exact"


# ------------------------------------------------------------------- exact
def exact(case, seed):
    s = prepare(case, seed)
    d, n, kind = case["d"], case["n"], case["kind"]
    out, sums = {}, torch.zeros(d, dtype=torch.float64, device=DEV)
    if kind == "round":
        out = {"q": [], "unsent": torch.zeros(n, dtype=torch.int32, device=DEV), "e": []}
        for g, e in zip(_gradients(s, 0), s["e"]):
            a = (e.double() + GAMMA * g.double()).float().double()
            q = torch.round(a * 2.0**20)
            out["q"].append(q.to(torch.int32))
            out["e"].append(a - q * 2.0**-20)
            sums += q
        out["dense"] = sums * 2.0**-20
        return out
    if kind == "exchange":
        for j, v in zip(s["idx"], s["val"]):
            sums.index_add_(0, j.long(), v.double())
    else:
        out = {"idx": [], "val": [], "counts": None, "e": []}
        counts, norms, tiles = [], [], []
        for w, (g, e) in enumerate(zip(_gradients(s, 0), s["e"])):
            a = e.double() + GAMMA * g.double()
            size = a.float().abs()   # the definition compares the rounded value
            j = _support(case, s, size)
            idx, val = s["idx"][w].clone(), s["val"][w].double()
            idx[:j.numel()] = j.to(torch.int32)
            val[:j.numel()] = a[j]
            sums[j] += a[j]
            a[j] = 0.0
            out["idx"].append(idx)
            out["val"].append(val)
            out["e"].append(a)
            counts.append(j.numel())
            norms.append(a.square().sum())
            if s["tiles"]:
                edges = torch.arange(efs.tiles_for(d) - 1, device=DEV) * efs.TILE
                first = torch.searchsorted(j, edges)
                tiles.append(torch.cat([first, first.new_tensor([j.numel()])]).to(torch.int32))
        out["counts"] = torch.tensor(counts, dtype=torch.int32, device=DEV)
        if s["tiles"]:
            out["tiles"] = tiles
        if case["norm"]:
            out["err"] = torch.stack(norms)
    if case["then"] == "sum":
        out["dense"] = sums
    elif case["then"] == "update":
        delta = sums * float(np.float32(1.0 / n))
        out["m"] = MU * s["m"].double() + delta
        out["x"] = s["x"].double() - LR * (delta + out["m"])
    return out


def _support(case, s, size):
    """The coordinates sent, ascending; ties to the lowest index."""
    if case["kind"] == "ht":
        return torch.nonzero((size >= s["lam"]) & (size > 0)).flatten()
    if case["kind"] == "topk":
        return _largest(size, s["k"])
    lo, got = 0, []
    for hi, k in zip(s["ends"].tolist(), s["ks"].tolist()):
        got.append(_largest(size[lo:hi], k) + lo)
        lo = hi
    return torch.cat(got)


def _largest(size, k):
    cut = torch.topk(size, k, sorted=True).values[-1]
    above = size > cut
    ties = torch.nonzero(size == cut).flatten()[:k - int(above.sum())]
    return torch.sort(torch.cat([torch.nonzero(above).flatten(), ties])).values
