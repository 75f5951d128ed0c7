"""What the Zeno library is used for, as cases that can be timed.

A case is one call (or one short chain of calls) that a parameter server makes through
`paper_1805_10032_b200.zeno`: the aggregation step of one model and one set of workers, the step with
the update, the server loop, a whole synchronous iteration with the workers' side, and the two baseline
rules on the same candidates.  Shapes come from the benchmark configurations (`synthetic.CONFIGS`),
from the tests' ragged shapes, or are generic sizes between them.

Inputs follow `synthetic.py`: honest rows are a worker's gradient plus noise, faulty rows are sign-flipped
copies, large Gaussian noise or an omniscient-style multiple of the honest mean, and b is the number of
faulty rows.
"""
from __future__ import annotations

import torch

from paper_1805_10032_b200 import synthetic as syn
from paper_1805_10032_b200 import zeno

DEVICE = "cuda"
LARGEST_BYTES = 64 * (1 << 26) * 4          # the candidates of the largest listed case
LARGEST_FLOPS = 1.0e11                      # CUDA-core or tensor operations a drawn case may ask for


def _case(name, call, model, dims, m, n_r, *, dtype="f32", b=None, faults="signflip", gamma=0.1, rho=5e-4,
          std=0.1, tight=False, steps=1, worker_batch=100):
    c = dict(call=call, model=model, dims="-".join(str(v) for v in dims), m=m, b=(2 * m) // 5 if b is None else b,
             n_r=n_r, dtype=dtype, faults=faults, gamma=gamma, rho=rho, std=std, tight=tight, steps=steps,
             worker_batch=worker_batch)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest model: softmax regression on 28 x 28 images, 20 workers, the paper's 4 server samples.
        # Launches and host time are all there is.
        _case("softmax_step", "step", "mlp", (784, 10), 20, 4),
        # The server loop of the same model, 20 iterations enqueued by one call.
        _case("softmax_run", "run", "mlp", (784, 10), 20, 4, steps=20),
        # A whole synchronous iteration on one GPU: the 20 workers' gradients on 100 samples each, the
        # bit-flipping failure, the step and the update.
        _case("softmax_iteration", "iteration", "mlp", (784, 10), 20, 4, faults="bitflip"),
        # The paper's experiment: a small convolutional network, 20 workers, 4 server samples.
        _case("cnn_step", "step", "cnn", (32, 3, 32, 32, 64, 64, 10), 20, 4, std=0.02),
        # The same network with bfloat16 storage, a larger server batch and the update in the same pass.
        _case("cnn_update_bf16", "update", "cnn", (32, 3, 32, 32, 64, 64, 10), 20, 32, dtype="bf16", std=0.02),
        # A fully connected network on flattened 32 x 32 x 3 images (1.8 M parameters), 20 workers.
        _case("mlp_step", "step", "mlp", (3072, 512, 512, 10), 20, 32, faults="noise200"),
        # The same network with 100 workers and 64 server samples, update in place.
        _case("mlp_update_100", "update", "mlp", (3072, 512, 512, 10), 100, 64, b=40, faults="mixed", gamma=0.05,
              rho=1e-3, std=0.02),
        # A network whose sizes are no multiple of anything, with rows packed without padding.
        _case("mlp_ragged", "step", "mlp", (1029, 301, 131, 11), 37, 19, faults="noise200", tight=True),
        # A wide bfloat16 network (37.7 M parameters) with a thousand classes.
        _case("wide_bf16_step", "step", "mlp", (4096, 4096, 4096, 1000), 32, 128, dtype="bf16", b=12, std=0.05),
        # The largest: least squares over 2^26 parameters, 64 workers, 17 GB of candidates.
        _case("least_squares_step", "step", "lsq", (1 << 26, 1), 64, 16, b=24, faults="noise100", gamma=0.01, rho=1e-4,
              std=0.01),
        # The baseline rules the paper compares with, on the candidates of the 1.8 M parameter network.
        _case("median_100", "median", "mlp", (3072, 512, 512, 10), 100, 64, b=40, faults="mixed"),
        _case("krum_20", "krum", "mlp", (3072, 512, 512, 10), 20, 32, faults="noise200"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    def size(lo, hi):                       # two of three as people choose them, one of three odd
        v = log(lo, hi)
        return v if rng.random() < 1 / 3 else max(8, v // 8 * 8)

    while True:
        kind = rng.choice(("softmax", "run", "iteration", "cnn", "cnn", "mlp", "mlp", "mlp_bf16", "lsq", "median", "krum"))
        tight = rng.random() < 0.25
        dtype = rng.choice(("f32", "f32", "bf16"))
        m, n_r = log(5, 128), log(1, 128)
        if kind in ("softmax", "run"):
            c = _case(None, "step" if kind == "softmax" else "run", "mlp", (size(32, 4096), rng.randint(2, 32)), m,
                      log(1, 64), dtype=dtype, faults=rng.choice(("signflip", "noise200")), tight=tight,
                      steps=1 if kind == "softmax" else rng.randint(2, 32))
        elif kind == "iteration":
            c = _case(None, "iteration", "mlp", (size(32, 2048), rng.randint(2, 20)), log(5, 64), log(1, 64), dtype=dtype,
                      faults="bitflip", tight=tight, worker_batch=log(10, 256))
        elif kind == "cnn":
            w = rng.choice((8, 16, 24, 32, rng.randint(5, 40)))
            side = rng.choice((8, 16, 24, 28, 32))
            chans = (w, w, 2 * w, 2 * w) if rng.random() < 2 / 3 else (w, w)
            c = _case(None, rng.choice(("step", "update")), "cnn", (side, rng.choice((1, 3)), *chans, rng.choice((10, 10, 43, 100))),
                      log(5, 64), log(1, 64), dtype=dtype, faults=rng.choice(("signflip", "noise20")), std=0.02, tight=tight)
        elif kind in ("mlp", "mlp_bf16"):
            top = 4096 if kind == "mlp_bf16" else 1024
            hidden = [size(48, top) for _ in range(rng.randint(1, 3))]
            c = _case(None, rng.choice(("step", "update")), "mlp", (size(64, 4096), *hidden, rng.choice((2, 10, 10, 47, 100, 1000))),
                      m, n_r, dtype="bf16" if kind == "mlp_bf16" else "f32", faults=rng.choice(("signflip", "noise200")), std=0.05,
                      tight=tight)
        elif kind == "lsq":
            c = _case(None, "step", "lsq", (size(1 << 14, 1 << 26), 1), m, log(1, 64), faults="noise100", gamma=0.01,
                      rho=1e-4, std=0.01, tight=tight)
        else:
            c = _case(None, kind, "mlp", (size(64, 4096), size(64, 2048), 10), m, 4, dtype=dtype,
                      faults=rng.choice(("signflip", "noise200", "mixed")), tight=tight)
        w = work(c)
        if w["bytes"] <= LARGEST_BYTES and w["flops"] <= LARGEST_FLOPS:
            return c


# ---- inputs ----------------------------------------------------------------------------------------------

def _dims(case):
    return tuple(int(v) for v in case["dims"].split("-"))


def _faults(case):
    b, kind = case["b"], case["faults"]
    if kind == "mixed":                     # half sign-flipped, half omniscient
        return [(b - b // 2, "signflip"), (b // 2, "omniscient")]
    return [(b, kind)]


def _workload(case, seed):
    dims = _dims(case)
    d = syn.param_count(case["model"], dims, case["model"] != "lsq")
    ldv = d if case["tight"] else None
    same = dict(m=case["m"], b=case["b"], n_r=case["n_r"], gamma=case["gamma"], rho=case["rho"],
                honest_std=case["std"], ldv=ldv, device=DEVICE)
    if case["model"] == "lsq":
        return syn.make_lsq_workload("case", seed, d, n_noise=case["b"], noise_std=100.0, **same)
    if case["model"] == "cnn":
        w = syn.make_cnn_workload("case", seed, dims, case["dtype"], faults=_as_signflip(case), **same)
    else:
        w = syn.make_mlp_workload("case", seed, dims, case["dtype"], faults=_as_signflip(case),
                                  x_init="he" if len(dims) > 2 else "normal0.1", **same)
    if case["faults"] == "noise20":         # noise whose models still have finite activations after five layers
        g = torch.Generator(device=DEVICE)
        g.manual_seed(seed + 1)
        for i in torch.nonzero(~w.honest).flatten().tolist():
            w.V[i, :w.d] = torch.randn(w.d, generator=g, device=DEVICE) * 20.0
    return w


def _as_signflip(case):
    return [(c, "signflip" if k in ("noise20", "bitflip") else k) for c, k in _faults(case) if c > 0]


def _inputs(case, seed):
    w = _workload(case, seed)
    s = dict(case=case, w=w)
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed + 104729)
    if case["call"] == "run":
        # candidates of every iteration: gradients of that iteration's worker batches, and its server batch
        T, (n_in, classes) = case["steps"], _dims(case)
        V = torch.empty((T, w.m, w.ldv), dtype=w.V.dtype, device=DEVICE)
        V[0] = w.V
        feats = torch.randn((T, w.n_r, n_in), generator=gen, device=DEVICE)
        labels = torch.randint(0, classes, (T, w.n_r), generator=gen, device=DEVICE, dtype=torch.int32)
        honest = w.honest.to(DEVICE)
        for t in range(1, T):
            wf = torch.randn((100, n_in), generator=gen, device=DEVICE)
            wl = torch.randint(0, classes, (100,), generator=gen, device=DEVICE, dtype=torch.int32)
            g = syn.mlp_gradient(w.x.float(), w.dims, w.has_bias, wf, wl)
            rows = g + torch.randn((w.m, w.d), generator=gen, device=DEVICE) * case["std"]
            bad = -4.0 * g if case["faults"] == "signflip" else 200.0 * torch.randn((w.m, w.d), generator=gen, device=DEVICE)
            V[t, :, :w.d] = torch.where(honest[:, None], rows, bad).to(V.dtype)
            V[t, :, w.d:] = float("nan")
        s.update(V=V, feats=feats, labels=labels)
    if case["call"] == "iteration":
        n, (n_in, classes) = case["worker_batch"], _dims(case)
        s.update(wfeats=torch.randn((w.m, n, n_in), generator=gen, device=DEVICE),
                 wlabels=torch.randint(0, classes, (w.m, n), generator=gen, device=DEVICE, dtype=torch.int32),
                 faulty=torch.nonzero(~w.honest).flatten().to(torch.int32).to(DEVICE))
    return s


def prepare(case, seed):
    """The server's inputs on the GPU and the handle it keeps for its model."""
    s = _inputs(case, seed)
    return dict(s, z=zeno.from_workload(s["w"]))


# ---- the calls -------------------------------------------------------------------------------------------
# The rank order of honest rows whose scores agree to the sixth digit is not an output two correct
# implementations share, so the steps ask for the average and the scores (the selected set shows in the average).

def run(state):
    case, w, z = state["case"], state["w"], state["z"]
    call, g, rho, b = case["call"], case["gamma"], case["rho"], case["b"]
    if call == "step":
        out, scores, _ = z.step(w.x, w.V, w.features, w.targets, g, rho, b, want_idx=False)
        return out, scores
    if call == "update":
        _, scores, _ = z.step_update(w.x, w.V, w.features, w.targets, g, rho, b, want_out=False, want_idx=False)
        return w.x, scores
    if call == "run":
        scores, _ = z.run(w.x, state["V"], state["feats"], state["labels"], g, rho, b)
        return w.x, scores
    if call == "iteration":
        z.worker_gradients(w.x, state["wfeats"], state["wlabels"], w.V)
        z.inject_faults(w.V, state["faulty"], zeno.FAULT_BIT_FLIP)
        _, scores, _ = z.step_update(w.x, w.V, w.features, w.targets, g, rho, b, want_out=False, want_idx=False)
        return w.x, w.V[:, :w.d], scores
    if call == "median":
        return z.median(w.V)
    return z.krum(w.V, b)


# ---- what a pass cannot do without -----------------------------------------------------------------------

def work(case):
    dims, m, b, n_r, T = _dims(case), case["m"], case["b"], case["n_r"], case["steps"]
    model = case["model"]
    d = syn.param_count(model, dims, model != "lsq")
    esz = 2 if case["dtype"] == "bf16" else 4
    if model == "cnn":
        side, chans, macs = dims[0], dims[1:-1], 0
        for l in range(1, len(chans)):
            macs += 9 * chans[l] * chans[l - 1] * side * side
            side //= 2 if l % 2 == 0 else 1
        macs += dims[-1] * chans[-1] * side * side
        feat = dims[1] * dims[0] ** 2
    else:
        macs = sum(dims[l] * dims[l + 1] for l in range(len(dims) - 1))
        feat = dims[0]
    if case["call"] == "median":            # one comparison an entry at the very least
        return {"bytes": m * d * esz + 4 * d, "flops": m * d}
    if case["call"] == "krum":              # difference, product, sum of every pair
        return {"bytes": m * d * esz + 4 * d + 4 * m, "flops": 3 * d * m * (m - 1) // 2}
    # scores: every model on every sample, the norms; the average of the rows that are kept
    bytes_ = m * d * esz + d * esz + n_r * (feat + 1) * 4 + (d * 4 if case["call"] == "step" else d * esz) + m * 4
    flops = 2 * (m + 1) * n_r * macs + 2 * m * d + (m - b) * d
    if case["call"] == "iteration":         # logits and weight gradients of every worker's samples; V is written first
        n = case["worker_batch"]
        return {"bytes": bytes_ + m * n * (feat + 1) * 4, "flops": flops + 4 * m * n * macs}
    return {"bytes": bytes_ * T, "flops": flops * T}


def tolerance(case):
    """Measured as the distance of the scores from a float64 evaluation of the same inputs (up to 1.5e-5 of
    their norm: a score is a difference of losses up to a hundred times larger) and as the distance between
    the tensor-core and the CUDA-core kernels, times about four."""
    if case["call"] == "median":            # a selection: the value of an entry, or the half sum of two
        return "exact"
    if case["dtype"] == "bf16" and case["call"] in ("update", "run", "iteration"):
        # results stored as bfloat16: where two binary32 values lie on the two sides of a rounding boundary
        # an entry moves by one spacing, 2^-8 of its value
        return {"rel": 1e-3, "max": 2e-2}
    return {"rel": 5e-5}


# ---- the same outputs in 64 bits -------------------------------------------------------------------------

def _stored(t, case):
    """Binary64 values rounded to the storage type of x and V."""
    return t.to(torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)


def _f32(v):
    return torch.tensor(v, dtype=torch.float32).double().item()      # a scalar as the C interface takes it


def _logits(case, p, feats):
    """Logits of one model, its parameters p as one binary64 vector."""
    dims, off = _dims(case), 0

    def take(*shape):
        nonlocal off
        n = 1
        for v in shape:
            n *= v
        off += n
        return p[off - n:off].view(shape)

    h = feats
    if case["model"] == "cnn":
        chans = dims[1:-1]
        for l in range(1, len(chans)):
            W, bias = take(chans[l], chans[l - 1], 3, 3), take(chans[l])
            h = torch.relu(torch.nn.functional.conv2d(h, W, bias, padding=1))
            h = torch.nn.functional.max_pool2d(h, 2) if l % 2 == 0 else h
        h = h.flatten(1)
        return h @ take(dims[-1], h.shape[1]).t() + take(dims[-1])
    for l in range(len(dims) - 1):
        W, bias = take(dims[l + 1], dims[l]), take(dims[l + 1])
        h = h @ W.t() + bias
        h = torch.relu(h) if l + 2 < len(dims) else h
    return h


def _exact_scores(case, x, V, feats, targets):
    g, rho, m, d = _f32(case["gamma"]), _f32(case["rho"]), case["m"], x.numel()
    if case["model"] == "lsq":              # A x, A v and v . v, a range of columns at a time
        a0 = torch.zeros(feats.shape[0], dtype=torch.float64, device=DEVICE)
        av, norms = torch.zeros(feats.shape[0], m, dtype=torch.float64, device=DEVICE), torch.zeros(m, dtype=torch.float64, device=DEVICE)
        for k in range(0, d, 1 << 22):
            A, v = feats[:, k:k + (1 << 22)].double(), V[:, k:min(d, k + (1 << 22))].double()
            a0 += A @ x[k:k + (1 << 22)].double()
            av += A @ v.t()
            norms += (v * v).sum(1)
        r = (a0 - targets.double())[:, None]
        f0, f = (r * r).mean(0) / 2, ((r - g * av) ** 2).mean(0) / 2
        return f0 - f - rho * norms
    x, feats, targets = x.double(), feats.double(), targets.long()
    f0 = torch.nn.functional.cross_entropy(_logits(case, x, feats), targets)
    scores = []
    for i in range(m):
        v = V[i, :d].double()
        w = x - g * v
        if case["dtype"] == "bf16":         # the candidate is itself a bfloat16 model
            w = w.float().to(torch.bfloat16).double()
        scores.append(f0 - torch.nn.functional.cross_entropy(_logits(case, w, feats), targets) - rho * (v * v).sum())
    return torch.stack(scores)


def _exact_mean(case, V, scores, d):
    keep = torch.sort(-scores.float(), stable=True).indices[:case["m"] - case["b"]].tolist()
    acc = torch.zeros(d, dtype=torch.float64, device=DEVICE)
    for i in keep:
        acc += V[i, :d].double()
    return acc / len(keep)


def exact(case, seed):
    s = _inputs(case, seed)
    w, call, g, b, m = s["w"], case["call"], _f32(case["gamma"]), case["b"], case["m"]
    d, V = w.d, w.V
    if call == "step":
        scores = _exact_scores(case, w.x, V, w.features, w.targets)
        return _exact_mean(case, V, scores, d), scores
    if call == "update":
        scores = _exact_scores(case, w.x, V, w.features, w.targets)
        return w.x.double() - g * _exact_mean(case, V, scores, d), scores
    if call == "run":                       # x is stored between the iterations, the last one is left in 64 bits
        x, rows = w.x, []
        for t in range(case["steps"]):
            rows.append(_exact_scores(case, x, s["V"][t], s["feats"][t], s["labels"][t]))
            new = x.double() - g * _exact_mean(case, s["V"][t], rows[-1], d)
            x = _stored(new, case)
        return new, torch.stack(rows)
    if call == "iteration":                 # worker i's gradient of softmax regression on its own samples
        n_in, classes = _dims(case)
        x = w.x.double()
        W, bias, n = x[:classes * n_in].view(classes, n_in), x[classes * n_in:], case["worker_batch"]
        G = torch.empty(m, d, dtype=torch.float64, device=DEVICE)
        for i in range(m):
            a = s["wfeats"][i].double()
            delta = torch.softmax(a @ W.t() + bias, 1)
            delta[torch.arange(n, device=DEVICE), s["wlabels"][i].long()] -= 1
            G[i] = torch.cat([(delta.t() @ a / n).flatten(), delta.sum(0) / n])
        if s["faulty"].numel():
            G[s["faulty"].long()] = -G[s["faulty"][0].long()]
        stored = _stored(G, case)
        scores = _exact_scores(case, w.x, stored, w.features, w.targets)
        return x - g * _exact_mean(case, stored, scores, d), G, scores
    if call == "median":
        out = torch.empty(d, dtype=torch.float64, device=DEVICE)
        for k in range(0, d, 1 << 20):
            c = torch.sort(V[:, k:min(d, k + (1 << 20))].double(), 0).values
            out[k:k + (1 << 20)] = (c[(m - 1) // 2] + c[m // 2]) / 2
        return out
    dist = torch.zeros(m, m, dtype=torch.float64, device=DEVICE)
    for k in range(0, d, 1 << 20):
        v = V[:, k:min(d, k + (1 << 20))].double()
        for i in range(m):
            dist[i] += ((v - v[i]) ** 2).sum(1)
    dist.fill_diagonal_(float("inf"))       # the m - b - 2 nearest of the others
    sums = torch.sort(dist, 1).values[:, :m - b - 2].sum(1)
    k = int(sums.float().argmin())
    return V[k, :d].double(), torch.tensor([k], dtype=torch.int32, device=DEVICE), sums
