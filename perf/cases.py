"""The measured cases: what a user has the library do, through its Python
binding, over the sizes that the repository's own configurations name.

Eight kinds of call (one pass is one call, or one training epoch):

  basis     Plan.basis: Alg. 1 on a snapshot matrix held on the GPU, outputs
            into buffers that the program keeps (as bench.py does)
  batch     Batch.run: independent instances (fields x parameter samples) as
            one unit
  project   Plan.project: coefficients of held-out snapshots
  fluct     fluctuations: per-sample centering before the basis
  grad      LSTM.loss_grad: one training batch's loss and gradients
  epoch     LSTM.train_epoch: a short epoch with Adam, the updated weights
  forward   LSTM.forward: one-step predictions (validation)
  rollout   LSTM.rollout: the online stage

The snapshot matrices are U diag(a) V^T plus noise of 1e-6 like the
repository's synthetic recipes: orthonormal spatial modes, each with one
strongest cell (the sign rule looks for it), cosine time coefficients of
distinct frequencies, amplitudes a_j = exp(-j / tau) with tau = k / 2.5
(bench.py's exp(-j / 40) at k = 100) or j^-1.5 (the paper's shape).  The
singular values are then the amplitudes, well apart, as in a resolved POD
spectrum.

The FP32 and 16-bit forms compute in 32 bits; their sigma is a double only by
its container, and `run` hands it on in the type of U and C, with which a
program combines it (V^T = C / sigma).
"""
import math

import numpy as np
import torch

import paper_2504_15350_gb300.rpod as R

_TYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def listed():
    return [
        # the smallest basis: 64 x 64 grid, 500 snapshots, in FP64 throughout
        dict(name="basis_f64_4096x500", kind="basis", form="f64", n=4096, m=500, k=20, p=10, q=1,
             decay="exp", seed=0),
        # the same shape with FP16 passes and FP32 refinement: latency counts
        dict(name="basis_f16_4096x500", kind="basis", form="f16", n=4096, m=500, k=20, p=10, q=1,
             decay="exp", seed=0),
        # the ROM driver's basis: 32 parameter samples x 2000 steps, FP32
        dict(name="basis_f32_4096x64000", kind="basis", form="f32", n=4096, m=64000, k=50, p=10, q=1,
             decay="exp", seed=1),
        # a larger FP32 basis at the rank of the benchmark (256 x 256 grid)
        dict(name="basis_f32_65536x4000", kind="basis", form="f32", n=65536, m=4000, k=100, p=20, q=2,
             decay="exp", seed=2),
        # the paper's own matrix: 8192 cells, 225 samples x 401 times
        dict(name="basis_bf16_8192x90225", kind="basis", form="bf16", n=8192, m=90225, k=10, p=75, q=1,
             decay="power", seed=3),
        # the benchmark: 512 x 512 grid, 10000 snapshots, BF16 passes
        dict(name="basis_bf16_262144x10000", kind="basis", form="bf16", n=262144, m=10000, k=100, p=20,
             q=2, decay="exp", seed=0),
        # four fields x four parameter samples on a 128 x 256 grid, ragged m
        dict(name="batch_bf16_16x32768", kind="batch", form="bf16", n=32768, count=16, m_lo=500,
             m_hi=3000, p=10, q=1, seed=5),
        # one held-out trajectory of 401 snapshots on the benchmark's basis
        dict(name="project_262144x401", kind="project", form="bf16", s_type="f32", n=262144, m=10000,
             m_new=401, k=100, seed=6),
        # centering: 25 samples of 400 snapshots, with the 16-bit copy
        dict(name="fluct_65536x10000", kind="fluct", s_type="f32", h_type="bf16", n=65536, samples=25,
             nt=400, seed=7),
        # the ROM driver's network and batch
        dict(name="lstm_grad_2x256_b512", kind="grad", inputs=54, hidden=256, layers=2, outputs=50,
             window=10, batch=512, dropout=0.0, seed=8),
        # the paper's stream-function network: 3 x 50, batch 16, dropout 0.1
        dict(name="lstm_epoch_3x50_b16", kind="epoch", inputs=14, hidden=50, layers=3, outputs=10,
             window=10, batch=16, steps=8, dropout=0.1, seed=9),
        # the online stage: 8 held-out parameters, 500 steps
        dict(name="lstm_rollout_2x256_b8", kind="rollout", inputs=54, hidden=256, layers=2, outputs=50,
             window=10, batch=8, steps=500, dropout=0.0, seed=10),
    ]


def _between(rng, lo, hi):
    """An integer of lo..hi, spread over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["basis"] * 5 + ["batch", "project", "fluct", "grad", "epoch", "forward", "rollout"])
    seed = rng.randrange(1 << 20)
    if kind == "basis":
        form = rng.choice(["f64", "f32", "f32", "bf16", "bf16", "f16"])
        q = rng.choice([1, 1, 2])
        # what the form's largest listed case multiplies and holds
        work, held = {"f64": (3.0e8, 1 << 22), "f32": (3.5e10, 1 << 28), "bf16": (3.5e11, 1 << 31),
                      "f16": (3.5e10, 1 << 28)}[form]
        while True:
            n, m = _between(rng, 1000, 262144), _between(rng, 300, 90225)
            k, p = _between(rng, 8, 100), rng.randint(2, 28)
            if k + p <= 128 and n * m <= held and n * m * (k + p) <= work and 3 * (k + p) <= m:
                return dict(kind=kind, form=form, n=n, m=m, k=k, p=p, q=q, decay="exp", seed=seed)
    if kind == "batch":
        return dict(kind=kind, form=rng.choice(["bf16", "bf16", "f32"]), n=_between(rng, 2000, 32768),
                    count=rng.randint(4, 16), m_lo=rng.randint(300, 800), m_hi=rng.randint(900, 3000),
                    p=rng.randint(5, 12), q=1, seed=seed)
    if kind == "project":
        form, s_type = rng.choice([("bf16", "f32"), ("f32", "f32"), ("bf16", "bf16"), ("f16", "f16")])
        while True:
            n, m_new = _between(rng, 1000, 262144), _between(rng, 1, 20000)
            if n * m_new <= 1 << 28:
                return dict(kind=kind, form=form, s_type=s_type, n=n, m=1000, m_new=m_new,
                            k=_between(rng, 5, 100), seed=seed)
    if kind == "fluct":
        s_type, h_type = rng.choice([("f32", "bf16"), ("f32", "f16"), ("f32", ""), ("f64", ""), ("bf16", "")])
        while True:
            n, samples, nt = _between(rng, 1000, 262144), _between(rng, 1, 225), _between(rng, 20, 2000)
            if n * samples * nt <= 1 << 29:
                return dict(kind=kind, s_type=s_type, h_type=h_type, n=n, samples=samples, nt=nt, seed=seed)
    outputs = _between(rng, 5, 60)
    case = dict(kind=kind, inputs=outputs + rng.randint(0, 6), hidden=_between(rng, 20, 256),
                layers=rng.randint(1, 3), outputs=outputs, window=rng.randint(4, 16),
                batch=_between(rng, 8, 512), dropout=0.0, seed=seed)
    if kind in ("grad", "epoch"):
        case["dropout"] = rng.choice([0.0, 0.1])
    if kind == "epoch":
        case.update(batch=_between(rng, 8, 64), steps=rng.randint(2, 8))
    if kind == "rollout":
        case.update(batch=_between(rng, 1, 16), steps=_between(rng, 50, 500))
    return case


# ---- inputs -------------------------------------------------------------
def _gen(*key):
    g = torch.Generator(device="cuda")
    g.manual_seed(hash(tuple(int(v) for v in key)) & 0x7FFFFFFFFFFF)
    return g


def _amplitudes(k, decay, J, dtype):
    j = torch.arange(1, J + 1, device="cuda", dtype=dtype)
    return j ** -1.5 if decay == "power" else torch.exp(-j * (2.5 / k))


def _snapshots(n, m, k, decay, dtype, gen):
    """n x m column-major snapshots with singular values close to
    sqrt(n m / 2) a_j."""
    wide = torch.float64 if dtype == torch.float64 else torch.float32
    J = min(400, n // 2, m // 2)
    phi = torch.randn(J, n, generator=gen, device="cuda", dtype=wide)
    # one strongest cell per mode (a vortex centre): the sign rule's choice
    peak = torch.randperm(n, generator=gen, device="cuda")[:J, None]
    phi.scatter_(1, peak, 9.0 * phi.gather(1, peak).sign())
    L = torch.linalg.cholesky(phi.double() @ phi.double().t()) if n <= 4096 else \
        torch.linalg.cholesky((phi @ phi.t()).double())
    phi = torch.linalg.solve_triangular(L.to(wide), phi, upper=False)   # orthonormal rows
    freq = torch.randperm(J, generator=gen, device="cuda").to(torch.float64) + 1.0
    t = torch.arange(m, device="cuda", dtype=torch.float64) + 0.5
    a = _amplitudes(k, decay, J, torch.float64) * math.sqrt(n)
    S = torch.empty(m, n, device="cuda", dtype=dtype)
    step = max(1, (1 << 27) // n)
    for c in range(0, m, step):
        coef = torch.cos(torch.outer(t[c:c + step], freq * (math.pi / m))) * a
        blk = coef.to(wide) @ phi
        blk += 1e-6 * torch.randn(blk.shape, generator=gen, device="cuda", dtype=wide)
        S[c:c + step] = blk.to(dtype)
    return S.t()


def _basis_input(c, seed):
    dtype = torch.float64 if c["form"] == "f64" else torch.float32
    return _snapshots(c["n"], c["m"], c["k"], c["decay"], dtype, _gen(1, seed, c["seed"]))


def _batch_shapes(c):
    rng = np.random.default_rng(c["seed"])
    ms = rng.integers(c["m_lo"], c["m_hi"] + 1, c["count"])
    ks = rng.choice([10, 20, 30, 50], c["count"])
    return [(int(m), int(k)) for m, k in zip(ms, ks)]


def _batch_input(c, seed):
    return [_snapshots(c["n"], m, k, "exp", torch.float32, _gen(2, seed, c["seed"], i))
            for i, (m, k) in enumerate(_batch_shapes(c))]


def _project_input(c, seed):
    g = _gen(3, seed, c["seed"])
    U = torch.randn(c["k"], c["n"], generator=g, device="cuda") / math.sqrt(c["n"])
    S = _snapshots(c["n"], max(c["m_new"], 2), c["k"], "exp", torch.float32, g)[:, :c["m_new"]]
    # new snapshots lie mostly in the basis' span, as held-out ones do
    S += U.t() @ torch.randn(c["k"], c["m_new"], generator=g, device="cuda") * math.sqrt(c["n"])
    return U.t(), S.t().to(_TYPES[c["s_type"]]).contiguous().t()


def _fluct_input(c, seed):
    g = _gen(4, seed, c["seed"])
    dtype = _TYPES[c["s_type"]]
    wide = torch.float64 if dtype == torch.float64 else torch.float32
    S = torch.empty(c["samples"], c["nt"], c["n"], device="cuda", dtype=dtype)
    for i in range(c["samples"]):   # a mean field per sample plus fluctuations
        mean = 2.0 + 4.0 * torch.randn(c["n"], generator=g, device="cuda", dtype=wide)
        S[i] = (mean + torch.randn(c["nt"], c["n"], generator=g, device="cuda", dtype=wide)).to(dtype)
    return S.reshape(-1, c["n"]).t()


def _lstm_sizes(c):
    out, I, H = [], c["inputs"], c["hidden"]
    for _ in range(c["layers"]):
        out += [(4 * H, I), (4 * H, H), (4 * H,)]
        I = H
    return out + [(c["outputs"], H), (c["outputs"],)]


def _lstm_theta(c, seed):
    """The usual initial weights: uniform in +-1/sqrt(hidden)."""
    P = sum(int(np.prod(s)) for s in _lstm_sizes(c))
    g = _gen(5, seed, c["seed"])
    return (torch.rand(P, generator=g, device="cuda") * 2 - 1) / math.sqrt(c["hidden"])


def _series(c, seed):
    """Standardised coefficient series (samples, steps, outputs) and their
    parameters: sums of a few oscillations, as POD coefficients are."""
    g = _gen(6, seed, c["seed"])
    samples, steps, d = 8, 200, c["inputs"] - c["outputs"]
    w = 0.1 + 1.9 * torch.rand(samples, 1, c["outputs"], 3, generator=g, device="cuda")
    ph = 2 * math.pi * torch.rand(samples, 1, c["outputs"], 3, generator=g, device="cuda")
    t = 0.1 * torch.arange(steps, device="cuda").reshape(1, -1, 1, 1)
    mu = torch.randn(samples, max(d, 1), generator=g, device="cuda")[:, :d].contiguous()
    return torch.cos(w * t + ph).sum(-1).mul_(0.8).contiguous(), mu


def _rows(c, seed, count):
    g = _gen(7, seed, c["seed"])
    s = torch.randint(0, 8, (count,), generator=g, device="cuda")
    t = torch.randint(0, 200 - c["window"], (count,), generator=g, device="cuda")
    return torch.stack([s, t], 1).to(torch.int32).contiguous()


def _windows(c, seed, count):
    """Windows (count, window, inputs) and targets, in plain torch."""
    series, mu = _series(c, seed)
    rows = _rows(c, seed, count).long()
    at = rows[:, 1:2] + torch.arange(c["window"] + 1, device="cuda")
    alpha = series[rows[:, :1], at]
    X = torch.cat([mu[rows[:, 0]][:, None].expand(-1, c["window"], -1), alpha[:, :-1]], -1)
    return X.contiguous(), alpha[:, -1].contiguous()


# ---- the call -----------------------------------------------------------
def _plan(c, m):
    flags = R.RPOD_FLAG_REFINE_FP32 if c["form"] in ("bf16", "f16") else 0
    return R.Plan(c["n"], m, c["k"], c.get("p", 0), c.get("q", 1), seed=c["seed"], compute=c["form"],
                  flags=flags)


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "basis":
        S = _basis_input(c, seed)
        plan = _plan(c, c["m"])
        out = (R.empty_colmajor(c["n"], c["k"], plan.out_dtype, "cuda"),
               torch.empty(c["k"] + c["p"], dtype=torch.float64, device="cuda"),
               R.empty_colmajor(c["k"], c["m"], plan.out_dtype, "cuda"))
        return dict(kind=kind, plan=plan, S=S, out=out)
    if kind == "batch":
        shapes = _batch_shapes(c)
        b = R.Batch(_batch_input(c, seed), [k for _, k in shapes], c["p"], c["q"],
                    [c["seed"] + i for i in range(len(shapes))], compute=c["form"],
                    flags=R.RPOD_FLAG_REFINE_FP32 if c["form"] == "bf16" else 0)
        b.configure(64, 25, 2)   # what the tuner finds for the benchmark's batch
        return dict(kind=kind, batch=b)
    if kind == "project":
        U, S = _project_input(c, seed)
        return dict(kind=kind, plan=_plan(c, c["m"]), U=U, S=S)
    if kind == "fluct":
        S = _fluct_input(c, seed)
        wide = torch.float64 if S.dtype == torch.float64 else torch.float32
        out = (R.empty_colmajor(c["n"], S.shape[1], S.dtype, "cuda"),
               R.empty_colmajor(c["n"], S.shape[1], _TYPES[c["h_type"]], "cuda") if c["h_type"] else None,
               R.empty_colmajor(c["n"], c["samples"], wide, "cuda"))
        return dict(kind=kind, S=S, nt=c["nt"], out=out)
    net = R.LSTM(c["inputs"], c["hidden"], c["layers"], c["outputs"], c["window"], max_batch=c["batch"],
                 theta=_lstm_theta(c, seed))
    if c["dropout"]:
        net.set_dropout(c["dropout"], c["seed"])
    if kind == "epoch":
        series, mu = _series(c, seed)
        return dict(kind=kind, net=net, series=series, mu=mu, batch=c["batch"],
                    rows=_rows(c, seed, c["steps"] * c["batch"]))
    X, Y = _windows(c, seed, c["batch"])
    return dict(kind=kind, net=net, X=X, Y=Y, d=c["inputs"] - c["outputs"], steps=c.get("steps", 0))


def run(state):
    kind = state["kind"]
    if kind == "basis":
        U, sigma, C = state["plan"].basis(state["S"], out=state["out"])
        return {"U": U, "sigma": sigma.to(U.dtype), "C": C}
    if kind == "batch":
        b = state["batch"]
        b.run()
        return {"U": b.U, "sigma": [s.to(U.dtype) for s, U in zip(b.sigma, b.U)], "C": b.C}
    if kind == "project":
        return state["plan"].project(state["U"], state["S"])
    if kind == "fluct":
        F, H, Sbar = R.fluctuations(state["S"], state["nt"], out=state["out"])
        return {"F": F, "H": H, "Sbar": Sbar}
    net = state["net"]
    if kind == "grad":
        loss, grad = net.loss_grad(state["X"], state["Y"])
        return {"loss": loss, "grad": grad}
    if kind == "epoch":
        loss = net.train_epoch(state["series"], state["mu"], state["rows"], state["batch"])
        return {"loss": loss, "weights": net.get_params()}
    if kind == "forward":
        return net.forward(state["X"])
    return net.rollout(state["X"], state["d"], state["steps"])


# ---- what a pass cannot do without --------------------------------------
def _size(name):
    return {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}[name]


def _basis_work(n, m, k, l, q, size):
    # S once, U, sigma and C once; 2 q + 2 products with S
    return size * (n * m + n * k + k * m) + 8 * l, (2 * q + 2) * 2.0 * n * m * l


def work(case):
    c, kind = case, case["kind"]
    if kind == "basis":
        b, f = _basis_work(c["n"], c["m"], c["k"], c["k"] + c["p"], c["q"], 8 if c["form"] == "f64" else 4)
    elif kind == "batch":
        each = [_basis_work(c["n"], m, k, k + c["p"], c["q"], 4) for m, k in _batch_shapes(c)]
        b, f = sum(x[0] for x in each), sum(x[1] for x in each)
    elif kind == "project":
        b = c["n"] * (_size(c["s_type"]) * c["m_new"] + 4 * c["k"]) + 4 * c["k"] * c["m_new"]
        f = 2.0 * c["n"] * c["m_new"] * c["k"]
    elif kind == "fluct":
        m, s = c["samples"] * c["nt"], _size(c["s_type"])
        b = c["n"] * (m * (2 * s + (2 if c["h_type"] else 0)) + c["samples"] * max(4, s))
        f = 2.0 * c["n"] * m
    else:
        sizes = _lstm_sizes(c)
        P = sum(int(np.prod(s)) for s in sizes)
        cell = sum(2.0 * a[0] * a[1] for a in sizes if len(a) == 2)   # multiply-adds of one step
        rows = c["batch"] * c["window"]
        if kind == "forward":
            b, f = 4 * (P + rows * c["inputs"] + c["batch"] * c["outputs"]), rows * cell
        elif kind == "grad":
            b, f = 4 * (2 * P + rows * c["inputs"] + c["batch"] * c["outputs"]), 3 * rows * cell
        elif kind == "epoch":
            b, f = 4 * (6 * P + c["steps"] * rows * c["inputs"]), c["steps"] * 3 * rows * cell
        else:
            b = 4 * (P + rows * c["inputs"] + c["batch"] * c["steps"] * c["outputs"])
            f = c["steps"] * rows * cell
    return {"bytes": float(b), "flops": float(f)}


# ---- the same in 64 bits, without the library ----------------------------
def _philox(key, start, blocks):
    """Words of numpy's Philox4x64-10 for `blocks` counters from `start`."""
    gen = np.random.Philox(key=np.array(key, dtype=np.uint64), counter=(start - 1) % (1 << 256))
    return gen.random_raw(4 * blocks).reshape(blocks, 4)


def _sketch(seed, m, l):
    blocks = (m * l + 1) // 2
    w = _philox((seed, 0), 0, blocks)[:, :2] >> np.uint64(11)
    r = np.sqrt(-2.0 * np.log((w[:, 0].astype(np.float64) + 1.0) * 2.0 ** -53))
    a = (2.0 * np.pi * 2.0 ** -53) * w[:, 1].astype(np.float64)
    z = np.stack([r * np.cos(a), r * np.sin(a)], 1).reshape(-1)[:m * l]
    return torch.from_numpy(z).cuda().reshape(l, m).t()


def _exact_basis(S, k, l, q, seed):
    n, m = S.shape
    St = S.t()
    step = max(1, (1 << 28) // n)
    part = [St[c:c + step].double() for c in range(0, m, step)]

    def times(Z):       # S Z
        return sum(b.t() @ Z[i * step:i * step + b.shape[0]] for i, b in enumerate(part))

    def transposed(Q):  # S^T Q
        return torch.cat([b @ Q for b in part])

    Q = torch.linalg.qr(times(_sketch(seed, m, l)))[0]
    for _ in range(q):
        Q = torch.linalg.qr(times(torch.linalg.qr(transposed(Q))[0]))[0]
    V, Rt = torch.linalg.qr(transposed(Q))        # T^T
    W, s, Xt = torch.linalg.svd(Rt)               # T = X s (V W)^T
    U = Q @ Xt.t()[:, :k]
    big = U.gather(0, U.abs().argmax(0, keepdim=True)).sign()
    C = (s[:k, None] * (V @ W[:, :k]).t()) * big.t()
    return {"U": U * big, "sigma": s, "C": C}


def _dropped(x, layer, at, c):
    """The input of a layer above the first in training pass `at`."""
    n = x.numel()
    words = _philox((c["seed"], 1), (at << 128) + (layer << 64), (n + 3) // 4).reshape(-1)[:n]
    keep = (words >> np.uint64(11)) >= np.uint64(math.ceil(c["dropout"] * 2.0 ** 53))
    return x * torch.from_numpy(keep).cuda().reshape(x.shape) / (1.0 - c["dropout"])


def _parts(theta, c):
    out, at = [], 0
    for s in _lstm_sizes(c):
        out.append(theta[at:at + int(np.prod(s))].reshape(s))
        at += int(np.prod(s))
    return out


def _exact_net(parts, X, c, at=None):
    """Predictions for the windows X (batch, window, inputs); the weight
    matrices enter as the 16-bit copies that the library documents."""
    x = X.transpose(0, 1)
    for layer in range(c["layers"]):
        Wx, Wh, b = parts[3 * layer:3 * layer + 3]
        if layer and at is not None and c["dropout"]:
            x = _dropped(x, layer, at, c)
        h = torch.zeros(x.shape[1], c["hidden"], dtype=x.dtype, device=x.device)
        cell, hs, gx = h, [], x @ Wx.t() + b
        for t in range(x.shape[0]):
            i, f, g, o = (gx[t] + h @ Wh.t()).chunk(4, 1)
            cell = torch.sigmoid(f) * cell + torch.sigmoid(i) * torch.tanh(g)
            h = torch.sigmoid(o) * torch.tanh(cell)
            hs.append(h)
        x = torch.stack(hs)
    return x[-1] @ parts[-2].t() + parts[-1]


def _entering(theta, c):
    return [(p.float().bfloat16().double() if p.dim() == 2 else p).detach().requires_grad_()
            for p in _parts(theta, c)]


def _exact_grad(theta, X, Y, c, at):
    parts = _entering(theta, c)
    loss = ((_exact_net(parts, X, c, at) - Y) ** 2).mean()
    return loss.detach().reshape(1), torch.cat([g.reshape(-1) for g in torch.autograd.grad(loss, parts)])


def _exact_epoch(c, seed):
    theta = _lstm_theta(c, seed).double()
    mean, square, total = torch.zeros_like(theta), torch.zeros_like(theta), 0.0
    X, Y = (v.double() for v in _windows(c, seed, c["steps"] * c["batch"]))
    for s in range(c["steps"]):
        at = slice(s * c["batch"], (s + 1) * c["batch"])
        loss, g = _exact_grad(theta, X[at], Y[at], c, s)
        g = g + 1e-5 * theta
        mean, square = 0.9 * mean + 0.1 * g, 0.999 * square + 0.001 * g * g
        theta = theta - 1e-3 * (mean / (1 - 0.9 ** (s + 1))) / \
            ((square / (1 - 0.999 ** (s + 1))).sqrt() + 1e-8)
        total = total + loss
    return {"loss": total / c["steps"], "weights": theta}


@torch.no_grad()
def _exact_rollout(c, seed):
    parts = _entering(_lstm_theta(c, seed).double(), c)
    x, _ = _windows(c, seed, c["batch"])
    x, d, out = x.double(), c["inputs"] - c["outputs"], []
    for _ in range(c["steps"]):
        y = _exact_net(parts, x, c)
        out.append(y)
        x = torch.cat([x[:, 1:], torch.cat([x[:, -1:, :d], y[:, None]], -1)], 1)
    return torch.stack(out, 1)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "basis":
        return _exact_basis(_basis_input(c, seed), c["k"], c["k"] + c["p"], c["q"], c["seed"])
    if kind == "batch":
        each = [_exact_basis(S, k, k + c["p"], c["q"], c["seed"] + i)
                for i, (S, (_, k)) in enumerate(zip(_batch_input(c, seed), _batch_shapes(c)))]
        return {key: [e[key] for e in each] for key in ("U", "sigma", "C")}
    if kind == "project":
        U, S = _project_input(c, seed)
        step = max(1, (1 << 27) // c["n"])
        return torch.cat([S[:, j:j + step].double().t() @ U.double()
                          for j in range(0, c["m_new"], step)]).t()
    if kind == "fluct":
        S = _fluct_input(c, seed).double().t().reshape(c["samples"], c["nt"], c["n"])
        mean = S.mean(1)
        F = (S - mean[:, None]).reshape(-1, c["n"]).t()
        return {"F": F, "H": F if c["h_type"] else None, "Sbar": mean.t()}
    if kind == "epoch":
        return _exact_epoch(c, seed)
    if kind == "rollout":
        return _exact_rollout(c, seed)
    X, Y = (v.double() for v in _windows(c, seed, c["batch"]))
    theta = _lstm_theta(c, seed).double()
    if kind == "forward":
        with torch.no_grad():
            return _exact_net(_entering(theta, c), X, c)
    loss, grad = _exact_grad(theta, X, Y, c, 0)
    return {"loss": loss, "grad": grad}
