"""The work this library is used for, as measurable cases.

A case names one use of the public API with its sizes:

  grad   the sampled loss and the whole gradient (one MTTKRP variant, one
         sampling scheme, FP32 or BF16 factors);
  loss   the objective estimate alone (the forward direction);
  steps  a stretch of a training loop (gradient + Adam per step, losses kept
         on the device), then the factors read out;
  fit    the whole GCP-Adam call from a starting guess;
  dense  the autograd binding on a dense tensor, forward and backward;
  fed    one federated round: tau local steps of every client, the server's
         Adam step, the clients' losses and the server model;
  list   a sample list drawn on the GPU, then its gradient through the entry
         point that allocates nothing.

`prepare` makes the tensor, the factors and the context; `run` is one pass;
`exact` restates the same arithmetic in FP64 with torch operations and
shares no code with the library.
"""
import math

import numpy as np
import torch

import paper_2605_20353_gb300 as gcp
from paper_2605_20353_gb300 import autograd as gcp_autograd

ADAM = dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, lower=0.0)
SERVER = dict(lr=1e-2, beta1=0.6, beta2=0.99, eps=1e-8, lower=0.0)


def _case(name, kind, dims, rank, loss, p, q, nnz=0, **more):
    c = dict(kind=kind, dims=dims, rank=rank, loss=loss, p=p, q=q, nnz=nnz, place="uniform", dtype="fp32",
             mttkrp="atomic", sampling="stratified")
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    K = 1 << 10
    return [
        # the smallest call of the tests: a gradient and its loss read by the
        # host, where launches and latency are all there is
        _case("grad-small", "grad", "50x40x30", 4, "gaussian", 1000, 1000, 2000, host=True),
        # an ordinary minibatch gradient with nothing round about it: odd mode
        # sizes, a rank that is no power of two, odd sample counts
        _case("grad-ragged-rank20", "grad", "4999x3001x777", 20, "gamma", 100003, 150001, 1500000),
        # a high-rank BF16 model of binary data with many samples
        _case("grad-binary-bf16", "grad", "10000x10000x1000", 64, "bernoulli", K * K, K * K, 4000000, dtype="bf16"),
        # the bit-reproducible gradient on the same data in FP32
        _case("grad-deterministic", "grad", "10000x10000x1000", 64, "bernoulli", K * K, K * K, 4000000,
              mttkrp="deterministic"),
        # semi-stratified sampling on the shape of the arXiv tensor, a modest
        # number of samples, a large rank that needs padding
        _case("grad-semi-rank50", "grad", "172x25000x300", 50, "poisson", 32 * K, 32 * K, 3000000, sampling="semi"),
        # the objective estimate of a skewed count tensor, BF16 factors
        _case("loss-zipf-bf16", "loss", "2000x1500x1000x200", 32, "poisson", 256 * K, 256 * K, 4000000, place="zipf",
              dtype="bf16"),
        # the benchmark's training loop: skewed counts, 2^21 samples a step
        _case("steps-zipf", "steps", "2000x1500x1000x200", 32, "poisson", K * K, K * K, 4000000, place="zipf", steps=8),
        # a model far larger than L2: 121.6 M parameters
        _case("steps-large-model", "steps", "4800000x1700000x1100000", 16, "poisson", K * K, K * K, 2000000, steps=2),
        # a whole small fit: many cheap iterations, rank 10, an odd shape
        _case("fit-rank10", "fit", "211x187x95x24", 10, "poisson", 5000, 5000, 60000, place="zipf", iters=50, epochs=2),
        # dense simulation-like data through autograd, 5 modes
        _case("dense-autograd", "dense", "100x100x100x20x50", 16, "gaussian", 4 * K * K, 0),
        # a federated round of 16 clients sharing one model
        _case("fed-16-clients", "fed", "2000x1200x500", 16, "poisson", 8 * K, 8 * K, 100000, clients=16, tau=8),
        # a caller that owns the sample list and all device memory
        _case("list-zipf", "list", "2000x1500x1000x200", 32, "poisson", 128 * K, 128 * K, 1000000, place="zipf"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: 2 to 6 modes, ranks 3 to 128, from
    hundreds of samples to millions, all losses, samplings and variants."""
    kind = rng.choice(["grad", "grad", "grad", "loss", "steps", "fit", "dense", "fed", "list"])
    loss = rng.choice(["gaussian", "poisson", "bernoulli", "gamma"])
    dtype = rng.choice(["fp32", "fp32", "bf16"])
    rank = rng.choice([rng.randint(3, 128), 8, 10, 16, 32, 64])
    place = rng.choice(["uniform", "zipf"])
    if kind == "dense":
        d = rng.randint(3, 5)
        dims = [_log(rng, 17, {3: 400, 4: 120, 5: 40}[d]) for _ in range(d)]
        return _case(None, kind, "x".join(map(str, dims)), rng.randint(3, 32), rng.choice(["gaussian", "gamma"]),
                     _log(rng, 1000, 2000000), 0, dtype=dtype)
    if kind == "fit":
        d = rng.randint(3, 4)
        dims = [_log(rng, 40, 900) for _ in range(d)]
        nnz = _log(rng, 10000, 200000)
        nnz = min(nnz, math.prod(dims) // 8)
        return _case(None, kind, "x".join(map(str, dims)), rng.randint(3, 32), "poisson", _log(rng, 700, 20000),
                     _log(rng, 700, 20000), nnz, place=place, iters=rng.randint(10, 60), epochs=rng.randint(1, 2))
    if kind == "fed":
        dims = [_log(rng, 200, 3000) for _ in range(3)]
        return _case(None, kind, "x".join(map(str, dims)), rng.randint(4, 32), "poisson", _log(rng, 1000, 16000),
                     _log(rng, 1000, 16000), _log(rng, 10000, 100000), dtype=dtype, clients=rng.randint(3, 16),
                     tau=rng.randint(2, 8))
    d = rng.randint(2, 6) if kind == "grad" else rng.randint(3, 4)
    dims = [_log(rng, 30, {2: 60000, 3: 20000, 4: 4000, 5: 700, 6: 200}[d]) for _ in range(d)]
    nnz = min(_log(rng, 20000, 2000000), max(100, math.prod(dims) // 8))
    most = int(min(2.0e6, 6.0e7 / rank / d))
    p, q = _log(rng, 500, most), _log(rng, 500, most)
    text = "x".join(map(str, dims))
    if kind == "steps":
        return _case(None, kind, text, rank, "poisson", p, q, nnz, place=place, dtype=dtype, steps=rng.randint(2, 8))
    if kind == "list":
        return _case(None, kind, text, rank, loss, p // 4 + 1, q // 4 + 1, nnz, place=place)
    more = {}
    if kind == "grad":
        more = dict(mttkrp=rng.choice(["atomic", "atomic", "deterministic", "nonfused"]), host=rng.random() < 0.3)
    return _case(None, kind, text, rank, loss, p, q, nnz, place=place, dtype=dtype,
                 sampling=rng.choice(["stratified", "stratified", "semi"]), **more)


# ------------------------------------------------------------------- inputs
def _dims(case):
    return [int(i) for i in case["dims"].split("x")]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(n, g):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _keys_of(case, g):
    """Sorted distinct linear indices of the nonzeros (last mode fastest)."""
    dims, want = _dims(case), case["nnz"]
    cdfs = []
    if case["place"] == "zipf":
        for I in dims:
            w = torch.arange(1, I + 1, device="cuda", dtype=torch.float64) ** -1.1
            cdfs.append(torch.cumsum(w, 0) / w.sum())
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    n = int(1.1 * want) + 64
    for _ in range(40):
        new = torch.zeros(n, dtype=torch.int64, device="cuda")
        for k, I in enumerate(dims):
            u = _rand(n, g)
            i = torch.searchsorted(cdfs[k], u) if cdfs else (u * I).to(torch.int64)
            new = new * I + i.clamp_(0, I - 1)
        keys = torch.unique(torch.cat([keys, new]))
        if keys.numel() >= want:
            break
        n = min(4 * n, 1 << 24)
    if keys.numel() > want:
        keys = keys[torch.randperm(keys.numel(), generator=g, device="cuda")[:want]].sort().values
    return keys


def _values(loss, n, g):
    if loss == "bernoulli":
        return torch.ones(n, device="cuda")
    if loss == "gamma":
        return (0.05 - torch.log(1.0 - _rand(n, g))).float()
    return 1.0 + torch.poisson(torch.full((n,), 3.0, device="cuda"), generator=g)


def _factors(case, g):
    dims, R = _dims(case), case["rank"]
    if case["kind"] == "dense" and case["loss"] == "gaussian" or case["loss"] == "bernoulli":
        std = (0.5 / math.sqrt(R)) ** (1.0 / len(dims))
        return [torch.randn((I, R), generator=g, device="cuda") * std for I in dims]
    return [0.1 + 0.9 * torch.rand((I, R), generator=g, device="cuda") for I in dims]


def _inputs(case, seed, shard=0):
    """(keys, values) of a sparse tensor; `shard` numbers the clients."""
    g = _gen(seed * 1000 + 17 + shard)
    keys = _keys_of(case, g)
    return keys, _values(case["loss"], keys.numel(), g)


def _dense_inputs(case, seed):
    dims, g = _dims(case), _gen(seed * 1000 + 17)
    X = torch.zeros(dims, device="cuda")
    for r in range(2):  # a smooth rank-2 signal and noise
        t = torch.ones((), device="cuda")
        for k, I in enumerate(dims):
            i = (torch.arange(I, device="cuda") + 0.5) / I
            v = torch.sin(2 * math.pi * (r + 1) * i + r)
            t = t.unsqueeze(-1) * v
        X += t
    X += 0.1 * torch.randn(dims, generator=g, device="cuda")
    return X if case["loss"] == "gaussian" else X.abs_().add_(0.05)


def _start(case, seed):
    return _factors(case, _gen(seed * 1000 + 5))


def _coords(dims, keys):
    out = torch.empty((keys.numel(), len(dims)), dtype=torch.int32, device=keys.device)
    for k in range(len(dims) - 1, -1, -1):
        out[:, k] = (keys % dims[k]).to(torch.int32)
        keys = torch.div(keys, dims[k], rounding_mode="floor")
    return out


def _context(case, seed, shard=0):
    keys, vals = _inputs(case, seed, shard)
    return gcp.gcp_create(_dims(case), _coords(_dims(case), keys).cpu().numpy(), vals.cpu().numpy(), case["rank"],
                          case["loss"], dtype=case["dtype"], mttkrp=case["mttkrp"], sampling=case["sampling"],
                          seed=seed + shard)


def prepare(case, seed):
    dims, R, kind = _dims(case), case["rank"], case["kind"]
    s = dict(case=case, it=0)
    A = _start(case, seed)
    if kind == "dense":
        s["ctx"] = gcp.gcp_create_dense(dims, _dense_inputs(case, seed), R, case["loss"], dtype=case["dtype"], seed=seed)
        s["A"] = [a.requires_grad_() for a in A]
        return s
    if kind == "fed":
        s["clients"] = [_context(case, seed, c) for c in range(case["clients"])]
        s["clients"][0].set_factors(A)
        n = len(s["clients"])
        s["batch"] = gcp.GcpBatch(s["clients"], [case["p"]] * n, [case["q"]] * n)
        s["batch"].server_init()
        return s
    s["ctx"] = ctx = _context(case, seed)
    ctx.set_factors(A)
    s["out"] = torch.empty(ctx.num_params, device="cuda")
    s["loss"] = torch.zeros(max(2, case.get("steps", 0)), dtype=torch.float64, device="cuda")
    if kind in ("fit", "list"):
        s["flat"] = torch.cat([a.reshape(-1) for a in A])
    return s


def run(s):
    case = s["case"]
    kind, p, q, it = case["kind"], case["p"], case["q"], s["it"]
    if kind == "grad":
        s["it"] += 1
        if case.get("host"):
            loss, G = s["ctx"].grad(it, p, q, G_out=s["out"])
            return {"loss": loss, "G": G}
        s["ctx"].grad_async(it, p, q, G_out=s["out"], dloss=s["loss"])
        return {"loss": s["loss"][:1], "G": s["out"]}
    if kind == "loss":
        s["it"] += 1
        return {"loss": s["ctx"].loss_value(it, p, q)}
    if kind == "steps":
        adam, n = gcp.AdamParams(**ADAM), case["steps"]
        for k in range(n):
            s["ctx"].step(it + k, p, q, adam, it + k + 1, dloss=s["loss"][k:k + 1])
        s["it"] += n
        # the factors, to a device buffer (gcp_get_factors takes either)
        rc = gcp.load().gcp_get_factors(s["ctx"].handle, s["out"].data_ptr())
        if rc:
            raise gcp.GcpError(rc, "gcp_get_factors")
        return {"loss": s["loss"][:n], "A": s["out"]}
    if kind == "fit":
        s["ctx"].set_factors(s["flat"])
        s["ctx"].reset_adam()
        rep = s["ctx"].fit(gcp.AdamParams(**ADAM), p, q, 2 * p, 2 * q, iters=case["iters"], max_epochs=case["epochs"],
                           iter0=it)
        s["it"] += case["iters"] * case["epochs"]
        return {"first": rep["objective0"], "trace": rep["trace"], "A": s["ctx"].get_factors()}
    if kind == "dense":
        s["it"] += 1
        loss = gcp_autograd.sampled_loss(s["ctx"], it, p, q, s["A"])
        return {"loss": loss.detach(), "G": list(torch.autograd.grad(loss, s["A"]))}
    if kind == "fed":
        tau = case["tau"]
        s["batch"].local_steps(tau, gcp.AdamParams(**ADAM), it * tau, it * tau)
        s["it"] += 1
        s["batch"].server_step(gcp.AdamParams(**SERVER), s["it"])
        return {"loss": s["batch"].losses(), "U": s["clients"][0].get_factors()}
    ctx = s["ctx"]
    s["it"] += 1
    idx, x, w = ctx.sample(it, p, q)
    gcp.gcp_grad_samples_noalloc(ctx.dims, ctx.rank, ctx.loss, idx, x, w, s["flat"], s["out"], s["loss"])
    return {"idx": idx, "x": x, "w": w, "G": s["out"], "loss": s["loss"]}


# ------------------------------------------------------------ what it takes
def work(case):
    """Bytes and operations one pass cannot do without: each sample's record
    or hash bucket, the factors read once, the gradient (or the updated model
    and moments) written once; products and sums of the model entry, the loss
    and the all-mode gradient."""
    d, R, kind = len(_dims(case)), case["rank"], case["kind"]
    params = sum(_dims(case)) * R
    elt = 2 if case["dtype"] == "bf16" else 4
    p, q = case["p"], case["q"]
    S = p + q
    sample = (p * 4 if kind == "dense" else p * 4 * (d + 1)) + q * (32 if case["sampling"] == "stratified" else 0)
    model, grad = (d + 1) * R + 10, (3 * d + 1) * R
    if kind == "loss":
        return {"bytes": sample + params * elt, "flops": S * model}
    one = {"bytes": sample + params * (elt + 4), "flops": S * (model + grad)}
    step = {"bytes": sample + params * 24, "flops": S * (model + grad) + 12 * params}
    if kind == "steps":
        n = case["steps"]
        return {"bytes": n * step["bytes"] + 4 * params, "flops": n * step["flops"]}
    if kind == "fit":
        n, e = case["iters"] * case["epochs"], case["epochs"] + 1
        return {"bytes": n * step["bytes"] + e * 2 * sample + 8 * params, "flops": n * step["flops"] + e * 2 * S * model}
    if kind == "fed":
        n = case["clients"]
        return {"bytes": n * (case["tau"] * step["bytes"] + 8 * params) + 24 * params,
                "flops": n * case["tau"] * step["flops"] + n * params}
    if kind == "list":
        return {"bytes": sample + S * 8 * (d + 2) + params * 8, "flops": S * (model + grad)}
    return one


def tolerance(case):
    """About four times what the FP32 products and sums, whose order is not
    fixed, were measured to differ by from the same in FP64: gradients 4e-7
    (1.2e-6 where hot rows are summed one term at a time), factors after Adam
    1e-6 and objectives along a fit 4e-6.  Adam divides by the gradient's own
    size, so single entries whose terms nearly cancel move by a
    rounding-dependent share of the rate."""
    if case["kind"] in ("steps", "fit", "fed"):
        return {"rel": 2e-5, "max": 0.02}
    if case["kind"] == "list":
        return {"rel": 5e-6, "max": 5e-4}
    return {"rel": 2e-6, "max": 2e-4}


# -------------------------------------------------- the same in 64 bits
_MASK = 0xFFFFFFFF


def _s64(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >= 1 << 63 else v


def _mulhi(a, b):
    """High 64 bits of the unsigned product; b is a Python integer."""
    b0, b1 = b & _MASK, (b >> 32) & _MASK
    a0, a1 = a & _MASK, (a >> 32) & _MASK
    m = a0 * b0
    t = a1 * b0 + ((m >> 32) & _MASK)
    u = a0 * b1 + (t & _MASK)
    return a1 * b1 + ((t >> 32) & _MASK) + ((u >> 32) & _MASK)


def _philox(j, sub, it, k0, k1):
    """Philox4x64-10 of the counters (j, sub, it, 0) under the key (k0, k1)."""
    M0, M1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157
    c = [j, torch.full_like(j, _s64(sub)), torch.full_like(j, _s64(it)), torch.zeros_like(j)]
    for r in range(10):
        if r:
            k0, k1 = k0 + 0x9E3779B97F4A7C15, k1 + 0xBB67AE8584CAA73B
        a, ah, b, bh = c[0] * _s64(M0), _mulhi(c[0], M0), c[2] * _s64(M1), _mulhi(c[2], M1)
        c = [bh ^ c[1] ^ _s64(k0), b, ah ^ c[3] ^ _s64(k1), a]
    return c


def _cells(dims, j, sub, it, seed, stream):
    out = []
    for b in range(0, len(dims), 4):
        w = _philox(j, sub + b // 4, it, seed, stream)
        out += [_mulhi(w[k - b], dims[k]) for k in range(b, min(b + 4, len(dims)))]
    return torch.stack(out, 1)


def _linear(dims, idx):
    key = torch.zeros(idx.shape[0], dtype=torch.int64, device=idx.device)
    for k, I in enumerate(dims):
        key = key * I + idx[:, k]
    return key


def _present(keys, cand):
    at = torch.searchsorted(keys, cand).clamp_(max=keys.numel() - 1)
    return keys[at] == cand


def _draw_set(case, data, seed, it, p, q):
    """(cells, values, weights in FP64, whether a nonzero) of one sample set."""
    dims = _dims(case)
    M = math.prod(dims)
    if case["kind"] == "dense":
        idx = _cells(dims, torch.arange(p, device="cuda"), 0, it, seed, 2)
        x = data.reshape(-1)[_linear(dims, idx)].double()
        return idx, x, torch.full((p,), M / p, dtype=torch.float64, device="cuda"), torch.zeros(p, dtype=torch.bool, device="cuda")
    keys, vals = data
    N = keys.numel()
    e = _mulhi(_philox(torch.arange(p, device="cuda"), 0, it, seed, 0)[0], N)
    semi = case["sampling"] == "semi"
    j = torch.arange(q, device="cuda")
    z = _cells(dims, j, 0, it, seed, 3 if semi else 1)
    if not semi:
        for a in range(1, 64):
            bad = _present(keys, _linear(dims, z)).nonzero().reshape(-1)
            if not bad.numel():
                break
            z[bad] = _cells(dims, j[bad], 4 * a, it, seed, 1)
    idx = torch.cat([_coords(dims, keys[e]).to(torch.int64), z])
    x = torch.cat([vals[e].double(), torch.zeros(q, dtype=torch.float64, device="cuda")])
    w = torch.empty(p + q, dtype=torch.float64, device="cuda")
    w[:p] = N / max(p, 1)
    w[p:] = (M if semi else M - N) / max(q, 1)
    return idx, x, w, torch.arange(p + q, device="cuda") < p


def _f(loss, x, m):
    """(loss, derivative)"""
    eps = 1e-10
    if loss == "gaussian":
        return (x - m) ** 2, 2.0 * (m - x)
    if loss == "poisson":
        return m - x * torch.log(m + eps), 1.0 - x / (m + eps)
    if loss == "bernoulli":
        return torch.nn.functional.softplus(m, threshold=700.0) - x * m, torch.sigmoid(m) - x
    return x / (m + eps) + torch.log(m + eps), 1.0 / (m + eps) - x / (m + eps) ** 2


def _loss_grad(case, A, sample, want_grad=True):
    """Sampled loss and the per-mode gradients in FP64."""
    idx, x, w, nz = sample
    if case["dtype"] == "bf16":
        A = [a.float().bfloat16().double() for a in A]
    semi = case["sampling"] == "semi" and case["kind"] != "dense"
    G = [torch.zeros_like(a) for a in A] if want_grad else None
    F = torch.zeros((), dtype=torch.float64, device="cuda")
    for lo in range(0, idx.shape[0], 1 << 19):
        i, xs, ws, isnz = (t[lo:lo + (1 << 19)] for t in (idx, x, w, nz))
        rows = [a[i[:, k]] for k, a in enumerate(A)]
        m = rows[0].clone()
        for r in rows[1:]:
            m *= r
        m = m.sum(1)
        f, df = _f(case["loss"], xs, m)
        if semi:
            f0, df0 = _f(case["loss"], torch.zeros_like(xs), m)
            f, df = torch.where(isnz, f - f0, f), torch.where(isnz, df - df0, df)
        F += (ws * f).sum()
        if not want_grad:
            continue
        y = (ws * df).unsqueeze(1)
        for k in range(len(A)):
            t = y.expand_as(rows[0]).clone()
            for j, r in enumerate(rows):
                if j != k:
                    t *= r
            G[k].index_add_(0, i[:, k], t)
    return F, G


def _adam(A, B, C, G, t, lr, beta1, beta2, eps, lower):
    for a, b, c, g in zip(A, B, C, G):
        b.mul_(beta1).add_(g, alpha=1 - beta1)
        c.mul_(beta2).addcmul_(g, g, value=1 - beta2)
        a.sub_(lr * (b / (1 - beta1 ** t)) / torch.sqrt(c / (1 - beta2 ** t) + eps)).clamp_(min=lower)


def _flat(A):
    return torch.cat([a.reshape(-1) for a in A])


def exact(case, seed):
    kind, p, q = case["kind"], case["p"], case["q"]
    A = [a.double() for a in _start(case, seed)]
    zeros = lambda: [torch.zeros_like(a) for a in A]  # noqa: E731
    if kind == "fed":
        clients, losses = [], []
        for c in range(case["clients"]):
            data, M, B, C = _inputs(case, seed, c), [a.clone() for a in A], zeros(), zeros()
            for t in range(case["tau"]):
                F, G = _loss_grad(case, M, _draw_set(case, data, seed + c, t, p, q))
                _adam(M, B, C, G, t + 1, **ADAM)
            losses.append(float(F))
            clients.append(M)
        D = [a - sum(M[k] for M in clients) / len(clients) for k, a in enumerate(A)]
        _adam(A, zeros(), zeros(), D, 1, **SERVER)
        return {"loss": np.array(losses), "U": [a.cpu().numpy() for a in A]}
    data = _dense_inputs(case, seed) if kind == "dense" else _inputs(case, seed)
    if kind == "steps":
        B, C, losses = zeros(), zeros(), []
        for t in range(case["steps"]):
            F, G = _loss_grad(case, A, _draw_set(case, data, seed, t, p, q))
            _adam(A, B, C, G, t + 1, **ADAM)
            losses.append(F.reshape(1))
        return {"loss": torch.cat(losses), "A": _flat(A)}
    if kind == "fit":
        fixed = _draw_set(case, data, seed, 2 ** 64 - 1, 2 * p, 2 * q)
        B, C, trace, t, lr, it = zeros(), zeros(), [], 0, ADAM["lr"], 0
        first = best = float(_loss_grad(case, A, fixed, False)[0])
        for _ in range(case["epochs"]):
            kept, t0 = [[a.clone() for a in X] for X in (A, B, C)], t
            for _ in range(case["iters"]):
                G = _loss_grad(case, A, _draw_set(case, data, seed, it, p, q))[1]
                it, t = it + 1, t + 1
                _adam(A, B, C, G, t, **dict(ADAM, lr=lr))
            trace.append(float(_loss_grad(case, A, fixed, False)[0]))
            if trace[-1] < best:
                best = trace[-1]
            else:
                (A, B, C), t, lr = kept, t0, lr * 0.1
        return {"first": first, "trace": trace, "A": [a.cpu().numpy() for a in A]}
    sample = _draw_set(case, data, seed, 0, p, q)
    F, G = _loss_grad(case, A, sample, kind != "loss")
    if kind == "loss":
        return {"loss": float(F)}
    if kind == "dense":
        return {"loss": F, "G": G}
    if kind == "list":
        # the weights are FP32 inputs of the gradient call
        idx, x, w, nz = sample
        F, G = _loss_grad(case, A, (idx, x, w.float().double(), nz))
        return {"idx": None, "x": x, "w": w, "G": _flat(G), "loss": torch.stack([F, torch.zeros_like(F)])}
    if case.get("host"):
        return {"loss": float(F), "G": _flat(G)}
    return {"loss": F.reshape(1), "G": _flat(G)}
