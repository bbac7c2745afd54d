"""The calls whose speed is followed: this framework's entry points as a user's program makes them,
over the sizes, key types, payloads, model shapes and forward-pass forms of its workloads.

A case is a dict of plain values; `kind` says which entry point it goes through:

  sort     nnsort_sort of a device array under a model trained beforehand (in place, so a pass
           first refreshes the array from the unsorted keys, as a caller that keeps its input does)
  job      nnsort_train followed by nnsort_sort: the whole method on one array
  train    nnsort_train alone
  batch    nnsort_train_batch followed by nnsort_sort_batch: every array has its own model
  serve    a burst of host arrays through the continuous-batching server
  predict  positions and F(x) of every key
  grad     forward and backward pass of f as a torch.autograd.Function (a user's own training loop)
  radix    the no-model radix sort

Inputs follow the distributions of the repository's workloads (lognormal with duplicates, uniform,
Zipf-weighted Gaussian mixture, clusters, ...), drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1907_08817_gb300 as nns
from paper_1907_08817_gb300 import F32, F64, U32, U64

_M64 = (1 << 64) - 1
_CODE = {"f32": F32, "f64": F64, "u32": U32, "u64": U64}
_BYTES = {"f32": 4, "f64": 8, "u32": 4, "u64": 8}


# ------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest serving request: 10,000 float64 keys under a ready model; launches and waits
        dict(name="sort_10k_f64", kind="sort", dtype="f64", n=10_000, dist="lognormal", payload=False,
             layers=2, h1=32, h2=32, precision="fp32", eps=3),
        # a million uniform keys with everything at its defaults: train f, then sort
        dict(name="job_1m_f32", kind="job", dtype="f32", n=1_000_000, dist="uniform", payload=False,
             layers=1, h1=32, h2=0, precision="fp32", eps=3, sample_n=10_000, steps=100, batch=0),
        # 100 MB of keys whose distribution has shifted since f was trained; default options
        dict(name="sort_26m_f32_shift", kind="sort", dtype="f32", n=26_214_400, dist="shift",
             payload=False, layers=1, h1=32, h2=0, precision="fp32", eps=3),
        # the large sort: 2^28 skewed keys with duplicates, split-BF16 tensor-core forward pass
        dict(name="sort_268m_f32", kind="sort", dtype="f32", n=1 << 28, dist="lognormal_dup",
             payload=False, layers=2, h1=64, h2=64, precision="bf16x2", eps="auto"),
        # ... and the training of its model on a 1% sample
        dict(name="train_268m_f32", kind="train", dtype="f32", n=1 << 28, dist="lognormal_dup",
             layers=2, h1=64, h2=64, sample_n=2_684_354, steps=100, batch=65_536),
        # a database's sort: 64-bit keys, each with the row it came from
        dict(name="sort_64m_u64_kv", kind="sort", dtype="u64", n=1 << 26, dist="gauss_mix",
             payload=True, layers=2, h1=32, h2=32, precision="bf16x2", eps="auto"),
        # record ids, an odd count, the compiled form of f
        dict(name="sort_50m_u64_pwl", kind="sort", dtype="u64", n=50_426_265, dist="uniform",
             payload=False, layers=1, h1=32, h2=0, precision="pwl", eps=3),
        # many arrays of uneven sizes, each with its own small model
        dict(name="batch_1024", kind="batch", dtype="f32", count=1024, lo=1000, hi=1_000_000, h1=16,
             steps=100),
        # a burst of requests to the server: per-request training, host memory to host memory
        dict(name="serve_16", kind="serve", dtype="f64", count=16, lo=10_000, hi=1_000_000, h1=32,
             h2=32, sample_n=20_000, steps=100, batch=4096),
        # positions of a ragged array in the plain binary32 form of the large model
        dict(name="predict_16m_fp32", kind="predict", dtype="f32", n=16_777_259, dist="lognormal_dup",
             layers=2, h1=64, h2=64, precision="fp32"),
        # one step of a user's own training loop on the large model
        dict(name="grad_65k", kind="grad", n=65_536, layers=2, h1=64, h2=64),
        # the sort without a model, 32-bit keys with payload, an odd count
        dict(name="radix_33m_u32_kv", kind="radix", dtype="u32", n=33_554_467, dist="uniform",
             payload=True),
    ]


def _log_int(rng, lo, hi):
    return int(math.floor(lo * (hi / lo) ** rng.random())) | (1 if rng.random() < 0.5 else 0)


def draw(rng):
    kind = rng.choice(["sort", "sort", "sort", "sort", "job", "train", "batch", "serve", "predict",
                       "grad", "radix"])
    dtype = rng.choice(["f32", "f32", "f64", "u32", "u64"])
    dist = rng.choice({"f32": ["uniform", "lognormal", "lognormal_dup", "normal", "exponential", "shift"],
                       "f64": ["uniform", "lognormal", "clustered"],
                       "u32": ["uniform"], "u64": ["uniform", "gauss_mix"]}[dtype])
    layers = rng.choice([1, 2])
    h1 = rng.choice([16, 32, 64] if layers == 1 else [32, 64])
    h2 = 0 if layers == 1 else h1
    if kind == "sort":
        precision = rng.choice(["fp32", "fp32", "pwl", "bf16x2"])
        # the binary32 form of the widest model is the dearest per key
        top = (1 << 26) if precision != "fp32" else (1 << 24)
        return dict(kind=kind, dtype=dtype, n=_log_int(rng, 10_000, top), dist=dist,
                    payload=rng.random() < 0.5, layers=layers, h1=h1, h2=h2, precision=precision,
                    eps=rng.choice([3, "auto"]))
    if kind == "job":
        n = _log_int(rng, 10_000, 1 << 24)
        return dict(kind=kind, dtype=dtype, n=n, dist=dist, payload=rng.random() < 0.5, layers=1,
                    h1=rng.choice([16, 32]), h2=0, precision=rng.choice(["fp32", "pwl"]), eps=3,
                    sample_n=min(20_000, max(1000, n // 100)), steps=100, batch=0)
    if kind == "train":
        sample = _log_int(rng, 10_000, 1 << 20)
        return dict(kind=kind, dtype=dtype, n=_log_int(rng, 1 << 20, 1 << 26), dist=dist, layers=layers,
                    h1=h1, h2=h2, sample_n=sample, steps=100,
                    batch=rng.choice([0, 4096]) if sample < 50_000 else rng.choice([4096, 65_536]))
    if kind == "batch":
        return dict(kind=kind, dtype="f32", count=_log_int(rng, 16, 1024), lo=1000,
                    hi=rng.choice([100_000, 1_000_000]), h1=rng.choice([16, 32]), steps=100)
    if kind == "serve":
        return dict(kind=kind, dtype="f64", count=rng.randrange(2, 25), lo=10_000,
                    hi=_log_int(rng, 100_000, 1_000_000), h1=32, h2=32, sample_n=20_000, steps=100,
                    batch=4096)
    if kind == "predict":
        precision = rng.choice(["fp32", "pwl", "bf16x2"])
        return dict(kind=kind, dtype=dtype, n=_log_int(rng, 10_000, 1 << 24), dist=dist, layers=layers,
                    h1=h1, h2=h2, precision=precision)
    if kind == "grad":
        return dict(kind=kind, n=_log_int(rng, 1000, 1 << 20), layers=layers, h1=h1, h2=h2)
    return dict(kind="radix", dtype=dtype, n=_log_int(rng, 10_000, 1 << 26), dist=dist,
                payload=rng.random() < 0.5)


# ---------------------------------------------------------------------------------------- inputs
def _gen(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + tag * 7_919 + 1) % (1 << 62))
    return g


def _keys(dist, dtype, n, seed, tag=0):
    """n keys on the GPU; unsigned types travel as same-width signed storage."""
    g = _gen(seed, tag)
    if dtype in ("u32", "u64"):
        if dist == "gauss_mix":
            w = torch.arange(1, 9, device="cuda", dtype=torch.float64) ** -1.1
            edges = torch.cumsum(w / w.sum(), 0)
            u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
            comp = torch.bucketize(u, edges).clamp_(max=7).to(torch.float64)
            v = (2.0 * comp + 1.0) / 16.0 * 2.0 ** 63
            v += torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * (2.0 ** 63 / 64.0)
            v.round_().clamp_(0.0, 2.0 ** 64 - 4096.0)
            k = torch.where(v >= 2.0 ** 63, v - 2.0 ** 64, v).to(torch.int64)
            return (k & ~0x7FF) | torch.randint(0, 2048, (n,), generator=g, device="cuda")
        hi = torch.randint(0, 1 << 32, (n,), generator=g, device="cuda")
        if dtype == "u32":
            return hi.to(torch.int32)  # the low 32 bits
        return (hi << 32) | torch.randint(0, 1 << 32, (n,), generator=g, device="cuda")
    t = torch.float32 if dtype == "f32" else torch.float64

    def normal(m):
        return torch.randn(m, generator=g, device="cuda", dtype=t)

    def uniform(m):
        return torch.rand(m, generator=g, device="cuda", dtype=t)
    if dist == "uniform":
        return uniform(n)
    if dist == "normal":
        return normal(n)
    if dist == "exponential":
        return -torch.log1p(-uniform(n))
    if dist == "lognormal":
        return torch.exp_(normal(n).mul_(2.0))
    if dist == "lognormal_dup":  # 5% exact copies of other keys, scattered
        k = torch.exp_(normal(n).mul_(2.0))
        return torch.where(uniform(n) < 0.05, k[torch.randint(0, n, (n,), generator=g, device="cuda")], k)
    if dist == "shift":  # 30% of the keys crowd around 0.5
        k = uniform(n)
        return torch.where(uniform(n) < 0.3, normal(n).mul_(0.1).add_(0.5), k)
    if dist == "clustered":
        centres = uniform(16) * 1e6
        return centres[torch.randint(0, 16, (n,), generator=g, device="cuda")] + normal(n)
    raise ValueError(dist)


def _order(k, dtype):
    """Signed integers in the keys' order (the order image less 2^63, or 2^31 for 32-bit keys)."""
    if dtype == "f32":
        b = k.view(torch.int32).to(torch.int64)
        return torch.where(b < 0, -b - (1 << 31) - 1, b)
    if dtype == "f64":
        b = k.view(torch.int64)
        return torch.where(b < 0, ~b ^ torch.iinfo(torch.int64).min, b)
    k = k.to(torch.int64)
    return k ^ (torch.iinfo(torch.int64).min if dtype == "u64" else -(1 << 31))


def _fit(keys, dtype, layers, h1, h2, seed):
    """A model that a program has trained earlier, elsewhere: Adam on a sample's empirical CDF (the
    training recipe of the workloads, in torch), so that it is the same model whatever the
    framework's own training does."""
    S = 16_384
    g = _gen(seed, 77)
    pick = torch.randint(0, keys.numel(), (S,), generator=g, device="cuda")
    o = torch.sort(_order(keys[pick], dtype)).values
    lo, hi = int(o[0]), int(o[-1])
    scale = 1.0 / (hi - lo) if hi > lo else 1.0
    x = ((o.double() - float(lo)) * scale).float().unsqueeze(1)
    y = (torch.arange(S, device="cuda") / S).float().unsqueeze(1)

    def uni(*shape):
        return torch.rand(*shape, generator=g, device="cuda") * 2.0 - 1.0
    w1 = uni(h1, 1) * math.sqrt(6.0)
    p = [w1, -w1[:, 0] * torch.rand(h1, generator=g, device="cuda")]
    if layers == 2:
        p += [uni(h2, h1) * math.sqrt(6.0 / h1), torch.zeros(h2, device="cuda")]
    last = h2 if layers == 2 else h1
    p += [uni(1, last) * math.sqrt(6.0 / last), torch.zeros(1, device="cuda")]
    for q in p:
        q.requires_grad_(True)
    opt = torch.optim.Adam(p, lr=1e-2)
    for _ in range(150):
        opt.zero_grad(set_to_none=True)
        h = x
        for i in range(0, len(p) - 2, 2):
            h = torch.relu(torch.addmm(p[i + 1], h, p[i].t()))
        loss = (torch.addmm(p[-1], h, p[-2].t()) - y).square().mean()
        loss.backward()
        opt.step()
    flat = torch.cat([q.detach().reshape(-1) for q in p]).cpu().numpy()
    off = (1 << 31) if dtype in ("f32", "u32") else (1 << 63)
    return nns.Model.create(_CODE[dtype], layers, h1, h2, flat, translate="ordbits",
                            lo_bits=(lo + off) & _M64, lo_val=0.0, scale=scale)


def _sizes(count, lo, hi):
    """The case's array sizes, spread over the logarithm of [lo, hi] (the same for every seed)."""
    u = np.random.Generator(np.random.PCG64(count + hi)).random(count)
    return np.floor(lo * (hi / lo) ** u).astype(np.int64)


def _key_type(dtype):
    return dtype if dtype in ("u32", "u64") else None


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": int(seed)}
    if kind == "grad":
        L, h1, h2 = case["layers"], case["h1"], case["h2"]
        g = _gen(seed, 3)
        w1 = (torch.rand(h1, generator=g, device="cuda") * 2 - 1) * math.sqrt(6.0)
        p = [w1, -w1 * torch.rand(h1, generator=g, device="cuda")]
        if L == 2:
            p += [(torch.rand(h2 * h1, generator=g, device="cuda") * 2 - 1) * math.sqrt(6.0 / h1),
                  (torch.rand(h2, generator=g, device="cuda") * 2 - 1) * 0.1]
        last = h2 if L == 2 else h1
        p += [(torch.rand(last, generator=g, device="cuda") * 2 - 1) * math.sqrt(6.0 / last),
              torch.zeros(1, device="cuda")]
        s["params"] = torch.cat(p).requires_grad_(True)
        s["x"] = torch.rand(case["n"], generator=g, device="cuda").requires_grad_(True)
        s["gy"] = torch.randn(case["n"], generator=g, device="cuda") / case["n"]
        return s
    if kind == "batch":
        sizes = _sizes(case["count"], case["lo"], case["hi"])
        dists = ("uniform", "normal", "lognormal", "exponential")
        s["keys"] = torch.cat([_keys(dists[j % 4], "f32", int(n), seed, j) for j, n in enumerate(sizes)])
        s["work"] = torch.empty_like(s["keys"])
        s["arrays"] = list(torch.split(s["work"], [int(n) for n in sizes]))
        s["sample_ns"] = [max(1, int(n) // 100) for n in sizes]
        return s
    if kind == "serve":
        sizes = _sizes(case["count"], case["lo"], case["hi"])
        dists = ("uniform", "lognormal", "clustered")
        s["keys"] = [_keys(dists[j % 3], "f64", int(n), seed, j).cpu().numpy() for j, n in enumerate(sizes)]
        s["work"] = [k.copy() for k in s["keys"]]
        s["server"] = nns.Server(workers=2, max_batch=32, train=dict(
            layers=2, h1=case["h1"], h2=case["h2"], sample_n=case["sample_n"], steps=case["steps"],
            batch=case["batch"]))
        return s
    s["keys"] = _keys(case["dist"], case["dtype"], case["n"], seed)
    if kind in ("sort", "job", "radix"):
        s["work"] = torch.empty_like(s["keys"])
        if case["payload"]:
            s["rows"] = torch.arange(case["n"], device="cuda", dtype=torch.int32)
            s["pay"] = torch.empty_like(s["rows"])
    if kind in ("sort", "predict"):
        # "shift": the model was trained before the crowd arrived
        old = _keys("uniform", case["dtype"], 1 << 20, seed, 9) if case["dist"] == "shift" else s["keys"]
        s["model"] = _fit(old, case["dtype"], case["layers"], case["h1"], case["h2"], seed)
    return s


# ------------------------------------------------------------------------------------- one pass
def _train(s, keys):
    c = s["case"]
    return nns.train(keys, key_type=_key_type(c["dtype"]), layers=c["layers"], h1=c["h1"], h2=c["h2"],
                     sample_n=c["sample_n"], steps=c["steps"], batch=c["batch"], lr=1e-2, seed=s["seed"])


def _refresh(s):
    s["work"].copy_(s["keys"])
    if "pay" in s:
        s["pay"].copy_(s["rows"])
    return s["work"], s.get("pay")


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "grad":
        p, x = state["params"], state["x"]
        y = nns.NNSortMLPFunction.apply(p, x, c["layers"], c["h1"], c["h2"])
        gp, gx = torch.autograd.grad(y, (p, x), state["gy"])
        return {"y": y.detach(), "gp": gp, "gx": gx}
    if kind == "batch":
        state["work"].copy_(state["keys"])
        models, loss = nns.train_batch(state["arrays"], sample_ns=state["sample_ns"], h1=c["h1"],
                                       steps=c["steps"], seed=state["seed"])
        nns.sort_batch(state["arrays"], models, eps="auto", stats=False)
        return {"keys": state["work"], "loss": loss}
    if kind == "serve":
        for a, b in zip(state["work"], state["keys"]):
            np.copyto(a, b)
        srv = state["server"]
        tickets = [srv.submit(a, seed=state["seed"] + j) for j, a in enumerate(state["work"])]
        for t in tickets:
            srv.wait(t)
        return list(state["work"])
    kt = _key_type(c["dtype"])
    if kind == "predict":
        slots, y = nns.predict(state["keys"], state["model"], precision=c["precision"], key_type=kt)
        return {"slots": slots, "y": y}
    if kind == "train":
        model, loss = _train(state, state["keys"])
        return {"params": model.describe()[1], "loss": loss}
    keys, pay = _refresh(state)
    if kind == "radix":
        nns.radix_sort(keys, pay, key_type=kt)
        return {"keys": keys, "pay": pay}
    if kind == "job":
        model, loss = _train(state, keys)
        nns.sort(keys, pay, model, eps=c["eps"], precision=c["precision"], key_type=kt)
        return {"keys": keys, "pay": pay, "params": model.describe()[1], "loss": loss}
    st = nns.sort(keys, pay, state["model"], eps=c["eps"], precision=c["precision"], key_type=kt)
    # the counts of the method's analysis: conflict arrays, placed and out-of-order elements, repairs
    counts = st["w_size"] + st["placed"] + st["out_of_order"] + [st["repaired"], st["repair_ranges"]]
    return {"keys": keys, "pay": pay, "counts": np.array(counts, dtype=np.int64)}


# ------------------------------------------------------------------------------- work and values
def _net_flops(layers, h1, h2):
    return 2 * (2 * h1) if layers == 1 else 2 * (h1 + h1 * h2 + h2)


def work(case):
    kind = case["kind"]
    net = _net_flops(case.get("layers", 1), case.get("h1", 0), case.get("h2", 0))
    if kind == "grad":  # x and gy in, y and gx out
        return {"bytes": 16.0 * case["n"], "flops": 3.0 * net * case["n"]}
    if kind in ("batch", "serve"):
        n = float(sum(_sizes(case["count"], case["lo"], case["hi"])))
        if kind == "batch":  # keys in and out; 100 full-batch steps on 1% samples
            net = _net_flops(1, case["h1"], 0)
            return {"bytes": 8.0 * n, "flops": net * n + 3.0 * net * case["steps"] * n / 100.0}
        net = _net_flops(2, case["h1"], case["h2"])
        return {"bytes": 16.0 * n, "flops": net * n + 3.0 * net * case["steps"] * case["batch"] * case["count"]}
    n, kb = float(case["n"]), _BYTES[case["dtype"]]
    moved = 2.0 * n * (kb + (4 if case.get("payload") else 0))  # each array in and out once
    if kind == "radix":
        return {"bytes": moved, "flops": 0.0}
    if kind == "predict":  # keys in; position and F(x) out
        return {"bytes": n * (kb + 8 + 4), "flops": n * (2.0 if case["precision"] == "pwl" else net)}
    learn = 3.0 * net * case.get("steps", 0) * (case.get("batch") or case.get("sample_n", 0))
    if kind == "train":
        return {"bytes": float(case["sample_n"]) * kb, "flops": learn}
    return {"bytes": moved, "flops": learn + n * (2.0 if case["precision"] == "pwl" else net)}


def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _draws(seed, start, count):
    """SplitMix64 draws start .. start + count - 1 of the stream `seed`."""
    with np.errstate(over="ignore"):
        i = np.arange(start + 1, start + count + 1, dtype=np.uint64)
        return _mix(np.uint64(seed & _M64) + i * np.uint64(0x9E3779B97F4A7C15))


def _below(u, n):
    """floor(u n / 2^64)"""
    lo, hi = u & np.uint64(0xFFFFFFFF), u >> np.uint64(32)
    return ((hi * np.uint64(n) + ((lo * np.uint64(n)) >> np.uint64(32))) >> np.uint64(32)).astype(np.int64)


def _unit(u):
    return (u >> np.uint64(11)).astype(np.float64) / 2.0 ** 53


def _train_exact(c, keys, seed):
    """The training recipe in 64 bits: (parameters, losses)."""
    S, steps, batch = c["sample_n"], c["steps"], c["batch"]
    layers, h1, h2 = c["layers"], c["h1"], c["h2"]
    rows = torch.from_numpy(_below(_draws(int(_draws(seed, 1, 1)[0]), 0, S), keys.numel())).cuda()
    o = torch.sort(_order(keys[rows], c["dtype"])).values
    lo, hi = int(o[0]), int(o[-1])
    scale = float(np.float32(1.0 / (hi - lo) if hi > lo else 1.0))
    x = ((o - lo) if hi - lo < 1 << 62 else (o.double() - float(lo))).double() * scale
    lab = torch.arange(S, device="cuda", dtype=torch.float64) / S
    s, k = int(_draws(seed, 2, 1)[0]), 0

    def uni(m):
        nonlocal k
        k += m
        return _unit(_draws(s, k - m, m))
    w1 = ((2.0 * uni(h1) - 1.0) * math.sqrt(6.0)).astype(np.float32)
    p = [w1, (-w1.astype(np.float64) * uni(h1)).astype(np.float32)]
    if layers == 2:
        p += [((2.0 * uni(h2 * h1) - 1.0) * math.sqrt(6.0 / h1)).astype(np.float32), np.zeros(h2, np.float32)]
    last = h2 if layers == 2 else h1
    p += [((2.0 * uni(last) - 1.0) * math.sqrt(6.0 / last)).astype(np.float32), np.zeros(1, np.float32)]
    p = torch.from_numpy(np.concatenate(p).astype(np.float64)).cuda().requires_grad_(True)
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    bs = int(_draws(seed, 3, 1)[0])
    b1, b2, lr, eps = (float(np.float32(q)) for q in (0.9, 0.999, 1e-2, 1e-8))
    for t in range(steps):
        xb, lb = x, lab
        if batch:
            at = torch.from_numpy(_below(_draws(bs, t * batch, batch), S)).cuda()
            xb, lb = x[at], lab[at]
        loss = (_net(p, xb, layers, h1, h2) - lb).square().mean()
        g, = torch.autograd.grad(loss, p)
        losses.append(loss.detach())
        with torch.no_grad():
            m.mul_(b1).add_(g, alpha=1 - b1)
            v.mul_(b2).addcmul_(g, g, value=1 - b2)
            p -= lr * (m / (1 - b1 ** (t + 1))) / ((v / (1 - b2 ** (t + 1))).sqrt() + eps)
    return p.detach(), torch.stack(losses)


def _net(p, x, layers, h1, h2):
    h = torch.relu(x[:, None] * p[:h1] + p[h1:2 * h1])
    at = 2 * h1
    if layers == 2:
        h = torch.relu(h @ p[at:at + h2 * h1].reshape(h2, h1).t() + p[at + h2 * h1:at + h2 * h1 + h2])
        at += h2 * h1 + h2
    return h @ p[at:-1] + p[-1]


def _sorted(keys, dtype):
    return torch.sort(keys).values.double() if dtype in ("f32", "f64") else None


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sort", "radix") and case["dtype"] not in ("f32", "f64"):
        return None  # whole numbers throughout
    s = prepare(case, seed)
    if kind == "grad":
        p = s["params"].detach().double().requires_grad_(True)
        x = s["x"].detach().double().requires_grad_(True)
        y = _net(p, x, case["layers"], case["h1"], case["h2"])
        gp, gx = torch.autograd.grad(y, (p, x), s["gy"].double())
        return {"y": y.detach(), "gp": gp, "gx": gx}
    if kind == "batch":
        parts = torch.split(s["keys"], [a.numel() for a in s["arrays"]])
        return {"keys": torch.cat([torch.sort(k).values for k in parts]).double(), "loss": None}
    if kind == "serve":
        return [np.sort(k) for k in s["keys"]]
    dt = case["dtype"]
    if kind == "predict":
        d, p = s["model"].describe()
        off = (1 << 31) if dt in ("f32", "u32") else (1 << 63)
        o, lo = _order(s["keys"], dt), d["lo_bits"] - off
        p = torch.from_numpy(p).cuda().double()
        y = torch.empty(case["n"], device="cuda", dtype=torch.float64)
        for a in range(0, case["n"], 1 << 21):
            part = o[a:a + (1 << 21)]
            y[a:a + (1 << 21)] = _net(p, (part.double() - float(lo)) * d["scale"], case["layers"],
                                      case["h1"], case["h2"])
        return {"slots": None, "y": y}
    if kind in ("train", "job"):
        params, loss = _train_exact(case, s["keys"], s["seed"])
        if kind == "train":
            return {"params": params, "loss": loss}
        return {"keys": _sorted(s["keys"], dt), "pay": None, "params": params, "loss": loss}
    return {"keys": _sorted(s["keys"], dt), "pay": None, "counts": None}
