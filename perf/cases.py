"""The work whose speed counts: what a user of the packed ensembles has the
library do, as cases that can be prepared, run and checked.

A training pass is a few consecutive steps of one pack (the call a training
loop repeats), after which every member's parameters are copied out (the
checkpoint that such a loop takes).  A prediction pass is one validation or
serving call, a selection pass one greedy ensemble selection.  Sizes are the
repository's own workloads (tiny, medium, large, narrow, wide); ``draw`` takes
sizes, tasks, precisions and options from the ranges around them.

Member hyperparameters follow from the case (its ``hp`` number), so that the
work does not depend on the seed; data, batches, initial parameters and
dropout masks follow from the seed.
"""
import math

import numpy as np
import torch

import paper_2607_05380_gb300 as tp

DEV = "cuda"
MASK32 = 0xFFFFFFFF
AUC_POOL, LOSS_POOL = 266, 96


# ------------------------------------------------------------------ the cases
def _train(name, **kw):
    c = dict(name=name, kind="train", task="regression", precision="bf16", d_in=64, d_out=1, m=8, depth_lo=1,
             depth_hi=3, w_lo=64, w_hi=256, w_step=16, p_lo=0.0, p_hi=0.3, batch=256, steps=4, stacked=False,
             muon=False, emb=False, hp=1)
    c.update(kw)
    return c


MEDIUM = dict(m=32, depth_lo=1, depth_hi=4, w_lo=128, w_hi=1024, w_step=64, p_hi=0.5)
LARGE = dict(task="multiclass", d_in=900, d_out=10, m=64, depth_lo=1, depth_hi=4, w_lo=256, w_hi=1024, w_step=128,
             p_hi=0.5)


def listed():
    return [
        # one epoch of a small table (2048 rows): launches and latency decide
        _train("tiny_epoch", task="binary", d_in=8, batch=256, steps=8),
        # an ordinary regression table, shared batches, AdamW
        _train("medium", batch=512, steps=2, **MEDIUM),
        # the same pack trained in 32-bit arithmetic, on a table of odd width and an odd batch
        _train("medium_fp32", precision="fp32", d_in=61, batch=500, steps=2, **MEDIUM),
        # members that read periodic feature embeddings of the table
        _train("medium_emb", emb=True, batch=512, steps=4, **MEDIUM),
        # many narrow ragged members: tile scheduling and many small optimizer segments
        _train("narrow", task="binary", d_in=128, m=256, w_lo=32, batch=256, steps=16),
        # a wide table with ten classes
        _train("large", batch=1024, steps=2, **LARGE),
        # the method's own training set-up on it: Muon on the hidden weights, a batch per member
        _train("large_muon_stacked", muon=True, stacked=True, batch=1024, steps=1, **LARGE),
        # wide members, near-dense matrix products
        _train("wide", d_in=512, m=16, depth_lo=4, depth_hi=4, w_lo=1024, w_hi=2048, w_step=256, p_hi=0.2,
               batch=2048, steps=1),
        # a validation pass over a table whose rows are no multiple of any tile
        dict(_train("predict_large", **LARGE), kind="predict", rows=20011),
        # a serving call: a few rows through every member
        dict(_train("predict_small", **MEDIUM), kind="predict", rows=37),
        # greedy selection by ROC-AUC from the narrow workload's pool at the end of an epoch
        dict(name="select_auc", kind="select", task="binary", score="auc", pool=AUC_POOL, rows=60000, d_out=1, m_ens=32),
        # greedy selection by cross-entropy from the large workload's pool
        dict(name="select_loss", kind="select", task="multiclass", score="loss", pool=LOSS_POOL, rows=100000, d_out=10,
             m_ens=32),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.999)) - 0.5 / hi)))))


def draw(rng):
    """One more case: its kind, task, precision and options at random, sizes
    spread over their logarithm, odd ones among them."""
    kind = rng.choice(["train", "train", "train", "train", "predict", "select"])
    task = rng.choice(["binary", "regression", "multiclass", "multiclass"])
    if kind == "select":
        scores = {"binary": ["loss", "accuracy", "auc", "auc"], "regression": ["loss", "rmse"],
                  "multiclass": ["loss", "accuracy"]}[task]
        d_out = rng.randint(2, 20) if task == "multiclass" else 1
        rows = _log_int(rng, 200, 100000)
        pool = max(4, min(_log_int(rng, 8, 300), int(9e7 / (rows * d_out)), int(1.6e7 / rows) + 4))
        return dict(kind="select", task=task, score=rng.choice(scores), pool=pool, rows=rows, d_out=d_out,
                    m_ens=rng.choice([4, 16, 32]))
    while True:
        w_hi = 16 * _log_int(rng, 2, 128)
        d_lo = rng.randint(1, 4)
        c = _train("", kind=kind, task=task, precision=rng.choice(["bf16", "bf16", "bf16", "fp32"]),
                   d_in=_log_int(rng, 4, 1000), d_out=rng.randint(2, 20) if task == "multiclass" else 1,
                   m=_log_int(rng, 2, 256), depth_lo=d_lo, depth_hi=rng.randint(d_lo, 4),
                   w_lo=16 * rng.randint(1, w_hi // 16), w_hi=w_hi, p_hi=rng.choice([0.0, 0.3, 0.5]),
                   batch=_log_int(rng, 32, 2048), steps=2, hp=rng.randrange(1 << 16))
        del c["name"]
        if kind == "train":
            c.update(stacked=rng.random() < 0.3, muon=rng.random() < 0.25)
            c.update(steps=1 if c["muon"] or w_hi >= 1024 else 2)
        else:
            c.update(rows=_log_int(rng, 1, 30000))
        c.update(emb=c["d_in"] <= 64 and rng.random() < 0.3)
        w = work(c)
        if w["flops"] <= (1e12 if c["precision"] == "bf16" else 1e11) and _param_bytes(c) <= 6e8:
            return c


# ----------------------------------------------- members of a case, its sizes
def _members(c):
    """Hyperparameters of the case's members (independent of the seed)."""
    r = np.random.default_rng([c["hp"], 11])
    m = c["m"]
    depth = r.integers(c["depth_lo"], c["depth_hi"] + 1, m).astype(np.int32)
    width = (c["w_step"] * r.integers(-(-c["w_lo"] // c["w_step"]), c["w_hi"] // c["w_step"] + 1, m)).astype(np.int32)
    h = dict(depth=depth, width=width, dropout=r.uniform(c["p_lo"], c["p_hi"], m).astype(np.float32),
             lr=np.exp(r.uniform(math.log(1e-4), math.log(3e-3), m)).astype(np.float32),
             wd=np.exp(r.uniform(math.log(1e-5), math.log(1e-2), m)).astype(np.float32),
             lr_muon=np.exp(r.uniform(math.log(1e-3), math.log(1e-1), m)).astype(np.float32))
    h["d_emb"] = (8 + 4 * r.integers(0, 7, m)).astype(np.int32)
    h["sigma"] = np.exp(r.uniform(math.log(1e-2), math.log(10.0), m))
    return h


def _in0(c, h, i):
    return c["d_in"] * (int(h["d_emb"][i]) if c["emb"] else 1)


def _blocks(c, h, i):
    """A member's parameter run as the library documents it: (kind, layer,
    offset, rows, columns, padded columns) of every block, and its length."""
    up = lambda v, a: -(-v // a) * a  # noqa: E731
    L, w, off, got = int(h["depth"][i]), int(h["width"][i]), 0, []
    for l in range(L + 1):
        n_in = _in0(c, h, i) if l == 0 else w
        pad = up(n_in, 8) if l == 0 else w
        out = c["d_out"] if l == L else w
        off = up(off, 32)
        got.append(("W", l, off, out, n_in, pad))
        off = up(off + out * pad, 32)
        got.append(("b", l, off, out, 1, 1))
        off += out
    if c["emb"]:
        off = up(off, 32)
        got.append(("e", L + 1, off, c["d_in"] * (4 * int(h["d_emb"][i]) - 2), 1, 1))
        off += c["d_in"] * (4 * int(h["d_emb"][i]) - 2)
    return got, off


def _param_bytes(c):
    h = _members(c)
    return 4.0 * sum(_blocks(c, h, i)[1] for i in range(c["m"]))


def work(c):
    if c["kind"] == "select":
        # every prediction and label read once; a term per candidate, row and member taken
        return {"bytes": 4.0 * c["pool"] * c["rows"] * c["d_out"] + 4.0 * c["rows"],
                "flops": 4.0 * c["m_ens"] * c["pool"] * c["rows"]}
    h = _members(c)
    fwd = bwd = ns = params = 0.0
    for i in range(c["m"]):
        L, w, n0 = float(h["depth"][i]), float(h["width"][i]), float(_in0(c, h, i))
        first, hidden, head = n0 * w, (L - 1) * w * w, w * c["d_out"]
        params += first + hidden + head + L * w + c["d_out"]
        fwd += 2 * (first + hidden + head)
        bwd += 2 * (first + 2 * hidden + 2 * head) + (2 * first if c["emb"] else 0)
        for k, n_in in ((1, n0), (L - 1, w)):
            r, q = min(n_in, w), max(n_in, w)
            ns += k * 5 * (4 * r * r * q + 2 * r * r * r)
    if c["kind"] == "predict":
        return {"bytes": 4.0 * params + 4.0 * c["rows"] * (c["d_in"] + c["m"] * c["d_out"]),
                "flops": c["rows"] * fwd}
    rows = c["batch"] * (c["m"] if c["stacked"] else 1)
    # parameters and optimizer state read and written once a step, the batch read, the members copied out once
    return {"bytes": c["steps"] * (24.0 * params + 4.0 * rows * (c["d_in"] + 2)) + 4.0 * params,
            "flops": c["steps"] * (c["batch"] * (fwd + bwd) + (ns if c["muon"] else 0))}


# -------------------------------------------------------------------- inputs
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _table(c, seed, n):
    """Features as tables have them (normal, some heavy-tailed columns, some
    one-hot ones where the table is wide) and labels from a random teacher."""
    g = _gen(seed, 1)
    d = c["d_in"]
    X = torch.randn(n, d, generator=g, device=DEV)
    heavy = min(8, d // 8)
    if heavy:
        chi2 = (torch.randn(n, heavy, 3, generator=g, device=DEV) ** 2).sum(-1)
        X[:, :heavy] /= torch.sqrt(chi2 / 3.0)
    if d >= 300:
        cats = 10 * (d // 30)
        X[:, d - cats:] = 0.0
        hot = torch.randint(0, 10, (n, cats // 10), generator=g, device=DEV)
        X.scatter_(1, d - cats + hot + 10 * torch.arange(cats // 10, device=DEV), 1.0)
    t = torch.randn(d, 64, generator=g, device=DEV) / math.sqrt(d)
    t = torch.relu(X @ t) @ (torch.randn(64, c["d_out"], generator=g, device=DEV) / 8.0)
    if c["task"] == "multiclass":
        y = torch.argmax(t, 1).to(torch.int32)
    elif c["task"] == "binary":
        y = (t[:, 0] > t[:, 0].median()).to(torch.int32)
    else:
        y = t[:, 0] + 0.1 * torch.randn(n, generator=g, device=DEV)
        y = ((y - y.mean()) / y.std()).float()
    return X.contiguous(), y.contiguous()


def _batches(c, seed, n):
    """Row indices [steps, B] (or [steps, m, B]: a batch per member)."""
    g = _gen(seed, 2)
    shape = (c["steps"], c["m"], c["batch"]) if c["stacked"] else (c["steps"], c["batch"])
    return torch.randint(0, n, shape, generator=g, device=DEV, dtype=torch.int32)


def _emb_values(c, h, seed):
    """Embedding parameters (w, b, alpha, beta) of every member, as training
    leaves them: w near its draw N(0, sigma), the others moved off zero."""
    r = np.random.default_rng([seed, 3])
    got = []
    for i in range(c["m"]):
        n, d = c["d_in"], int(h["d_emb"][i])
        got.append([a.astype(np.float32) for a in (r.normal(0, h["sigma"][i], (n, d - 1)), r.normal(0, 0.3, (n, d - 1)),
                                                   r.normal(0.3, 0.2, (n, d)), r.normal(0, 0.1, (n, d)))])
    return got


def _trained_run(c, h, i, g):
    """A member's parameter run with weights of a trained member's size."""
    blocks, n = _blocks(c, h, i)
    run = torch.zeros(n, device=DEV)
    for kind, l, off, out, n_in, pad in blocks:
        v = run[off:off + out * pad].view(out, pad)[:, :n_in]
        if kind == "W":
            v.copy_(torch.randn(out, n_in, generator=g, device=DEV) * math.sqrt(2.0 / n_in))
        else:
            v.copy_(torch.randn(out, n_in, generator=g, device=DEV) * 0.1)
    return run


def _pack_seed(seed):
    return int(seed) * 2654435761 % (1 << 48) + 5


def _pool(c, seed):
    """Candidates' predictions [P, N, d_out] that share the signal and part
    of their error, and the labels."""
    g = _gen(seed, 4)
    N, P, C = c["rows"], c["pool"], c["d_out"]
    t = 1.5 * torch.randn(N, C, generator=g, device=DEV)
    common = 0.5 * torch.randn(N, C, generator=g, device=DEV)
    if c["task"] == "regression":
        y = (t[:, 0] + 0.3 * torch.randn(N, generator=g, device=DEV)).contiguous()
    elif c["task"] == "binary":
        y = (torch.rand(N, generator=g, device=DEV) < torch.sigmoid(2.0 * t[:, 0])).to(torch.int32)
    else:
        e = -torch.log(-torch.log(torch.rand(N, C, generator=g, device=DEV).clamp(1e-9, 1 - 1e-7)))
        y = torch.argmax(2.0 * t + e, 1).to(torch.int32)
    preds = torch.empty(P, N, C, device=DEV)
    for p in range(P):
        own = torch.randn(N, C, generator=g, device=DEV)
        z = t + common + (0.6 + 0.8 * p / max(1, P - 1)) * own
        preds[p] = z if c["task"] == "regression" else torch.sigmoid(z) if C == 1 else torch.softmax(z, 1)
    return preds, y


# -------------------------------------------------------------- prepare, run
def _new_pack(c, h, seed, batch):
    kw = {}
    if c["emb"]:
        values = _emb_values(c, h, seed)
        kw = dict(d_emb=h["d_emb"], freq=np.concatenate([v[0].ravel() for v in values]))
    pack = tp.Pack(c["d_in"], c["d_out"], c["task"], h["depth"], h["width"], h["dropout"], h["lr"], h["wd"], batch,
                   seed=_pack_seed(seed), precision=c["precision"], **kw)
    if c["emb"]:
        for i, v in enumerate(values):
            pack.set_emb(i, *v)
    return pack


def _n_rows(c):
    return max(2 * c["batch"], min(200000, int(2e8 / (4 * c["d_in"]))))


def prepare(case, seed):
    c = case
    if c["kind"] == "select":
        preds, y = _pool(c, seed)
        return dict(case=c, preds=preds, y=y)
    h = _members(c)
    if c["kind"] == "predict":
        X, _ = _table(c, seed, c["rows"])
        pack = _new_pack(c, h, seed, c["batch"])
        g = _gen(seed, 5)
        for i in range(c["m"]):
            pack.restore(i, _trained_run(c, h, i, g))
        return dict(case=c, pack=pack, X=X, out=torch.empty(c["m"], c["rows"], c["d_out"], device=DEV))
    n = _n_rows(c)
    X, y = _table(c, seed, n)
    idx = _batches(c, seed, n)
    pack = _new_pack(c, h, seed, c["batch"])
    if c["muon"]:
        pack.set_muon(h["lr_muon"])
    sizes = [pack.member_size(i) for i in range(c["m"])]
    params = torch.empty(sum(sizes), device=DEV)
    runs, o = [], 0
    for s in sizes:
        runs.append(params[o:o + s])
        o += s
    return dict(case=c, pack=pack, X=X, y=y, idx=list(idx.unbind(0)), step=0, params=params, runs=runs,
                loss=torch.empty(c["steps"], c["m"], device=DEV))


def _slots(sel, m_ens):
    """The selection in m_ens slots, unused ones -1."""
    out = np.full(m_ens, -1, dtype=np.int32)
    out[:len(sel)] = sel
    return out


def run(state):
    c = state["case"]
    if c["kind"] == "select":
        sel, score = tp.select_greedy(state["preds"], state["y"], c["task"], c["score"], m_ens=c["m_ens"])
        return {"selected": _slots(sel, c["m_ens"]), "score": score}
    pack = state["pack"]
    if c["kind"] == "predict":
        return {"pred": pack.predict(state["X"], state["out"])}
    X, y, loss = state["X"], state["y"], state["loss"]
    for k, idx in enumerate(state["idx"]):
        pack.train_step(X, idx, y, state["step"], loss[k])
        state["step"] += 1
    for i, r in enumerate(state["runs"]):
        pack.snapshot(i, r)
    return {"loss": loss, "params": state["params"]}


def tolerance(case):
    """Training: Adam's first steps divide each gradient by its own size, so a
    gradient entry within rounding of zero may step either way, and ReLU
    decisions at near-ties follow.  Initial parameters moved by 6e-8 of
    themselves end 0.003 to 0.009 apart in bf16 (norm-wise; single entries up
    to 0.85 of the largest of rms and value; 1e-4 on the smallest packs) and
    2e-6 to 2.5e-5 apart in fp32 (entries up to 0.011).  Prediction in bf16
    storage is 0.0035 to 0.006 off the exact values."""
    c = case
    if c["kind"] == "select":
        return {"rel": 1e-6}
    if c["kind"] == "predict":
        return {"rel": 0.02, "max": 0.5} if c["precision"] == "bf16" else {"rel": 1e-5, "max": 1e-3}
    if c["precision"] == "bf16":
        return {"rel": 0.01 if c["m"] <= 16 and c["w_hi"] <= 256 else 0.03, "max": 0.99}
    return {"rel": 1e-4, "max": 0.05}


# ---------------------------------------------------------- the same in 64 bits
def _mulhilo(a, b):
    p = a * b
    return (p >> 32) & MASK32, p & MASK32


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors of 32-bit words."""
    k0, k1 = seed & MASK32, seed >> 32
    for _ in range(10):
        ha, la = _mulhilo(c0, 0xD2511F53)
        hb, lb = _mulhilo(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = hb ^ c1 ^ k0, lb, ha ^ c3 ^ k1, la
        k0, k1 = (k0 + 0x9E3779B9) & MASK32, (k1 + 0xBB67AE85) & MASK32
    return torch.stack([c0, c1, c2, c3], -1)


def _words(c0, c1, c2, c3, seed):
    c0, c1 = torch.broadcast_tensors(c0, c1)
    z = torch.zeros_like(c0)
    return _philox(c0, c1, z + c2, z + c3, seed)


def _keep(seed, i, l, step, B, w, p):
    """Dropout keep mask [B, w]: word >= floor(p 2^32)."""
    r = torch.arange(B, device=DEV)[:, None]
    q = torch.arange(w // 4, device=DEV)[None]
    return _words(r, q, step, i << 4 | l, seed).reshape(B, w) >= int(math.floor(float(p) * 4294967296.0))


def _initial(c, h, seed):
    """Initial parameters of every member: U(-1, 1) / sqrt(fan_in) from the
    Philox word of each element, rounded to fp32."""
    got = []
    values = _emb_values(c, h, seed) if c["emb"] else None
    for i in range(c["m"]):
        p = {}
        fan = 1
        for kind, l, _, out, n_in, _ in _blocks(c, h, i)[0]:
            if kind == "e":
                for key, v in zip(("ew", "eb", "ea", "et"), values[i]):
                    p[key] = torch.from_numpy(v).to(DEV).double()
                continue
            if kind == "W":
                fan, e0, n = n_in, 0, out * n_in
            else:
                e0, n = e0 + out * fan, out
            e = torch.arange(e0, e0 + n, device=DEV)
            q = torch.arange((e0 + n + 3) // 4, device=DEV)
            word = _words(q, torch.zeros_like(q), 0, 1 << 28 | i << 4 | l, _pack_seed(seed)).reshape(-1)[e]
            u = ((word >> 8).double() + 0.5) * 2.0 ** -24
            v = ((2 * u - 1) * (1.0 / math.sqrt(fan))).float().double()
            p[kind, l] = v.view(out, n_in) if kind == "W" else v
        got.append(p)
    return got


def _forward(c, h, i, p, x, keep):
    if c["emb"]:
        u = torch.cos(p["ew"] * x[:, :, None] + p["eb"])
        x = (p["ea"] * torch.cat([x[:, :, None], u], 2) + p["et"]).reshape(x.shape[0], -1)
    L = int(h["depth"][i])
    for l in range(L):
        x = torch.relu(x @ p["W", l].T + p["b", l])
        if keep is not None and h["dropout"][i] > 0:
            x = x * keep(l) / (1.0 - float(h["dropout"][i]))
    return x @ p["W", L].T + p["b", L]


def _loss(c, z, y):
    F = torch.nn.functional
    if c["task"] == "multiclass":
        return F.cross_entropy(z, y.long())
    if c["task"] == "binary":
        return F.binary_cross_entropy_with_logits(z[:, 0], y.double())
    return ((z[:, 0] - y.double()) ** 2).mean()


def _muon(g, buf, w, lr, wd):
    buf.mul_(0.95).add_(g, alpha=0.05)
    u = 0.05 * g + 0.95 * buf
    tall = u.shape[0] > u.shape[1]
    x = (u.T if tall else u) / max(float(u.norm()), 1e-7)
    for _ in range(5):
        a = x @ x.T
        x = 3.4445 * x + (-4.7750 * a + 2.0315 * a @ a) @ x
    w.mul_(1 - lr * wd).sub_(x.T if tall else x, alpha=lr * math.sqrt(max(1.0, w.shape[0] / w.shape[1])))


def _exact_train(c, h, seed):
    n = _n_rows(c)
    X, y = _table(c, seed, n)
    idx = _batches(c, seed, n)
    params = _initial(c, h, seed)
    loss = torch.empty(c["steps"], c["m"], device=DEV, dtype=torch.float64)
    out = []
    for i, p in enumerate(params):
        lr, wd, L = float(h["lr"][i]), float(h["wd"][i]), int(h["depth"][i])
        m = {k: torch.zeros_like(v) for k, v in p.items()}
        v2 = {k: torch.zeros_like(v) for k, v in p.items()}
        for t in range(c["steps"]):
            rows = (idx[t, i] if c["stacked"] else idx[t]).long()
            for v in p.values():
                v.requires_grad_(True)
                v.grad = None
            z = _forward(c, h, i, p, X[rows].double(),
                         lambda l: _keep(_pack_seed(seed), i, l, t, len(rows), int(h["width"][i]), h["dropout"][i]))
            e = _loss(c, z, y[rows])
            e.backward()
            loss[t, i] = e.detach()
            with torch.no_grad():
                for k, v in p.items():
                    if c["muon"] and k[0] == "W" and k[1] < L:
                        _muon(v.grad, m[k], v, float(h["lr_muon"][i]), wd)
                        continue
                    v.mul_(1 - lr * wd)
                    m[k].mul_(0.9).add_(v.grad, alpha=0.1)
                    v2[k].mul_(0.999).addcmul_(v.grad, v.grad, value=0.001)
                    v.sub_(lr * (m[k] / (1 - 0.9 ** (t + 1))) / ((v2[k] / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8))
        blocks, size = _blocks(c, h, i)
        flat = torch.zeros(size, device=DEV, dtype=torch.float64)
        for kind, l, off, r, n_in, pad in blocks:
            if kind == "e":
                v = torch.cat([p[k].detach().reshape(-1) for k in ("ew", "eb", "ea", "et")])
            else:
                v = p[kind, l].detach()
            flat[off:off + r * pad].view(r, pad)[:, :n_in] = v.reshape(r, n_in)
        out.append(flat)
        p.clear()
    return {"loss": loss, "params": torch.cat(out)}


def _exact_predict(c, h, seed):
    X, _ = _table(c, seed, c["rows"])
    g = _gen(seed, 5)
    got = []
    for i in range(c["m"]):
        run_, p = _trained_run(c, h, i, g).double(), {}
        for kind, l, off, out, n_in, pad in _blocks(c, h, i)[0]:
            v = run_[off:off + out * pad].view(out, pad)[:, :n_in]
            if kind == "e":
                n, d = c["d_in"], int(h["d_emb"][i])
                k, v = n * (d - 1), v.reshape(-1)
                p["ew"], p["eb"] = v[:k].view(n, d - 1), v[k:2 * k].view(n, d - 1)
                p["ea"], p["et"] = v[2 * k:2 * k + n * d].view(n, d), v[2 * k + n * d:].view(n, d)
            else:
                p[kind, l] = v if kind == "W" else v[:, 0]
        z = torch.cat([_forward(c, h, i, p, x.double(), None) for x in X.split(4096)])
        got.append(torch.softmax(z, 1) if c["task"] == "multiclass" else torch.sigmoid(z) if c["task"] == "binary" else z)
    return {"pred": torch.stack(got)}


def _scores(c, E, y):
    """Score (lower is better) of each ensemble prediction [P, N, d_out]."""
    if c["score"] == "accuracy":
        hit = (E.argmax(-1) if c["task"] == "multiclass" else (E[..., 0] > 0.5).int()) == y
        return -hit.double().mean(-1)
    if c["score"] == "auc":
        s = E[..., 0].float()
        pos = y == 1
        n_pos = int(pos.sum())
        got = []
        for q in s.split(32):
            v = q.sort(-1)[0]
            t = q[:, pos].contiguous()
            mid = 0.5 * (torch.searchsorted(v, t) + 1 + torch.searchsorted(v, t, right=True)).double()
            got.append(-(mid.sum(-1) - 0.5 * n_pos * (n_pos + 1)) / (n_pos * (len(y) - n_pos)))
        return torch.cat(got)
    if c["task"] == "regression":
        v = ((E[..., 0] - y.double()) ** 2).mean(-1)
        return v.sqrt() if c["score"] == "rmse" else v
    e = E.gather(-1, y.long()[None, :, None].expand(E.shape[0], -1, 1))[..., 0] if c["task"] == "multiclass" else \
        torch.where(y == 1, E[..., 0], 1 - E[..., 0])
    return -e.clamp(1e-7, 1 - 1e-7).log().mean(-1)


def _exact_select(c, seed):
    preds, y = _pool(c, seed)
    P, sel, best = c["pool"], [], math.inf
    total = torch.zeros(preds.shape[1:], device=DEV, dtype=torch.float64)
    while len(sel) < c["m_ens"]:
        s = torch.cat([_scores(c, (total + q.double()) / (len(sel) + 1), y) for q in preds.split(max(1, 32 // c["d_out"]))])
        if sel:
            s[sel] = math.inf
        k = int(torch.argmin(s))
        if len(sel) == P or not float(s[k]) < best:
            break
        best = float(s[k])
        sel.append(k)
        total += preds[k]
    return {"selected": _slots(sel, c["m_ens"]), "score": best}


def exact(case, seed):
    c = case
    if c["kind"] == "select":
        return _exact_select(c, seed)
    h = _members(c)
    return _exact_predict(c, h, seed) if c["kind"] == "predict" else _exact_train(c, h, seed)
