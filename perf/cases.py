"""The workloads this library's speed is measured on, through its public Python entry points.

Every case is a kind of call with a model shape:

  period    what a decode loop does between two evictions: the period's K/V rows are appended (by the
            model; here a copy), its queries go to the beacons in one call, the cache is compressed and
            the beacon state is read back for a checkpoint
  update    one batched beacon update with its assignments
  steps     one update call per generated token, for ``n_steps`` tokens
  seq       the same tokens handed over in one call
  seed      prefill: the beacons seeded from the prompt's queries
  ragged    period without the update, every sequence with a cache length and positions of its own
  static    the context-free compress of an engine that lets nobody allocate device memory
  cfps      period with Continual FPS buffers instead of centroids

A state holds ``POOL`` periods' worth of inputs, which successive passes take in turn, so that no pass sees
the queries or the appended rows of the pass before it.  Shapes are those of workloads.py, or generic.
"""
from __future__ import annotations

import math

import torch

from paper_2609_04971_gb300 import bkv

POOL = 4
DEV = "cuda"


def _case(name, kind, *, layers, batch, q_heads, kv_heads, d, L=0, budget=0, W=8, nb=8, n_new=0, n_steps=0, n_init=0,
          theta=1e6, prefix=0, scores=False, mean=False, causal=False):
    c = dict(kind=kind, layers=layers, batch=batch, q_heads=q_heads, kv_heads=kv_heads, d=d, L=L, budget=budget, W=W,
             nb=nb, n_new=n_new, n_steps=n_steps, n_init=n_init, theta=theta, prefix=prefix, scores=scores, mean=mean,
             causal=causal)
    if name:
        c["name"] = name
    return c


def listed():
    qwen4 = dict(layers=36, batch=16, q_heads=32, kv_heads=8, d=128)
    return [
        # one layer of a test-size model: launches and host work are all there is
        _case("tiny_period", "period", layers=1, batch=1, q_heads=4, kv_heads=2, d=64, L=1088, budget=512, nb=4,
              n_new=64, theta=1e4, scores=True),
        # one user's sequence on a 4B model
        _case("one_sequence_period", "period", layers=36, batch=1, q_heads=32, kv_heads=8, d=128, L=4224, budget=4096,
              n_new=128, scores=True),
        # the headline step: a batch of 16 long reasoning traces on a 4B model
        _case("qwen3_4b_period", "period", **qwen4, L=4224, budget=4096, n_new=128),
        # five query heads per KV head, 8K caches
        _case("qwen3_14b_period", "period", layers=40, batch=8, q_heads=40, kv_heads=8, d=128, L=8320, budget=8192,
              nb=16, n_new=128),
        # a server's batched update: 32 sequences on an 8B model, 16 beacons
        _case("llama_8b_update", "update", layers=32, batch=32, q_heads=32, kv_heads=8, d=128, nb=16, n_new=128,
              theta=5e5),
        # a decode loop that calls the library with every token
        _case("decode_steps", "steps", **qwen4, nb=16, n_steps=32),
        # a decode loop that hands a period's tokens over at once
        _case("decode_seq", "seq", **qwen4, nb=16, n_steps=128),
        # prefill of a batch of short prompts
        _case("prefill_seed", "seed", **qwen4, n_init=64),
        # batched serving: 16 sequences, each with its own length, the shortest of them not yet full
        _case("ragged_batch", "ragged", layers=12, batch=16, q_heads=32, kv_heads=8, d=128, L=4352, budget=4001,
              scores=True),
        # one long document: window of 16 (72 scoring queries), mean form, causal inside the window
        _case("long_cache_mean_causal", "period", layers=36, batch=1, q_heads=32, kv_heads=8, d=128, L=32700,
              budget=28613, W=16, n_new=37, prefix=4, scores=True, mean=True, causal=True),
        # an engine compressing four layers at a time inside its own memory
        _case("static_four_layers", "static", layers=4, batch=16, q_heads=32, kv_heads=8, d=128, L=4224, budget=4096,
              scores=True),
        # the paper's own beacon maintenance, a third of the model
        _case("continual_fps_period", "cfps", layers=12, batch=16, q_heads=32, kv_heads=8, d=128, L=4224, budget=4096,
              n_new=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["period", "period", "period", "update", "steps", "seq", "seed", "ragged", "static", "cfps"])
    d = rng.choice([64, 128, 128])
    kv = rng.choice([1, 2, 4, 8, 8])
    G = rng.choice([1, 2, 4, 4, 5, 7, 8])
    W = rng.choice([4, 8, 8, 16, 11])
    nb = rng.choice([4, 8, 8, 13, 16, 32])
    if kind == "cfps":  # b_max <= 32 rows per head, at most 128 scoring queries per group
        G, nb = rng.choice([1, 2, 4]), rng.choice([4, 8, 13])
        W = rng.choice([4, 8, 11, 16])
    while G * (W + (nb if kind == "cfps" else 0)) + nb > 128:
        W = max(1, W // 2)
    layers, batch = _log(rng, 1, 40), _log(rng, 1, 32)
    L = 600 if kind in ("update", "steps", "seq", "seed") else _log(rng, 600, 32768)
    budget = L - max(1, int(L * rng.uniform(0.01, 0.4)))
    most = 2 << 30  # bytes of K and V
    if kind == "static":
        L = min(L, 9000)
        layers, batch = rng.choice([1, 2, 4]), rng.choice([1, 2, 8, 16])
        budget = min(budget, L - 7)
        most = (14 << 20) * 4 * d // (4 + 256 * d // 600)  # the scratch array holds 16 MiB
    while layers * batch * kv * L * d * 4 > most and layers * batch * kv > 1:
        if layers > 1:
            layers = max(1, layers * 3 // 4)
        elif batch > 1:
            batch = max(1, batch * 3 // 4)
        else:
            kv = max(1, kv // 2)
    return _case(None, kind, layers=layers, batch=batch, q_heads=G * kv, kv_heads=kv, d=d, L=L, budget=budget, W=W,
                 nb=nb, n_new=_log(rng, 1, 256), n_steps=_log(rng, 4, 128), n_init=max(-(-nb // G), _log(rng, 16, 512)),
                 theta=rng.choice([1e4, 5e5, 1e6]), prefix=rng.choice([0, 0, 4]), scores=rng.random() < 0.7,
                 mean=rng.random() < 0.2, causal=rng.random() < 0.2)


# ------------------------------------------------------------------ inputs
def _unit(x):
    return x / x.norm(dim=-1, keepdim=True).clamp_min(1e-30)


def _gen(seed, tag):
    return torch.Generator(device=DEV).manual_seed((seed * 1000003 + tag) & 0x7FFFFFFFFFFFFFFF)


def _queries(c, centres, n, g):
    """Pre-RoPE queries [layers, batch, q_heads, n, d]: 70 % around the instance's centres, the rest isotropic."""
    G, d = c["q_heads"] // c["kv_heads"], c["d"]
    out = torch.empty(c["layers"], c["batch"], c["q_heads"], n, d, dtype=torch.bfloat16, device=DEV)
    for l in range(c["layers"]):
        cen = centres[l].repeat_interleave(G, dim=1)
        k = torch.randint(0, cen.shape[2], (c["batch"], c["q_heads"], n), generator=g, device=DEV)
        k[torch.rand(k.shape, generator=g, device=DEV) < 0.3] = cen.shape[2] - 1
        noise = torch.full((cen.shape[2],), 0.15, device=DEV)
        noise[-1] = 1.0  # the last "centre" is zero: isotropic queries
        pick = torch.gather(cen, 2, k.unsqueeze(-1).expand(*k.shape, d))
        xi = torch.randn(*k.shape, d, generator=g, device=DEV)
        out[l] = (pick * math.sqrt(d) + noise[k].unsqueeze(-1) * xi).to(torch.bfloat16)
    return out


def _cache_rows(c, n, g, mu=None):
    out = torch.empty(c["layers"], c["batch"], c["kv_heads"], n, c["d"], dtype=torch.bfloat16, device=DEV)
    for l in range(c["layers"]):
        x = torch.randn(out.shape[1:], generator=g, device=DEV)
        out[l] = (x if mu is None else x.add_(mu[l])).to(torch.bfloat16)
    return out


def _inputs(c, seed):
    """Everything a pass reads, from the seed alone, in torch (no code of the library)."""
    kind, d, nb, W = c["kind"], c["d"], c["nb"], c["W"]
    head = (c["layers"], c["batch"], c["kv_heads"])
    g = _gen(seed, 1)
    centres = _unit(torch.randn(*head, max(4, nb) + 1, d, generator=g, device=DEV))
    centres[:, :, :, -1] = 0.0
    x = {}
    if kind == "seed":
        x["q_init"] = [_queries(c, centres, c["n_init"], g) for _ in range(POOL)]
        return x
    if kind == "cfps":  # a buffer between two compressions holds n_beacons to n_beacons + window - 1 queries
        x["buffers"] = _queries(c, centres, nb + W, g)
        x["sizes"] = torch.randint(nb, nb + W, (c["layers"], c["batch"], c["q_heads"]), generator=g, device=DEV,
                                   dtype=torch.int32)
    else:  # centroids in mid-decode: sums of some hundred queries near the centres
        x["counts"] = torch.randint(16, 400, (*head, nb), generator=g, device=DEV, dtype=torch.int64)
        mean = math.sqrt(d) * centres[:, :, :, :nb] + 0.1 * torch.randn(*head, nb, d, generator=g, device=DEV)
        x["sums"] = torch.round(mean.double() * x["counts"].unsqueeze(-1) * 65536.0) / 65536.0
        x["cent"] = (x["sums"] / x["counts"].unsqueeze(-1)).float()
    if kind in ("steps", "seq"):
        q = [_queries(c, centres, c["n_steps"], g) for _ in range(POOL)]
        x["q_steps"] = [t.permute(3, 0, 1, 2, 4).contiguous() for t in q]
        return x
    if kind in ("period", "update", "cfps"):
        x["q_new"] = [_queries(c, centres, c["n_new"], g) for _ in range(POOL)]
    if kind == "update":
        return x
    L, budget = c["L"], c["budget"]
    mu = 0.5 * torch.randn(c["layers"], 1, c["kv_heads"], 1, d, generator=g, device=DEV)
    x["K"], x["V"] = _cache_rows(c, L, g, mu), _cache_rows(c, L, g)
    x["q_recent"] = [_queries(c, centres, W, g) for _ in range(POOL)]
    x["K_new"] = [_cache_rows(c, L - budget, g, mu) for _ in range(POOL)]
    x["V_new"] = [_cache_rows(c, L - budget, g) for _ in range(POOL)]
    x["t_pos"] = 2 * L + 17  # earlier evictions: positions run ahead of the cache length
    x["recent_pos"] = [x["t_pos"] - W + 1 + w for w in range(W)]
    if kind == "ragged":  # one length per sequence; about one in eight has not reached the budget
        hc = torch.Generator().manual_seed(seed + 5)
        ln = torch.randint(budget + 1, L + 1, (c["batch"],), generator=hc)
        short = torch.rand(c["batch"], generator=hc) < 0.125
        ln = torch.where(short, (budget * 0.9 * torch.ones(c["batch"])).long(), ln)
        ln[0] = L
        x["lens"] = ln.tolist()
        x["Ls"] = ln.to(DEV, torch.int32).view(1, -1, 1).expand(*head).contiguous()
        x["t_row"] = [2 * int(v) + 3 for v in ln]
        x["recent_row"] = [[t - W + 1 + w for w in range(W)] for t in x["t_row"]]
    return x


def prepare(case, seed):
    c = case
    x = _inputs(c, seed)
    x.update(case=c, i=0)
    shape = (c["layers"], c["batch"], c["kv_heads"])
    if "L" in c and "K" in x:
        x["kept"] = torch.zeros(*shape, c["budget"], dtype=torch.int32, device=DEV)
        x["scores"] = torch.zeros(*shape, c["L"], device=DEV) if c["scores"] else None
    flags = (bkv.BKV_F_MEAN_AGG if c["mean"] else 0) | (bkv.BKV_F_CAUSAL_WINDOW if c["causal"] else 0)
    if c["kind"] == "static":
        x["cfg"] = bkv.BkvConfig(c["layers"], c["batch"], c["q_heads"], c["kv_heads"], c["d"], c["nb"], c["W"],
                                 c["prefix"], c["L"], c["theta"], flags)
        x["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        return x
    bk = x["bk"] = bkv.BeaconKV(
        n_layers=c["layers"], batch=c["batch"], n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"], head_dim=c["d"],
        n_beacons=c["nb"], window=c["W"], capacity=c["L"] or 4224, rope_theta=c["theta"], n_prefix=c["prefix"],
        mean_agg=c["mean"], causal_window=c["causal"], continual_fps=c["kind"] == "cfps")
    if c["kind"] == "cfps":
        bk.set_cfps_state(x["buffers"], x["sizes"])
    elif c["kind"] != "seed":
        bk.set_state(x["cent"], x["sums"], x["counts"])
    heads = (c["layers"], c["batch"], c["q_heads"])
    if c["kind"] in ("period", "update"):
        x["assign"] = torch.zeros(*heads, c["n_new"], dtype=torch.int32, device=DEV)
    elif c["kind"] in ("steps", "seq"):
        x["assign"] = torch.zeros(c["n_steps"], *heads, dtype=torch.int32, device=DEV)
    return x


def _append(x, p):
    """The model's part of a period: its K/V rows behind the kept ones."""
    b = x["case"]["budget"]
    x["K"][:, :, :, b:].copy_(x["K_new"][p])
    x["V"][:, :, :, b:].copy_(x["V_new"][p])


def run(state):
    x, c = state, state["case"]
    kind, p = c["kind"], x["i"] % POOL
    x["i"] += 1
    if kind == "seed":
        x["bk"].init_beacons(x["q_init"][p])
        return list(x["bk"].state())
    if kind == "update":
        x["bk"].update(x["q_new"][p], x["assign"])
        return [x["assign"], *x["bk"].state()]
    if kind == "seq":
        x["bk"].update_seq(x["q_steps"][p], x["assign"])
        return [x["assign"], *x["bk"].state()]
    if kind == "steps":
        for t in range(c["n_steps"]):
            x["bk"].update(x["q_steps"][p][t].unsqueeze(3), x["assign"][t])
        return [x["assign"], *x["bk"].state()]
    _append(x, p)
    out = [x["kept"], x["K"], x["V"]] + ([x["scores"]] if c["scores"] else [])
    if kind == "ragged":
        x["bk"].compress_ragged(x["K"], x["V"], L=x["Ls"], budget=c["budget"], t_pos=x["t_row"],
                                q_recent=x["q_recent"][p], recent_pos=x["recent_row"], kept_out=x["kept"],
                                scores_out=x["scores"])
        return out
    if kind == "static":
        bkv.bkv_compress_static(x["cfg"], x["cent"], x["counts"], x["K"], x["V"], c["L"], c["budget"], x["t_pos"],
                                x["q_recent"][p], x["recent_pos"], x["kept"], x["scores"], x["status"])
        return out + [x["status"]]
    bk = x["bk"]
    bk.update(x["q_new"][p], x.get("assign"))
    bk.compress(x["K"], x["V"], L=c["L"], budget=c["budget"], t_pos=x["t_pos"], q_recent=x["q_recent"][p],
                recent_pos=x["recent_pos"], kept_out=x["kept"], scores_out=x["scores"])
    return out + (list(bk.cfps_state()) if kind == "cfps" else [x["assign"], *bk.state()])


# ------------------------------------------------------------------ work
def work(case):
    c, kind, d, nb, W = case, case["kind"], case["d"], case["nb"], case["W"]
    G = c["q_heads"] // c["kv_heads"]
    inst = c["layers"] * c["batch"] * c["kv_heads"]
    state = nb * (12 * d + 8)  # centroids, sums and counts of an instance
    by = fl = 0
    if kind == "seed":
        nq = G * c["n_init"]
        by, fl = nq * d * 2 + 2 * state, 2 * nq * d * nb
    elif kind in ("update", "steps", "seq", "period"):
        nq = G * (c["n_steps"] if kind in ("steps", "seq") else c["n_new"])
        by, fl = nq * (d * 2 + 4) + 3 * state, 2 * nq * nb * d
    elif kind == "cfps":
        nq, buf = G * c["n_new"], G * ((nb + W) * d * 2 + 4)
        by, fl = nq * d * 2 + 3 * buf, 2 * nq * (nb + W) * d
    if kind in ("period", "ragged", "static", "cfps"):
        L, B = c["L"], c["budget"]
        M = G * W + (G * nb if kind == "cfps" else nb)
        by += L * d * 2 + B * d * 8 + G * W * d * 2 + B * 4 + (L * 4 if c["scores"] else 0) + (L - B) * d * 8
        fl += 2 * M * L * d
    return {"bytes": float(by * inst), "flops": float(fl * inst)}


# ------------------------------------------------------------------ the same in 64 bits
def _update64(q, cent, sums, counts):
    """One call's update: q [I, n, d] against the centroids at its start (all fp64); returns the assignment."""
    a = torch.bmm(q, _unit(cent).transpose(1, 2)).argmax(-1)
    hot = torch.nn.functional.one_hot(a, cent.shape[1]).double()
    sums += torch.bmm(hot.transpose(1, 2), q)
    counts += hot.sum(1).long()
    cent.copy_((sums / counts.unsqueeze(-1)).float().double())
    return a


def _rotate(x, pos, theta):
    """x [..., d] (fp64) turned to the positions pos [...] (rotate-half pairs), rounded as the scoring takes it."""
    h = x.shape[-1] // 2
    inv = theta ** (-torch.arange(h, dtype=torch.float64, device=DEV) / h)
    ang = pos.double().unsqueeze(-1) * inv
    a, b = x[..., :h], x[..., h:]
    y = torch.cat([a * ang.cos() - b * ang.sin(), b * ang.cos() + a * ang.sin()], -1)
    return y.float().to(torch.bfloat16).double()


def _scores64(c, x, cent, K):
    """Scores [layers, batch, kv_heads, L] of the pass's cache K (rows past an instance's length: 0)."""
    G, W, d, nb = c["q_heads"] // c["kv_heads"], c["W"], c["d"], c["nb"]
    out = torch.zeros(K.shape[:4], dtype=torch.float64, device=DEV)
    j = torch.arange(c["L"], device=DEV)
    for l in range(c["layers"]):
        for b in range(c["batch"]):
            L = x["lens"][b] if c["kind"] == "ragged" else c["L"]
            if L <= c["budget"]:
                continue
            t = x["t_row"][b] if c["kind"] == "ragged" else x["t_pos"]
            rp = torch.tensor(x["recent_row"][b] if c["kind"] == "ragged" else x["recent_pos"], device=DEV)
            qr = x["q_recent"][0][l, b].double().view(c["kv_heads"], G * W, d)
            qr = _rotate(qr, rp.repeat(G).expand(c["kv_heads"], -1), c["theta"])
            bc = _rotate(cent[l, b], torch.full((c["kv_heads"], nb), t, device=DEV), c["theta"])
            s = torch.bmm(torch.cat([qr, bc], 1), K[l, b, :, :L].double().transpose(1, 2)) / math.sqrt(d)
            if c["causal"]:
                late = (j[:L] >= L - W) & ((t - (L - 1 - j[:L])) > rp.repeat(G).unsqueeze(-1))
                s[:, :G * W] = s[:, :G * W].masked_fill(late, -math.inf)
            w = s.softmax(-1)
            out[l, b, :, :L] = w.mean(1) if c["mean"] else w.amax(1)
    return out


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "cfps":
        return None  # buffers hold selected queries: no computed numbers
    x = _inputs(c, seed)
    I, G, d, nb = c["layers"] * c["batch"] * c["kv_heads"], c["q_heads"] // c["kv_heads"], c["d"], c["nb"]
    head = (c["layers"], c["batch"], c["kv_heads"])
    if kind == "seed":
        q = x["q_init"][0].view(I, -1, d)
        cent = torch.empty(I, nb, d, dtype=torch.float64, device=DEV)
        for i0 in range(0, I, 512):
            v = q[i0:i0 + 512].double()
            u = _unit(v)
            first = torch.bmm(u, u.sum(1).unsqueeze(-1)).squeeze(-1)
            far = torch.full_like(first, -math.inf)
            for k in range(nb):
                r = (first if k == 0 else far).argmin(-1)
                pick = r.view(-1, 1, 1).expand(-1, 1, d)
                cent[i0:i0 + 512, k] = torch.gather(v, 1, pick).squeeze(1)
                far = torch.maximum(far, torch.bmm(u, torch.gather(u, 1, pick).transpose(1, 2)).squeeze(-1))
                far.scatter_(1, r.unsqueeze(-1), math.inf)
        return [cent, cent, torch.ones(I, nb, dtype=torch.int64, device=DEV)]
    cent, sums = x["cent"].double().view(I, nb, d), x["sums"].clone().view(I, nb, d)
    counts = x["counts"].clone().view(I, nb)
    assign = None
    if kind in ("steps", "seq"):
        for t in range(c["n_steps"]):
            _update64(x["q_steps"][0][t].view(I, G, d).double(), cent, sums, counts)
    elif kind in ("update", "period"):
        q = x["q_new"][0].view(I, G * c["n_new"], d)
        for i0 in range(0, I, 512):
            e = slice(i0, i0 + 512)
            _update64(q[e].double(), cent[e], sums[e], counts[e])
    state = [cent, sums, counts]
    if kind in ("update", "steps", "seq"):
        return [assign, *state]
    out = [None, None, None]
    if c["scores"]:
        x["K"][:, :, :, c["budget"]:] = x["K_new"][0]
        out.append(_scores64(c, x, cent.view(*head, nb, d), x["K"]))
    return out + ([None, *state] if kind == "period" else [None] if kind == "static" else [])
