"""The calls whose time is measured, over the range in which a routing service makes them.

A case is a dict of plain values.  `kind` says which call a pass makes:

  route       one routing batch (ls_route_batch, or its guarded form), issued
              directly or as a replay of a captured graph
  sequential  a burst of requests routed one after the other, each decision
              committed before the next (ls_route_sequential)
  snapshot    a full cluster snapshot (every instance's cached-block keys) and
              the first routing batch on it
  train       one minibatch step of the predictor
  round       the online-learning round: log new records, admit evicted ones to
              the replay pool, refresh the feature bounds, train, publish

Prompts share prefixes through templates drawn from a Zipf law, and an
instance caches the first blocks of the templates it has served, so the hit
length of a request on an instance is known from the draws alone; `exact`
uses that and evaluates the predictor in 64 bits without the library.
"""
import math

import torch

from paper_2606_00946_gb300 import harness as H
from paper_2606_00946_gb300 import lodestar as L

BLOCK = 16
PAIR = 6
VOCAB = 32000
SPEEDS = (1.0, 1.7, 3.1)
RHO = (0.1, 0.3, 0.5, 0.7)      # share of a prompt that is its template's prefix
DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _route(name, hidden, d_inst, d_req, n_inst, n_req, len_lo, len_hi, templates, cache_blocks, dtype="bf16",
           guarded=False, graph=False, scores=False, n_types=1, kind="route"):
    c = dict(kind=kind, hidden=hidden, d_inst=d_inst, d_req=d_req, n_inst=n_inst, n_req=n_req, len_lo=len_lo,
             len_hi=len_hi, templates=templates, cache_blocks=cache_blocks, dtype=dtype, guarded=guarded,
             graph=graph, scores=scores, n_types=n_types)
    if name:
        c["name"] = name
    return c


def _train(name, hidden, d_inst, d_req, batch, ring, len_lo, len_hi, dtype="bf16", opt="adam", lr=3e-4,
           dropout=0.0, graph=False, n_types=1):
    c = dict(kind="train", hidden=hidden, d_inst=d_inst, d_req=d_req, batch=batch, ring=ring, len_lo=len_lo,
             len_hi=len_hi, dtype=dtype, opt=opt, lr=lr, dropout=dropout, graph=graph, n_types=n_types)
    if name:
        c["name"] = name
    return c


def _round(name, hidden, d_inst, d_req, pool, new, batch, steps, len_lo, len_hi, dropout):
    c = dict(kind="round", hidden=hidden, d_inst=d_inst, d_req=d_req, pool=pool, new=new, batch=batch, steps=steps,
             len_lo=len_lo, len_hi=len_hi, dtype="bf16", dropout=dropout, n_types=1)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a gateway that asks for one decision at a time over 16 instances, with the paper's predictor (three hidden
        # layers of 128), the route captured once and replayed per request: latency
        _route("route_one", "128-128-128", 34, 24, 16, 1, 64, 4096, 256, 16384, graph=True, scores=True),
        # a small deployment on an fp32 predictor: 8 instances, 64 short requests, issued call by call
        _route("route_tiny_f32", "64-64", 10, 0, 8, 64, 32, 640, 4, 2048, dtype="f32", scores=True),
        # a burst of requests over an instance count that divides nothing, with Algorithm 4's guards (cold start,
        # feature bounds, K-filter) and the pre-computed fallback heuristic
        _route("route_guarded", "128-128-128", 34, 24, 24, 777, 64, 4096, 256, 16384, guarded=True, scores=True),
        # the homogeneous cluster: 32 instances, batches of 4096
        _route("route_homogeneous", "256-256", 34, 24, 32, 4096, 64, 4096, 256, 16384),
        # long contexts on three GPU types: 64 instances, batches of 8192, a deeper predictor
        _route("route_heterogeneous", "256-256-256", 66, 56, 64, 8192, 8192, 32768, 256, 65536, n_types=3),
        # the largest cluster one GPU serves: 256 instances with a million cached blocks each, batches of 16384
        _route("route_large", "512-512", 66, 56, 256, 16384, 128, 16384, 4096, 1 << 20, n_types=3),
        # a burst routed request by request at the paper's operating point: every decision is committed (queue and
        # cache of the chosen instance) before the next request is scored
        _route("sequential_paper", "128-128-128", 34, 24, 16, 64, 64, 4096, 256, 16384, kind="sequential",
               scores=True),
        # a gateway that has lost its tracker state takes a full snapshot of 32 instances' caches and routes on it
        _route("snapshot_rebuild", "256-256", 34, 24, 32, 256, 64, 4096, 256, 16384, kind="snapshot"),
        # the online-training configuration: Adam, batch 4096 over a million logged records
        _train("train_online", "256-256-256", 66, 56, 4096, 1 << 20, 8192, 32768, n_types=3),
        # the step that runs beside the largest cluster's route: hidden layers of 512
        _train("train_wide", "512-512", 66, 56, 4096, 65536, 128, 16384, n_types=3),
        # the small fp32 predictor's SGD step over all its 256 records
        _train("train_tiny_f32", "64-64", 10, 0, 256, 256, 32, 640, dtype="f32", opt="sgd", lr=1e-3),
        # the paper's online round: 1000 new samples, FIFO and replay pools of 5000, dropout 0.1, one pass of three
        # minibatches over both pools, then the publish
        _round("round_paper", "128-128-128", 34, 24, 5000, 1000, 4096, 3, 64, 4096, 0.1),
    ]


BF16_HIDDEN = ("64", "128-64", "128-128-128", "192-192", "256-256", "256-256-256", "384-384", "512-512")
F32_HIDDEN = ("64-64", "100-50", "128-128-128", "256-256")
DIMS = ((10, 0), (34, 24), (66, 56), (23, 9))  # (instance state, request extras): widths 16, 64, 128, 38


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_shape(rng, dtype):
    hidden = rng.choice(F32_HIDDEN if dtype == "f32" else BF16_HIDDEN)
    d_inst, d_req = rng.choice(DIMS)
    return hidden, d_inst, d_req


def draw(rng):
    u = rng.random()
    dtype = "f32" if rng.random() < 0.25 else "bf16"
    hidden, d_inst, d_req = _draw_shape(rng, dtype)
    if u < 0.5:  # route
        while True:
            n_inst = _log_int(rng, 1, 256)
            n_req = _log_int(rng, 1, 16384)
            len_hi = _log_int(rng, 256, 16384)
            w = [int(x) for x in hidden.split("-")]
            per_row = sum(a * b for a, b in zip([PAIR + d_inst + d_req] + w, w + [1]))
            # no dearer than the largest listed case; fp32 runs on CUDA cores
            cap = 2e9 if dtype == "f32" else 3e11
            if n_inst * n_req * per_row <= cap and n_req * len_hi <= 1.5e8:
                break
        small = n_req <= 512
        return _route(None, hidden, d_inst, d_req, n_inst, n_req, max(1, len_hi // 64), len_hi,
                      rng.choice((16, 256, 1024)), _log_int(rng, 1024, 65536), dtype=dtype,
                      guarded=rng.random() < 0.25, graph=small and rng.random() < 0.5, scores=rng.random() < 0.5,
                      n_types=rng.choice((1, 3)))
    if u < 0.6:  # sequential
        hidden = rng.choice(("64-64", "128-128-128", "256-256"))
        return _route(None, hidden, 34, 24, _log_int(rng, 2, 32), _log_int(rng, 4, 48), 64, _log_int(rng, 256, 8192),
                      256, _log_int(rng, 1024, 16384), kind="sequential", scores=True)
    if u < 0.7:  # snapshot
        return _route(None, rng.choice(("128-128-128", "256-256")), 34, 24, _log_int(rng, 8, 128),
                      _log_int(rng, 16, 512), 64, 4096, 256, _log_int(rng, 1024, 32768), kind="snapshot")
    if u < 0.95:  # train
        f32 = dtype == "f32"
        n_hidden = hidden.count("-")
        fast = not f32 and max(int(x) for x in hidden.split("-")) <= 256
        return _train(None, hidden, d_inst, d_req, _log_int(rng, 64, 1024 if f32 else 8192), _log_int(rng, 8192, 1 << 18),
                      64, 8192, dtype=dtype, opt=rng.choice(("adam", "adam", "sgd")), lr=rng.choice((1e-4, 3e-4, 1e-3)),
                      dropout=0.1 if fast and n_hidden and rng.random() < 0.3 else 0.0, graph=rng.random() < 0.3)
    return _round(None, rng.choice(("128-128-128", "256-256")), 34, 24, _log_int(rng, 1000, 5000),
                  _log_int(rng, 100, 1000), _log_int(rng, 512, 4096), rng.choice((1, 2, 3)), 64, 4096,
                  rng.choice((0.0, 0.1)))


# ---------------------------------------------------------------------------
# inputs (plain torch, made on the GPU from the seed)
# ---------------------------------------------------------------------------

def _widths(case):
    return [PAIR + case["d_inst"] + case["d_req"]] + [int(x) for x in case["hidden"].split("-")] + [1]


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFF)
    return g


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo


def _ints(g, lo, hi, *shape):
    return torch.randint(lo, hi, shape, generator=g, device=DEV)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _instance_rows(g, case, n):
    """Instance states: queued, running, inflight prefill and decode tokens, KV use, free blocks, GPU type (one-hot)
    and speed, then other metrics."""
    st = torch.zeros(n, case["d_inst"], device=DEV, dtype=torch.float64)
    run = _ints(g, 0, 65, n).double()
    util = torch.rand(2, n, generator=g, device=DEV, dtype=torch.float64).mean(0)
    st[:, 0] = torch.poisson(torch.full((n,), 4.0, device=DEV), generator=g).double()
    st[:, 1] = run
    st[:, 2] = run * _uniform(g, 0, 4096, n)
    st[:, 3] = run * _uniform(g, 0, 1024, n)
    st[:, 4] = util
    st[:, 5] = torch.floor((1 - util) * case.get("cache_blocks", 16384))
    typ = torch.arange(n, device=DEV) % case["n_types"]
    st[torch.arange(n, device=DEV), 6 + typ] = 1.0
    st[:, 9] = torch.tensor(SPEEDS, device=DEV, dtype=torch.float64)[typ]
    if case["d_inst"] > 10:
        st[:, 10:] = _normal(g, n, case["d_inst"] - 10).double()
    return st.float()


def _records(g, case, n):
    """Logged records: raw feature rows of routed pairs and the observed TTFT (seconds)."""
    length = _ints(g, case["len_lo"], case["len_hi"] + 1, n).double()
    nb = torch.floor(length / BLOCK)
    h = torch.floor(_uniform(g, 0, 1, n) * (nb + 1))
    x = torch.zeros(n, PAIR + case["d_inst"] + case["d_req"], device=DEV)
    for k, v in enumerate((length, h, BLOCK * h, BLOCK * h / length, length - BLOCK * h,
                           torch.ceil(length / BLOCK) - h)):
        x[:, k] = v.float()
    x[:, PAIR:PAIR + case["d_inst"]] = _instance_rows(g, case, n)
    if case["d_req"]:
        x[:, PAIR + case["d_inst"]:] = _normal(g, n, case["d_req"])
    y = (0.02 + 5e-5 * length + 1e-9 * length ** 2 + 0.03 * x[:, PAIR].double() - 4e-5 * BLOCK * h
         + 0.05 * torch.exp(0.3 * _normal(g, n).double()))
    return x, y.clamp(min=1e-3).float()


def _normaliser(seed, case):
    x = _records(_gen(seed, 7), case, 16384)[0].double()
    return x.mean(0).float(), x.std(0, unbiased=False).float()


def _params(seed, case):
    """Weights as a trained predictor has them: Xavier-uniform scale, small biases."""
    g, w, parts = _gen(seed, 3), _widths(case), []
    for a, b in zip(w[:-1], w[1:]):
        s = math.sqrt(6.0 / (a + b))
        parts += [_uniform(g, -s, s, b * a).float(), _uniform(g, -0.05, 0.05, b).float()]
    return torch.cat(parts)


def _layers(case, flat):
    """[(W, b)] of the flat parameter vector, in 64 bits."""
    out, o, w = [], 0, _widths(case)
    flat = flat.double()
    for a, b in zip(w[:-1], w[1:]):
        out.append((flat[o:o + a * b].view(b, a), flat[o + a * b:o + a * b + b]))
        o += a * b + b
    return out


def _zipf(n):
    p = torch.arange(1, n + 1, device=DEV, dtype=torch.float64) ** -1.1
    return p / p.sum()


def _batch(case, seed):
    """A routing batch and the caches it meets.  `cached[i, t]`: leading blocks of template t that instance i holds;
    `blocks[r]`: full blocks of prompt r inside its template's prefix."""
    g = _gen(seed, 1)
    n_req, n_inst, n_t, lo, hi = case["n_req"], case["n_inst"], case["templates"], case["len_lo"], case["len_hi"]
    n_tb = max(1, hi // BLOCK)
    templates = _ints(g, 0, VOCAB, n_t, hi).int()
    length = _ints(g, lo, hi + 1, n_req)
    off = torch.zeros(n_req + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(length, 0)
    t = torch.multinomial(_zipf(n_t), n_req, replacement=True, generator=g)
    rho = torch.tensor(RHO, device=DEV, dtype=torch.float64)[_ints(g, 0, len(RHO), n_req)]
    shared = torch.floor(rho * length).long()
    tok = torch.randint(0, VOCAB, (int(off[-1]),), generator=g, device=DEV, dtype=torch.int32)
    for r0 in range(0, n_req, 1024):  # the template's prefix, then a token that differs from the template's
        r1 = min(n_req, r0 + 1024)
        seg = tok[int(off[r0]):int(off[r1])]
        req = torch.repeat_interleave(torch.arange(r0, r1, device=DEV), length[r0:r1])
        pos = torch.arange(seg.numel(), device=DEV) - (off[req] - off[r0])
        of_t = templates[t[req], pos]
        first = (of_t + 1 + seg % (VOCAB - 1)) % VOCAB
        seg.copy_(torch.where(pos < shared[req], of_t, torch.where(pos == shared[req], first, seg)))
    # half of an instance's cache is template prefixes (templates in a Zipf-weighted random order, the first k blocks
    # of each until the half is full), the rest blocks that no request shares
    half = case["cache_blocks"] // 2
    order = torch.argsort(torch.log(_zipf(n_t))[None] - torch.log(-torch.log(_uniform(g, 1e-12, 1, n_inst, n_t))), 1,
                          descending=True)
    k = _ints(g, 1, n_tb + 1, n_inst, n_t)
    before = torch.cumsum(k, 1) - k
    k = torch.minimum(k, (half - before).clamp(min=0))
    cached = torch.zeros_like(k).scatter_(1, order, k)
    return dict(tok=tok, off=off, length=length, t=t, blocks=shared // BLOCK, cached=cached, templates=templates,
                req=_normal(g, n_req, case["d_req"]) if case["d_req"] else torch.zeros(n_req, 0, device=DEV),
                inst=_instance_rows(_gen(seed, 2), case, n_inst))


def _cache_keys(router, case, seed, b):
    """Every instance's cached-block keys: its template prefixes hashed by the library, then random ones."""
    n_t, hi = b["templates"].shape
    toff = torch.arange(n_t + 1, dtype=torch.int64, device=DEV) * hi
    keys, _ = router.hash_blocks(b["templates"].reshape(-1).contiguous(), toff)
    keys = keys.view(n_t, -1)
    col = torch.arange(keys.shape[1], device=DEV)[None]
    g, parts, off = _gen(seed, 4), [], [0]
    for i in range(case["n_inst"]):
        chain = keys[col < b["cached"][i][:, None]]
        rest = case["cache_blocks"] - chain.numel()
        parts += [chain, torch.randint(1, 2 ** 63 - 1, (rest,), generator=g, device=DEV)]
        off.append(off[-1] + case["cache_blocks"])
    return torch.cat(parts), torch.tensor(off, dtype=torch.int64, device=DEV)


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    return {"train": _prepare_train, "round": _prepare_round}.get(case["kind"], _prepare_route)(case, seed)


def _router(case, **caps):
    base = dict(max_instances=case.get("n_inst", 16), max_requests=case.get("n_req", 16), max_keys_per_instance=1024,
                ring_capacity=1024, max_train_batch=case.get("batch", 256), max_batch_tokens=1 << 16)
    base.update(caps)
    return H.Router(_widths(case), case["d_inst"], case["d_req"], case["dtype"], **base)


def _prepare_route(case, seed):
    b = _batch(case, seed)
    total = int(b["off"][-1])
    keys_cap = case["cache_blocks"] + (total // BLOCK if case["kind"] == "sequential" else 0)
    r = _router(case, max_keys_per_instance=keys_cap, max_batch_tokens=max(total, 1))
    keys, key_off = _cache_keys(r, case, seed, b)
    del b["templates"]
    r.set_normalizer(*_normaliser(seed, case))
    r.snapshot(case["n_inst"], b["inst"], keys, key_off)
    r.set_params(_params(seed, case))
    if case.get("guarded"):
        x, y = _records(_gen(seed, 5), dict(case, len_lo=max(1, case["len_lo"])), 1024)
        x[:case["n_inst"], PAIR:PAIR + case["d_inst"]] = b["inst"][:1024]  # the instances' states are known ones
        x[0, :PAIR] = 0.0
        x[1, :PAIR] = float(case["len_hi"])
        r.log(x, y)
        r.refresh_bounds()
        r.set_guards(n_min=100, ood=True, k=min(4, case["n_inst"]), kv_col=4, tau_sat=0.3, tau_ben=64.0,
                     heuristic=L.LS_HEUR_PREFIX_LOAD, count_cols=(0, 1), theta_imbal=8.0, k_overload=1.0)
    r.publish()
    s = dict(case=case, r=r, b=b)
    if case["kind"] == "snapshot":
        s.update(keys=keys, key_off=key_off)
    if case["graph"]:
        _route_pass(s)
        torch.cuda.synchronize()
        s["graph"] = H.StepGraph(lambda: s.update(out=_route_pass(s)))
    torch.cuda.synchronize()
    return s


def _route_pass(s):
    c, r, b = s["case"], s["r"], s["b"]
    call = r.route_guarded if c["guarded"] else r.route
    o = call(b["tok"], b["off"], b["req"], c["n_inst"], want_scores=c["scores"], want_hits=True)
    return {k: v for k, v in o.items() if k != "version" and v is not None}


def _prepare_train(case, seed):
    r = _router(case, max_requests=1, ring_capacity=case["ring"], max_train_batch=case["batch"],
                dropout=case["dropout"], dropout_seed=17)
    x, y = _records(_gen(seed, 5), case, case["ring"])
    mean, std = _normaliser(seed, case)
    r.set_normalizer(mean, std)
    r.set_params(_params(seed, case))
    if case["opt"] == "adam":  # the middle of a training run
        m, v = _opt_state(case, seed)
        r.set_opt_state(m, v, 1000)
    r.log(x, y)
    s = dict(case=case, r=r, loss=torch.zeros(1, device=DEV))
    torch.cuda.synchronize()
    if case["graph"]:
        # one pass outside capture on another context of the same shape (kernels are loaded outside capture)
        w = _router(case, max_requests=1, ring_capacity=case["batch"], max_train_batch=case["batch"],
                    dropout=case["dropout"], dropout_seed=17)
        w.set_normalizer(mean, std)
        w.set_params(_params(seed, case))
        w.log(x[:case["batch"]], y[:case["batch"]])
        w.train(case["batch"], None, opt=case["opt"], lr=case["lr"])
        torch.cuda.synchronize()
        w.close()
        s["graph"] = H.StepGraph(lambda: s.update(out=_train_pass(s)))
        torch.cuda.synchronize()
    return s


def _opt_state(case, seed):
    n = sum(a * b + b for a, b in zip(_widths(case)[:-1], _widths(case)[1:]))
    g = _gen(seed, 6)
    return 1e-4 * _normal(g, n), _uniform(g, 0.5e-6, 1.5e-6, n).float()


def _train_pass(s):
    c, r = s["case"], s["r"]
    r.train(c["batch"], None, opt=c["opt"], lr=c["lr"], loss_out=s["loss"])
    return {"loss": s["loss"], "params": r.get_params()}


def _prepare_round(case, seed):
    n = case["pool"]
    r = _router(case, max_requests=1, ring_capacity=n, pending_capacity=n, replay_capacity=n,
                max_train_batch=case["batch"], dropout=case["dropout"], dropout_seed=17)
    chunks = 16
    x, y = _records(_gen(seed, 5), case, 2 * n + chunks * case["new"])
    r.set_normalizer(*_normaliser(seed, case))
    r.set_params(_params(seed, case))
    r.log(x[:n], y[:n])
    r.log(x[n:2 * n], y[n:2 * n])
    r.replay_admit()  # the first n records fill the replay pool, in order
    r.refresh_bounds()
    r.publish()
    torch.cuda.synchronize()
    return dict(case=case, r=r, x=x, y=y, k=0, chunks=chunks, losses=torch.zeros(case["steps"], device=DEV))


def run(state):
    s = state
    c, r = s["case"], s["r"]
    if "graph" in s:
        s["graph"].replay()
        return s["out"]
    if c["kind"] == "route":
        return _route_pass(s)
    b = s.get("b")
    if c["kind"] == "sequential":
        r.snapshot(c["n_inst"], b["inst"])  # the instances' states as last reported
        o = r.route_sequential(b["tok"], b["off"], b["req"], c["n_inst"], queue_col=0)
        return {k: v for k, v in o.items() if k != "version"}
    if c["kind"] == "snapshot":
        r.snapshot(c["n_inst"], b["inst"], s["keys"], s["key_off"])
        return _route_pass(s)
    if c["kind"] == "train":
        return _train_pass(s)
    at = 2 * c["pool"] + (s["k"] % s["chunks"]) * c["new"]
    s["k"] += 1
    r.log(s["x"][at:at + c["new"]], s["y"][at:at + c["new"]])
    d, n = r.replay_admit(diag=True)
    r.refresh_bounds()
    for k in range(c["steps"]):
        r.train(c["batch"], None, opt="adam", lr=3e-4, loss_out=s["losses"][k:k + 1])
    r.publish()
    return {"d": d, "n": n, "losses": s["losses"], "params": r.get_params()}


# ---------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------

def _mlp_macs(w):
    return sum(a * b for a, b in zip(w[:-1], w[1:]))


def work(case):
    w = _widths(case)
    n_par = _mlp_macs(w) + sum(w[1:])
    if case["kind"] == "train":
        # a minibatch's records, the parameters (and Adam's two moments) read and written
        mom = 3 if case["opt"] == "adam" else 1
        return {"bytes": 4 * case["batch"] * (w[0] + 1) + 8 * n_par * mom,
                "flops": 2 * case["batch"] * (3 * _mlp_macs(w) - w[0] * w[1])}
    if case["kind"] == "round":
        n, new, hid = case["pool"], case["new"], w[-2]
        rows = n + new  # embedded records: candidates and kept
        return {"bytes": 4 * (2 * new * w[0] + rows * w[0] + case["steps"] * case["batch"] * w[0] + 2 * n) + 24 * n_par,
                "flops": 2 * rows * _mlp_macs(w) + 2 * rows * n * hid
                + 2 * case["steps"] * case["batch"] * (3 * _mlp_macs(w) - w[0] * w[1])}
    n_inst, n_req = case["n_inst"], case["n_req"]
    # tokens of the shared prefixes (the mean share of a prompt): no instance matches past them
    tokens = n_req * (case["len_lo"] + case["len_hi"]) / 2 * sum(RHO) / len(RHO)
    pairs = n_inst * n_req
    byt = 4 * tokens + 4 * (n_req * case["d_req"] + n_inst * case["d_inst"] + n_par) + 8 * n_req + 8 * n_req
    byt += 4 * pairs * (2 if case["scores"] else 1)
    if case["kind"] == "snapshot":
        byt += 2 * 8 * n_inst * case["cache_blocks"]
    # the instance and request columns of the first layer once per instance and per request, the six pair columns
    # and the later layers per pair
    macs = pairs * (_mlp_macs(w) - (w[0] - PAIR) * w[1]) + (n_inst * case["d_inst"] + n_req * case["d_req"]) * w[1]
    return {"bytes": byt, "flops": 2 * macs}


def tolerance(case):
    if case["kind"] == "train":
        # the updated parameters and the loss: a step moves the parameters by a few thousandths, and a bf16 step's
        # gradient is good to about a percent
        return {"rel": 1e-5, "max": 1e-4} if case["dtype"] == "f32" else {"rel": 3e-4, "max": 1e-2}
    if case["kind"] == "round":
        # distances of bf16 embeddings, and three of Adam's first steps, whose size does not follow the gradient's
        return {"rel": 5e-3, "max": 0.1}
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.002}
    return {"rel": 1e-2, "max": 5e-2, "differ": 0.005}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _bf(x):
    return x.float().bfloat16().double()


def _forward(layers, x, rounded=False):
    for k, (w, b) in enumerate(layers):
        x = (_bf(x) if rounded else x) @ (_bf(w) if rounded else w).T + b
        if k + 1 < len(layers):
            x = x.clamp(min=0)
    return x[:, 0]


def _features(length, h, inst, req, mean, std):
    """Normalised rows of every (request, instance) pair: [n_req * n_inst, d]."""
    n_req, n_inst = h.shape
    ln = length.double()[:, None].expand(n_req, n_inst)
    h = h.double()
    pair = torch.stack((ln, h, BLOCK * h, BLOCK * h / ln, ln - BLOCK * h, torch.ceil(ln / BLOCK) - h), 2)
    x = torch.cat((pair, inst.double()[None].expand(n_req, -1, -1), req.double()[:, None].expand(-1, n_inst, -1)), 2)
    std = std.double()
    return ((x - mean.double()) / torch.where(std < 1e-12, torch.ones_like(std), std)).reshape(n_req * n_inst, -1)


def _exact_route(case, seed):
    b = _batch(case, seed)
    mean, std = _normaliser(seed, case)
    layers = _layers(case, _params(seed, case))
    n_inst, n_req = case["n_inst"], case["n_req"]
    hits = torch.minimum(b["blocks"][:, None], b["cached"].T[b["t"]])
    step = max(1, 131072 // n_inst)
    sc = torch.cat([_forward(layers, _features(b["length"][a:a + step], hits[a:a + step], b["inst"],
                                               b["req"][a:a + step], mean, std)).view(-1, n_inst)
                    for a in range(0, n_req, step)])
    best, choice = sc.min(1)
    out = {"hits": hits.int()}
    # a guarded route picks among hashed candidates and hands some requests back: no such value without the hash
    out["choice"] = None if case["guarded"] else choice.int()
    out["best"] = None if case["guarded"] else best
    if case["scores"]:
        out["scores"] = sc
    return out


def _exact_sequential(case, seed):
    """Decisions feed on one another, so the predictor's bf16 operands are rounded as its type says; sums in 64 bits."""
    b = _batch(case, seed)
    mean, std = _normaliser(seed, case)
    layers = _layers(case, _params(seed, case))
    inst, cached = b["inst"].clone(), b["cached"].clone()
    rows, hit_rows, choice = [], [], []
    for r in range(case["n_req"]):
        t = b["t"][r]
        h = torch.minimum(b["blocks"][r], cached[:, t])
        sc = _forward(layers, _features(b["length"][r:r + 1], h[None], inst, b["req"][r:r + 1], mean, std),
                      case["dtype"] == "bf16")
        c = int(sc.argmin())
        inst[c, 0] += 1
        cached[c, t] = torch.maximum(cached[c, t], b["blocks"][r])
        rows.append(sc)
        hit_rows.append(h)
        choice.append(c)
    sc = torch.stack(rows)
    return {"choice": torch.tensor(choice, dtype=torch.int32), "best": sc.min(1)[0], "scores": sc,
            "hits": torch.stack(hit_rows).int()}


def _exact_train(case, seed):
    if case["dropout"]:
        return None  # the masks are the library's own stream
    x, y = _records(_gen(seed, 5), case, case["ring"])
    mean, std = _normaliser(seed, case)
    flat = _params(seed, case).double()
    step = 1000 if case["opt"] == "adam" else 0
    idx = (step * case["batch"] + torch.arange(case["batch"], device=DEV)) % case["ring"]
    sd = std.double()
    z = (x[idx].double() - mean.double()) / torch.where(sd < 1e-12, torch.ones_like(sd), sd)
    flat.requires_grad_(True)
    loss = ((_forward(_layers(case, flat), z) - y[idx].double()) ** 2).mean()
    (g,) = torch.autograd.grad(loss, flat)
    with torch.no_grad():
        if case["opt"] == "sgd":
            new = flat - case["lr"] * g
        else:
            m, v = (a.double() for a in _opt_state(case, seed))
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            t = step + 1
            new = flat - case["lr"] * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"loss": loss.detach().view(1), "params": new}


def _exact_round(case, seed):
    n, new = case["pool"], case["new"]
    x, y = _records(_gen(seed, 5), case, 2 * n + 16 * new)
    mean, std = _normaliser(seed, case)
    layers = _layers(case, _params(seed, case))
    sd = std.double()
    z = (x[:n + new].double() - mean.double()) / torch.where(sd < 1e-12, torch.ones_like(sd), sd)
    for w, bias in layers[:-1]:
        z = (z @ w.T + bias).clamp(min=0)
    w, bias = layers[-1]
    emb = (z @ w.T + bias - y[:n + new, None].double()) * z
    kept, cand = emb[:n], emb[n:]
    far = torch.full((n,), math.inf, dtype=torch.float64, device=DEV)
    far[:new] = torch.cdist(cand, kept, compute_mode="donot_use_mm_for_euclid_dist").square().min(1)[0]
    own = torch.cdist(kept, kept, compute_mode="donot_use_mm_for_euclid_dist").square()
    own.fill_diagonal_(math.inf)
    # the training steps draw their dropout masks from the library's own stream
    return {"d": far, "n": own.min(1)[0], "losses": None, "params": None}


def exact(case, seed):
    return {"train": _exact_train, "round": _exact_round,
            "sequential": _exact_sequential}.get(case["kind"], _exact_route)(case, seed)
