"""The generic tensor-core scorer at the edges of its 128-row tiles: instance
counts that divide a tile, leave rows of it unused or exceed it, one tile to
several per CTA, one or two CTAs an SM, with and without the selection inside
the scorer."""
import numpy as np
import pytest
import torch

from paper_2606_00946_gb300 import build as B
from paper_2606_00946_gb300 import harness as H
from paper_2606_00946_gb300 import lodestar as L

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def forward(flat, widths, x):
    """fp64 sums of bf16 operands (the output layer's weights stay fp32)."""
    r = lambda t: t.float().bfloat16().double()
    x, o = x.double(), 0
    for k, (a, b) in enumerate(zip(widths[:-1], widths[1:])):
        w, bias = flat[o:o + a * b].view(b, a).double(), flat[o + a * b:o + a * b + b].double()
        o += a * b + b
        x = r(x) @ (r(w) if k + 2 < len(widths) else w).T + bias
        if k + 2 < len(widths):
            x = x.clamp(min=0)
    return x[:, 0]


CASES = [  # instances, requests, hidden
    (16, 1, (128, 128, 128)), (16, 4096, (128, 128, 128)), (24, 5, (128, 128, 128)), (24, 6, (128, 128, 128)),
    (128, 2, (128, 128, 128)), (200, 400, (128, 128, 128)), (1, 129, (64,)), (64, 3001, (64,)), (3, 42, (64,)),
    (32, 1999, (192, 192, 192)), (127, 1, (192, 192, 192)),
]


@pytest.mark.parametrize("n_inst,n_req,hidden", CASES)
def test_scores_and_selection(n_inst, n_req, hidden):
    d_inst, d_req = 11, 5
    widths = [6 + d_inst + d_req, *hidden, 1]
    g = torch.Generator(device="cuda").manual_seed(n_inst * 1000 + n_req)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda")
    r = H.Router(widths, d_inst, d_req, "bf16", max_instances=n_inst, max_requests=n_req, max_keys_per_instance=64,
                 max_batch_tokens=n_req * 80, ring_capacity=16, max_train_batch=16)
    lens = torch.randint(0, 80, (n_req,), generator=g, device="cuda")
    off = torch.zeros(n_req + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(lens, 0)
    tok = torch.randint(0, 32000, (int(off[-1]) + 1,), generator=g, device="cuda", dtype=torch.int32)
    keys, ko = r.hash_blocks(tok, off)
    state, req = n(n_inst, d_inst), n(n_req, d_req)
    flat = torch.cat([torch.cat([n(b * a) / a ** 0.5, n(b) * 0.1]) for a, b in zip(widths[:-1], widths[1:])])
    mean, std = n(widths[0]), n(widths[0]).abs() + 0.5
    mean[:6], std[:6] = 20.0, 30.0
    r.set_normalizer(mean, std)
    some = keys[torch.randperm(keys.numel(), generator=g, device="cuda")[:60]]
    r.snapshot(n_inst, state, some, torch.tensor([0] + [some.numel()] * n_inst, dtype=torch.int64, device="cuda"))
    r.set_params(flat)
    r.publish()
    out = r.route(tok, off, req, n_inst)
    assert r.sync() == L.LS_OK
    x = r.features(off, out["hits"], req)
    want = forward(flat, widths, x)
    got = out["scores"].reshape(-1).double()
    # fp32 sums; a rounding point of a hidden layer may go the other way (2^-9 of one unit)
    assert float((got - want).abs().max()) <= 1e-2 * float(want.abs().max().clamp(min=1.0))
    s = out["scores"].cpu().numpy()
    ch = out["choice"].cpu().numpy()
    assert np.array_equal(ch, s.argmin(1)) and np.array_equal(out["best"].cpu().numpy(), s[np.arange(n_req), ch])
    # without the optional outputs: the same selection
    o2 = r.route(tok, off, req, n_inst, want_scores=False, want_hits=False)
    assert torch.equal(o2["choice"], out["choice"]) and torch.equal(o2["best"], out["best"])
    r.close()
