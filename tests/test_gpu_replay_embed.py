"""Replay admission's embeddings over predictor shapes and pool sizes: the
distances of a round against fp64 embeddings (operands rounded to bf16), with
hidden layers of different widths and pools that end inside a row tile."""
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


# hidden layers (operand images; 320 and 96 through the general forward), FIFO, pending and replay sizes, new records
@pytest.mark.parametrize("hidden,fifo,pending,replay,new", [
    ((64, 256), 300, 300, 300, 200), ((256, 64), 129, 128, 130, 100), ((384, 128), 700, 520, 257, 300),
    ((192,), 64, 200, 1, 64), ((128, 128, 128), 1000, 1000, 999, 1), ((320, 128), 200, 150, 140, 90),
    ((96, 64), 200, 150, 140, 90)])
def test_round_distances(hidden, fifo, pending, replay, new):
    d_inst, d_req = 20, 10
    widths = [6 + d_inst + d_req, *hidden, 1]
    g = torch.Generator(device="cuda").manual_seed(fifo + new)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda")
    r = H.Router(widths, d_inst, d_req, "bf16", max_instances=2, max_requests=2, max_keys_per_instance=16,
                 ring_capacity=fifo, pending_capacity=pending, replay_capacity=replay, max_train_batch=256,
                 max_batch_tokens=64)
    x, y = n(2 * fifo + replay + new, widths[0]), n(2 * fifo + replay + new)
    flat = torch.cat([torch.cat([n(b * a) / a ** 0.5, n(b) * 0.1]) for a, b in zip(widths[:-1], widths[1:])])
    r.set_normalizer(torch.zeros(widths[0], device="cuda"), torch.ones(widths[0], device="cuda"))
    r.set_params(flat)
    r.log(x[:fifo], y[:fifo])
    kept = min(replay, pending, fifo)
    r.log(x[fifo:fifo + kept], y[fifo:fifo + kept])  # evicts the first records, all of which are admitted
    r.replay_admit()
    assert r.info().replay_count == kept
    at = fifo + kept
    r.log(x[at:at + new], y[at:at + new])
    m = min(new, pending)
    d, nn = r.replay_admit(diag=True)
    assert r.sync() == L.LS_OK
    rb = lambda t: t.float().bfloat16().double()
    a, o = rb(x[:kept + new]), 0
    for p, q in zip(widths[:-2], widths[1:-1]):
        a = rb((a @ rb(flat[o:o + p * q].view(q, p)).T + flat[o + p * q:o + p * q + q].double()).clamp(min=0))
        o += p * q + q
    yhat = a @ rb(flat[o:o + widths[-2]]) + flat[-1].double()
    emb = rb((yhat - y[:kept + new].double())[:, None] * a)
    cand, keep = emb[kept + new - m:], emb[:kept]
    # products of bf16 embeddings with fp32 sums; a rounding point that goes the other way moves a component by 2^-8
    # of itself, a distance by a few 2^-8 of the norms that nearly cancel in it
    scale = emb.square().sum(1).max().item()
    want = torch.cdist(cand, keep, compute_mode="donot_use_mm_for_euclid_dist").square().min(1)[0]
    assert float((d[:m].double() - want).abs().max()) <= 5e-3 * scale
    assert bool(torch.isinf(d[m:]).all())
    if kept > 1:
        own = torch.cdist(keep, keep, compute_mode="donot_use_mm_for_euclid_dist").square().fill_diagonal_(np.inf)
        assert float((nn[:kept].double() - own.min(1)[0]).abs().max()) <= 5e-3 * scale
    r.close()
