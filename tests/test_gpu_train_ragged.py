"""Training steps whose batch is not a whole number of weight-gradient splits:
every row of the minibatch reaches the gradient."""
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


def reference_gradient(flat, widths, x, y, bf16=True):
    """Gradient of the minibatch loss (the products' operands in bf16 where asked), sums in fp64."""
    r = lambda t: t.float().bfloat16().double() if bf16 else t.double()
    layers, o = [], 0
    for a, b in zip(widths[:-1], widths[1:]):
        layers.append((flat[o:o + a * b].view(b, a).double(), flat[o + a * b:o + a * b + b].double()))
        o += a * b + b
    acts, z = [r(x)], None
    for k, (w, b) in enumerate(layers):
        z = acts[-1] @ r(w).T + b
        if k + 1 < len(layers):
            acts.append(r(z.clamp(min=0)))
    dz = 2.0 * (z[:, 0] - y.double())[:, None] / len(y)
    grads = []
    for k in reversed(range(len(layers))):
        grads = [r(dz).T @ acts[k], dz.sum(0)] + grads
        if k:
            dz = (r(dz) @ r(layers[k][0])) * (acts[k] > 0)
    return torch.cat([g.reshape(-1) for g in grads])


# batches whose 64-row blocks leave a short last split (and some that do not)
@pytest.mark.parametrize("hidden,batch", [((256, 256), 3200), ((256, 256), 4096), ((256, 256, 256), 3900),
                                          ((128, 128), 1), ((64,), 129), ((256, 256), 8100),
                                          # wider than 256: K-blocks streamed through the stages, parts of 128 (or,
                                          # for few rows, 64) columns, clusters of two and four
                                          ((512, 512), 4096), ((512, 512), 130), ((384, 384), 3200), ((128, 512), 700),
                                          ((512, 64, 384), 1100), ((512,), 1), ((448, 512), 300)])
def test_every_row_reaches_the_gradient(hidden, batch):
    d_inst, d_req = 34, 24
    widths = [6 + d_inst + d_req, *hidden, 1]
    r = H.Router(widths, d_inst, d_req, "bf16", max_instances=4, max_requests=4, max_keys_per_instance=64,
                 ring_capacity=batch, max_train_batch=batch, max_batch_tokens=64)
    g = torch.Generator(device="cuda").manual_seed(batch)
    x = torch.randn(batch, widths[0], generator=g, device="cuda")
    y = torch.randn(batch, generator=g, device="cuda")
    y[-128:] += 30.0  # the last rows carry most of the gradient
    flat = torch.cat([torch.cat([torch.randn(b * a, generator=g, device="cuda") / a ** 0.5,
                                 torch.randn(b, generator=g, device="cuda") * 0.1])
                      for a, b in zip(widths[:-1], widths[1:])])
    r.set_normalizer(torch.zeros(widths[0], device="cuda"), torch.ones(widths[0], device="cuda"))
    r.set_params(flat)
    r.log(x, y)
    lr = 1e-2
    r.train(batch, None, opt="sgd", lr=lr)
    got = (flat.double() - r.get_params().double()) / lr
    assert r.sync() == 0
    want = reference_gradient(flat, widths, x, y)
    # bf16 operands agree on both sides; what differs is fp32 sums, the bf16
    # values they put on the other side of a rounding midpoint (2^-8 of a few),
    # and the fp32 subtraction of the update (2^-24 |p| / lr)
    bound = 5e-3 * want.norm() + 2.0 ** -23 * flat.double().norm() / lr
    assert float((got - want).norm()) <= float(bound)
    r.close()


# fp32 tiles of 4, 8, 16 and 32 rows, several tiles per CTA, odd widths,
# weights resident and staged in chunks, no hidden layer
@pytest.mark.parametrize("hidden,batch", [((64, 64), 1), ((64, 64), 256), ((64, 64), 700), ((64, 64), 1300),
                                          ((64, 64), 3001), ((64, 64), 6000), ((100, 50), 333), ((33, 7, 65), 130),
                                          ((128, 128, 128), 1024), ((256, 256), 515), ((1000,), 90), ((), 257),
                                          ((300, 200, 100), 64)])
def test_every_row_reaches_the_fp32_gradient(hidden, batch):
    d_inst, d_req = 34, 24
    widths = [6 + d_inst + d_req, *hidden, 1]
    ring = batch + 37
    r = H.Router(widths, d_inst, d_req, "f32", max_instances=4, max_requests=4, max_keys_per_instance=64,
                 ring_capacity=ring, max_train_batch=batch, max_batch_tokens=64)
    g = torch.Generator(device="cuda").manual_seed(batch)
    x = torch.randn(ring, widths[0], generator=g, device="cuda")
    y = torch.randn(ring, generator=g, device="cuda")
    flat = torch.cat([torch.cat([torch.randn(b * a, generator=g, device="cuda") / a ** 0.5,
                                 torch.randn(b, generator=g, device="cuda") * 0.1])
                      for a, b in zip(widths[:-1], widths[1:])])
    idx = torch.randperm(ring, generator=g, device="cuda")[:batch].int()
    y[idx[-1]] += 50.0  # the last row carries much of the gradient
    r.set_normalizer(torch.zeros(widths[0], device="cuda"), torch.ones(widths[0], device="cuda"))
    r.set_params(flat)
    r.log(x, y)
    lr, loss = 1e-2, torch.zeros(1, device="cuda")
    r.train(batch, idx, opt="sgd", lr=lr, loss_out=loss)
    got = (flat.double() - r.get_params().double()) / lr
    assert r.sync() == 0
    xi, yi = x[idx.long()], y[idx.long()]
    want = reference_gradient(flat, widths, xi, yi, bf16=False)
    # fp32 sums of up to `batch` terms (2^-24 sqrt(n) of the norm, a few layers deep; a ReLU whose input lies within
    # rounding of 0 may go the other way for a row) and the update's fp32 subtraction
    bound = 2e-5 * want.norm() + 2.0 ** -23 * flat.double().norm() / lr
    assert float((got - want).norm()) <= float(bound)
    # twice the same step from the same state: the same bits
    p1 = r.get_params()
    r.set_params(flat)
    r.train(batch, idx, opt="sgd", lr=lr, loss_out=loss)
    assert torch.equal(p1, r.get_params())
    r.close()


def test_dropout_needs_hidden_widths_up_to_256():
    with pytest.raises(L.LodestarError):
        H.Router([64, 512, 512, 1], 34, 24, "bf16", dropout=0.1)
