"""Which way an fp32 training step goes by its batch: in two launches up to the
batch where the general path's products become the faster ones, and the
gradient on either side of that line."""
import pytest
import torch

from paper_2606_00946_gb300 import build as B
from paper_2606_00946_gb300 import harness as H
from paper_2606_00946_gb300 import lodestar as L
from test_gpu_train_ragged import reference_gradient

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


# rows a CTA takes in one tile while the step stays in two launches (None: at any batch)
@pytest.mark.parametrize("hidden,rows", [((), 32), ((64, 20), None), ((300,), 32), ((128, 128, 128), 32),
                                         ((192, 96), 32), ((256, 256), 16), ((100, 500), 16), ((900,), 16)])
def test_both_sides_of_the_line(hidden, rows):
    d_inst, d_req = 10, 0
    widths = [6 + d_inst + d_req, *hidden, 1]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    line = 20000 if rows is None else rows * sms
    g = torch.Generator(device="cuda").manual_seed(len(hidden))
    r = H.Router(widths, d_inst, d_req, "f32", max_instances=4, max_requests=4, max_keys_per_instance=64,
                 ring_capacity=line + 1, max_train_batch=line + 1, max_batch_tokens=64)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda")
    x, y = n(line + 1, widths[0]), n(line + 1)
    flat = torch.cat([torch.cat([n(b * a) / a ** 0.5, n(b) * 0.1]) for a, b in zip(widths[:-1], widths[1:])])
    r.set_normalizer(torch.zeros(widths[0], device="cuda"), torch.ones(widths[0], device="cuda"))
    r.log(x, y)
    for batch in (line, line + 1):
        idx = torch.randperm(line + 1, generator=g, device="cuda")[:batch].int()
        r.set_params(flat)
        assert L.ls_trace_enable(r.h, True) == L.LS_OK
        r.train(batch, idx, opt="sgd", lr=1e-2)
        rc, entries = L.ls_trace_read(r.h)
        assert rc == L.LS_OK and L.ls_trace_enable(r.h, False) == L.LS_OK
        names = {k for k, v in entries.items() if v[0]}
        assert ("train_gather" in names) == (rows is not None and batch > line), (batch, names)
        got = (flat.double() - r.get_params().double()) / 1e-2
        want = reference_gradient(flat, widths, x[idx.long()], y[idx.long()], bf16=False)
        # (the bound of the fp32 gradients in test_gpu_train_ragged)
        bound = 2e-5 * want.norm() + 2.0 ** -23 * flat.double().norm() / 1e-2
        assert float((got - want).norm()) <= float(bound)
    assert r.sync() == L.LS_OK
    r.close()
