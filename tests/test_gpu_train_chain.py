"""The training step's forward and input-gradient passes in one launch: the
same bits as the persistent step, whose products run one after the other over
the whole batch, for clusters of one and two CTAs a tile, layers of unlike
widths (two to four of them), one layer to four, short last tiles, dropout and a bad slot."""
import pytest
import torch

from paper_2606_00946_gb300 import build as B
from paper_2606_00946_gb300 import harness as H
from paper_2606_00946_gb300 import lodestar as L

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


CASES = [  # hidden, instance and request widths, batch, dropout
    ((64,), 10, 0, 1, 0.0), ((128,), 34, 24, 129, 0.0), ((256,), 120, 120, 300, 0.0), ((128, 64), 23, 9, 2048, 0.0),
    ((256, 128), 34, 24, 257, 0.1), ((128, 256), 34, 24, 640, 0.1), ((64, 192), 34, 24, 384, 0.0),
    ((192, 192), 66, 56, 4096, 0.1), ((128, 128, 128), 34, 24, 4096, 0.1), ((128, 128), 34, 24, 10000, 0.0),
    ((256, 256, 256), 66, 56, 4096, 0.0), ((256, 256, 256, 256), 66, 56, 130, 0.1),
    # clusters of two whose columns of one product are not those of the next, three and four products in a row
    ((128, 256, 256), 34, 24, 8192, 0.0), ((256, 128, 128), 34, 24, 8192, 0.1), ((256, 256, 128), 34, 24, 4096, 0.0),
    ((128, 128, 256), 34, 24, 4096, 0.1), ((256, 128, 256), 120, 120, 9000, 0.0),
    ((128, 256, 128, 256), 34, 24, 8192, 0.1), ((256, 128, 128, 256), 10, 3, 4096, 0.0),
]


@pytest.mark.parametrize("hidden,d_inst,d_req,batch,dropout", CASES)
def test_same_bits_as_the_persistent_step(hidden, d_inst, d_req, batch, dropout):
    widths = [6 + d_inst + d_req, *hidden, 1]
    g = torch.Generator(device="cuda").manual_seed(batch)
    n = lambda *s: torch.randn(*s, generator=g, device="cuda")
    ring = batch + 50
    x, y = n(ring, widths[0]), n(ring)
    flat = torch.cat([torch.cat([n(b * a) / a ** 0.5, n(b) * 0.1]) for a, b in zip(widths[:-1], widths[1:])])
    idx = torch.randint(0, ring, (batch,), generator=g, device="cuda", dtype=torch.int32)
    seen = []
    for ctas in (0, 16):
        r = H.Router(widths, d_inst, d_req, "bf16", max_instances=4, max_requests=4, max_keys_per_instance=64,
                     ring_capacity=ring, max_train_batch=batch, max_batch_tokens=64, dropout=dropout, train_ctas=ctas)
        r.set_normalizer(torch.zeros(widths[0], device="cuda"), torch.ones(widths[0], device="cuda"))
        r.set_params(flat)
        r.log(x, y)
        loss = torch.zeros(4, device="cuda")
        for k in range(3):
            r.train(batch, idx if k == 1 else None, opt="adam", lr=1e-3, loss_out=loss[k:k + 1])
        assert r.sync() == L.LS_OK
        p = r.get_params()
        bad = idx.clone()
        bad[batch // 2] = ring
        r.train(batch, bad, opt="adam", lr=1e-3, loss_out=loss[3:])
        assert r.sync() == L.LS_ERR_ARG and torch.equal(r.get_params(), p) and bool(loss[3].isnan())
        seen.append((p, loss[:3].clone()))
        r.close()
    assert bool(seen[0][0].isfinite().all()) and not torch.equal(seen[0][0], flat)
    assert torch.equal(seen[0][0], seen[1][0]) and torch.equal(seen[0][1], seen[1][1])
