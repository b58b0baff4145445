"""The prefix-index walk over its launch shapes (a CTA per request, a warp per
request, requests sorted by length), mask words and token alignments, against
the per-instance tables' two-phase kernels on the same keys: equal hit lengths."""
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


# requests: CTAs of eight and four warps, warps, warps taking sorted requests; instances: one to eight mask words;
# first token of the batch at every position in 16 bytes
@pytest.mark.parametrize("n_req,n_inst,max_len,shift", [
    (1, 3, 9000, 1), (608, 64, 900, 2), (609, 65, 700, 3), (1216, 16, 600, 1), (1217, 16, 600, 0), (1300, 130, 300, 2),
    (152, 300, 1200, 3), (153, 300, 1200, 1), (5000, 10, 700, 1), (5000, 100, 200, 3), (4900, 200, 150, 0),
    (6000, 1, 100, 2), (2000, 500, 100, 1)])
def test_hits_equal_the_two_phase_kernels(n_req, n_inst, max_len, shift):
    g = np.random.default_rng(n_req + n_inst)
    tmpl = g.integers(0, 32000, size=(4, max_len)).astype(np.int32)
    lens = g.integers(0, max_len + 1, size=n_req)
    lens[: min(n_req, 40)] = (np.arange(40) * 16 + g.integers(-1, 2, 40)).clip(0, max_len)[: min(n_req, 40)]
    lens[-1] = max_len
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    tok = g.integers(0, 32000, size=int(off[-1])).astype(np.int32)
    for r in range(n_req):
        n = int(lens[r] * g.choice([0, 0.3, 0.7, 1.0]))
        tok[off[r]:off[r] + n] = tmpl[r % 4, :n]
    flat = torch.zeros(int(off[-1]) + 8, dtype=torch.int32, device="cuda")
    view = flat[shift:shift + int(off[-1])]
    view.copy_(torch.from_numpy(tok))
    toff = torch.from_numpy(off).cuda()
    routers = [H.Router([16, 64, 1], 10, 0, "bf16", max_instances=n_inst, max_requests=n_req, prefix_mode=mode,
                        max_keys_per_instance=4096, max_batch_tokens=int(off[-1]) + 16, ring_capacity=16,
                        max_train_batch=64) for mode in ("index", "two_phase")]
    tk, to = torch.from_numpy(tmpl.reshape(-1)).cuda(), torch.arange(5, dtype=torch.int64, device="cuda") * max_len
    keys, ko = routers[0].hash_blocks(tk, to)
    nb = max_len // 16
    held = []
    for i in range(n_inst):  # the first blocks of some templates, with a hole now and then
        for t in range(4):
            k = keys[ko[t]:ko[t] + int(g.integers(0, nb + 1))]
            held.append(torch.cat([k[:7], k[8:]]) if g.random() < 0.2 else k)
    ioff = np.concatenate([[0], np.cumsum([sum(len(held[4 * i + t]) for t in range(4)) for i in range(n_inst)])])
    hits = []
    for r in routers:
        r.set_normalizer(torch.zeros(16, device="cuda"), torch.ones(16, device="cuda"))
        r.set_params(torch.zeros(r.n_params, device="cuda"))
        r.snapshot(n_inst, torch.zeros(n_inst, 10, device="cuda"), torch.cat(held), torch.from_numpy(ioff).cuda())
        r.publish()
        for _ in range(2):  # the second call finds the counters the first one left
            out = r.route(view, toff, torch.zeros(n_req, 0, device="cuda"), n_inst)
        assert r.sync() == L.LS_OK
        hits.append(out["hits"])
    assert torch.equal(hits[0], hits[1])
    assert int(hits[0].max()) > 0
    for r in routers:
        r.close()


def test_the_trace_lists_the_sort():
    """A traced route's launches: the walk alone, or the sort by length and the walk."""
    for n_req, want in ((64, 0), (1300, 0), (6000, 1)):
        r = H.Router([16, 64, 1], 10, 0, "bf16", max_instances=4, max_requests=n_req, max_keys_per_instance=64,
                     max_batch_tokens=16 * n_req, ring_capacity=16, max_train_batch=64)
        r.set_normalizer(torch.zeros(16, device="cuda"), torch.ones(16, device="cuda"))
        r.set_params(torch.zeros(r.n_params, device="cuda"))
        r.snapshot(4, torch.zeros(4, 10, device="cuda"))
        r.publish()
        tok = torch.zeros(16 * n_req, dtype=torch.int32, device="cuda")
        off = torch.arange(n_req + 1, dtype=torch.int64, device="cuda") * 16
        assert L.ls_trace_enable(r.h, True) == L.LS_OK
        r.route(tok, off, torch.zeros(n_req, 0, device="cuda"), 4)
        rc, entries = L.ls_trace_read(r.h)
        assert rc == L.LS_OK and entries["prefix_index"][0] == 1, (n_req, entries)
        assert entries.get("walk_order", (0,))[0] == want, (n_req, entries)
        r.close()
