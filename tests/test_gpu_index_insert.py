"""Index insertion at the edges of its key chunks: membership of every key on
every instance, and the distinct-key count that max_keys bounds."""
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


def router(n_inst, max_keys, n_req):
    r = H.Router([16, 64, 1], 10, 0, "bf16", max_instances=n_inst, max_requests=n_req,
                 max_keys_per_instance=max_keys, max_batch_tokens=n_req * 16, ring_capacity=16, max_train_batch=64)
    r.set_normalizer(torch.zeros(16, device="cuda"), torch.ones(16, device="cuda"))
    r.set_params(torch.zeros(r.n_params, device="cuda"))
    r.publish()
    return r


# keys per instance around one warp's chunk (128 keys), empty instances, one
# to four mask words
COUNTS = [[1], [127], [128], [129, 0, 127], [0, 256, 0, 1], [5] * 70, [0, 640] + [33] * 200]


@pytest.mark.parametrize("spare,counts", [(s, c) for s in (0, -1) for c in COUNTS if max(c) + s >= 1])
def test_membership_and_distinct_counts(counts, spare):
    n_inst, n_req = len(counts), 700
    g = np.random.default_rng(sum(counts) + n_inst)
    toks = torch.from_numpy(g.integers(0, 32000, size=(n_req, 16)).astype(np.int32)).cuda()
    off = torch.arange(n_req + 1, dtype=torch.int64, device="cuda") * 16
    probe = router(1, 16, n_req)
    keys, _ = probe.hash_blocks(toks.reshape(-1), off)
    held = [g.choice(n_req, size=c, replace=False) for c in counts]
    # every key of the first non-empty instance twice: distinct keys count once
    rows = [np.concatenate([h, h]) if i == next(k for k, c in enumerate(counts) if c) else h
            for i, h in enumerate(held)]
    koff = torch.tensor(np.concatenate([[0], np.cumsum([len(x) for x in rows])]), dtype=torch.int64, device="cuda")
    flat = keys[torch.from_numpy(np.concatenate(rows).astype(np.int64)).cuda()]
    cap = max(counts) + spare
    r = router(n_inst, cap, n_req)
    state = torch.zeros(n_inst, 10, device="cuda")
    r.snapshot(n_inst, state, flat, koff)
    out = r.route(toks.reshape(-1), off, torch.zeros(n_req, 0, device="cuda"), n_inst)
    assert r.sync() == (L.LS_OK if spare == 0 else L.LS_ERR_TABLE_FULL)
    want = np.zeros((n_req, n_inst), np.int32)
    for i, h in enumerate(held):
        want[h, i] = 1
    assert np.array_equal(out["hits"].cpu().numpy(), want)
    # an insert of the same keys changes nothing
    if spare == 0:
        r.snapshot(n_inst, state, flat, koff, mode=L.LS_INSERT)
        again = r.route(toks.reshape(-1), off, torch.zeros(n_req, 0, device="cuda"), n_inst)
        assert r.sync() == L.LS_OK
        assert np.array_equal(again["hits"].cpu().numpy(), want)


# more keys than a GPU of 152 SMs has threads: four a thread into a cleared
# table, one a thread into a filled one
@pytest.mark.parametrize("counts", [[200_000, 0, 150_001], [330_000], [4000] * 70 + [40_000]])
@pytest.mark.parametrize("spare", [0, -1])
def test_many_keys(counts, spare):
    n_inst, n_req = len(counts), 700
    g = np.random.default_rng(sum(counts))
    toks = torch.from_numpy(g.integers(0, 32000, size=(n_req, 16)).astype(np.int32)).cuda()
    off = torch.arange(n_req + 1, dtype=torch.int64, device="cuda") * 16
    r = router(n_inst, max(counts) + spare, n_req)
    keys, _ = r.hash_blocks(toks.reshape(-1), off)
    # each instance: some of the prompts' keys, the rest distinct others, in any order
    held = [np.sort(g.choice(n_req, size=min(c, 300), replace=False)) for c in counts]
    flat = []
    for h, c in zip(held, counts):
        fill = torch.from_numpy(g.integers(1 << 20, 1 << 62, size=c - len(h)) | 1).cuda()
        k = torch.cat([keys[torch.from_numpy(h).cuda()], fill])
        assert len(torch.unique(k)) == c
        flat.append(k[torch.from_numpy(g.permutation(c)).cuda()])
    koff = torch.tensor(np.concatenate([[0], np.cumsum(counts)]), dtype=torch.int64, device="cuda")
    flat, state = torch.cat(flat), torch.zeros(n_inst, 10, device="cuda")
    want = np.zeros((n_req, n_inst), np.int32)
    for i, h in enumerate(held):
        want[h, i] = 1
    for mode in (L.LS_REPLACE, L.LS_INSERT):  # (the insert changes nothing)
        r.snapshot(n_inst, state, flat, koff, mode=mode)
        out = r.route(toks.reshape(-1), off, torch.zeros(n_req, 0, device="cuda"), n_inst)
        assert r.sync() == (L.LS_OK if spare == 0 or mode == L.LS_INSERT else L.LS_ERR_TABLE_FULL)
        assert np.array_equal(out["hits"].cpu().numpy(), want)
    r.close()
