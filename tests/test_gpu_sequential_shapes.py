"""Sequential-commit routing over the shapes its cluster splits differently
(instances per CTA, mask words, odd widths, weights beyond shared memory) and
over prompts that share prefixes with the one or two requests before them,
long ones included: every step equals a one-request batch route from the state
the earlier decisions left (snapshot rows and inserted keys)."""
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


def prompts(g, long):
    """Requests that repeat, extend and leave the prompts one and two before them."""
    t = lambda n: g.integers(0, 32000, size=n).astype(np.int32)
    a, b = t(9000 if long else 700), t(13000 if long else 333)
    cat = np.concatenate
    return [a, a, cat([a[:-7], t(40)]), b, a, b, cat([b, t(100)]), t(0), cat([b, t(64)]), t(15), t(16),
            cat([a[:len(a) // 2], t(50)]), a, a, a, b[:31], cat([b[:200], a])]


CASES = [  # instances, state columns, extras, hidden, dtype, long prompts
    (1, 4, 3, (20, 33), "bf16", False), (2, 5, 0, (64,), "f32", False), (3, 4, 3, (33, 7, 21), "f32", True),
    (7, 10, 5, (64, 64), "bf16", True), (8, 34, 24, (128, 128, 128), "bf16", False),
    (9, 34, 24, (256, 256), "bf16", True), (17, 4, 3, (40,), "bf16", True), (33, 10, 0, (64, 64), "f32", True),
    (16, 66, 56, (512, 512), "bf16", False), (70, 10, 2, (64, 32), "bf16", True), (130, 4, 2, (48,), "f32", True),
    (300, 4, 2, (16, 16), "bf16", True), (5, 3, 1, (), "f32", False),
    # a step that is shorter than its inserts: one instance, no hidden layer, hundreds of blocks
    (1, 3, 1, (), "f32", True), (1, 3, 1, (), "bf16", True),
]


@pytest.mark.parametrize("n_inst,d_inst,d_req,hidden,dtype,long", CASES)
def test_every_step_is_a_batch_route_of_the_committed_state(n_inst, d_inst, d_req, hidden, dtype, long):
    g = np.random.default_rng(n_inst)
    seqs = prompts(g, long)
    R = len(seqs)
    off = np.concatenate([[0], np.cumsum([len(s) for s in seqs])]).astype(np.int64)
    tok = torch.from_numpy(np.concatenate(seqs)).cuda()
    toff = torch.from_numpy(off).cuda()
    widths = [6 + d_inst + d_req, *hidden, 1]
    mk = lambda **kw: H.Router(widths, d_inst, d_req, dtype, max_instances=n_inst, max_requests=R,
                               max_keys_per_instance=1 << 15, max_batch_tokens=int(off[-1]) + 16 * R,
                               ring_capacity=16, max_train_batch=16, scorer="cuda_cores", **kw)
    a, b = mk(), mk()
    keys, koff = a.hash_blocks(tok, toff)
    kh = koff.cpu().numpy()
    f = lambda *s: torch.from_numpy(g.standard_normal(s).astype(np.float32)).cuda()
    state, req, params = f(n_inst, d_inst), f(R, d_req), f(a.n_params) * 0.3
    mean, std = f(widths[0]), f(widths[0]).abs() + 0.5
    mean[:6] = torch.tensor([900.0, 30, 500, 0.5, 400, 25])
    std[:6] = torch.tensor([900.0, 30, 500, 0.5, 400, 25])
    # some instances hold the first blocks of some prompts beforehand
    held = [keys[kh[q]:kh[q] + (kh[q + 1] - kh[q]) * (i + 1) // (n_inst + 1)]
            for i in range(n_inst) for q in [int(g.integers(0, R))]]
    ioff = torch.tensor(np.concatenate([[0], np.cumsum([len(x) for x in held])]), dtype=torch.int64).cuda()
    for r in (a, b):
        r.set_normalizer(mean, std)
        r.snapshot(n_inst, state, torch.cat(held + [keys[:0]]), ioff)
        r.set_params(params)
        r.publish()
    col = d_inst - 1
    out = a.route_sequential(tok, toff, req, n_inst, queue_col=col)
    assert a.sync() == L.LS_OK
    choice = out["choice"].cpu().numpy()
    rows = state.clone()
    tol = 1e-5 if dtype == "f32" else 2e-2
    for q in range(R):
        one = b.route(tok[off[q]:], torch.tensor([0, off[q + 1] - off[q]]).cuda(), req[q:q + 1].contiguous(), n_inst)
        assert torch.equal(one["hits"][0], out["hits"][q]), q
        want, got = one["scores"][0].double(), out["scores"][q].double()
        assert float((got - want).abs().max()) <= tol * float(want.abs().clamp(min=want.abs().mean()).max()), q
        s = out["scores"][q].cpu().numpy()
        assert choice[q] == int(np.argmin(s)) and out["best"][q].item() == s[choice[q]]
        rows[choice[q], col] += 1.0
        mine = keys[kh[q]:kh[q + 1]]
        io = torch.zeros(n_inst + 1, dtype=torch.int64)
        io[choice[q] + 1:] = len(mine)
        b.snapshot(n_inst, rows, mine, io.cuda(), mode=L.LS_INSERT)
    # the state left behind: one batch route on both contexts
    x, y = (r.route(tok, toff, req, n_inst) for r in (a, b))
    assert torch.equal(x["hits"], y["hits"]) and torch.equal(x["scores"], y["scores"])
    assert a.sync() == L.LS_OK and b.sync() == L.LS_OK
    a.close()
    b.close()
