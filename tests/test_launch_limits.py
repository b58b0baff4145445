"""Shared-memory limits of the kernels are a property of the process, not of a
context: every context allows the most a CTA can have (common.cuh, allow_smem)
before its first launch, and no call sets a limit of its own shape, which
another thread's context of a larger shape would trip over at its next launch."""
import glob
import os
import re
import threading

import pytest

from paper_2606_00946_gb300 import build as B


def test_limits_are_set_in_one_place():
    found = {}
    for path in sorted(glob.glob(os.path.join(B.CSRC, "*.cu*"))):
        n = len(re.findall(r"\bcudaFuncSetAttribute\s*\(", re.sub(r"//[^\n]*", "", open(path).read())))
        if n:
            found[os.path.basename(path)] = n
    assert found == {"common.cuh": 1}


@pytest.mark.gpu
def test_threads_of_different_shapes_train_and_route():
    """Two threads, each with a context of its own and of another size: fp32
    steps, admission rounds and sequential routes all succeed."""
    import torch

    from paper_2606_00946_gb300 import harness as H
    from paper_2606_00946_gb300 import lodestar as L

    B.build()

    def context(hidden, dtype, n_inst, seed):
        w = [16, *hidden, 1]
        r = H.Router(w, 10, 0, dtype, max_instances=n_inst, max_requests=2, max_keys_per_instance=64,
                     ring_capacity=64, replay_capacity=256, pending_capacity=256, max_train_batch=512,
                     max_batch_tokens=64)
        g = torch.Generator(device="cuda").manual_seed(seed)
        r.set_normalizer(torch.zeros(16, device="cuda"), torch.ones(16, device="cuda"))
        r.set_params(torch.randn(r.n_params, generator=g, device="cuda") * 0.1)
        r.snapshot(n_inst, torch.randn(n_inst, 10, generator=g, device="cuda"))
        r.publish()
        for _ in range(8):  # (a log call holds at most the ring)
            r.log(torch.randn(64, 16, generator=g, device="cuda"), torch.randn(64, generator=g, device="cuda"))
        return r

    errors = []

    def work(r, n_inst, stop):
        try:
            tok = torch.arange(32, device="cuda", dtype=torch.int32)
            off = torch.tensor([0, 16, 32], device="cuda")
            req = torch.zeros(2, 0, device="cuda")
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for k in range(300):
                    if stop.is_set():
                        break
                    r.train(512 if k & 1 else 100, lr=1e-4)
                    if k % 8 == 0:
                        r.route_sequential(tok, off, req, n_inst)
                        r.replay_admit()
                stream.synchronize()
        except Exception as e:  # noqa: BLE001 -- reported by the test below
            errors.append(e)
            stop.set()

    for pair in ([((64, 64), "f32", 4), ((16,), "f32", 1)], [((128, 256), "bf16", 8), ((64,), "bf16", 2)]):
        rs = [context(h, dt, n, k) for k, (h, dt, n) in enumerate(pair)]
        stop = threading.Event()
        ts = [threading.Thread(target=work, args=(r, p[2], stop)) for r, p in zip(rs, pair)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not errors, errors
        for r in rs:
            assert r.sync() == L.LS_OK
            r.close()
