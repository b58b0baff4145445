"""Device memory that a replay pool's capacity costs: the records, the images
their embeddings are formed on and the distances' partial minima, and nothing
that the round does not read."""
import pytest
import torch

from paper_2606_00946_gb300 import build as B
from paper_2606_00946_gb300 import harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


@pytest.mark.parametrize("hidden", [(256,), (128, 256)])
def test_bytes_a_record(hidden):
    d, n = 64, 200_000
    widths = [d, *hidden, 1]

    def used(cap):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        r = H.Router(widths, 34, 24, "bf16", max_instances=4, max_requests=4, max_keys_per_instance=64,
                     ring_capacity=1024, pending_capacity=1024, replay_capacity=cap, max_train_batch=256,
                     max_batch_tokens=64)
        after = torch.cuda.mem_get_info()[0]
        r.close()
        return before - after

    used(1024)  # (the library's kernels and pools are loaded)
    per = (used(2 * n) - used(n)) / n
    # features and target; bf16 embedding row; two bf16 activation rows and a target; 256 partial minima; norm,
    # distance, rank and its inverse
    want = 4 * (d + 1) + 2 * hidden[-1] + 2 * 2 * max(d, *hidden) + 4 + 4 * 256 + 4 * 4
    # (the allocator's granularity of 2 MB for each of a dozen buffers)
    assert abs(per - want) <= 12 * 2 * 2 ** 20 / n, (per, want)
