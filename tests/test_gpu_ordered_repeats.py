"""Ordered calls on a batch of one key alone cost no more than on as many distinct
keys (with a swap on the one entry by every occurrence they cost ten times that).
The results of such batches are compared with the oracle elsewhere."""
import pytest
import torch

from paper_1908_05936_gb300.table import Table
from test_gpu_bulk import CODE, KINDS, keys_of, vals_of

pytestmark = pytest.mark.gpu


def call_us(fn, after, reps=5):
    best = float("inf")
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
        after()
    return best


@pytest.mark.parametrize("name", KINDS)
def test_one_key_costs_no_more_than_distinct_keys(name):
    kind, n = CODE[name], 1 << 22
    t = Table(kind, 2 * n)
    try:
        scratch = torch.empty(int(t.lib.hc_ordered_scratch_bytes(n)) + 256, dtype=torch.uint8, device="cuda")
        st = torch.empty(n, dtype=torch.uint8, device="cuda")
        us = []
        for idx in (torch.arange(n, device="cuda"), torch.full((n,), 77, device="cuda")):
            k = keys_of(idx, kind)
            v = vals_of(k, kind)
            us.append(call_us(lambda: t.insert_ordered(k, v, status=st, scratch=scratch), t.clear))
            us.append(call_us(lambda: t.erase_ordered(k, status=st, scratch=scratch), lambda: None))
        assert us[2] < us[0] and us[3] < us[1], us
    finally:
        t.close()
