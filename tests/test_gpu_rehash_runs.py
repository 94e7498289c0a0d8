"""Rehash of small tables and of spatial-hash ones, whose stored keys become runs of
the insert loop: table sizes at the edges of a warp's 256 and a block's 2048 slots,
empty, sparse and full, grown, shrunk to what is stored and purged of tombstones."""
import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.table import Table
from test_gpu_bulk import CODE, KINDS, keys_of, vals_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,mode", [(k, L.HASH_MIX64) for k in KINDS] + [("map_i64_i32", L.HASH_TESCHNER),
                                                                             ("map_i64_i32", L.HASH_TESCHNER_SHORT3)])
@pytest.mark.parametrize("bb", (32, 128))
@pytest.mark.parametrize("slots", (1, 255, 256, 257, 2047, 2049, 70001))
@pytest.mark.parametrize("share", (0.0, 0.03, 0.6, 1.0))
def test_rehash_of_runs(name, mode, bb, slots, share):
    kind = CODE[name]
    n = int(slots * share)
    t = Table(kind, slots, bucket_bytes=bb, hash_mode=mode)
    try:
        k = keys_of(torch.arange(1, n + 1, device="cuda"), kind)
        v = vals_of(k, kind)
        assert not bool(t.insert(k, v).any())
        t.erase(k[::3].contiguous())
        gone = torch.zeros(n, dtype=torch.bool, device="cuda")
        gone[::3] = True
        live = n - int(gone.sum())
        for new in (slots, 2 * slots + 1, max(live, 1), slots):
            t.rehash(new)
            s = t.stats()
            assert (s["live"], s["used"], s["capacity"], s["error_bits"]) == (live, live, new, 0)
            f, w = t.find(k)
            assert torch.equal(f == 0, gone) and (w is None or torch.equal(w[~gone], v[~gone]))
    finally:
        t.close()
