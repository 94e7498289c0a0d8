"""Ordered calls on both sides of the batch size up to which first occurrences
are found through plain indices: position by position against the first
occurrences computed by torch."""
import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.table import Table
from test_gpu_bulk import CODE, keys_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ("set_u32", "map_u64_u64"))
@pytest.mark.parametrize("n", ((1 << 22) - 1, 1 << 22, (1 << 22) + 1))
def test_first_occurrences(name, n):
    kind = CODE[name]
    g = torch.Generator(device="cuda").manual_seed(n)
    pick = torch.randint(0, n // 3, (n,), generator=g, device="cuda")
    i = torch.arange(n, device="cuda")
    first = torch.full((n // 3,), n, device="cuda").scatter_reduce_(0, pick, i, "amin")
    leads = first[pick] == i
    k = keys_of(pick, kind)
    t = Table(kind, 1 << 23, bucket_bytes=64)
    try:
        st = t.insert_ordered(k, i if kind == L.MAP_U64_U64 else None)
        assert torch.equal(st == L.INSERTED, leads) and torch.equal(st == L.EXISTS, ~leads)
        f, v = t.find(k)
        assert bool(f.all()) and (v is None or torch.equal(v, first[pick]))
        st = t.erase_ordered(k)
        assert torch.equal(st == L.ERASED, leads) and torch.equal(st == L.NOT_FOUND, ~leads)
        assert t.size() == 0 and t.status() == L.OK
    finally:
        t.close()
