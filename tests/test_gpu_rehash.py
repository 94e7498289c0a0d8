"""Rehash region by region (tables of 16 MB and more) against the contents from
before it: the same size, other sizes up and down, load factors at which keys
leave their region, padding, tombstones, and the keys with patterns of their
own."""
import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.table import KEY_BYTES, KEY_TORCH, VAL_BYTES, Table
from test_gpu_bulk import CODE, KINDS, keys_of, vals_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", KINDS)
@pytest.mark.parametrize("bb", (32, 64, 128))
@pytest.mark.parametrize("load", (0.5, 0.999))
def test_rehash_keeps_the_contents(name, bb, load):
    kind = CODE[name]
    per = 16 if kind in VAL_BYTES else KEY_BYTES[kind]
    slots = (20 << 20) // per - 3
    t = Table(kind, slots, bucket_bytes=bb, seed=7)
    reserved = torch.tensor([-1, -2, -3], dtype=KEY_TORCH[KEY_BYTES[kind]], device="cuda")
    try:
        n = int(slots * load) - 1
        k = torch.cat([keys_of(torch.arange(n, device="cuda"), kind), reserved])
        v = vals_of(k, kind)
        t.insert(k, v, status=False)
        gone = k[:n // 3].clone()
        t.erase(gone)
        kept, kept_v = k[n // 3:], (None if v is None else v[n // 3:])
        live = t.size()
        assert live == kept.numel()
        for new in (slots, slots * 2 + 1, (live + slots) // 2, live - 2):   # the last: every slot taken
            t.rehash(new)
            s = t.stats()
            assert s["live"] == live and s["used"] == live - 2 and s["capacity"] == new and not s["error_bits"]
            f, w = t.find(kept)
            assert bool(f.all()) and (w is None or torch.equal(w, kept_v))
            assert not bool(t.find(gone[:100000], vals_out=False)[0].any())
            dk, _ = t.dump()
            assert torch.equal(torch.sort(dk)[0], torch.sort(kept)[0])
        st = t.insert(gone[:1000], None if v is None else v[:1000])
        assert bool((st == L.OVERFLOW).all())
        t.rehash(slots)
        st = t.insert(gone[:1000], None if v is None else v[:1000])
        assert not bool(st.any()) and t.size() == live + 1000
        assert not bool((t.insert(kept, kept_v) != L.EXISTS).any())
    finally:
        t.close()
