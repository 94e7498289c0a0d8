"""Inserts that lose claim after claim to other keys: on a table without an EMPTY
slot a key reads every bucket before each claim, and all keys of a batch make for
the first free slots they have passed.  As long as slots are free every new key is
stored, however many steps its run has taken."""
import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.batch import Batch, Item
from paper_1908_05936_gb300.table import KEY_BYTES, VAL_BYTES, Table
from test_gpu_bulk import CODE, KINDS, keys_of, vals_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", KINDS)
@pytest.mark.parametrize("form", ("range", "ordered", "batched 128", "batched 256"))
def test_tombstones_only(name, form):
    """2^15 buckets filled to capacity, half of the keys erased, as many others
    inserted: in runs of 32 keys (what so small a call takes), in the batched form's
    runs of 128 and 256, and through the ordered call."""
    kind = CODE[name]
    slots = (32 // (16 if kind in VAL_BYTES else KEY_BYTES[kind])) << 15
    n = slots // 2
    t = Table(kind, slots)
    try:
        k = keys_of(torch.arange(slots + n, device="cuda"), kind)
        v = vals_of(k, kind)
        old, new, new_v = k[:slots], k[slots:], (None if v is None else v[slots:])
        assert not bool(t.insert(old, None if v is None else v[:slots]).any())
        gone = old[::2].contiguous()
        assert bool((t.erase(gone) == L.ERASED).all())
        if form == "range":
            st = t.insert(new, new_v)
        elif form == "ordered":
            st = t.insert_ordered(new, new_v)
        else:
            st = torch.empty(n, dtype=torch.uint8, device="cuda")
            b = Batch([Item(t, L.OP_INSERT, new, new_v, st)], keys_per_group=8 if form == "batched 256" else 4,
                      tile=int(form[-3:]), use_graph=False)
            b.launch()
            torch.cuda.synchronize()
            b.close()
        assert int((st != L.INSERTED).sum()) == 0
        assert t.status() == L.OK
        s = t.stats()
        assert s["live"] == slots and s["used"] == slots
        dk, dv = t.dump()
        order = torch.argsort(dk)
        want = torch.cat([old[1::2], new])
        worder = torch.argsort(want)
        assert torch.equal(dk[order], want[worder])
        assert dv is None or torch.equal(dv[order], vals_of(want, kind)[worder])
        assert bool((t.insert(gone[:33], None if v is None else vals_of(gone[:33], kind)) == L.OVERFLOW).all())
    finally:
        t.close()
