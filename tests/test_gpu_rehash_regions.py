"""Rehash region by region on tables just above the size from which it is used, at
loads below and around its limit, and with keys that crowd the regions' ends so that
more of them leave their region than its list holds (the runs take over)."""
import numpy as np
import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.table import KEY_BYTES, VAL_BYTES, Table, to_device
from test_gpu_bulk import CODE, KINDS, keys_of, vals_of
from test_gpu_mixed_long_run import mix_inverse

pytestmark = pytest.mark.gpu


def contents_kept(t, k, v, new):
    live = t.size()
    t.rehash(new)
    s = t.stats()
    assert (s["live"], s["used"], s["capacity"], s["error_bits"]) == (live, live, new, 0)
    f, w = t.find(k)
    assert bool(f.all()) and (w is None or torch.equal(w, v))
    dk, _ = t.dump()
    assert torch.equal(torch.sort(dk)[0], torch.sort(k)[0])


@pytest.mark.parametrize("name", KINDS)
@pytest.mark.parametrize("bb", (32, 64, 128))
@pytest.mark.parametrize("load", (0.4, 0.75, 0.9))
def test_rehash_above_the_least_size(name, bb, load):
    kind = CODE[name]
    slot = 16 if kind in VAL_BYTES else KEY_BYTES[kind]
    least = (max(64, 256 * slot // bb) if kind in VAL_BYTES else max(16, 192 * slot // bb)) << 20
    slots = least // slot + 12345
    n = int(slots * load)
    t = Table(kind, slots, bucket_bytes=bb, seed=5)
    try:
        k = keys_of(torch.arange(n, device="cuda"), kind)
        v = vals_of(k, kind)
        t.insert(k, v, status=False)
        t.erase(k[:n // 4].contiguous(), status=False)
        kept, kept_v = k[n // 4:], (None if v is None else v[n // 4:])
        for new in (slots, slots + slots // 3, slots):
            contents_kept(t, kept, kept_v, new)
        assert bool((t.find(k[:n // 4], vals_out=False)[0] == 0).all())
    finally:
        t.close()


def test_more_keys_leave_their_regions_than_the_list_holds():
    """300 keys from the last bucket of every 32 KB region of a 128 MB map."""
    lg, per = 21, 300
    t = Table(L.MAP_U64_U64, 4 << lg, bucket_bytes=64)
    try:
        last = np.arange(511, 1 << lg, 512, dtype=np.uint64)
        k = mix_inverse((last[:, None] << np.uint64(64 - lg)) + np.arange(1, per + 1, dtype=np.uint64)[None, :])
        k = to_device(k.reshape(-1))
        v = vals_of(k, L.MAP_U64_U64)
        assert not bool(t.insert(k, v).any())
        contents_kept(t, k, v, 4 << lg)
    finally:
        t.close()
