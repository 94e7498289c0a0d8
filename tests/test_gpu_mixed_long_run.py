"""A mixed batch whose inserts lose swaps late in a long run: what ends an insert is
the swaps that it loses and the claims that it waits for, not the steps of its run."""
import numpy as np
import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.table import Table, to_device
from test_gpu_bulk import CODE, vals_of

pytestmark = pytest.mark.gpu


def mix_inverse(h):
    """The key whose 64-bit mix (MurmurHash3's finaliser) is h."""
    m1, m2 = pow(0xFF51AFD7ED558CCD, -1, 1 << 64), pow(0xC4CEB9FE1A85EC53, -1, 1 << 64)
    h = h ^ (h >> np.uint64(33))
    h = h * np.uint64(m2)
    h = h ^ (h >> np.uint64(33))
    h = h * np.uint64(m1)
    return h ^ (h >> np.uint64(33))


def keys_at(bucket, which, log2_nb):
    """Keys of 2^log2_nb buckets whose first bucket is `bucket`, one per entry of `which`."""
    return mix_inverse((np.uint64(bucket) << np.uint64(64 - log2_nb)) + which.astype(np.uint64) + np.uint64(1))


@pytest.mark.parametrize("name", ("set_u64", "map_u64_u64"))
def test_inserts_at_the_end_of_a_long_run(name):
    """One warp's run of 128 operations on a table whose only EMPTY slots are in
    one bucket: lookups of absent keys from the bucket after it, then as many
    inserts as there are slots, from the same bucket and for the same slot first.
    They lose swaps to each other after more steps than the table has buckets
    several times over, and are all stored."""
    kind, lg = CODE[name], 20
    nb, spb = 1 << lg, 2 if name == "map_u64_u64" else 4
    e = 12345
    t = Table(kind, nb * spb)
    try:
        buckets = np.delete(np.arange(nb, dtype=np.uint64), e)
        fill = mix_inverse((buckets[:, None] << np.uint64(64 - lg)) + np.arange(1, spb + 1, dtype=np.uint64)[None, :])
        fill = to_device(fill.reshape(-1))
        assert not bool(t.insert(fill, vals_of(fill, kind)).any())
        far = keys_at(e + 1, np.arange(100, 1100), lg)
        with np.errstate(over="ignore"):
            h = far ^ np.uint64(0x9E3779B97F4A7C15)
            h = (h ^ (h >> np.uint64(33))) * np.uint64(0xFF51AFD7ED558CCD)
            h = (h ^ (h >> np.uint64(33))) * np.uint64(0xC4CEB9FE1A85EC53)
            h = h ^ (h >> np.uint64(33))
        first = far[(h & np.uint64(spb - 1)) == 0][:spb]       # keys that start at the same slot of a bucket
        rest = np.setdiff1d(far, first)[:128 - spb]
        k = to_device(np.concatenate([rest, first]))
        ops = torch.tensor([1] * (128 - spb) + [0] * spb, dtype=torch.uint8, device="cuda")
        # as many operations as make the grid's runs 128 long; the others look up stored keys
        more = 4096 * 128 - 128
        k = torch.cat([k, fill[:more]])
        ops = torch.cat([ops, torch.ones(more, dtype=torch.uint8, device="cuda")])
        v = vals_of(k, kind)
        st, _ = t.apply_mixed(ops, k, v)
        assert not bool(st[:128 - spb].any()) and bool((st[128:] == 1).all())
        assert int((st[128 - spb:128] != L.INSERTED).sum()) == 0
        assert t.status() == L.OK and t.size() == nb * spb
        f, w = t.find(k[128 - spb:128])
        assert bool(f.all()) and (w is None or torch.equal(w, v[128 - spb:128]))
    finally:
        t.close()
