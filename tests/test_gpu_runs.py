"""The warp-run kernels where their probe loops end: tables without an EMPTY
slot, probes that come round the whole table, and batches at the edges of a
step (32 keys) and of a run."""
import numpy as np
import pytest

from gpu_pair import Pair, random_keys, value_for
from oracle import oracle as O

pytestmark = pytest.mark.gpu

KINDS = (O.SET_U32, O.SET_U64, O.MAP_I64_I32, O.MAP_U64_U64)
SPB = {O.SET_U32: lambda bb: bb // 4, O.SET_U64: lambda bb: bb // 8, O.MAP_I64_I32: lambda bb: bb // 16,
       O.MAP_U64_U64: lambda bb: bb // 16}


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("bb", (32, 64, 128))
@pytest.mark.parametrize("nb", (1, 2, 31, 32, 33, 65))
@pytest.mark.parametrize("pad", (0, 1))
def test_full_table_and_tombstones_only(kind, bb, nb, pad):
    """32 buckets and more share the end of a run among several lanes per key;
    fewer do not.  A full table answers absent keys after reading every bucket
    once, refuses inserts, and takes them again once its slots are tombstones;
    `pad` leaves the last bucket's last slot outside the capacity."""
    slots = nb * SPB[kind](bb) - pad
    if slots < 1:
        pytest.skip("no slot")
    rng = np.random.default_rng(1000 * nb + 10 * bb + kind)
    keys = np.unique(random_keys(kind, 3 * slots + 40, rng))
    rng.shuffle(keys)
    stored, other = keys[:slots], keys[slots:2 * slots + 20]
    p = Pair(kind, slots, bucket_bytes=bb)
    try:
        p.insert(stored, value_for(kind, stored))
        p.find(np.concatenate([stored, other]))
        p.insert(other[:7], value_for(kind, other[:7]))                 # every one overflows
        p.insert(np.concatenate([stored, other]), value_for(kind, np.concatenate([stored, other]), salt=1))
        p.check()
        p.erase(np.concatenate([other, stored]))
        p.find(np.concatenate([stored, other]))                         # tombstones only
        p.erase(other)
        p.insert(other[:slots], value_for(kind, other[:slots]))         # reuses them
        p.check()
        p.erase(other[:slots:2])
        p.insert(np.concatenate([other[:slots]] * 2), value_for(kind, np.concatenate([other[:slots]] * 2), salt=2))
        p.check()
    finally:
        p.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("bb", (32, 128))
@pytest.mark.parametrize("kpt", (4, 8))
def test_batches_at_the_edges_of_steps_and_runs(kind, bb, kpt):
    """Batch sizes around a step and a run, with arrays that start one element
    off a 16-byte boundary, at a load factor with long probe sequences."""
    import torch

    from paper_1908_05936_gb300.table import to_device, to_numpy
    rng = np.random.default_rng(bb + kpt + kind)
    p = Pair(kind, 9000, bucket_bytes=bb)
    for op in (0, 1, 2):
        p.g.set_launch(op, keys_per_group=kpt, block=128)
    keys = np.unique(random_keys(kind, 12000, rng))
    rng.shuffle(keys)
    try:
        at = 0
        for n in (1, 31, 32, 33, 32 * kpt - 1, 32 * kpt, 32 * kpt + 1, 4 * 32 * kpt + 1, 6000):
            k = keys[at:at + n]
            at += n
            p.insert(k, value_for(kind, k))
            p.find(np.concatenate([k, keys[-n:]]))
            dev = torch.empty(n + 1, dtype=to_device(k).dtype, device="cuda")[1:]
            dev.copy_(to_device(k))
            f, v = p.g.find(dev)
            of, ov = p.o.find(k)
            assert np.array_equal(to_numpy(f, np.uint8), of)
            if p.is_map:
                assert np.array_equal(to_numpy(v, O.VAL_DTYPE[kind]), ov)
            p.erase(k[::4])
        p.check()
    finally:
        p.close()


@pytest.mark.parametrize("kind", (O.MAP_I64_I32, O.MAP_U64_U64))
@pytest.mark.parametrize("slots", ((1 << 24) - 1, (1 << 24) + 1))
def test_whole_bucket_lookups(kind, slots):
    """Maps with 32-byte buckets just below and from 256 MB on, where a lookup
    reads keys and values together, against the lookup of one key per lane
    group: hits in either slot, misses, tombstones and reserved keys."""
    import torch

    from paper_1908_05936_gb300.table import VAL_BYTES, Table
    width = torch.int64 if VAL_BYTES[kind] == 8 else torch.int32
    g = torch.Generator(device="cuda").manual_seed(kind)
    keys = torch.randint(-(1 << 62), 1 << 62, (1 << 23,), generator=g, device="cuda")
    keys[:3] = torch.tensor([-1, -2, -3], device="cuda")
    vals = (keys >> 20).to(width)
    t = Table(kind, slots, bucket_bytes=32)
    try:
        t.insert(keys, vals)
        t.erase(keys[5::7].contiguous())
        q = torch.cat([keys[:200001], keys[:200001] + 1])
        t.set_launch(1, keys_per_group=1)
        want = [t.find(q[:n]) for n in (1, 33, 4097, q.numel())]
        t.set_launch(1, keys_per_group=8)
        for (f, v), n in zip(want, (1, 33, 4097, q.numel())):
            gf, gv = t.find(q[:n])
            assert torch.equal(gf, f) and torch.equal(gv, v)
            assert torch.equal(t.find(q[:n], vals_out=False)[0], f)
        assert 0 < int(want[-1][0].sum()) < q.numel()
    finally:
        t.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", (33, 4097, (1 << 21) - 1, 1 << 21))
def test_page_locked_arrays(kind, n):
    """Calls on page-locked host arrays, on both sides of the size where their
    runs get longer, against the same calls on device arrays."""
    import torch

    from paper_1908_05936_gb300.table import KEY_BYTES, KEY_NUMPY, KEY_TORCH, VAL_BYTES, VAL_NUMPY, Table
    kb, vb = KEY_BYTES[kind], VAL_BYTES.get(kind, 0)
    keys = torch.randperm(2 * n, generator=torch.Generator().manual_seed(n), dtype=torch.int64)
    keys = (keys * 40503 % (1 << 32)).to(KEY_TORCH[kb])
    vals = (keys.to(torch.int64) * 3 + 1).to(KEY_TORCH[vb]) if vb else None

    def pinned(t, dtype):
        return t.clone().pin_memory().numpy().view(dtype)

    def room(dtype):
        return torch.zeros(2 * n * np.dtype(dtype).itemsize, dtype=torch.uint8).pin_memory().numpy().view(dtype)

    def same(t, a):
        return np.array_equal(t.cpu().numpy(), a.view(t.cpu().numpy().dtype)[:t.numel()])

    a, b = Table(kind, 3 * n, bucket_bytes=64), Table(kind, 3 * n, bucket_bytes=64)
    try:
        k, hk, st = keys.cuda(), pinned(keys, KEY_NUMPY[kind]), room(np.uint8)
        dv, hv = (vals.cuda(), pinned(vals, VAL_NUMPY[kind])) if vb else (None, None)
        b.insert_host(hk[:n], hv[:n] if vb else None, st)
        assert same(a.insert(k[:n], dv[:n] if vb else None), st)
        hvo = room(VAL_NUMPY[kind]) if vb else None
        b.find_host(hk, st, hvo)
        f, v = a.find(k)
        assert same(f, st) and (not vb or same(v, hvo))
        b.erase_host(hk[n // 2:], st)
        assert same(a.erase(k[n // 2:]), st)
        assert a.size() == b.size() == n // 2
    finally:
        a.close(), b.close()
