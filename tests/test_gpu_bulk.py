"""Bulk calls (split by table part, probe part by part, join) against the range
kernels on a table of the same contents.  An explicit launch shape keeps a table
on the range kernels, whose results the other tests compare with the oracle."""
import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.table import KEY_BYTES, KEY_TORCH, VAL_BYTES, Table

pytestmark = pytest.mark.gpu

KINDS = ("set_u32", "set_u64", "map_i64_i32", "map_u64_u64")
CODE = {"set_u32": L.SET_U32, "set_u64": L.SET_U64, "map_i64_i32": L.MAP_I64_I32, "map_u64_u64": L.MAP_U64_U64}


def keys_of(idx, kind):
    """A bijective mix of idx, as key bits."""
    if kind == L.SET_U32:
        x = idx
        for _ in range(2):
            x = ((x ^ (x >> 16)) * 0x45D9F3B) & 0xFFFFFFFF
        return (x ^ (x >> 16)).to(torch.int32)
    x = idx.clone()
    for m in (-0x61C8864680B583EB, -0x40A7B892E31B1A47):
        x *= m
        x ^= (x >> 32) & 0xFFFFFFFF
    return x


def vals_of(keys, kind):
    if kind not in VAL_BYTES:
        return None
    v = keys * 3 + 1
    return v if VAL_BYTES[kind] == 8 else (v >> 7).to(torch.int32)


def off_by_one(t):
    """The same values in an array that starts one element off a 16-byte boundary."""
    if t is None:
        return None
    r = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")[1:]
    r.copy_(t)
    return r


def by_key(keys, status):
    """Statuses ordered by (key, status): what equal keys of a batch share."""
    s, o = torch.sort(status.to(torch.int64), stable=True)
    k, p = torch.sort(keys[o], stable=True)
    return k, s[p]


def same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("name", KINDS)
@pytest.mark.parametrize("bb", (32, 64, 128))
@pytest.mark.parametrize("hash_mode", (L.HASH_MIX64, L.HASH_TESCHNER))
def test_bulk_equals_range(name, bb, hash_mode):
    kind = CODE[name]
    if hash_mode == L.HASH_TESCHNER and kind != L.MAP_I64_I32:
        pytest.skip("the spatial hash is for packed block keys")
    slot = KEY_BYTES[kind] + VAL_BYTES.get(kind, 0)
    slots = (800 << 20) // (16 if kind in VAL_BYTES else slot) - 5      # 800 MB of buckets, the last one padded
    lines = (800 << 20) // 128
    a, b = Table(kind, slots, bucket_bytes=bb, hash_mode=hash_mode), Table(kind, slots, bucket_bytes=bb,
                                                                          hash_mode=hash_mode)
    for op in (0, 1, 2):
        b.set_launch(op, keys_per_group=4, block=64)
    reserved = torch.tensor([-1, -2, -3], dtype=KEY_TORCH[KEY_BYTES[kind]], device="cuda")
    try:
        g = torch.Generator(device="cuda").manual_seed(bb + kind)
        start = torch.cuda.mem_get_info()[0]
        for n in (lines // 2 + 1, 2 * lines + 4097):
            idx = torch.arange(n, dtype=torch.int64, device="cuda")
            idx[::20] = torch.randint(0, n, (idx[::20].numel(),), generator=g, device="cuda")   # equal keys in a batch
            k = torch.cat([keys_of(idx, kind), reserved])
            v = vals_of(k, kind)
            k, v = off_by_one(k), off_by_one(v)
            assert same(by_key(k, a.insert(k, v)), by_key(k, b.insert(k, v)))
            assert a.size() == b.size()
        assert torch.cuda.mem_get_info()[0] < start - (8 << 20), "no bulk call has taken scratch"
        q = keys_of(torch.randint(0, 3 * n, (2 * lines + 1,), generator=g, device="cuda"), kind)
        q = torch.cat([q, reserved])
        fa, va = a.find(q)
        fb, vb = b.find(q)
        assert torch.equal(fa, fb) and 0 < int(fa.sum()) < q.numel()
        assert va is None or torch.equal(va, vb)
        assert torch.equal(a.find(q, vals_out=False)[0], fb)
        e = torch.cat([q[:lines + 11], q[:50], reserved])
        assert same(by_key(e, a.erase(e)), by_key(e, b.erase(e)))
        assert a.size() == b.size()
        # tombstones are used again; no status asked for
        a.insert(e, vals_of(e, kind), status=False)
        b.insert(e, vals_of(e, kind), status=False)
        assert a.size() == b.size()
        fa, va = a.find(q)
        fb, vb = b.find(q)
        assert torch.equal(fa, fb) and (va is None or torch.equal(va, vb))
        if kind in VAL_BYTES:                            # values may replace the keys they were looked up by
            if VAL_BYTES[kind] == KEY_BYTES[kind]:
                r = q.clone()
                a.find(r, vals_out=r)
                assert torch.equal(r, vb)
        assert a.status() == L.OK and b.status() == L.OK
    finally:
        a.close()
        b.close()


def test_captured_call_keeps_the_range_kernels():
    """A capturing stream takes no scratch; the captured call replays."""
    t = Table(L.MAP_U64_U64, (800 << 20) // 16, bucket_bytes=64)
    try:
        n = 2 * (800 << 20) // 128
        k = keys_of(torch.arange(n, device="cuda"), L.MAP_U64_U64)
        t.insert(k, vals_of(k, L.MAP_U64_U64), status=False)
        f, v = torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty_like(k)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            t.find(k, found=f, vals_out=v)
        f.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert bool(f.all()) and torch.equal(v, vals_of(k, L.MAP_U64_U64))
    finally:
        t.close()


def test_bulk_calls_on_two_streams():
    """Lookups of one table and inserts of another at once, each with a scratch of its own."""
    slots = (800 << 20) // 16
    t, u = Table(L.MAP_U64_U64, slots, bucket_bytes=64), Table(L.MAP_U64_U64, slots, bucket_bytes=64)
    n = 2 * (800 << 20) // 128
    k = keys_of(torch.arange(n, device="cuda"), L.MAP_U64_U64)
    v = vals_of(k, L.MAP_U64_U64)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    try:
        t.insert(k, v, status=False)
        st = torch.empty(n, dtype=torch.uint8, device="cuda")
        outs = [(torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty_like(v)) for _ in range(3)]
        torch.cuda.synchronize()
        u.insert(k, v, status=st, stream=s1)
        for f, w in outs:
            t.find(k, found=f, vals_out=w, stream=s2)
        torch.cuda.synchronize()
        assert not bool(st.any()) and u.size() == n
        for f, w in outs:
            assert bool(f.all()) and torch.equal(w, v)
    finally:
        t.close()
        u.close()
