"""Bulk calls on keys that crowd into few table parts, so that a warp's part takes many
passes and runs are cut in the middle, and on more keys than one piece holds, against
the range kernels."""
import numpy as np
import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.table import Table, to_device
from test_gpu_bulk import CODE, by_key, keys_of, same, vals_of
from test_gpu_mixed_long_run import mix_inverse

pytestmark = pytest.mark.gpu

BYTES = 800 << 20


def pair(kind, bb):
    slots = BYTES // (16 if kind in (L.MAP_I64_I32, L.MAP_U64_U64) else 4 if kind == L.SET_U32 else 8)
    a, b = Table(kind, slots, bucket_bytes=bb), Table(kind, slots, bucket_bytes=bb)
    for op in (0, 1, 2):
        b.set_launch(op, keys_per_group=4, block=64)
    return a, b


def compare(a, b, k, kind):
    v = vals_of(k, kind)
    assert same(by_key(k, a.insert(k, v)), by_key(k, b.insert(k, v)))
    q = torch.cat([k, k + 1])
    fa, va = a.find(q)
    fb, vb = b.find(q)
    assert torch.equal(fa, fb) and (va is None or torch.equal(va, vb))
    assert same(by_key(k, a.erase(k)), by_key(k, b.erase(k)))
    assert a.size() == b.size() and a.status() == L.OK


@pytest.mark.parametrize("name", ("set_u32", "map_i64_i32", "map_u64_u64"))
@pytest.mark.parametrize("bb", (32, 128))
@pytest.mark.parametrize("crowd", (0.3, 1.0))
def test_one_key_many_times(name, bb, crowd):
    kind, n = CODE[name], 2 * BYTES // 128 + 4097
    a, b = pair(kind, bb)
    try:
        g = torch.Generator(device="cuda").manual_seed(bb)
        idx = torch.randint(0, n, (n,), generator=g, device="cuda")
        idx[torch.rand(n, generator=g, device="cuda") < crowd] = 77
        compare(a, b, keys_of(idx, kind), kind)
    finally:
        a.close(), b.close()


@pytest.mark.parametrize("name", ("set_u64", "map_u64_u64"))
def test_keys_of_one_part(name):
    """20,000 keys from the first thousandth of the table."""
    kind, n = CODE[name], 2 * BYTES // 128 + 1
    a, b = pair(kind, 64)
    try:
        h = np.random.default_rng(3).integers(0, (1 << 64) // 1000, 20_000, dtype=np.uint64)
        few = to_device(mix_inverse(h))
        g = torch.Generator(device="cuda").manual_seed(5)
        compare(a, b, few[torch.randint(0, few.numel(), (n,), generator=g, device="cuda")].contiguous(), kind)
    finally:
        a.close(), b.close()


def test_more_keys_than_a_piece():
    kind, n = L.MAP_U64_U64, (1 << 26) + 4099
    a, b = pair(kind, 64)
    try:
        g = torch.Generator(device="cuda").manual_seed(9)
        compare(a, b, keys_of(torch.randint(0, 1 << 25, (n,), generator=g, device="cuda"), kind), kind)
    finally:
        a.close(), b.close()
