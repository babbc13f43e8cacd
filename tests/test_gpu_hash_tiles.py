"""The digest kernel at the edges of its 16 KiB tiles and 16-byte vectors, at every alignment,
and with more ranges than one launch takes, against the oracle's digest (whole numbers: equal)."""
import pytest

import paper_2604_22228_gb300 as mpt
import payload
from oracle import transfer as T

pytestmark = pytest.mark.gpu

TILE = 16384
SIZES = [1, 8, 15, 16, 17, 24, 512, 513, 2047, 2048, 2049, TILE - 16, TILE - 1, TILE, TILE + 1, TILE + 17, 2 * TILE,
         2 * TILE + 2049, 3 * TILE - 9, 40 * TILE + 5]


@pytest.mark.parametrize("offset", list(range(16)))
def test_tile_edges_at_every_alignment(offset):
    import torch
    ctx = mpt.mpt_ctx_create(0)
    host = payload.fill("u8", 0x5EED0009 + offset, SIZES[-1] + 64)
    t = torch.from_numpy(host).cuda()
    got = mpt.mpt_hash_ranges_noalloc([(t.data_ptr() + offset, n) for n in SIZES])
    want = [T.hash64(host[offset:offset + n]) for n in SIZES]
    assert got == want
    assert [mpt.mpt_hash_device(ctx, t.data_ptr() + offset, n) for n in SIZES] == want
    mpt.mpt_ctx_destroy(ctx)


@pytest.mark.parametrize("n", [1, 4, 5, 159, 160, 161, 321, 1024])
def test_many_ranges(n):
    import torch
    sizes = [0 if i % 7 == 3 else (i * 37) % 900 + (TILE * 3 if i % 50 == 0 else 0) for i in range(n)]
    host = payload.fill("u8", 0x5EED000A, sum(sizes) + 16)
    t = torch.from_numpy(host).cuda()
    offs = [sum(sizes[:i]) for i in range(n)]
    got = mpt.mpt_hash_ranges_noalloc([(t.data_ptr() + o, k) for o, k in zip(offs, sizes)])
    assert got == [T.hash64(host[o:o + k]) for o, k in zip(offs, sizes)]


def test_device_and_host_ranges_in_one_call():
    """Ranges of device and page-locked host memory in turns: one launch for every run of
    neighbours of one kind."""
    import torch
    host = payload.fill("u8", 0x5EED000B, 12 * 70000)
    pinned = torch.from_numpy(host).pin_memory()
    dev = pinned.cuda()
    kinds = [0, 0, 1, 0, 1, 1, 1, 0, 0, 0, 1, 1]
    sizes = [70000 - 13 * i if i % 5 else 0 for i in range(12)]
    at = [(70000 * i + i) for i in range(12)]
    got = mpt.mpt_hash_ranges_noalloc([((pinned if k else dev).data_ptr() + a, n) for k, a, n in zip(kinds, at, sizes)])
    assert got == [T.hash64(host[a:a + n]) for a, n in zip(at, sizes)]


def test_large_device_and_host_ranges_in_one_call():
    """Above 1 MiB a call asks where its ranges lie: launches of their own for each run of
    neighbours of one kind, those over host memory by a small grid whose CTAs take several tiles
    each, off 16-byte boundaries as well."""
    import torch
    size = 5 << 20
    host = payload.fill("u8", 0x5EED000D, 3 * size)
    pinned = torch.from_numpy(host).pin_memory()
    dev = pinned.cuda()
    ranges = [("dev", 0, 400001), ("host", 16, size), ("host", size + 5, size - 9), ("dev", size + 3, size), ("host", 7, 0),
              ("pageable", 2 * size + 1, 3 * TILE * 32 + 11), ("dev", 0, 0), ("dev", 2 * size, 100), ("host", 1, 33)]
    at = {"dev": dev.data_ptr(), "host": pinned.data_ptr(), "pageable": host.ctypes.data}
    ctx = mpt.mpt_ctx_create(0)
    if not mpt.mpt_ctx_info(ctx)["pageable_access"]:
        ranges = [r for r in ranges if r[0] != "pageable"]
    want = [T.hash64(host[o:o + n]) for _, o, n in ranges]
    assert mpt.mpt_hash_ranges_noalloc([(at[k] + o, n) for k, o, n in ranges]) == want
    assert [mpt.mpt_hash_device(ctx, at[k] + o, n) for k, o, n in ranges] == want
    mpt.mpt_ctx_destroy(ctx)
