"""The vector copy kernels around their tiles (16, 32 and 64 KiB), 32-byte units and 128-byte
lines, with source and destination agreeing modulo 32, modulo 16 or at no boundary, on the device
and over the host link: bytes equal the oracle's copy and the guard bytes stay."""
import numpy as np
import pytest

import paper_2604_22228_gb300 as mpt
from gpu_util import Buf, seeded
from oracle import transfer as T

pytestmark = pytest.mark.gpu
KiB = 1024
SIZES = [1, 31, 32, 33, 63, 64, 95, 96, 127, 128, 129, 4096 - 33, 16 * KiB - 1, 16 * KiB, 16 * KiB + 31, 32 * KiB + 97,
         64 * KiB - 32, 64 * KiB + 64, 200 * KiB + 5]
# around the sizes at which a launch on 152 SMs takes larger tiles, and small grids that take them early
EDGES = [608 * 16 * KiB - 1, 608 * 16 * KiB + 1, 304 * 64 * KiB - 32, 304 * 64 * KiB + 33, 1064 * 32 * KiB - 64, 1064 * 32 * KiB + 3]
OFFSETS = [(0, 0), (32, 32), (96, 32), (16, 16), (0, 16), (16, 0), (48, 112), (1, 0), (0, 1), (3, 11), (4, 8), (8, 0), (20, 4),
           (31, 31), (127, 64), (5, 28)]


@pytest.fixture(scope="module")
def ctx():
    import torch
    torch.cuda.init()
    c = mpt.mpt_ctx_create(0)
    yield c
    st, site = mpt.mpt_ctx_status(c)
    mpt.mpt_ctx_destroy(c)
    assert st == mpt.MPT_OK, (st, site)


def _check(ctx, n, so, do, where, variant, ctas):
    src, dst = Buf(n, where[0], so), Buf(n, where[1], do)
    data = seeded("u8", 0xC0FFEE + n + 7 * so + do, n)
    src.fill(data)
    mpt.mpt_sm_copy(ctx, dst.ptr, src.ptr, n, variant, ctas)
    assert np.array_equal(dst.numpy(), T.copy(data)), (n, so, do, where, variant, ctas)
    assert dst.guards_intact(), (n, so, do, where, variant, ctas)


@pytest.mark.parametrize("offsets", OFFSETS, ids=lambda o: f"{o[0]}_{o[1]}")
@pytest.mark.parametrize("where", [("dev", "dev"), ("host", "dev"), ("dev", "host")], ids=["d2d", "h2d", "d2h"])
def test_unit_line_and_tile_edges(ctx, where, offsets):
    for n in SIZES:
        for variant, ctas in ((mpt.MPT_SM_VEC128, 0), (mpt.MPT_SM_VEC128, 1), (mpt.MPT_SM_TILE8K, 3)):
            _check(ctx, n, *offsets, where, variant, ctas)


@pytest.mark.parametrize("shift", list(range(32)))
def test_every_shift(ctx, shift):
    for n in (200 * KiB + 77, 3 * 1024 * KiB + 1):
        _check(ctx, n, shift, 0, ("dev", "dev"), mpt.MPT_SM_VEC128, 0)
        _check(ctx, n, 0, shift, ("dev", "dev"), mpt.MPT_SM_TILE8K, 0)


@pytest.mark.parametrize("n", EDGES)
@pytest.mark.parametrize("offsets", [(0, 0), (0, 16), (9, 2)], ids=lambda o: f"{o[0]}_{o[1]}")
def test_tile_size_rule(ctx, n, offsets):
    for ctas in (0, 100, 608):
        _check(ctx, n, *offsets, ("dev", "dev"), mpt.MPT_SM_VEC128, ctas)


@pytest.mark.parametrize("offsets", [(0, 0), (0, 16), (3, 12)], ids=lambda o: f"{o[0]}_{o[1]}")
def test_many_ranges_in_one_launch(ctx, offsets):
    """Interleaved chunks: the kernel's part of the message is up to 16 ranges by value a launch."""
    import torch
    n = 37 * 96 * KiB + 1001
    src, dst = Buf(n, "dev", offsets[0]), Buf(n, "dev", offsets[1])
    data = seeded("u8", 0xC0FFEE, n)
    src.fill(data)
    plan = mpt.mpt_plan(ctx, n, mpt.MPT_D2D, [(mpt.MPT_PATH_CE, 32768, 48 * KiB), (mpt.MPT_PATH_SM, 32768, 48 * KiB)], 16,
                        mpt.MPT_LAYOUT_INTERLEAVE)
    h = mpt.mpt_capture(ctx, plan, dst.ptr, src.ptr)
    mpt.mpt_launch(h, torch.cuda.current_stream())
    assert np.array_equal(dst.numpy(), T.copy(data)) and dst.guards_intact()
    mpt.mpt_graph_release(h)
    mpt.mpt_plan_destroy(plan)


@pytest.mark.parametrize("paths", [[(mpt.MPT_PATH_SM, 65536, 64 * KiB)], [(mpt.MPT_PATH_CE, 65536, 1024 * KiB)],
                                   [(mpt.MPT_PATH_SM, 65536, 64 * KiB, 0, mpt.MPT_SM_BULK)],
                                   [(mpt.MPT_PATH_CE, 32768, 64 * KiB), (mpt.MPT_PATH_SM, 32768, 64 * KiB)]],
                         ids=["sm", "ce", "bulk", "split"])
def test_direct_issue_handle_retargeted(ctx, paths):
    """A handle prepared for direct issue moves between its newest addresses, in a stream capture
    as well."""
    import torch
    n = 300 * KiB + 9
    pairs = []
    for so, do in ((0, 0), (16, 0), (3, 40)):
        src, dst = Buf(n, "dev", so), Buf(n, "dev", do)
        data = seeded("u8", 0xD1 + so, n)
        src.fill(data)
        pairs.append((src, dst, data))
    plan = mpt.mpt_plan(ctx, n, mpt.MPT_D2D, paths)
    h = mpt.mpt_prepare(ctx, plan, pairs[0][1].ptr, pairs[0][0].ptr, mpt.MPT_PREPARE_EAGER)
    s = torch.cuda.Stream()
    for i, (src, dst, data) in enumerate(pairs):
        if i:
            mpt.mpt_graph_rebind(h, plan, dst.ptr, src.ptr)
        mpt.mpt_launch(h, s)
        assert np.array_equal(dst.numpy(), T.copy(data)) and dst.guards_intact(), i
    src, dst, data = pairs[2]
    dst.view.zero_()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        mpt.mpt_launch(h, s)
    g.replay()
    assert np.array_equal(dst.numpy(), T.copy(data))
    mpt.mpt_graph_release(h)
    mpt.mpt_plan_destroy(plan)


MOVES = [8 * KiB - 1, 8 * KiB + 17, 16 * KiB, 16 * KiB + 1, 1024 * KiB - 16, 1024 * KiB, 1024 * KiB + 1, 1024 * KiB + 47,
         152 * 16 * KiB, 152 * 16 * KiB + 1, 152 * 32 * KiB - 5, 152 * 32 * KiB + 64]


@pytest.mark.parametrize("offsets", [(0, 0), (0, 16), (16, 0), (112, 96), (48, 48), (5, 0), (17, 1)], ids=lambda o: f"{o[0]}_{o[1]}")
@pytest.mark.parametrize("variant", [mpt.MPT_SM_VEC128, mpt.MPT_SM_TILE8K], ids=["vec", "small_tiles"])
def test_words_and_units(ctx, variant, offsets):
    """Both sides of the sizes at which words give way to units and tiles grow, on grids of one
    CTA to many, with source and destination agreeing modulo 32, 16 or not."""
    for n in MOVES:
        for ctas in (0, 1, 16, 152):
            _check(ctx, n, *offsets, ("dev", "dev"), variant, ctas)
    for where in (("host", "dev"), ("dev", "host")):
        for n in MOVES[1:8:2]:
            _check(ctx, n, *offsets, where, variant, 0)
