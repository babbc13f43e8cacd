"""Copy-engine paths over the host link: neighbouring chunks merged into one memcpy and, from
4 MiB, the bytes before the source's first 128-byte line apart, in graphs, by direct issue, in
splits with the zero-copy kernel and after a graph was retargeted to another alignment."""
import numpy as np
import pytest

import paper_2604_22228_gb300 as mpt
from gpu_util import Buf, seeded
from oracle import transfer as T

pytestmark = pytest.mark.gpu
MiB = 1 << 20
CE, ZC = mpt.MPT_PATH_CE, mpt.MPT_PATH_ZC
WHERE = {mpt.MPT_H2D: ("host", "dev"), mpt.MPT_D2H: ("dev", "host")}


@pytest.fixture(scope="module")
def ctx():
    import torch
    torch.cuda.init()
    c = mpt.mpt_ctx_create(0)
    yield c
    mpt.mpt_ctx_destroy(c)


def _buffers(n, direction, so, do, seed):
    src, dst = Buf(n, WHERE[direction][0], so), Buf(n, WHERE[direction][1], do)
    data = seeded("u8", seed, n)
    src.fill(data)
    return src, dst, T.copy(data)


@pytest.mark.parametrize("direction", list(WHERE), ids=["h2d", "d2h"])
@pytest.mark.parametrize("mode", [mpt.MPT_PREPARE_GRAPH, mpt.MPT_PREPARE_EAGER], ids=["graph", "eager"])
@pytest.mark.parametrize("layout", [mpt.MPT_LAYOUT_CONTIG, mpt.MPT_LAYOUT_INTERLEAVE], ids=["contig", "interleave"])
@pytest.mark.parametrize("paths", [[(CE, 65536, 64 * 1024)], [(CE, 65536, 5 * MiB)],
                                   [(CE, 49152, 2 * MiB), (ZC, 16384, MiB)]], ids=["small", "large", "split"])
def test_chunks_and_alignments(ctx, direction, mode, layout, paths):
    import torch
    for n in (100, 4 * MiB - 1, 4 * MiB, 9 * MiB + 77):
        for so, do in ((0, 0), (4, 4), (127, 3), (128, 64)):
            src, dst, want = _buffers(n, direction, so, do, 0xCE + n + so)
            plan = mpt.mpt_plan(ctx, n, direction, paths, 16, layout)
            h = mpt.mpt_prepare(ctx, plan, dst.ptr, src.ptr, mode)
            mpt.mpt_launch(h, torch.cuda.current_stream())
            assert np.array_equal(dst.numpy(), want) and dst.guards_intact(), (n, so, do)
            mpt.mpt_graph_release(h)
            mpt.mpt_plan_destroy(plan)
            mpt.mpt_graph_evict(ctx, src.ptr)


@pytest.mark.parametrize("first,second", [(0, 4), (4, 0), (4, 100), (64, 64)])
def test_retargeted_to_another_alignment(ctx, first, second):
    import torch
    n = 6 * MiB + 33
    plan = mpt.mpt_plan(ctx, n, mpt.MPT_H2D, [(CE, 65536, MiB)])
    a, b = (_buffers(n, mpt.MPT_H2D, o, 0, 0xCE0 + o) for o in (first, second))
    h = mpt.mpt_capture(ctx, plan, a[1].ptr, a[0].ptr)
    mpt.mpt_launch(h, torch.cuda.current_stream())
    assert np.array_equal(a[1].numpy(), a[2])
    mpt.mpt_graph_rebind(h, plan, b[1].ptr, b[0].ptr)
    mpt.mpt_launch(h, torch.cuda.current_stream())
    assert np.array_equal(b[1].numpy(), b[2]) and b[1].guards_intact()
    mpt.mpt_graph_release(h)
    mpt.mpt_graph_evict(ctx, b[0].ptr)
    mpt.mpt_plan_destroy(plan)
