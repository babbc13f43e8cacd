"""The batch kernel's tiles: sizes around the tile and line boundaries at every kind of
alignment and direction, and batch lengths around the steps of the descriptor search and the
longest table that a launch carries.  Whole
arenas are compared with the oracle's copies, so bytes between the transfers must stay as they
were."""
import numpy as np
import pytest

import paper_2604_22228_gb300 as mpt
import payload
from oracle import transfer as T

pytestmark = pytest.mark.gpu
KINDS = {mpt.MPT_D2D: ("dev", "dev"), mpt.MPT_H2D: ("host", "dev"), mpt.MPT_D2H: ("dev", "host")}
EDGES = [0, 1, 15, 16, 17, 111, 112, 127, 128, 129, 2047, 2048, 4080, 4096, 4097, 4096 + 112, 8192 - 16, 16384 - 1, 16384,
         16384 + 129, 3 * 16384 + 5]


@pytest.fixture(scope="module")
def ctx():
    import torch
    torch.cuda.init()
    c = mpt.mpt_ctx_create(0)
    yield c
    st, site = mpt.mpt_ctx_status(c)
    mpt.mpt_ctx_destroy(c)
    assert st == mpt.MPT_OK, (st, site)


def _run(ctx, xs, seed):
    """xs: (bytes, source offset, destination offset, direction), the offsets modulo 256."""
    import torch
    place = {(side, where): 0 for side in "sd" for where in ("dev", "host")}
    items = []
    for n, so, do, d in xs:
        row = [n, d]
        for side, where, off in (("s", KINDS[d][0], so), ("d", KINDS[d][1], do)):
            at = (place[side, where] + 255) // 256 * 256 + 256 + off
            place[side, where] = at + n
            row.append((side, where, at))
        items.append(row)
    src = {w: payload.fill("u8", seed + i, place["s", w] + 512) for i, w in enumerate(("dev", "host"))}
    dst = {w: np.full(place["d", w] + 512, 0x5A, dtype=np.uint8) for w in ("dev", "host")}
    ts = {"dev": torch.from_numpy(src["dev"]).cuda(), "host": torch.from_numpy(src["host"]).pin_memory()}
    td = {"dev": torch.from_numpy(dst["dev"]).cuda(), "host": torch.from_numpy(dst["host"]).pin_memory()}
    xf = [(ts[s[1]].data_ptr() + s[2], td[o[1]].data_ptr() + o[2], n, d) for n, d, s, o in items]
    b = mpt.mpt_batch_submit(ctx, xf, torch.cuda.current_stream())
    mpt.mpt_batch_wait(b)
    done, flags = mpt.mpt_batch_poll(b, len(xf))
    times = mpt.mpt_batch_times(b, len(xf))
    mpt.mpt_batch_release(b)
    assert done == len(xf) and all(flags) and all(0 <= t < 10 ** 10 for t in times)
    for n, d, s, o in items:
        dst[o[1]][o[2]:o[2] + n] = T.copy(src[s[1]][s[2]:s[2] + n])
    torch.cuda.synchronize()
    for w in ("dev", "host"):
        assert np.array_equal(td[w].cpu().numpy(), dst[w]), w


@pytest.mark.parametrize("direction", list(KINDS), ids=["d2d", "h2d", "d2h"])
@pytest.mark.parametrize("offsets", [(0, 0), (16, 16), (112, 112), (48, 112), (127, 127), (1, 1), (0, 5), (9, 0), (121, 66)],
                         ids=lambda o: f"{o[0]}_{o[1]}")
def test_tile_and_line_edges(ctx, direction, offsets):
    _run(ctx, [(n, *offsets, direction) for n in EDGES], 0xE0000 + 64 * direction + offsets[0])


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 1023, 1024, 1025, 1057, 4096])
@pytest.mark.parametrize("step", [16, 1])
def test_batch_lengths_and_mixed_directions(ctx, n, step):
    r = np.random.RandomState(n + step)
    xs = []
    for i in range(n):
        off = int(r.randint(0, 128 // step)) * step
        xs.append((int(r.randint(0, 9000 if n < 2000 else 700)), off, off if step == 16 else int(r.randint(0, 128)),
                   int(r.randint(0, 3))))
    _run(ctx, xs, 0xF0000 + n)


def test_overlaps_are_found_in_any_order(ctx):
    """Destinations that overlap one another, and sources that overlap a destination, are refused
    wherever they stand in the batch and whatever the others' order; the same batch without the
    offending transfer is accepted."""
    import torch
    dev = torch.zeros(1 << 20, dtype=torch.uint8, device="cuda")
    host = torch.zeros(1 << 20, dtype=torch.uint8).pin_memory()
    d, h = dev.data_ptr(), host.data_ptr()
    d2d, h2d, d2h = mpt.MPT_D2D, mpt.MPT_H2D, mpt.MPT_D2H
    good = [(d + 4096 * i, d + (512 << 10) + 4096 * i, 4000, d2d) for i in range(20)]
    good += [(h + 4096 * i, d + (640 << 10) + 4096 * i, 4000, h2d) for i in range(20)]
    good += [(d + 4096 * i, h + (512 << 10) + 4096 * i, 4000, d2h) for i in range(20)]
    bad = [(d, d + (512 << 10) + 4096 * 7 + 3999, 2, d2d),   # the last byte of a destination
           (h, d + (640 << 10) - 1, 2, h2d),                 # the first byte of one
           (d, h + (512 << 10) + 4096 * 19 + 100, 5, d2h),   # inside the last one
           (d + (512 << 10) + 4096 * 3, d + (900 << 10), 8, d2d),      # a source inside a destination
           (h + (512 << 10) - 4, d + (900 << 10), 8, h2d),             # reaching into the first
           (d + (512 << 10) - 4000, d + (900 << 10), 200 << 10, d2d)]  # spanning several
    for order in (list(good), good[::-1], good[1::2] + good[::2]):
        for x in bad:
            for at in (0, 31, len(order)):
                with pytest.raises(mpt.MptError) as e:
                    mpt.mpt_batch_submit(ctx, order[:at] + [x] + order[at:])
                assert e.value.status == mpt.MPT_EINVAL, x
        b = mpt.mpt_batch_submit(ctx, order + [(d + (900 << 10), d + (900 << 10), 0, d2d)])
        mpt.mpt_batch_wait(b)
        assert mpt.mpt_batch_poll(b)[0] == len(order) + 1
        mpt.mpt_batch_release(b)
