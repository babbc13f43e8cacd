"""The stencil kernels' strips: row counts at and around a strip's height, widths at and around
a warp's columns, and each side of the grid sizes at which the strip height changes, against
the oracle's sweep (bit-exact: every step is rounded to fp32 in the stated order)."""
import numpy as np
import pytest

import paper_2604_22228_gb300 as mpt
import payload
from oracle import jacobi as J

pytestmark = pytest.mark.gpu

VEC = [(1, 4), (1, 132), (2, 128), (2, 1028), (3, 4), (4, 124), (5, 1152), (7, 132), (767, 1024), (768, 1024), (770, 1024),
       (4, 1 << 21), (5, 1677720), (8, 1 << 20), (9, 1048580), (2049, 4096)]
ANY = [(1, 2), (1, 31), (2, 33), (5, 127), (64, 1023), (65, 1023), (3, 70001), (4, 129), (66, 1025), (769, 1023), (767, 1025),
       (771, 1025), (4, 262149), (6, 131073), (1, 200003)]


@pytest.mark.parametrize("rows,cols,offset", [(r, c, 0) for r, c in VEC] + [(r, c, 0) for r, c in ANY] +
                         [(4, 128, 1), (771, 1024, 3), (2, 40000, 2)])
def test_sweep_at_strip_edges(rows, cols, offset):
    import torch
    n = (rows + 2) * cols
    grid = payload.fill("f32", 0x5EED0008 + rows * 131 + cols, n * 4).view(np.float32).reshape(rows + 2, cols)
    buf_in = torch.zeros(n + offset, dtype=torch.float32, device="cuda")
    buf_out = torch.full((n + offset + 8,), 7.0, dtype=torch.float32, device="cuda")
    buf_in[offset:offset + n].copy_(torch.from_numpy(grid.reshape(-1)))
    mpt.mpt_demo_jacobi_step(buf_in[offset:], buf_out[offset:], rows, cols, torch.cuda.current_stream())
    torch.cuda.synchronize()
    got = buf_out[offset:offset + n].cpu().numpy().reshape(rows + 2, cols)
    assert np.array_equal(got[1:rows + 1], J.step(grid)[1:rows + 1])
    assert (got[0] == 7.0).all() and (got[rows + 1] == 7.0).all()  # halo rows are not written
    assert (buf_out[:offset].cpu().numpy() == 7.0).all() and (buf_out[offset + n:].cpu().numpy() == 7.0).all()


@pytest.mark.parametrize("rows,cols", [(3, 64), (40, 513), (600, 2048)])
def test_chain_of_sweeps_and_copies(rows, cols):
    """Back-to-back sweeps between two buffers, each reading what the one before wrote, with a
    directly issued copy of the grid after every fourth: launches overlap, memory does not."""
    import torch
    n = (rows + 2) * cols
    grid = payload.fill("f32", 0x5EED000C + rows, n * 4).view(np.float32).reshape(rows + 2, cols)
    want = grid.copy()
    a, b = torch.from_numpy(grid.copy()).cuda(), torch.from_numpy(grid.copy()).cuda()
    c = torch.zeros_like(a)
    ctx = mpt.mpt_ctx_create(0)
    plan = mpt.mpt_plan(ctx, n * 4, mpt.MPT_D2D, [(mpt.MPT_PATH_SM, 65536, n * 4 // 16 * 16)])
    out = [mpt.mpt_prepare(ctx, plan, c, x, mpt.MPT_PREPARE_EAGER) for x in (a, b)]
    back = [mpt.mpt_prepare(ctx, plan, x, c, mpt.MPT_PREPARE_EAGER) for x in (a, b)]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    for it in range(40):
        mpt.mpt_demo_jacobi_step(a, b, rows, cols, s)
        new = want.copy()
        new[1:rows + 1] = J.step(want)[1:rows + 1]
        want = new
        a, b = b, a
        out.reverse()
        back.reverse()
        if it % 4 == 3:  # a -> c -> b: the next sweep overwrites b from a
            mpt.mpt_launch(out[0], s)
            mpt.mpt_launch(back[1], s)
    s.synchronize()
    assert np.array_equal(a.cpu().numpy(), want)
    assert np.array_equal(c.cpu().numpy(), want) and np.array_equal(b.cpu().numpy(), want)
    for h in out + back:
        mpt.mpt_graph_release(h)
    mpt.mpt_plan_destroy(plan)
    mpt.mpt_ctx_destroy(ctx)


@pytest.mark.parametrize("rows,cols", [(191, 1029), (192, 1025), (1, 196607), (70000, 2), (4095, 31), (4096, 32), (4097, 31), (4103, 17),
                                       (4096, 33), (65541, 5), (600001, 3)])
@pytest.mark.parametrize("offset", [0, 1])
def test_small_and_narrow_grids(rows, cols, offset):
    """Around the grid size up to which a thread takes a point, and rows of at most 32 columns in
    tall strips, more of them than a grid has blocks across too."""
    test_sweep_at_strip_edges(rows, cols, offset)
