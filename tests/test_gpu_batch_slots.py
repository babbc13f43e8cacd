"""Batch slots that are used again: a ring of one slot submitted on two streams in turns, each time
right after mpt_batch_wait saw the last flag (the kernel ahead may still be putting its counters
back), and short batches after an error that an earlier call left behind, on a stream under capture
(refused), without the split into classes and with copy-engine lanes that no transfer is large
enough for.  Bytes equal the oracle's
copies."""
import numpy as np
import pytest

import paper_2604_22228_gb300 as mpt
import payload
from oracle import transfer as T

pytestmark = pytest.mark.gpu


def _buffers(n, seed):
    import torch
    data = payload.fill("u8", seed, n)
    return data, torch.from_numpy(data).cuda(), torch.zeros(n, dtype=torch.uint8, device="cuda")


def _submit_and_check(ctx, stream, count, size, data, src, dst):
    import torch
    dst.zero_()
    torch.cuda.synchronize()
    xs = [(src.data_ptr() + size * i, dst.data_ptr() + size * (count - 1 - i), size, mpt.MPT_D2D) for i in range(count)]
    b = mpt.mpt_batch_submit(ctx, xs, stream)
    mpt.mpt_batch_wait(b)
    done, flags = mpt.mpt_batch_poll(b, count)
    mpt.mpt_batch_release(b)
    assert done == count and all(flags)
    want = T.copy(data[:count * size]).reshape(count, size)[::-1].reshape(-1)
    return want, dst


@pytest.mark.parametrize("count", [1, 8, 9, 200])
def test_one_slot_on_two_streams(count):
    import torch
    ctx = mpt.mpt_ctx_create(0)
    mpt.mpt_batch_configure(ctx, 1)
    size = 3 * 4096 + 16
    data, src, dst = _buffers(200 * size, 0xBA7C0 + count)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    xs = [(src.data_ptr() + size * i, dst.data_ptr() + size * i, size, mpt.MPT_D2D) for i in range(count)]
    for i in range(100):  # no wait on the host between a batch and the next but the flags
        b = mpt.mpt_batch_submit(ctx, xs, streams[i % 2])
        mpt.mpt_batch_wait(b)
        mpt.mpt_batch_release(b)
    for s in streams:
        want, got = _submit_and_check(ctx, s, count, size, data, src, dst)
        torch.cuda.synchronize()
        assert np.array_equal(got[:count * size].cpu().numpy(), want)
    mpt.mpt_ctx_destroy(ctx)


def test_short_batch_after_an_error_left_behind():
    """A digest asked for inside a stream capture is refused and leaves the runtime's last error;
    the batch after it must not take that for its own."""
    import torch
    ctx = mpt.mpt_ctx_create(0)
    data, src, dst = _buffers(8 * 4096, 0xBA7C9)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with pytest.raises(Exception):
        with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
            with pytest.raises(mpt.MptError):
                mpt.mpt_hash_device(ctx, src, 4096, s)
    for count in (1, 8):
        want, got = _submit_and_check(ctx, torch.cuda.Stream(), count, 4096, data, src, dst)
        assert np.array_equal(got[:count * 4096].cpu().numpy(), want)
    mpt.mpt_ctx_destroy(ctx)


@pytest.mark.parametrize("count", [1, 9])
def test_batch_is_refused_inside_a_capture(count):
    import torch
    ctx = mpt.mpt_ctx_create(0)
    mpt.mpt_batch_configure(ctx, 1)
    data, src, dst = _buffers(9 * 4096, 0xBA7CB)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        with pytest.raises(mpt.MptError):
            _submit(ctx, s, count, src, dst)
        dst.add_(0)
    g.replay()
    torch.cuda.synchronize()
    assert not dst.any()
    want, got = _submit_and_check(ctx, s, count, 4096, data, src, dst)
    assert np.array_equal(got[:count * 4096].cpu().numpy(), want)
    mpt.mpt_ctx_destroy(ctx)


def _submit(ctx, stream, count, src, dst):
    mpt.mpt_batch_submit(ctx, [(src.data_ptr() + 4096 * i, dst.data_ptr() + 4096 * i, 4096, mpt.MPT_D2D) for i in range(count)],
                         stream)


@pytest.mark.parametrize("setting", ["split off", "idle lanes"])
def test_short_batches_of_other_rings(setting, monkeypatch):
    import torch
    ctx = mpt.mpt_ctx_create(0)
    if setting == "split off":
        monkeypatch.setenv("MPT_BATCH_SPLIT", "0")
        mpt.mpt_batch_configure(ctx)
    else:
        mpt.mpt_batch_configure_dma(ctx, 2, 4, 1 << 20)
    n = 70001
    host = payload.fill("u8", 0xBA7CA, 3 * n)
    dev = torch.from_numpy(host).cuda()
    pin, out = torch.from_numpy(host).pin_memory(), torch.zeros(3 * n, dtype=torch.uint8).pin_memory()
    dst = torch.zeros(3 * n, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    xs = [(dev.data_ptr(), dst.data_ptr() + n, n, mpt.MPT_D2D), (pin.data_ptr() + n, dst.data_ptr() + 2 * n, n, mpt.MPT_H2D),
          (dev.data_ptr() + 2 * n, out.data_ptr(), n, mpt.MPT_D2H)]
    b = mpt.mpt_batch_submit(ctx, xs)
    mpt.mpt_batch_wait(b)
    mpt.mpt_batch_release(b)
    got = dst.cpu().numpy()
    assert np.array_equal(got[n:2 * n], T.copy(host[:n])) and np.array_equal(got[2 * n:], T.copy(host[n:2 * n]))
    assert not got[:n].any()
    assert np.array_equal(out.numpy()[:n], T.copy(host[2 * n:])) and not out.numpy()[n:].any()
    mpt.mpt_ctx_destroy(ctx)
