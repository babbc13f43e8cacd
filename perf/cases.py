"""The work that a program has this library do, as cases that can be timed.

Every case goes through the public calls of ``paper_2604_22228_gb300``: prepared transfers
(``mpt_plan`` / ``mpt_prepare`` / ``mpt_launch``), descriptor-table batches
(``mpt_batch_submit`` / ``mpt_batch_wait``), the stencil sweep with its halo transfers
(``mpt_demo_jacobi_step``) and digests (``mpt_hash_ranges_noalloc`` / ``mpt_hash_device``).

A case is a dict of plain values.  ``kind`` says which path it takes:

* ``window``  ``n`` messages posted one after another on a stream, each with its own buffers
  and its own prepared handle; sizes log-uniform on [lo, hi] in multiples of ``step``;
  ``src_off`` / ``dst_off`` shift every source and destination off a 256-byte boundary.
* ``sweep``   one message of every power of two from 8 bytes to ``top``.
* ``batch``   ``n`` transfers in one descriptor table; sizes log-uniform on [lo, hi], the
  fractions ``d2d`` and ``h2d`` (the rest device-to-host), addresses multiples of ``align``.
* ``jacobi``  two iterations over a ring of ``sub`` subdomains of ``rows`` x ``cols``: a sweep
  of each subdomain, then the halo rows moved between neighbours as transfers.
* ``digest``  digests of ``n`` ranges, in one call or one call per range.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2604_22228_gb300 as mpt

KiB, MiB, GiB = 1 << 10, 1 << 20, 1 << 30
DIRS = {"d2d": mpt.MPT_D2D, "h2d": mpt.MPT_H2D, "d2h": mpt.MPT_D2H}
_STREAM = None


def listed():
    return [
        # many small tensors moved between buffers: the short half of the message-size sweep,
        # where each message costs a launch rather than its bytes
        dict(name="d2d_short_window", kind="window", dir="d2d", n=64, lo=8, hi=64 * KiB, step=1, src_off=0, dst_off=0, mix=1),
        # the benchmark's headline: one message of every size from 8 bytes to 1 GiB
        dict(name="d2d_sweep", kind="sweep", top=GiB),
        # a window of 16 ordinary messages in flight (activations, gradient buckets)
        dict(name="d2d_medium_window", kind="window", dir="d2d", n=16, lo=MiB, hi=32 * MiB, step=1, src_off=0, dst_off=0, mix=2),
        # messages cut out of larger buffers at byte offsets, so that source and destination
        # differ modulo 16
        dict(name="d2d_shifted_window", kind="window", dir="d2d", n=6, lo=4 * MiB, hi=128 * MiB, step=1, src_off=11, dst_off=3, mix=3),
        # uploads from page-locked memory
        dict(name="h2d_window", kind="window", dir="h2d", n=8, lo=256 * KiB, hi=64 * MiB, step=4, src_off=0, dst_off=0, mix=4),
        # downloads to page-locked memory
        dict(name="d2h_window", kind="window", dir="d2h", n=8, lo=256 * KiB, hi=64 * MiB, step=4, src_off=0, dst_off=0, mix=5),
        # what a serving loop launches at a time: a few requests of mixed directions, waited for
        dict(name="batch_short", kind="batch", n=8, lo=16 * KiB, hi=4 * MiB, d2d=0.5, h2d=0.25, align=16, mix=6),
        # thousands of small blocks gathered or scattered on the device in one launch
        dict(name="batch_small_blocks", kind="batch", n=4096, lo=256, hi=64 * KiB, d2d=1.0, h2d=0.0, align=16, mix=7),
        # the batched workload's sizes and direction mix, over the host link and on the device
        dict(name="batch_mixed", kind="batch", n=2048, lo=256, hi=16 * MiB, d2d=0.7, h2d=0.3, align=16, mix=8),
        # the application study: flat subdomains whose halo rows are large messages
        dict(name="jacobi_strips", kind="jacobi", sub=4, rows=8, cols=4 * MiB),
        # the same solver on an ordinary square grid cut into four
        dict(name="jacobi_square", kind="jacobi", sub=4, rows=1024, cols=4096),
        # checking a set of received messages against their senders' digests
        dict(name="digest_ranges", kind="digest", n=64, lo=4 * KiB, hi=64 * MiB, align=16, one_call=True, mix=9),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["short", "window", "shifted", "host", "host", "sweep", "batch", "batch", "small", "jacobi", "jacobi", "digest"])
    mix = rng.randrange(1 << 30)
    if kind == "short":
        return dict(kind="window", dir="d2d", n=rng.randint(8, 96), lo=8, hi=log(4 * KiB, 512 * KiB), step=1, src_off=0, dst_off=0, mix=mix)
    if kind in ("window", "shifted"):
        hi = log(2 * MiB, 256 * MiB)
        n = max(2, min(32, GiB // hi))
        so, do = (rng.randrange(64), rng.randrange(64)) if kind == "shifted" else (0, 0)
        return dict(kind="window", dir="d2d", n=rng.randint(2, n), lo=max(8, hi // rng.choice([2, 16, 64])), hi=hi, step=1, src_off=so, dst_off=do, mix=mix)
    if kind == "host":
        hi = log(64 * KiB, 96 * MiB)
        off = rng.choice([0, 0, 4, 20])
        return dict(kind="window", dir=rng.choice(["h2d", "d2h"]), n=rng.randint(2, 6), lo=max(4 * KiB, hi // 16), hi=hi, step=4, src_off=off, dst_off=off, mix=mix)
    if kind == "sweep":
        return dict(kind="sweep", top=1 << rng.randint(20, 30))
    if kind == "batch":
        d2d = rng.choice([0.5, 0.7, 1.0, rng.uniform(0.3, 1.0)])
        n = log(1, 512)
        hi = log(64 * KiB, 16 * MiB)
        return dict(kind="batch", n=n, lo=log(256, 16 * KiB), hi=hi, d2d=d2d, h2d=(1.0 - d2d) * rng.choice([0.5, 1.0]), align=rng.choice([16, 16, 2]), mix=mix)
    if kind == "small":
        return dict(kind="batch", n=log(256, 4096), lo=log(16, 1024), hi=log(4 * KiB, 256 * KiB), d2d=1.0, h2d=0.0, align=rng.choice([16, 16, 2]), mix=mix)
    if kind == "jacobi":
        points = log(1 << 16, 1 << 25)
        rows = log(2, 4096)
        cols = max(64, points // rows)
        cols = cols // 4 * 4 if rng.random() < 0.6 else cols
        return dict(kind="jacobi", sub=rng.randint(1, 4), rows=rows, cols=cols)
    hi = log(64 * KiB, 128 * MiB)
    return dict(kind="digest", n=rng.randint(1, max(1, min(200, 2 * GiB // hi))), lo=max(16, hi // 1024), hi=hi, align=rng.choice([16, 8, 1]), one_call=rng.random() < 0.6, mix=mix)


def _sizes(case):
    """The message sizes of a case (the same for every seed)."""
    if case["kind"] == "sweep":
        return [1 << k for k in range(3, case["top"].bit_length())]
    r = random.Random(case["mix"])
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    step = case.get("step", 2 if case["kind"] == "batch" else 1)
    return [max(step, int(math.exp(r.uniform(lo, hi))) // step * step) for _ in range(case["n"])]


def _directions(case):
    r = random.Random(case["mix"] ^ 0x5EED)
    u = [r.random() for _ in range(case["n"])]
    return ["d2d" if x < case["d2d"] else "h2d" if x < case["d2d"] + case["h2d"] else "d2h" for x in u]


def _bytes(n, seed, host=False):
    """n seeded random bytes in device or page-locked host memory."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.empty((n + 7) // 8, dtype=torch.int64, device="cuda")
    t.random_(-(1 << 62), (1 << 62) - 1, generator=g)
    t = t.view(torch.uint8)[:n]
    if not host:
        return t
    h = torch.empty(n, dtype=torch.uint8, pin_memory=True)
    h.copy_(t)
    return h


def _zeros(n, host=False):
    return torch.zeros(n, dtype=torch.uint8, pin_memory=True) if host else torch.zeros(n, dtype=torch.uint8, device="cuda")


def _stream():
    """The program's own stream; every case issues its work there."""
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream()
    return _STREAM


class State:
    """A context with the buffers, plans and handles a program keeps for one case."""

    def __init__(self):
        self.ctx = mpt.mpt_ctx_create(0)
        self.plans, self.handles = {}, []

    def transfer(self, dst, src, nbytes, direction, eager=None):
        """A prepared transfer of the tuned plan, as a graph or by direct issue, whichever the
        tuner measured faster for its size."""
        d = DIRS[direction]
        if eager is None:
            try:
                eager = (mpt.mpt_tune_get(self.ctx, d, nbytes, mpt.MPT_MODE_EAGER)[1]
                         < mpt.mpt_tune_get(self.ctx, d, nbytes, mpt.MPT_MODE_GRAPH)[1])
            except mpt.MptError:
                eager = False
        key = (nbytes, d, eager)
        if key not in self.plans:
            layout = mpt.MPT_LAYOUT_CONTIG | (mpt.MPT_PLAN_EAGER if eager else 0)
            self.plans[key] = mpt.mpt_plan(self.ctx, nbytes, d, None, 16, layout)
        mode = mpt.MPT_PREPARE_EAGER if eager else mpt.MPT_PREPARE_GRAPH
        h = mpt.mpt_prepare(self.ctx, self.plans[key], dst, src, mode)
        self.handles.append(h)
        return h

    def __del__(self):
        try:
            torch.cuda.synchronize()
            for h in self.handles:
                mpt.mpt_graph_release(h)
            for p in self.plans.values():
                mpt.mpt_plan_destroy(p)
            mpt.mpt_ctx_destroy(self.ctx)
        except Exception:  # the interpreter is on its way out
            pass


def _prepare_window(st, case, seed):
    sizes = _sizes(case)
    direction, so, do = case.get("dir", "d2d"), case.get("src_off", 0), case.get("dst_off", 0)
    offs, pos = [], 0
    for n in sizes:
        offs.append(pos)
        pos = (pos + n + 64 + 4095) // 4096 * 4096
    st.src = _bytes(pos + 4096, seed, direction == "h2d")
    st.dst = _zeros(pos + 4096, direction == "d2h")
    st.out = [st.dst[o + do:o + do + n] for o, n in zip(offs, sizes)]
    st.launches = [st.transfer(st.dst.data_ptr() + o + do, st.src.data_ptr() + o + so, n, direction) for o, n in zip(offs, sizes)]
    if len(st.out) > 64:
        st.out = [st.dst]


def _prepare_batch(st, case, seed):
    sizes, dirs, align = _sizes(case), _directions(case), case["align"]
    r = random.Random(case["mix"] ^ 0xA119)
    end = {("src", 0): 0, ("src", 1): 0, ("dst", 0): 0, ("dst", 1): 0}
    items = []
    for n, d in zip(sizes, dirs):
        a, b = ("src", int(d == "h2d")), ("dst", int(d == "d2h"))
        at = []
        for k in (a, b):
            # a gap of 1 to 7 units of the alignment after the one before it
            end[k] = (end[k] + align - 1) // align * align + align * r.randint(1, 7)
            at.append(end[k])
            end[k] += n
        items.append((a, at[0], b, at[1], n, d))
    st.mem = {k: (_bytes(v + 64, seed + 7 * k[1], bool(k[1])) if k[0] == "src" else _zeros(v + 64, bool(k[1])))
              for k, v in end.items() if v}
    mpt.mpt_batch_configure(st.ctx)
    for t in st.mem.values():
        mpt.mpt_batch_register(st.ctx, t, t.numel())
    st.xfers = mpt.make_xfers([(st.mem[a].data_ptr() + ao, st.mem[b].data_ptr() + bo, n, DIRS[d]) for a, ao, b, bo, n, d in items])
    st.out = [t for k, t in sorted(st.mem.items()) if k[0] == "dst"]


def _grid(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.empty((case["sub"] * case["rows"], case["cols"]), dtype=torch.float32, device="cuda")
    return t.uniform_(-1, 1, generator=g)


def _with_halos(grid, case):
    """Every subdomain of the ring with its neighbours' boundary rows around it."""
    rows, n = case["rows"], case["sub"] * case["rows"]
    return [torch.cat([grid[(i * rows - 1) % n][None], grid[i * rows:(i + 1) * rows], grid[(i + 1) * rows % n][None]])
            for i in range(case["sub"])]


def _prepare_jacobi(st, case, seed):
    sub, rows, cols = case["sub"], case["rows"], case["cols"]
    st.bufs = [_with_halos(_grid(case, seed), case)]
    st.bufs.append([torch.zeros_like(t) for t in st.bufs[0]])
    st.halos = []
    for b in st.bufs:
        hs = []
        for i in range(sub):  # first row to the neighbour above, last row to the one below
            hs.append(st.transfer(b[(i - 1) % sub][rows + 1].data_ptr(), b[i][1].data_ptr(), cols * 4, "d2d", True))
            hs.append(st.transfer(b[(i + 1) % sub][0].data_ptr(), b[i][rows].data_ptr(), cols * 4, "d2d", True))
        st.halos.append(hs)
    st.rows, st.cols = rows, cols


def _ranges(case):
    sizes, align = _sizes(case), case["align"]
    at, pos = [], 0
    for n in sizes:
        at.append(pos + align)
        pos = (pos + align + n + 255) // 256 * 256
    return at, sizes, pos + 256


def _prepare_digest(st, case, seed):
    at, sizes, total = _ranges(case)
    st.mem = _bytes(total, seed)
    st.ranges = [(st.mem.data_ptr() + o, n) for o, n in zip(at, sizes)]
    st.one_call = case["one_call"]


def prepare(case, seed):
    st = State()
    st.kind = case["kind"]
    {"window": _prepare_window, "sweep": _prepare_window, "batch": _prepare_batch, "jacobi": _prepare_jacobi,
     "digest": _prepare_digest}[st.kind](st, case, seed)
    return st


def run(st):
    s = _stream()
    if st.kind in ("window", "sweep"):
        for h in st.launches:
            mpt.mpt_launch(h, s)
        return st.out
    if st.kind == "batch":
        b = mpt.mpt_batch_submit(st.ctx, st.xfers, s)
        mpt.mpt_batch_wait(b)
        mpt.mpt_batch_release(b)
        return st.out
    if st.kind == "jacobi":
        for b in (0, 1):
            for i, o in zip(st.bufs[b], st.bufs[1 - b]):
                mpt.mpt_demo_jacobi_step(i, o, st.rows, st.cols, s)
            for h in st.halos[1 - b]:
                mpt.mpt_launch(h, s)
        return st.bufs[0]
    if st.one_call:
        got = mpt.mpt_hash_ranges_noalloc(st.ranges, s)
    else:
        got = [mpt.mpt_hash_device(st.ctx, p, n, s) for p, n in st.ranges]
    return np.array(got, dtype=np.uint64).view(np.int64)


def work(case):
    if case["kind"] == "jacobi":
        # per iteration and subdomain: rows + 2 rows read, rows written; two halo rows read and written
        sub, rows, cols = case["sub"], case["rows"], case["cols"]
        return {"bytes": 2 * sub * cols * 4 * (2 * rows + 2 + 4), "flops": 2 * sub * rows * cols * 4}
    n = sum(_sizes(case))
    return {"bytes": n if case["kind"] == "digest" else 2 * n, "flops": 0}


def _mix64(z):
    def shr(x, k):  # logical shift of int64 words
        return (x >> k) & ((1 << (64 - k)) - 1)

    z = (z ^ shr(z, 30)) * -0x40A7B892E31B1A47
    z = (z ^ shr(z, 27)) * -0x6B2FB644ECCEEE15
    return z ^ shr(z, 31)


def exact(case, seed):
    if case["kind"] == "jacobi":
        g = _grid(case, seed).double()
        for _ in range(2):
            up, down = torch.roll(g, 1, 0), torch.roll(g, -1, 0)
            new = g.clone()
            new[:, 1:-1] = ((up + down)[:, 1:-1] + (g[:, :-2] + g[:, 2:])) * 0.25
            g = new
        return _with_halos(g, case)
    if case["kind"] == "digest":
        at, sizes, total = _ranges(case)
        mem, out = _bytes(total, seed), []
        for o, n in zip(at, sizes):
            words = torch.zeros((n + 7) // 8 * 8, dtype=torch.uint8, device="cuda")
            words[:n] = mem[o:o + n]
            w = words.view(torch.int64)
            i = torch.arange(w.numel(), device="cuda") * -0x61C8864680B583EB
            h = _mix64(w ^ i).sum() + _mix64(torch.tensor(n, device="cuda"))
            out.append(int(h))
        return np.array(out, dtype=np.int64)
    return None  # bytes moved: nothing is computed
