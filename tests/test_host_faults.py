"""Host code of the library when a CUDA call fails, linked against a stand-in runtime
(tests/native/fake_cudart.cpp) that fails calls on request and logs launches: no GPU needed."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

import paper_2604_22228_gb300 as mpt
from paper_2604_22228_gb300 import _ffi, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MiB = 1 << 20
ERROR = 700  # any error code


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    build.build()
    objs = [os.path.join(build.OBJDIR, s + ".o") for s in build.SOURCES]
    for s, o in zip(build.SOURCES, objs):
        if not os.path.exists(o):
            os.makedirs(build.OBJDIR, exist_ok=True)
            build._compile(build._nvcc(), s)
    include = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    out = str(tmp_path_factory.mktemp("fake") / "libmpt_fake.so")
    subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", include,
                    os.path.join(ROOT, "tests", "native", "fake_cudart.cpp"), *objs, "-ldl", "-pthread", "-o", out],
                   check=True, capture_output=True, text=True)
    return out


@pytest.fixture
def fake(library, tmp_path, monkeypatch):
    """The stand-in's controls; the package calls the library linked against it meanwhile."""
    path = str(tmp_path / "libmpt_fake.so")  # a copy of its own: every test starts with fresh state
    shutil.copy(library, path)
    monkeypatch.setattr(_ffi, "_lib", None)
    lib = _ffi.load(path)
    lib.fake_fail.argtypes = [C.c_char_p, C.c_int, C.c_int]
    lib.fake_count.argtypes = lib.fake_loaded.argtypes = [C.c_char_p]
    lib.fake_capturing.argtypes = [C.c_void_p]
    lib.fake_copied_to.restype = C.c_void_p
    lib.fake_launches.argtypes = [C.c_char_p, C.POINTER(C.c_uint), C.POINTER(C.c_int)]
    return lib


@pytest.fixture
def ctx(fake):
    c = mpt.mpt_ctx_create(0)
    yield c
    mpt.mpt_ctx_destroy(c)


def _alloc(lib, n, host=False):
    p = C.c_void_p()
    assert (lib.cudaHostAlloc(C.byref(p), C.c_size_t(n), 0) if host else lib.cudaMalloc(C.byref(p), C.c_size_t(n))) == 0
    return p.value


def _short(lib):
    a, b = _alloc(lib, MiB), _alloc(lib, MiB)
    return [(a, b, 4096, mpt.MPT_D2D)]


# ---- batches ---------------------------------------------------------------------------------

def _batch(ctx, xs, stream=None):
    b = mpt.mpt_batch_submit(ctx, xs, stream)
    mpt.mpt_batch_wait(b)
    mpt.mpt_batch_release(b)


@pytest.mark.parametrize("n", [1, 8, 9])
def test_batch_after_an_error_left_behind(fake, ctx, n):
    """An earlier call's error, which the runtime keeps until it is asked for, is no failure of a
    batch's launch."""
    x = _short(fake)[0]
    fake.fake_leave_error(ERROR)
    _batch(ctx, [(x[0] + 4096 * i, x[1] + 4096 * i, 4096, mpt.MPT_D2D) for i in range(n)])


@pytest.mark.parametrize("n,call,name", [(1, "launch", "k_batch_short"), (8, "cudaEventRecord", "k_batch_short"),
                                         (9, "cudaGraphLaunch", None), (9, "cudaEventRecord", None)])
def test_slot_after_a_failed_submission(fake, ctx, n, call, name):
    """A submission that fails leaves nothing of its own running: what was launched before the
    failure is waited for, and the slot serves the next batch."""
    mpt.mpt_batch_configure(ctx, 1)
    x = _short(fake)[0]
    xs = [(x[0] + 4096 * i, x[1] + 4096 * i, 4096, mpt.MPT_D2D) for i in range(n)]

    def launched():
        return fake.fake_launches(name.encode(), None, None) if name else fake.fake_count(b"cudaGraphLaunch")

    _batch(ctx, xs)
    before, syncs = launched(), fake.fake_count(b"cudaStreamSynchronize")
    fake.fake_fail(call.encode(), 0, ERROR)
    with pytest.raises(mpt.MptError) as e:
        mpt.mpt_batch_submit(ctx, xs)
    assert e.value.status == mpt.MPT_ECUDA
    if call == "cudaEventRecord":
        assert launched() == before + 1 and fake.fake_count(b"cudaStreamSynchronize") == syncs + 1
    queries = fake.fake_count(b"cudaEventQuery")
    _batch(ctx, xs)
    # the slot was asked before it was used again, beside the query of the wait
    assert fake.fake_count(b"cudaEventQuery") >= queries + 2


# ---- digests ---------------------------------------------------------------------------------

@pytest.mark.parametrize("sizes", [[100], [MiB] * 5, [100] * 200])
def test_digest_after_an_error_left_behind(fake, ctx, sizes):
    a = _alloc(fake, max(sizes))
    calls = [lambda: mpt.mpt_hash_ranges_noalloc([(a, n) for n in sizes])]
    if len(sizes) == 1:
        calls.append(lambda: mpt.mpt_hash_device(ctx, a, sizes[0]))
    for call in calls:
        fake.fake_leave_error(ERROR)
        call()
        fake.fake_fail(b"launch", 0, ERROR)
        with pytest.raises(mpt.MptError) as e:
            call()
        assert e.value.status == mpt.MPT_ECUDA
        call()


# ---- stream captures -------------------------------------------------------------------------

@pytest.mark.parametrize("n", [1, 8, 9])
def test_batch_is_refused_inside_a_capture(fake, ctx, n):
    """A batch submitted to a stream under capture would run at every replay, with this batch's
    epoch and table, and never for the caller: it is refused, and the slot stays free."""
    mpt.mpt_batch_configure(ctx, 1)
    x = _short(fake)[0]
    xs = [(x[0] + 4096 * i, x[1] + 4096 * i, 4096, mpt.MPT_D2D) for i in range(n)]
    s = _alloc(fake, 16, host=True)  # any handle
    fake.fake_capturing(s)
    with pytest.raises(mpt.MptError) as e:
        mpt.mpt_batch_submit(ctx, xs, s)
    assert e.value.status == mpt.MPT_ECUDA
    assert fake.fake_launches(b"k_batch", None, None) == 0
    fake.fake_capturing(None)
    _batch(ctx, xs, s)


# ---- handles for direct issue ----------------------------------------------------------------

def test_rebind_that_fails_leaves_the_handle_as_it_was(fake, ctx):
    n = 66 * 4096
    old, new, src = _alloc(fake, n), _alloc(fake, n), _alloc(fake, n)
    plan = mpt.mpt_plan(ctx, n, mpt.MPT_D2D, [(mpt.MPT_PATH_SM, 65536, n)])
    h = mpt.mpt_prepare(ctx, plan, old, src, mpt.MPT_PREPARE_EAGER)
    fake.fake_fail(b"cudaGetFuncBySymbol", 0, ERROR)
    with pytest.raises(mpt.MptError):
        mpt.mpt_graph_rebind(h, plan, new, src)
    for k, to in ((1, old), (2, new)):
        mpt.mpt_launch(h)
        assert fake.fake_launches(b"k_sm_copy", None, None) == k and fake.fake_copied_to() == to
        mpt.mpt_graph_rebind(h, plan, new, src)
    mpt.mpt_graph_release(h)
    mpt.mpt_plan_destroy(plan)


# ---- overlapped launches ---------------------------------------------------------------------

@pytest.mark.parametrize("value,overlap", [(None, 1), ("1", 1), ("0", 0), ("0x0", 0), ("", 1)])
@pytest.mark.parametrize("cols", [64, 63])
def test_stencil_follows_the_overlap_switch(fake, monkeypatch, value, overlap, cols):
    """MPT_PDL=0 turns overlapped launches off for the stencil's sweeps too, as for the contexts'
    direct copies."""
    monkeypatch.delenv("MPT_PDL", raising=False)
    if value is not None:
        monkeypatch.setenv("MPT_PDL", value)
    a, b = _alloc(fake, MiB), _alloc(fake, MiB)
    mpt.mpt_demo_jacobi_step(a, b, 4, cols)
    got = C.c_int(-1)
    assert fake.fake_launches(b"k_jacobi", None, C.byref(got)) == 1 and got.value == overlap
    s = _alloc(fake, 16, host=True)
    fake.fake_capturing(s)
    mpt.mpt_demo_jacobi_step(a, b, 4, cols, s)
    assert fake.fake_launches(b"k_jacobi", None, C.byref(got)) == 2 and got.value == 0
    n = 4096
    c = mpt.mpt_ctx_create(0)
    plan = mpt.mpt_plan(c, n, mpt.MPT_D2D, [(mpt.MPT_PATH_SM, 65536, n)])
    mpt.mpt_launch_eager(c, plan, b, a)
    assert fake.fake_launches(b"k_sm_copy", None, C.byref(got)) == 1 and got.value == overlap
    mpt.mpt_ctx_destroy(c)


# ---- contexts --------------------------------------------------------------------------------

def test_context_page_locks_no_memory_for_digests(fake):
    """Page-locking costs a tenth of a millisecond, which a program that creates a context and
    asks for no digest must not pay, nor one that asks for its first."""
    c = mpt.mpt_ctx_create(0)
    assert fake.fake_count(b"cudaHostAlloc") == 0
    mpt.mpt_hash_device(c, _alloc(fake, 4096), 4096)
    assert fake.fake_count(b"cudaHostAlloc") == 0
    mpt.mpt_ctx_destroy(c)


@pytest.mark.parametrize("n", [1, 9])
def test_ring_loads_its_kernels(fake, ctx, n):
    """A ring's kernels are loaded when it is built, not by the first batch that needs one."""
    mpt.mpt_batch_configure(ctx)
    loaded = fake.fake_loaded(b"")
    assert fake.fake_loaded(b"k_batch") >= 4
    x = _short(fake)[0]
    for shift in (0, 1):
        _batch(ctx, [(x[0] + 4096 * i + shift, x[1] + 4096 * i, 4000, mpt.MPT_D2D) for i in range(n)])
    assert fake.fake_loaded(b"") == loaded


def test_batch_tune_reports_a_grid_that_runs(fake, ctx):
    """The last setting measured is the fastest here; what is reported and applied is what its
    kernels ran with, at most two CTAs per SM."""
    x = _short(fake)[0]
    xs = [(x[0] + 4096 * i, x[1] + 4096 * i, 4000, mpt.MPT_D2D) for i in range(4)]
    r = mpt.mpt_batch_tune(ctx, xs, mpt.MPT_BATCH_TUNE_TIME, 1)
    assert r["candidates"] == 30 and r["ctas"] == 2 * 152
    _batch(ctx, [(x[0] + 8192 * i, x[1] + 8192 * i, 8192, mpt.MPT_D2D) for i in range(8)])
    ran = C.c_uint()
    fake.fake_launches(b"k_batch_short", C.byref(ran), None)
    assert ran.value <= r["ctas"]


def test_launch_takes_streams_only(fake, ctx):
    """A stream is an int, None or an object with cuda_stream; anything else is refused before it
    is taken for a pointer."""
    n = 4096
    plan = mpt.mpt_plan(ctx, n, mpt.MPT_D2D, [(mpt.MPT_PATH_SM, 65536, n)])
    h = mpt.mpt_prepare(ctx, plan, _alloc(fake, n), _alloc(fake, n), mpt.MPT_PREPARE_EAGER)

    class Stream:
        cuda_stream = 0

    for good in (None, 0, Stream()):
        mpt.mpt_launch(h, good)
    for bad in (b"stream", "stream", C.c_void_p(64)):
        with pytest.raises(AttributeError):
            mpt.mpt_launch(h, bad)
    assert fake.fake_launches(b"k_sm_copy", None, None) == 3
