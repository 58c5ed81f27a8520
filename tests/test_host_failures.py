"""The library's host code on a stand-in for the CUDA runtime (fake_cudart.cpp): every call of a scenario is made to fail
in turn.  Whatever fails, no device block may go back to the pool of idle blocks while work is queued that can still use it
(another thread's context would get it), and what a failed call left half made is not taken for finished by the next.
Then what contexts make of a memory limit and of an allocation that fails."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2408_11376_gb300 import FDiRW, FDiRWBatch, FDiRWCoarse, build, fdirw

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    """The library's objects linked with the stand-in, in the place of the library."""
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    build.build()
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    so = str(tmp_path_factory.mktemp("fake") / "libfdirw_fake.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include, "-o", so,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    saved = fdirw._lib
    fdirw._lib = None
    lib = fdirw.load(so)
    lib.fake_calls.restype = lib.fake_violations.restype = lib.fake_launched.restype = lib.fake_blocks.restype = ctypes.c_long
    lib.fake_held.restype = ctypes.c_uint64
    lib.fake_fail_at.argtypes = [ctypes.c_long, ctypes.c_long]
    lib.fake_scalar.argtypes = [ctypes.c_double]
    lib.fake_free_bytes.argtypes = [ctypes.c_uint64]
    yield lib
    fdirw._lib = saved


def _stream(lib):
    s = ctypes.c_void_p()
    assert lib.cudaStreamCreateWithFlags(ctypes.byref(s), 0) == 0
    return s.value


def _each_failure(lib, prepare, act, finish):
    """act(state) with each of its runtime calls made to fail in turn, then finish(state); the calls that it made."""
    k = 0
    while True:
        lib.fake_reset()
        st = prepare()
        lib.fake_fail_at(k, 0)
        try:
            act(st)
        except fdirw.FdirwError:
            pass
        n = lib.fake_calls()
        lib.fake_fail_at(-1, 0)
        finish(st)
        assert lib.fake_violations() == 0, f"call {k}: a block was given back under queued work"
        k += 1
        if k > n:
            return n


def _close(st):
    for f in st:
        f.close()


# Sizes: the arrays that matter are above 64 MB, so that they go to cudaFree, where the stand-in looks, not to the pool.
BIG = (256, 256, 257)
MID = (143, 143, 143)


def test_create(fake):
    D = np.empty(int(np.prod(BIG)))
    stream = _stream(fake)
    for prec in ("fp32", "fp64"):
        def act(st):
            st.append(FDiRW(BIG, D, 0.1, 1, 1, prec, stream=stream))
            st[0].kernels()
            st[0].step(D, D, 1, want_mass=True)
        assert _each_failure(fake, list, act, _close) > 30


@pytest.mark.parametrize("per_cell", range(8, 45, 4))
def test_create_at_a_memory_limit(fake, per_cell):
    D = np.empty(int(np.prod(BIG)))
    fake.fake_reset()
    with pytest.raises(fdirw.FdirwError) as e:
        FDiRW(BIG, D, 0.1, 1, 1, stream=_stream(fake), mem_limit=per_cell * D.size + 64)
    assert e.value.code == fdirw.FDIRW_ERR_NOMEM
    assert fake.fake_violations() == 0


def test_set_velocity(fake):
    D = np.empty(int(np.prod(MID)))
    w = np.empty(3 * D.size)
    stream = _stream(fake)
    assert _each_failure(fake, lambda: [FDiRW(MID, D, 0.1, 1, 1, stream=stream)], lambda st: st[0].set_velocity(w), _close) > 8


BATCH = [MID, (9, 8, 7)]


def _batch(fake, stream):
    fake.fake_fill(1)                                # the radius of every source
    f = FDiRWBatch(BATCH, [np.empty(int(np.prod(s))) for s in BATCH], 0.1, 1, 1, 1, "bf16", stream=stream)
    fake.fake_fill(0)
    return f


def test_batch_create(fake):
    stream = _stream(fake)
    assert _each_failure(fake, list, lambda st: st.append(_batch(fake, stream)), _close) > 30


def test_batch_work(fake):
    stream = _stream(fake)
    c = np.zeros(sum(int(np.prod(s)) for s in BATCH))

    def work(st):
        st[0].kernels()
        st[0].step(c, c, 2)
    assert _each_failure(fake, lambda: [_batch(fake, stream)], work, _close) > 30


def test_coarse(fake):
    D = np.empty(int(np.prod(MID)))
    stream = _stream(fake)

    def act(st):
        fake.fake_fill(1)                            # liquid cells of every block
        st.append(FDiRWCoarse(MID, D, None, 3, 0.1, 1, 1, stream=stream))
        st[0].far_field(10.0, 0.1)
        st[0].coupled_step(D, 1, 1e-7, 1.0, 1e-5, 0.1, 1)
        st[0].coupled_step(D, 3, 1e-7, 1.0, 1e-5, 0.1, 1)
        st[0].read_coarse([0, 1])
    assert _each_failure(fake, list, act, _close) > 40


def test_read_back(fake):
    """Read-back buffers that grow after a call that failed with its kernel queued."""
    D = np.empty(int(np.prod(MID)))
    stream = _stream(fake)

    def prepare():
        f = FDiRW(MID, D, 0.1, 1, 1, stream=stream)
        f.kernels()
        return [f]

    def act(st):
        st[0].read_kernels(np.zeros(330000, dtype=np.int64))

    def grow(st):
        st[0].read_kernels(np.zeros(330001, dtype=np.int64))
        _close(st)
    assert _each_failure(fake, prepare, act, grow) > 3


def test_solid_stability_check_after_a_failed_call(fake):
    """A call that failed while the solid faces were being made leaves no bound that the next one takes for checked."""
    D = np.ones(12 * 11 * 10)
    stream = _stream(fake)

    def prepare():
        f = FDiRWCoarse((12, 11, 10), D, None, 3, 0.1, 1, 1, stream=stream)
        f.far_field(10.0, 0.1)
        f.kernels()
        fake.fake_scalar(1e6)                        # the largest sum of a cell's solid faces, as read from the device
        return [f]

    def act(st):
        st[0].coupled_step(np.ones(D.size), 1, 1e-7, 1.0, 1e-5, 0.1, 1)

    def again(st):
        with pytest.raises(fdirw.FdirwError) as e:
            act(st)
        assert e.value.code == fdirw.FDIRW_ERR_UNSTABLE
        _close(st)
    assert _each_failure(fake, prepare, act, again) > 3


def _ragged_batch(fake, n, **kw):
    fake.fake_fill(1)
    f = FDiRWBatch([(17, 9, 9)] * n, [np.empty(1377)] * n, 0.1, 1, 1, 1, "bf16", stream=_stream(fake), **kw)
    fake.fake_fill(0)
    return f


def _packed_bytes(n):
    return 27 * 2 * 1392 * n                         # 1377 cells of a structure in slots of 16


def test_batch_padding_does_not_split_it(fake):
    """Cache rows of 17 values are padded to 24 where there is room, and never at the price of a chunk."""
    fake.fake_reset()
    n, c = 4, np.zeros(4 * 1377)
    with _ragged_batch(fake, n) as f:
        f.step(c, c)
        i = f.info()
        assert i["n_chunks"] == 1 and i["cache_bytes"] > _packed_bytes(n)
        fixed = i["device_bytes"] - i["cache_bytes"]
    for extra in (0, 256, _packed_bytes(n) // 8):
        with _ragged_batch(fake, n, mem_limit=fixed + _packed_bytes(n) + 11 * 256 + extra) as f:
            f.step(c, c)
            i = f.info()
            assert i["n_chunks"] == 1 and i["cache_bytes"] <= _packed_bytes(n) + 256


def test_batch_drops_the_padding_when_its_allocation_fails(fake):
    fake.fake_reset()
    c = np.zeros(9 * 1377)
    with _ragged_batch(fake, 9) as f:
        fake.fake_fail_at(1, 2)                      # the arena (after the field's copy), also without idle blocks
        f.step(c, c)
        i = f.info()
        assert i["n_chunks"] == 1 and i["cache_bytes"] <= _packed_bytes(9) + 256
        f.read_kernels([0, 9 * 1377 - 1])


def _limited(fake, make, cells, W):
    """What a context of packed rows leaves for later calls at a memory limit, its padded one leaves as well."""
    fake.fake_reset()
    n_all, read = np.arange(cells), cells * (8 + 8 * W)
    with make(0) as f:
        f.kernels()
        i = f.info()
        padded, fixed = i["cache_bytes"], i["device_bytes"] - i["cache_bytes"]
    with make(fixed + (1 << 30)) as f:               # room for everything
        f.kernels()
        assert f.info()["cache_bytes"] == padded
    for later in (0, read, read // 2, 60 * cells + 8, read + 62 * cells):
        with make(fixed + 27 * 2 * 17 * (cells // 17 + 15) + 11 * 256 + later) as f:
            f.kernels()
            assert f.info()["n_chunks"] == 1 and f.info()["cache_bytes"] < padded
            if later >= read:
                f.read_kernels(n_all)
            elif later == read // 2:
                f.read_kernels(n_all[:cells // 2])
            elif later:
                f.set_velocity(np.zeros(3 * cells))


def test_padding_leaves_a_memory_limit_to_later_calls(fake):
    D, stream = np.empty(17 * 81), _stream(fake)
    _limited(fake, lambda limit: FDiRW((17, 9, 9), D, 0.1, 1, 1, "bf16", stream=stream, mem_limit=limit), D.size, 27)


def test_batch_padding_leaves_a_memory_limit_to_later_calls(fake):
    _limited(fake, lambda limit: _ragged_batch(fake, 4, mem_limit=limit), 4 * 1377, 27)


def test_idle_blocks_are_bounded_and_given_back(fake):
    fake.fake_reset()
    fdirw.fdirw_release_idle()
    held = fake.fake_held()
    D, stream = np.empty(160 ** 3), _stream(fake)    # arrays of 16 and 32 MB
    live = [FDiRW((160,) * 3, D, 0.1, 0, 1, stream=stream) for _ in range(6)]
    assert fake.fake_held() - held > 3 * (256 << 20)
    _close(live)
    idle = fake.fake_held() - held
    assert 128 << 20 < idle <= 256 << 20
    with FDiRW((160,) * 3, D, 0.1, 0, 1, stream=stream) as f:
        assert fake.fake_held() - held <= idle + f.info()["device_bytes"] // 4      # the blocks are used again
        assert fdirw.fdirw_release_idle() > 0
        assert 0 <= fake.fake_held() - held - f.info()["device_bytes"] < 4096      # (a block can be some bytes larger)
    fdirw.fdirw_release_idle()
    assert fake.fake_held() == held and fdirw.fdirw_release_idle() == 0


def test_idle_blocks_are_bounded_in_number(fake):
    """Many small contexts destroyed at once do not leave a list that every later allocation has to search."""
    fake.fake_reset()
    fdirw.fdirw_release_idle()
    held, stream = fake.fake_blocks(), _stream(fake)
    _close([FDiRW((9, 9, 9), np.empty(729), 0.1, 1, 1, stream=stream) for _ in range(100)])
    assert 100 < fake.fake_blocks() - held <= 512
    fdirw.fdirw_release_idle()
    assert fake.fake_blocks() == held


def test_network_takes_the_idle_blocks_memory(fake):
    """Allocations outside the contexts find the memory that destroyed contexts left with the library."""
    fake.fake_reset()
    fdirw.fdirw_release_idle()
    held, stream = fake.fake_held(), _stream(fake)
    FDiRW((9, 9, 9), np.empty(729), 0.1, 1, 1, stream=stream).close()
    assert fake.fake_held() > held
    fake.fake_fail_at(2, 1)
    net = fdirw.Net(np.zeros(fdirw.NET_NPARAM, dtype=np.float32))
    fake.fake_fail_at(-1, 0)
    idle = fdirw.fdirw_release_idle()
    net.close()
    assert idle == 0 and fake.fake_held() == held
