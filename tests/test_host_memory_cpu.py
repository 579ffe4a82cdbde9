"""The library's host code when device memory runs out, on a stand-in for the CUDA runtime (no device):
whatever allocation fails, the call returns QEW_ENOMEM, and neither that handle's later calls nor a retry
launch a kernel on an array that is not there (on a device that would be a memory fault)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1211_7275_gb300 import _build, _capi

HERE = os.path.dirname(os.path.abspath(__file__))
WRAPPED = """Malloc Free MallocHost FreeHost Memcpy MemcpyAsync Memset MemsetAsync GetDevice SetDevice GetLastError
PeekAtLastError GetErrorString StreamCreateWithFlags StreamDestroy StreamSynchronize StreamBeginCapture StreamEndCapture
GraphInstantiate GraphDestroy GraphExecDestroy GraphLaunch EventCreate EventCreateWithFlags EventDestroy EventRecord
EventSynchronize EventElapsedTime""".split()
OK, ENOMEM, ESTATE = 0, -2, -6
FP32, FP64 = 0, 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("fake")
    cc, procs, objs = _build.nvcc(), [], []
    for src, lang in ((os.path.join(_build.CSRC, "qew_capi.cu"), "cu"), (os.path.join(HERE, "fake", "fake_cuda.cpp"), "cu"),
                      (os.path.join(HERE, "fake", "fake_new.cpp"), "c++")):
        objs.append(str(tmp / (os.path.basename(src) + ".o")))
        procs.append(subprocess.Popen([cc, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-I", _build.INCLUDE, "-I", _build.CSRC,
                                       *_build.ARCH, "-x", lang, "-c", src, "-o", objs[-1]]))
    assert all(p.wait() == 0 for p in procs)
    out = str(tmp / "libqew_fake.so")
    wrap = [x for n in WRAPPED for x in ("-Xlinker", f"--wrap=cuda{n}")]
    subprocess.run([cc, "-shared", *_build.ARCH, "-o", out, *objs, *wrap, "-Xlinker", "-Bsymbolic"], check=True)
    lib = ctypes.CDLL(out)
    for name, (res, args) in _capi.SIGNATURES.items():
        if hasattr(lib, name):
            getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    lib.fake_fail_after.argtypes = [ctypes.c_int64]
    lib.fake_throw_after.argtypes = [ctypes.c_int64]
    lib.fake_capacity.argtypes = [ctypes.c_size_t]
    for n in ("fake_held", "fake_peak"):
        getattr(lib, n).restype = ctypes.c_size_t
    for n in ("fake_launches", "fake_bad", "fake_off_stream"):
        getattr(lib, n).restype = ctypes.c_int64
    lib.fake_first_bad.restype = ctypes.c_char_p
    return lib


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def create(lib, L, kind, precision, f=0.9):
    L = np.ascontiguousarray(np.atleast_1d(L), dtype=np.int64)
    f = np.full(L.size, f)
    kind = np.ascontiguousarray(np.broadcast_to(np.asarray(kind, np.int32), (L.size,)))
    h = ctypes.c_void_p()
    rc = lib.qew_create_batch(ctypes.byref(h), L.size, _p(L), _p(f), _p(kind), 0.1, 1, precision)
    return rc, h


def calls(lib, h, n_sites):
    """Statuses of the calls that would launch kernels on the state."""
    steps = np.array([40, 41, 100], dtype=np.int64)
    v, u, c = np.empty(3 * 64), np.empty(n_sites), np.empty(n_sites, dtype=np.int32)
    S = np.empty(8)
    rc = [lib.qew_advance(h, 1)]
    t = ctypes.c_int64()
    lib.qew_get_state(h, None, ctypes.byref(t))
    rc.append(lib.qew_observe(h, _p(steps + t.value), 3, _p(v), _p(v)))
    rc.append(lib.qew_get_state(h, _p(u), None))
    rc.append(lib.qew_get_cells(h, _p(c)))
    rc.append(lib.qew_structure_factor(h, 8, _p(S)))
    rc.append(lib.qew_set_state(h, _p(np.zeros(n_sites))))
    rc.append(lib.qew_reset(h))
    return rc


RECONFIGURE = {
    "to FP64": (FP32, lambda lib, h: lib.qew_set_precision(h, FP64)),
    "to FP32": (FP64, lambda lib, h: lib.qew_set_precision(h, FP32)),
    "period": (FP32, lambda lib, h: lib.qew_set_disorder_period(h, 64)),
    "period64": (FP64, lambda lib, h: lib.qew_set_disorder_period(h, 64)),
    "samples": (FP32, lambda lib, h: lib.qew_set_samples(h, _p(np.arange(2, dtype=np.uint32)))),
    "tuning": (FP32, lambda lib, h: lib.qew_set_tuning(h, 224, 8, 1)),
}


@pytest.mark.parametrize("kind", [0, 1, 3])
@pytest.mark.parametrize("what", sorted(RECONFIGURE))
@pytest.mark.parametrize("L", [5000, 600001])   # below and above the look-ahead shape's line
def test_a_handle_whose_reconfiguration_fails(lib, what, kind, L):
    precision, change = RECONFIGURE[what]
    for fail in range(40):
        lib.fake_reset()
        rc, h = create(lib, [L, L], kind, precision)
        assert rc == OK
        lib.fake_reset()
        lib.fake_fail_after(fail)
        rc = change(lib, h)
        lib.fake_fail_after(-1)
        assert rc in (OK, ENOMEM)
        after = calls(lib, h, 2 * L)
        assert lib.fake_bad() == 0, lib.fake_first_bad()
        assert set(after) <= ({OK} if rc == OK else {OK, ESTATE}), after
        assert change(lib, h) == OK              # a retry with memory to be had
        assert calls(lib, h, 2 * L) == [OK] * 7
        assert lib.fake_bad() == 0, lib.fake_first_bad()
        lib.qew_destroy(h)
        if rc == OK and fail > 20:
            break


@pytest.mark.parametrize("what", ["period", "period64", "samples"])
def test_a_new_layout_is_not_a_new_state(lib, what):
    """After a failed change of the disorder the caches are of the old one: another call that makes a layout
    does not let the chains go on with them, a reset does."""
    precision, change = RECONFIGURE[what]
    for fail in range(12):
        lib.fake_reset()
        rc, h = create(lib, [5000, 5000], 0, precision)
        assert rc == OK and lib.qew_advance(h, 10) == OK
        lib.fake_fail_after(fail)
        rc = change(lib, h)
        lib.fake_fail_after(-1)
        assert rc in (OK, ENOMEM)
        assert lib.qew_set_tuning(h, 224, 8, 1) == OK
        assert lib.qew_advance(h, 10) == (OK if rc == OK else ESTATE)
        assert lib.qew_reset(h) == OK
        assert calls(lib, h, 10000) == [OK] * 7
        assert lib.fake_bad() == 0, lib.fake_first_bad()
        lib.qew_destroy(h)


def test_autotuning_that_runs_out_of_memory(lib):
    for fail in range(0, 400, 7):
        lib.fake_reset()
        rc, h = create(lib, [5003 + fail] * 2, 0, FP32)   # (the shape found is remembered by size)
        assert rc == OK and lib.qew_advance(h, 1100) == OK
        assert lib.qew_set_tuning(h, 0, 0, 0) == OK
        lib.fake_fail_after(fail)
        v = np.empty(2)
        rc = lib.qew_observe(h, _p(np.array([1200], dtype=np.int64)), 1, _p(v), None)
        lib.fake_fail_after(-1)
        assert rc in (OK, ENOMEM)
        assert calls(lib, h, 2 * (5003 + fail)) == [OK] * 7   # in the shape it had
        assert lib.fake_bad() == 0, lib.fake_first_bad()
        lib.qew_destroy(h)


@pytest.mark.parametrize("what", sorted(RECONFIGURE))
def test_host_allocations_that_fail(lib, what):
    """No exception leaves a C entry: QEW_ENOMEM, and the handle is as after a failed device allocation."""
    precision, change = RECONFIGURE[what]
    L = 5000
    v, zero = np.empty(8), np.zeros(2 * L)
    others = [lambda h: lib.qew_reset(h), lambda h: lib.qew_set_state(h, _p(zero)), lambda h: lib.qew_advance(h, 40),
              lambda h: lib.qew_observe(h, _p(np.array([2000, 2001], dtype=np.int64)), 2, _p(v), None)]
    lib.fake_reset()
    rc, h = create(lib, [L, L], 3, precision)
    assert rc == OK
    assert lib.qew_enable_stats(h, 1) == OK
    for fail in range(40):
        for call in [lambda h: change(lib, h)] + others:
            lib.qew_reset(h)
            lib.fake_throw_after(fail)
            rc = call(h)
            lib.fake_throw_after(-1)
            assert rc in (OK, ENOMEM)
            assert set(calls(lib, h, 2 * L)) <= ({OK} if rc == OK else {OK, ESTATE})
            assert lib.fake_bad() == 0, lib.fake_first_bad()
            lib.qew_reset(h)
            assert change(lib, h) == OK
            assert lib.qew_set_precision(h, precision) in (OK, ESTATE)
    lib.qew_destroy(h)


@pytest.mark.parametrize("kind", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("precision", [FP32, FP64])
@pytest.mark.parametrize("L", [300, 600001])
def test_creation_fails_cleanly(lib, kind, precision, L):
    for fail in range(40):
        lib.fake_reset()
        held = lib.fake_held()
        lib.fake_fail_after(fail)
        rc, h = create(lib, [L, 77], kind, precision)
        lib.fake_fail_after(-1)
        assert lib.fake_bad() == 0, lib.fake_first_bad()
        if rc == OK:
            lib.qew_destroy(h)
            assert lib.fake_held() == held
            if fail > 20:
                break
        else:
            assert rc == ENOMEM and h.value is None and lib.fake_held() == held


@pytest.mark.parametrize("precision", [FP32, FP64])
def test_uploads_and_fills_are_ordered_with_the_kernels(lib, precision):
    """The handle's stream does not wait for the legacy default stream, where a copy from pageable memory
    may still be under way when the call returns: nothing but reads of finished results goes there."""
    lib.fake_reset()
    rc, h = create(lib, [3000, 3000], 0, precision)
    assert rc == OK and calls(lib, h, 6000) == [OK] * 7
    assert lib.qew_enable_stats(h, 1) == OK and calls(lib, h, 6000) == [OK] * 7
    assert lib.qew_get_stats(h, None, None, None, None, None) == OK
    assert lib.qew_set_precision(h, 1 - precision) == OK and calls(lib, h, 6000) == [OK] * 7
    assert lib.fake_off_stream() == 0
    lib.qew_destroy(h)


@pytest.mark.parametrize("precision", [FP32, FP64])
def test_allocations_inside_the_calls(lib, precision):
    L = 5000
    lib.fake_reset()
    rc, h = create(lib, [L, L], 3, precision)
    v = np.empty(64 * 2)
    for fail in range(4):
        # a first observation, and one with more of them than the buffers hold
        for n in (1, 2, 10 + 4 * fail):
            lib.fake_fail_after(fail)
            t = ctypes.c_int64()
            lib.qew_get_state(h, None, ctypes.byref(t))
            steps = t.value + 1 + np.arange(n, dtype=np.int64)
            assert lib.qew_observe(h, _p(steps), n, _p(v), _p(v)) in (OK, ENOMEM)
            lib.fake_fail_after(fail)
            assert set(calls(lib, h, 2 * L)) <= {OK, ENOMEM}
            lib.fake_fail_after(-1)
            assert lib.qew_observe(h, _p(np.array([50], dtype=np.int64)), 1, _p(v), _p(v)) == OK
            assert calls(lib, h, 2 * L) == [OK] * 7
            assert lib.fake_bad() == 0, lib.fake_first_bad()
    lib.qew_destroy(h)


@pytest.mark.parametrize("kind,per_site", [(0, 36), (1, 52), (3, 36)])
def test_fp64_batch_with_room_for_one_copy_of_the_caches(lib, kind, per_site):
    """Per site: two displacements, the cache's cell and its nodes; one step per launch then."""
    L = (1 << 21) + 5
    lib.fake_reset()
    lib.fake_capacity(lib.fake_held() + int(1.02 * per_site * L))
    rc, h = create(lib, [L], kind, FP64)
    assert rc == OK
    assert lib.qew_advance(h, 20) == OK
    assert lib.fake_bad() == 0, lib.fake_first_bad()
    assert lib.fake_last_K() == 1 and lib.fake_last_in_place() == 1
    # with the memory back, setting the precision again takes the second copy
    lib.fake_reset()
    assert lib.qew_reset(h) == OK
    assert lib.qew_set_precision(h, FP64) == OK
    assert lib.qew_advance(h, 20) == OK
    assert lib.fake_bad() == 0, lib.fake_first_bad()
    assert lib.fake_last_K() == 8 and lib.fake_last_in_place() == 0
    lib.qew_destroy(h)


@pytest.mark.parametrize("kind,L,per_site,per_chain", [
    (0, [(1 << 22) + 5], 32, 0), (3, [(1 << 22) + 5], 32, 0), (1, [(1 << 22) + 5], 64, 0), (2, [(1 << 22) + 5], 16, 0),
    (0, [1] * 50000, 32, 200), (3, [37] * 50000, 32, 200), (4, [101] * 20000, 64, 200)])
def test_fp32_batch_with_room_for_the_state(lib, kind, L, per_site, per_chain):
    """Two buffers of cells, offsets and caches and little beside them: what only makes a relaxation faster
    (tile lists of a second shape, the partials of many observations, Case 3's third node) gives way."""
    n = sum(L)
    lib.fake_reset()
    lib.fake_capacity(lib.fake_held() + int(1.015 * per_site * n) + per_chain * len(L))
    rc, h = create(lib, L, kind, FP32)
    assert rc == OK
    assert lib.qew_advance(h, 100) == OK
    lib.fake_capacity(2 ** 62)
    v = np.empty(30 * len(L))
    t = np.arange(100, 130, dtype=np.int64)
    assert lib.qew_observe(h, _p(t), 30, _p(v), None) == OK
    assert lib.fake_max_n_obs() == 1 and lib.fake_bad() == 0, lib.fake_first_bad()
    if kind == 3:
        assert lib.fake_last_has_q3() == 0
    # with the memory back, setting the precision again takes the rest
    assert lib.qew_reset(h) == OK and lib.qew_set_precision(h, FP32) == OK
    assert lib.qew_observe(h, _p(t), 30, _p(v), None) == OK
    assert lib.fake_max_n_obs() > 1 and lib.fake_bad() == 0, lib.fake_first_bad()
    if kind == 3:
        assert lib.fake_last_has_q3() == 1
    lib.qew_destroy(h)
