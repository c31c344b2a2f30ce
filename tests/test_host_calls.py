"""What the library's host code asks of the CUDA runtime, on a runtime that is not there (tests/fake_cudart.cpp):
the order of work between streams, what is left behind by a call that fails, and how often memory is
allocated.  The library's own object files are linked with it; no kernel runs."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

import paper_1710_10420_gb300 as prs
from paper_1710_10420_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    _build.build()
    objs = [os.path.join(_build.OBJDIR, os.path.basename(s) + ".o") for s in _build.sources()]
    if not all(os.path.exists(o) for o in objs):
        _build.build(force=True)
    cuda = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
    out = str(tmp_path_factory.mktemp("fake") / "libprs_fake.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", out], check=True)
    fake = ctypes.CDLL(out)
    for name, (res, args) in prs._SIGS.items():
        fn = getattr(fake, name)
        fn.restype, fn.argtypes = res, args
    fake.fake_log.restype = ctypes.c_char_p
    fake.fake_fail.argtypes = [ctypes.c_char_p, ctypes.c_int, ctypes.c_int]
    fake.fake_limit.argtypes = [ctypes.c_size_t]
    return fake


@pytest.fixture(autouse=True)
def _clean(lib):
    lib.fake_reset()


def _log(lib):
    return [line.split() for line in lib.fake_log().decode().splitlines()]


def _batch(lib, runs, stream):
    arr = (prs.prs_params * len(runs))(*runs)
    b = ctypes.c_void_p()
    assert lib.prs_batch_create(arr, len(runs), stream, ctypes.byref(b)) == prs.PRS_OK
    lib.fake_reset()
    return b


STREAM = 77  # the caller's


def _ordered(log, first, second):
    """Whether work on stream `second` at the end of the log comes after all work on stream `first`."""
    if first == second:
        return True
    events = {line[2] for line in log if line[0] == "record" and line[1] == first}
    return any(line[0] == "wait" and line[1] == second and line[2] in events for line in log)


@pytest.mark.parametrize("write", [True, False])
def test_ensemble_state_copies_follow_the_callers_stream(lib, write):
    """The copies of prs_batch_set_state and prs_batch_get_state come after what the caller queued on the
    stream given to prs_batch_create (the fill of a pinned buffer, a kernel that reads one)."""
    b = _batch(lib, [prs.make_params((128, 128)), prs.make_params((256, 64))], STREAM)
    for run, shape in ((0, (128, 128)), (1, (64, 256))):
        phi, v = np.zeros(shape, np.float32), np.zeros(shape, np.float32)
        lib.fake_reset()
        if write:
            assert lib.prs_batch_set_state(b, run, phi.ctypes.data, v.ctypes.data, 3) == prs.PRS_OK
        else:
            assert lib.prs_batch_get_state(b, run, phi.ctypes.data, v.ctypes.data, None) == prs.PRS_OK
        log = _log(lib)
        copies = [i for i, line in enumerate(log) if line[0] == "copy"]
        assert len(copies) == 2
        for i in copies:
            assert _ordered(log[:i], str(STREAM), log[i][1]), log
        assert any(line[0] == "sync" and line[1] == log[copies[-1]][1] for line in log[copies[-1]:])
    assert lib.prs_batch_destroy(b) == prs.PRS_OK


@pytest.mark.parametrize("call,nth", [("record", 1), ("wait", 1), ("wait", 2), ("wait", 3), ("launch", 2),
                                      ("launch", 5), ("copy", 1), ("copy", 2), ("copy", 3), ("record", 2),
                                      ("record", 3), ("sync", 1)])
def test_nothing_is_in_flight_behind_an_ensemble_error(lib, call, nth):
    """When a CUDA call fails in the middle of prs_batch_run, every stream that was given work is waited
    for before the error is returned (the caller may free its memory, and the groups are not joined)."""
    b = _batch(lib, [prs.make_params((128, 128)), prs.make_params((256, 64))], STREAM)
    ns = (ctypes.c_int64 * 2)(12, 12)
    out = np.zeros((2, 4, 4))
    lib.fake_fail(call.encode(), nth, 719)
    assert lib.prs_batch_run(b, ns, 4, out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 4) == prs.PRS_ECUDA
    log = _log(lib)
    at = log.index(["FAIL", call])
    for stream in {line[1] for line in log[:at] if line[0] in ("launch", "copy", "memset")}:
        assert ["sync", stream] in log[at:], stream
    assert not np.any(out)
    lib.fake_reset()
    assert lib.prs_batch_run(b, ns, 4, out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 4) == prs.PRS_OK
    assert lib.prs_batch_destroy(b) == prs.PRS_OK


def _run(lib, shape, **kw):
    h = ctypes.c_void_p()
    assert lib.prs_create(ctypes.byref(prs.make_params(shape, **kw)), STREAM, ctypes.byref(h)) == prs.PRS_OK
    return h


def _state(lib, h):
    p, v, n = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_int64()
    assert lib.prs_device_state(h, ctypes.byref(p), ctypes.byref(v), ctypes.byref(n)) == prs.PRS_OK
    return p.value, v.value, n.value


@pytest.mark.parametrize("shape,kw", [((128, 128), {}), ((50, 40), dict(precision=prs.PRS_FP64)),
                                      ((50, 40), dict(precision=prs.PRS_FP64, flags=prs.PRS_REPRO)),
                                      ((128, 64, 64), {}), ((21, 20, 19), dict(tblock=1))])
def test_a_launch_that_fails_leaves_the_state_where_it_is(lib, shape, kw):
    h = _run(lib, shape, **kw)
    assert lib.prs_init(h, None, None) == prs.PRS_OK
    before = _state(lib, h)
    lib.fake_fail(b"launch", 1, 9)  # an invalid configuration: the context stays usable
    assert lib.prs_step(h, 1) == prs.PRS_ECUDA
    assert _state(lib, h) == before
    assert lib.prs_step(h, 1) == prs.PRS_OK
    assert _state(lib, h)[0] != before[0] and _state(lib, h)[2] == 1
    assert lib.prs_destroy(h) == prs.PRS_OK


@pytest.mark.parametrize("shape,kw", [((128, 128), {}), ((50, 40), dict(precision=prs.PRS_FP64)), ((128, 64, 64), {})])
def test_a_launch_that_fails_is_reported_once(lib, shape, kw):
    h = _run(lib, shape, **kw)
    assert lib.prs_init(h, None, None) == prs.PRS_OK
    lib.fake_fail(b"launch", 1, 9)
    assert lib.prs_step(h, 1) == prs.PRS_ECUDA
    J = ctypes.c_double()
    assert lib.prs_observable(h, 0, 0.1, ctypes.byref(J)) == prs.PRS_OK
    assert lib.prs_destroy(h) == prs.PRS_OK


def test_a_wait_that_gave_up_is_reported_before_the_state_is_stepped(lib):
    """Correctly rounded diagnostics on a box of the staged passes: prs_step_measure returns the timeout of an
    earlier pass (the test writes the error word the diagnostics would bring) and queues no step."""
    h = _run(lib, (512, 512, 64), flags=prs.PRS_FP32_CR)
    status = next(int(line[2]) for line in _log(lib) if line[0] == "mallochost")  # result (48 bytes), counter, error
    assert lib.prs_init(h, None, None) == prs.PRS_OK
    assert lib.prs_step(h, 1) == prs.PRS_OK
    before = _state(lib, h)
    ctypes.c_uint.from_address(status + 52).value = 1
    lib.fake_reset()
    d = prs.prs_diag()
    assert lib.prs_step_measure(h, 3, ctypes.byref(d)) == prs.PRS_ETIMEOUT
    assert len([line for line in _log(lib) if line[0] == "launch"]) == 1  # the diagnostics
    assert _state(lib, h) == before
    assert lib.prs_step_measure(h, 3, ctypes.byref(d)) == prs.PRS_OK and _state(lib, h)[2] == 4
    assert lib.prs_destroy(h) == prs.PRS_OK


@pytest.mark.parametrize("shape", [(256, 32, 32), (256, 64, 64), (1024, 32, 32), (256, 256, 32), (768, 128, 32),
                                   (256, 512, 32)])
@pytest.mark.parametrize("steps", [20, 13, 2])
def test_small_boxes_take_no_staged_pairs(lib, shape, steps):
    """The staged two-step tiles take 25 us on a box of few of them, several times the march's passes."""
    h = _run(lib, shape)
    assert lib.prs_init(h, None, None) == prs.PRS_OK
    lib.fake_reset()
    assert lib.prs_step(h, steps) == prs.PRS_OK
    names = [line[2] for line in _log(lib) if line[0] == "launch"]
    assert names and not any("step3d_t2" in name for name in names)
    assert lib.prs_destroy(h) == prs.PRS_OK


def _mallocs(lib):
    return [int(line[1]) for line in _log(lib) if line[0] == "malloc"]


@pytest.mark.parametrize("shape,kw", [((128, 128, 128), {}), ((250, 170), {}), ((256, 256), {}), ((45, 42, 38), {}),
                                      ((64, 64), dict(precision=prs.PRS_FP64)), ((100, 90), dict(tblock=1))])
@pytest.mark.parametrize("bound", [True, False])
def test_a_run_allocates_once(lib, shape, kw, bound):
    """Creation and the first state take one device allocation, and the first state of bound buffers none
    (so it may be captured)."""
    nbytes = int(np.prod(shape)) * (8 if kw.get("precision") else 4)
    phi, v = np.zeros(nbytes, np.uint8), np.zeros(nbytes, np.uint8)
    h = _run(lib, shape, **kw)
    bufs = [np.zeros(nbytes + 64, np.uint8) for _ in range(3)]
    if bound:
        assert lib.prs_bind(h, *[b.ctypes.data + -b.ctypes.data % 16 for b in bufs]) == prs.PRS_OK
        assert len(_mallocs(lib)) == 1
    assert lib.prs_set_state_device(h, phi.ctypes.data, v.ctypes.data, 0) == prs.PRS_OK
    assert lib.prs_step(h, 7) == prs.PRS_OK
    assert len(_mallocs(lib)) == 1
    assert lib.prs_destroy(h) == prs.PRS_OK
    assert len([line for line in _log(lib) if line[0] == "free"]) == 1


@pytest.mark.parametrize("fields", [4, 3])
def test_a_run_without_room_for_the_second_dphi_buffer(lib, fields):
    """Where four fields do not fit in one allocation the run takes three and asks for the fourth apart."""
    n = 4 * 64 ** 3
    h = _run(lib, (64, 64, 64))
    lib.fake_limit(4 * n if fields == 4 else 3 * n)  # with the scratch, neither fits whole
    assert lib.prs_init(h, None, None) == (prs.PRS_OK if fields == 4 else prs.PRS_ENOMEM)
    if fields == 4:
        assert len(_mallocs(lib)) == 2
        assert lib.prs_step(h, 6) == prs.PRS_OK and _state(lib, h)[2] == 6
    lib.fake_limit(0)
    assert lib.prs_init(h, None, None) == prs.PRS_OK
    assert lib.prs_destroy(h) == prs.PRS_OK
    assert len([line for line in _log(lib) if line[0] == "free"]) == len(_mallocs(lib))


@pytest.mark.parametrize("tblocks", [[0, 0, 1, 0], [1, 1, 1, 1], [3, 2, 0, 1]])
@pytest.mark.parametrize("shape", [(256, 64), (128, 32, 16)])
def test_runs_of_an_ensemble_share_their_launches_whatever_their_tblock(lib, shape, tblocks):
    counts = []
    for tbs in (tblocks, [0] * len(tblocks)):
        b = _batch(lib, [prs.make_params(shape, tblock=t) for t in tbs], STREAM)
        ns = (ctypes.c_int64 * len(tbs))(*[20] * len(tbs))
        assert lib.prs_batch_run(b, ns, 0, None, 0) == prs.PRS_OK
        counts.append([line[2] for line in _log(lib) if line[0] == "launch"])
        assert lib.prs_batch_destroy(b) == prs.PRS_OK
    assert counts[0] == counts[1] and len(counts[1]) <= 20


@pytest.mark.parametrize("shape,tiles", [((4096, 3), 32), ((256, 256), 16), ((64, 64, 64), 32)])
def test_noalloc_diagnostics_fill_the_gpu(lib, shape, tiles):
    phi = np.zeros(tuple(reversed(shape)), np.float32)
    d = prs.prs_diag()
    p, at = ctypes.byref(prs.make_params(shape)), phi.ctypes.data
    assert lib.prs_measure_noalloc(p, at, at, STREAM, ctypes.byref(d)) == prs.PRS_OK
    assert [int(line[3]) >= tiles for line in _log(lib) if line[0] == "launch"] == [True]
    assert not _mallocs(lib)


@pytest.mark.parametrize("shape,kw,integers", [((40, 5, 40), {}, False), ((40, 3, 90), {}, False),
                                               ((40, 6, 40), {}, True), ((40, 3), {}, True),
                                               ((64, 64), dict(dx=10.0, W0=1.2), False),
                                               ((64, 64), dict(flags=prs.PRS_REPRO), False)])
def test_fp64_steps_take_the_integers_where_they_serve(lib, shape, kw, integers):
    h = _run(lib, shape, precision=prs.PRS_FP64, **kw)
    assert lib.prs_init(h, None, None) == prs.PRS_OK
    lib.fake_reset()
    assert lib.prs_step(h, 2) == prs.PRS_OK
    names = [line[2] for line in _log(lib) if line[0] == "launch"]
    assert len(names) == 2 and all(("step_fix64" if integers else "step_generic") in name for name in names)
    assert lib.prs_destroy(h) == prs.PRS_OK


@pytest.mark.parametrize("shape", [(100000, 3), (60000, 5)])
def test_a_step_of_a_few_long_rows_fills_the_gpu(lib, shape):
    h = _run(lib, shape, precision=prs.PRS_FP64, flags=prs.PRS_REPRO)
    assert lib.prs_init(h, None, None) == prs.PRS_OK
    lib.fake_reset()
    assert lib.prs_step(h, 1) == prs.PRS_OK
    assert [int(line[3]) >= 152 for line in _log(lib) if line[0] == "launch"] == [True]
    assert lib.prs_destroy(h) == prs.PRS_OK


def test_an_observable_of_a_small_box_has_a_block_for_every_row(lib):
    h = _run(lib, (65, 65))
    assert lib.prs_init(h, None, None) == prs.PRS_OK
    J, before = ctypes.c_double(), len(_mallocs(lib))
    lib.fake_reset()
    assert lib.prs_observable(h, 1, 0.1, ctypes.byref(J)) == prs.PRS_OK
    assert [int(line[3]) >= 65 for line in _log(lib) if line[0] == "launch"] == [True]
    assert before == 1 and not _mallocs(lib)  # its gradient goes to the idle dphi buffer
    assert lib.prs_destroy(h) == prs.PRS_OK


def test_the_benchmark_counts_the_passes_the_library_takes(lib):
    """bench.py divides the time of an interval's steps by passes of three (3D) and five (2D) steps."""
    import bench

    for shape, calls in (((1024, 1024, 1024), [(18, 3, 6), (2, 2, 1)]), ((512, 512, 512), [(18, 3, 6), (2, 2, 1)]),
                         ((4096, 4096), [(20, 5, 4)])):
        h = _run(lib, shape)
        assert lib.prs_init(h, None, None) == prs.PRS_OK  # memory that nothing touches
        tb = 3 if len(shape) == 3 else 5
        assert bench.interval_calls(21, tb)[:2] == (calls[0][0], calls[1][0] if len(calls) > 1 else 0)
        for steps, t, passes in calls:
            lib.fake_reset()
            assert lib.prs_step(h, steps) == prs.PRS_OK
            names = [line[2] for line in _log(lib) if line[0] == "launch"]
            assert len(names) == passes, (shape, names)
            assert all(f"Fold32ELi{t}E" in n or (t == 2 and "t2tma" in n) for n in names), names
        assert lib.prs_destroy(h) == prs.PRS_OK


def test_bound_runs_reuse_small_memory_while_runs_exist(lib):
    """What a small bound run gives back serves the next one; the last run gives everything back, and 64 MB
    and 16 pieces are the most that is kept."""
    bufs = [np.zeros((64, 64), np.float32) for _ in range(3)]

    def bind(shape):
        h = _run(lib, shape)
        assert lib.prs_bind(h, *[b.ctypes.data + -b.ctypes.data % 16 for b in bufs]) == prs.PRS_OK
        return h

    def done(*runs):
        for h in runs:
            assert lib.prs_destroy(h) == prs.PRS_OK

    def held():
        return len(_mallocs(lib)) - len([line for line in _log(lib) if line[0] == "free"])

    first, a = bind((64, 60)), bind((100, 90, 80))
    done(a)
    assert len(_mallocs(lib)) == 2 and held() == 2  # kept
    b = bind((100, 90, 79))
    assert len(_mallocs(lib)) == 2  # taken again
    c, large = bind((100, 90, 80)), bind((512, 512, 40))
    assert len(_mallocs(lib)) == 4
    done(large)
    assert held() == 3  # 42 MB go back
    done(*[bind((64, 64)) for _ in range(3)], b, c)
    assert held() == 1 + 3 + 2  # the first's; kept: three of 64 x 64, b's and c's
    runs = [bind((180, 160, 160)) for _ in range(8)]  # 19 MB each
    done(*runs)
    assert held() == 6 + 3  # 64 MB are 67.1e6 bytes, of which 7.7e6 were kept before
    done(first)
    assert held() == 0
    done(bind((64, 60)))
    assert held() == 0


def test_kept_memory_stays_with_its_device(lib):
    bufs = [np.zeros((64, 64), np.float32) for _ in range(3)]

    def bind(device):
        lib.fake_device(device)
        h = _run(lib, (64, 60))
        assert lib.prs_bind(h, *[b.ctypes.data + -b.ctypes.data % 16 for b in bufs]) == prs.PRS_OK
        return h

    try:
        first, a = bind(0), bind(0)
        lib.fake_device(1)
        assert lib.prs_destroy(a) == prs.PRS_OK  # made on device 0, released with device 1 current
        b = bind(1)
        assert len(_mallocs(lib)) == 3
        c = bind(0)
        assert len(_mallocs(lib)) == 3
        for h in (first, b, c):
            assert lib.prs_destroy(h) == prs.PRS_OK
    finally:
        lib.fake_device(0)
