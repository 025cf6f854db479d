"""The library's host side against a stand-in for the CUDA runtime (fake_cuda.cpp), on the CPU: what it does when calls
fail, when a wait runs out, and when memory it has kept is gone.  No GPU is used and none of the kernels."""
import ctypes as C
import os
import subprocess

import pytest

import mmee_inputs as mi
import paper_2604_03446_b200.binding as mm
from paper_2604_03446_b200 import build as lib_build

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(lib_build._nvcc()))), "include")


@pytest.fixture(scope="session")
def fake_path(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake_runtime") / "host_side.so")
    sources = [os.path.join(lib_build.CSRC, s) for s in ("mmee_api.cu", "mmee_workspace.cu", "mmee_plan.cu", "mmee_prune.cu")]
    subprocess.check_call(["g++", "-x", "c++", "-std=c++17", "-O1", "-shared", "-fPIC", "-pthread", "-Wl,-Bsymbolic", "-I", CUDA_INCLUDE,
                           "-o", out] + sources + [os.path.join(HERE, "fake_cuda.cpp")])
    return out


@pytest.fixture
def fake(fake_path, tmp_path):
    """A copy of its own for each test: the library's and the stand-in's state start fresh."""
    import shutil
    lib = C.CDLL(shutil.copy(fake_path, str(tmp_path / "host_side.so")))
    lib.mmee_destroy.argtypes = [C.c_void_p]
    return lib


def problem(topk=2):
    cfg = mi.config1()
    return (C.byref(mm._fill(mm.Workload(), cfg["workload"])), C.byref(mm._fill(mm.Arch(), cfg["arch"])),
            C.byref(mm._fill(mm.Objective(), mi.objective(mi.OBJ_ENERGY, topk))))


def solve(lib):
    best, topk = mm.Result(), (mm.Result * 2)()
    return lib.mmee_solve_host(*problem(), C.byref(best), topk, None, None), best.idx


def test_a_kept_workspace_does_not_outlive_its_context(fake):
    """A device reset takes kept device and pinned memory with it: the next call gets memory of its own, and nothing that is
    gone is used or freed again, whether it was idle at the reset or came back with its handle afterwards."""
    assert solve(fake) == (mm.OK, 7) and fake.fake_live() == 2
    fake.fake_device_reset()
    assert solve(fake) == (mm.OK, 7) and fake.fake_bad_pointers() == 0 and fake.fake_live() == 2
    fake.fake_device_reset()
    assert fake.mmee_trim() == mm.OK and fake.fake_bad_pointers() == 0 and fake.fake_live() == 0

    handles = []
    for _ in range(10):                              # more than are kept
        h = C.c_void_p()
        assert fake.mmee_create(*problem(), C.byref(h)) == mm.OK
        handles.append(h)
    fake.fake_device_reset()
    for h in handles:
        assert fake.mmee_destroy(h) == mm.OK
    assert solve(fake) == (mm.OK, 7) and fake.fake_bad_pointers() == 0 and fake.fake_live() == 2


def test_a_kept_workspace_stays_in_its_context(fake):
    """Several contexts on one device: each gets memory of its own, and keeps it."""
    for c in (1, 2, 1, 2):
        fake.fake_set_context(c)
        assert solve(fake) == (mm.OK, 7)
    assert fake.fake_bad_pointers() == 0 and fake.fake_live() == 4
    assert fake.mmee_trim() == mm.OK and fake.fake_live() == 0


@pytest.mark.parametrize("front", ["mmee_pareto_front", "mmee_pareto_front_bs_da"])
@pytest.mark.parametrize("missing", [1, 2, 4, 8, 0b1010])
def test_a_front_whose_wait_ran_out_returns_no_older_record(fake, front, missing):
    """Records that a front's kernel did not get to make are not read from what an earlier call left in the same memory: the
    status says that the wait ran out.  The next call starts clean."""
    def call():
        pts, n = (mm.Result * 8)(), C.c_uint32()
        return getattr(fake, front)(*problem(), pts, 8, C.byref(n)), n.value, [r.e_key for r in pts[:n.value]]

    fake.fake_chain(3, 0)
    assert call() == (mm.OK, 3, [0, 1, 2])
    fake.fake_chain(3, missing)
    assert call()[0] == mm.ERR_TIMEOUT
    fake.fake_chain(2, 0)
    assert call() == (mm.OK, 2, [0, 1]) and fake.fake_bad_pointers() == 0


@pytest.mark.parametrize("front", ["mmee_pareto_front", "mmee_pareto_front_bs_da"])
def test_fronts_take_the_ctas_that_can_be_resident_together(fake, front):
    """A context with a part of the SMs holds fewer CTAs at once than the device: the front runs on those, from four on (one
    that searches, one that merges, two that make the records)."""
    for resident, status in ((296, mm.OK), (295, mm.OK), (64, mm.OK), (4, mm.OK), (3, mm.ERR_CUDA), (2, mm.ERR_CUDA), (1000, mm.OK)):
        fake.fake_resident(resident)
        fake.fake_chain(3, 0)
        pts, n = (mm.Result * 8)(), C.c_uint32()
        assert getattr(fake, front)(*problem(), pts, 8, C.byref(n)) == status and n.value == (3 if status == mm.OK else 0)
        assert fake.fake_last_error() == 0 or status != mm.OK
    assert fake.fake_bad_pointers() == 0


@pytest.mark.parametrize("mallocs,host_allocs", [(1, 0), (0, 1)])
def test_a_failed_allocation_is_tried_again_without_the_idle_workspaces(fake, mallocs, host_allocs):
    """An allocation that fails once succeeds after the idle workspaces are freed; its error does not come back as the
    status of a later launch."""
    fake.fake_set_context(1)
    assert solve(fake) == (mm.OK, 7)                 # leaves an idle workspace of another context
    fake.fake_set_context(2)
    fake.fake_fail(mallocs, host_allocs)
    assert solve(fake) == (mm.OK, 7)
    assert fake.fake_live() == 2 and fake.fake_last_error() == 0 and fake.fake_bad_pointers() == 0


def test_an_allocation_that_keeps_failing_is_reported_once(fake):
    fake.fake_fail(2, 0)
    assert solve(fake)[0] == mm.ERR_CUDA and fake.fake_live() == 0 and fake.fake_last_error() == 0
    assert solve(fake) == (mm.OK, 7)
    h = C.c_void_p()
    assert fake.mmee_create(*problem(), C.byref(h)) == mm.OK
    fake.fake_fail(2, 0)
    other = C.c_void_p()
    assert fake.mmee_create(*problem(), C.byref(other)) == mm.ERR_CUDA and not other.value
    assert fake.mmee_decode(h, C.c_uint64(0), C.byref(mm.Result())) == mm.OK       # not that call's error
    assert fake.mmee_destroy(h) == mm.OK


def test_bytes_that_a_one_shot_call_says_it_moved(fake):
    """To the device the parameters of the launches it makes: one plan for one search; back the records."""
    best, topk, h2d, d2h = mm.Result(), (mm.Result * 2)(), C.c_uint64(), C.c_uint64()
    assert fake.mmee_solve_host(*problem(), C.byref(best), topk, C.byref(h2d), C.byref(d2h)) == mm.OK
    assert fake.fake_searches() == 1 and d2h.value == 3 * mm.RESULT_BYTES
    assert fake.fake_plan_bytes() <= h2d.value < fake.fake_plan_bytes() + 512


def launches(lib):
    """Searches and header resets in order: (capture that records it or 0, scratch or -1 for a reset, overlap, hold)."""
    out = []
    v = [C.c_ulonglong()] + [C.c_int() for _ in range(3)]
    while lib.fake_launch(len(out), *map(C.byref, v)):
        out.append(tuple(x.value for x in v))
    return out


def assert_scratches_are_free(log):
    """Among the searches that are launched, and among those that one capture records: of two with the same scratch the second
    starts after the first has ended, because a search between them lets the next one start only after the kernel before it has
    ended, or because it or one between them does not overlap with what is before it."""
    for capture in {c for c, *_ in log}:
        own = [(t, overlap, hold) for c, t, overlap, hold in log if c == capture]
        for y, (turn, _, _) in enumerate(own):
            for x in range(y):
                if turn >= 0 and own[x][0] == turn:
                    assert any(h for _, _, h in own[x + 1:y]) or not all(o for _, o, _ in own[x + 1:y + 1]), (capture, x, y)


def searching(lib, h):
    out = mm.Result()
    lib.mmee_search.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
    return lambda stream: lib.mmee_search(h, stream, C.addressof(out), None)


EAGER, GRAPH, OTHER = 16, 32, 48        # streams


@pytest.mark.parametrize("order", [[EAGER] * 40, [GRAPH] * 40, [EAGER, GRAPH, EAGER] * 13, [EAGER, EAGER, GRAPH] * 13,
                                   [EAGER, GRAPH, OTHER] * 13, [GRAPH, OTHER, GRAPH, GRAPH] * 10, [EAGER, GRAPH, GRAPH, GRAPH] * 10, None])
def test_a_scratch_is_free_when_its_turn_comes(fake, order):
    """Searches of one handle take the scratches in turn, whether they are launched or recorded by a stream capture: what is
    recorded is not part of the sequence of launches around it, and the other way round."""
    import random
    h = C.c_void_p()
    assert fake.mmee_create(*problem(), C.byref(h)) == mm.OK
    search = searching(fake, h)
    fake.fake_capture(C.c_void_p(GRAPH), C.c_ulonglong(7))
    fake.fake_capture(C.c_void_p(OTHER), C.c_ulonglong(9))
    rng = random.Random(11)
    for stream in order or [rng.choice((EAGER, EAGER, GRAPH, OTHER)) for _ in range(400)]:
        assert search(stream) == mm.OK
    log = launches(fake)
    assert_scratches_are_free(log)
    if order and len(set(order)) == 1:
        assert len({t for _, t, _, _ in log}) == 5 and all(o for _, t, o, _ in log[2:] if t >= 0)      # (the first may be without)
    fake.fake_capture(C.c_void_p(GRAPH), C.c_ulonglong(0))
    fake.fake_capture(C.c_void_p(OTHER), C.c_ulonglong(0))
    assert fake.mmee_destroy(h) == mm.OK and fake.fake_bad_pointers() == 0


def test_a_header_is_clean_only_after_a_reset_that_was_launched(fake):
    """After a launch that failed the header is reset before the next search; a reset that a capture has recorded has not
    happened when that search is followed by one that is launched."""
    h = C.c_void_p()
    assert fake.mmee_create(*problem(), C.byref(h)) == mm.OK
    search = searching(fake, h)
    fake.fake_capture(C.c_void_p(GRAPH), C.c_ulonglong(7))
    fake.fake_fail_launch(1)
    assert search(EAGER) == mm.ERR_CUDA
    n = len(launches(fake))
    for stream in (GRAPH, GRAPH, EAGER, EAGER, GRAPH):
        assert search(stream) == mm.OK
    log = launches(fake)[n:]
    kinds = [(c, t < 0) for c, t, _, _ in log]
    assert kinds == [(7, True), (7, False), (7, True), (7, False), (0, True), (0, False), (0, False), (7, False)]
    assert not any(o for (_, t, o, _), before in zip(log[1:], log) if t >= 0 and before[1] < 0)
    assert_scratches_are_free(log)
    fake.fake_capture(C.c_void_p(GRAPH), C.c_ulonglong(0))
    assert fake.mmee_destroy(h) == mm.OK and fake.fake_bad_pointers() == 0


def test_records_are_taken_when_their_signal_comes_or_the_stream_has_ended(fake):
    """A call with host records returns when the search's word is in host memory; where that does not come in time it waits for
    the stream, and a wait that fails is the call's status.  With kernel timing on it waits for the stream at once."""
    h = C.c_void_p()
    assert fake.mmee_create(*problem(), C.byref(h)) == mm.OK
    fake.mmee_search_host.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p]
    fake.mmee_kernel_timing.argtypes = [C.c_void_p, C.c_int]
    best = mm.Result()

    def call():
        before, best.idx = fake.fake_syncs(), 0
        return fake.mmee_search_host(h, C.addressof(best), None), best.idx, fake.fake_syncs() - before

    for _ in range(3):
        assert call() == (mm.OK, 7, 0)
        fake.fake_late(1, 0)
        assert call() == (mm.OK, 7, 1)
    fake.fake_late(1, 1)
    assert call() == (mm.ERR_CUDA, 0, 1)
    fake.fake_late(0, 0)
    assert call() == (mm.OK, 7, 0)
    assert fake.mmee_kernel_timing(h, 1) == mm.OK and call() == (mm.OK, 7, 1)
    assert fake.mmee_destroy(h) == mm.OK and solve(fake) == (mm.OK, 7) and fake.fake_bad_pointers() == 0
