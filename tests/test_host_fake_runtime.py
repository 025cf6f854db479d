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
    """A context with a part of the SMs holds fewer CTAs at once than the device: the front runs on those."""
    for resident, status in ((296, mm.OK), (295, mm.OK), (64, mm.OK), (3, mm.OK), (2, mm.ERR_CUDA), (1000, mm.OK)):
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
