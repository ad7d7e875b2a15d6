"""Recorded call sequences on a fake CUDA runtime: when the graph of a plan's launches is
made, what happens where it cannot be made, and that a capture in another thread is left
alone."""
import ctypes as C
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
FIELDS = ("launches graph_launches captured streams graphs execs instantiate_calls fail_instantiate "
          "fail_stream capture_elsewhere broken caller_capturing mode_changes no_memory").split()
N = 5                                     # launches of the plan


class Fake(C.Structure):
    _fields_ = [(n, C.c_int) for n in FIELDS]


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("plan") / "plan_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-fPIC", "-shared", "-Wl,-Bsymbolic",
                    "-I", os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"),
                    os.path.join(HERE, "plan_host.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    lib.fake.restype = C.POINTER(Fake)
    lib.dsq_plan_run.argtypes = [C.c_void_p, C.c_void_p]
    lib.dsq_plan_free.argtypes = [C.c_void_p]
    return lib


@pytest.fixture
def lib(built):
    C.memset(built.fake(), 0, C.sizeof(Fake))
    return built


def record(lib):
    plan = C.c_void_p()
    assert lib.dsq_plan_begin() == 0
    for _ in range(N):
        assert lib.record_launch() == 0
    assert lib.dsq_plan_end(C.byref(plan)) == 0
    return plan


def run(lib, plan):
    """Runs the plan; True when it went as a graph.  Either way its launches went once."""
    f = lib.fake().contents
    before = f.launches, f.graph_launches
    assert lib.dsq_plan_run(plan, None) == 0
    went = f.launches - before[0], f.graph_launches - before[1]
    assert went in ((N, 0), (0, 1))
    return went == (0, 1)


def all_given_back(lib, plan):
    f = lib.fake().contents
    lib.dsq_plan_free(plan)
    assert (f.streams, f.graphs, f.execs) == (0, 0, 0)
    assert lib.fake_mode() == 0           # the thread's capture mode is the caller's again


def test_graph_from_the_third_run(lib):
    plan = record(lib)
    assert [run(lib, plan) for _ in range(5)] == [False, False, True, True, True]
    f = lib.fake().contents
    assert (f.instantiate_calls, f.captured) == (1, N)
    f.caller_capturing = 1                # into a caller's capture: one by one
    assert not run(lib, plan)
    all_given_back(lib, plan)


@pytest.mark.parametrize("what", ["fail_instantiate", "fail_stream"])
def test_failed_graph_is_tried_again(lib, what):
    plan = record(lib)
    f = lib.fake().contents
    setattr(f, what, 1)
    assert not any(run(lib, plan) for _ in range(11))
    setattr(f, what, 0)                   # the third and the sixth run tried, the twelfth does
    assert [run(lib, plan) for _ in range(3)] == [True] * 3
    assert f.instantiate_calls == (3 if what == "fail_instantiate" else 1)
    all_given_back(lib, plan)


def test_capture_in_another_thread_is_left_alone(lib):
    plan = record(lib)
    f = lib.fake().contents
    f.capture_elsewhere = 1
    assert [run(lib, plan) for _ in range(4)] == [False, False, True, True]
    all_given_back(lib, plan)
    assert not f.broken


def test_no_memory_for_a_record(lib):
    """An entry point returns a status, and throws nothing, where its launch cannot be kept."""
    f = lib.fake().contents
    plan = C.c_void_p()
    assert lib.dsq_plan_begin() == 0
    f.no_memory = 1
    assert lib.record_launch() == -5
    f.no_memory = 0
    assert lib.dsq_plan_end(C.byref(plan)) == -5 and not plan
    all_given_back(lib, record(lib))
