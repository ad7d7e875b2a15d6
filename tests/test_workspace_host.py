"""The read of a workspace's status on a fake CUDA runtime: without page-locked memory,
with a workspace of another device, beside a capture in another thread."""
import ctypes as C
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
FIELDS = ("host_allocs host_frees kernels copies syncs fail_host_alloc device_of_ws capture_elsewhere "
          "broken pdl dependent schedule late waited").split()


class Fake(C.Structure):
    _fields_ = [(n, C.c_int) for n in FIELDS]


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("workspace") / "workspace_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-fPIC", "-shared", "-pthread", "-Wl,-Bsymbolic",
                    "-I", os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"),
                    os.path.join(HERE, "workspace_host.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    lib.fake.restype = C.POINTER(Fake)
    return lib


@pytest.mark.parametrize("change,by_kernel", [({}, True), (dict(capture_elsewhere=1), True),
                                              (dict(fail_host_alloc=1), False),
                                              (dict(device_of_ws=1), False)])
def test_status(built, change, by_kernel):
    C.memset(built.fake(), 0, C.sizeof(Fake))
    f = built.fake().contents
    for k, v in change.items():
        setattr(f, k, v)
    ws = (C.c_int * 64)()
    for status in (0, -10, -6):
        ws[0], ws[1] = status, 31
        assert built.status_of_new_thread(ws, 3) == status
        if status:
            assert (ws[0], ws[1]) == (0, 0)
    assert (f.kernels, f.copies) == ((9, 0) if by_kernel else (0, 9))
    assert f.syncs == 9 and not f.broken
    # one word a thread, given back when the thread ends
    assert f.host_allocs == f.host_frees == (0 if "fail_host_alloc" in change else 3)


@pytest.mark.parametrize("pdl", [0, 1])
def test_dependent_launch_hook(built, pdl):
    C.memset(built.fake(), 0, C.sizeof(Fake))
    f = built.fake().contents
    f.pdl = pdl
    assert built.status_of_new_thread((C.c_int * 64)(), 3) == 0
    assert (f.kernels, f.dependent) == (3, 3 * pdl)


@pytest.mark.parametrize("schedule,watched", [(0, True), (1, True), (2, False), (4, False)])
def test_watch_follows_the_schedule_flags(built, schedule, watched):
    """cudaDeviceScheduleAuto, Spin, Yield, BlockingSync: the word is watched (up to 200 us) only
    where CUDA's own wait would spin, too."""
    C.memset(built.fake(), 0, C.sizeof(Fake))
    f = built.fake().contents
    f.schedule, f.late = schedule, 1
    ws = (C.c_int * 64)()
    ws[0] = -10
    assert built.status_of_new_thread(ws, 20) == -10 and f.syncs == 20
    assert (f.waited >= 200) == watched       # the shortest of the twenty
