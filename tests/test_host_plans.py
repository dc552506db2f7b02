"""The launches that the library's host side makes of a call, on the CPU:
csrc/apc_host.cpp is compiled as it is against a stand-in for the CUDA
runtime and the kernels (host_stub.cpp) that records what it is asked."""
import ctypes
import os
import shutil
import subprocess

import pytest

import oracle
import paper_2609_18178_gb300 as apc
from paper_2609_18178_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
BASE = 1 << 40   # fake device addresses, one GB apart per kind of buffer
SMS = 152


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc")) or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    so = str(tmp_path_factory.mktemp("host") / "libhost.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-fvisibility=hidden", "-Wl,-Bsymbolic", "-I", cuda,
                    "-I", _build.CSRC, os.path.join(_build.CSRC, "apc_host.cpp"), os.path.join(HERE, "host_stub.cpp"),
                    "-o", so], check=True)
    out = ctypes.CDLL(so)
    out.apc_last_error.restype = ctypes.c_char_p
    for f in (out.stub_runtime_queries, out.stub_range_queries, out.stub_launches):
        f.restype = ctypes.c_long
    out.stub_limit.restype = ctypes.c_float
    out.stub_reset.argtypes = [ctypes.c_uint64, ctypes.c_int]
    yield out
    out.apc_set_reserved_sms(0)


def call(lib, what, count, n=300, step=3, **hp):
    """One call over `count` tensors or buffers of n elements each; its status."""
    out = ctypes.c_void_p(BASE + (7 << 30))
    if what == "commit":
        h = dict(oracle.DEFAULT_HP, **hp)
        hp = apc._HParams(h["lr"], h["beta1"], h["beta2"], h["eps"], h["weight_decay"])
        arr = (apc._Tensor * count)()
        for k in range(count):
            at = [BASE + (i << 30) + (4 if i < 3 else 2) * k * (n + 4) for i in range(5)]
            arr[k] = apc._Tensor(*at, n, k * n)
        return lib.apc_commit_step(arr, count, ctypes.byref(hp), ctypes.c_int64(step), None, out)
    arr = (apc._Buffer * count)()
    for k in range(count):
        arr[k] = apc._Buffer(BASE + 4 * k * (n + 4), n, k * n, apc.F32, 0)
    return (lib.apc_digest if what == "digest" else lib.apc_count_nonzero)(arr, count, 1, None, out)


def launches(lib):
    buf = (ctypes.c_int64 * 64)()
    k = lib.stub_launches(buf, 16)
    return [dict(zip(("count", "grid", "more", "chained"), buf[4 * i:4 * i + 4])) for i in range(k)]


PER_SM = dict(commit=1, digest=1, count=2)   # resident CTAs, as the stand-in answers


@pytest.mark.parametrize("what,count", [("commit", 1100), ("digest", 2300), ("count", 2300)])
@pytest.mark.parametrize("reserved,limit", [(0, None), (8, None), (0, 20), (0, 10_000), (151, 1)])
def test_long_tables_leave_the_sms_free_that_they_are_told_to(lib, monkeypatch, what, count, reserved, limit):
    """A launch that lets the next one start early hands it every SM that is
    free, also those that the grid's cap was to leave free: a call's launches
    are chained only where their grid may take the whole GPU."""
    monkeypatch.delenv("APC_GRID_LIMIT", raising=False)
    if limit:
        monkeypatch.setenv("APC_GRID_LIMIT", str(limit))
    lib.stub_reset(0, 0)
    assert lib.apc_set_reserved_sms(reserved) == 0
    assert call(lib, what, count) == 0
    got = launches(lib)
    assert len(got) == 3 and sum(x["count"] for x in got) == count
    whole = SMS * PER_SM[what]
    cap = min((SMS - reserved) * PER_SM[what], limit or whole)
    assert all(x["grid"] <= cap for x in got)
    chained = cap == whole
    assert [x["more"] for x in got] == [int(chained)] * 2 + [0]
    assert [x["chained"] for x in got] == [0] + [int(chained)] * 2


@pytest.mark.parametrize("what,count,addresses,arenas", [("commit", 1100, 5501, 6), ("digest", 2300, 2301, 2), ("count", 2300, 2301, 2)])
@pytest.mark.parametrize("virtual", ["none", "all", "some"])
def test_pointer_queries_by_kind_of_memory(lib, what, count, addresses, arenas, virtual):
    """One attribute query and one range query per allocation of cudaMalloc's.
    Memory of the virtual-memory interface is asked address by address, and the
    failed range queries beside that stay a handful, however long the table; a
    list that begins in such memory still finds its way back."""
    lib.stub_reset({"none": 0, "all": 1 << 63, "some": BASE + (1 << 30)}[virtual], 0)
    assert call(lib, what, count) == 0
    asked, ranges = lib.stub_runtime_queries(), lib.stub_range_queries()
    if virtual == "none":
        assert asked == ranges == arenas
    elif virtual == "all":
        assert asked == addresses and ranges <= 13
    else:     # the first arena, p's or the whole list's, is virtual memory
        assert count <= asked <= 2 * count + 2 * arenas and ranges <= 13 + arenas


@pytest.mark.parametrize("what", ["commit", "digest", "count"])
def test_a_refused_launch_leaves_no_error_pending(lib, what):
    """An error that a call has returned is not left with the runtime for the
    caller's next check, or this library's next launch, to find."""
    lib.stub_reset(0, 9)
    assert call(lib, what, 3) == 4                      # APC_ECUDA
    assert b"launch" in lib.apc_last_error()
    assert lib.stub_pending() == 0


@pytest.mark.parametrize("hp,step,limit", [
    (dict(), 1, 2.0**30), (dict(eps=1e-6, beta2=0.999), 5, 2.0**30), (dict(eps=2.0**-32), 9, 2.0**30),
    (dict(eps=1e-15), 3, 1e-15 * 2**62), (dict(eps=1e-16), 3, 1e-16 * 2**62), (dict(eps=2.0**-60), 100, 4.0),
    (dict(lr=0.0), 1, 2.0**30), (dict(beta2=1 - 1e-12), 1, 2.0**30), (dict(eps=300.0), 1, 2.0**30),
    # the root of the addend in den, a step or a quotient out of binary32's normal range: the general operations
    (dict(eps=2.0**-69, beta2=0.95), 1, -1), (dict(eps=1e-30), 5, -1), (dict(eps=1e-16, beta2=1 - 1e-15), 1, -1),
    (dict(lr=1e-25), 5, -1), (dict(lr=1e7), 5, -1)])
def test_bounds_of_the_grouped_update(lib, hp, step, limit):
    """Up to which |m'| + den a group's square root and quotient keep to the
    grouped form: what a job sets, and moments of unscaled or summed gradients,
    lie well inside."""
    lib.stub_reset(0, 0)
    assert call(lib, "commit", 3, step=step, **hp) == 0
    assert lib.stub_limit() == pytest.approx(limit, rel=1e-6)
