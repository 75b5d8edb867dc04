"""Host logic of the C ABI on a machine without a GPU: csrc/qs_api.cu compiled
as C++ against a stand-in CUDA runtime (fake_cuda.cpp)."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2306_09537_gb300", "csrc")
DEVICE, PAGE_LOCKED, MANAGED = 2, 1, 3  # cudaMemoryType
STREAM = 0x1000  # any stream but the legacy default one


@pytest.fixture(scope="module")
def api(tmp_path_factory):
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))),
                        "include")
    out = str(tmp_path_factory.mktemp("api") / "libapi.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-fPIC", "-shared", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC,
                    "-I" + cuda, "-x", "c++", os.path.join(CSRC, "qs_api.cu"), os.path.join(HERE, "fake_cuda.cpp"), "-o", out,
                    "-Wl,-Bsymbolic", "-lpthread"], check=True)
    from paper_2306_09537_gb300 import qs  # for the configuration's layout
    lib = C.CDLL(out)
    V, I = C.c_void_p, C.c_int32
    lib.qs_create.argtypes = [C.POINTER(qs.qs_config), V, C.POINTER(V)]
    lib.qs_step.argtypes = [V, V, V, V, V]
    lib.qs_rollout.argtypes = [V, I, V, V, V, V]
    lib.qs_reset.argtypes = [V, C.c_uint64, V, V]
    lib.qs_destroy.argtypes = [V]
    lib.fake_set_kind.argtypes = [V, I]
    lib.qs = qs
    return lib


@pytest.fixture
def handle(api, request):
    swarm = getattr(request, "param", 8)
    cfg = api.qs.make_config(4, swarm, 0 if swarm == 1 else 2, ("floor", "walls"), 1)
    h = C.c_void_p()
    assert api.qs_create(C.byref(cfg), STREAM, C.byref(h)) == 0
    yield h
    assert api.qs_destroy(h) == 0


def buffers(n=1 << 16):
    raw = (C.c_char * (2 * n + 64))()
    act = (C.addressof(raw) + 63) & ~63
    return raw, act, act + n


@pytest.mark.parametrize("handle", [1, 8], indirect=True)
def test_replayed_rollout_follows_the_kind_of_its_buffer(api, handle):
    """A graph holds whether rows may leave by bulk copies; an address that comes
    back as another kind of memory is captured again."""
    keep, act, obs = buffers()
    seen = []
    for kind in (DEVICE, DEVICE, PAGE_LOCKED, PAGE_LOCKED, MANAGED, DEVICE):
        api.fake_set_kind(obs, kind)
        before = api.fake_captures()
        assert api.qs_rollout(handle, 3, act, obs, None, None) == 0
        seen.append((api.fake_captures() - before, api.fake_bulk()))
    assert seen == [(1, 1), (0, 1), (1, 0), (0, 0), (0, 0), (1, 1)]


def test_replayed_rollout_follows_the_seed(api, handle):
    """A captured launch holds the Philox keys; a full reset that changes them is
    captured again, the same seed or a masked reset is not."""
    keep, act, obs = buffers()
    mask = (C.c_uint8 * 4)(1, 0, 0, 1)
    seen = []
    for seed, masked in ((None, False), (5, False), (5, False), (6, True), (5 + (1 << 32), False), (None, False)):
        if seed is not None:
            assert api.qs_reset(handle, seed, C.addressof(mask) if masked else None, None) == 0
        before = api.fake_captures()
        assert api.qs_rollout(handle, 3, act, obs, None, None) == 0
        seen.append(api.fake_captures() - before)
    assert seen == [1, 1, 0, 0, 1, 0]


def test_a_failed_launch_is_reported_once(api, handle):
    """The error a failed launch leaves with the runtime is taken by the call that
    reports it: later calls, whose launches check for one, must not find it."""
    keep, act, obs = buffers()
    calls = [lambda: api.qs_step(handle, act, obs, None, None), lambda: api.qs_rollout(handle, 2, act, obs, None, None),
             lambda: api.qs_reset(handle, 3, None, None)]
    for call in calls:
        api.fake_fail_next_launch(1)
        assert call() != 0
        assert api.fake_pending_error() == 0
        assert call() == 0
