"""The library's host side on a fake CUDA runtime (tests/host/fake_cudart.cpp):
calls that fail, several devices, little memory.  Nothing here needs a GPU."""
import ctypes
import glob
import os
import subprocess
import time

import numpy as np
import pytest

from paper_2405_02603_gb300 import build as B

OK = 0
F64, F32, F64_DF = 0, 1, 2
HE = 0
VP = ctypes.c_void_p


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    here = os.path.dirname(os.path.abspath(__file__))
    objects = lambda: glob.glob(os.path.join(B.OUT_DIR, "*.o"))  # noqa: E731
    B.build(force=len(objects()) < len(B.sources()))
    names = {os.path.basename(s)[:-3] + ".o" for s in B.sources()}
    out = str(tmp_path_factory.mktemp("fake") / "libfsp_fake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    # its own CUDA runtime, whatever else the process has loaded
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", cuda,
                    os.path.join(here, "host", "fake_cudart.cpp")] +
                   [o for o in objects() if os.path.basename(o) in names] + ["-o", out], check=True)
    L = ctypes.CDLL(out)
    i, d = ctypes.c_int, ctypes.c_double
    L.fsp_plan_create.argtypes = [ctypes.POINTER(VP), i, d, d, i, i, VP]
    L.fsp_solve.argtypes = [VP, VP, VP, VP]
    L.fsp_plan_destroy.argtypes = [VP]
    L.fsp_batch_create.argtypes = [ctypes.POINTER(VP), ctypes.POINTER(VP), ctypes.POINTER(VP), ctypes.POINTER(VP), i, VP]
    for f in ("launch", "wait", "autotune"):
        getattr(L, "fsp_batch_" + f).argtypes = [VP, VP]
    L.fsp_batch_set_timeout.argtypes = [VP, d]
    L.fsp_batch_set_form.argtypes = [VP, i]
    L.fsp_batch_destroy.argtypes = [VP]
    L.fsp_server_create.argtypes = [ctypes.POINTER(VP), ctypes.c_size_t, i]
    L.fsp_server_submit.argtypes = [VP, i, d, i, i, VP, VP, ctypes.POINTER(ctypes.c_uint64)]
    L.fsp_server_poll.argtypes = [VP, ctypes.c_uint64, ctypes.POINTER(i), ctypes.POINTER(d)]
    L.fsp_server_destroy.argtypes = [VP]
    for f in ("fake_used", "fake_idle"):
        getattr(L, f).restype = ctypes.c_size_t
    L.fake_violations.restype = ctypes.c_long
    L.fake_capacity.argtypes = [ctypes.c_size_t]
    L.fake_fail.argtypes = [ctypes.c_char_p, i, i]
    L.fake_failed.argtypes = [ctypes.c_char_p]
    return L


def plan(L, N, dtype=F64, algo=HE):
    p = VP()
    assert L.fsp_plan_create(ctypes.byref(p), N, 1.0, 1.0 / N, algo, dtype, None) == OK
    return p


class Arrays:
    """16-byte aligned arrays of N^3 reals."""

    def __init__(self, Ns, dtype):
        self.keep = [np.zeros(n ** 3 + 4, np.float32 if dtype == F32 else np.float64) for n in Ns]
        self.ptrs = (VP * len(Ns))(*[(a.ctypes.data + 15) // 16 * 16 for a in self.keep])


class BatchOf:
    def __init__(self, L, Ns, dtype):
        self.L, self.plans = L, [plan(L, N, dtype) for N in Ns]
        self.rho, self.phi = Arrays(Ns, dtype), Arrays(Ns, dtype)
        self.b = VP()
        assert L.fsp_batch_create(ctypes.byref(self.b), (VP * len(Ns))(*[p.value for p in self.plans]), self.rho.ptrs,
                                  self.phi.ptrs, len(Ns), None) == OK

    def usable(self):
        """Launches, on live memory."""
        before = self.L.fake_violations()
        return self.L.fsp_batch_launch(self.b, None) == OK and self.L.fsp_batch_wait(self.b, None) == OK and \
            self.L.fake_violations() == before

    def close(self):
        assert self.L.fsp_batch_destroy(self.b) == OK
        for p in self.plans:
            assert self.L.fsp_plan_destroy(p) == OK


@pytest.mark.parametrize("dtype,Ns", [(F32, [160, 128]), (F64, [75, 128])])
def test_batches_of_different_sizes_live_together(fake, dtype, Ns):
    """The kernel's shared-memory attribute belongs to the process: a batch of
    small plans must not take it from one of large plans."""
    L = fake
    L.fake_reset(1)
    big = BatchOf(L, Ns, dtype)
    small = BatchOf(L, [32, 32], dtype)
    assert L.fsp_batch_set_timeout(big.b, 500.0) == OK
    assert big.usable() and small.usable()
    big.close()
    small.close()


@pytest.mark.parametrize("dtype", [F64, F32])
@pytest.mark.parametrize("call", [b"alloc", b"copy", b"stream", b"capture", b"instantiate"])
def test_failed_rebuild_leaves_the_batch(fake, dtype, call):
    """Whichever of its calls fails, the autotuner returns an error and the
    batch runs on, with live memory; so do set_timeout and set_form."""
    L = fake
    L.fake_reset(1)
    b = BatchOf(L, [32, 64] if dtype == F32 else [16, 20], dtype)
    assert b.usable()
    nth, failed = 0, 0
    while True:
        L.fake_fail(call, nth, 3 if call == b"alloc" else 1)  # an allocation is tried three times
        st = L.fsp_batch_autotune(b.b, None)
        hit = L.fake_failed(call)
        L.fake_fail_none()
        assert b.usable(), nth
        if not hit:
            break
        failed += st != OK
        nth += 1 if nth < 12 else 7
    assert failed >= 3 and st == OK
    if call in (b"stream", b"capture", b"instantiate"):
        for change in (lambda: L.fsp_batch_set_timeout(b.b, 20.0), lambda: L.fsp_batch_set_form(b.b, 1)):
            L.fake_fail(call, 0, 1)
            assert change() != OK
            L.fake_fail_none()
            assert b.usable()
            assert change() == OK and b.usable()
    b.close()


def test_buffers_wait_for_their_own_device(fake):
    """A buffer goes back to the pool when the work on its own device is done,
    whichever device is current, also when a capture kept it from going at first."""
    L = fake
    L.fake_reset(2)
    used = [L.fake_used(d) for d in (0, 1)]
    a = Arrays([16, 16], F64)
    on = {}
    for d in (0, 1):
        assert L.cudaSetDevice(d) == 0
        on[d] = [plan(L, 16), plan(L, 16)]
    assert L.fsp_solve(on[1][0], a.ptrs[0], a.ptrs[1], None) == OK  # device 1 is current
    L.cudaSetDevice(0)
    assert L.fsp_plan_destroy(on[1][0]) == OK
    assert L.fake_violations() == 0
    # device 0: refused while a stream is in capture, then freed from device 1
    stream, graph = VP(), VP()
    assert L.cudaStreamCreateWithFlags(ctypes.byref(stream), 1) == 0
    assert L.fsp_solve(on[0][0], a.ptrs[0], a.ptrs[1], None) == OK
    L.cudaStreamBeginCapture(stream, 1)
    L.fsp_plan_destroy(on[0][0])
    L.cudaStreamEndCapture(stream, ctypes.byref(graph))
    L.cudaSetDevice(1)
    assert L.fsp_plan_destroy(on[1][1]) == OK
    assert L.fake_violations() == 0
    assert L.fake_used(0) > used[0]
    L.cudaSetDevice(0)
    assert L.fsp_plan_destroy(on[0][1]) == OK
    assert L.fake_violations() == 0
    assert [L.fake_used(d) for d in (0, 1)] == used


def test_kept_memory_is_within_reach(fake):
    """What the library keeps of destroyed plans serves its other allocations
    on a full device, and goes back on request."""
    L = fake
    L.fake_reset(2)  # as many as the tests before made pools on
    used = L.fake_used(0)
    assert L.fsp_memory_trim() == OK and L.fake_idle(0) == 0
    for _ in range(3):
        p = plan(L, 96, F32)
        most = L.fake_used(0)
        assert L.fsp_plan_destroy(p) == OK
    kept = L.fake_idle(0)
    assert L.fake_used(0) == used and 0 < most - used <= kept <= 1 << 30
    # a server's workspace (N = 64: 7.9 MB), with half that much free
    L.fake_capacity(used + kept + (4 << 20))
    v, ticket, state = VP(), ctypes.c_uint64(), ctypes.c_int()
    a = Arrays([64, 64], F32)
    assert L.fsp_server_create(ctypes.byref(v), 1 << 30, 1) == OK
    assert L.fsp_server_submit(v, 64, 1.0, HE, F32, a.ptrs[0], a.ptrs[1], ctypes.byref(ticket)) == OK
    for _ in range(1000):
        assert L.fsp_server_poll(v, ticket, ctypes.byref(state), None) == OK
        if state.value >= 2:
            break
        time.sleep(0.01)
    assert state.value == 2
    assert L.fsp_server_destroy(v) == OK
    assert L.fake_idle(0) > 0
    # another allocator, which needs all of it
    q = VP()
    left = used + kept + (4 << 20) - L.fake_used(0)
    assert L.cudaMalloc(ctypes.byref(q), ctypes.c_size_t(left)) != 0
    assert L.fsp_memory_trim() == OK and L.fake_idle(0) == 0
    assert L.cudaMalloc(ctypes.byref(q), ctypes.c_size_t(left)) == 0
    assert L.cudaFree(q) == 0 and L.fake_violations() == 0
