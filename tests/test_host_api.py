"""The host side of the C ABI (csrc/sim_api.cpp) on the CPU, compiled against a fake CUDA runtime
(tests/host/fake_cuda.cpp): what is ordered before what, and what happens when memory runs out."""
import ctypes
import shutil
import subprocess
from pathlib import Path

import numpy as np
import pytest

from tests.conftest import ROOT

A_MIN, NOMEM = 1, -6


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2508_14544_gb300.build import nvcc
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    cuda = Path(nvcc()).resolve().parent.parent / "include"
    so = tmp_path_factory.mktemp("host") / "libhost.so"
    csrc = ROOT / "paper_2508_14544_gb300" / "csrc"
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", f"-I{ROOT / 'include'}", f"-I{csrc}",
                    f"-I{cuda}", str(csrc / "sim_api.cpp"), str(ROOT / "tests" / "host" / "fake_cuda.cpp"), "-o", str(so)],
                   check=True)
    lib = ctypes.CDLL(str(so))
    for f in ("fake_used", "fake_seed"):
        getattr(lib, f).restype = ctypes.c_uint64
    for f in ("fake_slots", "fake_rho_calls"):
        getattr(lib, f).restype = ctypes.c_int64
    lib.fake_stream.restype = ctypes.c_void_p
    lib.fake_limits.argtypes = [ctypes.c_size_t, ctypes.c_size_t]
    lib.sim_last_error.restype = ctypes.c_char_p
    yield lib
    lib.fake_limits(1 << 40, (1 << 64) - 1)


class Ctx:
    def __init__(self, lib, n_inst, policy=A_MIN):
        self.lib, self.n, self.h = lib, n_inst, ctypes.c_void_p()
        assert lib.sim_create(policy, ctypes.c_int64(1000), n_inst, ctypes.byref(self.h)) == 0

    def load(self, sizes):
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        x = np.ones(16, np.int32)  # device pointers: never read here
        p = ctypes.c_void_p(x.ctypes.data)
        return self.lib.sim_load_csr(self.h, ctypes.c_void_p(off.ctypes.data), p, p, p, p, p, 1)

    def run(self, stream=None):
        self.out = np.zeros(7 * self.n, np.int64)
        return self.lib.sim_run(self.h, ctypes.c_void_p(self.out.ctypes.data), ctypes.c_void_p(stream))

    def seeds(self, values):
        v = np.array(values, np.uint64)
        return self.lib.sim_set_tie_seeds(self.h, ctypes.c_void_p(v.ctypes.data))

    def close(self):
        self.lib.sim_destroy(self.h)


@pytest.mark.parametrize("n_inst", [2, 20000])
def test_a_run_finds_the_tie_seeds_just_set(lib, n_inst):
    """Also on a stream that does not wait for the legacy default stream, with or without a load between, and
    when they are set twice."""
    c = Ctx(lib, n_inst)
    stream = lib.fake_stream()
    for first, load in ((7, True), (8, False), (9, True), (10, False)):
        assert c.seeds([99] * n_inst) == 0 and c.seeds([first] * n_inst) == 0
        assert not load or c.load([3] * n_inst) == 0
        assert c.run(stream) == 0
        assert lib.fake_seed() == first
    c.close()


def test_a_load_that_fits_succeeds_after_one_that_did_not(lib):
    """The failed allocation is reported once: no later launch takes it for an error of its own."""
    c = Ctx(lib, 1)
    lib.fake_limits(lib.fake_used() + 10**6, (1 << 64) - 1)
    assert c.load([1_000_000]) == NOMEM
    assert c.load([100]) == 0 and c.run() == 0
    lib.fake_limits(1 << 40, (1 << 64) - 1)
    c.close()
    assert lib.fake_used() == 0
    lib.fake_limits(10**6, (1 << 64) - 1)
    u, out = np.array([1 << 20], np.int32), np.zeros(1)
    rho = lambda: lib.sim_cr_amin_rho(1, ctypes.c_void_p(u.ctypes.data), ctypes.c_void_p(out.ctypes.data))
    assert rho() == NOMEM
    u[0] = 9
    assert rho() == 0 and out[0] == 9
    lib.fake_limits(1 << 40, (1 << 64) - 1)


def test_runs_with_fewer_warps_when_the_queue_buffers_do_not_fit(lib):
    """The queue buffers of a launch take 32 bytes x largest instance per simulating warp: 292 GB for one of five
    million on 12 warps per SM.  With 100 GB left fewer warps simulate, also in the global-memory re-run, whose
    workspace needs room too."""
    for status in (0, -100):  # -100: every instance outgrew the shared-memory slots
        c = Ctx(lib, 3000)
        assert c.load([5_000_000] + [2] * 2999) == 0
        lib.fake_status(status)
        lib.fake_limits(lib.fake_used() + 100 * 10**9, (1 << 64) - 1)
        assert c.run() == 0 and 200 <= lib.fake_slots() <= 600
        lib.fake_limits(lib.fake_used() + 10**6, (1 << 64) - 1)
        assert c.run() == 0  # the same buffers again
        c.close()
        lib.fake_status(0)
        lib.fake_limits(1 << 40, (1 << 64) - 1)
    assert lib.fake_used() == 0


def test_rho_works_in_smaller_batches_when_its_scratch_does_not_fit(lib):
    """18 values of 2^20 ask for 1 GB of scratch at once (59 MB each): with 300 MB left they are computed in
    batches of a few, with the same results."""
    u, out = np.full(18, 1 << 20, np.int32) - np.arange(18, dtype=np.int32), np.zeros(18)
    for room in (1 << 40, lib.fake_used() + 300 * 10**6):
        lib.fake_limits(room, (1 << 64) - 1)
        out[:] = 0
        assert lib.sim_cr_amin_rho(18, ctypes.c_void_p(u.ctypes.data), ctypes.c_void_p(out.ctypes.data)) == 0
        assert np.array_equal(out, u)
    lib.fake_limits(1 << 40, (1 << 64) - 1)
    assert lib.fake_used() == 0


@pytest.mark.parametrize("entry", ["csr", "uniform", "redo"])
def test_host_memory_that_runs_out_is_an_error_code(lib, entry):
    """No exception leaves the C entry points, and the context works again once there is memory."""
    n = 20000  # results above 16384 instances are kept in ordinary memory: 1.1 MB
    c = Ctx(lib, n)
    one = np.ones(16, np.int32)
    p = ctypes.c_void_p(one.ctypes.data)
    if entry == "redo":  # the list of the instances to run again takes 80 kB
        lib.fake_status(-100)
        assert c.load([2] * n) == 0
    lib.fake_limits(1 << 40, 50_000)
    for _ in range(2):
        assert (c.run() if entry == "redo" else c.load([2] * n) if entry == "csr" else
                lib.sim_load(c.h, 2, p, p, p, p, p, 1)) == NOMEM
    lib.fake_limits(1 << 40, (1 << 64) - 1)
    assert c.load([2] * n) == 0 and c.run() == 0
    lib.fake_status(0)
    c.close()
