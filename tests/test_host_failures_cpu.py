"""What the library's host code does when a runtime call or a device-side wait
fails, on the CPU: fredopt_api.cu compiled over a stand-in CUDA runtime whose
"kernels" compute nothing (fake_cuda.cpp).  No GPU is involved."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2509_20012_gb300 import fredopt

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    if not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I",
                           os.path.join(ROOT, "include"), "-I", os.path.join(CUDA, "include"),
                           os.path.join(ROOT, "tests", "fake_cuda.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    for name, (res, args) in fredopt._SIGS.items():
        if hasattr(lib, name):
            getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    lib.fake_used.restype = lib.fake_peak.restype = ctypes.c_size_t
    lib.fake_limit.argtypes = [ctypes.c_size_t]
    yield lib
    lib.fake_limit(2 ** 63)


class Plan:
    """A handle of the stand-in library with n_vox rows of `per` nonzeros."""

    def __init__(self, lib, n_vox, per, n=64):
        self.lib, self.n = lib, n
        self.h = ctypes.c_void_p()
        assert lib.fredopt_create(ctypes.byref(self.h), 0, None) == 0
        assert self.load(n_vox, per) == 0

    def load(self, n_vox, per, fmt=0):
        rp = np.arange(n_vox + 1, dtype=np.int64) * per
        col = np.zeros(n_vox * per, np.int32)
        val = np.zeros(n_vox * per, np.float32)
        mask = np.ones(n_vox, np.uint32)
        return self.lib.fredopt_load_influence(self.h, n_vox, self.n, n_vox * per, rp.ctypes.data, col.ctypes.data,
                                               val.ctypes.data, val.ctypes.data, mask.ctypes.data, fmt, 0)

    def begin(self, **kw):
        p = fredopt.Params(beta0=-1.0, eta=1.0, reductions=1, max_trials=50, c_cdl=0.04, use_graphs=0, tile_balance=1)
        for k, v in kw.items():
            setattr(p, k, v)
        w0 = np.ones(self.n, np.float32)
        return self.lib.fredopt_begin(self.h, w0.ctypes.data, 0.99, 1.0, ctypes.byref(p), 0)

    def end(self):
        return self.lib.fredopt_end(self.h, None, None, None, None, 0)

    def close(self):
        self.lib.fredopt_destroy(self.h)


def test_begin_drops_the_error_of_an_abandoned_solve(fake):
    """A wait that gave up in a solve that is never ended belongs to that solve:
    the next one on the handle, alone or in a batch, does not report it."""
    a = Plan(fake, 50, 3)
    assert a.begin() == 0
    fake.fake_fail_waits(1)
    assert fake.fredopt_iterate(a.h, 2) == 0
    assert a.begin() == 0
    assert fake.fredopt_iterate(a.h, 2) == 0
    assert a.end() == 0
    # in a batch: reported by its synchronisation, and by that call alone
    b = ctypes.c_void_p()
    hs = (ctypes.c_void_p * 1)(a.h)
    for give_up in (1, 0):
        assert a.begin() == 0
        fake.fake_fail_waits(give_up)
        assert fake.fredopt_batch_create(ctypes.byref(b), hs, 1) == 0  # the stand-in runs what is captured
        assert fake.fredopt_batch_sync(b, None) == (fredopt.ERR_TIMEOUT if give_up else 0)
        assert fake.fredopt_batch_destroy(b) == 0
    a.close()


@pytest.mark.parametrize("per", [1, 40])
def test_reload_frees_the_old_plan_when_memory_runs_out(fake, per):
    """A reload for which there is no room beside the old plan's buffers, from the
    first allocation on, frees them and loads: whatever fits on its own fits."""
    sizes = (4000, 3000)
    alone = []  # peak of each plan in a fresh handle
    for n_vox in sizes:
        fake.fake_limit(2 ** 63)
        before = fake.fake_used()
        p = Plan(fake, n_vox, per)
        alone.append(fake.fake_peak() - before)
        p.close()
        assert fake.fake_used() == before
    p = Plan(fake, sizes[0], per)
    assert p.begin() == 0 and p.end() == 0
    held = fake.fake_used()
    base = held  # every handle before is closed
    for room in list(range(0, 4 * alone[1], alone[1] // 16)):
        limit = max(held + room, 0)
        fake.fake_limit(limit)
        rc = p.load(sizes[1], per)
        if limit >= alone[1]:
            assert rc == 0, (room, rc)
        fake.fake_limit(2 ** 63)
        assert p.load(sizes[0], per) == 0
        held = fake.fake_used()
    p.close()
    assert fake.fake_used() < base


def test_checked_lengths_hold_for_every_array(fake):
    """The element count that checked builds test ranges against is one that each of
    the arrays has, also where a reload kept longer buffers for some of them."""
    INDEX32, ROI = 0x200, 0x100
    p = Plan(fake, 300, 20)
    x, a, u = np.ones(p.n, np.float32), np.ones(2000, np.float32), np.zeros(2000, np.float32)
    con = (fredopt.Constraint * 1)(fredopt.Constraint(0, 0, 1.0, 1.0))
    for n_vox, per, fmt in ((300, 20, INDEX32), (200, 20, 0), (300, 20, 1), (250, 21, INDEX32 | 2), (300, 20, 0),
                            (160, 20, INDEX32 | ROI), (160, 39, 1), (1200, 20, 0), (700, 20, 2)):
        assert p.load(n_vox, per, fmt) == 0
        assert p.lib.fredopt_set_constraints(p.h, 1, con) == 0
        assert p.lib.fredopt_forward(p.h, x.ctypes.data, u.ctypes.data, None, 0) == 0
        assert p.lib.fredopt_backward(p.h, a.ctypes.data, a.ctypes.data, u.ctypes.data, 0) == 0
        assert p.lib.fredopt_sweep_step(p.h, x.ctypes.data, 1.0, 1.0, 0, 3, u.ctypes.data, 0) == 0
        assert fake.fake_long_checks() == 0, (n_vox, per, fmt)
    p.close()


@pytest.mark.parametrize("fmt", [0, 1, 2])
def test_autotune_can_keep_the_weights_of_a_load(fake, fmt):
    """The tile weights that a load sets are among those that fredopt_autotune times
    and returns (rows 16..512 and chunks 4..1024, as test_gpu_batch has them)."""
    p = Plan(fake, 100, 20)
    assert p.load(100, 20, fmt) == 0
    r, c = ctypes.c_int64(), ctypes.c_int64()
    assert fake.fredopt_get_tuning(p.h, ctypes.byref(r), ctypes.byref(c)) == 0
    assert r.value in (16, 32, 64, 128, 256, 512) and c.value in (4, 16, 64, 256, 1024)
    p.close()


def test_the_barrier_of_the_forward_product_has_its_own_place(fake):
    """Behind x (4 bytes per spot) and behind the 512 bytes of the reduction that is
    written over x, on an 8-byte boundary, for every padded number of spots."""
    fake.fake_bar_offset.restype = ctypes.c_size_t
    for n_pad in (4, 8, 60, 124, 128, 132, 30000, 58100):
        at = fake.fake_bar_offset(n_pad)
        assert at == max(4 * n_pad, 512) and at % 8 == 0


def test_a_capture_that_cannot_start_leaves_plain_launches(fake):
    """After a begin whose stream capture is refused, a begin without graphs runs and
    times its iterations as plain launches: no event is recorded as a graph node."""
    p = Plan(fake, 50, 3)
    assert fake.fredopt_set_timing(p.h, 1) == 0
    fake.fake_fail_captures(1)
    assert p.begin(use_graphs=1) == -7
    assert p.begin(use_graphs=0) == 0
    assert fake.fredopt_iterate(p.h, 2) == 0
    assert p.end() == 0
    assert fake.fake_stray_external() == 0
    p.close()


def test_a_single_sweep_leaves_the_solve_its_blocks(fake):
    """A begun solve that sweeps 4 blocks, in plain launches or captured in a batch,
    goes on with its own 4 after a single sweep of 7, whose tables are not built in
    the place of the solve's."""
    p = Plan(fake, 100, 3)
    con = (fredopt.Constraint * 1)(fredopt.Constraint(0, 0, 1.0, 1.0))
    assert fake.fredopt_set_constraints(p.h, 1, con) == 0
    x, w = np.ones(p.n, np.float32), np.zeros(p.n, np.float32)
    sweep = lambda n: fake.fredopt_sweep_step(p.h, x.ctypes.data, 1.0, 1.0, 0, n, w.ctypes.data, 0)
    assert p.begin(sweep_blocks=4) == 0
    b = ctypes.c_void_p()
    fake.fake_sweep_blocks()
    assert fake.fredopt_batch_create(ctypes.byref(b), (ctypes.c_void_p * 1)(p.h), 1) == 0
    assert fake.fake_sweep_blocks() == 4
    fake.fake_capture_pos()
    assert sweep(7) == 0 and fake.fake_sweep_blocks() == 7
    assert fake.fake_captured_alive() == 1
    assert fake.fredopt_iterate(p.h, 2) == 0 and fake.fake_sweep_blocks() == 8
    assert sweep(4) == 0 and fake.fake_sweep_blocks() == 4
    assert fake.fredopt_batch_destroy(b) == 0
    # a captured solve refuses another number, as it did
    assert p.begin(sweep_blocks=4, use_graphs=1) == 0
    assert sweep(7) == -1
    p.close()
