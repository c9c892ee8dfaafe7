"""The handle's device scratch, on the CPU: the library's host side over a CUDA
runtime that only counts (fake_cuda.cpp)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_17018_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
GB = 1 << 30

pytestmark = pytest.mark.skipif(not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")), reason="no CUDA headers")


class _Hits(C.Structure):
    _fields_ = [("y", C.c_void_p), ("z", C.c_void_p), ("rowsec", C.c_void_p), ("n_hits", C.c_int64)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I" + os.path.join(ROOT, "include"),
                    "-I" + CSRC, "-I" + CUDA, os.path.join(CSRC, "tpcfit_host.cpp"),
                    os.path.join(ROOT, "tests", "fake_cuda.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    for f in ("fake_bytes", "fake_used", "fake_used_live"):
        getattr(L, f).restype = C.c_longlong
    return L


class Handle:
    """A handle over the fake, with `limit` bytes of device memory."""

    def __init__(self, lib, limit=256 * GB):
        from paper_2511_17018_gb300 import synth
        from paper_2511_17018_gb300 import tpcfit as tf
        fr = synth.generate(2, 1)
        rx = np.ascontiguousarray(fr.geometry.row_x, dtype=np.float64)
        g = tf._Geometry(36, rx.shape[0], rx.ctypes.data_as(C.POINTER(C.c_double)), 20.0, 250.0)
        self.L, self.h = lib, C.c_void_p()
        lib.fake_limit(C.c_longlong(limit))
        lib.fake_capture(0)
        lib.fake_forget()
        assert lib.tpcfit_create(C.byref(g), C.c_double(5.0), C.byref(self.h)) == 0
        lib.tpcfit_set_record(self.h, 1)

    def args(self, n, per):
        p = C.c_void_p(4096)  # (never followed: nothing runs)
        return [self.h, C.byref(_Hits(4096, 4096, 4096, n * per)), p, C.c_int32(n)], p

    def fit(self, n, per=100):
        a, p = self.args(n, per)
        return self.L.tpcfit_fit(*a, p, p, p, p, p, None)

    def backward(self, n, per=100):
        a, p = self.args(n, per)
        return self.L.tpcfit_fit_backward(*a, p, p, p, p, None, None)

    def smooth(self, n, per=100):
        a, p = self.args(n, per)
        return self.L.tpcfit_smooth(*a, p, p, p, p, None)

    def reject(self, n, per=100):
        a, p = self.args(n, per)
        return self.L.tpcfit_reject_outliers(*a, p, C.c_float(9.0), p, p, p, p, None)

    def close(self):
        self.L.fake_capture(0)
        self.L.tpcfit_destroy(self.h)
        assert self.L.fake_bytes() == 0  # everything is given back


def test_a_captured_call_keeps_its_scratch(lib):
    # fit + adjoint + smoother + rejection captured; whatever the handle does
    # afterwards, a replay finds the buffers that the graph holds
    h = Handle(lib)
    try:
        def calls(n):
            assert [h.fit(n), h.backward(n), h.smooth(n), h.reject(n)] == [0] * 4

        for det in (0, 1):
            lib.tpcfit_set_mode(h.h, det)
            calls(5000)
        lib.fake_forget()
        lib.fake_capture(1)
        for det in (0, 1):
            lib.tpcfit_set_mode(h.h, det)
            calls(5000)
        lib.fake_capture(0)
        used = lib.fake_used()
        assert lib.fake_taped() and used >= 8 and lib.fake_used_live() == used
        for n in (20000, 60000, 400000):
            for det in (1, 0):
                lib.tpcfit_set_mode(h.h, det)
                calls(n)
                lib.tpcfit_set_det_reduction(h.h, 1)
                assert h.backward(n) == 0
        assert lib.fake_used() > used  # they have grown, and
        assert lib.fake_used_live() == lib.fake_used()  # nothing that was in use since is gone
    finally:
        h.close()


def test_a_captured_handle_that_keeps_growing_stays_bounded(lib):
    sizes = [5000 + 400 * k for k in range(200)]
    total = []
    for capture in (0, 1):
        h = Handle(lib)
        try:
            assert h.fit(sizes[0]) == 0
            lib.fake_capture(capture)
            assert h.fit(sizes[0]) == 0
            lib.fake_capture(0)
            for n in sizes:
                assert h.fit(n) == 0 and h.backward(n) == 0
            total.append(lib.fake_bytes())
        finally:
            h.close()
    # a quarter more each time: the last one at most 1.25 times the need, those before
    # it together at most four times the last
    assert total[1] <= 5 * 1.25 * total[0]


def test_a_refused_allocation_leaves_nothing_behind(lib):
    # ENOMEM is that call's answer; the next call, which fits, does not report it
    h = Handle(lib, limit=GB)
    try:
        assert h.fit(10_000_000, per=200) == 3
        assert h.fit(5000) == 0 and h.backward(5000) == 0
        assert lib.tpcfit_reserve(h.h, C.c_int64(2_000_000_000), C.c_int64(0)) == 3
        assert h.fit(5000) == 0
    finally:
        h.close()


def test_the_tape_gives_way_to_what_a_fit_cannot_do_without(lib):
    # 4.6 GB: a recorded fit of 200,000 tracks takes 1.9 GB for its tape; checkpoints of
    # 1.6 million tracks (3.0 GB) fit without it, in a handle that never had one too
    limit = 4600 << 20
    for first in (False, True):
        h = Handle(lib, limit)
        try:
            if first:
                assert h.fit(200_000) == 0 and lib.fake_taped()
                assert h.backward(200_000) == 0
            lib.fake_forget()
            assert h.fit(1_600_000) == 0 and not lib.fake_taped()
            assert h.backward(1_600_000) == 0
            assert lib.fake_used_live() == lib.fake_used()
        finally:
            h.close()


def test_the_tape_stays_while_its_recording_does(lib):
    # scratch of other calls that finds no room is refused; the recording goes on
    h = Handle(lib, 2500 << 20)
    try:
        assert h.fit(100_000) == 0 and lib.fake_taped()
        assert lib.tpcfit_reserve(h.h, C.c_int64(1_000_000_000), C.c_int64(0)) == 3
        assert h.backward(100_000) == 0 and h.smooth(100_000) == 0
    finally:
        h.close()
