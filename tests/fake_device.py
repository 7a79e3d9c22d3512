"""The library's host code on a fake CUDA runtime (tests/fake_cudart.cpp): no
GPU, no kernels, but every allocation, copy, event and wait is followed."""
import ctypes
import itertools
import os
import shutil
import subprocess

import numpy as np

from paper_1609_08094_gb300 import _build, tcorr

HERE = os.path.dirname(os.path.abspath(__file__))
OUT_OF_MEMORY, LAUNCH_FAILURE = 2, 719  # cudaError_t
OK, EINVAL, ENOMEM, ECUDA = 0, 1, 2, 3
_count = itertools.count()


def build(folder):
    _build.build()
    lib = os.path.join(folder, "libfake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    objs = [os.path.join(_build.OBJ, s.replace(".cu", ".o")) for s in _build.SOURCES]
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-I", inc, "-Wl,-Bsymbolic", "-o", lib,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    return lib


class Device:
    """One copy of the library with a device of its own."""

    def __init__(self, lib):
        own = "%s.%d" % (lib, next(_count))
        shutil.copyfile(lib, own)
        self.lib = lib = ctypes.CDLL(own)
        for f in ("tcorr_last_error", "tcorr_server_last_error", "tcorr_mp2_last_error", "fake_log", "fake_bad"):
            getattr(lib, f).restype = ctypes.c_char_p
        for f in ("tcorr_device_bytes", "tcorr_mp2_device_bytes", "tcorr_num_tasks"):
            getattr(lib, f).restype = ctypes.c_int64
        for f in ("fake_free", "fake_blocks"):
            getattr(lib, f).restype = ctypes.c_size_t
        lib.fake_stream.restype = ctypes.c_void_p
        self.stream = ctypes.c_void_p(lib.fake_stream())

    def log(self):
        return self.lib.fake_log().decode().splitlines()

    def bad(self):
        return self.lib.fake_bad().decode()

    def capacity(self, n):
        self.lib.fake_capacity(ctypes.c_size_t(n))

    def fail(self, fn, nth=1, code=OUT_OF_MEMORY):
        self.lib.fake_fail(fn.encode(), nth, code)

    def free(self):
        return self.lib.fake_free()


def _p(a):
    return ctypes.c_void_p(a.ctypes.data)


class Handle:
    """tcorr_create on host arrays of zeros (device=True: passed as device arrays)."""

    def __init__(self, dev, o, v, prec=0, device=False, **opts):
        self.dev, self.o, self.v = dev, o, v
        self.a = [np.zeros(n) for n in (o, v, o * v, o * o * v * v, v ** 3 * o, o ** 3 * v, o * v * o * v)]
        self.opts = tcorr.Opts(prec=prec, host_inputs=0 if device else 1, **opts)
        self.h = ctypes.c_void_p()
        self.status = dev.lib.tcorr_create(ctypes.byref(self.h), o, v, *[_p(x) for x in self.a],
                                           ctypes.byref(self.opts), dev.stream)

    def range(self, first, count):
        e = (ctypes.c_double * 3)()
        return self.dev.lib.tcorr_energy_range(self.h, ctypes.c_int64(first), ctypes.c_int64(count), e, None)

    def energy(self):
        return self.dev.lib.tcorr_energy(self.h, (ctypes.c_double * 3)())

    def bytes(self):
        return self.dev.lib.tcorr_device_bytes(self.h)

    def close(self):
        return self.dev.lib.tcorr_destroy(self.h)


class Mp2:
    def __init__(self, dev, o, v, naux, prec=0):
        self.dev = dev
        self.a = [np.zeros(n) for n in (o, v, naux * v * o)]
        self.opts = tcorr.Opts(prec=prec, host_inputs=1)
        self.h = ctypes.c_void_p()
        self.status = dev.lib.tcorr_mp2_create(ctypes.byref(self.h), o, v, naux, *[_p(x) for x in self.a],
                                               ctypes.byref(self.opts), dev.stream)

    def energy(self):
        return self.dev.lib.tcorr_mp2_energy(self.h, (ctypes.c_double * 3)())

    def close(self):
        return self.dev.lib.tcorr_mp2_destroy(self.h)


class Server:
    def __init__(self, dev, prec=1, hbm=0, **opts):
        self.dev, self.keep = dev, []
        self.opts = tcorr.Opts(prec=prec, **opts)
        self.h = ctypes.c_void_p()
        self.status = dev.lib.tcorr_server_create(ctypes.byref(self.h), ctypes.byref(self.opts), ctypes.c_int64(hbm),
                                                  dev.stream)

    def submit(self, o, v):
        a = [np.zeros(n) for n in (o, v, o * v, o * o * v * v, v ** 3 * o, o ** 3 * v, o * v * o * v)]
        self.keep.append(a)
        p, i = tcorr.Problem(o, v, *[x.ctypes.data for x in a]), ctypes.c_int64()
        assert self.dev.lib.tcorr_server_submit(self.h, ctypes.byref(p), ctypes.byref(i)) == OK
        return i.value

    def step(self):
        return self.dev.lib.tcorr_server_step(self.h, None)

    def drain(self):
        return self.dev.lib.tcorr_server_drain(self.h)

    def state(self, i):
        st, js = ctypes.c_int(), ctypes.c_int()
        assert self.dev.lib.tcorr_server_poll(self.h, ctypes.c_int64(i), ctypes.byref(st), None, ctypes.byref(js)) == OK
        return tcorr.JOB_STATES[st.value], js.value

    def close(self):
        return self.dev.lib.tcorr_server_destroy(self.h)

    def waves(self):
        st = (ctypes.c_int64 * 8)()
        assert self.dev.lib.tcorr_server_stats(self.h, st) == OK
        return st[7]
