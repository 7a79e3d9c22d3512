"""Blocks from the handles' memory pool are only used in the order of the
handle's own stream: on a stream that does not wait for the default one, every
copy into a block comes after the block's allocation, and its give-back after
every copy (the host code on a fake runtime, tests/fake_device.py)."""
import ctypes

import numpy as np
import pytest

from tests import fake_device as fd


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fd.build(str(tmp_path_factory.mktemp("fake")))


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("tune", [0, 1])
@pytest.mark.parametrize("device", [False, True])
def test_handle(lib, prec, tune, device):
    dev = fd.Device(lib)
    for o, v in ((4, 20), (1, 1), (3, 130)):
        h = fd.Handle(dev, o, v, prec=prec, tune=tune, device=device)
        assert h.status == fd.OK, dev.lib.tcorr_last_error(None)
        assert h.energy() == fd.OK and h.range(0, 1) == fd.OK and h.energy() == fd.OK
        h.close()
    assert dev.bad() == ""


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_mp2(lib, prec):
    dev = fd.Device(lib)
    for o, v, naux in ((3, 30, 20), (1, 1, 1), (2, 300, 7)):
        h = fd.Mp2(dev, o, v, naux, prec=prec)
        assert h.status == fd.OK
        assert h.energy() == fd.OK and h.close() == fd.OK
    assert dev.bad() == ""


@pytest.mark.parametrize("prec", [0, 2])
def test_batch(lib, prec):
    from paper_1609_08094_gb300 import tcorr
    dev = fd.Device(lib)
    keep, probs = [], (tcorr.Problem * 3)()
    for n, (o, v) in enumerate(((4, 20), (2, 33), (3, 7))):
        a = [np.zeros(k) for k in (o, v, o * v, o * o * v * v, v ** 3 * o, o ** 3 * v, o * v * o * v)]
        keep.append(a)
        probs[n] = tcorr.Problem(o, v, *[x.ctypes.data for x in a])
    h = ctypes.c_void_p()
    opts = tcorr.Opts(prec=prec, host_inputs=1, eager=1, tune=1)
    assert dev.lib.tcorr_batch_create(ctypes.byref(h), 3, probs, ctypes.byref(opts), dev.stream) == fd.OK
    assert dev.lib.tcorr_batch_energy(h, (ctypes.c_double * 9)()) == fd.OK
    assert dev.lib.tcorr_batch_destroy(h) == fd.OK
    assert dev.bad() == ""


@pytest.mark.parametrize("prec", [0, 2, 3])
@pytest.mark.parametrize("fn", ["cudaStreamWaitEvent", "cudaEventRecord"])
def test_no_copy_is_left_in_a_block_given_back(lib, prec, fn):
    """An error between a chunk's copy and the stream's wait for it ends the
    creation; the staging block (20 MB, kept for reuse) then goes to the next one."""
    dev = fd.Device(lib)
    o, v = 12, 60
    dev.fail(fn, nth=2, code=fd.LAUNCH_FAILURE)
    assert fd.Handle(dev, o, v, prec=prec).status == fd.ECUDA
    h = fd.Handle(dev, o, v, prec=prec)
    assert h.status == fd.OK and h.close() == fd.OK
    assert dev.bad() == ""
