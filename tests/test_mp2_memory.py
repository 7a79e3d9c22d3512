"""RI-MP2 in split precision takes what memory there is (the host code on a fake
runtime, tests/fake_device.py): waves of g of at most 1 GiB, smaller ones where less
is free, and the form without g where no two pairs of it fit."""
import pytest

from tests import fake_device as fd

MB = 1 << 20


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fd.build(str(tmp_path_factory.mktemp("fake")))


def launches(dev, h):
    n = len(dev.log())
    assert h.energy() == fd.OK
    return len([x for x in dev.log()[n:] if x.startswith("launch")])


# free memory beyond C^T (hi and lo) and the 64 MiB of slack -> one wave of two kernels, several (2), or the one kernel (0)
@pytest.mark.parametrize("o,v,naux,extra,waves", [
    (20, 450, 8, 400, 1), (20, 450, 8, 200, 2), (2, 4000, 8, 300, 1), (2, 4000, 8, 140, 2), (2, 4000, 8, 10, 0),
    (2, 9000, 8, 4000, 0)])
@pytest.mark.parametrize("prec", [1, 2])
def test_what_fits(lib, o, v, naux, extra, waves, prec):
    dev = fd.Device(lib)
    host = o * v * naux * 8  # the staged copy of C
    dev.capacity(2 * o * v * 32 * 4 + host + (64 + extra) * MB)
    h = fd.Mp2(dev, o, v, naux, prec=prec)
    assert h.status == fd.OK, dev.lib.tcorr_mp2_last_error(None)
    got = launches(dev, h)
    assert got == 2 if waves == 0 else got >= 1 + 2 * waves
    if waves == 1:
        assert got == 3
    h.close()
    assert dev.bad() == ""
