"""What tcorr_create counts before it allocates is enough for what it allocates
(the host code on a fake runtime, tests/fake_device.py): a device with just the
footprint free takes the handle."""
import re

import pytest

from tests import fake_device as fd


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fd.build(str(tmp_path_factory.mktemp("fake")))


@pytest.mark.parametrize("o,v,prec", [(4, 20, 0), (4, 20, 3), (20, 150, 1), (250, 8, 1), (250, 8, 2)])
def test_a_device_with_the_footprint_free(lib, o, v, prec):
    dev = fd.Device(lib)
    dev.capacity(1 << 20)
    h = fd.Handle(dev, o, v, prec=prec, device=True, batch_tasks=64)
    assert h.status == fd.ENOMEM
    need = int(re.search(rb"footprint (\d+) bytes", dev.lib.tcorr_last_error(None)).group(1))
    dev.capacity(need)
    h = fd.Handle(dev, o, v, prec=prec, device=True, batch_tasks=64)
    assert h.status == fd.OK, dev.lib.tcorr_last_error(None)
    assert h.energy() == fd.OK and h.bytes() <= need
    h.close()
    assert dev.bad() == ""
