"""Plan tables of task ranges (the host code on a fake runtime, tests/fake_device.py):
a handle has room for the plan of any range from its creation on, so that energy
calls neither allocate nor can run out of memory, and no table is ever written to
memory that was given back."""
import pytest

from tests import fake_device as fd


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fd.build(str(tmp_path_factory.mktemp("fake")))


# v = 150 and 169: whether a wave's columns are packed depends on its tasks
@pytest.mark.parametrize("o,v,wave", [(8, 150, 40), (10, 169, 96), (13, 20, 7), (6, 64, 1), (9, 40, 0), (5, 257, 10)])
@pytest.mark.parametrize("prec", [1, 2])
def test_ranges_do_not_allocate(lib, o, v, wave, prec):
    dev = fd.Device(lib)
    h = fd.Handle(dev, o, v, prec=prec, device=True, batch_tasks=wave)
    assert h.status == fd.OK
    n = o * (o + 1) * (o + 2) // 6
    start = len(dev.log())
    step = max(1, n // 24)
    ranges = [(f, l - f) for f in range(0, n, step) for l in list(range(f + 1, n + 1, step)) + [n]]
    dev.capacity(0)  # were a call to allocate, it would fail, and the next one write to what it gave back
    failed = [r for r in ranges if h.range(*r) != fd.OK]
    assert dev.bad() == ""
    assert failed == []
    assert not [x for x in dev.log()[start:] if "Alloc" in x or "Malloc" in x]
    h.close()
    assert dev.bad() == ""
