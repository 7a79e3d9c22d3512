"""Memory that closed handles leave for later ones (the host code on a fake runtime,
tests/fake_device.py): what else allocates through the library gets it back, and a
program can take it back with tcorr_trim."""
import pytest

from tests import fake_device as fd

GB = 1 << 30


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fd.build(str(tmp_path_factory.mktemp("fake")))


def leave(dev):
    """A handle whose U scratch (2.8 GiB) and smaller blocks are kept after it is closed."""
    h = fd.Handle(dev, 10, 100, prec=1, device=True)
    assert h.status == fd.OK and h.energy() == fd.OK
    assert 2 * GB < h.bytes()
    before = dev.free()
    h.close()
    return dev.free() - before


def test_a_server_counts_it_as_free(lib):
    dev = fd.Device(lib)
    dev.capacity(40 * GB)
    leave(dev)
    s = fd.Server(dev, hbm=37 * GB)  # 2 GiB of scratch aside
    assert s.status == fd.OK, dev.lib.tcorr_server_last_error(None)
    s.close()
    assert dev.bad() == ""


def test_a_job_gets_it(lib):
    dev = fd.Device(lib)
    dev.capacity(40 * GB)
    s = fd.Server(dev)
    leave(dev)
    dev.capacity(40 * GB - dev.free())  # nothing but what is kept
    i = s.submit(6, 100)
    assert s.drain() == fd.OK and s.state(i) == ("done", fd.OK)
    s.close()
    assert dev.bad() == ""


def test_trim_gives_it_back(lib):
    dev = fd.Device(lib)
    start = dev.free()
    leave(dev)
    kept = start - dev.free()
    assert 2 * GB < kept <= 4 * GB
    h = fd.Handle(dev, 4, 20, prec=1)
    assert dev.lib.tcorr_trim() == fd.OK
    assert h.energy() == fd.OK  # an open handle keeps its blocks
    assert start - dev.free() <= h.bytes() + (64 << 20)
    h.close()
    assert dev.lib.tcorr_trim() == fd.OK and dev.free() == start
    assert dev.bad() == ""


def test_bytes_of_a_reused_block(lib):
    dev = fd.Device(lib)
    start = dev.free()
    leave(dev)
    dev.lib.fake_clear()
    h = fd.Handle(dev, 10, 100, prec=1, device=True, batch_tasks=190)  # 190 tasks' scratch in the block of 220
    assert h.status == fd.OK
    assert [x for x in dev.log() if x.startswith("cudaMalloc ")] == []
    assert h.bytes() >= 220 * 3 * 104 ** 3 * 4
    h.close()
    assert dev.lib.tcorr_trim() == fd.OK and dev.free() == start
