"""Host allocations that fail (the host code on a fake runtime, tests/fake_device.py):
every entry of the C ABI answers with a status, no exception leaves one, closing a
handle allocates nothing that could fail, and the next call works again.  Each test
runs in a process of its own: an exception at a C entry ends the process."""
import subprocess
import sys
import textwrap

import pytest

from tests import fake_device as fd


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fd.build(str(tmp_path_factory.mktemp("fake")))


def run(lib, body):
    code = "import sys\nsys.path.insert(0, %r)\nfrom tests import fake_device as fd\ndev = fd.Device(%r)\n" % (
        fd.os.path.dirname(fd.HERE), lib)
    r = subprocess.run([sys.executable, "-c", code + textwrap.dedent(body)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("prec", [0, 1])
def test_calls_and_close(lib, prec):
    run(lib, """
        h = fd.Handle(dev, 6, 40, prec=%d, batch_tasks=10)
        assert h.status == fd.OK
        seen = set()
        for n in range(1, 200):
            assert h.range(0, 56) == fd.OK
            dev.lib.fake_fail_new(n)
            st = h.range(1 + n %% 40, 10 + n %% 5)
            left = dev.lib.fake_new_left()
            dev.lib.fake_fail_new(-1)
            assert st == (fd.ENOMEM if left == 0 else fd.OK), (n, st, left)
            seen.add(st)
            if left > 0:
                break
        assert seen == {fd.OK, fd.ENOMEM}
        g = fd.Handle(dev, 10, 100, prec=%d, device=True, batch_tasks=20)
        assert g.status == fd.OK and g.energy() == fd.OK
        for x in (h, g):
            dev.lib.fake_fail_new(1)
            assert x.close() == fd.OK
            dev.lib.fake_fail_new(-1)
        dev.lib.fake_fail_new(1)
        assert dev.lib.tcorr_trim() == fd.OK
        assert dev.bad() == ""
    """ % (prec, prec))


def test_create(lib):
    run(lib, """
        h = fd.Handle(dev, 4, 20, prec=1)
        h.close()
        dev.lib.tcorr_trim()
        free, n = dev.free(), 0
        while True:
            n += 1
            dev.lib.fake_fail_new(n)
            h = fd.Handle(dev, 4, 20, prec=1)
            left = dev.lib.fake_new_left()
            dev.lib.fake_fail_new(-1)
            if left > 0:
                break
            assert h.status == fd.ENOMEM
            dev.lib.tcorr_trim()
            assert dev.free() == free, n  # nothing is left behind
        assert h.status == fd.OK and n > 10
        assert h.close() == fd.OK and dev.bad() == ""
    """)
