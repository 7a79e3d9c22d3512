"""A server's wave that an error ends before it is launched as a whole (the host code
on a fake runtime, tests/fake_device.py): its tasks stay with their jobs, the next
drain schedules them, and no job is done with tasks left out."""
import pytest

from tests import fake_device as fd

WAVES = 7  # 35 tasks, 5 to a wave


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fd.build(str(tmp_path_factory.mktemp("fake")))


def drained(s, i):
    assert s.drain() == fd.OK
    assert s.state(i) == ("done", fd.OK) and s.waves() == WAVES


@pytest.mark.parametrize("prec", [0, 1])
def test_host_allocations(lib, prec):
    dev = fd.Device(lib)
    for n in range(1, 400):
        s = fd.Server(dev, prec=prec, batch_tasks=5)
        i = s.submit(5, 30)
        dev.lib.fake_fail_new(n)
        st = s.drain()
        left = dev.lib.fake_new_left()
        dev.lib.fake_fail_new(-1)
        assert st == fd.OK or (st == fd.ENOMEM and left == 0)
        if s.state(i) != ("failed", fd.ENOMEM):  # a job whose admission found no memory
            drained(s, i)
        s.close()
        if left > 0:
            break
    assert left > 0 and dev.bad() == ""


# launches of the job's admission come first; those after them are of its waves
@pytest.mark.parametrize("fn,code,status", [("launch", fd.LAUNCH_FAILURE, fd.ECUDA),
                                            ("cudaMemcpyAsync", fd.LAUNCH_FAILURE, fd.ECUDA),
                                            ("cudaEventRecord", fd.LAUNCH_FAILURE, fd.ECUDA),
                                            ("cudaMalloc", fd.OUT_OF_MEMORY, fd.ENOMEM)])
def test_device_calls(lib, fn, code, status):
    dev = fd.Device(lib)
    reached = 0
    for nth in range(1, 80):
        s = fd.Server(dev, prec=1, batch_tasks=5)
        i = s.submit(5, 30)
        dev.fail(fn, nth=nth, code=code)
        st = s.drain()
        hit = dev.lib.fake_pending_fails() == 0
        dev.lib.fake_clear()
        assert st in (fd.OK, status)
        if s.state(i)[0] != "failed":
            drained(s, i)
            reached += st != fd.OK
        s.close()
        if not hit:
            break
    assert not hit
    if fn != "cudaMalloc":
        assert reached >= WAVES
