"""Operand layouts at sizes where the transposes can go wrong: o and v around the
16-, 32- and 64-wide tiles, and host arrays streamed in chunks that start on odd
rows.  Device and host inputs give the same bits; energies against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("tf32x3", 1e-6), ("fp64_oz", 1e-10)])
@pytest.mark.parametrize("o,v", [(2, 1), (3, 15), (2, 33), (17, 16), (33, 9), (4, 63), (3, 65)])
def test_layouts_from_device_and_host(prec, tol, o, v):
    import oracle
    from paper_1609_08094_gb300 import synth, tcorr
    inst = synth.make_instance(o, v, 3 * (o + v), seed=o * 100 + v)
    ref = oracle.energy(inst)
    with tcorr.Tcorr.from_instance(inst, prec=prec) as t:
        host = t.energy()
    with tcorr.Tcorr.from_instance(inst.to("cuda:0"), prec=prec) as t:
        dev = t.energy()
    assert host == dev
    if v > 1:  # with one virtual orbital the energy is exactly zero: nothing to be relative to
        assert abs(dev[2] - ref[2]) <= tol * abs(ref[2])


@pytest.mark.parametrize("prec", ["fp64", "bf16x3", "fp64_oz"])
def test_host_chunks_that_start_on_odd_rows(prec):
    """vvvo above 512 MiB is copied in chunks of d rows: 231^2 x 6 doubles per row give 209 rows."""
    from paper_1609_08094_gb300 import synth, tcorr
    o, v = 6, 231
    inst = synth.make_instance(o, v, 12, seed=5, device="cuda:0")
    n = 6
    with tcorr.Tcorr.from_instance(inst, prec=prec) as t:
        dev = t.energy_range(3, n, per_task=True)
    with tcorr.Tcorr.from_instance(inst.numpy(), prec=prec) as t:
        host = t.energy_range(3, n, per_task=True)
    assert np.array_equal(dev[1], host[1])
