"""Packed columns of the SM-pair contraction (tasks that share (p, q) computed
side by side): the same per-task energies, bit for bit, as the single-SM kernel,
which computes every group on its own, at the edges of the 16-column entries, the
256-column passes and v = 256, and over task ranges that cut the runs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,o,v", [
    ("tf32x3", 2, 1), ("tf32x3", 5, 15), ("tf32x3", 5, 16), ("tf32x3", 7, 17), ("tf32x3", 3, 33), ("tf32x3", 9, 64),
    ("tf32x3", 4, 97), ("tf32x3", 3, 128), ("tf32x3", 3, 129), ("tf32x3", 2, 240), ("tf32x3", 2, 241),
    ("tf32x3", 2, 256), ("tf32x3", 2, 257), ("tf32x3", 33, 18), ("bf16x3", 6, 128)])
def test_per_task_energies_equal_the_single_sm_kernels(prec, o, v):
    from paper_1609_08094_gb300 import synth, tcorr
    inst = synth.make_instance(o, v, 3 * (o + v), seed=o * 1000 + v, device="cuda:0")
    n = tcorr.num_tasks(o)
    with tcorr.Tcorr.from_instance(inst, prec=prec, single_sm=True) as t:
        ref = t.energy_range(0, n, per_task=True)
    with tcorr.Tcorr.from_instance(inst, prec=prec) as t:
        got = t.energy_range(0, n, per_task=True)
        first = n // 3
        part = t.energy_range(first, n - first - 1, per_task=True)
    assert got[0] == ref[0]
    assert np.array_equal(got[1], ref[1])
    assert np.array_equal(part[1], ref[1][first:n - 1])
    with tcorr.Tcorr.from_instance(inst, prec=prec, batch_tasks=3) as t:
        cut = t.energy_range(0, n, per_task=True)
    assert np.array_equal(cut[1], ref[1])
