"""FP64 emulation with an infinity or a NaN among its operands (GPU): the digit
planes hold neither, so the problem's energies are NaN, as FP64's are, and not
finite numbers; other problems of a batch are not touched."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _with(inst, which, value):
    arrays = [np.array(a) for a in inst.arrays()]
    arrays[which].reshape(-1)[arrays[which].size // 3] = value
    return arrays


@pytest.mark.parametrize("which", [3, 4, 5], ids=["t2", "vvvo", "ooov"])
@pytest.mark.parametrize("value", [math.nan, math.inf, -math.inf])
@pytest.mark.parametrize("device", [True, False])
def test_energies_are_nan(which, value, device):
    import torch

    from paper_1609_08094_gb300 import synth, tcorr
    inst = synth.make_instance(4, 20, 72, 1)
    arrays = _with(inst, which, value)
    if device:
        arrays = [torch.from_numpy(a).cuda() for a in arrays]
    with tcorr.Tcorr(inst.o, inst.v, *arrays, prec="fp64_oz") as h:
        e, tasks = h.energy_range(0, h.num_tasks, per_task=True)
        ijk = [h.task(n) for n in range(h.num_tasks)]
    assert all(math.isnan(x) for x in e)
    for (i, j, k), t in zip(ijk, tasks):
        assert np.isnan(t).all() if i != k else (t == 0).all()


def test_other_problems_of_a_batch():
    import torch

    from paper_1609_08094_gb300 import synth, tcorr
    inst = synth.make_instance(4, 20, 72, 1)
    good = [torch.from_numpy(np.array(a)).cuda() for a in inst.arrays()]
    bad = [torch.from_numpy(a).cuda() for a in _with(inst, 3, math.nan)]
    with tcorr.Tcorr(inst.o, inst.v, *good, prec="fp64_oz") as h:
        want = h.energy()
    with tcorr.Batch([(inst.o, inst.v, *good), (inst.o, inst.v, *bad), (inst.o, inst.v, *good)], prec="fp64_oz") as b:
        e = b.energy()
    assert tuple(e[0]) == want and tuple(e[2]) == want and np.isnan(e[1]).all()
