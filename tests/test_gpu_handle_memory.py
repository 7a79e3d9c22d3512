"""Handles on reused device memory (GPU).

A handle's larger device blocks (above 16 MiB) may be ones that an earlier
handle gave back, with that handle's values in them, and up to a quarter larger
than asked for.  Energies must not depend on it: handles kept side by side,
closed, and created again one at a time or from several threads give the same
bits.
"""
import threading

import pytest

pytestmark = pytest.mark.gpu
SIZES = [(7, 61), (7, 60), (6, 64), (7, 61)]


@pytest.mark.parametrize("prec", ["fp64", "fp64_oz", "tf32x3"])
def test_energies_on_reused_blocks(prec):
    from paper_1609_08094_gb300 import synth, tcorr

    insts = [synth.make_instance(o, v, 2 * (o + v), 11 + n, device="cuda:0") for n, (o, v) in enumerate(SIZES)]
    kept = [tcorr.Tcorr.from_instance(i, prec=prec) for i in insts]
    want = [h.energy() for h in kept]
    for h in kept:
        h.close()

    def again(order):
        got = {}
        for n in order:
            with tcorr.Tcorr.from_instance(insts[n], prec=prec) as h:
                got[n] = h.energy()
        return got

    assert again(range(len(insts))) == dict(enumerate(want))
    results = [None] * 3

    def work(t):
        results[t] = again([(n + t) % len(insts) for n in range(len(insts))])

    threads = [threading.Thread(target=work, args=(t,)) for t in range(len(results))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert results == [dict(enumerate(want))] * len(results)
