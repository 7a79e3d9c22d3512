"""Handles on a stream that does not wait for the default one, with work queued on
it: the same bits as on the default stream (GPU).  The stream's operations are in
order, so a handle's tables and operands are complete before its kernels read them
however late the stream gets to them."""
import pytest

pytestmark = pytest.mark.gpu


def _busy(torch, stream):
    with torch.cuda.stream(stream):
        a = torch.randn(4096, 4096, device="cuda")
        for _ in range(20):
            a = torch.tanh(a @ a)
    return a


@pytest.mark.parametrize("prec", ["fp64", "fp64_oz", "tf32x3", "bf16x3"])
def test_tcorr_on_a_side_stream(prec):
    import torch

    from paper_1609_08094_gb300 import synth, tcorr
    inst = synth.make_instance(7, 45, 104, 3, device="cuda:0")
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for tune in (False, True):
        keep = _busy(torch, side)
        with tcorr.Tcorr.from_instance(inst, prec=prec, tune=tune, stream=side) as h:
            keep = _busy(torch, side)
            e = h.energy()
        with tcorr.Tcorr.from_instance(inst, prec=prec, tune=tune) as h:  # the tile found above
            assert h.energy() == e
        del keep


@pytest.mark.parametrize("prec", ["fp64", "tf32x3", "bf16x3"])
def test_mp2_on_a_side_stream(prec):
    import torch

    from paper_1609_08094_gb300 import synth, tcorr
    m = synth.make_mp2_instance(5, 150, 90, seed=2).to("cuda:0")
    torch.cuda.synchronize()
    with tcorr.Mp2.from_instance(m, prec=prec) as h:
        want = h.energy()
    side = torch.cuda.Stream()
    keep = _busy(torch, side)
    with tcorr.Mp2.from_instance(m, prec=prec, stream=side) as h:
        keep = _busy(torch, side)
        assert h.energy() == want
    del keep
