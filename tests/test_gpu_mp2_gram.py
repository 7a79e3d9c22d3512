"""RI-MP2 in split precision from Gram-matrix tiles: against the FP64 kernel at
the edges of the 256-row tiles of the flattened (i, a), with several waves of g
(1 GiB each) and with waves that cut the j of one i.  Tolerance: the split
precisions' 1e-6 (the scheme's error is 1.2e-7 .. 2.3e-7 in TF32)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("o,v,naux", [
    (1, 1, 1), (1, 255, 5), (1, 257, 40), (2, 128, 33), (4, 64, 16), (3, 86, 70), (5, 51, 31), (7, 73, 97),
    (60, 300, 8), (17, 4096, 8)])
def test_gram_form_matches_the_fp64_kernel(o, v, naux):
    import torch

    from paper_1609_08094_gb300 import tcorr
    g = torch.Generator(device="cuda").manual_seed(o * 10000 + v)
    eo = torch.sort(-2.0 + 1.7 * torch.rand(o, dtype=torch.float64, device="cuda", generator=g)).values
    ev = torch.sort(0.1 + 4.9 * torch.rand(v, dtype=torch.float64, device="cuda", generator=g)).values
    C = 0.1 * torch.randn(naux, v, o, dtype=torch.float64, device="cuda", generator=g)
    with tcorr.Mp2(o, v, naux, eo, ev, C) as h:
        ref = h.energy()
    for prec in ("tf32x3", "bf16x3"):
        with tcorr.Mp2(o, v, naux, eo, ev, C, prec=prec) as h:
            e = h.energy()
            assert h.energy() == e
        assert abs(e[2] - ref[2]) <= 1e-6 * abs(ref[2])
