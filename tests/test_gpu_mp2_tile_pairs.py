"""RI-MP2 in split precision where g is not stored (v > 8192, GPU): the tile-pair
kernel against the FP64 kernel, at a ragged last tile and with i = j and i < j.
Tolerance: the split precisions' 1e-6."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("o,v,naux", [(1, 8200, 8), (2, 8193, 33)])
def test_tile_pair_form_matches_the_fp64_kernel(o, v, naux):
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
            assert tcorr.load().tcorr_mp2_device_bytes(h._h) < 4 * v * v  # no room for g of a pair
            e = h.energy()
            assert h.energy() == e
        for a, b in zip(e, ref):
            assert abs(a - b) <= 1e-6 * abs(ref[2])
