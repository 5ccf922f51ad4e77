"""The operand images of D_c in a mixed setup: made in the form that the solves of its own
vectors use, and read by the other counts too."""
import numpy as np
import pytest
import torch

import oracle
from paper_1601_03184_gb300 import MRHS_F32, MRHS_PREC_FP32, MRHS_PREC_MIX_BF16, Lattice, inputs

pytestmark = pytest.mark.gpu


def setup(dims, agg, ntv, prec, tv=None, U=None):
    lat = Lattice(dims, agg, ntv, prec)
    lat.set_gauge(inputs.unit_gauge_field(dims) if U is None else U)
    lat.build_clover(-0.1, 1.2)
    if tv is None:
        tv = torch.randn(lat.V * 24 * ntv, device="cuda", generator=torch.Generator("cuda").manual_seed(7))
    lat.set_tv(tv, MRHS_F32)
    lat.build_P()
    lat.build_Dc()
    return lat


def test_stencil_of_the_setups_vectors_reads_the_images():
    """24 vectors: the same split form as in an FP32 setup and as fast as there (a stencil
    that converts every block itself takes 14 % longer at this size)."""
    n, best = 24, []
    lats = [setup((16, 16, 16, 32), (4, 4, 4, 4), n, p) for p in (MRHS_PREC_FP32, MRHS_PREC_MIX_BF16)]
    x = torch.randn(lats[0].nagg * 4 * n * n, device="cuda", generator=torch.Generator("cuda").manual_seed(8))
    y = torch.zeros_like(x)
    times = [[], []]
    for _ in range(6):
        for lat, t in zip(lats, times):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            lat.apply_Dc(x, y, n, MRHS_F32)
            a.record()
            for _ in range(40):
                lat.apply_Dc(x, y, n, MRHS_F32)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
    best = [min(t) for t in times]
    for lat in lats:
        lat.close()
    assert best[1] <= 1.07 * best[0]


# vectors whose solves take split images (20, 24; 32 in blocks of 20), and single ones (16);
# counts of the split and of the single form on either
@pytest.mark.parametrize("ntv,block", [(20, 0), (24, 0), (32, 20), (16, 0)])
def test_every_count_on_either_images(ntv, block):
    """against the oracle's stencil on the same D_c: |dy| <= gamma sum |D| |x|, gamma = 2 (2 e
    + 2 * 9 * 2ntv * 2^-24) with the operand error e = 2^-22 (split) or 2^-11 (single)"""
    dims, agg = (4, 8, 4, 8), (2, 4, 2, 2)
    lat = Lattice(dims, agg, ntv, MRHS_PREC_MIX_BF16)
    lat.set_block_length(block)
    lat.set_gauge(inputs.gauge_field(dims, 0.5, 1403))
    lat.build_clover(-0.1, 1.2)
    lat.set_tv(lat.to_device(inputs.test_vectors(ntv, dims, 2403), MRHS_F32), MRHS_F32)
    lat.build_P()
    lat.build_Dc()
    Dc = lat.get_Dc()
    for n in (9, 16, 20, 24, 32):
        x = inputs.gaussian_field((n, lat.nagg, 2 * ntv), 4405).astype(np.complex64).astype(np.complex128)
        yd = lat.field(n, MRHS_F32, coarse=True)
        lat.apply_Dc(lat.to_device(x, MRHS_F32, coarse=True), yd, n, MRHS_F32)
        ref = oracle.apply_Dc(dims, agg, Dc, x)
        size = oracle.apply_Dc(dims, agg, np.abs(Dc).astype(np.complex128), np.abs(x).astype(np.complex128)).real
        gamma = 2 * (2 * (2.0 ** -11 if n % 16 == 0 else 2.0 ** -22) + 2 * 9 * 2 * ntv * 2.0 ** -24)
        assert np.all(np.abs(lat.to_host(yd, n, MRHS_F32, coarse=True) - ref) <= gamma * size), n
    lat.close()
