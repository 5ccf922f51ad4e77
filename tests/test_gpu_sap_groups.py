"""The on-chip smoother on tile copies with more right-hand sides than one group of copies
takes. A right-hand side's arithmetic does not depend on the others, so each comes out as
in a smoothing of its own group of four."""
import pytest
import torch

import paper_1601_03184_gb300 as pkg
from paper_1601_03184_gb300 import MRHS_F32, MRHS_PREC_FP32, Lattice, inputs

pytestmark = pytest.mark.gpu

DIMS, AGG = (8, 8, 8, 8), (4, 4, 4, 4)


@pytest.fixture(scope="module")
def lat():
    lat = Lattice(DIMS, AGG, 4, MRHS_PREC_FP32)
    lat.set_gauge(inputs.gauge_field(DIMS, 0.4, 1801))
    lat.build_clover(-0.1, 1.2)
    yield lat
    lat.close()


def test_thousands_of_right_hand_sides(lat):
    """6148 = 2048 three times and 4: whole rows of one site of more than 6142 are larger
    than a block's shared memory without a request."""
    n = 6148
    gen = torch.Generator("cuda").manual_seed(8)
    b, x = (torch.randn(lat.V * 24, n, device="cuda", generator=gen) for _ in range(2))
    four = [(k, b[:, k:k + 4].contiguous(), x[:, k:k + 4].contiguous()) for k in (0, 2044, 2048, 4096, 6140, 6144)]
    pkg.mrhs_profile(lat.ctx, 1)
    lat.sap(b, x, n, MRHS_F32, 2, 2)
    assert "sap_tiles" in pkg.mrhs_profile_read(lat.ctx)
    pkg.mrhs_profile(lat.ctx, 0)
    for k, bk, xk in four:
        lat.sap(bk, xk, 4, MRHS_F32, 2, 2)
        assert torch.equal(x[:, k:k + 4], xk), k
