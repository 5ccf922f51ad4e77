"""The on-chip smoother on tile copies with more right-hand sides than one group of copies
takes. A right-hand side's arithmetic does not depend on the others, so each comes out as
in a smoothing of its own group of four."""
import numpy as np
import pytest
import torch

import oracle
import paper_1601_03184_gb300 as pkg
from paper_1601_03184_gb300 import MRHS_BF16, MRHS_F32, MRHS_PREC_FP32, MRHS_PREC_MIX_BF16, Lattice, inputs

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


def limited(monkeypatch, ntv, prec, groups_of):
    """a lattice whose workspace takes groups_of right-hand sides and half of four more"""
    V = int(np.prod(DIMS))
    monkeypatch.setenv("MRHS_TILE_BYTES", str(V * 320 + (groups_of + 2) * V * 24 * 4 * 2))
    lat = Lattice(DIMS, AGG, ntv, prec)
    U = inputs.gauge_field(DIMS, 0.4, 1802)
    lat.set_gauge(U)
    lat.build_clover(-0.1, 1.2)
    return lat, U, oracle.clover(DIMS, U, -0.1, 1.2)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("groups_of,groups", [(4, 5), (8, 3), (12, 3), (16, 2)])
def test_groups(monkeypatch, groups_of, groups):
    """20 right-hand sides in groups of 4, of 8 (also where 12 would fit) and of 16, the
    last one shorter, against the oracle at the bound of the FP32 forms."""
    n = 20
    lat, U, A = limited(monkeypatch, 4, MRHS_PREC_FP32, groups_of)
    b = inputs.gaussian_field((n, lat.V, 12), 783)
    x0 = 0.1 * inputs.gaussian_field((n, lat.V, 12), 784)
    xd = lat.to_device(x0, MRHS_F32)
    pkg.mrhs_profile(lat.ctx, 1)
    lat.sap(lat.to_device(b, MRHS_F32), xd, n, MRHS_F32, 2, 3)
    assert pkg.mrhs_profile_read(lat.ctx)["sap_tiles"][0] == 2 * groups
    ref = oracle.sap(DIMS, AGG, U, A, b, x0, 2, 3)
    x = lat.to_host(xd, n, MRHS_F32)
    for r in range(n):
        assert rel(x[r], ref[r]) < 1e-5, r
    lat.close()


def test_groups_of_the_initial_phase(monkeypatch):
    """the same from x0 = 0 and b in bf16, rounded once to bf16 at the end"""
    n = 20
    lat, U, A = limited(monkeypatch, n, MRHS_PREC_MIX_BF16, 8)
    tv = lat.to_device(inputs.test_vectors(n, DIMS, 2802), MRHS_BF16)
    b = lat.to_host(tv, n, MRHS_BF16)
    pkg.mrhs_profile(lat.ctx, 1)
    lat.setup_init(tv, MRHS_BF16, 0, 2, 3)
    assert pkg.mrhs_profile_read(lat.ctx)["sap_tiles"][0] == 6
    ref = oracle.sap(DIMS, AGG, U, A, b, 0 * b, 2, 3)
    x = lat.get_tv()
    for r in range(n):
        assert rel(x[r], ref[r] / np.linalg.norm(ref[r])) < 2.0 ** -8 + 1e-5, r
    lat.close()
