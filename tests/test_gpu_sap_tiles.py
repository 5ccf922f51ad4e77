"""The on-chip smoother on tile copies (domains of 129 to 256 sites, at least two
sweeps) at the edges of its face slots, against the FP64 oracle at the bound of
the other FP32 smoother forms.

4^4: two faces beside the rho tile, four in it; 4^3 x 3: idle threads and faces of
48 and 64 sites; (2,8,4,4): faces of half the domain; (1,16,4,4): both faces of
every site, one direction at a time; (8,8,2,2): the wide directions first."""
import numpy as np
import pytest
import torch

import oracle
import paper_1601_03184_gb300 as pkg
from paper_1601_03184_gb300 import MRHS_BF16, MRHS_F32, MRHS_PREC_FP32, MRHS_PREC_MIX_BF16, Lattice, inputs

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("nrhs,n_mr", [(4, 3), (12, 0), (20, 1)])
@pytest.mark.parametrize("agg,dims", [((4, 4, 4, 4), (8, 8, 8, 8)), ((4, 4, 4, 3), (8, 8, 8, 6)),
                                      ((2, 8, 4, 4), (4, 16, 8, 8)), ((1, 16, 4, 4), (2, 32, 8, 8)),
                                      ((8, 8, 2, 2), (16, 16, 4, 4))])
def test_sap_on_tiles(agg, dims, nrhs, n_mr):
    U = inputs.gauge_field(dims, 0.4, 1501)
    A = oracle.clover(dims, U, -0.1, 1.2)
    lat = Lattice(dims, agg, 4, MRHS_PREC_FP32)
    lat.set_gauge(U)
    lat.build_clover(-0.1, 1.2)
    b = inputs.gaussian_field((nrhs, lat.V, 12), 781)
    x0 = 0.1 * inputs.gaussian_field((nrhs, lat.V, 12), 782)
    xd = lat.to_device(x0, MRHS_F32)
    pkg.mrhs_profile(lat.ctx, 1)
    lat.sap(lat.to_device(b, MRHS_F32), xd, nrhs, MRHS_F32, 2, n_mr)
    assert "sap_tiles" in pkg.mrhs_profile_read(lat.ctx)
    ref = oracle.sap(dims, agg, U, A, b, x0, 2, n_mr)
    assert rel(lat.to_host(xd, nrhs, MRHS_F32), ref) < 1e-5
    lat.close()


def test_copies_give_way_to_needed_memory():
    """What the smoother holds only to run faster is released for what a later step
    cannot do without: with the device filled up after a smoothing, the test vectors
    (more than is left) are still stored, and the smoother still gives its result
    (to the bound of the FP32 forms, twice)."""
    dims, agg, ntv = (16, 16, 16, 16), (4, 4, 4, 4), 16
    lat = Lattice(dims, agg, ntv, MRHS_PREC_FP32)
    lat.set_gauge(inputs.gauge_field(dims, 0.4, 1503))
    lat.build_clover(-0.1, 1.2)
    b = torch.randn(lat.V * 24 * ntv, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    first, again = torch.zeros_like(b), torch.zeros_like(b)
    lat.sap(b, first, ntv, MRHS_F32, 2, 2)
    lat.sync()
    torch.cuda.empty_cache()
    held = pkg.mrhs_info(lat.ctx)[5]
    rest = torch.cuda.mem_get_info()[0] - (48 << 20)
    fill = torch.empty(rest, dtype=torch.uint8, device="cuda")  # 48 MB left, 100 MB needed
    try:
        lat.set_tv(b, MRHS_F32)
        assert pkg.mrhs_info(lat.ctx)[5] < held  # 200 MB of copies gone, 100 MB of vectors there
        lat.sap(b, again, ntv, MRHS_F32, 2, 2)
        lat.sync()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert torch.linalg.vector_norm((first - again).double()) <= 2e-5 * torch.linalg.vector_norm(first.double())
    lat.close()


def test_initial_phase_from_reduced_storage():
    """b in bf16 (the mixed setup's vectors) and x0 = 0: the smoothed, normalised
    vectors, rounded once to bf16, against the oracle's from the same rounded b."""
    dims, agg, ntv = (8, 8, 8, 8), (4, 4, 4, 4), 8
    U = inputs.gauge_field(dims, 0.4, 1502)
    A = oracle.clover(dims, U, -0.1, 1.2)
    lat = Lattice(dims, agg, ntv, MRHS_PREC_MIX_BF16)
    lat.set_gauge(U)
    lat.build_clover(-0.1, 1.2)
    tv = lat.to_device(inputs.test_vectors(ntv, dims, 2502), MRHS_BF16)
    b = lat.to_host(tv, ntv, MRHS_BF16)
    lat.setup_init(tv, MRHS_BF16, 0, 2, 3)
    ref = oracle.sap(dims, agg, U, A, b, 0 * b, 2, 3)
    ref /= np.linalg.norm(ref.reshape(ntv, -1), axis=1)[:, None, None]
    assert rel(lat.get_tv(), ref) < 2.0 ** -8 + 1e-5
    lat.close()
