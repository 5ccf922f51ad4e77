"""Device memory after a smoothing: what the smoother took for its tile copies does not
keep another context, or the caller's own allocator, from what it could have before."""
import pytest
import torch

import paper_1601_03184_gb300 as pkg
from paper_1601_03184_gb300 import MRHS_F32, MRHS_PREC_FP32, Lattice, inputs

pytestmark = pytest.mark.gpu

DIMS, N = (16, 16, 16, 32), 128  # 128 vectors: 3.2 GB of copies


def lattice(agg):
    lat = Lattice(DIMS, agg, 8, MRHS_PREC_FP32)
    lat.set_gauge(inputs.unit_gauge_field(DIMS))
    lat.build_clover(-0.1, 1.0)
    pkg.mrhs_trim(lat.ctx)  # (the gauge field's staging)
    return lat


def left(n):
    """all of the device's memory but n bytes"""
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - n, dtype=torch.uint8, device="cuda")


@pytest.fixture
def smoothed():
    """a context after a smoothing, its result, and the memory that was free before it"""
    lat = lattice((4, 4, 4, 4))
    b = torch.randn(lat.V * 24 * N, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    x = torch.zeros_like(b)
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    pkg.mrhs_profile(lat.ctx, 1)
    lat.sap(b, x, N, MRHS_F32, 2, 2)
    lat.sync()
    assert "sap_tiles" in pkg.mrhs_profile_read(lat.ctx)  # (on copies)
    yield lat, b, x, free
    lat.close()
    torch.cuda.empty_cache()


def test_the_callers_allocator_gets_it(smoothed):
    """and the smoother works on without it, to the bound of the FP32 forms (twice)"""
    lat, b, x, free = smoothed
    y = torch.zeros_like(x)
    take = torch.empty(free - y.numel() * 4 - (256 << 20), dtype=torch.uint8, device="cuda")
    lat.sap(b, y, N, MRHS_F32, 2, 2)
    lat.sync()
    del take
    torch.cuda.empty_cache()
    assert torch.linalg.vector_norm((x - y).double()) <= 2e-5 * torch.linalg.vector_norm(x.double())
    x.zero_()
    lat.sap(b, x, N, MRHS_F32, 2, 2)
    lat.sync()
    assert torch.linalg.vector_norm((x - y).double()) <= 2e-5 * torch.linalg.vector_norm(x.double())


def test_another_context_gets_it(smoothed):
    fill = left(64 << 20)  # of some 500 MB that the second context needs
    other = lattice((4, 4, 4, 4))
    other.sync()
    other.close()
    del fill


def test_trim_gives_it_back(smoothed):
    lat = smoothed[0]
    held = pkg.mrhs_info(lat.ctx)[5]
    pkg.mrhs_trim(lat.ctx)
    assert held - pkg.mrhs_info(lat.ctx)[5] > 3 << 30
    assert torch.cuda.mem_get_info()[0] > smoothed[3] - (256 << 20)


def test_gauge_field_takes_the_same_room_for_every_domain():
    held = []
    for agg in ((4, 4, 4, 4), (4, 4, 4, 2)):
        lat = lattice(agg)
        held.append(pkg.mrhs_info(lat.ctx)[5])
        lat.close()
    assert held[0] <= held[1]
