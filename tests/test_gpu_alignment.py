"""Caller's fields that start on the alignment of their numbers only: the calls whose
usual forms copy wider pieces give the same results (to FP32 rounding: any order of at
most a few hundred terms, each part's error below 2e-5 of the field)."""
import pytest
import torch

from paper_1601_03184_gb300 import MRHS_F32, MRHS_PREC_FP32, Lattice, inputs

pytestmark = pytest.mark.gpu

DIMS, AGG, NTV = (8, 8, 8, 8), (4, 4, 4, 4), 8


@pytest.fixture(scope="module")
def lat():
    lat = Lattice(DIMS, AGG, NTV, MRHS_PREC_FP32)
    lat.set_gauge(inputs.gauge_field(DIMS, 0.4, 1701))
    lat.build_clover(-0.1, 1.2)
    lat.set_tv(lat.to_device(inputs.test_vectors(NTV, DIMS, 2701), MRHS_F32), MRHS_F32)
    lat.build_P()
    lat.build_Dc()
    yield lat
    lat.close()


def normal(n, seed):
    return torch.randn(n, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))


def shifted(x, floats):
    """the same numbers, `floats` numbers after a 16-byte boundary"""
    y = torch.empty(x.numel() + 4, device="cuda")[floats:floats + x.numel()]
    y.copy_(x)
    assert y.data_ptr() % 16 == 4 * floats
    return y


def close(a, b):
    return torch.linalg.vector_norm((a - b).double()) <= 2e-5 * torch.linalg.vector_norm(b.double())


@pytest.mark.parametrize("nrhs", [1, 5, 12])
def test_restriction(lat, nrhs):
    v = normal(lat.V * 24 * nrhs, 11)
    a, b = (torch.zeros(lat.nagg * 4 * NTV * nrhs, device="cuda") for _ in range(2))
    lat.restrict(v, a, nrhs, MRHS_F32)
    lat.restrict(shifted(v, 1), b, nrhs, MRHS_F32)
    assert close(b, a)


@pytest.mark.parametrize("nrhs", [5, 9, 16, 20])
def test_coarse_stencil(lat, nrhs):
    x = normal(lat.nagg * 4 * NTV * nrhs, 12)
    a, b = (torch.zeros_like(x) for _ in range(2))
    lat.apply_Dc(x, a, nrhs, MRHS_F32)
    lat.apply_Dc(shifted(x, 1), b, nrhs, MRHS_F32)
    lat.sync()
    assert close(b, a)


def test_smoother(lat):
    n = 8
    b = normal(lat.V * 24 * n, 13)
    x, y = (normal(lat.V * 24 * n, 14) for _ in range(2))
    lat.sap(b, x, n, MRHS_F32, 2, 3)
    lat.sap(shifted(b, 2), y, n, MRHS_F32, 2, 3)
    assert close(y, x)
