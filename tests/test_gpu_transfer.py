"""Restriction and prolongation of FP32 coarse fields at the edges of their tiles,
against the products of the GPU's own P written out in FP64.

One entry is a sum of 6 |A| (restriction) or ntv (prolongation) complex products:
in any order its error is below sqrt(2) gamma_n (|P| |x|), n = 2 * terms + 2 with the
FP32 unit roundoff; reduced storage of P and v is read exactly."""
import numpy as np
import pytest

from lattice_helpers import aggregate_of_sites
from paper_1601_03184_gb300 import MRHS_F32, MRHS_PREC_FP32, MRHS_PREC_MIX_BF16, Lattice, inputs

pytestmark = pytest.mark.gpu

DIMS, AGG = (6, 4, 4, 8), (3, 2, 2, 2)
U = 2.0 ** -24


def bound(terms, size):
    n = 2 * terms + 2
    return 2 ** 0.5 * n * U / (1 - n * U) * size + 1e-300


# vectors: 1, 3 and 6 (not a multiple of four), 4 (one tile), 20, 32; right-hand sides:
# 1 to 3 (one per thread), 4, 5 (ragged tile), 12, 33, and 200 (32 vectors: columns in
# two pieces) for the prolongation
@pytest.mark.parametrize("ntv", [1, 3, 4, 6, 20, 32])
@pytest.mark.parametrize("prec", [MRHS_PREC_FP32, MRHS_PREC_MIX_BF16])
def test_restriction_and_prolongation(ntv, prec):
    lat = Lattice(DIMS, AGG, ntv, prec)
    lat.set_gauge(inputs.unit_gauge_field(DIMS))
    lat.build_clover(0.1, 1.0)
    lat.set_tv(lat.to_device(inputs.test_vectors(ntv, DIMS, 2701), MRHS_F32), MRHS_F32)
    lat.build_P()
    ag = aggregate_of_sites(DIMS, AGG)
    P = lat.get_P().reshape(ntv, lat.V, 2, 6)
    sites = [np.flatnonzero(ag == a) for a in range(lat.nagg)]
    for nrhs in (1, 2, 3, 4, 5, 12, 33, 200):
        v = inputs.gaussian_field((nrhs, lat.V, 12), 4701).astype(np.complex64).astype(np.complex128)
        uc = inputs.gaussian_field((nrhs, lat.nagg, 2 * ntv), 4702).astype(np.complex64).astype(np.complex128)
        vcd, ud = lat.field(nrhs, MRHS_F32, coarse=True), lat.field(nrhs, MRHS_F32)
        if nrhs <= 64:
            lat.restrict(lat.to_device(v, MRHS_F32), vcd, nrhs, MRHS_F32)
        lat.prolong(lat.to_device(uc, MRHS_F32, coarse=True), ud, nrhs, MRHS_F32)
        vc = lat.to_host(vcd, nrhs, MRHS_F32, coarse=True).reshape(nrhs, lat.nagg, 2, ntv)
        u = lat.to_host(ud, nrhs, MRHS_F32).reshape(nrhs, lat.V, 2, 6)
        v, uc = v.reshape(nrhs, lat.V, 2, 6), uc.reshape(nrhs, lat.nagg, 2, ntv)
        for a, s in enumerate(sites):
            Pa, va = P[:, s], v[:, s]
            if nrhs <= 64:
                ref = np.einsum("ishc,rshc->rhi", Pa.conj(), va)
                size = np.einsum("ishc,rshc->rhi", np.abs(Pa), np.abs(va))
                assert np.all(np.abs(vc[:, a] - ref) <= bound(6 * len(s), size)), (nrhs, a)
            ref = np.einsum("ishc,rhi->rshc", Pa, uc[:, a])
            size = np.einsum("ishc,rhi->rshc", np.abs(Pa), np.abs(uc[:, a]))
            assert np.all(np.abs(u[:, s] - ref) <= bound(ntv, size)), (nrhs, a)
    lat.close()
