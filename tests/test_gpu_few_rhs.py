"""The coarse stencil of few right-hand sides (a warp per coarse row) at the
edges of its range, against the oracle's stencil on the GPU's own D_c.

Every output is a sum of 9 * 2ntv complex products: in any order of the sums
the error of one entry is below gamma_n (|D_c| |x|) with n = 2 * 9 * 2ntv + 2
real terms of unit roundoff u (and sqrt(2) for the two parts of an entry)."""
import numpy as np
import pytest

import oracle
from paper_1601_03184_gb300 import (MRHS_F32, MRHS_F64, MRHS_PREC_FP32, MRHS_PREC_FP64, MRHS_PREC_MIX_BF16, Lattice,
                                    inputs, mrhs_profile, mrhs_profile_read)

pytestmark = pytest.mark.gpu

DIMS, AGG = (4, 8, 4, 8), (2, 4, 2, 2)


# 2ntv = 2, 10 and 32 (one column per lane), 34 and 64 (two), 66 and 72 (two, twice)
# (D_c of an FP64 context is built up to ntv = 32)
@pytest.mark.parametrize("ntv,prec", [(n, MRHS_PREC_FP32) for n in (1, 5, 16, 17, 32, 33, 36)]
                         + [(n, MRHS_PREC_FP64) for n in (1, 5, 16, 17, 32)])
def test_coarse_stencil_of_few_vectors(ntv, prec):
    wd = MRHS_F32 if prec == MRHS_PREC_FP32 else MRHS_F64
    u = 2.0 ** (-24 if prec == MRHS_PREC_FP32 else -53)
    lat = Lattice(DIMS, AGG, ntv, prec)
    lat.set_gauge(inputs.gauge_field(DIMS, 0.5, 1401))
    lat.build_clover(-0.1, 1.2)
    lat.set_tv(lat.to_device(inputs.test_vectors(ntv, DIMS, 2401), wd), wd)
    lat.build_P()
    lat.build_Dc()
    Dc = lat.get_Dc()
    n = 2 * 9 * 2 * ntv + 2
    for nrhs in (1, 2, 3, 4, 5, 8, 9):
        x = inputs.gaussian_field((nrhs, lat.nagg, 2 * ntv), 4401)
        if wd == MRHS_F32:
            x = x.astype(np.complex64).astype(np.complex128)
        xd, yd = lat.to_device(x, wd, coarse=True), lat.field(nrhs, wd, coarse=True)
        lat.apply_Dc(xd, yd, nrhs, wd)
        ref = oracle.apply_Dc(DIMS, AGG, Dc, x)
        size = oracle.apply_Dc(DIMS, AGG, np.abs(Dc).astype(np.complex128), np.abs(x).astype(np.complex128)).real
        err = np.abs(lat.to_host(yd, nrhs, wd, coarse=True) - ref)
        assert np.all(err <= 2 ** 0.5 * n * u / (1 - n * u) * size + 1e-300), nrhs
    lat.close()


# The reductions of the coarse GMRES at the edges of their forms: four right-hand
# sides per thread (4, 12, 20: rows joined in a warp; 128: a row is a whole warp),
# one per thread (1, 3, 33, 132: a row spans warps), each as a cluster of CTAs
# per chunk (1024 and 32768 rows of 256 aggregates are few); seven steps with a
# restart after five. The oracle's solve of the same D_c; bounds of the coarse
# solve's other parity tests.
@pytest.mark.parametrize("prec,tol", [(MRHS_PREC_FP32, 2e-5), (MRHS_PREC_FP64, 1e-10)])
@pytest.mark.parametrize("nrhs", [1, 3, 4, 12, 20, 33, 128, 132])
def test_coarse_gmres_reductions(nrhs, prec, tol):
    dims, agg, ntv = (8, 8, 8, 8), (2, 2, 2, 2), 2
    wd = MRHS_F32 if prec == MRHS_PREC_FP32 else MRHS_F64
    lat = Lattice(dims, agg, ntv, prec)
    lat.set_gauge(inputs.gauge_field(dims, 0.5, 1402))
    lat.build_clover(0.1, 1.2)
    lat.set_tv(lat.to_device(inputs.test_vectors(ntv, dims, 2402), wd), wd)
    lat.build_P()
    lat.build_Dc()
    b = inputs.gaussian_field((nrhs, lat.nagg, 2 * ntv), 4402)
    xd = lat.field(nrhs, wd, coarse=True)
    its = lat.coarse_solve(lat.to_device(b, wd, coarse=True), xd, nrhs, wd, 0.0, 5, 7)
    ref, rits = oracle.coarse_solve(dims, agg, lat.get_Dc(), b, 0.0, 5, 7)
    x = lat.to_host(xd, nrhs, wd, coarse=True)
    assert list(its) == list(rits)
    for r in range(nrhs):
        assert np.linalg.norm(x[r] - ref[r]) <= tol * np.linalg.norm(ref[r]), r
    lat.close()


# The tensor-core stencil with columns filled up to 16: 9 (the fewest), 20 and 24
# (the configurations' N_tv), 33 (five column groups for one slice), and 16 beside
# them. The entries' bound is the few-vector test's with the split operands' 2^-21
# in place of the unit roundoff of a product.
@pytest.mark.parametrize("prec", [MRHS_PREC_FP32, MRHS_PREC_MIX_BF16])
@pytest.mark.parametrize("ntv", [8, 20, 32])
def test_coarse_stencil_of_other_counts(ntv, prec):
    lat = Lattice(DIMS, AGG, ntv, prec)
    lat.set_gauge(inputs.gauge_field(DIMS, 0.5, 1403))
    lat.build_clover(-0.1, 1.2)
    lat.set_tv(lat.to_device(inputs.test_vectors(ntv, DIMS, 2403), MRHS_F32), MRHS_F32)
    lat.build_P()
    lat.build_Dc()
    Dc = lat.get_Dc()
    n = 2 * 9 * 2 * ntv + 2
    rel = n * 2.0 ** -24 / (1 - n * 2.0 ** -24) + 2 * 2.0 ** -21
    for nrhs in (9, 16, 20, 24, 33):
        if prec == MRHS_PREC_MIX_BF16 and nrhs % 16 == 0:
            continue  # single tf32 there
        x = inputs.gaussian_field((nrhs, lat.nagg, 2 * ntv), 4403).astype(np.complex64).astype(np.complex128)
        xd, yd = lat.to_device(x, MRHS_F32, coarse=True), lat.field(nrhs, MRHS_F32, coarse=True)
        mrhs_profile(lat.ctx, 1)
        lat.apply_Dc(xd, yd, nrhs, MRHS_F32)
        assert "apply_dc_tc" in mrhs_profile_read(lat.ctx)
        mrhs_profile(lat.ctx, 0)
        ref = oracle.apply_Dc(DIMS, AGG, Dc, x)
        size = oracle.apply_Dc(DIMS, AGG, np.abs(Dc).astype(np.complex128), np.abs(x).astype(np.complex128)).real
        assert np.all(np.abs(lat.to_host(yd, nrhs, MRHS_F32, coarse=True) - ref) <= 2 ** 0.5 * rel * size + 1e-300), nrhs
    lat.close()
