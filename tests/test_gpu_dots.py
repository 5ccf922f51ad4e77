"""The per right-hand-side dot products on whole numbers, where they have to be exact: the
FP32 sums of a thread stay below 2^24 (32 rows of values up to 511 with one right-hand side
per thread, 128 rows of values up to 255 with four), and every sum across threads has
more bits than the result. And the range: sums beyond FP32's of summands within it."""
import ctypes

import numpy as np
import pytest
import torch

import paper_1601_03184_gb300 as pkg
from paper_1601_03184_gb300 import MRHS_BF16, MRHS_F32, MRHS_F64, MRHS_PREC_FP32, Lattice, inputs

pytestmark = pytest.mark.gpu

TORCH = {MRHS_F32: torch.float32, MRHS_F64: torch.float64, MRHS_BF16: torch.bfloat16}


@pytest.fixture(scope="module")
def lat():
    lat = Lattice((4, 4, 4, 4), (2, 2, 2, 2), 2, MRHS_PREC_FP32)
    yield lat
    lat.close()


def multi_dot(lat, X, Y, K, rows, N, dtype):
    """out[k][r] = sum over the rows of conj(X_k) Y, as (re, im)"""
    f = pkg.lib()["_ZN4mrhs9multi_dotEP10mrhs_ctx_sPKvmiS3_miiPdPf"]
    f.restype = None
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int, ctypes.c_void_p, ctypes.c_size_t,
                  ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    out = torch.empty(K, N, 2, dtype=torch.float64, device="cuda")
    f(lat.ctx, X.data_ptr(), rows * 2 * N, K, Y.data_ptr(), rows, N, dtype, out.data_ptr(), None)
    lat.sync()
    return out


# N = 1, 5, 33, 132: one right-hand side per thread, rows within a warp and across warps;
# 4, 20, 64, 68, 128: four per thread, 16 rows each and, in the last two, the most (128,
# with chunks capped) and one too many for them (one per thread again); few rows (clusters of
# eight CTAs per chunk), more (of four and of two) and many (one CTA per chunk); one vector
# and a group with a remainder
@pytest.mark.parametrize("N,rows,K,dtype", [
    (1, 4096, 5, MRHS_F32), (1, 5200000, 1, MRHS_F32), (5, 4100, 5, MRHS_F32), (5, 1100000, 1, MRHS_F32),
    (33, 4100, 5, MRHS_F32), (132, 4100, 2, MRHS_F32), (20, 4100, 5, MRHS_BF16), (5, 1100000, 1, MRHS_BF16),
    (5, 4100, 5, MRHS_F64), (4, 4100, 5, MRHS_F32), (20, 4100, 5, MRHS_F32), (20, 300000, 1, MRHS_F32),
    (64, 4100, 5, MRHS_F32), (68, 4100, 5, MRHS_F32), (128, 4100, 5, MRHS_F32),
    (32, 16384, 5, MRHS_F32), (32, 16384, 10, MRHS_F32), (5, 105000, 5, MRHS_F32), (5, 105000, 10, MRHS_F32),
    (64, 2048 * 16 * 127, 1, MRHS_F32), (64, 2048 * 16 * 129, 1, MRHS_F32)])
def test_whole_numbers(lat, N, rows, K, dtype):
    top = 255 if dtype == MRHS_BF16 or N % 4 == 0 and N <= 128 else 511
    gen = torch.Generator("cuda").manual_seed(N)
    X = torch.randint(0, top + 1, (K, rows, 2, N), device="cuda", generator=gen, dtype=torch.int16).to(TORCH[dtype])
    Y = torch.randint(top // 2, top + 1, (rows, 2, N), device="cuda", generator=gen, dtype=torch.int16).to(TORCH[dtype])
    got = multi_dot(lat, X, Y, K, rows, N, dtype)
    for k in range(K):
        re = im = 0
        for x, y in zip(X[k].split(1 << 20), Y.split(1 << 20)):
            x, y = x.double(), y.double()
            re = re + (x * y).sum((0, 1))
            im = im + (x[:, 0] * y[:, 1] - x[:, 1] * y[:, 0]).sum(0)
        assert torch.equal(got[k], torch.stack((re, im), -1)), k


@pytest.mark.parametrize("N", [1, 4, 20, 64, 128])
def test_range(lat, N):
    """Squares of 2^63: two rows' sum is 2^127 times two, in FP32's range with one row per
    thread; the sum of all is not. An infinite number gives an infinite sum in its own
    right-hand side and leaves the others alone."""
    rows = 8
    X = torch.zeros(rows, 2, N, device="cuda")
    X[:, 0] = 2.0 ** 63
    got = multi_dot(lat, X, X, 1, rows, N, MRHS_F32)[0]
    assert bool((got[:, 0] == rows * 2.0 ** 126).all()) and bool((got[:, 1] == 0).all())
    Y = torch.ones_like(X)
    Y[3, 0, 0] = float("inf")
    X.fill_(1)
    X[:, 1] = 0
    got = multi_dot(lat, X, Y, 1, rows, N, MRHS_F32)[0]
    assert got[0, 0] == float("inf") and bool((got[1:, 0] == rows).all())


@pytest.mark.parametrize("nrhs", [1, 5, 16])
def test_solve_of_large_numbers(nrhs):
    """coarse GMRES of 2^62 b, numbers of modulus 2^62 (norms beyond FP32's range): 2^62
    times the solution for b, to the bound of the coarse solve's parity tests"""
    dims, agg, ntv = (8, 8, 8, 8), (2, 2, 2, 2), 2
    lat = Lattice(dims, agg, ntv, MRHS_PREC_FP32)
    lat.set_gauge(inputs.gauge_field(dims, 0.5, 1402))
    lat.build_clover(0.1, 1.2)
    lat.set_tv(lat.to_device(inputs.test_vectors(ntv, dims, 2402), MRHS_F32), MRHS_F32)
    lat.build_P()
    lat.build_Dc()
    b = inputs.gaussian_field((nrhs, lat.nagg, 2 * ntv), 4402)
    b /= np.abs(b)
    x = []
    for s in (1.0, 2.0 ** 62):
        xd = lat.field(nrhs, MRHS_F32, coarse=True)
        lat.coarse_solve(lat.to_device(s * b, MRHS_F32, coarse=True), xd, nrhs, MRHS_F32, 0.0, 5, 7)
        x.append(lat.to_host(xd, nrhs, MRHS_F32, coarse=True) / s)
    assert np.linalg.norm(x[1] - x[0]) <= 2e-5 * np.linalg.norm(x[0])
    lat.close()
