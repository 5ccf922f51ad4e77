"""The coarse stencil of numbers at the end of FP32's range: the tensor-core form of 9 and
more right-hand sides gives infinities, not-a-numbers and finite results where the form
for few right-hand sides does."""
import numpy as np
import pytest

from paper_1601_03184_gb300 import MRHS_F32, MRHS_PREC_FP32, MRHS_PREC_MIX_BF16, Lattice, inputs

pytestmark = pytest.mark.gpu

DIMS, AGG, NTV = (4, 8, 4, 8), (2, 4, 2, 2), 8


@pytest.mark.parametrize("prec", [MRHS_PREC_FP32, MRHS_PREC_MIX_BF16])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, np.finfo(np.float32).max])
def test_coarse_stencil(value, prec):
    lat = Lattice(DIMS, AGG, NTV, prec)
    lat.set_gauge(inputs.gauge_field(DIMS, 0.5, 1403))
    lat.build_clover(-0.1, 1.2)
    lat.set_tv(lat.to_device(inputs.test_vectors(NTV, DIMS, 2403), MRHS_F32), MRHS_F32)
    lat.build_P()
    lat.build_Dc()
    n = 20
    x = inputs.gaussian_field((n, lat.nagg, 2 * NTV), 4403).astype(np.complex64)
    for r in (1, 7, 19):  # one number of three vectors; 2^-8 of the others, so that finite sums stay finite
        x[r] *= 2.0 ** -8
        x.imag[r, r, 3] = value

    def apply(v):
        xd, yd = lat.to_device(v, MRHS_F32, coarse=True), lat.field(len(v), MRHS_F32, coarse=True)
        lat.apply_Dc(xd, yd, len(v), MRHS_F32)
        return lat.to_host(yd, len(v), MRHS_F32, coarse=True)

    got = apply(x)
    few = np.concatenate([apply(x[r:r + 5]) for r in range(0, n, 5)])
    for a, b in ((got.real, few.real), (got.imag, few.imag)):
        assert np.array_equal(np.isnan(a), np.isnan(b))
        inf = np.isinf(b)
        assert np.array_equal(np.isinf(a), inf) and np.array_equal(a[inf], b[inf])
    fin = np.isfinite(few.real) & np.isfinite(few.imag)
    for r in range(n):  # FP32 accuracy, each form to 1e-5
        a, b = got[r][fin[r]], few[r][fin[r]]
        assert np.linalg.norm(a - b) <= 2e-5 * np.linalg.norm(b), r
    lat.close()
