"""The split-tf32 D_c assembly at the edges of its chunks, column groups and site
table, against the oracle's contraction of the GPU's own P (1e-5 relative, the
bound of FP32 work here; the split form measures 4e-7).

ntv 1, 3, 20 and 32: part of a warp, two rows of a chirality, a ragged last group
and full warps; (2,2,2,2): 16 sites, faces of 8; (1,4,4,4): no hop inside a
direction, both faces of every site; (3,2,2,2): a chunk of four that does not
divide the 24 sites' faces of 8 and 12; (8,8,2,4): 512 sites, beyond the table."""
import numpy as np
import pytest

import oracle
from paper_1601_03184_gb300 import MRHS_F32, MRHS_PREC_FP32, Lattice, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ntv", [1, 3, 20, 32])
@pytest.mark.parametrize("agg,dims", [((2, 2, 2, 2), (4, 4, 4, 8)), ((1, 4, 4, 4), (2, 8, 8, 8)),
                                      ((3, 2, 2, 2), (6, 4, 4, 4)), ((8, 8, 2, 4), (16, 16, 4, 8))])
def test_coarse_operator_blocks(agg, dims, ntv):
    U = inputs.gauge_field(dims, 0.5, 1601)
    A = oracle.clover(dims, U, -0.1, 1.2)
    lat = Lattice(dims, agg, ntv, MRHS_PREC_FP32)
    lat.set_gauge(U)
    lat.build_clover(-0.1, 1.2)
    lat.set_tv(lat.to_device(inputs.test_vectors(ntv, dims, 2601), MRHS_F32), MRHS_F32)
    lat.build_P()
    lat.build_Dc()
    ref = oracle.coarse_op(dims, agg, U, A, lat.get_P())
    got = lat.get_Dc()
    for k in range(9):
        assert np.linalg.norm(got[:, k] - ref[:, k]) <= 1e-5 * np.linalg.norm(ref[:, k]), k
    lat.close()
