"""Restriction and prolongation of odd counts of vectors on either side of the line between
the prolongation's two forms (7), with the checks of the transfer tests."""
import pytest

from paper_1601_03184_gb300 import MRHS_PREC_FP32, MRHS_PREC_MIX_BF16
from test_gpu_transfer import test_restriction_and_prolongation as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ntv", [5, 7, 9, 13])
@pytest.mark.parametrize("prec", [MRHS_PREC_FP32, MRHS_PREC_MIX_BF16])
def test_odd_counts(ntv, prec):
    check(ntv, prec)
