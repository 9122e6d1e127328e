"""Slice products of small operands: the low half of the double-float sum is a subnormal FP32 number."""
import numpy as np
import pytest

import paper_2303_00689_gb300 as kx
from tests.test_gpu_tc import kept_pairs, slices

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 131])
@pytest.mark.parametrize("scale", [0, -106, -109])
def test_small_products_keep_their_low_half(n, scale):
    """Sums of about 2^(scale + 3) whose last slice product counts units of 2^(scale - 25): FP64 holds
    the sum of the six slice products exactly, and hi + lo does as far as lo has FP32's units of 2^-149."""
    rng = np.random.default_rng(n)
    A, B = rng.normal(size=(n, n)), np.ldexp(rng.normal(size=(n, n)), scale)
    A, B = np.ldexp(A, scale // 2), np.ldexp(B, -(scale // 2))
    C = kx.sim_debug_tc_gemm(A, B, terms=6)
    pa, pb = slices(A, 3), slices(B, 3)
    ref = sum(pa[i] @ pb[j].T for i, j in kept_pairs(3))
    assert np.max(np.abs(C - ref) / (np.abs(A) @ np.abs(B).T)) < 2.0 ** -40
