"""The line phase's forms give the same bits: few pairs (points shared by the
warps of a block, solves in shared memory) and many pairs (a warp per 32 pairs,
solves in registers).  A case alone takes the first, the same case in a batch
with a large one the second.  Radial sizes: the smallest, around the rows of a
block and of a ring, and the longest line that fits shared memory and the next.
"""
import numpy as np
import pytest

import paper_0711_1429_gb300 as tc

from helpers import ensure_lib, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nr", [9, 10, 11, 12, 13, 18, 20, 35, 36, 37, 69, 133, 281, 282])
@pytest.mark.parametrize("prec", [tc.TC_PREC_FP64, tc.TC_PREC_MIXED, tc.TC_PREC_DF64])
def test_few_and_many_pairs_same_bits(Nr, prec):
    ensure_lib()
    Nt, Nz = 12, 14                             # 84 pairs: the last block of 16 is ragged
    args = (Nr, Nt, Nz, 0.8, 300.0, -20.0, 2e-3)
    v, e = inputs(Nr, Nt, Nz, 0.8, 3 + Nr, "box", 1e-2, jmax=Nt // 4, nmax=Nz // 4)
    get = lambda h: [tc.tc_get_field(h, w) for w in (tc.TC_FIELD_V, tc.TC_FIELD_ETA, tc.TC_FIELD_U, tc.TC_FIELD_W,
                                                     tc.TC_FIELD_MEAN_U, tc.TC_FIELD_MEAN_W)]
    h = tc.tc_create_ex(*args, precision=prec)
    big = tc.make_params(9, 256, 160, 0.8, 300.0, 0.0, 2e-3, precision=prec)      # 20480 pairs
    b = tc.tc_batch_create([tc.make_params(*args, precision=prec), big])
    try:
        for x in (h, tc.tc_batch_case(b, 0)):
            tc.tc_set_field(x, tc.TC_FIELD_V, v)
            tc.tc_set_field(x, tc.TC_FIELD_ETA, e)
        tc.tc_step(h, 2)
        tc.tc_batch_step(b, 2)
        for x, y in zip(get(h), get(tc.tc_batch_case(b, 0))):
            assert np.all(np.isfinite(x)) and np.any(x != 0.0) or np.array_equal(x, y)
            assert np.array_equal(x, y)
    finally:
        tc.tc_destroy(h)
        tc.tc_batch_destroy(b)
