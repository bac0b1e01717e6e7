"""The line phase's kernels for many pairs (1216 blocks of 16 and more, also in a
column group of half of them): every launch plan of a step gives the bits of the
substeps one after the other.  Short lines, so that the pairs are what is large."""
import numpy as np
import pytest

import paper_0711_1429_gb300 as tc

from helpers import gpu_case, gpu_state, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nr", [9, 14])
@pytest.mark.parametrize("prec", [tc.TC_PREC_FP64, tc.TC_PREC_MIXED, tc.TC_PREC_DF64])
def test_launch_plans_change_no_bits_at_many_pairs(Nr, prec):
    Nt, Nz = 512, 320                           # 81920 pairs: 5120 blocks, 2560 in a group of two
    v, e = inputs(Nr, Nt, Nz, 0.883, 7, "k2", 0.05)

    def run(step):
        h = gpu_case(Nr, Nt, Nz, 0.883, 3000.0, 20.0, 1e-3, v=v, eta=e, precision=prec)
        try:
            step(h)
            return gpu_state(h, Nr, Nz, Nt // 2)
        finally:
            tc.tc_destroy(h)

    def planned(groups, deferral):
        def step(h):
            tc.tc_set_tiles(h, 0, 0, groups)
            tc.tc_set_rk_deferral(h, deferral)
            tc.tc_step(h, 1)                    # a step by itself, and two chained ones
            tc.tc_step(h, 2)
        return step

    ref = run(lambda h: tc.tc_advance_substeps(h, 9))
    for x in ref.values():
        assert np.all(np.isfinite(x)) and np.any(x != 0.0)
    for groups in (1, 2):
        for deferral in ((0,) if prec == tc.TC_PREC_FP64 else (0, 1)):
            g = run(planned(groups, deferral))
            for k in ref:
                assert np.array_equal(g[k], ref[k]), (groups, deferral, k)


@pytest.mark.parametrize("Nr", [9, 37, 282])
@pytest.mark.parametrize("prec", [tc.TC_PREC_FP64, tc.TC_PREC_MIXED, tc.TC_PREC_DF64])
def test_few_pairs_give_finite_fields_that_are_not_zero(Nr, prec):
    """(The comparison of few and many pairs elsewhere would hold for zeros too.)"""
    Nt, Nz = 12, 14
    v, e = inputs(Nr, Nt, Nz, 0.8, 3 + Nr, "box", 1e-2, jmax=Nt // 4, nmax=Nz // 4)
    h = gpu_case(Nr, Nt, Nz, 0.8, 300.0, -20.0, 2e-3, v=v, eta=e, precision=prec)
    try:
        tc.tc_step(h, 2)
        for k, x in gpu_state(h, Nr, Nz, Nt // 2).items():
            assert np.all(np.isfinite(x)) and np.any(x != 0.0), k
    finally:
        tc.tc_destroy(h)
