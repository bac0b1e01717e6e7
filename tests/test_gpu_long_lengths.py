"""Grids with a padded length beyond the planned ones (1536), which take the
float64 and double-float transforms instead of the fixed-point ones, in both
directions and with factors other than 2 and 3: one step against the oracle,
within the bound of the other parity tests."""
import pytest

import paper_0711_1429_gb300 as tc
from oracle.grid import Case
from oracle.rk import OracleSolver

from helpers import compare, gpu_case, gpu_state, inputs, oracle_state

pytestmark = pytest.mark.gpu


# padded: 1728 x 12, 12 x 1560, 24 x 1728, 1944 x 15, 36 x 1575 and one below the limit
@pytest.mark.parametrize("Nt,Nz", [(1152, 8), (8, 1040), (16, 1152), (1296, 10), (24, 1050), (1024, 8)])
@pytest.mark.parametrize("prec", [tc.TC_PREC_FP64, tc.TC_PREC_DF64])
def test_one_step_matches_the_oracle(Nt, Nz, prec):
    Nr = 9
    v, e = inputs(Nr, Nt, Nz, 0.8, 3 + Nt, "box", 1e-2, jmax=min(Nt // 4, 40), nmax=min(Nz // 4, 40))
    h = gpu_case(Nr, Nt, Nz, 0.8, 300.0, -20.0, 1e-3, v=v, eta=e, precision=prec)
    try:
        tc.tc_step(h, 1)
        g = gpu_state(h, Nr, Nz, Nt // 2)
    finally:
        tc.tc_destroy(h)
    s = OracleSolver(Case(Nr, Nt, Nz, 0.8, 300.0, -20.0, 1e-3))
    s.set_fields(v=v, eta=e)
    s.step(1)
    for k, err in compare(g, oracle_state(s)).items():
        assert err < 1e-10, (k, err)
