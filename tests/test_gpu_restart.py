"""A set state made ready to step: the initial Runge-Kutta memory
H_1 = (M + alpha_1 dt L) x and u, w, as the state image holds them, against the
oracle's bands, at the radial sizes where the sharing of rows over warps and lanes
can go wrong and on both sides of the rule between the two launch shapes (1216
blocks of 16 pairs).  Tolerance: that of one step, 1e-10."""
import numpy as np
import pytest

import paper_0711_1429_gb300 as tc
from oracle import operators as op
from oracle.grid import Case
from oracle.rk import SMR91, OracleSolver

from helpers import gpu_case, inputs, relerr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nr,Nt,Nz", [(9, 12, 14), (10, 12, 14), (11, 12, 14), (15, 16, 16), (16, 16, 16), (33, 16, 16),
                                      (64, 16, 16), (9, 256, 160), (10, 256, 160), (13, 256, 160), (22, 256, 160)])
@pytest.mark.parametrize("prec", [tc.TC_PREC_FP64, tc.TC_PREC_MIXED, tc.TC_PREC_DF64])
def test_initial_memory_and_velocity(Nr, Nt, Nz, prec):
    args = (Nr, Nt, Nz, 0.8, 300.0, -20.0, 2e-3)
    v, e = inputs(Nr, Nt, Nz, 0.8, 3 + Nr, "box", 1e-2, jmax=Nt // 4, nmax=Nz // 4)
    h = gpu_case(*args, v=v, eta=e, precision=prec)
    try:
        img = np.frombuffer(tc.tc_save_state(h), np.uint8)
    finally:
        tc.tc_destroy(h)
    f = img[40:40 + 96 * Nr * Nz * Nt // 2].view(np.complex128).reshape(6, Nr, Nz, Nt // 2)     # v, eta, u, w, Hv, He
    s = OracleSolver(Case(*args))
    s.set_fields(v=v, eta=e)
    adt = SMR91.floats()[0][0] * s.case.dt
    va, ea = s._gather(s.v), s._gather(s.eta)
    Hv = op.band_apply(s.S, s.Mv, va) + adt * op.band_apply(s.S, s.Lv, va)
    He = op.band_apply(s.S, s.Me, ea) + adt * op.band_apply(s.S, s.Le, ea)
    Hv[[0, 1, Nr - 2, Nr - 1]] = 0.0
    He[[0, Nr - 1]] = 0.0
    u, _, w = s.velocity()
    for got, want in ((s._gather(f[4]), Hv), (s._gather(f[5]), He), (f[2], u), (f[3], w)):
        assert np.any(want != 0.0) and relerr(got, want) < 1e-10
