"""Physical output in fixed point: both routes (a handle's tc_get_field, the
allocation-free entry point, which builds its tables on the device) against
numpy, at the planned lengths from the shortest to the longest, with odd row
counts and several radial planes a pass.

Tolerance: two transforms within 2^-52 of their norm each and one float64
rounding here, about 2 eps log2(Mt Mz) in numpy: below 1e-14 of the largest
value (20 lengths' bits at most, eps = 1.1e-16)."""
import numpy as np
import pytest

import paper_0711_1429_gb300 as tc

from helpers import ensure_lib, inputs

pytestmark = pytest.mark.gpu


def _phys(F, Mz, Mt):
    Nr, Nz, Nh = F.shape
    p = np.zeros((Nr, Mz, Mt // 2 + 1), dtype=complex)
    h = Nz // 2
    p[:, :h, :Nh], p[:, Mz - h + 1:, :Nh] = F[:, :h], F[:, h + 1:]
    return np.fft.irfft2(p, s=(Mz, Mt), axes=(1, 2)) * (Mz * Mt)


@pytest.mark.parametrize("Nr,Nt,Nz", [(9, 8, 8), (11, 8, 1024), (9, 1024, 8), (17, 12, 24), (10, 24, 12), (33, 96, 16),
                                      (13, 16, 288), (9, 576, 192), (21, 144, 48), (15, 384, 768), (9, 48, 10)])
@pytest.mark.parametrize("prec", [tc.TC_PREC_FP64, tc.TC_PREC_MIXED])
def test_physical_matches_numpy(Nr, Nt, Nz, prec):
    torch = pytest.importorskip("torch")
    ensure_lib()
    Nh, Mt, Mz = Nt // 2, 3 * Nt // 2, 3 * Nz // 2
    v, e = inputs(Nr, Nt, Nz, 0.8, 3 + Nt + Nz, "k2", 3e-2)
    h = tc.tc_create_ex(Nr, Nt, Nz, 0.8, 700.0, -50.0, 1e-3, precision=prec)
    try:
        tc.tc_set_field(h, tc.TC_FIELD_V, v)
        tc.tc_set_field(h, tc.TC_FIELD_ETA, e)
        for which in (tc.TC_FIELD_V, tc.TC_FIELD_W):
            F = tc.tc_get_field(h, which).reshape(Nr, Nz, Nh)
            ref = _phys(F, Mz, Mt)
            bound = 1e-14 * np.abs(ref).max()
            assert np.abs(tc.tc_get_field(h, which, tc.TC_PHYSICAL).reshape(ref.shape) - ref).max() <= bound
            x = torch.from_numpy(np.ascontiguousarray(F)).cuda()
            out = torch.full((Nr, Mz, Mt), float("nan"), dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            tc.tc_to_physical_noalloc(Nr, Nt, Nz, x.data_ptr(), out.data_ptr(), torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            assert np.abs(out.cpu().numpy() - ref).max() <= bound
    finally:
        tc.tc_destroy(h)
