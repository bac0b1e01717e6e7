"""Fields at the ends of the float64 range on the GPU, against numpy on the same
fields times a power of two that keeps its sums in range (both exact).

Tolerance: that of the physical output elsewhere, 1e-14 of the largest value."""
import numpy as np
import pytest

import paper_0711_1429_gb300 as tc

from helpers import ensure_lib

pytestmark = pytest.mark.gpu


def _phys(F, Mz, Mt):
    Nr, Nz, Nh = F.shape
    p = np.zeros((Nr, Mz, Mt // 2 + 1), dtype=complex)
    h = Nz // 2
    p[:, :h, :Nh], p[:, Mz - h + 1:, :Nh] = F[:, :h], F[:, h + 1:]
    return np.fft.irfft2(p, s=(Mz, Mt), axes=(1, 2)) * (Mz * Mt)


def _both_routes(F, Nt):
    """Physical field of F from a handle and from the allocation-free call."""
    torch = pytest.importorskip("torch")
    ensure_lib()
    Nr, Nz, _ = F.shape
    Mt, Mz = 3 * Nt // 2, 3 * Nz // 2
    h = tc.tc_create_ex(Nr, Nt, Nz, 0.8, 700.0, -50.0, 1e-3)
    try:
        tc.tc_set_field(h, tc.TC_FIELD_V, F)
        a = tc.tc_get_field(h, tc.TC_FIELD_V, tc.TC_PHYSICAL).reshape(Nr, Mz, Mt)
    finally:
        tc.tc_destroy(h)
    x = torch.from_numpy(np.ascontiguousarray(F)).cuda()
    out = torch.full((Nr, Mz, Mt), float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    tc.tc_to_physical_noalloc(Nr, Nt, Nz, x.data_ptr(), out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return a, out.cpu().numpy()


@pytest.mark.parametrize("Nt,Nz", [(8, 8), (24, 16), (96, 48)])     # two and three passes
def test_sums_beyond_the_range_are_infinite(Nt, Nz):
    Nr = 9
    F = np.zeros((Nr, Nz, Nt // 2), complex)
    F[:, 0, 1], F[:, 1, 1], F[:, 2, 1] = 1.5e308, -1.1e308, 0.3e308j
    F[4:] *= 2.0 ** -8                                  # planes that stay in range
    big = np.finfo(float).max
    ref = _phys(F * 2.0 ** -8, 3 * Nz // 2, 3 * Nt // 2)            # / 2^8
    tol = 1e-14 * np.abs(ref).max()
    over = np.abs(ref) > big * 2.0 ** -8 + tol
    under = np.abs(ref) < big * 2.0 ** -8 - tol
    assert over.any() and under[4:].all()
    for got in _both_routes(F, Nt):
        assert np.array_equal(got[over], np.sign(ref[over]) * np.inf)
        assert np.all(np.abs(got[under] * 2.0 ** -8 - ref[under]) <= tol)


# Beyond the relative bound: a column of subnormal numbers has the scale of the largest
# subnormal, so its fixed-point unit is up to 2^-1071 (96 x 48: 2^-1023 2^2 for the
# value, 2^10 for the sum of up to 72 x 2 of them, 2^-62), and some 2^6 of them round.
@pytest.mark.parametrize("scale", [2.0 ** -950, 2.0 ** -1000, 2.0 ** -1035, 2.0 ** -1050])
@pytest.mark.parametrize("Nt,Nz", [(8, 8), (24, 16), (96, 48)])
def test_tiny_fields_are_not_taken_for_zero(Nt, Nz, scale):
    Nr, Nh = 9, Nt // 2
    rng = np.random.default_rng(Nt)
    F = rng.standard_normal((Nr, Nz, Nh)) + 1j * rng.standard_normal((Nr, Nz, Nh))
    F[:, Nz // 2], F[:, 0, 0] = 0.0, 0.0
    F[:, 0, 0] = 0.0
    for n in range(1, Nz // 2):
        F[:, Nz - n, 0] = F[:, n, 0].conj()
    F = (F * scale) / scale * scale                     # rounded to what is stored
    ref = _phys(F / scale, 3 * Nz // 2, 3 * Nt // 2)
    tol = 1e-14 * np.abs(ref).max() + 2.0 ** -1065 / scale
    for got in _both_routes(F, Nt):
        assert np.abs(got / scale - ref).max() <= tol
