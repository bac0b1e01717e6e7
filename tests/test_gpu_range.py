"""Fields at the ends of the float64 range on the GPU, against numpy on the same
fields times a power of two that keeps its sums in range (both exact).

Tolerance: that of the physical output elsewhere, 1e-14 of the largest value."""
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


def _times(F, e):
    """F 2^e, exactly (a division by a subnormal number would overflow on the way)."""
    return np.ldexp(F.view(float), e).view(F.dtype)


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
@pytest.mark.parametrize("scale", [-950, -1000, -1035, -1050])
@pytest.mark.parametrize("Nt,Nz", [(8, 8), (24, 16), (96, 48)])
def test_tiny_fields_are_not_taken_for_zero(Nt, Nz, scale):
    Nr, Nh = 9, Nt // 2
    rng = np.random.default_rng(Nt)
    F = rng.standard_normal((Nr, Nz, Nh)) + 1j * rng.standard_normal((Nr, Nz, Nh))
    F[:, Nz // 2], F[:, 0, 0] = 0.0, 0.0
    F[:, 0, 0] = 0.0
    for n in range(1, Nz // 2):
        F[:, Nz - n, 0] = F[:, n, 0].conj()
    F = _times(F, scale)                                # rounded to what is stored
    ref = _phys(_times(F, -scale), 3 * Nz // 2, 3 * Nt // 2)
    tol = 1e-14 * np.abs(ref).max() + 2.0 ** (-1065 - scale)
    for got in _both_routes(F, Nt):
        assert np.abs(_times(got, -scale) - ref).max() <= tol


def _products(F, eta, Nt, prec):
    """u, v, w and the five spectral products of one plane phase."""
    torch = pytest.importorskip("torch")
    ensure_lib()
    Nr, Nz, Nh = F.shape
    h = tc.tc_create_ex(Nr, Nt, Nz, 0.8, 700.0, -50.0, 1e-3, precision=prec)
    try:
        tc.tc_set_field(h, tc.TC_FIELD_MEAN_U, np.zeros(Nr))
        tc.tc_set_field(h, tc.TC_FIELD_MEAN_W, np.zeros(Nr))
        tc.tc_set_field(h, tc.TC_FIELD_V, F)
        tc.tc_set_field(h, tc.TC_FIELD_ETA, eta)
        tc.tc_split_set(h, 0, Nr, 0, Nh)
        f = [tc.tc_get_field(h, w).reshape(Nr, Nz, Nh) for w in (tc.TC_FIELD_U, tc.TC_FIELD_V, tc.TC_FIELD_W)]
        tc.tc_split_planes(h)
        tc.tc_split_finish(h)

        class A:
            pass
        a = A()
        a.__cuda_array_interface__ = {"shape": (5, Nr, Nz, Nh, 2), "typestr": "<f8", "version": 3,
                                      "data": (tc.tc_device_array(h, tc.TC_ARRAY_PROD_SLAB), False)}
        raw = torch.as_tensor(a, device="cuda").cpu().numpy()
    finally:
        tc.tc_destroy(h)
    return f, raw[..., 0] + 1j * raw[..., 1]


# peak: log2 of the largest physical velocity, so that the largest products lie just
# below 2^1024 in the first case and are subnormal in the last.  Tolerance: that of the
# products elsewhere (2e-15 of their norm) and the last place of a subnormal number.
@pytest.mark.parametrize("peak", [511, 480, -500, -528])
@pytest.mark.parametrize("Nt,Nz", [(24, 16), (96, 48)])
def test_products_at_the_ends_of_the_range(Nt, Nz, peak):
    Nr, Nh, Mz, Mt = 9, Nt // 2, 3 * Nz // 2, 3 * Nt // 2
    v, e = (x.reshape(Nr, Nz, Nh) for x in inputs(Nr, Nt, Nz, 0.8, 11, "k2", 3e-2))
    f, _ = _products(v, e, Nt, tc.TC_PREC_FP64)
    top = int(np.ceil(np.log2(max(np.abs(_phys(F, Mz, Mt)).max() for F in f))))
    f, got = _products(_times(v, peak - top), _times(e, peak - top), Nt, tc.TC_PREC_FP64)
    u, v_, w = (_phys(_times(F, -peak), Mz, Mt) for F in f)
    for k, p in enumerate((u * u - v_ * v_, u * v_, u * w, v_ * w, w * w - v_ * v_)):
        S = np.fft.rfft2(p, axes=(1, 2))[:, :, :Nh] / (Mz * Mt)
        want = np.zeros((Nr, Nz, Nh), dtype=complex)
        want[:, :Nz // 2], want[:, Nz // 2 + 1:] = S[:, :Nz // 2], S[:, Mz - Nz // 2 + 1:]
        assert np.all(np.isfinite(got[k]))
        for r in range(Nr):
            norm = max(np.sqrt(np.sum(p[r] ** 2) / (Mz * Mt)), np.linalg.norm(want[r]))
            tol = 2e-15 * norm + 2.0 ** (-1073 - 2 * peak) * np.sqrt(Nz * Nh)
            assert np.linalg.norm(_times(got[k, r], -2 * peak) - want[r]) <= tol, (k, r)


def test_products_of_a_spot():
    """Velocities that fall off in z by many orders from a spot: the theta rows of a plane
    share one scale, so the quiet rows keep fewer bits than the spot's, and the
    products, sums over all rows, must not show it (bound as in the tests of fields
    that fill the box)."""
    Nr, Nt, Nz = 9, 48, 96
    Nh, Mz, Mt = Nt // 2, 3 * Nz // 2, 3 * Nt // 2
    rng = np.random.default_rng(3)
    n = np.minimum(np.arange(Nz), Nz - np.arange(Nz))
    spot = np.exp(-(n / 8.0) ** 2)[:, None] * np.exp(-np.arange(Nh) / 6.0)         # all modes in phase at z = 0
    s = np.linspace(-1, 1, Nr)[:, None, None]
    a = 1 + 0.1 * rng.standard_normal((Nr, 1, Nh)) + 0.1j * rng.standard_normal((Nr, 1, Nh))
    a[:, :, 0] = 0.0                                    # (the slot (0, 0) is not a field's, and its lack is not local)
    v, e = 1e-2 * (1 - s * s) ** 2 * spot * a, 3e-2 * (1 - s * s) * spot * a.imag
    for F in (v, e):
        F[:, Nz // 2] = 0.0
    f, got = _products(v.astype(complex), e.astype(complex), Nt, tc.TC_PREC_FP64)
    u, v_, w = (_phys(F, Mz, Mt) for F in f)
    rows = np.abs(v_[Nr // 2]).max(axis=1)
    assert rows.min() < 1e-6 * rows.max()
    for k, p in enumerate((u * u - v_ * v_, u * v_, u * w, v_ * w, w * w - v_ * v_)):
        S = np.fft.rfft2(p, axes=(1, 2))[:, :, :Nh] / (Mz * Mt)
        want = np.zeros((Nr, Nz, Nh), dtype=complex)
        want[:, :Nz // 2], want[:, Nz // 2 + 1:] = S[:, :Nz // 2], S[:, Mz - Nz // 2 + 1:]
        for r in range(Nr):
            norm = max(np.sqrt(np.sum(p[r] ** 2) / (Mz * Mt)), np.linalg.norm(want[r]))
            assert np.linalg.norm(got[k, r] - want[r]) <= 2e-15 * norm, (k, r)
