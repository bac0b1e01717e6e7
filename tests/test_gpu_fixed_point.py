"""The plane phase of the float64 and double-float forms (fixed-point
transforms) on the GPU: the spectral products of one substep against numpy,
at the transform lengths where a plan, a pad or a block shape can go wrong.

Tolerance: the products pass six transforms (two inverse, two forward, two
operands), each within 2^-52 of its norm, and one float64 rounding at each
of three stores: below 2e-15 of the product's norm; the double-float form
truncates the result to 46 bits (2^-45 = 2.8e-14)."""
import numpy as np
import pytest

import paper_0711_1429_gb300 as tc

from helpers import ensure_lib, inputs

pytestmark = pytest.mark.gpu

# theta lengths 12 .. 1536 and axial lengths 12 .. 1536, among them odd ones
# that are padded (Nz = 10, 14, 26, 34, 50, 170) and odd numbers of rows
SHAPES = [(8, 8), (12, 10), (16, 14), (24, 18), (32, 26), (36, 34), (48, 50), (64, 66), (72, 24), (96, 102),
          (108, 12), (128, 128), (144, 44), (192, 16), (216, 170), (256, 20), (288, 48), (324, 22), (384, 10),
          (512, 28), (576, 8), (768, 12), (1024, 8), (8, 512), (12, 768), (16, 1024), (4, 4)]


def _phys(F, Mz, Mt):
    Nr, Nz, Nh = F.shape
    p = np.zeros((Nr, Mz, Mt // 2 + 1), dtype=complex)
    h = Nz // 2
    p[:, :h, :Nh], p[:, Mz - h + 1:, :Nh] = F[:, :h], F[:, h + 1:]
    return np.fft.irfft2(p, s=(Mz, Mt), axes=(1, 2)) * (Mz * Mt)


def _device(torch, h, which, shape):
    class A:
        pass
    a = A()
    a.__cuda_array_interface__ = {"shape": shape, "typestr": "<f8", "data": (tc.tc_device_array(h, which), False), "version": 3}
    return torch.as_tensor(a, device="cuda").cpu().numpy()


@pytest.mark.parametrize("Nt,Nz", SHAPES)
@pytest.mark.parametrize("prec", [tc.TC_PREC_FP64, tc.TC_PREC_DF64])
def test_products_match_numpy(Nt, Nz, prec):
    torch = pytest.importorskip("torch")
    ensure_lib()
    Nr, Nh = 9, Nt // 2
    v, e = inputs(Nr, Nt, Nz, 0.8, 5 + Nt + Nz, "k2", 3e-2)
    h = tc.tc_create_ex(Nr, Nt, Nz, 0.8, 700.0, -50.0, 1e-3, precision=prec)
    try:
        tc.tc_set_field(h, tc.TC_FIELD_V, v)
        tc.tc_set_field(h, tc.TC_FIELD_ETA, e)
        tc.tc_split_set(h, 0, Nr, 0, Nh)
        f = [tc.tc_get_field(h, w).reshape(Nr, Nz, Nh) for w in (tc.TC_FIELD_U, tc.TC_FIELD_V, tc.TC_FIELD_W)]
        tc.tc_split_planes(h)
        tc.tc_split_finish(h)
        raw = _device(torch, h, tc.TC_ARRAY_PROD_SLAB, (5, Nr, Nz, Nh, 2))
    finally:
        tc.tc_destroy(h)
    if prec == tc.TC_PREC_DF64:
        pair = raw.view(np.float32).reshape(5, Nr, Nz, Nh, 2, 2).astype(np.float64)
        raw = pair[..., 0] + pair[..., 1]
    got = raw[..., 0] + 1j * raw[..., 1]
    Mz, Mt = 3 * Nz // 2, 3 * Nt // 2
    u, v_, w = (_phys(F, Mz, Mt) for F in f)
    tol = 2e-15 if prec == tc.TC_PREC_FP64 else 6e-14
    for k, p in enumerate((u * u - v_ * v_, u * v_, u * w, v_ * w, w * w - v_ * v_)):
        S = np.fft.rfft2(p, axes=(1, 2))[:, :, :Nh] / (Mz * Mt)
        want = np.zeros((Nr, Nz, Nh), dtype=complex)
        want[:, :Nz // 2], want[:, Nz // 2 + 1:] = S[:, :Nz // 2], S[:, Mz - Nz // 2 + 1:]
        # plane by plane, against the norm of the products formed there
        for r in range(Nr):
            scale = np.sqrt(np.sum(p[r] ** 2) / (Mz * Mt)) + 1e-300
            assert np.linalg.norm(got[k, r] - want[r]) < tol * max(scale, np.linalg.norm(want[r])), (k, r)


def test_a_resting_perturbation_stays_zero():
    ensure_lib()
    h = tc.tc_create_ex(17, 24, 16, 0.7, 300.0, 0.0, 1e-3)
    try:
        tc.tc_step(h, 2)
        assert not tc.tc_get_field(h, tc.TC_FIELD_V).any() and not tc.tc_get_field(h, tc.TC_FIELD_ETA).any()
    finally:
        tc.tc_destroy(h)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_nonfinite_fields_are_flagged(bad):
    ensure_lib()
    Nr, Nt, Nz = 17, 24, 16
    v, e = inputs(Nr, Nt, Nz, 0.7, 3, "k2", 1e-2)
    e[5, 2, 3] = bad
    h = tc.tc_create_ex(Nr, Nt, Nz, 0.7, 300.0, 0.0, 1e-3)
    try:
        tc.tc_set_field(h, tc.TC_FIELD_V, v)
        tc.tc_set_field(h, tc.TC_FIELD_ETA, e)
        with pytest.raises(tc.TcError) as err:
            tc.tc_step(h, 1)
        assert err.value.code == tc.TC_ERR_NONFINITE
    finally:
        tc.tc_destroy(h)
