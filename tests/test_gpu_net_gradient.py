"""Arithmetic of the network's weight gradient, on its hop 0 (no transport, so that the sums
alone are seen): rounding no larger than that of FP32 sums of 48 rows with one rounding per
product, added up in FP64; infinities stay infinities."""
import numpy as np
import pytest
import torch

from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def gradient(dims, x, u):
    fat, lng = I.hisq_links(dims, 3, 0.4)
    ctx = H.hisq_create(dims, True, 0, torch.cuda.current_stream().cuda_stream)
    try:
        H.hisq_load_links(ctx, fat, lng)
        gw = torch.empty(u.shape[0], x.shape[0], 9, dtype=torch.complex64, device="cuda")
        H.hisq_net_wgrad(ctx, torch.from_numpy(x).cuda(), torch.from_numpy(u).cuda(), gw)
        return gw.cpu().numpy()[:, :, 0]
    finally:
        ctx.close()


def rows(a):
    """(C, V, 3) -> (V / 16, 48, C) real and imaginary parts: 16 sites at a time"""
    c = a.reshape(a.shape[0], -1, 48).transpose(1, 2, 0)
    return np.ascontiguousarray(c.real), np.ascontiguousarray(c.imag)


def fp32_rows_fp64_total(x, u):
    """sum_x u_b conj(x_a): p = fma(re, re, im * im), sum += p over 48 rows in FP32, the sums
    of the groups in FP64, the result in FP32"""
    (xr, xi), (ur, ui) = rows(x), rows(u)
    f32, f64 = np.float32, np.float64
    sr = np.zeros((xr.shape[0], u.shape[0], x.shape[0]), f32)
    si = sr.copy()
    for r in range(48):
        tr, ti = xr[:, r, None, :], xi[:, r, None, :]
        gr, gi = ur[:, r, :, None], ui[:, r, :, None]
        sr = sr + (gr.astype(f64) * tr + gi * ti).astype(f32)
        si = si + (gi.astype(f64) * tr - gr * ti).astype(f32)
    return (sr.sum(0, dtype=f64).astype(f32) + 1j * si.sum(0, dtype=f64).astype(f32)).astype(np.complex64)


@pytest.mark.parametrize("cin,cout", [(16, 16), (12, 16)])
def test_rounding(cin, cout):
    """10 % of room: the rms is over at least 384 sums, good to 4 %."""
    dims = (12, 12, 12, 14)  # 24,192 sites = 1,512 groups of 16
    x = np.stack([I.gaussian_field(dims, 20 + a) for a in range(cin)]).astype(np.complex64)
    u = np.stack([I.gaussian_field(dims, 60 + b) for b in range(cout)]).astype(np.complex64)
    ref = u.astype(complex).reshape(cout, -1) @ x.astype(complex).reshape(cin, -1).conj().T
    rms = lambda a: np.sqrt(np.mean(np.abs(a - ref) ** 2))
    assert rms(gradient(dims, x, u)) <= 1.1 * rms(fp32_rows_fp64_total(x, u))


@pytest.mark.parametrize("value", [np.inf, -np.inf, 3e38])
def test_infinities(value):
    """An infinite (or overflowing) entry gives the infinite sums of its products, with their
    signs, in the weights of its channel and leaves the others finite."""
    dims = (6, 4, 6, 8)
    x = np.stack([I.gaussian_field(dims, 20 + a) for a in range(3)]).astype(np.complex64)
    u = np.stack([I.gaussian_field(dims, 60 + b) for b in range(5)]).astype(np.complex64)
    x[:, 37, 1] = [4 - 2j, -3 + 5j, 2 + 7j]
    u[3, 37, 1] = complex(value, 0.5)
    g = gradient(dims, x, u)
    assert np.all(np.isfinite(np.delete(g, 3, axis=0).view(np.float32)))
    s = np.sign(value)
    assert np.array_equal(g[3].real, s * np.sign(x[:, 37, 1].real) * np.float32(np.inf))
    assert np.array_equal(g[3].imag, -s * np.sign(x[:, 37, 1].imag) * np.float32(np.inf))
