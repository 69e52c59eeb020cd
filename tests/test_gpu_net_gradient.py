"""Arithmetic of the network's weight gradient, on its hop 0 (no transport, so that the sums
alone are seen): infinities stay infinities."""
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
