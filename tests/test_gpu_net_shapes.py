"""The network layer and its weight gradient at the channel counts and volumes where their
tiling changes: one thread per site for 2, 4, 8 or 16 output channels (odd counts, counts
split over several passes on small lattices), 4 x 4 gradient tiles with rows dealt to up to
12 groups of threads, and volumes that are not whole blocks of 128 or 16 sites."""
import numpy as np
import pytest
import torch

from gpu_common import rel
from oracle.oracle import net_layer, net_wgrad
from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 6), (6, 10, 6, 4), (12, 12, 12, 14)])
@pytest.mark.parametrize("cin,cout", [(1, 1), (2, 5), (3, 16), (5, 3), (7, 9), (16, 16)])
@pytest.mark.parametrize("recon", [18, 12])
def test_layer_adjoint_and_gradient(dims, cin, cout, recon):
    """FP32 sums of at most 9 x 16 x 3 x 4 products: 2e-6 of the result, as for the layer's
    other tests; the gradient sums FP32 products over 48 terms at a time, the rest in
    higher precision."""
    fat, lng = I.hisq_links(dims, 3, 0.4)
    ctx = H.hisq_create(dims, True, 0, torch.cuda.current_stream().cuda_stream)
    try:
        H.hisq_load_links(ctx, fat, lng, long_recon=recon, long_scale=I.C3_NAIK if recon != 18 else 1.0)
        r = np.random.default_rng(cin * 100 + cout)
        w = ((r.standard_normal((cout, cin, 9)) + 1j * r.standard_normal((cout, cin, 9))) / 3).astype(np.complex64)
        x = np.stack([I.gaussian_field(dims, 20 + a) for a in range(cin)]).astype(np.complex64)
        u = np.stack([I.gaussian_field(dims, 60 + b) for b in range(cout)]).astype(np.complex64)
        wd, xd, ud = (torch.from_numpy(v).cuda() for v in (w, x, u))
        out, back, gw = torch.empty_like(ud), torch.empty_like(xd), torch.empty_like(wd)
        H.hisq_net_layer(ctx, wd, xd, out)
        H.hisq_net_layer(ctx, wd, ud, back, adjoint=True)
        H.hisq_net_wgrad(ctx, xd, ud, gw)
        w8, x8, u8 = (v.astype(np.complex128) for v in (w, x, u))
        assert rel(out.cpu().numpy(), net_layer(dims, fat, w8, x8)) <= 2e-6
        assert rel(gw.cpu().numpy(), net_wgrad(dims, fat, x8, u8)) <= 2e-6
        # the adjoint layer has weights conj(w) transposed, forward and backward hops swapped and negated
        wt = np.conj(w8).transpose(1, 0, 2)
        wa = np.empty_like(wt)
        wa[..., 0] = wt[..., 0]
        for mu in range(4):
            wa[..., 1 + 2 * mu], wa[..., 2 + 2 * mu] = -wt[..., 2 + 2 * mu], -wt[..., 1 + 2 * mu]
        assert rel(back.cpu().numpy(), net_layer(dims, fat, wa, u8)) <= 2e-6
    finally:
        ctx.close()
