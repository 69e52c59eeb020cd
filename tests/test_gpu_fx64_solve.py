"""The FP64 operator inside a solve.  When device memory runs out: its scratch (the mantissas
of one field, 50 B per site) is asked for once per solve, after the buffers the solve needs
and never inside the iterations that are captured into a CUDA graph; refused, the whole
solve runs on FP64 FMAs.  For a batch on a half-volume that is not whole groups of 32 sites:
its residuals are the oracle's."""
import numpy as np
import pytest
import torch

from gpu_common import make
from oracle.oracle import Oracle, project_parity
from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DIMS = (6, 4, 6, 8)
VH = 6 * 4 * 6 * 8 // 2


@pytest.mark.parametrize("sloppy,reliable", [(64, 64), (32, 64), (16, 48)])
def test_solve_without_room_for_the_mantissas(sloppy, reliable):
    """Allocations are let through one at a time until the solve lacks only its optional
    scratch.  It then converges past the first captured iterations (the fifth on), and the
    scratch is what the context still lacked."""
    m = 0.02
    ctx, o = make(DIMS, seed=5, eps=0.3, mass=m)
    try:
        eta = I.gaussian_source(DIMS, 13, 0)
        prm = H.hisq_default_solve_params(batch=0, precision_sloppy=sloppy, precision_reliable=reliable)

        def attempt(after):
            H.hisq_inject_alloc_failure(ctx, after)
            try:
                return H.hisq_solve(ctx, eta, prm)
            except H.HisqError as e:
                assert e.status == H.HISQ_ERR_OOM, e
                return None
            finally:
                H.hisq_inject_alloc_failure(ctx, -1)

        for _ in range(40):
            got = attempt(0)
            if got is not None:
                break
            held = H.hisq_device_bytes(ctx)
            attempt(1)
            if H.hisq_device_bytes(ctx) == held:
                attempt(2)  # the double-float links of both parities come together
        psi, st, status = got
        assert status == H.HISQ_OK and st[0]["iterations"] > 8
        assert o.full_residual(m, psi.reshape(-1, 3), eta) <= 1e-10
        before = H.hisq_device_bytes(ctx)
        psi2, st2, status = H.hisq_solve(ctx, eta, prm)
        assert status == H.HISQ_OK and o.full_residual(m, psi2.reshape(-1, 3), eta) <= 1e-10
        assert 48 * VH <= H.hisq_device_bytes(ctx) - before <= 52 * VH + 512
        assert np.linalg.norm(psi - psi2) <= 1e-7 * np.linalg.norm(psi)
    finally:
        ctx.close()


def test_allocation_in_a_callers_capture_does_not_outlast_it():
    """A call that needs memory while its caller captures the stream is refused with a message
    and leaves the capture usable; a later solve captures its own iterations as usual."""
    m = 0.02
    fat, lng = I.hisq_links(DIMS, 5, 0.3)
    o = Oracle(DIMS, fat, lng, t_antiperiodic=True)
    s = torch.cuda.Stream()
    ctx = H.hisq_create(DIMS, True, 0, s.cuda_stream)
    try:
        H.hisq_load_links(ctx, fat, lng)
        H.hisq_set_mass(ctx, m)
        x = torch.zeros(2, 2 * VH, 3, dtype=torch.complex64, device="cuda")
        gw = torch.zeros(2, 2, 9, dtype=torch.complex64, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s):
            g.capture_begin()
            try:
                with pytest.raises(H.HisqError) as e:
                    H.hisq_net_wgrad(ctx, x, x, gw)  # its partial sums have no buffer yet
            finally:
                g.capture_end()
        assert "captured" in str(e.value)
        eta = I.gaussian_source(DIMS, 13, 0)
        psi, st, status = H.hisq_solve(ctx, eta, H.hisq_default_solve_params(batch=0, precision_sloppy=64))
        assert status == H.HISQ_OK and st[0]["iterations"] > 8
        assert o.full_residual(m, psi, eta) <= 1e-10
    finally:
        ctx.close()


@pytest.mark.parametrize("nrhs", [2, 3, 5, 8, 12, 13, 17])
def test_batched_residuals_on_a_ragged_volume(nrhs):
    """6^3 x 10: 33 groups of 32 sites and one of 24.  Source preparation, the reliable update
    and the full residual of fields of sizes from 1 to 1e4, in groups of up to 12 with a
    remainder; two FP64 evaluations of a residual of order 1 agree to far better than 1e-9."""
    dims, m = (6, 6, 6, 10), 0.02
    ctx, o = make(dims, seed=5, eps=0.3, mass=m)
    try:
        etas = np.stack([I.gaussian_source(dims, 13, j) * 10.0 ** (j % 5) for j in range(nrhs)])
        prm = H.hisq_default_solve_params(batch=1, max_iter=3, tol=1e-14, precision_sloppy=32)
        psi, st, status = H.hisq_solve(ctx, etas, prm)
        assert status == H.HISQ_ERR_NOT_CONVERGED
        for j in range(nrhs):
            y = project_parity(dims, o.prepare_source(m, etas[j]), 0)
            ref = o.even_residual(m, project_parity(dims, psi[j], 0), y)
            assert abs(st[j]["even_residual"] - ref) <= 1e-9 * ref
            full = o.full_residual(m, psi[j], etas[j])
            assert abs(st[j]["full_residual"] - full) <= 1e-9 * full
    finally:
        ctx.close()
