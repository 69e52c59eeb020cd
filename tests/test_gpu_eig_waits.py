"""A wait that runs out in the block eigensolver's operator: the call reports it instead of
returning pairs of a Krylov block that was left unfinished, and leaves no status behind for
the next call."""
import numpy as np
import pytest

from gpu_common import make
from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree", [0, 8])
def test_operator_wait_timeout_is_reported_and_recovered(degree):
    dims, m = (6, 6, 6, 8), 0.05
    ctx, o = make(dims, seed=21, eps=0.3, mass=m)
    try:
        prm = H.hisq_default_eig_params(n_ev=6, n_kr=60, tol=1e-5, max_restarts=200, cheby_degree=degree, a_min=-2.0,
                                        block_size=4)
        H.hisq_set_batched_kernel(ctx, 4, 2, 1)  # the ring kernel, whose waits are bounded
        H.hisq_inject_wait_timeout(ctx, 2)
        with pytest.raises(H.HisqError) as e:
            H.hisq_eigensolve(ctx, prm)
        assert e.value.status == H.HISQ_ERR_TIMEOUT and "ran out" in str(e.value)
        H.hisq_apply_dslash(ctx, 1, 64, I.gaussian_field(dims, 3))  # nothing left behind
        eps, n = H.hisq_eigensolve(ctx, prm)
        assert n == 6
        lam, _ = o.eig_dense(0.0, 6)
        assert np.all(np.abs(eps - lam) <= 1e-6 * lam[-1])
    finally:
        ctx.close()
