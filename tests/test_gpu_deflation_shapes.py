"""The CUDA-core deflation at the sizes where its launch changes: 8, 4, 2 or 1 vectors per
block of the projection (fewer blocks than half the SMs), ragged vector groups and site
chunks, and expansion blocks of 64 or 256 threads."""
import numpy as np
import pytest

from gpu_common import make, orthonormal_even_set, rel, stored_vectors
from oracle.oracle import deflation_guess, project_parity
from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,n", [((8, 8, 8, 8), 5), ((12, 12, 12, 16), 41), ((16, 16, 16, 16), 37),
                                    ((16, 16, 16, 16), 83), ((24, 16, 16, 26), 17)])
@pytest.mark.parametrize("storage", [32, 16, 15, 14])
def test_guess_matches_oracle(dims, n, storage):
    """FP32 products and sums of 16 sites per thread, then FP64: 1e-5 as for the other
    tests of this path (the stored values are the oracle's vectors)."""
    m = 0.01
    ctx, _ = make(dims, seed=21, eps=0.3, mass=m)
    try:
        lam, vecs = orthonormal_even_set(dims, n, seed=5)
        H.hisq_set_eigvecs(ctx, vecs, lam, storage)
        b = project_parity(dims, I.gaussian_field(dims, 31), 0)
        ref = deflation_guess(stored_vectors(vecs, storage, I.volume(dims) // 2), lam + 4 * m * m, b)
        assert rel(H.hisq_deflate(ctx, b), ref) <= 1e-5
    finally:
        ctx.close()
