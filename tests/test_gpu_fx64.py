"""The FP64 operator's block floating-point sums (fx64.cuh) where they can go wrong:
half-volumes that are not whole groups of 32 sites, sites split over four warps and not
(below and above 16 warps per SM), neighbouring vectors of very different size, values
outside the block format (huge, tiny, denormal, Inf, NaN) and links outside it."""
import numpy as np
import pytest

from gpu_common import dslash_ref, make, rel
from oracle.oracle import project_parity
from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# An output component is a sum of 96 products.  Oracle: 2 x 96 roundings of 2^-53 of the
# sum of the products' magnitudes at most; the operator's own error is below that.
TOL_SUM = 4 * 96 * 2.0 ** -53


def site_errors(o, dims, field, out, par):
    """largest |out - ref| per site and a bound of the sum of its terms' magnitudes: 16 hops
    of matrices with entries below 1.2 (fat) and 0.05 (long)"""
    V = int(np.prod(dims))
    ref = dslash_ref(o, dims, field, par)
    big = np.abs(field).max(axis=1).reshape(dims[::-1])
    near = np.zeros(dims[::-1])
    for ax in range(4):
        for n, w in ((1, 1.2), (3, 0.05)):
            for d in (n, -n):
                near += 12 * w * np.roll(big, d, axis=ax)
    near = near.reshape(V)
    x, y, z, t = dims
    s = np.arange(V)
    p = (s % x + s // x % y + s // (x * y) % z + s // (x * y * z)) % 2 == par
    return np.abs(out - ref).max(axis=1)[p], near[p]


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (6, 4, 6, 10), (14, 10, 12, 22), (16, 16, 16, 32), (18, 16, 16, 34)])
@pytest.mark.parametrize("spread", [0, 40, 300])
def test_sums_are_local(dims, spread):
    """Site vectors scaled by 2^k, k uniform in +-spread: the error at a site stays
    relative to its own neighbours, not to the field's largest entry."""
    ctx, o = make(dims, seed=5)
    try:
        f = I.gaussian_field(dims, 3)
        k = np.random.default_rng(1).integers(-spread, spread + 1, f.shape[0])
        f = f * np.ldexp(1.0, k)[:, None]
        f[np.random.default_rng(2).random(f.shape[0]) < 0.1] = 0
        for par in (0, 1):
            err, near = site_errors(o, dims, f, H.hisq_apply_dslash(ctx, par, 64, f), par)
            assert np.all(err <= TOL_SUM * near)
    finally:
        ctx.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e290, 1e-290, 5e-324])
@pytest.mark.parametrize("dims", [(6, 6, 4, 8), (18, 16, 16, 34)])
def test_values_outside_the_block_format(dims, value):
    """One entry of one site replaced: the sites that touch it get what FP64 gives them
    (Inf and NaN where the oracle has them), all others keep their values."""
    ctx, o = make(dims, seed=5)
    try:
        f = I.gaussian_field(dims, 3)
        ref0 = H.hisq_apply_dslash(ctx, 1, 64, f)
        f[0, 1] = complex(value, f[0, 1].imag)  # site 0 is even
        with np.errstate(all="ignore"):
            ref = dslash_ref(o, dims, f, 1)
        out = H.hisq_apply_dslash(ctx, 1, 64, f)
        touched = np.any(ref != dslash_ref(o, dims, np.where(np.arange(f.shape[0])[:, None] == 0, 0, f), 1), axis=1)
        assert np.array_equal(out[~touched], ref0[~touched])
        if np.isfinite(value):
            assert np.all(np.abs(out - ref)[touched] <= 1e-13 * (1 + abs(value)))
        else:
            a, b = out[touched].view(float), ref[touched].view(float)
            assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
            assert np.array_equal(a[np.isinf(a)], b[np.isinf(b)])
    finally:
        ctx.close()


@pytest.mark.parametrize("scale", [1e-40, 1e40, 0.0])
def test_links_outside_the_block_format(scale):
    """The links of some sites scaled out of 2^+-100 (or to zero) keep FP64 accuracy."""
    dims = (6, 4, 6, 8)
    fat, lng = I.hisq_links(dims, 5, 0.4)
    for s in (0, 17, 400):
        fat[s] *= scale
        lng[s] *= scale
    from oracle.oracle import Oracle

    o = Oracle(dims, fat, lng, t_antiperiodic=True)
    ctx = H.hisq_create(dims, True, 0)
    try:
        H.hisq_load_links(ctx, fat, lng)
        f = I.gaussian_field(dims, 3)
        for par in (0, 1):
            out, ref = H.hisq_apply_dslash(ctx, par, 64, f), dslash_ref(o, dims, f, par)
            far = np.abs(ref).max(axis=1) > 1e10
            assert np.all(np.abs(out - ref)[far] <= 1e-13 * np.abs(ref).max())
            assert np.abs(out - ref)[~far].max() <= 1e-12
        # the double-float operator's links come from the same copy
        d = H.hisq_apply_dslash(ctx, 1, H.HISQ_PREC_DF64, f) if scale < 1 else None
        assert d is None or rel(d, dslash_ref(o, dims, f, 1)) <= 2e-12
    finally:
        ctx.close()


def test_without_room_for_the_mantissas():
    """The operator still runs, in FP64 from the field itself, when its scratch is refused."""
    dims = (6, 4, 6, 8)
    ctx, o = make(dims, seed=5)
    try:
        f = I.gaussian_field(dims, 3)
        H.hisq_apply_dslash(ctx, 1, 32, f)  # every scratch field but the mantissas, FP32
        H.hisq_inject_alloc_failure(ctx, 2)  # two fields grow to FP64, the mantissas are refused
        out = H.hisq_apply_dslash(ctx, 1, 64, f)
        H.hisq_inject_alloc_failure(ctx, -1)
        ref = dslash_ref(o, dims, f, 1)
        assert rel(out, ref) <= 1e-13
        assert rel(H.hisq_apply_dslash(ctx, 1, 64, f), ref) <= 1e-13
        assert rel(project_parity(dims, H.hisq_apply_dslash(ctx, 0, 64, f), 0), dslash_ref(o, dims, f, 0)) <= 1e-13
    finally:
        ctx.close()


@pytest.mark.parametrize("nrhs", [2, 5, 7, 8, 12, 13, 25])
@pytest.mark.parametrize("guess", [0, 1])
def test_batched_residuals_match_oracle(nrhs, guess):
    """A batched solve stopped by max_iter: source preparation, the reliable update of every
    right-hand side and the full residual run as batched launches (groups of up to 12 fields
    of 1 to 8 warps, Vh = 576 = 18 groups of 32 sites).  Its residuals are the oracle's."""
    dims, m = (6, 6, 4, 8), 0.02
    ctx, o = make(dims, seed=5, eps=0.3, mass=m)
    try:
        etas = np.stack([I.gaussian_source(dims, 13, j) for j in range(nrhs)])
        start = 0.1 * np.stack([I.gaussian_source(dims, 17, j) for j in range(nrhs)]) if guess else None
        prm = H.hisq_default_solve_params(batch=1, max_iter=3, tol=1e-14, precision_sloppy=32, guess=guess)
        psi, st, status = H.hisq_solve(ctx, etas, prm, guess=start)
        assert status == H.HISQ_ERR_NOT_CONVERGED
        for j in range(nrhs):
            y = project_parity(dims, o.prepare_source(m, etas[j]), 0)
            ref = o.even_residual(m, project_parity(dims, psi[j], 0), y)
            assert abs(st[j]["even_residual"] - ref) <= 1e-9 * ref
            full = o.full_residual(m, psi[j], etas[j])
            assert abs(st[j]["full_residual"] - full) <= 1e-9 * full
    finally:
        ctx.close()
