"""The batched operator's default kernel (links of a site group and direction through a
shared-memory ring) shape by shape: 2, 3 or 4 right-hand sides per thread, 1, 2 or 4
blocks per SM, both vector precisions, both link formats, both parities, 1 to 64
right-hand sides (64 come in two parts of the grid), against the FP64 oracle's D; its sums
over a solve; and its waits, and those of the batched FP64 operator, made to run out.

14^3 x 18 has Vh = 24,696 = 771 full site groups of 32 and a ragged one of 24; 6^3 x 10 has
Vh = 1,080 = 33 and a ragged one of 24."""
import numpy as np
import pytest

from gpu_common import dslash_ref, make, rel
from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DIMS = (14, 14, 14, 18)
NF = 12


def warps(R):
    return 12 if R == 4 else 16


def exists(R, blocks, k):
    """the shapes the tuner chooses from: as many right-hand sides as a thread takes, and
    with several blocks per SM all fields in each"""
    return (R == 2 or k >= R) and (blocks == 1 or -(-k // R) <= warps(R) // blocks)


@pytest.fixture(scope="module", params=[12, 18])
def lat(request):
    ctx, o = make(DIMS, seed=8, eps=0.3, recon=request.param, mass=0.01)
    fields = np.stack([I.gaussian_field(DIMS, 300 + j) for j in range(NF)])
    refs = {par: [dslash_ref(o, DIMS, fields[j], par) for j in range(NF)] for par in (0, 1)}
    yield ctx, fields, refs
    ctx.close()


def batch(fields, k):
    """k fields, all different: the NF given ones, their multiples by 2, 3, ..."""
    return np.stack([fields[j % NF] * (1 + j // NF) for j in range(k)])


@pytest.mark.parametrize("R,blocks", [(R, b) for R in (2, 3, 4) for b in (1, 2, 4)])
@pytest.mark.parametrize("prec,tol", [(32, 1e-6), (16, 5e-3)])  # as for the other shapes of this operator
def test_shapes_match_oracle(lat, R, blocks, prec, tol):
    ctx, fields, refs = lat
    H.hisq_set_batched_kernel(ctx, 4, R, blocks)
    try:
        for k, par in ((1, 1), (5, 0), (12, 1), (33, 0), (64, 1)):
            if not exists(R, blocks, k):
                with pytest.raises(H.HisqError) as e:
                    H.hisq_apply_dslash_batch(ctx, par, prec, batch(fields, k))
                assert e.value.status == H.HISQ_ERR_INVALID_ARG
                continue
            out = H.hisq_apply_dslash_batch(ctx, par, prec, batch(fields, k))
            for j in range(k):
                assert rel(out[j], refs[par][j % NF] * (1 + j // NF)) <= tol, (k, par, j)
    finally:
        H.hisq_set_batched_kernel(ctx, 0)


def test_other_budgets_and_links_are_refused():
    ctx, _ = make((6, 6, 6, 10), seed=8, eps=0.3, recon=8)
    try:
        for R, blocks in ((1, 1), (5, 1), (2, 0), (2, 3), (2, 5)):
            with pytest.raises(H.HisqError):
                H.hisq_set_batched_kernel(ctx, 4, R, blocks)
        H.hisq_set_batched_kernel(ctx, 4, 2, 1)  # the ring holds 18- and 12-real links only
        with pytest.raises(H.HisqError) as e:
            H.hisq_apply_dslash_batch(ctx, 0, 32, np.zeros((2, 6 ** 3 * 10, 3), complex))
        assert e.value.status == H.HISQ_ERR_INVALID_ARG
    finally:
        ctx.close()


def solves(dims, m, k, prm, shapes):
    """the same k right-hand sides, of sizes from 1 to 1e6, under each launch shape"""
    ctx, o = make(dims, seed=13, eps=0.3, recon=12, mass=m)
    try:
        etas = np.stack([I.gaussian_source(dims, 21, j) * 10.0 ** (j % 7) for j in range(k)])
        got = []
        for shape in shapes:
            H.hisq_set_batched_kernel(ctx, *shape)
            got.append(H.hisq_solve(ctx, etas, prm))
        return o, etas, got
    finally:
        ctx.close()


@pytest.mark.parametrize("sloppy,tol", [(32, 1e-4), (16, 1e-3)])
@pytest.mark.parametrize("R,blocks,k", [(2, 1, 33), (2, 4, 5), (3, 1, 64), (3, 2, 7), (4, 1, 64), (4, 2, 9)])
def test_sums_of_an_iteration(R, blocks, k, sloppy, tol):
    """CG takes its alpha and beta from the per-field sums of these launches (33 and 64
    fields: two parts with an offset of their own).  After six iterations of every field the
    true residuals are those the register kernel leads to.  The two differ in rounding:
    FP32 sums by less than 1e-6 an iteration, FP16 fields by the roundings of 2^-11 that fall
    the other way; another field's sum would be off by a factor of 10."""
    dims, m = (6, 6, 6, 10), 0.05
    prm = H.hisq_default_solve_params(batch=1, precision_sloppy=sloppy, max_iter=6, tol=1e-14)
    _, _, got = solves(dims, m, k, prm, ((4, R, blocks), (1, 4, 0)))
    (_, ring, s0), (_, reg, s1) = got
    assert s0 == s1 == H.HISQ_ERR_NOT_CONVERGED
    for a, b in zip(ring, reg):
        assert abs(a["even_residual"] - b["even_residual"]) <= tol * b["even_residual"]


@pytest.mark.parametrize("sloppy", [32, 16])
@pytest.mark.parametrize("blocks,k", [(1, 33), (4, 5)])
def test_whole_solve(blocks, k, sloppy):
    """Every field converges to the true residual (fields finish at different times, so the
    batch shrinks to one), in as many iterations as with the register kernel but for an
    update one reliable step earlier or later."""
    dims, m = (6, 6, 6, 10), 0.05
    prm = H.hisq_default_solve_params(batch=1, precision_sloppy=sloppy)
    o, etas, got = solves(dims, m, k, prm, ((4, 2, blocks), (1, 4, 0)))
    for psi, _, status in got:
        assert status == H.HISQ_OK
        for j in range(k):
            assert o.full_residual(m, psi[j], etas[j]) <= 1e-10
    for a, b in zip(got[0][1], got[1][1]):
        assert abs(a["iterations"] - b["iterations"]) <= max(4, 0.05 * b["iterations"])


@pytest.mark.parametrize("R,blocks", [(2, 1), (3, 2), (4, 1)])
def test_operator_wait_timeout_is_reported_and_recovered(lat, R, blocks):
    """Every warp gives up at its first wait, the copies in flight land, the launch ends."""
    ctx, fields, refs = lat
    H.hisq_set_batched_kernel(ctx, 4, R, blocks)
    try:
        H.hisq_inject_wait_timeout(ctx, 2)
        with pytest.raises(H.HisqError) as e:
            H.hisq_apply_dslash_batch(ctx, 1, 16, fields[:4])
        assert e.value.status == H.HISQ_ERR_TIMEOUT and "ran out" in str(e.value)
        out = H.hisq_apply_dslash_batch(ctx, 1, 16, fields[:4])  # the injection was one-shot
        for j in range(4):
            assert rel(out[j], refs[1][j]) <= 5e-3
    finally:
        H.hisq_set_batched_kernel(ctx, 0)


@pytest.mark.parametrize("k", [2, 5, 12])
def test_fp64_batch_wait_timeout_is_reported_and_recovered(k):
    """The first ring of a batched solve is that of the FP64 source preparation."""
    dims, m = (6, 6, 6, 10), 0.05
    ctx, o = make(dims, seed=13, eps=0.3, mass=m)
    try:
        etas = np.stack([I.gaussian_source(dims, 22, j) for j in range(k)])
        prm = H.hisq_default_solve_params(batch=1, precision_sloppy=32)
        H.hisq_inject_wait_timeout(ctx, 2)
        with pytest.raises(H.HisqError) as e:
            H.hisq_solve(ctx, etas, prm)
        assert e.value.status == H.HISQ_ERR_TIMEOUT and "ran out" in str(e.value)
        psi, st, status = H.hisq_solve(ctx, etas, prm)
        assert status == H.HISQ_OK
        for j in range(k):
            assert o.full_residual(m, psi[j], etas[j]) <= 1e-10
    finally:
        ctx.close()
