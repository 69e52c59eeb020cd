"""Accuracy of the two FP64 forms of the operator against sums in extended precision.

hisq_apply_dslash runs on FP64 FMAs: each component is within 96 roundings of the sum of
its products' magnitudes, however small it is beside the others of its site.

A solve runs on fixed-point sums: 56 bits below the largest of the 16 hops' powers of two
(largest matrix entry times largest vector entry).  Its operator is read out of a solve that converges
at once: with m = 1/2, eta zero on odd sites, the field as the guess and a tolerance above
any residual, the odd part of psi is -D_oe of the guess.

6^3 x 10: four warps per site group and a ragged last group; 18 x 16^2 x 34: one thread per
site."""
import numpy as np
import pytest

from gpu_common import dslash_ref, rel
from oracle.oracle import Oracle, project_parity
from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import inputs as I

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
SMALL, LARGE = (6, 6, 6, 10), (18, 16, 16, 34)


def links(dims, depth):
    """links, with entries scaled by 2^-k, k uniform in 0 .. depth, and one in ten zero"""
    fat, lng = I.hisq_links(dims, 5, 0.4)
    if depth:
        r = np.random.default_rng(1)
        for w in (fat, lng):
            w.real *= np.ldexp(1.0, -r.integers(0, depth + 1, w.shape))
            w.imag *= np.ldexp(1.0, -r.integers(0, depth + 1, w.shape))
            w[r.random(w.shape) < 0.1] = 0
    return fat, lng


def field(dims, kind):
    f = I.gaussian_field(dims, 3)
    r = np.random.default_rng(2)
    if kind == "components":  # each real of its own size
        f.real *= np.ldexp(1.0, r.integers(-60, 1, f.shape))
        f.imag *= np.ldexp(1.0, r.integers(-60, 1, f.shape))
    elif kind in ("sites40", "sites300"):
        k = int(kind[5:])
        f *= np.ldexp(1.0, r.integers(-k, k + 1, f.shape[0]))[:, None]
        f[r.random(f.shape[0]) < 0.1] = 0
    elif kind == "tiny":  # sites below the block format's range
        f[r.random(f.shape[0]) < 0.1] *= 1e-290
    elif kind == "point":
        f[:] = 0
        f[r.choice(f.shape[0], 20, replace=False), 1] = 1
    elif kind == "wall":
        f = I.z2_wall_source(dims, 5, 2, 0)
    else:
        assert kind == "gauss"
    return f


class Extended:
    """D at some sites of one parity: sums in extended precision, the sums of the products'
    magnitudes, and the error bound of the fixed-point form"""

    def __init__(self, dims, fat, lng, f, par, nsites):
        X, Y, Z, T = dims
        s = np.arange(X * Y * Z * T)
        x = np.stack([s % X, s // X % Y, s // (X * Y) % Z, s // (X * Y * Z)])
        p = np.flatnonzero(x.sum(0) % 2 == par)
        if len(p) > nsites:
            p = np.sort(np.random.default_rng(4).choice(p, nsites, replace=False))
        self.sites, x = p, x[:, p]
        f = project_parity(dims, f, 1 - par)
        stride = (1, X, X * Y, X * Y * Z)
        big = lambda a: np.maximum(np.abs(a.real), np.abs(a.imag)).reshape(len(p), -1).max(1)
        mats, vecs = [], []
        for mu in range(4):
            eta = 1.0 - 2.0 * (x[:mu].sum(0) % 2)
            for n, u in ((1, fat), (3, lng)):
                for sign in (1, -1):
                    c = x[mu] + sign * n
                    nb = p + (c % dims[mu] - x[mu]) * stride[mu]
                    phase = eta * np.where((mu == 3) & ((c < 0) | (c >= dims[mu])), -1.0, 1.0)
                    w = u[p, mu] if sign > 0 else -u[nb, mu].conj().transpose(0, 2, 1)
                    mats.append(phase[:, None, None] * w)
                    vecs.append(f[nb])
        self.hits = np.sum([np.any(v != 0, axis=1) for v in vecs], axis=0)
        two = lambda q: np.where(q > 0, np.ldexp(1.0, np.frexp(q)[1]), 0)[:, None]
        A, B = [two(big(w)) for w in mats], [two(big(v)) for v in vecs]
        P = np.max([a * b for a, b in zip(A, B)], axis=0)  # what all products are aligned to
        L = np.longdouble
        self.re, self.im = np.zeros((2, len(p), 3), L)
        self.mag_re, self.mag_im, part = np.zeros((3, len(p), 3))
        for w, v, scale in zip(mats, vecs, A):
            a, b = w.real, w.imag
            c, d = (q[:, None, :] for q in (v.real, v.imag))
            self.re += (a.astype(L) * c - b.astype(L) * d).sum(-1)
            self.im += (a.astype(L) * d + b.astype(L) * c).sum(-1)
            self.mag_re += (np.abs(a * c) + np.abs(b * d)).sum(-1)
            self.mag_im += (np.abs(a * d) + np.abs(b * c)).sum(-1)
            part += (scale * (np.abs(c) + np.abs(d))[:, 0, :].sum(-1, keepdims=True)
                     + P / np.where(scale > 0, scale, 1) * (np.abs(a) + np.abs(b)).sum(-1) + 3 * P / 2)
        # a link real of a hop is cut to 2^-56 of its scale A, a neighbour's (after rounding to 2^-60
        # of its own) to 2^-56 P / A, a product of two low limbs (below 2^-58 P) is dropped, the sum
        # rounded to 2^-56 P and to FP64
        self.bound_re = 1.1 * 2.0 ** -56 * part + U * np.abs(self.re)
        self.bound_im = 1.1 * 2.0 ** -56 * part + U * np.abs(self.im)
        # sites next to a vector outside the format (2^+-700) are summed in FP64
        out = np.any([(big(v) > 0) & (big(v) < 2.0 ** -699) for v in vecs], axis=0)
        self.bound_re[out], self.bound_im[out] = 97 * U * self.mag_re[out], 97 * U * self.mag_im[out]

    def errors(self, out):
        o = out[self.sites]
        return np.abs(o.real - self.re), np.abs(o.imag - self.im)


def solve_operator(ctx, dims, f):
    """D_oe f as a solve computes it"""
    H.hisq_set_mass(ctx, 0.5)
    eta = np.zeros((int(np.prod(dims)), 3), complex)
    eta[0, 0] = 1
    prm = H.hisq_default_solve_params(batch=0, guess=1, tol=1e200)
    psi, st, status = H.hisq_solve(ctx, eta, prm, guess=project_parity(dims, f, 0))
    assert status == H.HISQ_OK and st[0]["iterations"] == 0
    return -project_parity(dims, psi, 1)


def context(dims, fat, lng):
    ctx = H.hisq_create(dims, True, 0)
    H.hisq_load_links(ctx, fat, lng)
    return ctx


@pytest.mark.parametrize("dims", [SMALL, LARGE])
@pytest.mark.parametrize("depth", [0, 60])
@pytest.mark.parametrize("kind", ["gauss", "components", "sites300", "point"])
def test_applied_operator_is_accurate_in_each_component(dims, depth, kind):
    fat, lng = links(dims, depth)
    f = field(dims, kind)
    o = Oracle(dims, fat, lng, t_antiperiodic=True)
    ctx = context(dims, fat, lng)
    try:
        for par in (0, 1):
            ref = Extended(dims, fat, lng, f, par, 3000)
            out = H.hisq_apply_dslash(ctx, par, 64, f)
            assert rel(out, dslash_ref(o, dims, f, par)) <= 1e-13  # the reference above has the same D
            er, ei = ref.errors(out)
            assert np.all(er <= 97 * U * ref.mag_re) and np.all(ei <= 97 * U * ref.mag_im)
            if kind == "point":  # where one source reaches a site: one product by 1 in each component
                one = ref.hits == 1
                assert dims == LARGE or one.sum() > 50
                assert np.array_equal(out[ref.sites][one], (ref.re + 1j * ref.im)[one].astype(complex))
    finally:
        ctx.close()


@pytest.mark.parametrize("dims", [SMALL, LARGE])
@pytest.mark.parametrize("depth", [0, 60])
@pytest.mark.parametrize("kind", ["gauss", "components", "sites40", "sites300", "tiny", "point", "wall"])
def test_solve_operator_is_accurate_at_each_site(dims, depth, kind):
    fat, lng = links(dims, depth)
    f = field(dims, kind)
    ctx = context(dims, fat, lng)
    try:
        ref = Extended(dims, fat, lng, f, 1, 3000)
        er, ei = ref.errors(solve_operator(ctx, dims, f))
        assert np.all(er <= ref.bound_re) and np.all(ei <= ref.bound_im)
    finally:
        ctx.close()


@pytest.mark.parametrize("kind", ["gauss", "sites40"])
def test_solve_operator_is_no_less_accurate_than_fp64(kind):
    """dense fields: relative to the largest product of a site, its rms error is below that of
    FP64 FMAs"""
    fat, lng = links(SMALL, 0)
    f = field(SMALL, kind)
    ctx = context(SMALL, fat, lng)
    try:
        ref = Extended(SMALL, fat, lng, f, 1, 3000)
        scale = np.maximum(ref.mag_re, ref.mag_im).max(1, keepdims=True)
        rms = lambda out: np.sqrt(np.mean([np.mean((e / scale) ** 2) for e in ref.errors(out)]))
        assert rms(solve_operator(ctx, SMALL, f)) <= rms(H.hisq_apply_dslash(ctx, 1, 64, f))
    finally:
        ctx.close()
