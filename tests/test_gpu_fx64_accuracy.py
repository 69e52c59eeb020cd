"""Accuracy of the FP64 operator against sums in extended precision: hisq_apply_dslash runs
on FP64 FMAs, so that each component is within 96 roundings of the sum of its products'
magnitudes, however small it is beside the others of its site."""
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
    elif kind == "sites300":
        f *= np.ldexp(1.0, r.integers(-300, 301, f.shape[0]))[:, None]
        f[r.random(f.shape[0]) < 0.1] = 0
    elif kind == "point":
        f[:] = 0
        f[r.choice(f.shape[0], 20, replace=False), 1] = 1
    else:
        assert kind == "gauss"
    return f


class Extended:
    """D at some sites of one parity: sums in extended precision and the sums of the products'
    magnitudes"""

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
        L = np.longdouble
        self.re, self.im = np.zeros((2, len(p), 3), L)
        self.mag_re, self.mag_im = np.zeros((2, len(p), 3))
        for w, v in zip(mats, vecs):
            a, b = w.real, w.imag
            c, d = (q[:, None, :] for q in (v.real, v.imag))
            self.re += (a.astype(L) * c - b.astype(L) * d).sum(-1)
            self.im += (a.astype(L) * d + b.astype(L) * c).sum(-1)
            self.mag_re += (np.abs(a * c) + np.abs(b * d)).sum(-1)
            self.mag_im += (np.abs(a * d) + np.abs(b * c)).sum(-1)

    def errors(self, out):
        o = out[self.sites]
        return np.abs(o.real - self.re), np.abs(o.imag - self.im)


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
