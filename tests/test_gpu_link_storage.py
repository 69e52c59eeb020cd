"""The FP64 links a context keeps are the ones it was given: entries far below the largest
of their site (the long links' coefficient, zeroed or nearly diagonal matrices) keep their
own 53 bits.  A unit point source reads them out one by one, since each output component is
then one link entry times 1; the double-float operator splits the stored links into pairs
of FP32 numbers, good to 2^-47."""
import numpy as np
import pytest

from gpu_common import dslash_ref
from oracle.oracle import Oracle
from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import inputs as I

DIMS = (8, 8, 8, 8)  # hops of 1 and 3 sites, forward and backward, all lead to different sites


def spread_links(depth, seed):
    """links whose entries are scaled by 2^-k, k uniform in 0 .. depth, one in ten zero"""
    fat, lng = I.hisq_links(DIMS, seed, 0.4)
    r = np.random.default_rng(seed)
    for w in (fat, lng):
        w.real *= np.ldexp(1.0, -r.integers(0, depth + 1, w.shape))
        w.imag *= np.ldexp(1.0, -r.integers(0, depth + 1, w.shape))
        w[r.random(w.shape) < 0.1] = 0
    return fat, lng


def point_sources(n, seed):
    """n unit point sources on random sites and colours"""
    r = np.random.default_rng(seed)
    V = int(np.prod(DIMS))
    for s, c in zip(r.choice(V, n, replace=False), r.integers(0, 3, n)):
        x, y, z, t = s % 8, s // 8 % 8, s // 64 % 8, s // 512
        f = np.zeros((V, 3), complex)
        f[s, c] = 1
        yield int(1 - (x + y + z + t) % 2), f


@pytest.mark.gpu
@pytest.mark.parametrize("depth", [0, 8, 40, 90, 120, 200])
def test_double_float_operator_reads_the_links(depth):
    """2^-44: the pair's 2^-47 and the roundings of one complex product.  From a depth of
    about 127 places below the site's largest entry on, sites are stored as plain FP64."""
    fat, lng = spread_links(min(depth, 100), 5)
    if depth > 100:  # FP32's exponents end at 2^-126: only the storage form of these sites differs
        lng[::7, 0, 0, 0] = 2.0 ** -depth
    o = Oracle(DIMS, fat, lng, t_antiperiodic=True)
    ctx = H.hisq_create(DIMS, True, 0)
    try:
        H.hisq_load_links(ctx, fat, lng)
        for par, f in point_sources(12, 7):
            out, ref = H.hisq_apply_dslash(ctx, par, H.HISQ_PREC_DF64, f), dslash_ref(o, DIMS, f, par)
            for a, b in ((out.real, ref.real), (out.imag, ref.imag)):
                seen = np.abs(b) > 2.0 ** -100
                assert np.all(np.abs(a - b)[seen] <= 2.0 ** -44 * np.abs(b)[seen])
    finally:
        ctx.close()
