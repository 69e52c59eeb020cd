"""The calls whose speed this framework is judged by, as a user's program makes them.

Sizes are those of the lattice configurations in paper_2502_00152_gb300/inputs.py
(8^4, 16^3x32, 24^3x48, 32^3x64) and ragged ones between them.  Every case is one call
(or one short sequence of calls) of the public binding on inputs made from the seed:
gauge links of the synthetic recipe (thin SU(3) links exp(i eps A), fat = c1 U, long =
c3 U U U), sources, eigenvectors and network weights.

Kinds of case:
  solve    hisq_solve_device / hisq_solve: M psi = eta to |eta - M psi| <= 1e-10 |eta|
  deflate  hisq_deflate_noalloc: x = V Lambda^-1 V^dag b over stored vectors
  layer    PTLayer: forward, adjoint and weight gradient of one network layer (training)
  guess    GuessNet: the network's prediction for three right-hand sides (inference)
  eig      hisq_eigensolve: the lowest eigenpairs of the even-site operator
"""
import math

import numpy as np
import torch

from paper_2502_00152_gb300 import hisq as H
from paper_2502_00152_gb300 import learned

C1, C3 = 9.0 / 8.0, -1.0 / 24.0
LARGEST = 32 ** 3 * 64 * 12  # sites x right-hand sides of the largest solve


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest whole solve: pure FP64 CG on a point source (validation runs, unit tests of an analysis)
        solve("point_8x8_fp64", (8, 8, 8, 8), 0.05, 0.4, source="point", sloppy=64, recon=18),
        # one propagator column on a small lattice in mixed precision: launches and latency count
        solve("point_16x32_half", (16, 16, 16, 32), 0.01, 0.3, source="point", sloppy=16, recon=12),
        # one stochastic source on the training lattice, reliable updates in double-float arithmetic
        solve("gauss_24x48_df64", (24, 24, 24, 48), 0.003, 0.3, sloppy=16, recon=12, reliable=48),
        # one stochastic source on the benchmark's single-source lattice, FP64 reliable updates
        solve("gauss_32x64_half", (32, 32, 32, 64), 0.002, 0.3, sloppy=16, recon=12),
        # the benchmark's batch (4 Gaussian sources x 3 colours together): the largest call
        solve("batch12_32x64_half", (32, 32, 32, 64), 0.002, 0.3, source="colour", nrhs=12, sloppy=16, recon=12),
        # library defaults from host memory: FP32 vectors, uncompressed links, an odd batch on a ragged lattice
        solve("host_batch5_ragged", (14, 10, 12, 22), 0.01, 0.3, nrhs=5, sloppy=32, recon=18, host=True),
        # wall sources on a small lattice with 64 eigenpairs: projection, expansion and re-deflation in the solve
        solve("deflated_walls12_16x32", (16, 16, 16, 32), 0.01, 0.3, source="z2", nrhs=12, sloppy=16, recon=12,
              n_ev=64, storage=14),
        # a deflated guess alone, 128 single-precision vectors (a caller with a solver of its own)
        deflate("deflate128_24x48", (24, 24, 24, 48), 128, 32),
        # the same call where it is short: few half-precision vectors, ragged lattice
        deflate("deflate37_ragged", (14, 6, 10, 22), 37, 14),
        # training of the guess network: forward, adjoint and weight gradient of its widest layer
        layer("layer16_24x48", (24, 24, 24, 48), 16, 16, True),
        # the network's guess for three right-hand sides before a solve
        guess("guess_16x32", (16, 16, 16, 32), True),
        # low modes of a new configuration (set-up of every deflated run)
        eig("eig16_8x16", (8, 8, 8, 16), 16, 64, 8),
    ]


def solve(name, dims, mass, eps, source="gauss", nrhs=1, sloppy=16, recon=12, reliable=64, host=False, n_ev=0,
          storage=32):
    return dict(name=name, kind="solve", X=dims[0], Y=dims[1], Z=dims[2], T=dims[3], mass=mass, eps=eps,
                source=source, nrhs=nrhs, sloppy=sloppy, recon=recon, reliable=reliable, host=host, n_ev=n_ev,
                storage=storage)


def deflate(name, dims, n, storage):
    return dict(name=name, kind="deflate", X=dims[0], Y=dims[1], Z=dims[2], T=dims[3], n=n, storage=storage)


def layer(name, dims, cin, cout, bf16):
    return dict(name=name, kind="layer", X=dims[0], Y=dims[1], Z=dims[2], T=dims[3], cin=cin, cout=cout, bf16=bf16)


def guess(name, dims, bf16):
    return dict(name=name, kind="guess", X=dims[0], Y=dims[1], Z=dims[2], T=dims[3], bf16=bf16)


def eig(name, dims, n_ev, n_kr, block):
    return dict(name=name, kind="eig", X=dims[0], Y=dims[1], Z=dims[2], T=dims[3], n_ev=n_ev, n_kr=n_kr, block=block)


def draw(rng):
    """One more case of the same ranges: volumes log-uniform up to 32^3x64, every extent even."""
    kind = rng.choice(("solve", "solve", "solve", "solve", "solve", "deflated", "deflate", "deflate", "layer", "layer",
                       "guess", "eig"))
    if kind == "solve":
        dims = _dims(rng, 8 ** 4, 32 ** 3 * 64)
        V = dims[0] * dims[1] * dims[2] * dims[3]
        nrhs = 1 if rng.random() < 0.4 else rng.randint(2, min(24, max(2, LARGEST // V)))
        sloppy = rng.choice((16, 16, 16, 32, 32, 64)) if nrhs == 1 and V < 2 ** 18 else rng.choice((16, 16, 32))
        c = solve("", dims, round(math.exp(rng.uniform(math.log(0.002), math.log(0.05))), 5),
                  rng.choice((0.25, 0.3, 0.4)), rng.choice(("point", "gauss", "colour", "z2")), nrhs, sloppy,
                  rng.choice((18, 12, 12, 8)), 48 if sloppy != 64 and rng.random() < 0.25 else 64,
                  V * nrhs < 2 ** 18 and rng.random() < 0.3)
    elif kind == "deflated":
        dims = _dims(rng, 8 ** 4, 16 ** 3 * 32)
        c = solve("", dims, round(rng.uniform(0.005, 0.03), 5), 0.3, rng.choice(("gauss", "colour", "z2")),
                  rng.randint(1, 16), rng.choice((16, 32)), rng.choice((18, 12)), 64, False, rng.choice((16, 24, 32)),
                  rng.choice((32, 15, 14)))
    elif kind == "deflate":
        dims = _dims(rng, 8 ** 4, 24 ** 3 * 48)
        V = dims[0] * dims[1] * dims[2] * dims[3]
        n = int(math.exp(rng.uniform(math.log(8), math.log(256))))
        c = deflate("", dims, max(8, min(n, 128 * 24 ** 3 * 48 // V)), rng.choice((32, 32, 16, 15, 14)))
    elif kind == "layer":
        c = layer("", _dims(rng, 6 ** 4, 24 ** 3 * 48), rng.choice((1, 3, 5, 8, 16, 16)),
                  rng.choice((1, 3, 7, 12, 16, 16)), rng.random() < 0.6)
    elif kind == "guess":
        c = guess("", _dims(rng, 6 ** 4, 16 ** 3 * 32), rng.random() < 0.7)
    else:
        c = eig("", _dims(rng, 8 ** 4, 2 * 8 ** 4), rng.choice((8, 12, 16)), rng.choice((64, 80)),
                rng.choice((4, 8, 16)))
    del c["name"]
    return c


def _dims(rng, lo, hi):
    """Even extents >= 6 whose volume is log-uniform in about [lo, hi]."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = target ** 0.25
    d = [max(6, 2 * round(side * math.exp(rng.uniform(-0.25, 0.25)) / 2)) for _ in range(3)]
    t = max(6, 2 * round(target / (d[0] * d[1] * d[2]) / 2))
    while d[0] * d[1] * d[2] * t > hi and t > 6:
        t -= 2
    while d[0] * d[1] * d[2] * t > hi:
        d[d.index(max(d))] -= 2
    return d[0], d[1], d[2], min(t, 64)


# ------------------------------------------------------------------ inputs
def _shape(case):
    return case["X"], case["Y"], case["Z"], case["T"]


def _normal(seed, stream, *size):
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 64 + stream)
    return torch.randn(*size, generator=g, device="cuda", dtype=torch.float64)


def _complex(seed, stream, *size):
    return torch.view_as_complex(_normal(seed, stream, *size, 2))


def _links(dims, seed, eps):
    """(fat, long) links [s][mu][3][3] complex128 on the GPU."""
    X, Y, Z, T = dims
    V = X * Y * Z * T
    w = _normal(seed, 1, V, 4, 8) * (0.5 * eps)
    a = torch.zeros(V, 4, 3, 3, dtype=torch.complex128, device="cuda")
    d8 = w[..., 7] / math.sqrt(3.0)
    for i, d in enumerate((w[..., 2] + d8, d8 - w[..., 2], -2 * d8)):
        a[..., i, i] = d.to(torch.complex128)
    for i, j, p, q in ((0, 1, 0, 1), (0, 2, 3, 4), (1, 2, 5, 6)):
        a[..., i, j] = torch.complex(w[..., p], -w[..., q])
        a[..., j, i] = torch.complex(w[..., p], w[..., q])
    del w
    # exp(i A) to third order, then Gram-Schmidt back onto SU(3)
    ia = 1j * a
    ia2 = ia @ ia
    u = torch.eye(3, dtype=torch.complex128, device="cuda") + ia + 0.5 * ia2 + (ia2 @ ia) / 6
    del a, ia, ia2
    r0 = u[..., 0, :] / torch.linalg.vector_norm(u[..., 0, :], dim=-1, keepdim=True)
    r1 = u[..., 1, :] - (r0.conj() * u[..., 1, :]).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = torch.stack([r0[..., 1] * r1[..., 2] - r0[..., 2] * r1[..., 1], r0[..., 2] * r1[..., 0] - r0[..., 0] * r1[..., 2],
                      r0[..., 0] * r1[..., 1] - r0[..., 1] * r1[..., 0]], dim=-1).conj()
    u = torch.stack([r0, r1, r2], dim=-2)
    lng = torch.empty_like(u)
    g = u.view(T, Z, Y, X, 4, 3, 3)
    for mu in range(4):
        n = g[..., mu, :, :]
        lng[:, mu] = (C3 * (n @ torch.roll(n, -1, 3 - mu) @ torch.roll(n, -2, 3 - mu))).reshape(V, 3, 3)
    return C1 * u, lng


def _context(dims, seed, eps, recon, stream):
    fat, lng = (x.cpu().numpy() for x in _links(dims, seed, eps))
    ctx = H.hisq_create(dims, t_antiperiodic=True, device=0, cuda_stream=stream)
    H.hisq_load_links(ctx, fat, lng, long_recon=recon, long_scale=C3 if recon != 18 else 1.0)
    return ctx


def _sources(case, seed):
    """eta [nrhs][V][3] complex128 on the GPU."""
    X, Y, Z, T = _shape(case)
    V, k = X * Y * Z * T, case["nrhs"]
    if case["source"] == "gauss":
        return _complex(seed, 2, k, V, 3)
    eta = torch.zeros(k, V, 3, dtype=torch.complex128, device="cuda")
    if case["source"] == "colour":  # colour-diluted Gaussian sources
        for j in range(k):
            eta[j, :, j % 3] = _complex(seed, 3 + j // 3, V)
    elif case["source"] == "z2":  # +-1 on one timeslice, one colour
        vs = X * Y * Z
        for j in range(k):
            t0 = (j // 3) * T // 8 % T
            eta[j, t0 * vs:(t0 + 1) * vs, j % 3] = torch.sign(_normal(seed, 3 + j // 3, vs)).to(torch.complex128)
    else:  # a point on an even site, one colour each
        rs = np.random.RandomState(seed % (1 << 31))
        for j in range(k):
            x, y, z, t = (int(rs.randint(0, n)) for n in (X, Y, Z, T))
            x = (x - (x + y + z + t) % 2) % X
            eta[j, x + X * (y + Y * (z + Z * t)), j % 3] = 1.0
    return eta


def _even(dims):
    """indices of the even sites, ascending"""
    X, Y, Z, T = dims
    s = torch.arange(X * Y * Z * T, device="cuda")
    return s[(s % X + s // X % Y + s // (X * Y) % Z + s // (X * Y * Z)) % 2 == 0]


def _vectors(case, seed):
    """stored vectors (n, V, 3) (unit Gaussian even-site fields), their eigenvalues and b (3, Vh)."""
    dims, n = _shape(case), case["n"]
    ev = _even(dims)
    v = torch.zeros(n, 2 * len(ev), 3, dtype=torch.complex128, device="cuda")
    for i in range(n):
        f = _complex(seed, 1000 + i, len(ev), 3)
        v[i, ev] = f / torch.linalg.vector_norm(f)
    g = torch.Generator().manual_seed(int(seed))
    eps = torch.sort(0.006 + 0.5 * torch.rand(n, generator=g, dtype=torch.float64)).values
    return v, eps, _complex(seed, 2, 3, len(ev))


def _weights(case, seed):
    w = _complex(seed, 4, case["cout"], case["cin"], 9) / math.sqrt(18.0 * case["cin"])
    return w.to(torch.complex64)


def _channels(case, seed, stream, c):
    X, Y, Z, T = _shape(case)
    return _complex(seed, stream, c, X * Y * Z * T, 3).to(torch.complex64)


# ------------------------------------------------------------------ prepare, run
def prepare(case, seed):
    dims, kind = _shape(case), case["kind"]
    st = {"case": case}
    if kind == "solve":
        st["stream"] = torch.cuda.Stream()
        st["ctx"] = ctx = _context(dims, seed, case["eps"], case["recon"], st["stream"].cuda_stream)
        H.hisq_set_mass(ctx, case["mass"])
        if case["n_ev"]:
            H.hisq_eigensolve(ctx, H.hisq_default_eig_params(n_ev=case["n_ev"], n_kr=case["n_ev"] * 3 // 2 + 32, tol=1e-6,
                                                             max_restarts=100, cheby_degree=40, a_min=-2.0,
                                                             storage_precision=case["storage"], seed=1000, block_size=16))
        st["params"] = H.hisq_default_solve_params(precision_sloppy=case["sloppy"], precision_reliable=case["reliable"],
                                                   deflate=1 if case["n_ev"] else 0)
        st["eta"] = _sources(case, seed)
        if case["host"]:
            st["eta"] = st["eta"].cpu().numpy()
        else:
            st["psi"] = torch.zeros_like(st["eta"])
    elif kind == "eig":
        st["ctx"] = _context(dims, seed, 0.3, 12, None)
        H.hisq_set_mass(st["ctx"], 0.01)
        st["params"] = H.hisq_default_eig_params(n_ev=case["n_ev"], n_kr=case["n_kr"], tol=1e-6, max_restarts=200,
                                                 cheby_degree=20, a_min=-2.0, seed=1000, block_size=case["block"])
    else:  # on torch's own stream, so that its tensors are ordered with the library's work
        st["ctx"] = ctx = _context(dims, seed, 0.3, 12, torch.cuda.current_stream().cuda_stream)
        H.hisq_set_mass(ctx, 0.003)
        if kind == "deflate":
            v, eps, st["b"] = _vectors(case, seed)
            H.hisq_set_eigvecs(ctx, v.cpu().numpy(), eps.numpy(), case["storage"])
            st["x"] = torch.zeros_like(st["b"])
        elif kind == "layer":
            st["x"] = _channels(case, seed, 2, case["cin"]).requires_grad_(True)
            st["w"] = _weights(case, seed).requires_grad_(True)
            st["gout"] = _channels(case, seed, 3, case["cout"])
        else:
            st["net"] = learned.GuessNet(ctx, seed=int(seed) % (1 << 31), bf16=case["bf16"])
            st["x"] = _channels(case, seed, 2, 3)
    torch.cuda.synchronize()
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "solve":
        if case["host"]:
            psi, _, status = H.hisq_solve(ctx, st["eta"], st["params"])
        else:
            _, status = H.hisq_solve_device(ctx, st["eta"], st["psi"], case["nrhs"], st["params"])
            psi = st["psi"]
        if status != H.HISQ_OK:
            raise RuntimeError("the solve did not converge")
        return psi
    if kind == "deflate":
        H.hisq_deflate_noalloc(ctx, st["b"], st["x"])
        return st["x"]
    if kind == "layer":
        out = learned.PTLayer.apply(st["x"], st["w"], ctx, case["bf16"])
        gx, gw = torch.autograd.grad(out, (st["x"], st["w"]), st["gout"])
        return {"out": out.detach(), "gx": gx, "gw": gw}
    if kind == "guess":
        with torch.no_grad():
            return st["net"](st["x"])
    eps, _ = H.hisq_eigensolve(ctx, st["params"])
    return eps


# ------------------------------------------------------------------ what a pass cannot do without
def _iterations(case):
    """CG iterations of the synthetic configurations: about 8 sqrt(condition number); deflation halves them."""
    lam = 4 * case["mass"] ** 2 + 2.4 * (math.pi / case["T"]) ** 2
    return (8 * math.sqrt(22 / lam) + 40) * (0.5 if case["n_ev"] else 1)


def work(case):
    X, Y, Z, T = _shape(case)
    V = X * Y * Z * T
    Vh, kind = V // 2, case["kind"]
    if kind == "solve":
        it, k = _iterations(case), case["nrhs"]
        sv = {64: 48, 32: 24, 16: 16}[case["sloppy"]]
        rb = 8 if case["sloppy"] == 64 else 4
        links = (8 * 18 + 8 * (18 if rb == 8 else case["recon"])) * rb  # all hops of one half-apply, per output site
        # an iteration: the links twice; p, tmp, r, x read and p, tmp, r, x written
        b = it * Vh * (2 * links + k * (6 * sv + 2 * max(sv, 24)))
        f = it * Vh * k * (2 * 1146 + 72)
        hi = 0 if case["sloppy"] == 64 else 12  # FP64 residuals: ten decades in steps of delta_rd, source, odd sites
        b += Vh * (hi + 2) * (2 * 2304 + k * 5 * 48)
        f += Vh * k * (hi + 2) * 2 * 1146
        b += 2 * k * V * 48
        if case["n_ev"]:
            per = 24 if case["storage"] == 32 else 12
            b += 2 * 4 * Vh * case["n_ev"] * per
            f += 4 * 2 * 24 * Vh * case["n_ev"] * k
        return {"bytes": b, "flops": f}
    if kind == "deflate":
        per = {32: 24, 16: 16, 15: 12, 14: 12}[case["storage"]]
        return {"bytes": Vh * (2 * case["n"] * per + 96), "flops": 2 * 24 * Vh * case["n"]}
    fat = V * 4 * 18 * 4
    if kind == "layer":
        ci, co = case["cin"], case["cout"]
        # forward: links, x -> out; adjoint: links, gout -> gx; gradient: links, x, gout -> gw
        return {"bytes": 3 * fat + V * 24 * 3 * (ci + co),
                "flops": V * (8 * 66 * (2 * ci + co) + 3 * 9 * ci * co * 24)}
    if kind == "guess":
        pairs = list(zip(learned.CHANNELS[:-1], learned.CHANNELS[1:]))
        return {"bytes": sum(fat + V * 24 * (a + b) for a, b in pairs),
                "flops": sum(V * (8 * 66 * a + 9 * a * b * 24) for a, b in pairs)}
    applies = 3 * case["n_kr"] * 20  # filtered Krylov vectors over the restarts
    return {"bytes": applies / case["block"] * Vh * 2 * (960 + case["block"] * 72), "flops": applies * Vh * 2 * 1146}


# ------------------------------------------------------------------ the same in 64 bits
class _Dirac:
    """D of the synthetic configuration in complex128, plain torch."""

    def __init__(self, dims, fat, lng):
        X, Y, Z, T = dims
        self.shape = (T, Z, Y, X)
        x = torch.arange(X, device="cuda").view(1, 1, 1, X)
        y = torch.arange(Y, device="cuda").view(1, 1, Y, 1)
        z = torch.arange(Z, device="cuda").view(1, Z, 1, 1)
        t = torch.arange(T, device="cuda").view(T, 1, 1, 1)
        self.even = ((x + y + z + t) % 2 == 0).to(torch.float64)[..., None]
        zero = 0 * (x + y + z + t)
        self.hops = []
        for mu, e in enumerate((zero, x + zero, x + y + zero, x + y + z + zero)):
            eta = 1.0 - 2.0 * (e % 2)
            for n, links in ((1, fat), (3, lng)):
                bc = torch.where(t + n >= T, -1.0, 1.0) if mu == 3 else 1.0
                w = (eta * bc)[..., None, None] * links[:, mu].reshape(self.shape + (3, 3))
                self.hops.append((n, 3 - mu, w, w.mH.contiguous()))

    def __call__(self, f):  # f (k, T, Z, Y, X, 3)
        out = torch.zeros_like(f)
        for n, ax, w, wd in self.hops:
            out += (w * torch.roll(f, -n, ax + 1).unsqueeze(-2)).sum(-1)
            # eta_mu(x) = eta_mu(x - n mu): the phase does not depend on the hop's own coordinate
            out -= torch.roll((wd * f.unsqueeze(-2)).sum(-1), n, ax + 1)
        return out

    def one_hop(self, f):
        """the eight one-hop transports of D, forward and backward of each direction"""
        for n, ax, w, wd in self.hops:
            if n == 1:
                yield (w * torch.roll(f, -1, ax + 1).unsqueeze(-2)).sum(-1)
                yield -torch.roll((wd * f.unsqueeze(-2)).sum(-1), 1, ax + 1)


def _dot(a, b):
    return (a.conj() * b).flatten(1).sum(1).real


def _exact_solve(D, m, eta):
    """M psi = eta by CG on the even sites to the limit of 64 bits."""
    e, o = D.even, 1 - D.even
    wide = (-1,) + (1,) * (eta.ndim - 1)
    x = torch.zeros_like(eta)
    y = e * (2 * m * eta - D(o * eta))
    r, best = y.clone(), None
    for _ in range(2):  # restarted once from the true residual
        p, rr = r.clone(), _dot(r, r)
        start = rr.clone()
        for it in range(4000):
            ap = 4 * m * m * p - e * D(o * D(p))
            alpha = torch.where(rr > 0, rr / _dot(p, ap).clamp_min(1e-300), torch.zeros_like(rr))
            x += alpha.view(wide) * p
            r -= alpha.view(wide) * ap
            new = _dot(r, r)
            p = r + torch.where(rr > 0, new / rr.clamp_min(1e-300), torch.zeros_like(rr)).view(wide) * p
            rr = new
            if it % 10 == 9 and bool((rr <= 1e-30 * start).all()):
                break
        r = y - (4 * m * m * x - e * D(o * D(x)))
    return x + o * (eta - D(x)) / (2 * m)


def _exact_eigenvalues(D, n, seed):
    """lowest n eigenvalues of -D_eo D_oe by filtered subspace iteration"""
    e, k = D.even, 3 * n
    shape = (k,) + D.shape + (3,)
    v = e * _complex(seed, 9, *shape)
    flat = v.numel() // k

    def apply(f):
        return -(e * D(D(f)))

    top, cut = 25.0, 1.5
    last = None
    for _ in range(12):
        q = torch.linalg.qr(v.reshape(k, flat).T)[0].T.contiguous()
        h = q.conj() @ apply(q.reshape(shape)).reshape(k, flat).T
        w, z = torch.linalg.eigh(0.5 * (h + h.mH))
        v = (z.T @ q).reshape(shape)
        if last is not None and float((w[:n] - last).abs().max()) < 1e-13 * float(w[n - 1]):
            return w[:n]
        last, cut = w[:n].clone(), min(cut, float(w[-1]))
        c, d = 0.5 * (top + cut), 0.5 * (top - cut)
        a, b = v, (apply(v) - c * v) / d
        for _ in range(79):
            a, b = b, 2 * (apply(b) - c * b) / d - a
        v = b
    return last


def exact(case, seed):
    dims, kind = _shape(case), case["kind"]
    V = dims[0] * dims[1] * dims[2] * dims[3]
    if kind == "solve":
        if V * case["nrhs"] > 700_000:
            return None
        D = _Dirac(dims, *_links(dims, seed, case["eps"]))
        eta = _sources(case, seed)
        psi = _exact_solve(D, case["mass"], eta.reshape((case["nrhs"],) + D.shape + (3,)))
        psi = psi.reshape(case["nrhs"], V, 3)
        return psi.cpu().numpy() if case["host"] else psi
    if kind == "deflate":
        v, eps, b = _vectors(case, seed)
        ev = _even(dims)
        u = v[:, ev].transpose(1, 2).reshape(case["n"], -1)  # [n][colour][Vh]
        del v
        c = (u.conj() @ b.reshape(-1)) / (eps.cuda() + 4 * 0.003 ** 2)
        return (u.T @ c).reshape(b.shape)
    fat, lng = _links(dims, seed, 0.3)
    D = _Dirac(dims, fat, lng)
    if kind == "eig":
        return _exact_eigenvalues(D, case["n_ev"], seed).cpu().numpy()

    def rounded(w):
        w = torch.view_as_real(w.detach())
        return torch.view_as_complex((w.bfloat16().float() if case["bf16"] else w).double().contiguous())

    def transports(f):  # (C, V, 3) -> 9 x (C, V, 3)
        g = f.to(torch.complex128).reshape((-1,) + D.shape + (3,))
        yield f.to(torch.complex128)
        for t in D.one_hop(g):
            yield t.reshape(f.shape)

    def forward(f, w):
        return sum(torch.einsum("ba,avc->bvc", w[:, :, h], t) for h, t in enumerate(transports(f)))

    if kind == "guess":
        f = _channels(case, seed, 2, 3)
        for w in learned.GuessNet(None, seed=int(seed) % (1 << 31), bf16=case["bf16"]).weights:
            f = forward(f, rounded(w))
        return f
    x, g, w = _channels(case, seed, 2, case["cin"]), _channels(case, seed, 3, case["cout"]), rounded(_weights(case, seed))
    g64 = g.to(torch.complex128)
    gw = torch.stack([torch.einsum("bvc,avc->ba", g64, t.conj()) for t in transports(x)], dim=-1)
    # the adjoint of a forward hop is minus the backward one
    wt = w.conj().transpose(0, 1)
    wa = torch.stack([wt[:, :, 0]] + [-wt[:, :, 1 + 2 * mu + 1 - d] for mu in range(4) for d in range(2)], dim=-1)
    return {"out": forward(x, w), "gx": forward(g, wa), "gw": gw}
