// dslash.cu -- the HISQ Dirac operator on one parity (Section 2 of the paper:
// M = D + 2m, D with one-hop fat links and three-hop Naik long links) and the
// fused kernels of one CG iteration on (M^dag M)_ee = 4m^2 - D_eo D_oe (Eq. 1).
//
// One thread computes one output site: 16 link matrices are streamed from the
// gathered per-parity link arrays (read once per half-apply, evict-first), the
// 16 neighbour colour vectors are gathered from the opposite parity (they stay
// in L2: a parity field is at most a few hundred MB and the sweep order keeps
// the +-3 time-slice window resident).
#include "fx64.cuh"

namespace hisq {

// ------------------------------------------------------------- epilogues
// out = a*x + b*y + c*acc; optional |out|^2
template <class S>
struct EpiXpay {
    S out, x, y;
    typename S::real a, b, c;
    int has_x, has_y, want_norm;
    template <typename R>
    __device__ __forceinline__ void operator()(int cb, const CVec<R> &acc, double &red) const
    {
        CVec<R> o;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            o.re[i] = c * acc.re[i];
            o.im[i] = c * acc.im[i];
        }
        if (has_x) {
            CVec<R> v = x.load(cb);
#pragma unroll
            for (int i = 0; i < 3; i++) {
                o.re[i] = fma(a, v.re[i], o.re[i]);
                o.im[i] = fma(a, v.im[i], o.im[i]);
            }
        }
        if (has_y) {
            CVec<R> v = y.load(cb);
#pragma unroll
            for (int i = 0; i < 3; i++) {
                o.re[i] = fma(b, v.re[i], o.re[i]);
                o.im[i] = fma(b, v.im[i], o.im[i]);
            }
        }
        out.store(cb, o);
        if (want_norm) red += double(o.norm2());
    }
};

// second half of a CG iteration: Ap = 4m^2 p - D_eo tmp; x += alpha p;
// r -= alpha Ap; |r|^2.  Ap is never stored.
template <class S, class SX>
struct EpiCG {
    S p, r;
    SX x;
    const DevScalars *scal;
    template <typename R>
    __device__ __forceinline__ void operator()(int cb, const CVec<R> &acc, double &red) const
    {
        const R alpha = R(scal->alpha);
        const R m4 = R(scal->m4);
        CVec<R> pv = p.load(cb);
        CVec<R> rv = r.load(cb);
        auto xv = x.load(cb);
        typedef typename SX::real XR;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            R apr = fma(m4, pv.re[i], -acc.re[i]);
            R api = fma(m4, pv.im[i], -acc.im[i]);
            rv.re[i] = fma(-alpha, apr, rv.re[i]);
            rv.im[i] = fma(-alpha, api, rv.im[i]);
            xv.re[i] = fma(XR(alpha), XR(pv.re[i]), xv.re[i]);
            xv.im[i] = fma(XR(alpha), XR(pv.im[i]), xv.im[i]);
        }
        x.store(cb, xv);
        r.store(cb, rv);
        red += double(rv.norm2());
    }
};

// ------------------------------------------------------------- link formats
// FP32, kinds per mu = 2 (fat + long, 18 reals) or 1 (fat only; long in recon 12)
struct LinksFv {
    const float4 *base;
    int Vh;
    int nk;
    typedef float real;
    __device__ __forceinline__ void load(int mu, int kind, int i, CMat<float> &f, CMat<float> &b) const
    {
        const float4 *q = base + link_index(i, (mu * nk + kind) * 9, nk * 36);
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const float4 a = __ldcs(q + 32 * k);
            f.re[k] = a.x;
            b.re[k] = a.y;
            f.im[k] = a.z;
            b.im[k] = a.w;
        }
    }
};

__device__ __forceinline__ float2 h2f(unsigned u)
{
    __half2 h = *reinterpret_cast<__half2 *>(&u);
    return __half22float2(h);
}

// FP16: uint2 = (fwd_k, bwd_k) as two half2
struct LinksHv {
    const uint2 *base;
    int Vh;
    int nk;
    typedef float real;
    __device__ __forceinline__ void load(int mu, int kind, int i, CMat<float> &f, CMat<float> &b) const
    {
        const uint2 *q = base + link_index(i, (mu * nk + kind) * 9, nk * 36);
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const uint2 a = __ldcs(q + 32 * k);
            float2 x = h2f(a.x), y = h2f(a.y);
            f.re[k] = x.x;
            f.im[k] = x.y;
            b.re[k] = y.x;
            b.im[k] = y.y;
        }
    }
};

// FP16 12-real long links: uint2 (fwd_k, bwd_k), rows 0,1 of the SU(3) factor
struct LinksH12 {
    const uint2 *base;
    int Vh;
    __device__ __forceinline__ void load(int mu, int i, CMat<float> &f, CMat<float> &b) const
    {
        const uint2 *q = base + link_index(i, mu * 6, 24);
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const uint2 a = __ldcs(q + 32 * k);
            float2 x = h2f(a.x), y = h2f(a.y);
            f.re[k] = x.x;
            f.im[k] = x.y;
            b.re[k] = y.x;
            b.im[k] = y.y;
        }
        su3_third_row(f);
        su3_third_row(b);
    }
};

// FP64 for the FP64-FMA form of the operator
struct LinksXv {
    LinksX L;
    typedef double real;
    __device__ __forceinline__ void load(int mu, int kind, int i, CMat<double> &f, CMat<double> &b) const
    {
        const int4 *q = L.w + fx_link_index(i, (mu * 2 + kind) * 18);
        const unsigned dl = __ldg(L.dl + size_t(4) * i + mu);
        const int ef = fx_hop_exponent(L.e[i], dl, 2 * kind), eb = fx_hop_exponent(L.e[i], dl, 2 * kind + 1);
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const double2 x = fx_link(__ldcs(q + 32 * k), ef), y = fx_link(__ldcs(q + 32 * (9 + k)), eb);
            f.re[k] = x.x;
            f.im[k] = x.y;
            b.re[k] = y.x;
            b.im[k] = y.y;
        }
    }
};

// ------------------------------------------------------------- the kernel
// At most 128 registers, two blocks per SM: the compiler then keeps enough link loads in
// flight (left to itself it chose 80 to 92 registers and three blocks).  32^3x64, D_oe and
// fused update, FP16 vectors and 12-real long links: 161 / 170 us, 171 / 172 without the
// bound; FP32 vectors, 18-real: 192 / 206 us, 202 / 222 without; three blocks 164 / 173
// and 194 / 208.  FP64 sums (bound by the FP64 pipe) take what registers they need.
template <class SIn, class Lk, class L12T, bool R12, class Epi>
__global__ void __launch_bounds__(256, sizeof(typename Lk::real) == 8 ? 1 : 2)
    k_dslash(Geom g, int par, Lk L, L12T L12, float c3, SIn in, Epi epi, RedArgs ra, int do_red)
{
    typedef typename Lk::real R;
    double red = 0;
    for (int cb = blockIdx.x * blockDim.x + threadIdx.x; cb < g.Vh; cb += gridDim.x * blockDim.x) {
        int c[4];
        cb_coords(g, par, cb, c);
        const int s = full_site(g, c);
        CVec<R> acc;
        acc.zero();
#pragma unroll
        for (int mu = 0; mu < 4; mu++) {
            CMat<R> f, b;
            L.load(mu, 0, cb, f, b);
            {
                CVec<R> vf = cvt<R>(in.load(nb_cb(g, c, s, mu, +1)));
                CVec<R> vb = cvt<R>(in.load(nb_cb(g, c, s, mu, -1)));
                mv_acc(acc, f, vf);
                mv_acc(acc, b, vb);
            }
            if constexpr (R12) {
                CMat<float> f3, b3;
                L12.load(mu, cb, f3, b3);
                const float eta = stag_phase(mu, c);
                float sf = eta * c3, sb = -eta * c3;
                if (mu == 3 && g.t_antiperiodic) {
                    if (c[3] + 3 >= g.T) sf = -sf;
                    if (c[3] < 3) sb = -sb;
                }
                CVec<float> vf = cvt<float>(in.load(nb_cb(g, c, s, mu, +3)));
                CVec<float> vb = cvt<float>(in.load(nb_cb(g, c, s, mu, -3)));
                mv_acc_scaled(acc, sf, f3, vf);
                mv_acc_scaled(acc, sb, b3, vb);
            } else {
                L.load(mu, 1, cb, f, b);
                CVec<R> vf = cvt<R>(in.load(nb_cb(g, c, s, mu, +3)));
                CVec<R> vb = cvt<R>(in.load(nb_cb(g, c, s, mu, -3)));
                mv_acc(acc, f, vf);
                mv_acc(acc, b, vb);
            }
        }
        epi(cb, acc, red);
    }
    if (do_red) {
        double v[1] = {red};
        grid_reduce<1>(v, ra);
    }
}

// ------------------------------------------------------------- launch glue
// ------------------------------------------------- the FP64 kernel
// Fixed-point sums (fx64.cuh) of FP64 links and one FP64 field, one thread per site, or
// SPLIT = 4 warps per group of 32 sites, one per direction, whose integer sums are added
// in shared memory (exact, so the result is the same bit for bit).
//
// Bound by the 2304 B of links per site.  Each thread holds the links and the neighbour
// of two hops (100 registers), so that a warp has 6.5 KB of loads in flight while it
// multiplies.  32^3x64, split of the input included: 439 us per application at 168
// registers (12 warps per SM); FP64 FMAs take 1058.  With links cut to 56-bit limbs
// beforehand, which saves the shift of each real but loses bits of the small ones: 417, at
// 128 registers (432 B spilled) 500, with the links in shared memory as the batch has them 513.
//
// Split where one thread per site leaves fewer than 16 warps per SM: 8^4 16 us per
// application instead of 23, 14x10x12x22 24 instead of 27, 16^3x32 even; on 24^3x48 (68
// warps per SM) the split costs 181 instead of 146.
constexpr int kFxSplitWarps = 16;

template <class Epi, int SPLIT>
__global__ void __launch_bounds__(128, 3)
    k_dslash_fx(Geom g, int par, LinksX L, FxField in, Epi epi, RedArgs ra, int do_red, int fp64)
{
    constexpr int kGroups = SPLIT == 1 ? 4 : 1; // site groups of a block
    __shared__ long long sh[SPLIT == 1 ? 1 : 3][18][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = SPLIT == 1 ? 0 : warp;
    double red = 0;
    for (int b0 = blockIdx.x * kGroups * 32; b0 < g.Vh; b0 += gridDim.x * kGroups * 32) {
        const int at = b0 + (SPLIT == 1 ? warp * 32 : 0) + lane;
        const int cb = min(at, g.Vh - 1);
        int c[4];
        cb_coords(g, par, cb, c);
        const int s = full_site(g, c);
        const int4 *w = L.w + fx_link_index(cb, 0);
        const unsigned *dl = L.dl + size_t(4) * cb;
        const int le = L.e[cb], E = fp64 ? kFxMark : fx_site_exponent(g, c, s, in.e, dl);
        const bool mark = E == kFxMark || le == kFxMark;
        FxAcc acc;
        acc.zero();
        if (!mark) fx_directions(g, c, s, SPLIT == 1 ? 0 : part, SPLIT == 1 ? 4 : part + 1, w, dl, in, E, acc);
        if (SPLIT > 1) {
            if (part > 0) {
#pragma unroll
                for (int k = 0; k < 9; k++) {
                    sh[part - 1][k][lane] = acc.h[k / 3][k % 3];
                    sh[part - 1][9 + k][lane] = acc.m[k / 3][k % 3];
                }
            }
            __syncthreads();
            if (part == 0) {
#pragma unroll
                for (int k = 0; k < 9; k++)
#pragma unroll
                    for (int u = 0; u < 3; u++) {
                        acc.h[k / 3][k % 3] += sh[u][k][lane];
                        acc.m[k / 3][k % 3] += sh[u][9 + k][lane];
                    }
            }
            __syncthreads();
        }
        if (at < g.Vh && part == 0) {
            CVec<double> o;
            if (!mark) {
                const double u = fx_unit(E, le);
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    o.re[i] = double(fx_sum(acc, 2 * i)) * u;
                    o.im[i] = double(fx_sum(acc, 2 * i + 1)) * u;
                }
            } else {
                o = fx_site_fp64(g, c, s, w, dl, le, in.src);
            }
            epi(cb, o, red);
        }
    }
    if (do_red) {
        double v[1] = {red};
        grid_reduce<1>(v, ra);
    }
}

template <class SIn, class Lk, class L12T, bool R12, class Epi>
static hisq_status run_dslash(hisq_ctx *ctx, int par, const Lk &L, const L12T &L12, const SIn &in, const Epi &epi,
                              RedArgs ra, int do_red)
{
    auto kern = k_dslash<SIn, Lk, L12T, R12, Epi>;
    static const int bps = blocks_per_sm(kern, 256);
    const int grid = grid_for(ctx, ctx->g.Vh, 256, bps);
    kern<<<grid, 256, 0, ctx->stream>>>(ctx->g, par, L, L12, float(ctx->long_scale), in, epi, ra, do_red);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_err(ctx, e, "dslash launch");
    return HISQ_OK;
}

void fx_reserve(hisq_ctx *ctx) { get_optional_buf(ctx, BUF_FX, fx_field_bytes(ctx->g.Vh)); }

// FP64: the input field to mantissas, then the fixed-point kernel.  Without room for
// the mantissas (50 B per site, fx_reserve) every site takes the FP64 path; the buffer is
// never asked for here, since the launches of an iteration are captured.
template <class Epi>
static hisq_status run_fx(hisq_ctx *ctx, int par, const SpinorD &in, const Epi &epi, RedArgs ra, int do_red)
{
    const int Vh = ctx->g.Vh;
    void *buf = ctx->buf_cap[BUF_FX] >= fx_field_bytes(Vh) ? ctx->bufs[BUF_FX] : nullptr;
    if (buf) {
        const hisq_status st = launch_fx_split(ctx, in.p, buf);
        if (st != HISQ_OK) return st;
    }
    const LinksX L = links_fx(ctx, par);
    const FxField f = fx_field(buf, in.p, Vh);
    auto launch = [&](auto kern, int sites, int bps) -> hisq_status {
        const int grid = grid_for(ctx, Vh, sites, bps);
        kern<<<grid, 128, 0, ctx->stream>>>(ctx->g, par, L, f, epi, ra, do_red, buf ? 0 : 1);
        const cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? HISQ_OK : cuda_err(ctx, e, "FP64 dslash launch");
    };
    if (Vh < ctx->num_sms * 32 * kFxSplitWarps) {
        static const int bps4 = blocks_per_sm(k_dslash_fx<Epi, 4>, 128);
        return launch(k_dslash_fx<Epi, 4>, 32, bps4);
    }
    static const int bps1 = blocks_per_sm(k_dslash_fx<Epi, 1>, 128);
    return launch(k_dslash_fx<Epi, 1>, 128, bps1);
}

// Run the Dslash with output parity `par` on links of precision link_prec
// (64, 32 or 16) in the context's long-link format; FMA64: FP64 on FP64 FMAs.
template <bool FMA64 = false, class S, class Epi>
static hisq_status run_any(hisq_ctx *ctx, int par, int link_prec, const S &in, const Epi &epi, RedArgs ra, int dored)
{
    typedef typename S::real R;
    const int Vh = ctx->g.Vh;
    const bool r12 = ctx->long_recon == 12, r8 = ctx->long_recon == 8;
    const int nk = (r12 || r8) ? 1 : 2;
    if (link_prec == 64) {
        if constexpr (sizeof(R) == 8 && !FMA64) return run_fx(ctx, par, in, epi, ra, dored);
        if constexpr (sizeof(R) == 8 && FMA64)
            return run_dslash<S, LinksXv, LinksF12, false>(ctx, par, LinksXv{links_fx(ctx, par)},
                                                           LinksF12{nullptr, Vh}, in, epi, ra, dored);
        return set_err(ctx, HISQ_ERR_INVALID_ARG, "FP64 links need FP64 vectors");
    }
    if constexpr (sizeof(R) == 4) {
        if (link_prec == 32) {
            LinksFv L{ctx->links_f[par], Vh, nk};
            if (r12) return run_dslash<S, LinksFv, LinksF12, true>(ctx, par, L, LinksF12{ctx->links_f12[par], Vh}, in, epi, ra, dored);
            if (r8) return run_dslash<S, LinksFv, LinksF8, true>(ctx, par, L, LinksF8{ctx->links_f12[par], Vh}, in, epi, ra, dored);
            return run_dslash<S, LinksFv, LinksF12, false>(ctx, par, L, LinksF12{nullptr, Vh}, in, epi, ra, dored);
        }
        if (link_prec == 16) {
            if (!ctx->links_h[par]) {
                const hisq_status hs = ensure_half_links(ctx);
                if (hs != HISQ_OK) return hs;
            }
            LinksHv L{ctx->links_h[par], Vh, nk};
            if (r12) return run_dslash<S, LinksHv, LinksH12, true>(ctx, par, L, LinksH12{ctx->links_h12[par], Vh}, in, epi, ra, dored);
            return run_dslash<S, LinksHv, LinksH12, false>(ctx, par, L, LinksH12{nullptr, Vh}, in, epi, ra, dored);
        }
        return set_err(ctx, HISQ_ERR_INVALID_ARG, "link precision must be 64, 32 or 16");
    }
    return set_err(ctx, HISQ_ERR_INVALID_ARG, "FP32/FP16 links need FP32 or FP16 vectors");
}

void fp64_prof_drain(hisq_ctx *ctx, bool all, bool discard)
{
    size_t n = 0;
    for (; n < ctx->fp64_pending.size(); n++) {
        const auto &e = ctx->fp64_pending[n];
        if (all || discard) {
            cudaEventSynchronize(e.second);
        } else if (cudaEventQuery(e.second) != cudaSuccess) {
            cudaGetLastError(); // not ready yet: later pairs are not either
            break;
        }
        float ms = 0;
        if (!discard && cudaEventElapsedTime(&ms, e.first, e.second) == cudaSuccess) {
            ctx->fp64_seconds += 1e-3 * ms;
            ctx->fp64_launches += e.fields;
        }
        cudaGetLastError();
        ctx->fp64_pool.push_back(e.first);
        ctx->fp64_pool.push_back(e.second);
    }
    ctx->fp64_pending.erase(ctx->fp64_pending.begin(), ctx->fp64_pending.begin() + n);
}

static hisq_status dslash_xpay(hisq_ctx *ctx, int out_parity, int prec, int link_prec, const void *in, void *out,
                               double a, const void *x, double b, const void *y, double c, int norm_slot, bool fma64);

// With profiling on, an FP64 launch outside stream capture is bracketed by a
// pair of events (from a pool); the pairs are summed once they have completed,
// so the host never waits for a launch it has just issued.
hisq_status launch_dslash(hisq_ctx *ctx, int out_parity, int prec, int link_prec, const void *in, void *out, double a,
                          const void *x, double b, const void *y, double c, int norm_slot, bool fma64)
{
    bool timed = false;
    if (prec == 64) {
        const hisq_status b0 = fp64_prof_begin(ctx, 1, &timed);
        if (b0 != HISQ_OK) return b0;
    }
    const hisq_status st = dslash_xpay(ctx, out_parity, prec, link_prec, in, out, a, x, b, y, c, norm_slot, fma64);
    const hisq_status e0 = fp64_prof_end(ctx, timed);
    return st != HISQ_OK ? st : e0;
}

hisq_status fp64_prof_begin(hisq_ctx *ctx, int fields, bool *on)
{
    *on = false;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (!ctx->profile || cudaStreamIsCapturing(ctx->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)
        return HISQ_OK;
    cudaEvent_t e[2];
    for (int i = 0; i < 2; i++) {
        if (!ctx->fp64_pool.empty()) {
            e[i] = ctx->fp64_pool.back();
            ctx->fp64_pool.pop_back();
        } else {
            HISQ_CUDA(cudaEventCreate(&e[i]));
        }
    }
    HISQ_CUDA(cudaEventRecord(e[0], ctx->stream));
    ctx->fp64_pending.push_back({e[0], e[1], fields});
    *on = true;
    return HISQ_OK;
}

hisq_status fp64_prof_end(hisq_ctx *ctx, bool on)
{
    if (!on) return HISQ_OK;
    HISQ_CUDA(cudaEventRecord(ctx->fp64_pending.back().second, ctx->stream));
    fp64_prof_drain(ctx, ctx->fp64_pending.size() > 4096);
    return HISQ_OK;
}

static hisq_status dslash_xpay(hisq_ctx *ctx, int out_parity, int prec, int link_prec, const void *in, void *out,
                               double a, const void *x, double b, const void *y, double c, int norm_slot, bool fma64)
{
    const int Vh = ctx->g.Vh;
    if (!ctx->links_loaded) return set_err(ctx, HISQ_ERR_STATE, "links not loaded");
    if ((prec == 64) != (link_prec == 64)) return set_err(ctx, HISQ_ERR_INVALID_ARG, "FP64 vectors go with FP64 links");
    void *xx = const_cast<void *>(x ? x : out), *yy = const_cast<void *>(y ? y : out);
    RedArgs ra = red_args(ctx, FIN_STORE, norm_slot < 0 ? 0 : norm_slot);
    const int dored = norm_slot >= 0;
    auto go = [&](auto in_, auto out_, auto x_, auto y_) -> hisq_status {
        typedef decltype(in_) S;
        typedef typename S::real R;
        EpiXpay<S> epi{out_, x_, y_, R(a), R(b), R(c), x != nullptr, y != nullptr, dored};
        if (fma64) return run_any<true>(ctx, out_parity, link_prec, in_, epi, ra, dored);
        return run_any(ctx, out_parity, link_prec, in_, epi, ra, dored);
    };
    void *ii = const_cast<void *>(in);
    switch (prec) {
    case 64: return go(make_spinorD(ii, Vh), make_spinorD(out, Vh), make_spinorD(xx, Vh), make_spinorD(yy, Vh));
    case 32: return go(make_spinorF(ii, Vh), make_spinorF(out, Vh), make_spinorF(xx, Vh), make_spinorF(yy, Vh));
    case 16: return go(make_spinorH(ii, Vh), make_spinorH(out, Vh), make_spinorH(xx, Vh), make_spinorH(yy, Vh));
    }
    return set_err(ctx, HISQ_ERR_INVALID_ARG, "precision must be 64, 32 or 16");
}

// ---------------------------------------------------------- CG iteration
// (1) tmp = D_oe p (odd output) with tt = |tmp|^2 -> alpha = rr / (4m^2 pp + tt)
//     using <p, A p> = 4m^2 |p|^2 + |D_oe p|^2 (D_eo = -D_oe^dag).
hisq_status launch_cg_dslash_tt(hisq_ctx *ctx, int prec, int link_prec, const void *p, void *tmp)
{
    const int Vh = ctx->g.Vh;
    RedArgs ra = red_args(ctx, FIN_CG_ALPHA);
    void *pp = const_cast<void *>(p);
    auto go = [&](auto in_, auto out_) -> hisq_status {
        typedef decltype(in_) S;
        typedef typename S::real R;
        EpiXpay<S> epi{out_, out_, out_, R(0), R(0), R(1), 0, 0, 1};
        return run_any(ctx, 1, link_prec, in_, epi, ra, 1);
    };
    switch (prec) {
    case 64: return go(make_spinorD(pp, Vh), make_spinorD(tmp, Vh));
    case 32: return go(make_spinorF(pp, Vh), make_spinorF(tmp, Vh));
    case 16: return go(make_spinorH(pp, Vh), make_spinorH(tmp, Vh));
    }
    return set_err(ctx, HISQ_ERR_INVALID_ARG, "bad sloppy precision");
}

// (2) even output: Ap = 4m^2 p - D_eo tmp; x += alpha p; r -= alpha Ap; rr_new = |r|^2,
//     beta = rr_new / rr.
hisq_status launch_cg_dslash_update(hisq_ctx *ctx, int prec, int link_prec, int xprec, const void *tmp,
                                    const void *p, void *x, void *r)
{
    const int Vh = ctx->g.Vh;
    RedArgs ra = red_args(ctx, FIN_CG_BETA);
    void *tt = const_cast<void *>(tmp), *pp = const_cast<void *>(p);
    switch (prec) {
    case 64: {
        EpiCG<SpinorD, SpinorD> epi{make_spinorD(pp, Vh), make_spinorD(r, Vh), make_spinorD(x, Vh), ctx->scal};
        return run_any(ctx, 0, link_prec, make_spinorD(tt, Vh), epi, ra, 1);
    }
    case 32: {
        if (xprec != 32) return set_err(ctx, HISQ_ERR_INVALID_ARG, "x precision");
        EpiCG<SpinorF, SpinorF> epi{make_spinorF(pp, Vh), make_spinorF(r, Vh), make_spinorF(x, Vh), ctx->scal};
        return run_any(ctx, 0, link_prec, make_spinorF(tt, Vh), epi, ra, 1);
    }
    case 16: {
        if (xprec != 32) return set_err(ctx, HISQ_ERR_INVALID_ARG, "x precision");
        EpiCG<SpinorH, SpinorF> epi{make_spinorH(pp, Vh), make_spinorH(r, Vh), make_spinorF(x, Vh), ctx->scal};
        return run_any(ctx, 0, link_prec, make_spinorH(tt, Vh), epi, ra, 1);
    }
    }
    return set_err(ctx, HISQ_ERR_INVALID_ARG, "bad sloppy precision");
}

} // namespace hisq
