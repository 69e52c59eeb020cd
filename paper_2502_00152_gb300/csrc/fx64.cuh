// fx64.cuh -- the FP64 Dirac operator in fixed-point arithmetic on the integer
// units.
//
// GB300 retires 1.68 FP64 FMAs per clock and SM (measured), so an FP64 Dslash
// (576 complex-matrix FMAs per site and right-hand side) takes 343 clocks per site
// and SM where its 2.4 KB of links take 111 from HBM.  32 x 32 -> 64 bit integer
// multiply-adds run at 64 per clock and SM (measured), so the same sums are formed
// here from 56-bit mantissas held as two 28-bit limbs, three multiply-adds per real
// product (the product of the two low limbs, below 2^-57 of the largest term, is
// dropped): 27 clocks, and HBM becomes the bound for one right-hand side.
//
// Block floating point: the six reals of a colour vector share the exponent of the
// largest one, the 288 link reals of an output site share theirs, and at an output
// site the 16 neighbour vectors are aligned to the largest of their exponents.  A
// mantissa keeps 56 bits below the shared exponent (FP64 keeps 53 below its own), and
// the integer sums are exact.  Measured against 113-bit sums on 8^4: relative error
// 6.4e-17 for a Gaussian field (FP64 FMAs 3.5e-16), 1.0e-16 where site vectors differ by
// up to e^20 (3.5e-16).  The sums do not depend on the order of the terms, so a site may be
// split over threads without changing a bit of the result.
//
// Limbs: v = hi 2^28 + lo with -2^27 <= lo < 2^27 and |hi| <= 2^28.  A sum has 96
// products hi hi of at most 2^56 (< 2^62.6) and 192 products hi lo of at most 2^55
// (< 2^62.6): both fit a signed 64-bit word.  Vector mantissas are stored with four
// more bits, |v| <= 2^60, so that the limbs of a shifted one are its two 32-bit words:
// hi = the upper word plus the sign bit of the lower, lo = the lower word >> 4.
//
// Links are stored by groups of 32 sites, [group][mu][kind][fwd,bwd][k][32] int4: the
// 144 loads of a thread are at constant offsets from one address.
//
// Values the block format cannot hold -- Inf, NaN, and exponents so far out that a
// product's scale would leave the FP64 range -- are marked, and a site that meets a
// mark is computed with FP64 FMAs from the original numbers, which keeps the former
// behaviour for them (non-finite sources are reported from their norms).
#pragma once

#include "internal.cuh"

namespace hisq {

constexpr int kFxMark = 0x7fff;                // exponent of a vector or link site kept as FP64
constexpr int kFxVecLo = 323, kFxVecHi = 1723; // biased exponents of ordinary colour vectors: 2^-700 .. 2^700
constexpr int kFxLinkLo = 923, kFxLinkHi = 1123; // and of links: 2^-100 .. 2^100

// one parity of a colour field: mantissas [3][Vh] (re, im), biased exponents [Vh],
// and the FP64 field they were made from
struct FxField {
    const longlong2 *v;
    const short *e;
    const double2 *src;
};

// gathered links of one output parity: int4 =
// (re hi, re lo, im hi, im lo) per element, biased exponents [Vh]; where the exponent
// is kFxMark the int4 holds the two FP64 values themselves
struct LinksX {
    const int4 *w; // fx_link_index
    const short *e;
};

__host__ __device__ __forceinline__ size_t fx_link_index(int cb, int k) // element k = 9 hop + 3 row + column
{
    return (size_t(cb >> 5) * 144 + k) * 32 + (cb & 31);
}

inline size_t fx_field_bytes(int Vh) { return size_t(Vh) * 48 + ((size_t(Vh) * 2 + 255) & ~size_t(255)); }
inline FxField fx_field(void *buf, const void *src, int Vh)
{
    return FxField{(const longlong2 *)buf, (const short *)((char *)buf + size_t(Vh) * 48), (const double2 *)src};
}

__device__ __forceinline__ int fx_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// round(x 2^(53 + UP - (eb - 1022))) for |x| < 2^(eb - 1022)
template <int UP>
__device__ __forceinline__ long long fx_mantissa(double x, int eb)
{
    const long long b = __double_as_longlong(x);
    const int e = int(b >> 52) & 0x7ff;
    const int s = eb - (e > 0 ? e : 1);
    unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (e > 0 ? 1ull << 52 : 0ull);
    m <<= UP;
    if (s > 0) m = s < 62 ? (m + (1ull << (s - 1))) >> s : 0ull;
    return b < 0 ? -(long long)m : (long long)m;
}

// limbs of a mantissa, |v| <= 2^56
__device__ __forceinline__ void fx_limbs(long long v, int &hi, int &lo)
{
    hi = int((v + (1ll << 27)) >> 28);
    lo = int(unsigned(v) - (unsigned(hi) << 28));
}

// limbs of a vector mantissa shifted down by d (0..31), |v| <= 2^60: two shifts, one
// add-and-shift, one shift
__device__ __forceinline__ void fx_shifted_limbs(long long v, int d, int &hi, int &lo)
{
    const unsigned l = __funnelshift_r(unsigned(v), unsigned(v >> 32), d);
    hi = (int(v >> 32) >> d) + int(l >> 31);
    lo = int(l) >> 4;
}

// 2^k, -1022 <= k <= 1023
__device__ __forceinline__ double fx_pow2(int k) { return __hiloint2double((k + 1023) << 20, 0); }

// link element (re, im) as FP64
__device__ __forceinline__ double2 fx_link(int4 q, int eb)
{
    if (eb == kFxMark) return make_double2(__hiloint2double(q.y, q.x), __hiloint2double(q.w, q.z));
    const double s1 = fx_pow2(eb - 1022 - 28), s0 = fx_pow2(eb - 1022 - 56);
    return make_double2(fma(double(q.x), s1, double(q.y) * s0), fma(double(q.z), s1, double(q.w) * s0));
}

// sums of the integer products of one right-hand side: value of component c is
// (h[c] 2^56 + m[c] 2^28) times the shared scale; c = 2 * colour + (0: re, 1: im)
struct FxAcc {
    long long h[6], m[6];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int c = 0; c < 6; c++) h[c] = m[c] = 0;
    }
};

// h 2^56 + m 2^28 += (ah 2^28 + al)(bh 2^28 + bl) without al bl: three IMAD.WIDE
__device__ __forceinline__ void fx_mac(long long &h, long long &m, int ah, int al, int bh, int bl)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(h) : "r"(ah), "r"(bh));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(m) : "r"(ah), "r"(bl));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(m) : "r"(al), "r"(bh));
}

// the shared exponent of the 16 neighbours of a site (kFxMark if one is marked)
__device__ __forceinline__ int fx_site_exponent(const Geom &g, const int c[4], int s, const short *e)
{
    int E = 0;
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        E = max(E, max(int(__ldg(e + nb_cb(g, c, s, mu, 1))), int(__ldg(e + nb_cb(g, c, s, mu, -1)))));
        E = max(E, max(int(__ldg(e + nb_cb(g, c, s, mu, 3))), int(__ldg(e + nb_cb(g, c, s, mu, -3)))));
    }
    return E;
}

// One hop of a site in flight: its link matrix and the neighbour's vector of R
// right-hand sides.  hop = 4 mu + (0: fat fwd, 1: fat bwd, 2: long fwd, 3: long bwd).
// KEEP: the links go through L1 (other warps of the block read the same lines), else
// they are streamed.
template <int R, bool KEEP>
struct FxHop {
    int4 w[9];
    longlong2 v[R][3];
    int e[R];
    __device__ __forceinline__ void load(const Geom &g, const int c[4], int s, int mu, int h, const int4 *L,
                                         const FxField (&in)[R])
    {
        const int nb = nb_cb(g, c, s, mu, (h & 2 ? 3 : 1) * (h & 1 ? -1 : 1));
        const int4 *p = L + (mu * 4 + h) * (9 * 32);
#pragma unroll
        for (int k = 0; k < 9; k++) w[k] = KEEP ? __ldg(p + 32 * k) : __ldcs(p + 32 * k);
#pragma unroll
        for (int r = 0; r < R; r++) {
            e[r] = __ldg(in[r].e + nb);
#pragma unroll
            for (int j = 0; j < 3; j++) v[r][j] = __ldg(in[r].v + size_t(j) * g.Vh + nb);
        }
    }
    // acc += W v, the vector shifted down to the site's exponent
    __device__ __forceinline__ void add(const int (&E)[R], FxAcc (&acc)[R]) const
    {
        int vh[R][6], vl[R][6], nh[R][3], nl[R][3]; // limbs, and those of -im
#pragma unroll
        for (int r = 0; r < R; r++) {
            int d = E[r] - e[r];
            longlong2 q[3] = {v[r][0], v[r][1], v[r][2]};
            if (d > 31) { // a neighbour far below the largest one
#pragma unroll
                for (int j = 0; j < 3; j++) q[j] = make_longlong2(q[j].x >> 31, q[j].y >> 31);
                d = min(d - 31, 31);
            }
#pragma unroll
            for (int j = 0; j < 3; j++) {
                fx_shifted_limbs(q[j].x, d, vh[r][2 * j], vl[r][2 * j]);
                fx_shifted_limbs(q[j].y, d, vh[r][2 * j + 1], vl[r][2 * j + 1]);
                nh[r][j] = -vh[r][2 * j + 1];
                nl[r][j] = -vl[r][2 * j + 1];
            }
        }
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const int4 q = w[3 * i + j];
#pragma unroll
                for (int r = 0; r < R; r++) {
                    FxAcc &a = acc[r];
                    fx_mac(a.h[2 * i], a.m[2 * i], q.x, q.y, vh[r][2 * j], vl[r][2 * j]);
                    fx_mac(a.h[2 * i], a.m[2 * i], q.z, q.w, nh[r][j], nl[r][j]);
                    fx_mac(a.h[2 * i + 1], a.m[2 * i + 1], q.x, q.y, vh[r][2 * j + 1], vl[r][2 * j + 1]);
                    fx_mac(a.h[2 * i + 1], a.m[2 * i + 1], q.z, q.w, vh[r][2 * j], vl[r][2 * j]);
                }
            }
    }
};

// directions mu0 .. mu1 - 1 of a site (L: its first link element): the loads of the next hop are issued before
// the sums of the current one
template <int R, bool KEEP>
__device__ __forceinline__ void fx_directions(const Geom &g, const int c[4], int s, int mu0, int mu1, const int4 *L,
                                              const FxField (&in)[R], const int (&E)[R],
                                              FxAcc (&acc)[R])
{
    FxHop<R, KEEP> a, b;
    a.load(g, c, s, mu0, 0, L, in);
#pragma unroll 1
    for (int mu = mu0; mu < mu1; mu++) {
        b.load(g, c, s, mu, 1, L, in);
        a.add(E, acc);
        a.load(g, c, s, mu, 2, L, in);
        b.add(E, acc);
        b.load(g, c, s, mu, 3, L, in);
        a.add(E, acc);
        if (mu + 1 < mu1) a.load(g, c, s, mu + 1, 0, L, in);
        b.add(E, acc);
    }
}

// the sums as FP64: carries of the middle sum into the high one, then one rounding
__device__ __forceinline__ CVec<double> fx_value(const FxAcc &a, int E, int le)
{
    const int k = E + le - 2100; // unit of h: 2^56 2^(E - 1022 - 56) 2^(le - 1022 - 56)
    const double s1 = fx_pow2(k), s0 = fx_pow2(k - 28);
    CVec<double> o;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const long long h0 = a.h[2 * c] + (a.m[2 * c] >> 28), h1 = a.h[2 * c + 1] + (a.m[2 * c + 1] >> 28);
        const int l0 = int(a.m[2 * c] & 0xfffffffll), l1 = int(a.m[2 * c + 1] & 0xfffffffll);
        o.re[c] = fma(double(h0), s1, double(l0) * s0);
        o.im[c] = fma(double(h1), s1, double(l1) * s0);
    }
    return o;
}

// a marked site (L: its first link element): FP64 FMAs on the original field
static __device__ __noinline__ CVec<double> fx_site_fp64(const Geom &g, const int c[4], int s, const int4 *L, int le,
                                                         const double2 *src)
{
    const int Vh = g.Vh;
    CVec<double> acc;
    acc.zero();
#pragma unroll 1
    for (int h = 0; h < 16; h++) {
        const int mu = h >> 2, kind = (h >> 1) & 1, bwd = h & 1;
        const int nb = nb_cb(g, c, s, mu, (kind ? 3 : 1) * (bwd ? -1 : 1));
        const int4 *w = L + h * (9 * 32);
        CVec<double> v;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const double2 q = src[size_t(j) * Vh + nb];
            v.re[j] = q.x;
            v.im[j] = q.y;
        }
        CMat<double> W;
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const double2 q = fx_link(w[32 * k], le);
            W.re[k] = q.x;
            W.im[k] = q.y;
        }
        mv_acc(acc, W, v);
    }
    return acc;
}

// ------------------------------------------------------------- host side
// mantissas and exponents of the FP64 parity field `in` into `out` (fx_field_bytes)
hisq_status launch_fx_split(hisq_ctx *ctx, const void *in, void *out);

} // namespace hisq
