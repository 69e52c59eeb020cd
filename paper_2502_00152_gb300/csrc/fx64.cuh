// fx64.cuh -- the FP64 Dirac operator in fixed-point arithmetic on the integer
// units.
//
// GB300 retires 1.68 FP64 FMAs per clock and SM (measured), so an FP64 Dslash
// (576 FMAs per site and right-hand side) takes 343 clocks per site and SM where its
// 2.4 KB of links take 111 from HBM.  32 x 32 + 64 bit integer multiply-adds run at 30
// per clock and SM (measured; the 64-bit additions of the ALU pipe pass beside them), so
// the same sums are formed here from 56-bit mantissas held as two 28-bit limbs.  A real
// product takes three multiply-adds (the product of the two low limbs, below 2^-57 of
// the largest term, is dropped) and a complex one three real products instead of four
// (Karatsuba's identity, see FxAcc): 1296 multiply-adds, 43 clocks per site.
//
// Block floating point: the six reals of a colour vector share the exponent of the
// largest one, the 18 reals of a hop's matrix theirs, and the 16 products of an output site
// are aligned to the largest sum of the two.  In the sums a matrix entry has 56 bits below
// its hop's exponent, a vector entry the same less what its product is shifted down (FP64
// keeps 53 below its own), and the integer sums are exact.  So an error is at most about
// 2.3 x 96 x 2^-56 of the largest product of a matrix's and a vector's power of two: small
// against the site's result, but not against a component that only small entries couple
// to.  The solves use this operator, whose residuals are norms over the lattice;
// hisq_apply_dslash and hisq_apply_normal_op, whose callers see each component, run on FP64
// FMAs.  Norm of the error against 113-bit sums on 6^3x10, relative to the result's (FP64
// FMAs): Gaussian field 6.9e-17 (3.5e-16), sites scaled by 2^+-40 1.0e-16 (2.9e-16), a wall
// of one colour 5.3e-17 (1.2e-16), unit points 3.3e-17 (1.7e-17: single products by 1 are
// exact there).  The sums do not depend on the order of the terms, so a site may be
// split over threads without changing a bit of the result.
//
// Limbs: v = hi 2^28 + lo with -2^27 <= lo < 2^27 and |hi| <= 2^28.  A sum has 96
// products hi hi of at most 2^56 (< 2^62.6) and 192 products hi lo of at most 2^55
// (< 2^62.6): both fit a signed 64-bit word.  Vector mantissas are stored with four
// more bits, |v| <= 2^60, so that the limbs of a shifted one are its two 32-bit words:
// hi = the upper word plus the sign bit of the lower, lo = the lower word >> 4.
//
// Links are stored by groups of 32 sites, [group][mu][kind][fwd,bwd][k][32] int4: the
// 144 loads of a thread are at constant offsets from one address.  A real keeps its own 53
// bits: its signed mantissa times 2^7 in 64 bits, with the number of places it lies below
// its hop's exponent in the seven low ones, so that one shift aligns it (links of the
// solves, of FP64 FMAs and of the double-float operator are the same values).
//
// Values the block format cannot hold -- Inf, NaN, and exponents so far out that a
// product's scale would leave the FP64 range -- are marked, and a site that meets a
// mark is computed with FP64 FMAs from the original numbers, which keeps the former
// behaviour for them (non-finite sources are reported from their norms).
#pragma once

#include "internal.cuh"
#include "tc.cuh"

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

// gathered links of one output parity: int4 = (re low, re high, im low, im high) words of an
// element (fx_encode); of each site the biased exponent of its largest entry and, one byte
// per hop, how far that of the hop's largest entry lies below it (fx_hop_exponent).  Where
// the site's exponent is kFxMark the int4 hold the two FP64 values themselves.
struct LinksX {
    const int4 *w;      // fx_link_index
    const unsigned *dl; // [Vh][mu], byte h = hop of the direction: fat fwd, fat bwd, long fwd, long bwd
    const short *e;     // [Vh]
};
inline LinksX links_fx(const hisq_ctx *ctx, int par)
{
    return LinksX{ctx->links_x[par], ctx->links_xe[par], (const short *)(ctx->links_xe[par] + size_t(4) * ctx->g.Vh)};
}
__device__ __forceinline__ int fx_depth(unsigned dl, int h) { return int((dl >> (8 * h)) & 255); }
__device__ __forceinline__ int fx_hop_exponent(int le, unsigned dl, int h) { return le == kFxMark ? le : le - fx_depth(dl, h); }

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

// round(x 2^(60 - (eb - 1022))) for |x| < 2^(eb - 1022)
__device__ __forceinline__ long long fx_mantissa(double x, int eb)
{
    const long long b = __double_as_longlong(x);
    const int e = int(b >> 52) & 0x7ff;
    const int s = eb - (e > 0 ? e : 1);
    unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (e > 0 ? 1ull << 52 : 0ull);
    m <<= 7;
    if (s > 0) m = s < 62 ? (m + (1ull << (s - 1))) >> s : 0ull;
    return b < 0 ? -(long long)m : (long long)m;
}

// one site's vector to mantissas and exponent; marked sites keep no mantissas
__device__ __forceinline__ void fx_store_site(longlong2 *v, short *e, int Vh, int i, const CVec<double> &q)
{
    int eb = 0;
    bool zero = true;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        eb = max(eb, max(fx_exponent(q.re[c]), fx_exponent(q.im[c])));
        zero = zero && q.re[c] == 0.0 && q.im[c] == 0.0;
    }
    if (!zero && (eb < kFxVecLo || eb > kFxVecHi)) {
        e[i] = short(kFxMark); // the operator reads the FP64 field at the sites this one touches
        return;
    }
    if (zero) eb = kFxVecLo; // below every other exponent, mantissas 0
    e[i] = short(eb);
#pragma unroll
    for (int c = 0; c < 3; c++)
        v[size_t(c) * Vh + i] = make_longlong2(fx_mantissa(q.re[c], eb), fx_mantissa(q.im[c], eb));
}

// a link real under its hop's exponent eb: signed mantissa (53 bits) 2^7, and in the low seven
// bits how far its own exponent lies below eb (at most kFxDepth); zero: 0
constexpr int kFxDepth = 127;
__device__ __forceinline__ long long fx_encode(double x, int eb)
{
    if (x == 0.0) return 0;
    const long long b = __double_as_longlong(x);
    const long long m = ((b & 0xfffffffffffffll) | (1ll << 52)) << 7;
    return (b < 0 ? -m : m) | (eb - fx_exponent(x));
}
__device__ __forceinline__ double fx_decode(int w0, int w1, int eb)
{
    const unsigned long long v = ((unsigned long long)unsigned(w1) << 32) | unsigned(w0 & ~kFxDepth);
    const unsigned long long m = (w1 < 0 ? 0ull - v : v) >> 7;
    const unsigned top = (unsigned(m >> 32) & 0xfffffu) | (unsigned(w1) & 0x80000000u) |
                         (v ? unsigned(eb - (w0 & kFxDepth)) << 20 : 0u);
    return eb == kFxMark ? __hiloint2double(w1, w0) : __hiloint2double(int(top), int(unsigned(m)));
}

// limbs of an encoded link real shifted down to its hop's exponent, |v| <= 2^60.  Below a
// shift of 16 the count takes bits that the low limb drops, from 16 on it is shifted out.
__device__ __forceinline__ void fx_link_limbs(int w0, int w1, int &hi, int &lo)
{
    long long v;
    asm("{\n\t.reg .s64 t;\n\tmov.b64 t, {%1, %2};\n\tshr.s64 %0, t, %3;\n\t}"
        : "=l"(v)
        : "r"(w0), "r"(w1), "r"(w0 & kFxDepth)); // a shift past 63 places leaves the sign
    const unsigned l = unsigned(v);
    hi = int(v >> 32) + int(l >> 31);
    lo = int(l) >> 4;
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

// link element (re, im) of a hop of exponent eb as FP64
__device__ __forceinline__ double2 fx_link(int4 q, int eb)
{
    return make_double2(fx_decode(q.x, q.y, eb), fx_decode(q.z, q.w, eb));
}

// Sums of the integer products of one right-hand side.  With W = a + ib and v = c + id,
//   k1 = c (a + b),  k2 = a (d - c),  k3 = b (c + d):  Re W v = k1 - k3,  Im W v = k1 + k2,
// and the three are summed separately over the 16 hops and 3 colours of row i, [row][k];
// value: (h 2^56 + m 2^28) times the shared scale.  Single sums may wrap around 2^64, the
// differences that are used at the end fit (above), so they are exact.
struct FxAcc {
    long long h[3][3], m[3][3];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int k = 0; k < 3; k++) h[i][k] = m[i][k] = 0;
    }
};

// the largest exponent of a neighbour's vector less its hop's depth, which the 16 products
// are aligned to (kFxMark if a neighbour is marked)
__device__ __forceinline__ int fx_site_exponent(const Geom &g, const int c[4], int s, const short *e, const unsigned *dl)
{
    const uint4 q = __ldg(reinterpret_cast<const uint4 *>(dl));
    const unsigned d[4] = {q.x, q.y, q.z, q.w};
    int E = 0;
#pragma unroll
    for (int mu = 0; mu < 4; mu++)
#pragma unroll
        for (int h = 0; h < 4; h++)
            E = max(E, int(__ldg(e + nb_cb(g, c, s, mu, (h & 2 ? 3 : 1) * (h & 1 ? -1 : 1)))) - fx_depth(d[mu], h));
    return E > kFxVecHi ? kFxMark : E; // a mark less a depth is still above every exponent
}

// the neighbour's vector of one hop.
// hop = 4 mu + h, h = 0: fat fwd, 1: fat bwd, 2: long fwd, 3: long bwd.
struct FxVec {
    longlong2 v[3];
    int e; // less the hop's depth
    __device__ __forceinline__ void load(const Geom &g, const SiteLine &line, int h, const FxField &in, unsigned dl)
    {
        const unsigned nb = unsigned(line.at(g, (h & 2 ? 3 : 1) * (h & 1 ? -1 : 1)));
        e = int(__ldg(in.e + nb)) - fx_depth(dl, h);
#pragma unroll
        for (int j = 0; j < 3; j++) v[j] = __ldg(in.v + size_t(j) * g.Vh + nb);
    }
};

// acc += W v, the vector shifted down to the site's exponent; link(k): element k of W
template <class F>
__device__ __forceinline__ void fx_add(const FxVec &x, int E, FxAcc &acc, F &&link)
{
    int d = E - x.e;
    longlong2 q[3] = {x.v[0], x.v[1], x.v[2]};
    if (d > 31) { // a neighbour far below the largest one
#pragma unroll
        for (int j = 0; j < 3; j++) q[j] = make_longlong2(q[j].x >> 31, q[j].y >> 31);
        d = min(d - 31, 31);
    }
    int vh[3][3], vl[3][3]; // limbs of c, d - c and c + d
#pragma unroll
    for (int j = 0; j < 3; j++) {
        int dh, dl;
        fx_shifted_limbs(q[j].x, d, vh[j][0], vl[j][0]);
        fx_shifted_limbs(q[j].y, d, dh, dl);
        vh[j][1] = dh - vh[j][0];
        vl[j][1] = dl - vl[j][0];
        vh[j][2] = dh + vh[j][0];
        vl[j][2] = dl + vl[j][0];
    }
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const int4 w = link(3 * i + j);
            int wh[3], wl[3]; // limbs of a + b, a, b
            fx_link_limbs(w.x, w.y, wh[1], wl[1]);
            fx_link_limbs(w.z, w.w, wh[2], wl[2]);
            wh[0] = wh[1] + wh[2];
            wl[0] = wl[1] + wl[2];
            // three independent sums between two additions to the same one
#pragma unroll
            for (int k = 0; k < 3; k++) acc.h[i][k] += (long long)wh[k] * vh[j][k];
#pragma unroll
            for (int k = 0; k < 3; k++) acc.m[i][k] += (long long)wh[k] * vl[j][k];
#pragma unroll
            for (int k = 0; k < 3; k++) acc.m[i][k] += (long long)wl[k] * vh[j][k];
        }
}

// Directions mu0 .. mu1 - 1 of a site (L: its first link element, dl: its depths), links in registers:
// the loads of the next hop are issued before the sums of the current one.
struct FxHop {
    int4 w[9];
    FxVec x;
    __device__ __forceinline__ void load(const Geom &g, const SiteLine &line, int mu, int h, const int4 *L,
                                         const FxField &in, unsigned dl)
    {
        const int4 *p = L + (mu * 4 + h) * (9 * 32);
#pragma unroll
        for (int k = 0; k < 9; k++) w[k] = __ldcs(p + 32 * k); // read once per launch
        x.load(g, line, h, in, dl);
    }
    __device__ __forceinline__ void add(int E, FxAcc &acc) const
    {
        fx_add(x, E, acc, [&](int k) { return w[k]; });
    }
};
__device__ __forceinline__ void fx_directions(const Geom &g, const int c[4], int s, int mu0, int mu1, const int4 *L,
                                              const unsigned *dl, const FxField &in, int E, FxAcc &acc)
{
    FxHop a, b;
    SiteLine line(g, c, s, mu0);
    unsigned d = __ldg(dl + mu0);
    a.load(g, line, mu0, 0, L, in, d);
#pragma unroll 1
    for (int mu = mu0; mu < mu1; mu++) {
        b.load(g, line, mu, 1, L, in, d);
        a.add(E, acc);
        a.load(g, line, mu, 2, L, in, d);
        b.add(E, acc);
        b.load(g, line, mu, 3, L, in, d);
        a.add(E, acc);
        if (mu + 1 < mu1) {
            line = SiteLine(g, c, s, mu + 1);
            d = __ldg(dl + mu + 1);
            a.load(g, line, mu + 1, 0, L, in, d);
        }
        b.add(E, acc);
    }
}

// the high sum with the carry of the middle one, rounded to the unit of h: at most 2^-57
// of the largest product is lost, as in every term.  c = 2 * colour + (0: re, 1: im)
__device__ __forceinline__ long long fx_sum(const FxAcc &a, int c)
{
    const int i = c >> 1;
    const long long h = c & 1 ? a.h[i][0] + a.h[i][1] : a.h[i][0] - a.h[i][2];
    const long long m = c & 1 ? a.m[i][0] + a.m[i][1] : a.m[i][0] - a.m[i][2];
    return h + ((m + (1ll << 27)) >> 28);
}

// unit of h: 2^56 2^(E - 1022 - 56) 2^(le - 1022 - 56)
__device__ __forceinline__ double fx_unit(int E, int le) { return fx_pow2(E + le - 2100); }

// a marked site (L: its first link element): FP64 FMAs on the original field
static __device__ __noinline__ CVec<double> fx_site_fp64(const Geom &g, const int c[4], int s, const int4 *L,
                                                         const unsigned *dl, int le, const double2 *src)
{
    const int Vh = g.Vh;
    CVec<double> acc;
    acc.zero();
#pragma unroll 1
    for (int h = 0; h < 16; h++) {
        const int mu = h >> 2, kind = (h >> 1) & 1, bwd = h & 1;
        const int eh = fx_hop_exponent(le, dl[mu], h & 3);
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
            const double2 q = fx_link(w[32 * k], eh);
            W.re[k] = q.x;
            W.im[k] = q.y;
        }
        mv_acc(acc, W, v);
    }
    return acc;
}

// ------------------------------------------------- links through shared memory
// A warp computes 32 consecutive sites of one field; nch warps (fields) share a site
// group, nsg groups share a block: warp = (group, field).  The links of a hop of a site
// group are one contiguous 4.6 KB piece: one bulk copy into a ring of `stages` slots of
// shared memory that the nch warps read, so that each link leaves HBM once for all of
// them and takes no registers while it travels; the next hop's vector is loaded while the
// current one is multiplied.  Every wait is bounded: one that runs out records its code
// in *status, the warp gives up the rest of its sites, and the launch ends.
constexpr int kFxHopBytes = 9 * 32 * 16;
constexpr int kFxWarps = 8; // warps of a block at most

struct FxTile {
    int nch, nsg, stages;
    __host__ __device__ size_t smem() const { return size_t(nsg) * stages * (kFxHopBytes + 2 * sizeof(uint64_t)); }
};

// site(cb, c, s, E, le, acc) for every site of this warp
template <class F>
__device__ __forceinline__ void fx_ring_sites(const Geom &g, int par, const LinksX &L, const FxField &in,
                                              const FxTile &tl, int bx, int nbx, unsigned char *dsm, int *status,
                                              uint32_t spin_limit, F &&site)
{
    const int Vh = g.Vh, stages = tl.stages;
    const int lane = threadIdx.x & 31, chunk = (threadIdx.x >> 5) % tl.nch, sg = (threadIdx.x >> 5) / tl.nch;
    unsigned char *ring = dsm + size_t(sg) * stages * kFxHopBytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(dsm + size_t(tl.nsg) * stages * kFxHopBytes) + 2 * sg * stages;
    uint64_t *empty = full + stages;
    const bool producer = chunk == 0 && lane == 0;
    if (producer) {
        for (int q = 0; q < stages; q++) {
            tc::mbar_init(&full[q], 1);
            tc::mbar_init(&empty[q], tl.nch);
        }
        tc::fence_mbar_init();
    }
    __syncthreads();
    const int ngroups = (Vh + 31) / 32;
    const int first = bx * tl.nsg + sg, gstride = nbx * tl.nsg;
    const int nitems = first < ngroups ? ((ngroups - 1 - first) / gstride + 1) * 16 : 0;
    // item j: hop j % 16 of this group's (j / 16)-th 32 sites
    int issued = 0, islot = 0; // items issued, and the slot of the next one
    uint32_t iphase = 1;       // parity to wait for before the next one's slot is refilled
    auto issue = [&]() {
        uint64_t *fb = &full[islot];
        tc::mbar_arrive_expect_tx(fb, kFxHopBytes);
        tc::bulk_load_1d(ring + size_t(islot) * kFxHopBytes,
                         L.w + fx_link_index((first + (issued >> 4) * gstride) * 32, (issued & 15) * 9), kFxHopBytes, fb);
        issued++;
        if (++islot == stages) {
            islot = 0;
            iphase ^= 1;
        }
    };
    if (producer)
        while (issued < min(stages, nitems)) issue();

    bool ok = true;
    int slot = 0;       // slot of the item in work
    uint32_t phase = 0; // its parity
#pragma unroll 1
    for (int it = 0; it < nitems && ok; it += 16) {
        const int at = (first + (it >> 4) * gstride) * 32 + lane;
        const int cb = min(at, Vh - 1);
        int c[4];
        cb_coords(g, par, cb, c);
        const int s = full_site(g, c);
        const int le = L.e[cb];
        const unsigned *dl = L.dl + size_t(4) * cb;
        const int E = fx_site_exponent(g, c, s, in.e, dl);
        FxAcc acc;
        acc.zero();
        // one hop: refill the ring, wait for the links, add
        auto hop = [&](int j, const FxVec &cur) {
            if (producer) {
                // a slot is refilled once every warp of the group has released it; the
                // producer blocks only when the hop its own warp needs now is not issued
                while (ok && issued < nitems && issued < it + j + stages) {
                    if (!tc::mbar_try_wait(&empty[islot], iphase)) {
                        if (issued > it + j) break;
                        ok = tc::mbar_wait(&empty[islot], iphase, status, tc::TC_TIMEOUT_EMPTY, spin_limit);
                        if (!ok) break;
                    }
                    issue();
                }
            }
            if (ok) ok = tc::mbar_wait(&full[slot], phase, status, tc::TC_TIMEOUT_FULL, spin_limit);
            const int4 *w = reinterpret_cast<const int4 *>(ring + size_t(slot) * kFxHopBytes) + lane;
            if (ok) fx_add(cur, E, acc, [&](int k) { return w[32 * k]; });
            tc::ring_release(&empty[slot], ok);
            if (++slot == stages) {
                slot = 0;
                phase ^= 1;
            }
        };
        FxVec a, b;
        SiteLine line(g, c, s, 0);
        unsigned d = __ldg(dl);
        a.load(g, line, 0, in, d);
#pragma unroll 1
        for (int mu = 0; mu < 4; mu++) {
            b.load(g, line, 1, in, d);
            hop(4 * mu, a);
            a.load(g, line, 2, in, d);
            hop(4 * mu + 1, b);
            b.load(g, line, 3, in, d);
            hop(4 * mu + 2, a);
            if (mu < 3) {
                line = SiteLine(g, c, s, mu + 1);
                d = __ldg(dl + mu + 1);
                a.load(g, line, 0, in, d);
            }
            hop(4 * mu + 3, b);
        }
        ok = __all_sync(0xffffffffu, ok); // the lanes leave the loop together
        if (ok && at < Vh) site(cb, c, s, E, le, acc);
    }
    // copies still in flight (only after a wait gave up) land before the block ends
    if (producer && !ok)
        for (int q = 0; q < stages; q++) {
            // the last item issued into slot q, if any: its parity follows from how often it was used
            const int uses = (issued + stages - 1 - q) / stages;
            if (uses > 0)
                for (int spin = 0; spin < (1 << 20) && !tc::mbar_try_wait(&full[q], (uses - 1) & 1); spin++) {
                }
        }
}

// ------------------------------------------------------------- host side
// Tile for k fields: ny launches' worth of blocks of nch fields and nsg site groups.  An SM
// holds 16 warps (128 registers); the tile keeps as many of them as it can on fields of
// their own, and each further reading of the links (ny) costs a little: 12 fields on
// 32^3x64 took 10 % longer with 12 warps at work than with 16.
inline FxTile fx_tile(int k, int *ny)
{
    FxTile t{1, kFxWarps, 0};
    double best = -1e9;
    for (int nch = 1; nch <= kFxWarps && nch <= k; nch++) {
        const int nsg = kFxWarps / nch, y = (k + nch - 1) / nch;
        const double score = double(16 / (nch * nsg) * nch * nsg) / 16 * k / (nch * y) - 0.03 * y;
        if (score >= best) {
            best = score;
            t.nch = nch;
            t.nsg = nsg;
            *ny = y;
        }
    }
    t.stages = t.nsg == 1 ? 8 : (t.nsg == 2 ? 6 : (t.nsg <= 4 ? 4 : 3));
    return t;
}

// mantissas and exponents of the FP64 parity field `in` into `out` (fx_field_bytes)
hisq_status launch_fx_split(hisq_ctx *ctx, const void *in, void *out);

// Several right-hand sides at once (at most kFxGroup): out_i = a x_i + b y_i + c D(in_i)
// on output parity par, and |out_i|^2.  Slot q of the group is right-hand side id[q];
// every FP64 field lies at base + 3 Vh double2 times its slot or its right-hand side.
constexpr int kFxGroup = 12;
struct FxArray {
    double2 *base; // null: not there
    bool by_slot;
};
struct FxGroup {
    int k;
    int id[kFxGroup];
};
struct FxBatch {
    FxArray in, out, x, y; // out null: norms only
    double a, b, c;
    void *mant;     // mantissas of in, fx_field_bytes per slot
    void *mant_out; // mantissas of out, or null
    bool norm;      // |out|^2 into ctx->bscal->out[id]
};
// in (FP64) to mantissas for every slot; with add, in += add first (FP32 fields at a
// stride of 24 Vh bytes by right-hand side)
hisq_status launch_fx_batch_split(hisq_ctx *ctx, const FxGroup &grp, FxArray in, void *mant, const void *add);
hisq_status launch_fx_batch(hisq_ctx *ctx, int par, const FxGroup &grp, const FxBatch &b);
hisq_status fx_blocks_per_sm(hisq_ctx *ctx, const void *kern, const FxTile &tl, int *bps);

} // namespace hisq
