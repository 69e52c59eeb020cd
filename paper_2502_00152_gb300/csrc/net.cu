// net.cu -- a gauge-covariant parallel-transport network that predicts an
// initial guess for CG (the learned part of the method, built on the paper's
// solver: CG still runs from the guess to the same true residual).
//
// One layer maps Cin complex colour-vector channels to Cout channels on the
// full lattice:
//   out_b(x) = sum_a sum_h w[b][a][h] (T_h in_a)(x)
//   T_0 = identity, T_{mu,fwd} in(x) = W_fwd(x) in(x+mu), T_{mu,bwd} in(x) = W_bwd(x) in(x-mu)
// with W the one-hop fat-link hop matrices of the Dirac operator (staggered
// phases, boundary signs and the backward minus sign included), so a layer with
// w = (0, 1, 1, ..., 1) is exactly the fat-link part of D and the map commutes
// with gauge transformations (scalar weights, covariant transports).
// Because T_{mu,fwd}^dag = -T_{mu,bwd}, the adjoint of a layer is the same layer
// with weights w'[a][b][0] = conj(w[b][a][0]), w'[a][b][mu,d] = -conj(w[b][a][mu,1-d]).
//
// Channel tensors: (C, V, 3) complex64, full lattice, s = x + X(y + Y(z + Z t)).
// Weights: (Cout, Cin, 9) complex64; optionally rounded to BF16 when staged.
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.cuh"

namespace hisq {

constexpr int kNetHops = 9;
constexpr int kNetMaxC = 16;

// two FP32 values as one operand of the packed FMA (each half an IEEE FMA)
typedef unsigned long long pairf;
__device__ __forceinline__ pairf pk(float a, float b)
{
    pairf d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ float2 upk(pairf a)
{
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(a));
    return d;
}
__device__ __forceinline__ void pfma(pairf &c, pairf a, pairf b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ pairf padd(pairf a, pairf b)
{
    pairf d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// coordinates of full-lattice site s
__device__ __forceinline__ void net_coords(const Geom &g, int s, int (&c)[4])
{
    int r = fdiv(s >> 1, g.dX2);
    c[0] = s - r * g.X;
    int q = fdiv(r, g.dY);
    c[1] = r - q * g.Y;
    r = q;
    q = fdiv(r, g.dZ);
    c[2] = r - q * g.Z;
    c[3] = q;
}

// neighbour of hop h (1 + 2 mu + d; 0: the site itself), full-lattice index
__device__ __forceinline__ int net_neighbour(const Geom &g, const int (&c)[4], int s, int h)
{
    if (h == 0) return s;
    const int mu = (h - 1) >> 1, d = (h - 1) & 1;
    const int L = dim_of(g, mu), cm = coord_of(c, mu);
    const int cn = d == 0 ? (cm + 1 == L ? 0 : cm + 1) : (cm == 0 ? L - 1 : cm - 1);
    return checked_index(g, s + (cn - cm) * stride_of(g, mu), g.V);
}

// fat hop matrix of hop h > 0 at site (parity arrays, nk kinds per direction)
__device__ __forceinline__ void net_link(const float4 *links_p, int nk, int cb, int h, CMat<float> &m)
{
    const int mu = (h - 1) >> 1;
    const bool bwd = (h - 1) & 1;
    const float4 *q = links_p + link_index(cb, mu * nk * 9, nk * 36);
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const float4 w = __ldg(q + 32 * k);
        m.re[k] = bwd ? w.y : w.x;
        m.im[k] = bwd ? w.w : w.z;
    }
}

__device__ __forceinline__ void net_load(const float2 *p, CVec<float> &v)
{
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const float2 a = __ldg(p + i);
        v.re[i] = a.x;
        v.im[i] = a.y;
    }
}

// weight of output b, input a, hop h of the layer as applied (adjoint: see above)
__device__ __forceinline__ float2 net_weight(const float2 *w, int cin, int b, int a, int h, int adjoint, int bf16)
{
    float2 v;
    if (!adjoint) {
        v = w[(size_t(b) * cin + a) * kNetHops + h];
    } else {
        const int hs = h == 0 ? 0 : (1 + (((h - 1) >> 1) << 1) + (1 - ((h - 1) & 1)));
        const float2 u = w[(size_t(a) * cin + b) * kNetHops + hs];
        v = h == 0 ? make_float2(u.x, -u.y) : make_float2(-u.x, u.y);
    }
    if (bf16) {
        v.x = __bfloat162float(__float2bfloat16_rn(v.x));
        v.y = __bfloat162float(__float2bfloat16_rn(v.y));
    }
    return v;
}

// out = layer(in) (adjoint = 0) or layer^dag(in) (adjoint = 1).  A thread computes one
// site for 2 P output channels (blockIdx.y: which): for each hop its matrix, for each
// input channel the transported vector, and for each pair of output channels 12 packed
// FMAs with the two weights as the halves, the vector's components repeated in both.  The
// weights are staged once per block and read as broadcasts; nothing else passes through
// shared memory.  The sums over the input channels of a hop are formed on their own and
// then added, which halves the rounding error of one long sum (1.9e-7 against 3.1e-7 of
// the result at 16 x 16 channels; 2.3e-7 before).  Bound by the FMA pipe: 9 ci co 12 +
// 8 ci 36 FMAs per site.  16 to 16 channels: 24^3x48 10.6 -> 1.0 ms, 16^3x32 2.1 -> 0.20 ms;
// 8 channels per thread 1.43 ms.
constexpr int kNetThreads = 128;

template <int P>
__global__ void __launch_bounds__(kNetThreads, P == 8 ? 2 : (P == 4 ? 3 : 4))
    k_net_layer(Geom g, const float4 *links0, const float4 *links1, int nk, const float2 *__restrict__ w, int cin,
                int cout, int adjoint, int bf16, const float2 *__restrict__ in, float2 *__restrict__ out)
{
    extern __shared__ float4 sw[]; // [hop][input channel][pair]: (re0, re1, im0, im1)
    const int co = adjoint ? cin : cout, ci = adjoint ? cout : cin;
    const int b0 = blockIdx.y * 2 * P;
    for (int t = threadIdx.x; t < kNetHops * ci * P; t += blockDim.x) {
        const int h = t / (ci * P), a = t / P % ci, b = b0 + 2 * (t % P);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (b < co) {
            const float2 u = net_weight(w, cin, b, a, h, adjoint, bf16);
            v.x = u.x;
            v.z = u.y;
        }
        if (b + 1 < co) {
            const float2 u = net_weight(w, cin, b + 1, a, h, adjoint, bf16);
            v.y = u.x;
            v.w = u.y;
        }
        sw[t] = v;
    }
    __syncthreads();
    const size_t V3 = size_t(g.V) * 3;
    for (int s0 = blockIdx.x * kNetThreads; s0 < g.V; s0 += gridDim.x * kNetThreads) {
        const int s = min(s0 + int(threadIdx.x), g.V - 1);
        int c[4];
        net_coords(g, s, c);
        const float4 *links_p = (c[0] + c[1] + c[2] + c[3]) & 1 ? links1 : links0;
        pairf re[P][3], im[P][3], sr[P][3], si[P][3]; // sums over the input channels of a hop, over all hops
#pragma unroll
        for (int p = 0; p < P; p++)
#pragma unroll
            for (int i = 0; i < 3; i++) sr[p][i] = si[p][i] = 0;
#pragma unroll 1
        for (int h = 0; h < kNetHops; h++) {
#pragma unroll
            for (int p = 0; p < P; p++)
#pragma unroll
                for (int i = 0; i < 3; i++) re[p][i] = im[p][i] = 0;
            CMat<float> m;
            if (h > 0) net_link(links_p, nk, s >> 1, h, m);
            const float2 *q = in + size_t(net_neighbour(g, c, s, h)) * 3;
            const ulonglong2 *wp = reinterpret_cast<const ulonglong2 *>(sw) + h * ci * P;
            CVec<float> nxt;
            net_load(q, nxt);
#pragma unroll 1
            for (int a = 0; a < ci; a++) {
                CVec<float> t = nxt;
                q += V3;
                if (a + 1 < ci) net_load(q, nxt);
                if (h > 0) {
                    const CVec<float> v = t;
                    t.zero();
                    mv_acc(t, m, v);
                }
                pairf tr[3], ti[3], tn[3];
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    tr[i] = pk(t.re[i], t.re[i]);
                    ti[i] = pk(t.im[i], t.im[i]);
                    tn[i] = pk(-t.im[i], -t.im[i]);
                }
#pragma unroll
                for (int p = 0; p < P; p++) {
                    const ulonglong2 u = wp[p]; // x: the two real parts, y: the imaginary ones
#pragma unroll
                    for (int i = 0; i < 3; i++) {
                        pfma(re[p][i], u.x, tr[i]);
                        pfma(im[p][i], u.x, ti[i]);
                        pfma(re[p][i], u.y, tn[i]);
                        pfma(im[p][i], u.y, tr[i]);
                    }
                }
                wp += P;
            }
#pragma unroll
            for (int p = 0; p < P; p++)
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    sr[p][i] = padd(sr[p][i], re[p][i]);
                    si[p][i] = padd(si[p][i], im[p][i]);
                }
        }
        if (s0 + int(threadIdx.x) < g.V) {
#pragma unroll
            for (int p = 0; p < P; p++) {
                const int b = b0 + 2 * p;
                float2 *o = out + size_t(b) * V3 + size_t(s) * 3;
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    const float2 r = upk(sr[p][i]), m = upk(si[p][i]);
                    if (b < co) o[i] = make_float2(r.x, m.x);
                    if (b + 1 < co) o[V3 + i] = make_float2(r.y, m.y);
                }
            }
        }
    }
}

// Weight gradients: G[b][a][h] = sum_x gout_b(x) . conj(T_h in_a(x)).  A block takes 16
// sites at a time: its 144 threads transport one (site, hop) each for every input channel
// into shared memory, then each accumulates a 4 x 4 tile of (b, (a, h)) over the 48 (site,
// colour) rows.  With fewer tiles than threads the rows are dealt to groups of threads.
// The products are summed in FP32 over kWgChain rows by chains of FMAs, the chains over
// kWgSum rows, and these sums in FP64, as the partial sums of groups and blocks are, in a
// fixed order.  Rounding, 16 x 16 channels, relative to the sums: 1.29e-7 with chains of 16
// rows; 1.8e-7 with one of all 48 (two roundings a product); 1.44e-7 with each product
// formed first, at half as many FP32 operations again.
// Bound by the FMA pipe and the latency of the transports' loads between two barriers, at
// three blocks per SM.  The FP64 sums of a thread stay in local memory, touched every
// fourth tile: in 64 registers they left an SM two blocks.  16 x 16 channels: 24^3x48 4.35
// -> 1.59 ms (FP64 sums after every tile 1.64, in registers 1.89), 16^3x32 0.33 ms.
constexpr int kWgSites = 16, kWgThreads = kWgSites * kNetHops, kWgRows = kWgSites * 3;
constexpr int kWgChain = 16, kWgSum = 192; // rows of one chain of FMAs, and of one FP32 sum of chains
constexpr int kWgPitch = kNetMaxC * kNetHops + 4; // floats per row of a plane: 16-byte rows, few conflicts

__global__ void __launch_bounds__(kWgThreads, 3)
    k_net_wgrad(Geom g, const float4 *links0, const float4 *links1, int nk, int cin, int cout,
                const float2 *__restrict__ in, const float2 *__restrict__ gout, int groups, double2 *part)
{
    extern __shared__ float4 dsm4[];
    float *st = reinterpret_cast<float *>(dsm4);      // [re, im][row][kWgPitch]: transports, row = 3 site + colour
    float2 *sg = reinterpret_cast<float2 *>(st + 2 * kWgRows * kWgPitch); // [row][kNetMaxC]: gout
    const int nah = cin * kNetHops, nta = (nah + 3) / 4, ntb = (cout + 3) / 4, ntile = nta * ntb;
    const int ls = threadIdx.x % kWgSites, h = threadIdx.x / kWgSites;
    // this thread's tile and rows
    const int tile = threadIdx.x % ntile, grp = threadIdx.x / ntile;
    const bool on = grp < groups;
    const int ta = tile % nta, tb = tile / nta;
    pairf ar[4][2], ai[4][2]; // FP32 sums [b][pair of (a, h)]
    double mem[32], *sr = mem; // FP64 sums
    asm("" : "+l"(sr));        // an address, so that they are not taken into registers
    double *si = sr + 16;
#pragma unroll
    for (int k = 0; k < 16; k++) {
        sr[k] = si[k] = 0;
        ar[k >> 2][k & 1] = ai[k >> 2][k & 1] = 0;
    }
    const int every = kWgSum / ((kWgRows + groups - 1) / groups); // tiles that make one FP32 sum
    int left = every;
    auto flush = [&]() {
#pragma unroll
        for (int b = 0; b < 4; b++)
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const float2 r = upk(ar[b][k]), m = upk(ai[b][k]);
                sr[4 * b + 2 * k] = sr[4 * b + 2 * k] + double(r.x);
                sr[4 * b + 2 * k + 1] = sr[4 * b + 2 * k + 1] + double(r.y);
                si[4 * b + 2 * k] = si[4 * b + 2 * k] + double(m.x);
                si[4 * b + 2 * k + 1] = si[4 * b + 2 * k + 1] + double(m.y);
                ar[b][k] = ai[b][k] = 0;
            }
        left = every;
    };
    const size_t V3 = size_t(g.V) * 3;
    // the columns past the last (a, h) and the channels past the last b stay zero
    for (int t = threadIdx.x; t < 2 * kWgRows * kWgPitch; t += blockDim.x) st[t] = 0.f;
    for (int t = threadIdx.x; t < kWgRows * kNetMaxC; t += blockDim.x) sg[t] = make_float2(0.f, 0.f);
    for (int blk = blockIdx.x; blk * kWgSites < g.V; blk += gridDim.x) {
        __syncthreads();
        const int s = blk * kWgSites + ls;
        const float live = s < g.V ? 1.f : 0.f;
        {
            const int sc = min(s, g.V - 1);
            int c[4];
            net_coords(g, sc, c);
            CMat<float> m;
            if (h > 0) net_link((c[0] + c[1] + c[2] + c[3]) & 1 ? links1 : links0, nk, sc >> 1, h, m);
            const float2 *q = in + size_t(net_neighbour(g, c, sc, h)) * 3;
            float *o = st + 3 * ls * kWgPitch + h;
            for (int a0 = 0; a0 < cin; a0 += 4) {
                CVec<float> v[4]; // four channels' loads in flight
#pragma unroll
                for (int k = 0; k < 4; k++) net_load(q + V3 * min(a0 + k, cin - 1), v[k]);
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    if (a0 + k >= cin) break;
                    CVec<float> t = v[k];
                    if (h > 0) {
                        t.zero();
                        mv_acc(t, m, v[k]);
                    }
#pragma unroll
                    for (int i = 0; i < 3; i++) {
                        o[i * kWgPitch + (a0 + k) * kNetHops] = live != 0.f ? t.re[i] : 0.f;
                        o[(kWgRows + i) * kWgPitch + (a0 + k) * kNetHops] = live != 0.f ? t.im[i] : 0.f;
                    }
                }
            }
        }
        for (int t = threadIdx.x; t < kWgRows * cout; t += blockDim.x) {
            const int b = t / kWgRows, r = t % kWgRows;
            const size_t x = size_t(blk) * kWgRows + r;
            sg[r * kNetMaxC + b] = x < V3 ? __ldg(gout + size_t(b) * V3 + x) : make_float2(0.f, 0.f);
        }
        __syncthreads();
        if (!on) continue;
#pragma unroll 1
        for (int r0 = grp; r0 < kWgRows; r0 += kWgChain * groups) {
            pairf cr[4][2], ci[4][2];
#pragma unroll
            for (int b = 0; b < 4; b++) cr[b][0] = cr[b][1] = ci[b][0] = ci[b][1] = 0;
            const int r1 = min(kWgRows, r0 + kWgChain * groups);
#pragma unroll 2
            for (int r = r0; r < r1; r += groups) {
                const ulonglong2 tr = *reinterpret_cast<const ulonglong2 *>(st + r * kWgPitch + 4 * ta);
                const ulonglong2 ti = *reinterpret_cast<const ulonglong2 *>(st + (kWgRows + r) * kWgPitch + 4 * ta);
                const float4 *gp = reinterpret_cast<const float4 *>(sg + r * kNetMaxC + 4 * tb);
                const float4 g0 = gp[0], g1 = gp[1];
                const float gr[4] = {g0.x, g0.z, g1.x, g1.z}, gi[4] = {g0.y, g0.w, g1.y, g1.w};
#pragma unroll
                for (int b = 0; b < 4; b++) { // g conj(t)
                    const pairf pr = pk(gr[b], gr[b]), pi = pk(gi[b], gi[b]), pn = pk(-gr[b], -gr[b]);
                    pfma(cr[b][0], pi, ti.x);
                    pfma(cr[b][1], pi, ti.y);
                    pfma(ci[b][0], pn, ti.x);
                    pfma(ci[b][1], pn, ti.y);
                    pfma(cr[b][0], pr, tr.x);
                    pfma(cr[b][1], pr, tr.y);
                    pfma(ci[b][0], pi, tr.x);
                    pfma(ci[b][1], pi, tr.y);
                }
            }
#pragma unroll
            for (int b = 0; b < 4; b++)
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    ar[b][k] = padd(ar[b][k], cr[b][k]);
                    ai[b][k] = padd(ai[b][k], ci[b][k]);
                }
        }
        if (--left == 0) flush();
    }
    flush();
    // the groups' sums through shared memory, in group order
    double2 *sd = reinterpret_cast<double2 *>(dsm4); // [group][tile][16]
    __syncthreads();
    if (on && grp > 0) {
#pragma unroll
        for (int k = 0; k < 16; k++)
            sd[(size_t(grp - 1) * ntile + tile) * 16 + k] =
                make_double2(sr[k], si[k]);
    }
    __syncthreads();
    if (!on || grp > 0) return;
    double2 *p = part + size_t(blockIdx.x) * cout * nah;
#pragma unroll
    for (int b = 0; b < 4; b++)
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const int bb = 4 * tb + b, aa = 4 * ta + a, k = 4 * b + a;
            if (bb >= cout || aa >= nah) continue;
            double2 t = make_double2(sr[k], si[k]);
            for (int w = 1; w < groups; w++) {
                const double2 o = sd[(size_t(w - 1) * ntile + tile) * 16 + k];
                t.x += o.x;
                t.y += o.y;
            }
            p[bb * nah + aa] = t;
        }
}

// gw[q] = sum of the nparts partial sums: 32 weights per block, each warp every eighth
// part, the eight sums in a fixed order
__global__ void __launch_bounds__(256) k_net_wgrad_finish(int nparts, int ntrip, const double2 *part, float2 *gw)
{
    __shared__ double2 sh[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = blockIdx.x * 32 + lane;
    double2 t = make_double2(0, 0);
    if (q < ntrip)
        for (int b = warp; b < nparts; b += 8) {
            const double2 v = part[size_t(b) * ntrip + q];
            t.x += v.x;
            t.y += v.y;
        }
    sh[warp][lane] = t;
    __syncthreads();
    if (warp > 0 || q >= ntrip) return;
    for (int w = 1; w < 8; w++) {
        t.x += sh[w][lane].x;
        t.y += sh[w][lane].y;
    }
    gw[q] = make_float2(float(t.x), float(t.y));
}

// Adam step on n real parameters (Kingma & Ba, ICLR 2015)
__global__ void k_adam(int n, float *w, const float *gr, float *m1, float *m2, float lr, float b1, float b2, float eps,
                       float bc1, float bc2)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gv = gr[i];
        m1[i] = b1 * m1[i] + (1.f - b1) * gv;
        m2[i] = b2 * m2[i] + (1.f - b2) * gv * gv;
        const float mh = m1[i] / bc1, vh = m2[i] / bc2;
        w[i] -= lr * mh / (sqrtf(vh) + eps);
    }
}

} // namespace hisq

using namespace hisq;

extern "C" {

hisq_status hisq_net_layer(hisq_ctx *ctx, int cin, int cout, const float *w_dev, int w_bf16, int adjoint,
                           const float *in_dev, float *out_dev)
{
    if (!ctx) return HISQ_ERR_INVALID_ARG;
    if (!w_dev || !in_dev || !out_dev || cin < 1 || cout < 1 || cin > kNetMaxC || cout > kNetMaxC)
        return set_err(ctx, HISQ_ERR_INVALID_ARG, "network layer: 1..16 channels, device pointers");
    if (!ctx->links_loaded) return set_err(ctx, HISQ_ERR_STATE, "links not loaded");
    HISQ_CUDA(cudaSetDevice(ctx->device));
    const int co = adjoint ? cin : cout, ci = adjoint ? cout : cin;
    const int nk = ctx->long_recon == 18 ? 2 : 1;
    const int nblk = (ctx->g.V + kNetThreads - 1) / kNetThreads;
    // output channels per thread: 16, fewer where the layer has fewer or the lattice
    // leaves fewer than four blocks per SM
    int P = (co + 1) / 2 <= 1 ? 1 : ((co + 1) / 2 <= 2 ? 2 : ((co + 1) / 2 <= 4 ? 4 : 8));
    while (P > 1 && nblk * ((co + 2 * P - 1) / (2 * P)) < 4 * ctx->num_sms) P /= 2;
    auto launch = [&](auto kern, int per_sm) -> hisq_status {
        const int ny = (co + 2 * P - 1) / (2 * P);
        const int gx = std::min(nblk, std::max(1, ctx->num_sms * per_sm / ny));
        const size_t smem = sizeof(float4) * kNetHops * ci * P;
        ctx->launches++;
        kern<<<dim3(gx, ny), kNetThreads, smem, ctx->stream>>>(ctx->g, ctx->links_f[0], ctx->links_f[1], nk,
                                                               (const float2 *)w_dev, cin, cout, adjoint, w_bf16,
                                                               (const float2 *)in_dev, (float2 *)out_dev);
        HISQ_CUDA(cudaGetLastError());
        return HISQ_OK;
    };
    switch (P) {
    case 1: return launch(k_net_layer<1>, 16);
    case 2: return launch(k_net_layer<2>, 8);
    case 4: return launch(k_net_layer<4>, 3);
    default: return launch(k_net_layer<8>, 2);
    }
}

hisq_status hisq_net_wgrad(hisq_ctx *ctx, int cin, int cout, const float *in_dev, const float *gout_dev, float *gw_dev)
{
    if (!ctx) return HISQ_ERR_INVALID_ARG;
    if (!in_dev || !gout_dev || !gw_dev || cin < 1 || cout < 1 || cin > kNetMaxC || cout > kNetMaxC)
        return set_err(ctx, HISQ_ERR_INVALID_ARG, "network gradient: 1..16 channels, device pointers");
    if (!ctx->links_loaded) return set_err(ctx, HISQ_ERR_STATE, "links not loaded");
    HISQ_CUDA(cudaSetDevice(ctx->device));
    const size_t smem = size_t(kWgRows) * (2 * kWgPitch * sizeof(float) + kNetMaxC * sizeof(float2));
    HISQ_CUDA(cudaFuncSetAttribute(k_net_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
    const int nblk = (ctx->g.V + kWgSites - 1) / kWgSites;
    const int grid = std::min(nblk, ctx->num_sms * 3);
    const int ntrip = cin * cout * kNetHops;
    const int ntile = ((cin * kNetHops + 3) / 4) * ((cout + 3) / 4);
    const int groups = std::max(1, std::min(kWgThreads / ntile, 12));
    double2 *part = (double2 *)get_buf(ctx, BUF_NET_PART, sizeof(double2) * size_t(grid) * ntrip);
    if (!part) return HISQ_ERR_OOM;
    const int nk = ctx->long_recon == 18 ? 2 : 1;
    ctx->launches += 2;
    k_net_wgrad<<<grid, kWgThreads, smem, ctx->stream>>>(ctx->g, ctx->links_f[0], ctx->links_f[1], nk, cin, cout,
                                                         (const float2 *)in_dev, (const float2 *)gout_dev, groups,
                                                         part);
    HISQ_CUDA(cudaGetLastError());
    k_net_wgrad_finish<<<(ntrip + 31) / 32, 256, 0, ctx->stream>>>(grid, ntrip, part, (float2 *)gw_dev);
    HISQ_CUDA(cudaGetLastError());
    return HISQ_OK;
}

hisq_status hisq_net_adam(hisq_ctx *ctx, int n, float *w_dev, const float *g_dev, float *m1_dev, float *m2_dev,
                          float lr, float beta1, float beta2, float eps, int step)
{
    if (!ctx) return HISQ_ERR_INVALID_ARG;
    if (n < 1 || !w_dev || !g_dev || !m1_dev || !m2_dev || step < 1)
        return set_err(ctx, HISQ_ERR_INVALID_ARG, "adam: bad arguments");
    HISQ_CUDA(cudaSetDevice(ctx->device));
    const float bc1 = 1.f - std::pow(beta1, float(step)), bc2 = 1.f - std::pow(beta2, float(step));
    ctx->launches++;
    k_adam<<<(n + 255) / 256, 256, 0, ctx->stream>>>(n, w_dev, g_dev, m1_dev, m2_dev, lr, beta1, beta2, eps, bc1, bc2);
    HISQ_CUDA(cudaGetLastError());
    return HISQ_OK;
}

} // extern "C"
