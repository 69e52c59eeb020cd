// fx64.cu -- block floating-point operands of the fixed-point FP64 operator
// (fx64.cuh): the links once, when they are loaded, and a colour field per
// application.
#include "fx64.cuh"

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

namespace hisq {

// One thread per site: 48 B read, 50 B written (HBM bound; 4 % of the operator's own
// traffic).
__global__ void __launch_bounds__(256) k_fx_split(int Vh, const double2 *__restrict__ in, longlong2 *__restrict__ v,
                                                  short *__restrict__ e)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Vh; i += gridDim.x * blockDim.x) {
        CVec<double> q;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double2 d = in[size_t(c) * Vh + i];
            q.re[c] = d.x;
            q.im[c] = d.y;
        }
        fx_store_site(v, e, Vh, i, q);
    }
}

hisq_status launch_fx_split(hisq_ctx *ctx, const void *in, void *out)
{
    const int Vh = ctx->g.Vh;
    const int grid = grid_for(ctx, Vh, 256, 8);
    k_fx_split<<<grid, 256, 0, ctx->stream>>>(Vh, (const double2 *)in, (longlong2 *)out,
                                              (short *)((char *)out + size_t(Vh) * 48));
    const cudaError_t err = cudaGetLastError();
    return err == cudaSuccess ? HISQ_OK : cuda_err(ctx, err, "fixed-point split");
}

// The gathered FP64 links of one parity to the operator's form, in place: each thread owns
// the 144 elements of its site.  Zero matrices get an ordinary exponent; sites whose
// largest entry lies outside 2^+-100, or that have one more than 127 binary places below
// it, stay FP64 and are marked.
__global__ void __launch_bounds__(256) k_links_fx(int Vh, int4 *w, unsigned *dl, short *e)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Vh; i += gridDim.x * blockDim.x) {
        int4 *p = w + fx_link_index(i, 0);
        int eb = 0, low = 0x7ff; // exponents of the largest entry and of the smallest that is not zero
        int hop[16];             // of the largest of each hop, 0 for a zero matrix
        bool zero = true;
#pragma unroll
        for (int h = 0; h < 16; h++) {
            hop[h] = 0;
            for (int k = 9 * h; k < 9 * h + 9; k++) {
                const int4 q = p[32 * k];
                for (const double x : {__hiloint2double(q.y, q.x), __hiloint2double(q.w, q.z)}) {
                    hop[h] = max(hop[h], fx_exponent(x));
                    if (x != 0.0) low = min(low, fx_exponent(x));
                    zero = zero && x == 0.0;
                }
            }
            eb = max(eb, hop[h]);
        }
        if (zero) eb = low = 1022;
        if (eb < kFxLinkLo || eb > kFxLinkHi || eb - low > kFxDepth) {
            e[i] = short(kFxMark);
            reinterpret_cast<uint4 *>(dl)[i] = make_uint4(0, 0, 0, 0);
            continue;
        }
        e[i] = short(eb);
        unsigned d[4] = {0, 0, 0, 0};
#pragma unroll
        for (int h = 0; h < 16; h++) {
            const int depth = min(eb - hop[h], kFxDepth);
            d[h >> 2] |= unsigned(depth) << (8 * (h & 3));
            for (int k = 9 * h; k < 9 * h + 9; k++) {
                const int4 q = p[32 * k];
                const long long re = fx_encode(__hiloint2double(q.y, q.x), eb - depth);
                const long long im = fx_encode(__hiloint2double(q.w, q.z), eb - depth);
                p[32 * k] = make_int4(int(re), int(re >> 32), int(im), int(im >> 32));
            }
        }
        reinterpret_cast<uint4 *>(dl)[i] = make_uint4(d[0], d[1], d[2], d[3]);
    }
}

hisq_status launch_links_fx(hisq_ctx *ctx, int par)
{
    const int grid = grid_for(ctx, ctx->g.Vh, 256, 8);
    k_links_fx<<<grid, 256, 0, ctx->stream>>>(ctx->g.Vh, ctx->links_x[par], ctx->links_xe[par],
                                              (short *)(ctx->links_xe[par] + size_t(4) * ctx->g.Vh));
    const cudaError_t err = cudaGetLastError();
    return err == cudaSuccess ? HISQ_OK : cuda_err(ctx, err, "fixed-point links");
}

// ------------------------------------------------- several right-hand sides
__device__ __forceinline__ double2 *fx_at(const FxArray &a, const FxGroup &g, int q, int Vh)
{
    return a.base + size_t(3) * Vh * (a.by_slot ? q : g.id[q]);
}

// in_q (+= add_q) to mantissas, one field per blockIdx.y
__global__ void __launch_bounds__(256) k_fx_batch_split(int Vh, FxGroup grp, FxArray in, char *mant, size_t ms,
                                                        const char *add)
{
    const int q = blockIdx.y;
    double2 *p = fx_at(in, grp, q, Vh);
    longlong2 *v = (longlong2 *)(mant + ms * q);
    short *e = (short *)(mant + ms * q + size_t(Vh) * 48);
    const SpinorF f{(float4 *)(add + size_t(24) * Vh * grp.id[q]),
                    (float2 *)(add + size_t(24) * Vh * grp.id[q] + size_t(16) * Vh), Vh};
    const SpinorD d{p, Vh};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Vh; i += gridDim.x * blockDim.x) {
        CVec<double> x = d.load(i);
        if (add) {
            const CVec<float> s = f.load(i);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                x.re[c] = fma(1.0, double(s.re[c]), x.re[c]);
                x.im[c] = fma(1.0, double(s.im[c]), x.im[c]);
            }
            d.store(i, x);
        }
        fx_store_site(v, e, Vh, i, x);
    }
}

hisq_status launch_fx_batch_split(hisq_ctx *ctx, const FxGroup &grp, FxArray in, void *mant, const void *add)
{
    const int Vh = ctx->g.Vh;
    const dim3 grid(grid_for(ctx, Vh, 256, 8), grp.k);
    k_fx_batch_split<<<grid, 256, 0, ctx->stream>>>(Vh, grp, in, (char *)mant, fx_field_bytes(Vh), (const char *)add);
    const cudaError_t err = cudaGetLastError();
    return err == cudaSuccess ? HISQ_OK : cuda_err(ctx, err, "fixed-point split (batch)");
}

// The operator for a group of fields (fx_ring_sites), blockIdx.y: fields blockIdx.y * nch ...
// Bound by instruction issue and the multiply-add pipe together (54 % busy at 12 warps):
// 32^3x64, per field and application, splits included: 386 us for 12 or 5 fields, one field
// at a time 439, FP64 FMAs 1058.  With one exponent per site instead of one per hop 377;
// with links cut to 56-bit limbs beforehand as well (bits of the small ones lost) 351 and
// 340; two fields per thread, with four real products per complex
// one, took 495.
__global__ void __launch_bounds__(32 * kFxWarps, 2)
    k_dslash_fx_batch(Geom g, int par, LinksX L, FxGroup grp, FxBatch o, size_t ms, FxTile tl, double *partials,
                      unsigned int *ticket, double *norms, int *status, uint32_t spin_limit)
{
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ double sh[kFxWarps];
    __shared__ bool am_last;
    const int Vh = g.Vh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // a warp past the group's last field computes that one again and writes nothing
    const int q0 = blockIdx.y * tl.nch + warp % tl.nch;
    const int q = min(q0, grp.k - 1);
    const char *mq = (const char *)o.mant + ms * q;
    const FxField in{(const longlong2 *)mq, (const short *)(mq + size_t(Vh) * 48), nullptr};
    double red = 0;
    fx_ring_sites(g, par, L, in, tl, blockIdx.x, gridDim.x, dsm, status, spin_limit,
                  [&](int cb, const int (&c)[4], int s, int E, int le, const FxAcc &acc) {
                      if (q0 >= grp.k) return;
                      CVec<double> v, t;
                      double u = o.c;
                      if (E != kFxMark && le != kFxMark) {
                          u *= fx_unit(E, le);
#pragma unroll
                          for (int i = 0; i < 3; i++) {
                              v.re[i] = double(fx_sum(acc, 2 * i));
                              v.im[i] = double(fx_sum(acc, 2 * i + 1));
                          }
                      } else {
                          v = fx_site_fp64(g, c, s, L.w + fx_link_index(cb, 0), L.dl + size_t(4) * cb, le,
                                             fx_at(o.in, grp, q, Vh));
                      }
                      t.zero();
                      if (o.y.base) {
                          const CVec<double> y = SpinorD{fx_at(o.y, grp, q, Vh), Vh}.load(cb);
#pragma unroll
                          for (int i = 0; i < 3; i++) {
                              t.re[i] = o.b * y.re[i];
                              t.im[i] = o.b * y.im[i];
                          }
                      }
                      if (o.x.base) {
                          const CVec<double> x = SpinorD{fx_at(o.x, grp, q, Vh), Vh}.load(cb);
#pragma unroll
                          for (int i = 0; i < 3; i++) {
                              t.re[i] = fma(o.a, x.re[i], t.re[i]);
                              t.im[i] = fma(o.a, x.im[i], t.im[i]);
                          }
                      }
#pragma unroll
                      for (int i = 0; i < 3; i++) {
                          t.re[i] = fma(u, v.re[i], t.re[i]);
                          t.im[i] = fma(u, v.im[i], t.im[i]);
                      }
                      if (o.out.base) SpinorD{fx_at(o.out, grp, q, Vh), Vh}.store(cb, t);
                      if (o.mant_out) {
                          char *m = (char *)o.mant_out + ms * q;
                          fx_store_site((longlong2 *)m, (short *)(m + size_t(Vh) * 48), Vh, cb, t);
                      }
                      if (o.norm) red += t.norm2();
                  });
    if (!o.norm) return;
    // per-field sums: lanes by a fixed shuffle tree, site groups in order, blocks in block order
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) red += __shfl_down_sync(0xffffffffu, red, off);
    if (lane == 0) sh[warp] = red;
    __syncthreads();
    if (threadIdx.x < tl.nch && blockIdx.y * tl.nch + threadIdx.x < grp.k) {
        double t = 0;
        for (int w = 0; w < tl.nsg; w++) t += sh[w * tl.nch + threadIdx.x];
        partials[size_t(blockIdx.x) * kMaxBatch + blockIdx.y * tl.nch + threadIdx.x] = t;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) am_last = (atomicAdd(ticket, 1u) == gridDim.x * gridDim.y - 1);
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    for (int f = warp; f < grp.k; f += blockDim.x >> 5) { // a warp per field
        double t = 0;
        for (int b = lane; b < int(gridDim.x); b += 32) t += __ldcg(partials + size_t(b) * kMaxBatch + f);
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) t += __shfl_down_sync(0xffffffffu, t, off);
        if (lane == 0) norms[grp.id[f]] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        *ticket = 0u;
        __threadfence();
    }
}

// blocks of a ring kernel per SM (its shared memory allowed first), kept per device, kernel and tile
hisq_status fx_blocks_per_sm(hisq_ctx *ctx, const void *kern, const FxTile &tl, int *bps)
{
    static std::mutex mu;
    static std::map<std::tuple<int, const void *, int, int>, int> cache;
    std::lock_guard<std::mutex> lock(mu);
    int &n = cache[std::make_tuple(ctx->device, kern, tl.nch, tl.nsg)];
    if (n == 0) {
        HISQ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 113 * 1024));
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, 32 * tl.nch * tl.nsg, tl.smem()) != cudaSuccess ||
            n < 1) {
            cudaGetLastError();
            n = 1;
        }
    }
    *bps = n;
    return HISQ_OK;
}

hisq_status launch_fx_batch(hisq_ctx *ctx, int par, const FxGroup &grp, const FxBatch &b)
{
    const int Vh = ctx->g.Vh;
    if (grp.k < 1 || grp.k > kFxGroup) return set_err(ctx, HISQ_ERR_INVALID_ARG, "FP64 batch of 1..%d", kFxGroup);
    int ny = 1;
    const FxTile tl = fx_tile(grp.k, &ny);
    const int threads = 32 * tl.nch * tl.nsg;
    const size_t smem = tl.smem();
    auto kern = k_dslash_fx_batch;
    int bps;
    hisq_status st = fx_blocks_per_sm(ctx, (const void *)kern, tl, &bps);
    if (st != HISQ_OK) return st;
    // all parts resident together, so that they sweep the sites in step
    const dim3 grid(std::max(1, std::min(grid_for(ctx, Vh, 32 * tl.nsg, bps), ctx->num_sms * bps / ny)), ny);
    bool timed = false;
    st = fp64_prof_begin(ctx, grp.k, &timed);
    if (st != HISQ_OK) return st;
    kern<<<grid, threads, smem, ctx->stream>>>(ctx->g, par, links_fx(ctx, par), grp, b,
                                               fx_field_bytes(Vh), tl, ctx->bpartials, ctx->ticket + 40, ctx->bscal->out,
                                               ctx->wait_status_d, ring_spin_limit(ctx));
    const cudaError_t err = cudaGetLastError();
    st = fp64_prof_end(ctx, timed);
    return err == cudaSuccess ? st : cuda_err(ctx, err, "FP64 dslash (batch) launch");
}

} // namespace hisq
