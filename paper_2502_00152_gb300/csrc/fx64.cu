// fx64.cu -- block floating-point operands of the fixed-point FP64 operator
// (fx64.cuh): the links once, when they are loaded, and a colour field per
// application.
#include "fx64.cuh"

namespace hisq {

// One thread per site: 48 B read, 50 B written (HBM bound; 4 % of the operator's own
// traffic).
__global__ void __launch_bounds__(256) k_fx_split(int Vh, const double2 *__restrict__ in, longlong2 *__restrict__ v,
                                                  short *__restrict__ e)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Vh; i += gridDim.x * blockDim.x) {
        double2 q[3];
        int eb = 0;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            q[c] = in[size_t(c) * Vh + i];
            eb = max(eb, max(fx_exponent(q[c].x), fx_exponent(q[c].y)));
        }
        bool zero = true;
#pragma unroll
        for (int c = 0; c < 3; c++) zero = zero && q[c].x == 0.0 && q[c].y == 0.0;
        if (!zero && (eb < kFxVecLo || eb > kFxVecHi)) {
            e[i] = short(kFxMark); // the operator reads the FP64 field at the sites this one touches
            continue;
        }
        if (zero) eb = kFxVecLo; // below every other exponent, mantissas 0
        e[i] = short(eb);
#pragma unroll
        for (int c = 0; c < 3; c++)
            v[size_t(c) * Vh + i] = make_longlong2(fx_mantissa<7>(q[c].x, eb), fx_mantissa<7>(q[c].y, eb));
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

// The gathered FP64 links of one parity to mantissas, in place: each thread owns the
// 144 elements of its site.  Zero matrices keep an ordinary exponent; sites whose
// largest entry lies outside 2^+-100 stay FP64 and are marked.
__global__ void __launch_bounds__(256) k_links_fx(int Vh, int4 *w, short *e)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Vh; i += gridDim.x * blockDim.x) {
        int4 *p = w + fx_link_index(i, 0);
        int eb = 0;
        for (int k = 0; k < 144; k++) {
            const int4 q = p[32 * k];
            eb = max(eb, max((q.y >> 20) & 0x7ff, (q.w >> 20) & 0x7ff));
        }
        if (eb < kFxLinkLo || eb > kFxLinkHi) {
            bool zero = eb == 0;
            for (int k = 0; k < 144 && zero; k++) {
                const int4 q = p[32 * k];
                zero = ((q.y | q.w) & 0x7fffffff) == 0 && (q.x | q.z) == 0;
            }
            if (!zero) {
                e[i] = short(kFxMark);
                continue;
            }
            eb = 1022;
        }
        e[i] = short(eb);
        for (int k = 0; k < 144; k++) {
            const int4 q = p[32 * k];
            int4 o;
            fx_limbs(fx_mantissa<3>(__hiloint2double(q.y, q.x), eb), o.x, o.y);
            fx_limbs(fx_mantissa<3>(__hiloint2double(q.w, q.z), eb), o.z, o.w);
            p[32 * k] = o;
        }
    }
}

hisq_status launch_links_fx(hisq_ctx *ctx, int par)
{
    const int grid = grid_for(ctx, ctx->g.Vh, 256, 8);
    k_links_fx<<<grid, 256, 0, ctx->stream>>>(ctx->g.Vh, ctx->links_x[par], ctx->links_xe[par]);
    const cudaError_t err = cudaGetLastError();
    return err == cudaSuccess ? HISQ_OK : cuda_err(ctx, err, "fixed-point links");
}

} // namespace hisq
