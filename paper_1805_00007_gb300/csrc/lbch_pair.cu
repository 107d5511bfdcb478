// lbch_pair.cu -- launch and set-up of the two-step kernel (periodic instances, tau_g = 1), f32 and f64.
#include "lbch_internal.h"
#include "lbch_pair.cuh"

namespace lbch {
namespace {

template <typename C, typename P, int TX, int TY, int NT>
cudaError_t launch_pair_v(lbch_handle* h, int parity)
{
    using L = PairShape<C, P, TX, TY>;
    const lbch_handle::PerShape& ps = h->pr[h->pshape];
    PairArgs<C, P> a;
    a.inst0 = h->inst[0];
    a.inst = h->d_inst;
    a.tile_begin = ps.d_tile_begin;
    a.ttabs = static_cast<const C*>(ps.d_ttabs);
    a.n_inst = h->n_inst;
    a.total_tiles = ps.total_tiles;
    a.pitch = h->pitch;
    a.phi_in = static_cast<const P*>(h->phi[parity]);
    a.lo_in = h->lo[parity];
    a.phi_out = static_cast<P*>(h->phi[parity ^ 1]);
    a.lo_out = h->lo[parity ^ 1];
    a.ctl = h->ctl;
    a.t_off = h->t_off;
    a.t_adv = h->t_adv;
    a.need_time = h->need_time;
    a.Tf = launch_T(h);
    a.read_n = launch_reads_n(h);
    a.debug_skip = h->debug_skip;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ps.grid);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = L::BYTES;
    cfg.stream = h->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = h->no_pdl ? 0 : 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return h->n_inst == 1 ? cudaLaunchKernelEx(&cfg, ch_pair_kernel<C, P, TX, TY, NT, true>, a)
                          : cudaLaunchKernelEx(&cfg, ch_pair_kernel<C, P, TX, TY, NT, false>, a);
}

template <typename C, typename P, int TX, int TY, int NT>
cudaError_t prepare_pair_v(lbch_handle* h, int k)
{
    using L = PairShape<C, P, TX, TY>;
    const void* kern = reinterpret_cast<const void*>(ch_pair_kernel<C, P, TX, TY, NT, false>);
    cudaError_t e = lbch_kernel_smem(kern, h->device, L::BYTES);
    if (e == cudaSuccess)
        e = lbch_kernel_smem(reinterpret_cast<const void*>(ch_pair_kernel<C, P, TX, TY, NT, true>), h->device, L::BYTES);
    if (e != cudaSuccess) return e;
    int per_sm = 0, sms = 0;
    e = lbch_kernel_fit(kern, h->device, NT, L::BYTES, &per_sm, &sms);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    h->pr[k].grid = std::max(1, std::min(h->pr[k].total_tiles, per_sm * sms));
    return cudaSuccess;
}

// Every tile's velocity tables over the tile + 6, periodically wrapped, contiguous per tile so that one bulk copy brings
// them: X1, X2 by column, Y1, Y2 by row, padded to 16 bytes.  One value per thread, once per handle.  (Formed on the host and copied, the
// four shapes' tables took 4.3 of the 9.1 ms in which a 1024^2 float handle is set up.)
template <typename C>
__global__ void __launch_bounds__(256) pair_tables_kernel(const InstDev* inst, int n_inst, const int* tile_begin, const C* tabs,
                                                          int pitch, int tx, int ty, int stride, long long count, C* out)
{
    const long long e = (long long)blockIdx.x * 256 + threadIdx.x;
    if (e >= count) return;
    const int t = (int)(e / stride), i = (int)(e - (long long)t * stride);
    const int k = find_inst(tile_begin, n_inst, t), local = t - tile_begin[k];
    const InstDev& I = inst[k];
    const int tiles_x = (I.nx + tx - 1) / tx, w6 = tx + 12, h6 = ty + 12;
    const C* X = tabs + I.tab;
    const C* Y = X + 2 * pitch;
    C v = C(0);
    if (i < 2 * w6) {
        const int q = i >= w6;
        v = X[q * pitch + GC + wrap(local % tiles_x * tx - 6 + i - q * w6, I.nx)];
    } else if (i < 2 * w6 + 2 * h6) {
        const int j = i - 2 * w6, q = j >= h6;
        v = Y[q * I.ylen + GR + wrap(local / tiles_x * ty - 6 + j - q * h6, I.ny)];
    }
    out[e] = v;
}

template <typename C> cudaError_t pair_tables_t(lbch_handle* h, int k)
{
    const Shape sh = pair_shape(h->prec, k);
    const int stride = pair_table_stride<C>(sh.tx, sh.ty);
    const long long count = (long long)h->pr[k].total_tiles * stride;
    pair_tables_kernel<C><<<(unsigned)((count + 255) / 256), 256, 0, h->stream>>>(
        h->d_inst, h->n_inst, h->pr[k].d_tile_begin, tables<C>(h), h->pitch, sh.tx, sh.ty, stride, count,
        static_cast<C*>(h->pr[k].d_ttabs));
    return cudaGetLastError();
}

}  // namespace
}  // namespace lbch

size_t lbch_pair_tables_bytes(const lbch_handle* h, int k)
{
    const Shape sh = pair_shape(h->prec, k);
    return h->prec == LBCH_F64 ? (size_t)h->pr[k].total_tiles * lbch::pair_table_stride<double>(sh.tx, sh.ty) * 8
                               : (size_t)h->pr[k].total_tiles * lbch::pair_table_stride<float>(sh.tx, sh.ty) * 4;
}

cudaError_t lbch_pair_tables(lbch_handle* h, int k)
{
    return h->prec == LBCH_F64 ? lbch::pair_tables_t<double>(h, k) : lbch::pair_tables_t<float>(h, k);
}

// The shapes are those of pair_shape() (lbch_internal.h), in its order.
cudaError_t lbch_launch_pair(lbch_handle* h, int parity)
{
    using namespace lbch;
    const int k = h->pshape;
    if (k < 0 || k >= kPairShapes || !h->pr[k].d_tile_begin || h->pr[k].grid < 1) return cudaErrorInvalidValue;
    if (h->prec == LBCH_F64)
        return k == 0 ? launch_pair_v<double, double, 32, 8, 512>(h, parity)
             : k == 1 ? launch_pair_v<double, double, 16, 8, 256>(h, parity)
             : k == 2 ? launch_pair_v<double, double, 16, 16, 512>(h, parity) : launch_pair_v<double, double, 32, 14, 1024>(h, parity);
    return k == 0 ? launch_pair_v<float, float, 32, 16, 512>(h, parity)
         : k == 1 ? launch_pair_v<float, float, 32, 14, 512>(h, parity)
         : k == 2 ? launch_pair_v<float, float, 16, 8, 256>(h, parity) : launch_pair_v<float, float, 32, 8, 512>(h, parity);
}

cudaError_t lbch_prepare_pair(lbch_handle* h, int k)
{
    using namespace lbch;
    if (h->prec == LBCH_F64)
        return k == 0 ? prepare_pair_v<double, double, 32, 8, 512>(h, k)
             : k == 1 ? prepare_pair_v<double, double, 16, 8, 256>(h, k)
             : k == 2 ? prepare_pair_v<double, double, 16, 16, 512>(h, k) : prepare_pair_v<double, double, 32, 14, 1024>(h, k);
    return k == 0 ? prepare_pair_v<float, float, 32, 16, 512>(h, k)
         : k == 1 ? prepare_pair_v<float, float, 32, 14, 512>(h, k)
         : k == 2 ? prepare_pair_v<float, float, 16, 8, 256>(h, k) : prepare_pair_v<float, float, 32, 8, 512>(h, k);
}
