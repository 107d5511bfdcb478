// lbch_sweep_launch.cuh -- launch and set-up of the row-sweep kernel for one precision; included by the
// per-precision translation units, so that their kernels compile in parallel.
#pragma once
#include "lbch_internal.h"
#include "lbch_sweep.cuh"

namespace lbch {

template <typename C, typename S, typename P, bool FF, bool GEN, bool SINGLE, bool WALLS, bool M3>
cudaError_t launch_sweep_v(lbch_handle* h, int parity)
{
    using L = SweepShape<S, P, FF, GEN, GEN && (WALLS || !SINGLE)>;
    const lbch_handle::SweepCut& sc = h->sw[h->shape][GEN];
    SweepArgs<C, S, P> a;
    a.inst0 = h->inst[0];
    a.inst = h->d_inst;
    a.items = static_cast<const SweepItem*>(sc.d_items);
    a.tabs = tables<C>(h);
    a.n_items = sc.n_items;
    a.strips = sc.strips;
    a.rows_per = sc.rows_per;
    a.pitch = h->pitch;
    a.phi_in = static_cast<const P*>(h->phi[parity]);
    a.lo_in = h->lo[parity];
    a.phi_out = static_cast<P*>(h->phi[parity ^ 1]);
    a.lo_out = h->lo[parity ^ 1];
    a.ctl = h->ctl;
    a.t_off = h->t_off;
    a.t_adv = h->t_adv;
    a.timed = h->timed;
    a.Tf = launch_T(h);
    a.read_n = launch_reads_n(h);
    a.g_in = static_cast<const S*>(h->g[parity]);
    a.g_out = static_cast<S*>(h->g[parity ^ 1]);
    a.H_in = M3 ? static_cast<const C*>(h->H[parity]) : nullptr;
    a.H_out = M3 ? static_cast<C*>(h->H[parity ^ 1]) : nullptr;
    a.H_plane = (long long)h->rows * h->pitch;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((sc.n_items + sc.nw - 1) / sc.nw);
    cfg.blockDim = dim3(sc.nw * 32);
    cfg.dynamicSmemBytes = L::bytes(sc.nw);
    cfg.stream = h->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = h->no_pdl ? 0 : 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, ch_sweep_kernel<C, S, P, FF, GEN, SINGLE, WALLS, M3>, a);
}

// F(GEN, SINGLE, WALLS) of the handle's form of the sweep, as compile-time constants
template <typename F> cudaError_t sweep_form(const lbch_handle* h, bool gen, F&& f)
{
    using T = std::true_type;
    using N = std::false_type;
    const bool single = h->n_inst == 1;
    if (gen) {
        if (single) return h->walls ? f(T(), T(), T()) : f(T(), T(), N());
        return h->walls ? f(T(), N(), T()) : f(T(), N(), N());
    }
    if (single) return h->walls ? f(N(), T(), T()) : f(N(), T(), N());
    return h->walls ? f(N(), N(), T()) : f(N(), N(), N());
}

template <typename C, typename S, typename P, bool FF, bool M3>
cudaError_t launch_sweep_t(lbch_handle* h, int parity)
{
    return sweep_form(h, sweep_gen(h), [&](auto gen, auto single, auto walls) {
        return launch_sweep_v<C, S, P, FF, decltype(gen)::value, decltype(single)::value, decltype(walls)::value, M3>(h, parity);
    });
}

// Dynamic shared memory of the sweep kernel the handle steps with (gen: with the populations), the warps of it that
// one SM holds, and the columns of its strips.
template <typename C, typename S, typename P, bool FF, bool M3>
cudaError_t prepare_sweep_t(lbch_handle* h, bool gen, SweepFit* fit)
{
    return sweep_form(h, gen, [&](auto g, auto single, auto walls) {
        constexpr bool G = decltype(g)::value;
        using L = SweepShape<S, P, FF, G, G && (decltype(walls)::value || !decltype(single)::value)>;
        const void* kern = reinterpret_cast<const void*>(
            ch_sweep_kernel<C, S, P, FF, G, decltype(single)::value, decltype(walls)::value, M3>);
        cudaError_t e = lbch_kernel_smem(kern, h->device, L::bytes(L::NW));
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        e = lbch_kernel_fit(kern, h->device, L::NW * 32, L::bytes(L::NW), &per_sm, &fit->sms);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        fit->warps = per_sm * L::NW;
        fit->nw = L::NW;
        fit->width = L::W;
        fit->lead = L::LEAD;
        return cudaSuccess;
    });
}

}  // namespace lbch
