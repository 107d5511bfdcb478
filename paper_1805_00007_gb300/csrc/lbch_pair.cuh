// lbch_pair.cuh -- two consecutive steps of the Cahn-Hilliard lattice Boltzmann equation per launch.
//
// For handles whose instances all have tau_g = 1 and periodic boundaries.  At tau_g = 1, Eq. LB gives
// g* = g_eq + S/2, so the state is phi alone (the populations are multiplied by 1 - 1/tau = 0).  The output
// phi(t+1) of a node depends on phi(t) three nodes out: mu and D = div(phi u) one node out (Eq. mu,
// Eq. mark3), their gradients, the force and the collision one node further (Eqs. liangFi, geq), and the
// pull of the streamed populations one more.  Two steps therefore need phi(t) on the tile + 6.
//
// A CTA loads phi(t) (and the low part of the float path) on tile + 6 with the domain indices wrapped
// periodically -- the stored ghost frame, three deep, is not used -- runs step t on tile + 3 and step t+1
// on the tile, entirely in shared memory, and stores phi(t+2) with the ghost images a one-step launch
// reads.  Each node value is formed by the same per-node helpers in the same order as in the one-step
// kernels (a halo node is computed as the periodic image it stands for), so the result is bit for bit
// that of two one-step launches.  The neighbouring tiles recompute the halo; what this buys is one
// launch -- fixed latency, dependency wait, prologue, load round trip -- per two steps, on grids small
// enough for a step to be latency-bound.
#pragma once
#include "lbch_kernels.cuh"

namespace lbch {

template <typename C, typename P>
struct PairArgs {
    InstDev inst0;          // the record of instance 0, for single-instance handles (read from the parameters)
    const InstDev* inst;
    const int* tile_begin;  // first tile of each instance for this launch's tile shape
    const C* ttabs;         // each tile's velocity tables over tile + 6, PairShape::TAB_STRIDE values per tile
    int n_inst;
    int total_tiles;
    int pitch;
    const P* phi_in;        // phi(t): the high part on the float path
    const float* lo_in;     // low part of phi(t) (float path)
    P* phi_out;             // phi(t+2), with its ghost images
    float* lo_out;
    Ctl* ctl;
    int t_off;              // the launch's first step is ctl->time + t_off, its second one step later
    int t_adv;              // when nonzero, the launch's last CTA advances ctl->time by t_adv
    int need_time;          // some instance's flow depends on the step index
    int read_n;             // ... and the launch reads it (no table of time factors)
    const double* Tf;       // the instances' time factors at the first step, then at the second, or null (step_T)
    int debug_skip;         // test hook: CTA 0 never issues its first table copy (its bounded wait runs out)
};

// Values of a tile's velocity tables: X1, X2 over the TX + 12 columns, Y1, Y2 over the TY + 12 rows, padded to 16 bytes
template <typename C> __host__ __device__ constexpr int pair_table_stride(int tx, int ty)
{
    return (int)((2 * (tx + ty + 24) * sizeof(C) + 15) / 16 * 16 / sizeof(C));
}

// Shared-memory regions, each centred on the tile: region k spans the tile plus k nodes on every side.
template <typename C, typename P, int TX, int TY>
struct PairShape {
    static constexpr bool FF = sizeof(C) == 4;  // float-float phi
    static constexpr int W6 = TX + 12, H6 = TY + 12, N6 = W6 * H6;  // phi(t), velocity tables
    static constexpr int W5 = TX + 10, H5 = TY + 10, N5 = W5 * H5;  // mu, D of step t
    static constexpr int W4 = TX + 8, H4 = TY + 8, N4 = W4 * H4;    // post-collision populations of step t
    static constexpr int W3 = TX + 6, H3 = TY + 6, N3 = W3 * H3;    // phi(t+1); low parts of phi(t), phi(t+1)
    static constexpr int W2 = TX + 4, H2 = TY + 4, N2 = W2 * H2;    // mu, D of step t+1
    static constexpr int W1 = TX + 2, H1 = TY + 2, N1 = W1 * H1;    // post-collision populations of step t+1
    __host__ __device__ static constexpr size_t a128(size_t b) { return (b + 127) / 128 * 128; }
    static constexpr size_t OFF_LO0 = a128(N6 * sizeof(P));
    static constexpr size_t OFF_HI1 = OFF_LO0 + (FF ? a128(N3 * 4) : 0);
    static constexpr size_t OFF_LO1 = OFF_HI1 + a128(N3 * sizeof(P));
    static constexpr size_t OFF_MU = OFF_LO1 + (FF ? a128(N3 * 4) : 0);
    static constexpr size_t OFF_D = OFF_MU + a128(N5 * sizeof(C));
    static constexpr size_t OFF_POST = OFF_D + a128(N5 * sizeof(C));
    static constexpr size_t OFF_TAB = OFF_POST + a128(9 * N4 * sizeof(C));
    static constexpr int TAB_STRIDE = pair_table_stride<C>(TX, TY);  // a tile's velocity tables
    static constexpr unsigned TAB_BYTES = TAB_STRIDE * sizeof(C);
    // the Y tables times the two steps' time factors (time-dependent flows): Y1, Y2 for step t, then for t + 1
    static constexpr size_t OFF_YT = OFF_TAB + a128(TAB_BYTES);
    static constexpr size_t BYTES = OFF_YT + a128(4 * H6 * sizeof(C)) + 128;  // + alignment slack
};

// i reduced into [0, n); i lies within a few periods of the domain
__device__ __forceinline__ int wrap_near(int i, int n)
{
    while (i < 0) i += n;
    while (i >= n) i -= n;
    return i;
}

// mu (Eq. mu) and D = div(phi u) on a region of width W, height H, from phi on the region one node wider
// (row stride PW); the velocity tables (Y with the step's time factor) are indexed by the phi region's
// columns/rows shifted by `to`.
template <typename C, typename P, int W, int H, int PW, int NT>
__device__ __forceinline__ void pair_mu_div(const P* ph, const C* sX1, const C* sX2, const C* sY1, const C* sY2,
                                            int to, const Consts<C>& K0, bool model2, C* s_mu, C* s_D)
{
    for_region<W, H, NT>([&](int e, int r, int c) {
        const P* q = ph + (r + 1) * PW + c + 1;
        const C ce = cvt<C>(q[0]);
        const C pE = cvt<C>(q[1]), pW = cvt<C>(q[-1]), pN = cvt<C>(q[PW]), pS = cvt<C>(q[-PW]);
        const C pNE = cvt<C>(q[PW + 1]), pNW = cvt<C>(q[PW - 1]), pSE = cvt<C>(q[-PW + 1]), pSW = cvt<C>(q[-PW - 1]);
        s_mu[e] = mu9(ce, pE, pW, pN, pS, pNE, pNW, pSE, pSW, K0);
        if (model2) {
            const int tc = c + to, tr = r + to;  // the table index of the node's column/row minus one
            s_D[e] = div9(pE, pW, pN, pS, pNE, pNW, pSE, pSW, sX1[tc], sX1[tc + 2], sX2[tc], sX2[tc + 1],
                          sX2[tc + 2], sY1[tr], sY1[tr + 1], sY1[tr + 2], sY2[tr], sY2[tr + 2]);
        }
    });
}

// Force, equilibrium, source and collision at tau = 1 (Eqs. liangFi, mark3, geq, LB) on a region of width
// W, height H; mu and D come from the region one node wider (stride MW), phi from the region two nodes
// wider (stride PW), the velocity at table index (row, col) + tu.  The nine post-collision populations
// are stored as planes of W * H values, the axis directions in a quarter (collide9).
template <typename C, typename P, int W, int H, int MW, int PW, int NT>
__device__ __forceinline__ void pair_collide(const P* ph_reg, const C* s_mu, const C* s_D, const C* sX1,
                                             const C* sX2, const C* sY1, const C* sY2, int tu, const Consts<C>& K0,
                                             bool model2, C* s_post)
{
    for_region<W, H, NT>([&](int e, int r, int c) {
        const int m = (r + 1) * MW + (c + 1);
        C gmx, gmy, gDx = C(0), gDy = C(0);
        grad9(s_mu[m + 1], s_mu[m - 1], s_mu[m + MW], s_mu[m - MW], s_mu[m + MW + 1], s_mu[m + MW - 1],
              s_mu[m - MW + 1], s_mu[m - MW - 1], gmx, gmy);
        if (model2)
            grad9(s_D[m + 1], s_D[m - 1], s_D[m + MW], s_D[m - MW], s_D[m + MW + 1], s_D[m + MW - 1], s_D[m - MW + 1],
                  s_D[m - MW - 1], gDx, gDy);
        const C ph = cvt<C>(ph_reg[(r + 2) * PW + c + 2]);
        const C ux = node_u(sX1[c + tu], sY1[r + tu]), uy = node_u(sX2[c + tu], sY2[r + tu]);
        C Px, Py, Jx, Jy, post[9];
        node_flow(ph, ux, uy, K0, Px, Py);
        node_force(ph, gmx, gmy, gDx, gDy, Px, Py, model2, K0, Jx, Jy);
        collide9<C, true>(s_mu[m], ux, uy, Px, Py, Jx, Jy, nullptr, K0, post);
        post[0] = rest_add(post[0], ph, K0);
#pragma unroll
        for (int q = 0; q < 9; q++) s_post[q * (W * H) + e] = post[q];
    });
}

// The streamed populations at node (r, c) of a region of width W, from the post-collision planes of the
// region one node wider (width W + 2, planes of NP values): g_q(x) = g*_q(x - c_q).  Returns g_0 and the
// sum of g_1..g_8 in the order of the one-step kernels.
template <typename C, int W, int NP>
__device__ __forceinline__ C pair_pull(const C* s_post, int r, int c, C& v0)
{
    constexpr int PW = W + 2;
    const int p = (r + 1) * PW + (c + 1);
    C v[9];
    v0 = s_post[p];
#pragma unroll
    for (int q = 1; q < 9; q++) v[q] = s_post[q * NP + p - cy(q) * PW - cx(q)];
    return stream_sum_q(v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8]);
}

// ---- the same phases with two neighbouring nodes per thread (the float path)
//
// In float the launch is bound by latency and instruction issue.  A thread that takes the pair (a, b) of a row loads the
// neighbourhood of both as aligned pairs of values (15 loads instead of 38 for mu and D, 17 instead of 44 for the
// collision, 12 instead of 18 for the pull), forms the column values they share once, and halves the index arithmetic,
// with the values and operations of the one-node phases (600 instructions per update instead of 780).  Half the threads
// take every phase of a 32 x 14 tile in one pass, and at 64 registers two blocks of 512 fit on an SM, so that a launch's
// blocks set up (tables, load offsets) beside the previous launch's last phases.  Us per step before -> with pairs ->
// with two blocks per SM: 256^2 2.55 -> 2.56 -> 2.10; 100^2 1.90 (32 x 8) -> 1.84 -> 1.56 (16 x 8); 360^2 4.7 -> 4.6 -> 3.6.
template <int W, int H, int NT, typename F> __device__ __forceinline__ void for_pairs(F&& f)
{
    static_assert(W % 2 == 0, "whole pairs");
    for (int i = threadIdx.x; i < H * (W / 2); i += NT) {
        const int r = i / (W / 2);
        f(r, 2 * (i - r * (W / 2)));
    }
}
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void st2(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }
// four neighbouring values from an even offset
struct Quad { float L, a, b, R; };
__device__ __forceinline__ Quad ld4(const float* p)
{
    const float2 u = ld2(p), v = ld2(p + 2);
    return {u.x, u.y, v.x, v.y};
}

template <int W, int H, int PW, int NT>
__device__ __forceinline__ void pair_mu_div2(const float* ph, const float* sX1, const float* sX2, const float* sY1,
                                             const float* sY2, int to, const Consts<float>& K0, bool model2, float* s_mu,
                                             float* s_D)
{
    for_pairs<W, H, NT>([&](int r, int c) {
        const float* q = ph + r * PW + c;
        const Quad S = ld4(q), M = ld4(q + PW), N = ld4(q + 2 * PW);
        float dl, dla, dlb;
        const float zL = node_z(S.L, M.L, N.L, dl), za = node_z(S.a, M.a, N.a, dla);
        const float zb = node_z(S.b, M.b, N.b, dlb), zR = node_z(S.R, M.R, N.R, dl);
        st2(s_mu + r * W + c, node_mu(M.a, dla, za, zb, zL, K0), node_mu(M.b, dlb, zb, zR, za, K0));
        if (model2) {
            const float *x1 = sX1 + c + to, *x2 = sX2 + c + to, *y1 = sY1 + r + to, *y2 = sY2 + r + to;
            const float y1S = y1[0], y14 = op_mul(4.0f, y1[1]), y1N = y1[2], y2S = y2[0], y2N = y2[2];
            float E, Ea, Eb, ER, WL, Wa, Wb, W_;
            node_flux(S.L, M.L, N.L, x1[0], x2[0], y1S, y14, y1N, y2S, y2N, E, WL);
            const float da = node_flux(S.a, M.a, N.a, x1[1], x2[1], y1S, y14, y1N, y2S, y2N, Ea, Wa);
            const float db = node_flux(S.b, M.b, N.b, x1[2], x2[2], y1S, y14, y1N, y2S, y2N, Eb, Wb);
            node_flux(S.R, M.R, N.R, x1[3], x2[3], y1S, y14, y1N, y2S, y2N, ER, W_);
            st2(s_D + r * W + c, node_div(da, Eb, WL), node_div(db, ER, Wa));
        }
    });
}

// 12 grad of a field at the pair from its values on the region one node wider (row stride MW), q at the south-west
template <int MW>
__device__ __forceinline__ void grad_pair(const float* q, float2& gx, float2& gy, float2& mid)
{
    const Quad S = ld4(q), M = ld4(q + MW), N = ld4(q + 2 * MW);
    const float wL = node_w(S.L, M.L, N.L), wa = node_w(S.a, M.a, N.a), wb = node_w(S.b, M.b, N.b), wR = node_w(S.R, M.R, N.R);
    const float da = N.a - S.a, db = N.b - S.b;
    gx = make_float2(wb - wL, wR - wa);
    gy = make_float2(node_gy(N.L - S.L, da, db), node_gy(da, db, N.R - S.R));
    mid = make_float2(M.a, M.b);
}

template <int W, int H, int MW, int PW, int NT>
__device__ __forceinline__ void pair_collide2(const float* ph_reg, const float* s_mu, const float* s_D, const float* sX1,
                                              const float* sX2, const float* sY1, const float* sY2, int tu,
                                              const Consts<float>& K0, bool model2, float* s_post)
{
    for_pairs<W, H, NT>([&](int r, int c) {
        float2 gmx, gmy, gDx = make_float2(0.0f, 0.0f), gDy = gDx, mu, D;
        grad_pair<MW>(s_mu + r * MW + c, gmx, gmy, mu);
        if (model2) grad_pair<MW>(s_D + r * MW + c, gDx, gDy, D);
        const float2 ph = ld2(ph_reg + (r + 2) * PW + c + 2);
        const float y1 = sY1[r + tu], y2 = sY2[r + tu];
        auto node = [&](float p, float m, float gx, float gy, float dx, float dy, int k, float* post) {
            const float ux = node_u(sX1[c + tu + k], y1), uy = node_u(sX2[c + tu + k], y2);
            float Px, Py, Jx, Jy;
            node_flow(p, ux, uy, K0, Px, Py);
            node_force(p, gx, gy, dx, dy, Px, Py, model2, K0, Jx, Jy);
            collide9<float, true>(m, ux, uy, Px, Py, Jx, Jy, nullptr, K0, post);
        };
        float pa[9], pb[9];
        node(ph.x, mu.x, gmx.x, gmy.x, gDx.x, gDy.x, 0, pa);
        node(ph.y, mu.y, gmx.y, gmy.y, gDx.y, gDy.y, 1, pb);
#pragma unroll
        for (int q = 0; q < 9; q++) st2(s_post + q * (W * H) + r * W + c, pa[q], pb[q]);
    });
}

// The streamed populations at the pair (r, c), (r, c + 1) of a region of width W: what comes from the columns to either
// side lies at even offsets of the region one node wider, what stays in its column at odd ones.
template <int W, int NP>
__device__ __forceinline__ float2 pair_pull2(const float* s_post, int r, int c, float2& v0)
{
    constexpr int PW = W + 2;
    const float* p = s_post + r * PW + c;
    const float2 v1 = ld2(p + 1 * NP + PW), v5 = ld2(p + 5 * NP), v8 = ld2(p + 8 * NP + 2 * PW);
    const float2 v3 = ld2(p + 3 * NP + PW + 2), v6 = ld2(p + 6 * NP + 2), v7 = ld2(p + 7 * NP + 2 * PW + 2);
    const float* p2 = p + 2 * NP + 1;
    const float* p4 = p + 4 * NP + 2 * PW + 1;
    v0 = make_float2(p[PW + 1], p[PW + 2]);
    return make_float2(stream_sum_q(v1.x, p2[0], v3.x, p4[0], v5.x, v6.x, v7.x, v8.x),
                       stream_sum_q(v1.y, p2[1], v3.y, p4[1], v5.y, v6.y, v7.y, v8.y));
}

// phi(t+1) = phi(t) + g_0 + sum_q g_q on the float path: hi + lo absorbs the increment exactly (TwoSum),
// as in the one-step kernels.  (On the double path phi(t+1) is the plain sum.)
__device__ __forceinline__ float pair_phi(float h, float lo_in, float v0, float sumq, float& lo_out)
{
    const float tt = lo_in + (v0 + sumq);
    const float sm = h + tt;
    const float bb = sm - h;
    lo_out = (h - (sm - bb)) + (tt - bb);
    return sm;
}

// Shared-memory views of one CTA's regions.
template <typename C, typename P, int TX, int TY>
struct PairSmem {
    P* phi0;     // phi(t) on tile + 6
    float* lo0;  // its low part on tile + 3 (float path)
    P* hi1;      // phi(t+1) on tile + 3
    float* lo1;
    C *mu, *D;   // mu and D of the step in progress
    C* post;     // post-collision populations of the step in progress, nine planes
    C *X1, *X2, *Y1, *Y2;  // velocity tables over the columns / rows of tile + 6
    C* YT;       // Y1, Y2 times the time factor of step t, then of step t + 1
    __device__ explicit PairSmem(unsigned char* raw)
    {
        using L = PairShape<C, P, TX, TY>;
        unsigned char* base = smem_aligned128(raw);
        phi0 = reinterpret_cast<P*>(base);
        lo0 = reinterpret_cast<float*>(base + L::OFF_LO0);
        hi1 = reinterpret_cast<P*>(base + L::OFF_HI1);
        lo1 = reinterpret_cast<float*>(base + L::OFF_LO1);
        mu = reinterpret_cast<C*>(base + L::OFF_MU);
        D = reinterpret_cast<C*>(base + L::OFF_D);
        post = reinterpret_cast<C*>(base + L::OFF_POST);
        X1 = reinterpret_cast<C*>(base + L::OFF_TAB);
        X2 = X1 + L::W6;
        Y1 = X2 + L::W6;
        Y2 = Y1 + L::H6;
        YT = reinterpret_cast<C*>(base + L::OFF_YT);
    }
};

// A tile's velocity tables (columns and rows of tile + 6, periodically wrapped; laid out per tile at
// set-up) arrive by one bulk copy on an mbarrier, issued by thread 0 first thing, so that the copy's
// latency overlaps the dependency wait and the phi loads.  Thread 0 waits for it (bounded: a copy that never
// lands is reported through ctl->err) before the barrier that precedes the first phase.
template <typename C, typename P, int TX, int TY>
__device__ __forceinline__ void pair_fetch_tables(const PairSmem<C, P, TX, TY>& S, const C* ttabs, int t, uint64_t* bar)
{
    using L = PairShape<C, P, TX, TY>;
    fence_proxy_async();  // the table region was last read through the generic proxy
    mbar_expect_tx(bar, L::TAB_BYTES);
    bulk_load(S.X1, ttabs + (size_t)t * L::TAB_STRIDE, L::TAB_BYTES, bar);
}

// The values one thread loads for a tile: phi on tile + 6 and (float path) its low part on tile + 3, at
// periodically wrapped domain positions.  The offsets, from the instance's first domain node, are computed
// once per tile; -1 marks no value.
template <typename C, typename P, int TX, int TY, int NT>
struct PairLoad {
    using L = PairShape<C, P, TX, TY>;
    static constexpr int IT6 = (L::N6 + NT - 1) / NT, IT3 = (L::N3 + NT - 1) / NT;
    long long o6[IT6], o3[IT3];
    __device__ void init(int nx, int ny, int pitch, int x0, int y0)
    {
#pragma unroll
        for (int i = 0; i < IT6; i++) {
            const int e = threadIdx.x + i * NT, r = e / L::W6, c = e - r * L::W6;
            o6[i] = e < L::N6 ? (long long)wrap_near(y0 - 6 + r, ny) * pitch + wrap_near(x0 - 6 + c, nx) : -1;
        }
#pragma unroll
        for (int i = 0; i < IT3; i++) {
            const int e = threadIdx.x + i * NT, r = e / L::W3, c = e - r * L::W3;
            o3[i] = e < L::N3 && L::FF ? (long long)wrap_near(y0 - 3 + r, ny) * pitch + wrap_near(x0 - 3 + c, nx) : -1;
        }
    }
    // every load is in flight before the first store to shared memory; L2 only (another CTA wrote them)
    __device__ void load(const PairSmem<C, P, TX, TY>& S, const P* phi, const float* lo) const
    {
        P v[IT6];
        float w[IT3];
#pragma unroll
        for (int i = 0; i < IT6; i++)
            if (o6[i] >= 0) v[i] = __ldcg(phi + o6[i]);
#pragma unroll
        for (int i = 0; i < IT3; i++)
            if (o3[i] >= 0) w[i] = __ldcg(lo + o3[i]);
#pragma unroll
        for (int i = 0; i < IT6; i++)
            if (o6[i] >= 0) S.phi0[threadIdx.x + i * NT] = v[i];
#pragma unroll
        for (int i = 0; i < IT3; i++)
            if (o3[i] >= 0) S.lo0[threadIdx.x + i * NT] = w[i];
    }
};

// Steps t and t+1 of one tile from phi(t) and the tables in shared memory (loaded and synchronised by the
// caller): phi(t+2) of the tile's domain nodes and their ghost images into phi_out (rb: the instance's first
// domain node).  timed: the flow depends on time; T0, T1: its time factor at the two steps (else 1).  Ends
// without a barrier.
template <typename C, typename P, int TX, int TY, int NT>
__device__ __forceinline__ void pair_steps(const PairSmem<C, P, TX, TY>& S, const InstDev& I, bool timed, C T0, C T1,
                                           int x0, int y0, int pitch, long long rb, P* phi_out, float* lo_out)
{
    using L = PairShape<C, P, TX, TY>;
    constexpr int W6 = L::W6, W3 = L::W3;
    const Consts<C>& K0 = consts<C>(I);
    const bool model2 = I.model == 2;

    const C *Ya1 = S.Y1, *Ya2 = S.Y2, *Yb1 = S.Y1, *Yb2 = S.Y2;  // the Y tables of the two steps
    if (timed) {
        for (int e = threadIdx.x; e < 2 * L::H6; e += NT) {
            const C y = S.Y1[e];
            S.YT[e] = op_mul(y, T0);
            S.YT[2 * L::H6 + e] = op_mul(y, T1);
        }
        __syncthreads();
        Ya1 = S.YT;
        Ya2 = Ya1 + L::H6;
        Yb1 = Ya2 + L::H6;
        Yb2 = Yb1 + L::H6;
    }

    const int nx = I.nx, ny = I.ny;
    // phi(t+2) of a domain node, with its periodic images in the ghost frame (three deep), read by one-step launches
    auto images = [&](int gx, int gy, P hi) {
        if (gx >= 3 && gx < nx - 3 && gy >= 3 && gy < ny - 3) return;
        for_images3(gx, gy, nx, ny, 0, [&](int xx, int yy) { phi_out[rb + (long long)yy * pitch + xx] = hi; });
    };

    if constexpr (L::FF) {
        // step t: mu, D on tile + 5; collision on tile + 4; streaming to phi(t+1) on tile + 3
        pair_mu_div2<L::W5, L::H5, W6, NT>(S.phi0, S.X1, S.X2, Ya1, Ya2, 0, K0, model2, S.mu, S.D);
        __syncthreads();
        pair_collide2<L::W4, L::H4, L::W5, W6, NT>(S.phi0, S.mu, S.D, S.X1, S.X2, Ya1, Ya2, 2, K0, model2, S.post);
        __syncthreads();
        for_pairs<W3, L::H3, NT>([&](int r, int c) {
            float2 v0;
            const float2 sum = pair_pull2<W3, L::N4>(S.post, r, c, v0);
            const float* h = S.phi0 + (r + 3) * W6 + c + 3;
            const float2 l = ld2(S.lo0 + r * W3 + c);
            float la, lb;
            const float ha = pair_phi(h[0], l.x, v0.x, sum.x, la), hb = pair_phi(h[1], l.y, v0.y, sum.y, lb);
            st2(S.hi1 + r * W3 + c, ha, hb);
            st2(S.lo1 + r * W3 + c, la, lb);
        });
        __syncthreads();

        // step t+1: mu, D on tile + 2; collision on tile + 1; streaming to phi(t+2) on the tile
        pair_mu_div2<L::W2, L::H2, W3, NT>(S.hi1, S.X1, S.X2, Yb1, Yb2, 3, K0, model2, S.mu, S.D);
        __syncthreads();
        pair_collide2<L::W1, L::H1, L::W2, W3, NT>(S.hi1, S.mu, S.D, S.X1, S.X2, Yb1, Yb2, 5, K0, model2, S.post);
        __syncthreads();
        for_pairs<TX, TY, NT>([&](int r, int c) {
            const int gx = x0 + c, gy = y0 + r;
            if (gx >= nx || gy >= ny) return;
            float2 v0;
            const float2 sum = pair_pull2<TX, L::N1>(S.post, r, c, v0);
            const int k = (r + 3) * W3 + c + 3;
            float la, lb;
            const float ha = pair_phi(S.hi1[k], S.lo1[k], v0.x, sum.x, la);
            const float hb = pair_phi(S.hi1[k + 1], S.lo1[k + 1], v0.y, sum.y, lb);
            const long long node = rb + (long long)gy * pitch + gx;
            if (gx + 1 < nx) {
                st2(phi_out + node, ha, hb);
                st2(lo_out + node, la, lb);
            } else {
                phi_out[node] = ha;
                lo_out[node] = la;
            }
            images(gx, gy, ha);
            if (gx + 1 < nx) images(gx + 1, gy, hb);
        });
    } else {
        pair_mu_div<C, P, L::W5, L::H5, W6, NT>(S.phi0, S.X1, S.X2, Ya1, Ya2, 0, K0, model2, S.mu, S.D);
        __syncthreads();
        pair_collide<C, P, L::W4, L::H4, L::W5, W6, NT>(S.phi0, S.mu, S.D, S.X1, S.X2, Ya1, Ya2, 2, K0, model2, S.post);
        __syncthreads();
        for_region<W3, L::H3, NT>([&](int e, int r, int c) {
            C v0;
            const C sumq = pair_pull<C, W3, L::N4>(S.post, r, c, v0);
            S.hi1[e] = v0 + sumq;
        });
        __syncthreads();
        pair_mu_div<C, P, L::W2, L::H2, W3, NT>(S.hi1, S.X1, S.X2, Yb1, Yb2, 3, K0, model2, S.mu, S.D);
        __syncthreads();
        pair_collide<C, P, L::W1, L::H1, L::W2, W3, NT>(S.hi1, S.mu, S.D, S.X1, S.X2, Yb1, Yb2, 5, K0, model2, S.post);
        __syncthreads();
        for_region<TX, TY, NT>([&](int e, int r, int c) {
            const int gx = x0 + c, gy = y0 + r;
            if (gx >= nx || gy >= ny) return;
            C v0;
            const C sumq = pair_pull<C, TX, L::N1>(S.post, r, c, v0);
            const P hi = v0 + sumq;
            phi_out[rb + (long long)gy * pitch + gx] = hi;
            images(gx, gy, hi);
        });
    }
}

// The instance and origin of tile t.
template <int TX, int TY>
__device__ __forceinline__ void pair_locate(const int* tile_begin, int n_inst, const InstDev* inst, int t, int& k,
                                            int& x0, int& y0)
{
    k = find_inst(tile_begin, n_inst, t);
    const int local = t - tile_begin[k];
    const int tiles_x = (inst[k].nx + TX - 1) / TX;
    x0 = (local % tiles_x) * TX;
    y0 = (local / tiles_x) * TY;
}

// One launch per two steps: a persistent CTA walks its tiles.  SINGLE (a handle of one instance): the
// instance record stays in the launch parameters, so the tile's origin, tables and load offsets need no
// memory round trip (the table loads start at once, the phi loads right after the dependency wait), and the
// per-node helpers take the instance's constants as constant-bank operands instead of loading them.
template <typename C, typename P, int TX, int TY, int NT, bool SINGLE>
__global__ void __launch_bounds__(NT, NT > 512 ? 1 : 2) ch_pair_kernel(const __grid_constant__ PairArgs<C, P> a)
{
    extern __shared__ unsigned char smem_raw[];
    const PairSmem<C, P, TX, TY> S(smem_raw);
    __shared__ long long s_time;
    __shared__ int s_k, s_x0, s_y0;
    __shared__ C s_T[2];
    __shared__ InstDev s_I;
    __shared__ __align__(8) uint64_t s_tbar;  // completion of the table copy
    __shared__ int s_abort;                    // a table wait ran out: the CTA stops after it
    const int tid = threadIdx.x;
    const int stride = gridDim.x;
    const bool any = (int)blockIdx.x < a.total_tiles;
    PairLoad<C, P, TX, TY, NT> ld;
    long long n = 0;
    int tuse = 0;  // table copies waited for so far (the mbarrier's phase)
    // thread 0: wait (bounded) for the tile's table copy.  When the wait runs out the kernel records the
    // error, lets the copy land if it was issued (bounded again) so that no copy into this CTA's shared
    // memory outlives it, and tells the CTA to stop; the step counter is still kept consistent below.
    auto wait_tables = [&]() {
        if (!mbar_wait_bounded(&s_tbar, (unsigned)(tuse & 1), WAIT_POLLS)) {
            atomicOr(&a.ctl->err, 1u);
            mbar_wait_bounded(&s_tbar, (unsigned)(tuse & 1), WAIT_POLLS);
            s_abort = 1;
        }
        tuse++;
    };
    if (tid == 0) s_abort = 0;
    if (tid == 0 && any) {
        mbar_init(&s_tbar, 1);
        fence_mbar_init();
        if (!(a.debug_skip && blockIdx.x == 0)) pair_fetch_tables<C, P, TX, TY>(S, a.ttabs, blockIdx.x, &s_tbar);
    }

    if constexpr (SINGLE) {
        const InstDev& I = a.inst0;
        const int tiles_x = (I.nx + TX - 1) / TX;
        const long long rb = (long long)I.row0 * a.pitch + GC;
        int x0 = ((int)blockIdx.x % tiles_x) * TX, y0 = ((int)blockIdx.x / tiles_x) * TY;
        if (any) ld.init(I.nx, I.ny, a.pitch, x0, y0);  // constant data: before the dependency wait
        grid_dependency_wait();
        grid_launch_dependents();
        if (any) ld.load(S, a.phi_in + rb, a.lo_in + rb);
        if (tid == 0) {
            if (any) wait_tables();
            s_time = a.read_n ? a.ctl->time : 0;
            if (a.need_time) {  // (forming the 1 of a steady flow takes its thread 0.2 us of the launch)
                s_T[0] = (C)step_T(a.Tf, 0, I, s_time + a.t_off);
                s_T[1] = (C)step_T(a.Tf, 1, I, s_time + a.t_off + 1);
            }
        }
        __syncthreads();
        n = s_time + a.t_off;
        for (int t = blockIdx.x; t < a.total_tiles && !s_abort; t += stride) {
            if (t != (int)blockIdx.x) {
                __syncthreads();  // the previous tile's shared data are read no more
                if (tid == 0) pair_fetch_tables<C, P, TX, TY>(S, a.ttabs, t, &s_tbar);
                x0 = (t % tiles_x) * TX;
                y0 = (t / tiles_x) * TY;
                ld.init(I.nx, I.ny, a.pitch, x0, y0);
                ld.load(S, a.phi_in + rb, a.lo_in + rb);
                if (tid == 0) wait_tables();
                __syncthreads();
                if (s_abort) break;
            }
            pair_steps<C, P, TX, TY, NT>(S, I, a.need_time, s_T[0], s_T[1], x0, y0, a.pitch, rb, a.phi_out, a.lo_out);
        }
    } else {
        // thread 0: tile t's instance (copied when it changes) and origin
        auto locate = [&](int t) {
            int k, x0, y0;
            pair_locate<TX, TY>(a.tile_begin, a.n_inst, a.inst, t, k, x0, y0);
            const bool changed = k != s_k;
            if (changed) s_I = a.inst[k];
            s_k = k;
            s_x0 = x0;
            s_y0 = y0;
            return changed;
        };
        // the first tile: instance, tables and load offsets are constant data, set up before the wait
        if (tid == 0) {
            s_k = -1;
            if (any) locate(blockIdx.x);
        }
        __syncthreads();
        if (any) ld.init(s_I.nx, s_I.ny, a.pitch, s_x0, s_y0);
        long long rb = (long long)s_I.row0 * a.pitch + GC;
        grid_dependency_wait();
        grid_launch_dependents();
        if (any) ld.load(S, a.phi_in + rb, a.lo_in + rb);
        if (tid == 0) {
            if (any) wait_tables();
            s_time = a.read_n ? a.ctl->time : 0;
            if (s_k >= 0 && a.need_time) {
                s_T[0] = (C)step_T(a.Tf, s_k, s_I, s_time + a.t_off);
                s_T[1] = (C)step_T(a.Tf, a.n_inst + s_k, s_I, s_time + a.t_off + 1);
            }
        }
        __syncthreads();
        n = s_time + a.t_off;
        for (int t = blockIdx.x; t < a.total_tiles && !s_abort; t += stride) {
            if (t != (int)blockIdx.x) {
                __syncthreads();  // the previous tile's shared data are read no more
                if (tid == 0) {
                    pair_fetch_tables<C, P, TX, TY>(S, a.ttabs, t, &s_tbar);
                    if (locate(t) && a.need_time) {
                        s_T[0] = (C)step_T(a.Tf, s_k, s_I, n);
                        s_T[1] = (C)step_T(a.Tf, a.n_inst + s_k, s_I, n + 1);
                    }
                }
                __syncthreads();
                ld.init(s_I.nx, s_I.ny, a.pitch, s_x0, s_y0);
                rb = (long long)s_I.row0 * a.pitch + GC;
                ld.load(S, a.phi_in + rb, a.lo_in + rb);
                if (tid == 0) wait_tables();
                __syncthreads();
                if (s_abort) break;
            }
            pair_steps<C, P, TX, TY, NT>(S, s_I, a.need_time, s_T[0], s_T[1], s_x0, s_y0, a.pitch, rb, a.phi_out, a.lo_out);
        }
    }

    // the last CTA of a batch's last launch advances the step counter (as in the one-step kernels)
    if (a.t_adv && tid == 0) {
        unsigned int prev = atomicAdd(&a.ctl->done, 1u);
        if (prev == gridDim.x - 1) {
            a.ctl->done = 0u;
            a.ctl->time = (a.read_n ? n - a.t_off : a.ctl->time) + a.t_adv;
        }
    }
}

}  // namespace lbch
