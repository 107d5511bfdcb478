// lbch_kernels.cuh -- sm_103a device code of the Cahn-Hilliard lattice Boltzmann step.
//
// Method: Zhang, Guo & Liang, arXiv:1805.00007, Sec. II (Eqs. LB, geq, liangFi, macroscopicg, mu, bulk,
// betakappa, rho, t0-phiu, mark3).  The step is one fused kernel; no tensor cores (a stencil has no contraction).  This file
// holds the arithmetic that every form of the step shares, and the tile kernel.
//
// Storage ("padded image layout").  Every stored row has the same pitch.  An instance occupies
// ny + 2*GR consecutive stored rows; domain node (x, y) sits at stored row row0 + y, column GC + x.  The
// ghost rows and columns around the domain hold copies of the nodes they stand for -- periodic images,
// or mirror images next to walls -- written by the step that produces those nodes, so that the halo of
// every tile is one contiguous box of the stored array.  The populations are interleaved by row:
// g[(row * nq + q) * pitch + col], so one 3-D TMA box (columns x planes x rows) brings a tile's planes.
// phi is a plain 2-D array phi[row * pitch + col].
//
// Per step a persistent CTA walks its tiles (TX x TY output nodes) with a two-stage TMA pipeline:
// while tile k is computed, the population box (tile + 1 halo) and the phi box (tile + 3 halo) of the
// next tile are in flight.  For each tile the CTA
//   1. computes mu = f'(phi) - kappa lap phi and D = div(phi u) on tile + 2 (velocity from per-instance separable tables;
//      stencils column first, in double through column sums in shared memory),
//   2. on tile + 1 computes grad mu, grad D, the force F, g_eq and S and collides, in place in the box,
//   3. pulls g*_i(x - c_i) from shared memory for every tile node (halfway bounce-back at walls) and
//      stores g(t+1) and phi(t+1), with the ghost images the next step's boxes need.
// HBM traffic per lattice update is one read and one write of the stored populations and of phi; the
// overlap of neighbouring tiles' boxes is served from L2.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace lbch {

constexpr int GC = 4;  // ghost columns on each side (keeps box starts 16-byte aligned)
constexpr int GR = 3;  // ghost rows on each side (phi halo of the stencil chain)

// ------------------------------------------------------------------------------------------ lattice
// D2Q9 (Sec. II.B): c0=(0,0), c1=-c3=(1,0), c2=-c4=(0,1), c5=-c7=(1,1), c6=-c8=(-1,1).
__host__ __device__ constexpr int cx(int q) { return (q == 1 || q == 5 || q == 8) ? 1 : ((q == 3 || q == 6 || q == 7) ? -1 : 0); }
__host__ __device__ constexpr int cy(int q) { return (q == 2 || q == 5 || q == 6) ? 1 : ((q == 4 || q == 7 || q == 8) ? -1 : 0); }
__host__ __device__ constexpr int opp(int q) { return q == 0 ? 0 : (q <= 4 ? ((q + 1) % 4) + 1 : ((q - 5 + 2) % 4) + 5); }
// Weights w0 = 4/9, w1..4 = 1/9, w5..8 = 1/36.
template <typename C> __host__ __device__ constexpr C wq(int q) { return q == 0 ? C(4) / C(9) : (q <= 4 ? C(1) / C(9) : C(1) / C(36)); }

enum Vel { VEL_UNIFORM = 0, VEL_ROTATION = 1, VEL_VORTEX = 2, VEL_SHEAR = 3, VEL_REV_SHEAR = 4, VEL_DEFORM = 5 };

// Derived constants of one instance in the arithmetic type of a kernel.
template <typename C>
struct Consts {
    C beta, kappa, eta, a, b, K, phiA, phiB;
    C itau, omt, src;  // 1/tau, 1 - 1/tau, 1 - 1/(2 tau)
    C cF1, cmu;        // Model III: 2 tau - 1 + 3K and 3 c_s^2 eta K, the coefficients of d_t F1 and d_t grad mu
    // Products of the above as the step's per-node arithmetic takes them (formed in double at set-up and rounded
    // once), so that no node multiplies by a constant that another constant could carry:
    C b4, b2s;         // 4 beta and -2 beta (phiA + phiB): f'(phi) = (phi - phiA)(phi - phiB)(b4 phi + b2s)
    C kM;              // (w_5 / tau) eta
    C ra, rb;          // -144 a / src, -144 b / src: 1/(ra phi + rb) = -(3 w_5 src)/(12 rho)
    C Kd;              // 3 w_5 src K / 12
    C k3;              // 3 w_5 src
    C hF, hG;          // Model III: cF1 / k3 and cmu / 12
};

// Per-instance parameters, derived constants and layout, resident in device memory.
struct InstDev {
    int nx, ny;
    int row0;          // stored row of domain row 0 (the instance's first ghost row is row0 - GR)
    int walls, model, vel;
    int ylen;          // length of each Y velocity table: ny rounded up to 16, plus 24 (ghost rows and the
                       // reach of the last tile's slice)
    int tab;           // offset of the velocity tables: X1, X2 [pitch]; Y1/12, Y2/12 [ylen]; W[4]
    int slab;          // a slab of a larger periodic grid: its ghost rows hold the neighbouring slabs' rows
                       // (imported between steps), not images of its own rows
    double Tper;
    Consts<double> cd;  // the constants in double (FP64 path, initial state)
    Consts<float> cf;   // and rounded once to float (float paths)
};

template <typename C> __device__ __forceinline__ const Consts<C>& consts(const InstDev& I);
template <> __device__ __forceinline__ const Consts<double>& consts<double>(const InstDev& I) { return I.cd; }
template <> __device__ __forceinline__ const Consts<float>& consts<float>(const InstDev& I) { return I.cf; }

// Step counter shared by the launches of one handle.  A launch's step is time + its offset; the launch
// that ends a batch (a captured graph of steps, or a single step) advances `time` from its last CTA.
struct Ctl {
    long long time;
    unsigned int done;
    unsigned int err;   // bit 0: a TMA wait timed out
};

// Time factor of the prescribed flows: u(x, y, t) = (X1(x) Y1(y), X2(x) Y2(y)) T(t).  The tables hold Y1/12 and
// Y2/12, and the kernels work with u/12 (node_u), the scale at which the stencils of div(phi u) take it.
__host__ __device__ inline double vel_t(int vel, double Tper, long long n)
{
    const double pi = 3.14159265358979323846;
    switch (vel) {
    case VEL_VORTEX:
    case VEL_DEFORM: return cos(pi * (double)n / Tper);
    case VEL_REV_SHEAR: return ((double)n < Tper) ? 1.0 : -1.0;
    default: return 1.0;
    }
}

// The time factor at step n of instance k: from the launch's table (time_table_kernel) or, without one, formed here.
// cos in double takes one thread about 1.4 us on a GPU with two FP64 lanes per SM, which a block would wait for
// at the head of every launch of a time-dependent flow (512^2 single vortex in float: 11.9 -> 10.9 us per step with
// the table, where the flow without a time factor takes 10.4).
__device__ __forceinline__ double step_T(const double* Tf, int k, const InstDev& I, long long n)
{
    return Tf ? Tf[k] : vel_t(I.vel, I.Tper, n);
}

// Time factors of every instance for `steps` steps from the current one: T[j * n_inst + k] for step time + j.
// One launch ahead of a batch of step launches, all factors side by side (in a graph, its first node).  E counts the
// entries: four million instances make more of them than an int does, and no others pay for a 64-bit division (a single
// step of a 450^2 float handle, table included: 10.8 us per call, 11.2 with it).
constexpr int TIME_NT = 128;
inline unsigned time_table_blocks(int steps, int n_inst) { return (unsigned)(((long long)steps * n_inst + TIME_NT - 1) / TIME_NT); }
template <typename E = long long>
__global__ void time_table_kernel(const InstDev* inst, int n_inst, const Ctl* ctl, int steps, double* T)
{
    const E e = (E)blockIdx.x * TIME_NT + threadIdx.x;
    if (e >= (E)steps * n_inst) return;
    const int j = (int)(e / n_inst), k = (int)(e - (E)j * n_inst);
    T[e] = vel_t(inst[k].vel, inst[k].Tper, ctl->time + j);
}

// ------------------------------------------------------------------------------------------ helpers
template <typename T> __device__ __forceinline__ float to_f(T v) { return (float)v; }
template <> __device__ __forceinline__ float to_f<__half>(__half v) { return __half2float(v); }
template <typename C, typename T> __device__ __forceinline__ C cvt(T v) { return (C)to_f(v); }
template <> __device__ __forceinline__ double cvt<double, double>(double v) { return v; }
template <typename T, typename C> __device__ __forceinline__ T to_s(C v) { return (T)v; }
template <> __device__ __forceinline__ __half to_s<__half, float>(float v) { return __float2half_rn(v); }

template <typename C> __device__ __forceinline__ C rcp(C v);
template <> __device__ __forceinline__ float rcp<float>(float v) { return __frcp_rn(v); }
// double reciprocal: a float seed refined by two Newton-Raphson steps r <- r (2 - v r); the error
// squares at each step (2^-23 -> 2^-46 -> below double rounding)
template <> __device__ __forceinline__ double rcp<double>(double v)
{
    double r = (double)__frcp_rn((float)v);
    r = r * fma(-v, r, 2.0);
    r = r * fma(-v, r, 2.0);
    return r;
}

template <typename C> __device__ __forceinline__ C dfdphi(C phi, C beta, C phiA, C phiB)
{
    // d/dphi of beta (phi - phiA)^2 (phi - phiB)^2 (Eq. bulk)
    return C(2) * beta * (phi - phiA) * (phi - phiB) * (C(2) * phi - phiA - phiB);
}

// The instance owning tile `tile`: tile_begin[k] is the first tile of instance k for the launch's shape.
__device__ __forceinline__ int find_inst(const int* tile_begin, int n_inst, int tile)
{
    int lo = 0, hi = n_inst - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (tile_begin[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int wrap(int i, int n) { i %= n; return i < 0 ? i + n : i; }
__device__ __forceinline__ int mirror(int j, int n)
{
    if (j < 0) j = -1 - j;
    if (j >= n) j = 2 * n - 1 - j;
    return j < 0 ? 0 : (j >= n ? n - 1 : j);
}

// ------------------------------------------------------------------------------------------ per-node arithmetic
// Used by every form of the step kernel (tiles in shared memory; row sweeps in registers; two steps per
// launch), so that every quantity is evaluated by the same operations in all of them.  Every product is an
// explicit rounded multiply or an explicit fused multiply-add: the compiler's own contraction of a*b + c
// depends on how often a product is reused, which differs between the forms, and would change the last bits.
//
// The isotropic nine-point stencils are products of one-dimensional ones, and are evaluated as such: first a few
// values per column from the nodes below, at and above a row, then their combination along the row.  A form
// that holds the column values (the row sweep) forms them once per node, and every constant that another can
// carry is folded into it at set-up.  A node's update at tau_g = 1, Model II, takes 86 operations this way
// in float (37 additions, 17 products, 32 fused multiply-adds, streaming and the float-float sum included) and 81 in double (30, 17
// and 34), and the reciprocal's approximation, where the nine-point forms direction by direction took 149.  The
// FP64 kernels, which the FP64 pipe bounds, and the row sweeps, which instruction issue bounds, gained most
// (us per step before -> after: FP64 500^2 row sweep 147 -> 94, FP64 256^2 two-step kernel 30.6 -> 23.8, float
// 3001 x 1999 row sweep 65.7 -> 53.3, half storage with the populations at 4096^2 267 -> 219; float with the
// populations, near its HBM bound, 297 -> 295), with the same distance from the 64-bit result.
__device__ __forceinline__ float op_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double op_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float op_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double op_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// Reciprocal for the force: the hardware's approximation (within one unit in the last place in float, about 20 bits in
// double) refined once: in float by a Newton-Raphson step r + r e, in double by the third-order step r + r (e + e^2) of the
// same family (Householder's, of order two), e = 1 - v r (2^-20 -> 2^-60).  Within one unit in the last place of the rounded
// quotient for every v whose reciprocal is a normal number, |v| < 2^126 in float and 2^1022 in double; the constants that
// form v are chosen to stay there (derive).  Against the correctly rounded __frcp_rn and 1.0 / v, us per step: FP64
// 256^2 15.8 and 16.6, float 3001 x 1999 32.6 and 34.7, 256^2 2.04 and 2.18, half storage with the populations at 4096^2 136 and 143.
__device__ __forceinline__ float node_rcp(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return op_fma(r, op_fma(-v, r, 1.0f), r);
}
__device__ __forceinline__ double node_rcp(double v)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(v));
    const double e = op_fma(-v, r, 1.0);
    return op_fma(r, op_fma(e, e, e), r);
}

// d/dphi of beta (phi - phiA)^2 (phi - phiB)^2 (Eq. bulk), direction by direction (the coupled flow)
template <typename C> __device__ __forceinline__ C node_dfdphi(C phi, C beta, C phiA, C phiB)
{
    const C s = op_fma(C(2), phi, -phiA) - phiB;
    return op_mul(op_mul(op_mul(op_mul(C(2), beta), phi - phiA), phi - phiB), s);
}

// Column values of phi for the Laplacian: dl = the second difference along y, and z = phi + dl/6.  The isotropic
// Laplacian sum_k 2 w_k (psi(x + c_k) - psi(x)) / c_s^2 is dl + (z(E) - 2 z + z(W)).
template <typename C> __device__ __forceinline__ C node_z(C pS, C ce, C pN, C& dl)
{
    dl = op_fma(C(-2), ce, pN + pS);
    return op_fma(C(1) / C(6), dl, ce);
}

// Eq. mu: mu = f'(phi) - kappa lap phi, with f' of Eq. bulk in its factors
template <typename C> __device__ __forceinline__ C node_mu(C ce, C dl, C z, C zE, C zW, const Consts<C>& K0)
{
    const C lap = dl + op_fma(C(-2), z, zE + zW);
    const C f1 = op_mul(op_mul(ce - K0.phiA, ce - K0.phiB), op_fma(K0.b4, ce, K0.b2s));
    return op_fma(-K0.kappa, lap, f1);
}

// Column values of the flux phi u for D = div(phi u) = sum_k w_k c_k . (phi u)(x + c_k) / c_s^2 in the separable flow
// u = (X1 Y1, X2 Y2) T: with y1 = Y1 T/12, y2 = Y2 T/12 of the rows below (S), at (y14 = 4 y1) and above (N), the
// column's share in D of the node to its west is E, to its east W, and of its own node 4 d.
template <typename C>
__device__ __forceinline__ C node_flux(C pS, C ce, C pN, C X1, C X2, C y1S, C y14, C y1N, C y2S, C y2N, C& E, C& W)
{
    const C t = op_fma(y1N, pN, op_fma(y1S, pS, op_mul(y14, ce)));
    const C d = op_mul(X2, op_fma(y2N, pN, -op_mul(y2S, pS)));
    E = op_fma(X1, t, d);
    W = op_fma(-X1, t, d);
    return d;
}
// ... its own node's alone
template <typename C> __device__ __forceinline__ C node_flux_d(C pS, C pN, C X2, C y2S, C y2N)
{
    return op_mul(X2, op_fma(y2N, pN, -op_mul(y2S, pS)));
}
// D from the node's own d, the E of the column to its east and the W of the column to its west
template <typename C> __device__ __forceinline__ C node_div(C d, C E, C W) { return op_fma(C(4), d, E + W); }

// Column values of a field for the isotropic gradient sum_k w_k c_k psi(x + c_k) / c_s^2 = (gx, gy)/12:
// w = psi(S) + 4 psi + psi(N) and d = psi(N) - psi(S); gx = w(E) - w(W), gy = d(E) + 4 d + d(W).
template <typename C> __device__ __forceinline__ C node_w(C s, C c, C n) { return op_fma(C(4), c, n + s); }
template <typename C> __device__ __forceinline__ C node_gy(C dW, C d, C dE) { return op_fma(C(4), d, dE + dW); }

// The same from the nine values of a node's neighbourhood (the forms that hold fields in shared memory).
template <typename C>
__device__ __forceinline__ C mu9(C ce, C pE, C pW, C pN, C pS, C pNE, C pNW, C pSE, C pSW, const Consts<C>& K0)
{
    C dl, dE, dW;
    const C z = node_z(pS, ce, pN, dl), zE = node_z(pSE, pE, pNE, dE), zW = node_z(pSW, pW, pNW, dW);
    return node_mu(ce, dl, z, zE, zW, K0);
}
// x1*, x2*: the X tables at the columns W, (C), E; y1*, y2*: the Y tables (times T) at the rows S, (C), N
template <typename C>
__device__ __forceinline__ C div9(C pE, C pW, C pN, C pS, C pNE, C pNW, C pSE, C pSW, C x1W, C x1E, C x2W, C x2C,
                                  C x2E, C y1S, C y1C, C y1N, C y2S, C y2N)
{
    const C y14 = op_mul(C(4), y1C);
    C EE, WE, EW, WW;
    node_flux(pSE, pE, pNE, x1E, x2E, y1S, y14, y1N, y2S, y2N, EE, WE);
    node_flux(pSW, pW, pNW, x1W, x2W, y1S, y14, y1N, y2S, y2N, EW, WW);
    return node_div(node_flux_d(pS, pN, x2C, y2S, y2N), EE, WW);
}
template <typename C>
__device__ __forceinline__ void grad9(C E, C W, C N, C S, C NE, C NW, C SE, C SW, C& gx, C& gy)
{
    gx = node_w(SE, E, NE) - node_w(SW, W, NW);
    gy = node_gy(NW - SW, N - S, NE - SE);
}

// The prescribed velocity over 12 at a node, X(x) y(y) with y = (Y/12) T.
template <typename C> __device__ __forceinline__ C node_u(C X, C y) { return op_mul(X, y); }
// ... and at a wall (the tables' W entries hold Y itself there)
template <typename C> __device__ __forceinline__ C wall_u(C X, C W, C T) { return op_mul(X, op_mul(W, T)); }

// 1/tau phi u, the momentum part of g_eq in the scale of the diagonal directions: 3 w_5 / tau phi u = 1/tau phi (u/12)
template <typename C>
__device__ __forceinline__ void node_flow(C ph, C ux, C uy, const Consts<C>& K0, C& Px, C& Py)
{
    const C pk = op_mul(K0.itau, ph);
    Px = op_mul(pk, ux);
    Py = op_mul(pk, uy);
}

// The part of g_eq / tau + (1 - 1/(2 tau)) S odd in c_i, in the scale of the diagonal directions: J = 3 w_5 (phi u/tau +
// (1 - 1/(2 tau)) F).  F1 = (phi / rho)(-phi grad mu) with rho = a phi + b (Eq. liangFi, with grad p = 0), plus
// F2 = 3 c_s^2 K grad(div(phi u)) for Model II (Eq. mark3).  gm, gD: 12 grad mu, 12 grad D.
template <typename C>
__device__ __forceinline__ void node_force(C ph, C gmx, C gmy, C gDx, C gDy, C Px, C Py, bool model2,
                                           const Consts<C>& K0, C& Jx, C& Jy)
{
    const C fct = op_mul(op_mul(ph, ph), node_rcp(op_fma(K0.ra, ph, K0.rb)));
    Jx = Px;
    Jy = Py;
    if (model2) {
        Jx = op_fma(K0.Kd, gDx, Jx);
        Jy = op_fma(K0.Kd, gDy, Jy);
    }
    Jx = op_fma(fct, gmx, Jx);
    Jy = op_fma(fct, gmy, Jy);
}

// Model III: the complete diffusive-scale force of Eq. F2-1, with the time derivatives on the convective
// scale replaced by backward differences over one step (Remarks I, II).  H = cF1 F1 + cmu grad mu is the
// part under the time derivative; F = F1 + (H - Hprev) + 3 c_s^2 K grad D.  Hprev = H at the first step.
template <typename C>
__device__ __forceinline__ void node_force_full(C ph, C gmx, C gmy, C gDx, C gDy, C Hpx, C Hpy, bool first, C Px, C Py,
                                                const Consts<C>& K0, C& Jx, C& Jy, C& Hx, C& Hy)
{
    const C fct = op_mul(op_mul(ph, ph), node_rcp(op_fma(K0.ra, ph, K0.rb)));
    Hx = op_fma(K0.hF, op_mul(fct, gmx), op_mul(K0.hG, gmx));
    Hy = op_fma(K0.hF, op_mul(fct, gmy), op_mul(K0.hG, gmy));
    const C dHx = first ? C(0) : Hx - Hpx, dHy = first ? C(0) : Hy - Hpy;
    Jx = op_fma(fct, gmx, op_fma(K0.k3, dHx, op_fma(K0.Kd, gDx, Px)));
    Jy = op_fma(fct, gmy, op_fma(K0.k3, dHy, op_fma(K0.Kd, gDy, Py)));
}

// Eq. LB as g* = (1 - 1/tau) g + g_eq / tau + (1 - 1/(2 tau)) S, with Eq. geq and the source
// S_i = w_i c_i . F / c_s^2 (Eq. liangFi), split into the parts even and odd in c_i (J, node_force).  ux, uy:
// u/12; Px, Py: node_flow.  The rest population leaves out phi/tau (it is carried as g_0 - phi in the float
// paths; rest_add puts it back in double).  Everything is formed in the scale of the diagonal directions
// (w_5 = w_1/4); q = 0: the full value.  With QUARTER (tau_g = 1, where the populations are not read) the axis
// directions 1..4 are returned in that scale, a quarter of g*, for stream_sum_q to multiply in its sums;
// otherwise every g* is returned in full, with the same bits (a multiplication by 4 is exact).
template <typename C, bool QUARTER>
__device__ __forceinline__ void collide9(C mu, C ux, C uy, C Px, C Py, C Jx, C Jy, const C* g, const Consts<C>& K0, C* post)
{
    const C M = op_mul(K0.kM, mu);
    const C tx = op_mul(Px, ux), ty = op_mul(Py, uy), r = op_mul(Px, uy);
    const C s = tx + ty;
    const C e = op_fma(C(-6), s, M), Ad = op_fma(C(12), s, M);
    // pairs (q, opp q): (1,3) c=(1,0); (2,4) c=(0,1); (5,7) c=(1,1); (6,8) c=(-1,1)
    const C A1 = op_fma(C(18), tx, e), A2 = op_fma(C(18), ty, e);
    const C A5 = op_fma(C(36), r, Ad), A6 = op_fma(C(-36), r, Ad);
    const C J5 = Jx + Jy, J6 = Jy - Jx;
    const C g0 = op_fma(C(-96), s, op_mul(C(-20), M));
    if constexpr (QUARTER) {
        post[0] = g0;
        post[1] = A1 + Jx; post[3] = A1 - Jx;
        post[2] = A2 + Jy; post[4] = A2 - Jy;
        post[5] = A5 + J5; post[7] = A5 - J5;
        post[6] = A6 + J6; post[8] = A6 - J6;
    } else {
        const C omt = K0.omt;
        post[0] = op_fma(omt, g[0], g0);
        post[1] = op_fma(omt, g[1], op_mul(C(4), A1 + Jx)); post[3] = op_fma(omt, g[3], op_mul(C(4), A1 - Jx));
        post[2] = op_fma(omt, g[2], op_mul(C(4), A2 + Jy)); post[4] = op_fma(omt, g[4], op_mul(C(4), A2 - Jy));
        post[5] = op_fma(omt, g[5], A5 + J5); post[7] = op_fma(omt, g[7], A5 - J5);
        post[6] = op_fma(omt, g[6], A6 + J6); post[8] = op_fma(omt, g[8], A6 - J6);
    }
}

// The rest population of the double path from collide9's: phi/tau added
template <typename C> __device__ __forceinline__ C rest_add(C g0, C ph, const Consts<C>& K0) { return op_fma(K0.itau, ph, g0); }

// Halfway bounce-back at a wall node: g_q arriving from the ghost row is the node's own post-collision
// g_opp(q) plus the moving-wall term 2 w_q phi (c_q . u_w) / c_s^2.
template <typename C, int q>
__device__ __forceinline__ C bounce(C post_opp, C ph, C uwx, C uwy)
{
    const C cuw = cx(q) == 0 ? (cy(q) > 0 ? uwy : -uwy)
                : (cy(q) == 0 ? (cx(q) > 0 ? uwx : -uwx)
                : (cx(q) > 0 ? (cy(q) > 0 ? uwx + uwy : uwx - uwy) : (cy(q) > 0 ? uwy - uwx : -(uwx + uwy))));
    const C g = op_fma(op_mul(C(6) * wq<C>(q), ph), cuw, post_opp);
    // 2 and 4 pass through a quarter, as which the sums at tau_g = 1 carry them: the same bits in every form, down to
    // the smallest numbers
    return q == 2 || q == 4 ? op_mul(C(4), op_mul(C(0.25), g)) : g;
}

// Sum of the streamed populations g_1..g_8(t+1) at a node, grouped by the column they come from: the
// three from x - 1 (1, 5, 8), the two from x (2, 4), the three from x + 1 (3, 6, 7).
template <typename C>
__device__ __forceinline__ C stream_sum(C v1, C v2, C v3, C v4, C v5, C v6, C v7, C v8)
{
    return (((v1 + v5) + v8) + (v2 + v4)) + ((v3 + v6) + v7);
}
// The same with 1..4 in a quarter (collide9's QUARTER): the same bits, since multiplications by 4 are exact
template <typename C>
__device__ __forceinline__ C stream_sum_q(C v1, C v2, C v3, C v4, C v5, C v6, C v7, C v8)
{
    const C R = op_fma(C(4), v1, v5) + v8, L = op_fma(C(4), v3, v6) + v7;
    return op_fma(C(4), v2 + v4, R) + L;
}

// ------------------------------------------------------------------------------------------ TMA / mbarrier
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// The dynamic shared memory of a kernel from its first 128-byte boundary.  The offset is added to the shared
// array itself (not formed by a round trip through an integer address), so the compiler still knows every
// pointer derived from it addresses shared memory and issues shared-memory loads and stores rather than
// generic ones.
__device__ __forceinline__ unsigned char* smem_aligned128(unsigned char* raw)
{
    return raw + ((128u - (unsigned)(reinterpret_cast<uintptr_t>(raw) & 127u)) & 127u);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: gives up after `limit` polls (each poll may suspend the thread for a short while, 3.7 us as measured: WAIT_POLLS
// run out after a second, where a copy takes microseconds).
constexpr unsigned WAIT_POLLS = 1u << 18;
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned parity, unsigned limit)
{
    for (unsigned k = 0; k < limit; k++)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
// programmatic dependent launch: wait for the prerequisite grid to complete with its writes visible (a
// no-op without a programmatic dependency), and allow the dependent grid to be scheduled
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, int c0, int c1, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(smem_u32(dst)), "l"(tm), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

// plain bulk copy (not tensor-mapped): 16-byte aligned source and destination, size a multiple of 16
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, int c0, int c1, int c2, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
            "r"(smem_u32(dst)), "l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

// f(xx, yy) for the ghost cells that stand for domain node (x, y): periodic images in x; periodic or (walls) mirror images in
// y, three deep.  A node has at most one image along each axis unless the domain is narrower than six nodes.  (Straight-line
// code: a tile on the edge sets the time of a launch of one tile per SM, and as a loop over all images that a node can have
// these tests were 1 to 5 % of a step on grids of 45 to 1024 squared.)
template <typename F>
__device__ __forceinline__ void for_images3(int x, int y, int nx, int ny, int walls, F&& f)
{
    const int xa = x < 3 ? x + nx : x >= nx - 3 ? x - nx : x;
    const int ya = y < 3 ? (walls ? -1 - y : y + ny) : y >= ny - 3 ? (walls ? 2 * ny - 1 - y : y - ny) : y;
    if (xa != x) f(xa, y);
    if (ya != y) {
        f(x, ya);
        if (xa != x) f(xa, ya);
    }
    if (nx >= 6 && ny >= 6) return;
    const int xb = x < 3 && x >= nx - 3 ? x - nx : x;  // the second image along an axis
    const int yb = y < 3 && y >= ny - 3 ? (walls ? 2 * ny - 1 - y : y - ny) : y;
    if (xb != x) {
        f(xb, y);
        if (ya != y) f(xb, ya);
    }
    if (yb != y) {
        f(x, yb);
        if (xa != x) f(xa, yb);
        if (xb != x) f(xb, yb);
    }
}

// The same one deep, for the populations: periodic images in x, and in y unless the instance has walls there.
template <typename F>
__device__ __forceinline__ void for_images1(int x, int y, int nx, int ny, int walls, F&& f)
{
    const int xa = x == 0 ? nx : x == nx - 1 ? -1 : x;
    const int ya = walls ? y : y == 0 ? ny : y == ny - 1 ? -1 : y;
    if (xa != x) f(xa, y);
    if (ya != y) {
        f(x, ya);
        if (xa != x) f(xa, ya);
    }
}

// Model III: H(t) of domain node (x, y) and its ghost images one deep (periodic in x; in y unless walls).
template <typename C>
__device__ __forceinline__ void store_h(C* H, long long plane, int row0, int pitch, int nx, int ny, int walls, int x,
                                        int y, C hx, C hy)
{
    const int xa = x == 0 ? nx : (x == nx - 1 ? -1 : x);
    const int ya = walls ? y : (y == 0 ? ny : (y == ny - 1 ? -1 : y));
    for (int iy = 0; iy < 2; iy++) {
        const int yy = iy == 0 ? y : ya;
        if (iy == 1 && yy == y) continue;
        for (int ix = 0; ix < 2; ix++) {
            const int xx = ix == 0 ? x : xa;
            if (ix == 1 && xx == x) continue;
            const long long k = (long long)(row0 + yy) * pitch + GC + xx;
            H[k] = hx;
            H[plane + k] = hy;
        }
    }
}

// The nodes of a W x H region that the CTA's NT threads take in one phase, consecutive threads consecutive nodes:
// f(e, r, c) for node e = r W + c.
template <int W, int H, int NT, typename F>
__device__ __forceinline__ void for_region(F&& f)
{
    for (int i = threadIdx.x; i < H * W; i += NT) {
        const int r = i / W;
        f(i, r, i - r * W);
    }
}

// ------------------------------------------------------------------------------------------ step
// Storage types: S populations, P phi (the high part on the float path), C arithmetic.  The float path
// (C = S = float) keeps phi as an unevaluated sum of two floats, phi = hi + lo: hi feeds the stencils,
// lo is carried only at the node, and phi(t+1) = phi(t) + increment is formed with an exact TwoSum.
template <typename C, typename S, typename P>
struct StepArgs {
    const InstDev* inst;
    const int* tile_begin;  // first tile of each instance for this launch's tile shape
    const C* tabs;       // velocity tables of all instances, indexed by stored column / instance row
    int n_inst;
    int total_tiles;
    int pitch;           // elements per stored row
    int debug_skip;      // test hook: when nonzero, CTA 0 never issues its first load (its wait runs out)
    S* g_out;
    P* phi_out;
    float* lo_out;       // low part of phi on the float path
    Ctl* ctl;
    const C* H_in;       // Model III: H(t - 1), two planes (x, y) of rows x pitch values; nullptr otherwise
    C* H_out;            // H(t), written for the tile's own nodes and their ghost images
    long long H_plane;   // values per plane of H
    int t_off;           // this launch's step is ctl->time + t_off
    int t_adv;           // when nonzero, the launch's last CTA advances ctl->time by t_adv
    int need_time;       // some instance's step depends on the step index (a time-dependent flow or Model III)
    int read_n;          // ... and the launch reads the index: Model III, or a time factor without a table
    const double* Tf;    // the instances' time factors at this launch's step, or null (see step_T)
};

template <typename C, typename S, typename P, int TX, int TY>
struct StepShape {
    static constexpr bool FF = sizeof(C) == 4 && sizeof(S) == 4;  // float-float phi
    static constexpr int NQ = (sizeof(S) == 2) ? 8 : 9;        // stored planes
    static constexpr int BW = TX + 8;                          // box width (x0-4 .. x0+TX+3)
    static constexpr int GBH = TY + 2, PBH = TY + 6;           // box heights
    static constexpr int PW = TX + 6, PH = TY + 6;             // tile + 3
    static constexpr int MW = TX + 4, MH = TY + 4;             // tile + 2
    static constexpr int GW = TX + 2, GH = TY + 2;             // tile + 1
    static constexpr int NP = PW * PH, NM = MW * MH, NG = GW * GH;  // region sizes
    static constexpr unsigned GBOX_BYTES = GBH * NQ * BW * sizeof(S);
    static constexpr unsigned PBOX_BYTES = PBH * BW * sizeof(P);
    static constexpr unsigned LBOX_BYTES = FF ? TX * TY * 4 : 0;
    // velocity-table slices of the tile: X1, X2 over the box columns, Y1, Y2 over TY + 8 rows
    static constexpr int YT = TY + 8;
    static constexpr unsigned XT_BYTES = BW * sizeof(C), YT_BYTES = YT * sizeof(C);
    static constexpr unsigned TAB_BYTES = 2 * XT_BYTES + 2 * YT_BYTES;
    __host__ __device__ static constexpr size_t a128(size_t b) { return (b + 127) / 128 * 128; }
    static constexpr size_t OFF_P = a128(GBOX_BYTES), OFF_L = OFF_P + a128(PBOX_BYTES);
    static constexpr size_t OFF_T = OFF_L + a128(LBOX_BYTES);
    static constexpr size_t STAGE = OFF_T + a128(TAB_BYTES);
    // the column passes of the double path: five column values of phi on tile + 3 by tile + 2 rows (then four of mu and D)
    static constexpr int AW = TX + 6, AN = AW * MH;
    static constexpr bool COLS = sizeof(C) == 8;
    static constexpr size_t OFF_COLS = a128(sizeof(C) * (2 * NM));
    static constexpr size_t WORK1 = OFF_COLS + (COLS ? a128(sizeof(C) * (5 * AN)) : 0);
    static constexpr size_t WORK = WORK1 + (sizeof(S) == 2 ? a128(sizeof(C) * NG) : 0);  // + h*_0 (half path)
    static constexpr size_t BYTES = 2 * STAGE + WORK + 128 + 128;  // mbarriers, alignment slack
};

// TAU1: the kernel for instances that all have tau_g = 1.  Then Eq. LB gives g* = g_eq + S/2: the
// populations are multiplied by 1 - 1/tau = 0, so they are neither loaded nor stored -- the state is phi
// alone, and the result is bit for bit the general kernel's (which multiplies them by exactly zero).
template <typename C, typename S, typename P, int TX, int TY, int NT, bool TAU1 = false>
__global__ void __launch_bounds__(NT, NT >= 512 ? 1 : (sizeof(C) == 8 ? 2 : 3)) ch_step_kernel(const __grid_constant__ CUtensorMap tm_g,
                                                     const __grid_constant__ CUtensorMap tm_phi,
                                                     const __grid_constant__ CUtensorMap tm_lo,
                                                     StepArgs<C, S, P> a)
{
    using L = StepShape<C, S, P, TX, TY>;
    constexpr int NQ = L::NQ, BW = L::BW, MW = L::MW, MH = L::MH, GW = L::GW;
    constexpr bool kHalf = sizeof(S) == 2;    // g_0 not stored: implied by phi
    constexpr bool kShift = sizeof(C) == 4;   // float arithmetic on g_0 - phi instead of g_0
    constexpr bool kFF = L::FF;
    constexpr int QOFF = kHalf ? 1 : 0;       // stored plane of population q is q - QOFF
    // at tau_g = 1 the axis populations are staged in a quarter (collide9); not where they round to half
    constexpr bool kQuarter = TAU1 && !kHalf;

    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_aligned128(smem_raw);
    auto stage = [&](int k) { return base + (size_t)k * L::STAGE; };
    C* s_mu = reinterpret_cast<C*>(base + 2 * L::STAGE);
    C* s_D = s_mu + L::NM;
    C* s_h0 = reinterpret_cast<C*>(base + 2 * L::STAGE + L::WORK1);
    uint64_t* mbar = reinterpret_cast<uint64_t*>(base + 2 * L::STAGE + L::WORK);

    __shared__ long long s_time;
    __shared__ int s_tile_inst;
    __shared__ int3 s_info[2];  // (instance, x0, y0) of the tile in each stage, written when it is issued
    __shared__ C s_T;
    __shared__ InstDev s_I;  // the current tile's instance, copied when the instance changes

    const int tid = threadIdx.x;
    const int stride = gridDim.x;
    if (tid == 0) {
        mbar_init(&mbar[0], 1);
        mbar_init(&mbar[1], 1);
        fence_mbar_init();
        s_tile_inst = -1;
        if ((int)blockIdx.x < a.total_tiles) {  // instance data are constant: read before the dependency wait
            const int k = find_inst(a.tile_begin, a.n_inst, blockIdx.x);
            s_I = a.inst[k];
            s_tile_inst = k;
        }
    }

    // producer: thread 0 issues the boxes of tile t into stage s
    auto issue = [&](int t, int s) {
        int k = find_inst(a.tile_begin, a.n_inst, t);
        const InstDev& I = a.inst[k];
        int local = t - a.tile_begin[k];
        int tiles_x = (I.nx + TX - 1) / TX;
        int x0 = (local % tiles_x) * TX, y0 = (local / tiles_x) * TY;
        s_info[s] = make_int3(k, x0, y0);
        fence_proxy_async();
        mbar_expect_tx(&mbar[s], (TAU1 ? 0u : L::GBOX_BYTES) + L::PBOX_BYTES + L::LBOX_BYTES + L::TAB_BYTES);
        // box column origin: domain x0 - 4 is stored column x0 - 4 + GC = x0
        if (!TAU1) tma_load_3d(stage(s), &tm_g, x0, 0, I.row0 + y0 - 1, &mbar[s]);
        tma_load_2d(stage(s) + L::OFF_P, &tm_phi, x0, I.row0 + y0 - 3, &mbar[s]);
        if (kFF) tma_load_2d(stage(s) + L::OFF_L, &tm_lo, x0 + GC, I.row0 + y0, &mbar[s]);
        // the velocity tables of the box's columns and rows (the Y tables start at the box's first row)
        const C* tX1 = a.tabs + I.tab;
        const C* tY1 = tX1 + 2 * a.pitch;
        unsigned char* tb = stage(s) + L::OFF_T;
        bulk_load(tb, tX1 + x0, L::XT_BYTES, &mbar[s]);
        bulk_load(tb + L::XT_BYTES, tX1 + a.pitch + x0, L::XT_BYTES, &mbar[s]);
        bulk_load(tb + 2 * L::XT_BYTES, tY1 + y0, L::YT_BYTES, &mbar[s]);
        bulk_load(tb + 2 * L::XT_BYTES + L::YT_BYTES, tY1 + I.ylen + y0, L::YT_BYTES, &mbar[s]);
    };

    // Launched as a programmatic dependent of the previous step: everything above overlaps its tail;
    // nothing it writes (phi, g, the step counter) is touched before this wait.  The first boxes are
    // issued before the counter is read, so the two latencies overlap.
    grid_dependency_wait();
    grid_launch_dependents();
    if (tid == 0) {
        for (int j = 0; j < 2; j++) {
            int t = blockIdx.x + j * stride;
            if (t < a.total_tiles && !(a.debug_skip && blockIdx.x == 0 && j == 0)) issue(t, j);
        }
        // the counter is read only when the launch needs the step index; otherwise nothing waits on that load
        s_time = a.read_n ? a.ctl->time : 0;
        if (s_tile_inst >= 0) s_T = a.need_time ? (C)step_T(a.Tf, s_tile_inst, s_I, s_time + a.t_off) : C(1);
    }
    __syncthreads();
    const long long n = s_time + a.t_off;
    int cur_inst = s_tile_inst;  // the instance in s_I (a register copy, so that no thread races thread 0)

    for (int it = 0;; it++) {
        const int t = blockIdx.x + it * stride;
        if (t >= a.total_tiles) break;
        const int s = it & 1;
        // every thread observes the completion of the stage's copies itself (bounded wait)
        bool ok = mbar_wait_bounded(&mbar[s], (unsigned)((it >> 1) & 1), WAIT_POLLS);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                atomicOr(&a.ctl->err, 1u);
                // let a copy already issued into the other stage land before the CTA exits (bounded)
                if (t + stride < a.total_tiles)
                    mbar_wait_bounded(&mbar[s ^ 1], (unsigned)(((it + 1) >> 1) & 1), WAIT_POLLS);
            }
            break;  // skip the remaining tiles; the step counter below is still kept consistent
        }
        if (s_info[s].x != cur_inst) {  // uniform: a tile of another instance (never the first tile)
            cur_inst = s_info[s].x;
            if (tid == 0) {
                s_I = a.inst[cur_inst];
                s_tile_inst = cur_inst;
                s_T = a.need_time ? (C)step_T(a.Tf, cur_inst, s_I, n) : C(1);  // time factor of the flow, once per instance
            }
            __syncthreads();
        }
        const InstDev& I = s_I;
        const Consts<C>& K0 = consts<C>(I);
        const int nx = I.nx, ny = I.ny, walls = I.walls, model = I.model;
        const int x0 = s_info[s].y, y0 = s_info[s].z;
        const C T = s_T;
        S* gb = reinterpret_cast<S*>(stage(s));
        const P* pb = reinterpret_cast<const P*>(stage(s) + L::OFF_P);  // phi on tile + 3 at box column c + 1
        // velocity tables: X by stored column, Y by row of the instance's stored band
        const C* tX1 = a.tabs + I.tab;
        const C* tX2 = tX1 + a.pitch;
        const C* tY1 = tX2 + a.pitch;
        const C* tY2 = tY1 + I.ylen;
        const C* tW = tY2 + I.ylen;

        // the velocity-table slices arrived with the boxes: X by box column, Y/12 by box row, multiplied here by
        // the time factor (1 for the flows without one); u/12 at box (row, col) is (X1[col] Y1[row], X2[col] Y2[row])
        const C* sX1 = reinterpret_cast<const C*>(stage(s) + L::OFF_T);
        const C* sX2 = sX1 + BW;
        const C* sY1 = sX2 + BW;
        const C* sY2 = sY1 + L::YT;
        if (a.need_time) {
            C* sY = const_cast<C*>(sY1);
            for (int e = tid; e < 2 * L::YT; e += NT) sY[e] = op_mul(sY[e], T);
            __syncthreads();
        }

        // 2. mu (Eq. mu) and D = div(phi u) on tile + 2
        // In double the stencils go through shared memory column first (lbch_kernels.cuh, per-node arithmetic): a pass for
        // the column values, then one along the rows, for phi and again for mu and D.  Two more barriers, but no
        // column value is formed three times, and it is the FP64 pipe that bounds these kernels (32 x 14
        // tiles at 256^2: 19.7 -> 16.0 us per step, 500^2 74.3 -> 59.3, about three quarters of the pipe's rate).
        // In float, where latency does, every thread forms what it needs from the nine neighbours.
        C* s_z = s_mu + L::OFF_COLS / sizeof(C);
        if constexpr (L::COLS) {
            constexpr int AW = L::AW, AN = L::AN;
            for_region<AW, MH, NT>([&](int e, int r, int c) {
                const P* q = pb + (r + 1) * BW + c + 1;
                const C pS = cvt<C>(q[-BW]), ce = cvt<C>(q[0]), pN = cvt<C>(q[BW]);
                C dl;
                s_z[e] = node_z(pS, ce, pN, dl);
                s_z[AN + e] = dl;
                if (model >= 2) {
                    C E, W;
                    s_z[2 * AN + e] = node_flux(pS, ce, pN, sX1[c + 1], sX2[c + 1], sY1[r], op_mul(C(4), sY1[r + 1]), sY1[r + 2],
                                                sY2[r], sY2[r + 2], E, W);
                    s_z[3 * AN + e] = E;
                    s_z[4 * AN + e] = W;
                }
            });
            __syncthreads();
            for_region<MW, L::MH, NT>([&](int e, int r, int c) {
                const int k = r * AW + c + 1;
                s_mu[e] = node_mu(cvt<C>(pb[(r + 1) * BW + c + 2]), s_z[AN + k], s_z[k], s_z[k + 1], s_z[k - 1], K0);
                if (model >= 2) s_D[e] = node_div(s_z[2 * AN + k], s_z[3 * AN + k + 1], s_z[4 * AN + k - 1]);
            });
        } else
        for_region<MW, L::MH, NT>([&](int e, int r, int c) {
            const P* q = pb + (r + 1) * BW + c + 2;
            C ce = cvt<C>(q[0]);
            C pE = cvt<C>(q[1]), pW = cvt<C>(q[-1]), pN = cvt<C>(q[BW]), pS = cvt<C>(q[-BW]);
            C pNE = cvt<C>(q[BW + 1]), pNW = cvt<C>(q[BW - 1]), pSE = cvt<C>(q[-BW + 1]), pSW = cvt<C>(q[-BW - 1]);
            s_mu[e] = mu9(ce, pE, pW, pN, pS, pNE, pNW, pSE, pSW, K0);
            if (model >= 2)  // the tables at box columns c+1..c+3 and box rows r..r+2
                s_D[e] = div9(pE, pW, pN, pS, pNE, pNW, pSE, pSW, sX1[c + 1], sX1[c + 3], sX2[c + 1], sX2[c + 2],
                              sX2[c + 3], sY1[r], sY1[r + 1], sY1[r + 2], sY2[r], sY2[r + 2]);
        });
        if (walls && (y0 < 2 || y0 + TY + 2 > ny)) {
            // every stencil operand takes at a ghost row the value at the mirror row: mu and D at rows
            // -2, -1, ny, ny+1 are copied from rows 1, 0, ny-1, ny-2 (interior rows, as ny >= 4)
            __syncthreads();
            for (int e = tid; e < 4 * MW; e += NT) {
                int k = e / MW, c = e - k * MW;
                int gy = (k == 0) ? -2 : (k == 1) ? -1 : (k == 2) ? ny : ny + 1;
                int r = gy - (y0 - 2);
                int rm = (gy < 0 ? -1 - gy : 2 * ny - 1 - gy) - (y0 - 2);
                if (r >= 0 && r < MH && rm >= 0 && rm < MH) {
                    C vmu = s_mu[rm * MW + c], vD = s_D[rm * MW + c];
                    s_mu[r * MW + c] = vmu;
                    if (model >= 2) s_D[r * MW + c] = vD;
                }
            }
        }
        __syncthreads();

        // the column values of mu and D (in the place of phi's)
        constexpr int CN = MW * L::GH;
        if constexpr (L::COLS) {
            for_region<MW, L::GH, NT>([&](int e, int r, int c) {
                const C mS = s_mu[e], mN = s_mu[e + 2 * MW];
                s_z[e] = node_w(mS, s_mu[e + MW], mN);
                s_z[CN + e] = mN - mS;
                if (model >= 2) {
                    const C dS = s_D[e], dN = s_D[e + 2 * MW];
                    s_z[2 * CN + e] = node_w(dS, s_D[e + MW], dN);
                    s_z[3 * CN + e] = dN - dS;
                }
            });
            __syncthreads();
        }

        // 3. force, equilibrium, source and collision on tile + 1, written back into the box
        for_region<GW, L::GH, NT>([&](int e, int r, int c) {
            int gy = y0 - 1 + r;
            if (walls && (gy < 0 || gy >= ny)) return;  // ghost rows: never pulled (bounce-back)
            int m = (r + 1) * MW + (c + 1);
            C gmx, gmy, gDx = C(0), gDy = C(0);
            if constexpr (L::COLS) {
                const C* w = s_z + r * MW + c + 1;
                gmx = w[1] - w[-1];
                gmy = node_gy(w[CN - 1], w[CN], w[CN + 1]);
                if (model >= 2) {
                    gDx = w[2 * CN + 1] - w[2 * CN - 1];
                    gDy = node_gy(w[3 * CN - 1], w[3 * CN], w[3 * CN + 1]);
                }
            } else {
                grad9(s_mu[m + 1], s_mu[m - 1], s_mu[m + MW], s_mu[m - MW], s_mu[m + MW + 1], s_mu[m + MW - 1],
                      s_mu[m - MW + 1], s_mu[m - MW - 1], gmx, gmy);
                if (model >= 2)
                    grad9(s_D[m + 1], s_D[m - 1], s_D[m + MW], s_D[m - MW], s_D[m + MW + 1], s_D[m + MW - 1],
                          s_D[m - MW + 1], s_D[m - MW - 1], gDx, gDy);
            }
            C ph = cvt<C>(pb[(r + 2) * BW + c + 3]);
            C mu = s_mu[m];
            const C ux = node_u(sX1[c + 3], sY1[r + 2]), uy = node_u(sX2[c + 3], sY2[r + 2]);  // box row r+2, col c+3
            C Px, Py, Jx, Jy;
            node_flow(ph, ux, uy, K0, Px, Py);
            if (model == 3) {
                // H(t - 1) at this node (halo nodes included: its images are stored one deep); H(t) is
                // stored for the tile's own nodes only
                const int gx = x0 - 1 + c;
                const long long hn = (long long)(I.row0 + gy) * a.pitch + GC + gx;
                const bool first = n == 0;
                const C Hpx = first ? C(0) : a.H_in[hn], Hpy = first ? C(0) : a.H_in[a.H_plane + hn];
                C Hx, Hy;
                node_force_full(ph, gmx, gmy, gDx, gDy, Hpx, Hpy, first, Px, Py, K0, Jx, Jy, Hx, Hy);
                if (r >= 1 && r <= TY && c >= 1 && c <= TX && gx < nx && gy < ny)
                    store_h(a.H_out, a.H_plane, I.row0, a.pitch, nx, ny, walls, gx, gy, Hx, Hy);
            } else {
                node_force(ph, gmx, gmy, gDx, gDy, Px, Py, model == 2, K0, Jx, Jy);
            }
            // the node's populations in the box: row r, plane q - QOFF, column c + 3
            S* gp = gb + (r * NQ) * BW + c + 3;
            C g[9];
            if (TAU1) {
#pragma unroll
                for (int q = 0; q < 9; q++) g[q] = C(0);   // multiplied by 1 - 1/tau = 0 below
            } else if (kHalf) {
                C rest = C(0);
#pragma unroll
                for (int q = 1; q < 9; q++) { g[q] = cvt<C>(gp[(q - QOFF) * BW]); rest += g[q]; }
                g[0] = -rest;  // g_0 - phi
            } else {
#pragma unroll
                for (int q = 0; q < 9; q++) g[q] = cvt<C>(gp[q * BW]);
            }
            C post[9];
            collide9<C, kQuarter>(mu, ux, uy, Px, Py, Jx, Jy, g, K0, post);
            if (!kShift) post[0] = rest_add(post[0], ph, K0);
            if (kHalf) {
                // the rest population takes what the half-rounded moving ones leave of phi (see the row sweep)
                C rest = C(0);
#pragma unroll
                for (int q = 1; q < 9; q++) rest += cvt<C>(to_s<S>(post[q]));
                s_h0[e] = -rest;
            }
#pragma unroll
            for (int q = QOFF; q < 9; q++) gp[(q - QOFF) * BW] = to_s<S>(post[q]);
        });
        __syncthreads();

        // 4. pull streaming from the box, bounce-back at walls; store g(t+1), phi(t+1) and ghost images.
        //    Interior nodes (no wall neighbour, no ghost image) take a straight path without the checks.
        const int pitch = a.pitch;
        const float* lb = reinterpret_cast<const float*>(stage(s) + L::OFF_L);
        for_region<TX, TY, NT>([&](int e, int r, int c) {
            int gx = x0 + c, gy = y0 + r;
            if (gx >= nx || gy >= ny) return;
            const bool wallrow = walls && (gy == 0 || gy == ny - 1);
            const bool edge = gx < 3 || gx >= nx - 3 || gy < 3 || gy >= ny - 3;
            const S* src = gb + ((r + 1) * NQ) * BW + c + 4;   // this node's box position, plane 0
            C v[9];
            v[0] = kHalf ? s_h0[(r + 1) * GW + (c + 1)] : cvt<C>(src[0]);
#pragma unroll
            for (int q = 1; q < 9; q++) v[q] = cvt<C>(src[(-cy(q) * NQ + q - QOFF) * BW - cx(q)]);
            if (wallrow) {
                // populations that would come from a ghost row are bounced back at the node
                const C ph = cvt<C>(pb[(r + 3) * BW + c + 4]);
                constexpr C ax = kQuarter ? C(4) : C(1);  // the staged axis populations in full
                v[1] = op_mul(ax, v[1]); v[2] = op_mul(ax, v[2]); v[3] = op_mul(ax, v[3]); v[4] = op_mul(ax, v[4]);
                if (gy == 0) {
                    const C uwx = wall_u(tX1[gx + GC], tW[0], T), uwy = wall_u(tX2[gx + GC], tW[2], T);
                    v[2] = bounce<C, 2>(op_mul(ax, cvt<C>(src[(4 - QOFF) * BW])), ph, uwx, uwy);
                    v[5] = bounce<C, 5>(cvt<C>(src[(7 - QOFF) * BW]), ph, uwx, uwy);
                    v[6] = bounce<C, 6>(cvt<C>(src[(8 - QOFF) * BW]), ph, uwx, uwy);
                }
                if (gy == ny - 1) {
                    const C uwx = wall_u(tX1[gx + GC], tW[1], T), uwy = wall_u(tX2[gx + GC], tW[3], T);
                    v[4] = bounce<C, 4>(op_mul(ax, cvt<C>(src[(2 - QOFF) * BW])), ph, uwx, uwy);
                    v[7] = bounce<C, 7>(cvt<C>(src[(5 - QOFF) * BW]), ph, uwx, uwy);
                    v[8] = bounce<C, 8>(cvt<C>(src[(6 - QOFF) * BW]), ph, uwx, uwy);
                }
            }
            const C sumq = kQuarter && !wallrow ? stream_sum_q(v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8])
                                                : stream_sum(v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8]);
            P hi;
            float lo = 0.0f;
            if (kFF) {
                // g_0(t+1) = phi(t) + v_0 stays at the node: phi(t+1) = phi(t) + (v_0 + sum_{q>0} g_q(t+1));
                // hi + lo absorbs the increment exactly (TwoSum); g_0 - phi is stored as -sum_{q>0} g_q
                float h = (float)pb[(r + 3) * BW + c + 4];
                float tt = lb[r * TX + c] + (float)(v[0] + sumq);
                float sm = h + tt;
                float bb = sm - h;
                lo = (h - (sm - bb)) + (tt - bb);
                hi = (P)sm;
                v[0] = -sumq;
            } else if (kShift) {
                // half path: phi(t+1) = phi(t) + v_0 + sum_{q>0} g_q(t+1) in float; g_0 stays implied
                hi = (P)((float)pb[(r + 3) * BW + c + 4] + (float)(v[0] + sumq));
            } else {
                hi = (P)(v[0] + sumq);
            }
            const long long node = (long long)(I.row0 + gy) * pitch + GC + gx;
            a.phi_out[node] = hi;
            if (kFF) a.lo_out[node] = lo;
            if (!TAU1) {
                S* o = a.g_out + ((long long)(I.row0 + gy) * NQ) * pitch + GC + gx;
#pragma unroll
                for (int q = QOFF; q < 9; q++) o[(q - QOFF) * pitch] = to_s<S>(v[q]);
            }
            if (edge) {
                // the node's images in the ghost columns/rows (phi three deep, the populations one deep;
                // in y only for periodic y, mirror images next to walls)
                for_images3(gx, gy, nx, ny, walls, [&](int xx, int yy) {
                    a.phi_out[(long long)(I.row0 + yy) * pitch + GC + xx] = hi;
                });
                if (!TAU1)
                    for_images1(gx, gy, nx, ny, walls, [&](int xx, int yy) {
                        S* oi = a.g_out + ((long long)(I.row0 + yy) * NQ) * pitch + GC + xx;
#pragma unroll
                        for (int q = QOFF; q < 9; q++) oi[(q - QOFF) * pitch] = to_s<S>(v[q]);
                    });
            }
        });
        // the stage takes the tile after next once every thread is done with it (the next iteration's
        // wait is a barrier too, so without a tile to issue nothing needs to wait here)
        const int t2 = t + 2 * stride;
        if (t2 < a.total_tiles) {
            __syncthreads();
            if (tid == 0) issue(t2, s);
        }
    }

    // the last CTA of a batch's last launch advances the step counter read by the next launch.  No
    // fence: the counter orders no other data, every CTA read the time before its increment, and the next
    // launch reads it only after this grid has completed (kernel boundary or the dependency wait).
    if (a.t_adv && tid == 0) {
        unsigned int prev = atomicAdd(&a.ctl->done, 1u);
        if (prev == gridDim.x - 1) {
            a.ctl->done = 0u;
            a.ctl->time = (a.read_n ? n - a.t_off : a.ctl->time) + a.t_adv;
        }
    }
}

// ------------------------------------------------------------------------------------------ init
// g_i(x, 0) = g_i^eq(phi0, mu(phi0), u(x, 0)); phi(0) = phi0 (hi + lo on the float path); the ghost
// images are written too.  phi0 arrives in the padded layout with its ghost frame filled; the
// velocity tables are the double ones, indexed like the step kernel's.
template <typename C, typename S, typename P>
__global__ void init_kernel(const InstDev* inst, int n_inst, const double* tabs, const double* phi0, int pitch,
                            S* g, P* phi, float* lo, long long nodes_total, const long long* node_begin)
{
    long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nodes_total) return;
    int lo_i = 0, hi_i = n_inst - 1;
    while (lo_i < hi_i) {
        int mid = (lo_i + hi_i + 1) >> 1;
        if (node_begin[mid] <= k) lo_i = mid; else hi_i = mid - 1;
    }
    const InstDev& I = inst[lo_i];
    const int NQ = (sizeof(S) == 2) ? 8 : 9, QOFF = (sizeof(S) == 2) ? 1 : 0;
    long long loc = k - node_begin[lo_i];
    int y = (int)(loc / I.nx), x = (int)(loc - (long long)y * I.nx);
    auto at = [&](int dx, int dy) -> double {
        int xx = wrap(x + dx, I.nx);
        int yy = I.slab ? y + dy : (I.walls ? mirror(y + dy, I.ny) : wrap(y + dy, I.ny));
        return phi0[(long long)(I.row0 + yy) * pitch + GC + xx];
    };
    double c0 = at(0, 0);
    double ax = at(1, 0) + at(-1, 0) + at(0, 1) + at(0, -1);
    double dg = at(1, 1) + at(-1, 1) + at(1, -1) + at(-1, -1);
    double lap = (2.0 / 3.0) * (ax - 4.0 * c0) + (1.0 / 6.0) * (dg - 4.0 * c0);
    C mu = (C)(dfdphi<double>(c0, I.cd.beta, I.cd.phiA, I.cd.phiB) - I.cd.kappa * lap);
    const double* tX1 = tabs + I.tab;
    const double* tX2 = tX1 + pitch;
    const double* tY1 = tX2 + pitch;
    const double* tY2 = tY1 + I.ylen;
    double T = vel_t(I.vel, I.Tper, 0);
    C ux = (C)(12.0 * tX1[x + GC] * tY1[y + GR] * T), uy = (C)(12.0 * tX2[x + GC] * tY2[y + GR] * T);
    C ph = (C)c0, eta = (C)I.cd.eta;
    C uu = ux * ux + uy * uy;
    C v[9];
#pragma unroll
    for (int q = 0; q < 9; q++) {
        if (q == 0) {
            // the float paths store g_0 - phi
            v[q] = (sizeof(C) == 4 ? C(0) : ph) + (wq<C>(0) - C(1)) * eta * mu - wq<C>(0) * C(1.5) * ph * uu;
        } else {
            C cu = (C)cx(q) * ux + (C)cy(q) * uy;
            v[q] = wq<C>(q) * eta * mu + wq<C>(q) * ph * (C(3) * cu + C(4.5) * cu * cu - C(1.5) * uu);
        }
    }
    const P hi = (P)c0;
    if (lo) lo[(long long)(I.row0 + y) * pitch + GC + x] = (float)(c0 - (double)hi);
    const int NONE = -0x40000000;
    const int xa = x < 3 ? x + I.nx : NONE, xb = x >= I.nx - 3 ? x - I.nx : NONE;
    // a slab's ghost rows are the neighbouring slabs' rows, imported before its first step
    const int ya = y < 3 && !I.slab ? (I.walls ? -1 - y : y + I.ny) : NONE;
    const int yb = y >= I.ny - 3 && !I.slab ? (I.walls ? 2 * I.ny - 1 - y : y - I.ny) : NONE;
    for (int iy = 0; iy < 3; iy++) {
        const int yy = iy == 0 ? y : (iy == 1 ? ya : yb);
        if (yy == NONE) continue;
        for (int ix = 0; ix < 3; ix++) {
            const int xx = ix == 0 ? x : (ix == 1 ? xa : xb);
            if (xx == NONE) continue;
            long long row = I.row0 + yy;
            phi[row * pitch + GC + xx] = hi;
            S* o = g + (row * NQ) * pitch + GC + xx;
            for (int q = QOFF; q < 9; q++) o[(q - QOFF) * pitch] = to_s<S>(v[q]);
        }
    }
}

// ------------------------------------------------------------------------------------------ reductions
// Observables in double: [0] sum phi, [1] sum (phi - phi0)^2, [2] sum phi0^2, [3] max, [4] min,
// [5] count of non-finite values.  Pass 1: grid (chunks, n_inst) writes per-block partials in a fixed
// order; pass 2: one block per instance reduces them in a fixed order, so results are reproducible.
constexpr int RED_NT = 256;
constexpr int RED_NV = 6;

__device__ __forceinline__ void red_combine(double* a, const double* b)
{
    a[0] += b[0]; a[1] += b[1]; a[2] += b[2];
    a[3] = fmax(a[3], b[3]); a[4] = fmin(a[4], b[4]); a[5] += b[5];
}

__device__ inline void block_reduce(double* v, double (*sh)[RED_NV])
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        double t[RED_NV];
#pragma unroll
        for (int k = 0; k < RED_NV; k++) t[k] = __shfl_down_sync(0xffffffffu, v[k], o);
        red_combine(v, t);
    }
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < RED_NV; k++) sh[w][k] = v[k];
    }
    __syncthreads();
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        double t[RED_NV];
        if (lane < nw) {
#pragma unroll
            for (int k = 0; k < RED_NV; k++) t[k] = sh[lane][k];
        } else {
            t[0] = t[1] = t[2] = t[5] = 0.0; t[3] = -INFINITY; t[4] = INFINITY;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            double u[RED_NV];
#pragma unroll
            for (int k = 0; k < RED_NV; k++) u[k] = __shfl_down_sync(0xffffffffu, t[k], o);
            red_combine(t, u);
        }
#pragma unroll
        for (int k = 0; k < RED_NV; k++) v[k] = t[k];
    }
}

template <typename P>
__global__ void __launch_bounds__(RED_NT) reduce_partials_kernel(const InstDev* inst, const P* phi, const float* lo,
                                                                 const double* phi0, int pitch,
                                                                 double* partials, int chunks)
{
    __shared__ double sh[RED_NT / 32][RED_NV];
    const InstDev& I = inst[blockIdx.y];
    const long long N = (long long)I.nx * I.ny;
    double v[RED_NV] = {0.0, 0.0, 0.0, -INFINITY, INFINITY, 0.0};
    for (long long k = (long long)blockIdx.x * RED_NT + threadIdx.x; k < N; k += (long long)chunks * RED_NT) {
        const int y = N <= 0x7fffffffLL ? (int)((unsigned)k / (unsigned)I.nx) : (int)(k / I.nx), x = (int)(k - (long long)y * I.nx);
        long long gi = (long long)(I.row0 + y) * pitch + GC + x;
        double p = (double)phi[gi] + (lo ? (double)lo[gi] : 0.0), p0 = phi0[gi];
        if (!isfinite(p)) { v[5] += 1.0; continue; }
        v[0] += p; v[1] += (p - p0) * (p - p0); v[2] += p0 * p0;
        v[3] = fmax(v[3], p); v[4] = fmin(v[4], p);
    }
    block_reduce(v, sh);
    if (threadIdx.x == 0) {
        double* out = partials + ((long long)blockIdx.y * chunks + blockIdx.x) * RED_NV;
#pragma unroll
        for (int k = 0; k < RED_NV; k++) out[k] = v[k];
    }
}

// The sums of an instance, and after those of all instances the error flags of the steps, into pinned host memory: the
// host reads them there once the stream is idle, without a copy of its own
static __global__ void __launch_bounds__(RED_NT) reduce_final_kernel(const double* partials, int chunks, const Ctl* ctl,
                                                                     double* result)
{
    __shared__ double sh[RED_NT / 32][RED_NV];
    double v[RED_NV] = {0.0, 0.0, 0.0, -INFINITY, INFINITY, 0.0};
    const double* base = partials + (long long)blockIdx.x * chunks * RED_NV;
    for (int c = threadIdx.x; c < chunks; c += RED_NT) red_combine(v, base + (long long)c * RED_NV);
    block_reduce(v, sh);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < RED_NV; k++) result[blockIdx.x * RED_NV + k] = v[k];
        if (blockIdx.x == 0) result[gridDim.x * RED_NV] = (double)ctl->err;
    }
}

// Rows [row, row + count / nx) of an instance's phi as contiguous doubles for the host (count < 2^31).  note[0] is set when
// one of them is not finite, note[1] to the error flags of the steps (pinned host memory, as above).
template <typename P>
__global__ void __launch_bounds__(256) gather_phi_kernel(const P* phi, const float* lo, int pitch, int nx, unsigned count,
                                                         const Ctl* ctl, double* out, double* note)
{
    const unsigned e = blockIdx.x * 256u + threadIdx.x;
    bool bad = false;
    if (e < count) {
        const unsigned y = e / (unsigned)nx;
        const long long k = (long long)y * pitch + (e - y * (unsigned)nx);
        const double p = (double)phi[k] + (lo ? (double)lo[k] : 0.0);
        out[e] = p;
        bad = !isfinite(p);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) note[0] = 1.0;
    if (e == 0) note[1] = (double)ctl->err;
}

}  // namespace lbch
