// lbch_adjoint.cuh -- reverse-mode adjoint of the step kernel (one instance, periodic domain).
//
// For a loss L of phi(T), lambda_q(x) = dL/dg_q(x).  One forward step (Eq. LB with Eqs. geq, liangFi,
// mu, t0-phiu, mark3) is
//   phi = sum_q g_q;  mu = f'(phi) - kappa lap phi;  F = -(phi^2/rho) grad mu [+ K grad div(phi u)];
//   post_q = (1 - 1/tau) g_q + g_eq_q(phi, mu, u)/tau + (1 - 1/(2 tau)) S_q(F);  g'_q(x + c_q) = post_q(x).
// Its Jacobian depends on the populations only through phi, so the backward sweep needs the forward phi
// of each step (a tape) and nothing else.  The transpose of every linear map is applied explicitly:
// streaming becomes a gather from x + c_q, the gradient stencil G becomes (G^T v)(x) = sum_k w_k c_k
// v(x - c_k)/c_s^2, the Laplacian L becomes (L^T v)(x) = sum_k 2 w_k (v(x - c_k) - v(x))/c_s^2.  The velocity
// is u = s u_ref and dL/ds (at s = 1) is accumulated in double.
//
// Layout: plain arrays over the instance, node index y*nx + x; lambda is [9][N].  The adjoint is carried
// in double for every storage precision (at tau = 1 all nine lambda_q are equal and dL/du is formed from
// differences of neighbouring lambda, which float storage would round away); the tape keeps the
// forward phi in the precision of the forward path, so the gradient is that of the path actually run.
// Two kernels per adjoint step on tiles of 32 x 8 nodes (local_kernel: forward mu and the local adjoints of collision,
// g_eq, S and F1; transpose_kernel: mu_bar and D_bar on tile + 1, phi_bar and the new lambda), and one deterministic sum of
// dL/ds at the end of the sweep.
//
// CF: the type the forward quantities are formed in (mu, its gradient, the velocity, rho and the force's
// coefficient, f''(phi)) -- float for a float tape, as the float forward step formed them, double for a double
// tape.  Everything that carries lambda is double in either case.
//
// ONE (tau_g = 1): lambda_q = (1 - 1/tau) lambda'_q(x + c_q) + phi_bar(x) is phi_bar(x) for every q, since
// 1 - 1/tau is exactly 0, so lambda is kept as one plane instead of nine.  The kernels read that plane where
// they would read plane q and write it once; the values are those of the nine-plane form bit for bit (for
// finite lambda, 0 * lambda' + phi_bar is phi_bar).

#pragma once
#include "lbch_kernels.cuh"

namespace lbch {
namespace adj {

struct AdjArgs {
    int nx, ny, model;
    int pitch;                 // of the velocity tables' X part
    int ylen;                  // length of each Y table
    long long n;               // forward step index of this adjoint step
    // constants of the adjoint step, formed once on the host: src/12, eta/tau, src/144, -K src/144
    double s12, ieta, s144, sK144;
};

__device__ __forceinline__ int wp(int i, int n) { return i >= n ? i - n : (i < 0 ? i + n : i); }

// the prescribed velocity at node (x, y) from the velocity tables of type CF (the forward step's), as the
// forward step forms it: X ((Y/12) T), times 12
template <typename CF>
__device__ __forceinline__ void vel_at(const InstDev& I, const CF* tabs, const AdjArgs& a, int x, int y, CF T, CF& ux,
                                       CF& uy)
{
    const CF* tX1 = tabs + I.tab;
    const CF* tX2 = tX1 + a.pitch;
    const CF* tY1 = tX2 + a.pitch;
    const CF* tY2 = tY1 + a.ylen;
    ux = op_mul(CF(12), node_u(tX1[x + GC], op_mul(tY1[y + GR], T)));
    uy = op_mul(CF(12), node_u(tX2[x + GC], op_mul(tY2[y + GR], T)));
}

template <typename C> __device__ __forceinline__ C d2f(C phi, C beta, C phiA, C phiB)
{
    // f''(phi) of f = beta (phi - phiA)^2 (phi - phiB)^2 (Eq. bulk)
    return C(2) * beta * ((phi - phiB) * (C(2) * phi - phiA - phiB) + (phi - phiA) * (C(2) * phi - phiA - phiB)
                          + C(2) * (phi - phiA) * (phi - phiB));
}

// The contractions sum_q l_q d g_eq_q / d(phi, mu, u) at one node (Eq. geq), for the adjoint l of the
// equilibria.  g_eq_q is quadratic in c_q . u, so they depend on l only through l_0 and its moments
// m0 = sum_q w_q l_q, m1 = sum_q w_q l_q c_q and m2 = sum_q w_q l_q c_q c_q, formed from the sums and
// differences of opposite directions.  m1 is returned too (the source term S_q is linear in c_q).
template <typename C>
__device__ __forceinline__ void geq_contract(const C* l, C phi, C ux, C uy, C eta, C& pl, C& ml, C& bx, C& by,
                                             C& m1x, C& m1y)
{
    // opposite pairs (1, 3) c = (1, 0); (2, 4) c = (0, 1); (5, 7) c = (1, 1); (6, 8) c = (-1, 1)
    const C E1 = l[1] + l[3], O1 = l[1] - l[3], E2 = l[2] + l[4], O2 = l[2] - l[4];
    const C E5 = l[5] + l[7], O5 = l[5] - l[7], E6 = l[6] + l[8], O6 = l[6] - l[8];
    const C wa = wq<C>(1), wd = wq<C>(5);
    const C Ed = wd * (E5 + E6);
    const C m2xx = wa * E1 + Ed, m2yy = wa * E2 + Ed, m2xy = wd * (E5 - E6);
    const C m0 = wq<C>(0) * l[0] + (wa * (E1 + E2) + Ed);
    m1x = wa * O1 + wd * (O5 - O6);
    m1y = wa * O2 + wd * (O5 + O6);
    const C vx = ux * m2xx + uy * m2xy, vy = ux * m2xy + uy * m2yy;  // sum_q w_q l_q (c_q . u) c_q
    const C uu = ux * ux + uy * uy;
    // d g_eq_0/d phi = 1 - (3/2) w_0 u^2;  d g_eq_q/d phi = w_q (3 c_q.u + (9/2)(c_q.u)^2 - (3/2) u^2)
    pl = l[0] + C(3) * (ux * m1x + uy * m1y) + C(4.5) * (ux * vx + uy * vy) - C(1.5) * uu * m0;
    // d g_eq_0/d mu = (w_0 - 1) eta;  d g_eq_q/d mu = w_q eta
    ml = eta * (m0 - l[0]);
    // d g_eq_q/d u = w_q phi (3 c_q + 9 (c_q.u) c_q - 3 u), q = 0 included
    bx = phi * (C(3) * m1x + C(9) * vx - C(3) * ux * m0);
    by = phi * (C(3) * m1y + C(9) * vy - C(3) * uy * m0);
}

// The isotropic Laplacian on the periodic lattice, grouped by axis and diagonal neighbours:
// (L v)(x) = sum_k 2 w_k (v(x + c_k) - v(x))/c_s^2.  Its transpose follows by substituting c_k -> -c_k: L^T = L (and
// G^T = -G for the gradient).
template <typename C, typename V>
__device__ __forceinline__ C at_nb(const V* v, int nx, int ny, int x, int y, int dx, int dy)
{
    return (C)v[(long long)wp(y + dy, ny) * nx + wp(x + dx, nx)];
}
template <typename C, typename V>
__device__ __forceinline__ C lap_c(const V* v, int nx, int ny, int x, int y)
{
    auto at = [&](int dx, int dy) { return at_nb<C>(v, nx, ny, x, y, dx, dy); };
    const C c = at(0, 0);
    const C ax = (at(1, 0) + at(-1, 0)) + (at(0, 1) + at(0, -1));
    const C dg = (at(1, 1) + at(-1, 1)) + (at(1, -1) + at(-1, -1));
    return C(2) / C(3) * (ax - C(4) * c) + C(1) / C(6) * (dg - C(4) * c);
}
// (L^T v)(x)
template <typename C>
__device__ __forceinline__ C lapT(const C* v, int nx, int ny, int x, int y)
{
    return lap_c<C>(v, nx, ny, x, y);
}

// ---- one adjoint step
//
// Everything that carries lambda is bound by the FP64 pipe, so the two kernels are built to take few operations: about 90
// per node, conversions of the forward quantities included, where four one-thread-per-node kernels took about 130 (us per
// step with a float tape: 512^2 84 -> 56, 1024^2 281 -> 189, 100^2 25 -> 19; the pipe is 83 % busy).
//   - The stencils go through shared memory column first (lbch_kernels.cuh): a pass for the column values, then one
//     along the rows.
//   - The moments of the gathered lambda' are stencils too.  With ONE they are, times 36: M0 = w(E) + 4 w + w(W),
//     M1 = (w(E) - w(W), d(E) + 4 d + d(W)), M2xx = w(E) + w(W), M2yy = v(E) + 4 v + v(W), M2xy = d(E) - d(W) with the column
//     values v = l(N) + l(S), w = 4 l + v, d = l(N) - l(S).
//   - With B = M1 + (3 M2 - M0) u, the contractions of lambda' with d g_eq (geq_contract) are d/du: phi B/12 and
//     d/dphi: l_0 + u.(B + M1)/24.  u.B is all that dL/ds needs of the former, so that one value is handed on.
//   - S is linear in F: F_bar = src M1/12, so grad_mu_bar = -coef F_bar and D_bar = K G^T F_bar come from M1, which
//     the first kernel hands to the second.
// What is handed on: M1 (two values), the local phi_bar, the local mu_bar and u.B/tau.
// Tiles of 32 x 8, one node per thread: four to six blocks per SM keep the pipe fed across each other's barriers, and
// 1024 of them at 512^2 spread evenly (32 x 16 recompute less of the halo but took 66 us per step there, 32 x 4 65).
constexpr int TX = 32, TY = 8, NT = 256;
// transpose_kernel's shared memory: the vectors on tile + 2, later mu_bar and D_bar on tile + 1 with their column values
constexpr int N_VEC = 4 * (TX + 4) * (TY + 4), N_BAR = 2 * (TX + 2) * (TY + 2) + 4 * (TX + 2) * TY;
constexpr int N_FIRST = N_VEC > N_BAR ? N_VEC : N_BAR;
constexpr size_t TRANSPOSE_SMEM = 8 * (N_FIRST + 6 * (TX + 4) * (TY + 2));

__device__ __forceinline__ int wrap_any(int v, int n)
{
    if (v < 0 || v >= n) {
        v %= n;
        if (v < 0) v += n;
    }
    return v;
}

// f(e, i, j) for the nodes (i, j) of a W x H region, e = j W + i
template <int W, int H, typename F> __device__ __forceinline__ void region(F&& f)
{
    for (int e = threadIdx.x; e < W * H; e += NT) {
        const int j = e / W;
        f(e, e - j * W, j);
    }
}

template <typename C, typename CF, typename TP, bool ONE>
__global__ void __launch_bounds__(NT, ONE ? 4 : 3) local_kernel(const InstDev* inst, const CF* tabs, AdjArgs a, CF T, const TP* phi,
                                                      const C* lam_next, C* M1, C* phib, C* mub, C* uB)
{
    constexpr int PW = TX + 4, PH = TY + 4;  // phi on tile + 2
    constexpr int ZW = TX + 4, ZH = TY + 2;  // its column values
    constexpr int MW = TX + 2, MH = TY + 2;  // mu (and lambda) on tile + 1
    constexpr int GW = TX + 2, GH = TY;      // the column values of mu (and lambda)
    __shared__ CF s_p[PW * PH], s_z[ZW * ZH], s_dl[ZW * ZH], s_m[MW * MH], s_wm[GW * GH], s_dm[GW * GH];
    __shared__ C s_l[ONE ? MW * MH : 1], s_v[ONE ? GW * GH : 1], s_w[ONE ? GW * GH : 1], s_d[ONE ? GW * GH : 1];
    const InstDev& I = inst[0];
    const Consts<C>& K0 = consts<C>(I);
    const Consts<CF>& KF = consts<CF>(I);
    const int nx = a.nx, ny = a.ny;
    const long long N = (long long)nx * ny;
    const int tiles_x = (nx + TX - 1) / TX;
    const int x0 = ((int)blockIdx.x % tiles_x) * TX, y0 = ((int)blockIdx.x / tiles_x) * TY;
    region<PW, PH>([&](int e, int i, int j) {
        s_p[e] = (CF)phi[(long long)wrap_any(y0 - 2 + j, ny) * nx + wrap_any(x0 - 2 + i, nx)];
    });
    if constexpr (ONE)
        region<MW, MH>([&](int e, int i, int j) {
            s_l[e] = lam_next[(long long)wrap_any(y0 - 1 + j, ny) * nx + wrap_any(x0 - 1 + i, nx)];
        });
    __syncthreads();
    region<ZW, ZH>([&](int e, int i, int j) {
        CF dl;
        s_z[e] = node_z(s_p[e], s_p[e + PW], s_p[e + 2 * PW], dl);
        s_dl[e] = dl;
    });
    if constexpr (ONE)
        region<GW, GH>([&](int e, int i, int j) {
            const C S = s_l[e], Nn = s_l[e + 2 * MW];
            const C v = Nn + S;
            s_v[e] = v;
            s_w[e] = fma(C(4), s_l[e + MW], v);
            s_d[e] = Nn - S;
        });
    __syncthreads();
    region<MW, MH>([&](int e, int i, int j) {
        const int k = j * ZW + i + 1;
        s_m[e] = node_mu(s_p[k + PW], s_dl[k], s_z[k], s_z[k + 1], s_z[k - 1], KF);
    });
    __syncthreads();
    region<GW, GH>([&](int e, int i, int j) {
        const CF S = s_m[e], Nn = s_m[e + 2 * MW];
        s_wm[e] = node_w(S, s_m[e + MW], Nn);
        s_dm[e] = Nn - S;
    });
    __syncthreads();
    region<TX, TY>([&](int e, int i, int j) {
        const int x = x0 + i, y = y0 + j;
        if (x >= nx || y >= ny) return;
        const long long k = (long long)y * nx + x;
        const int c = j * GW + i + 1;  // the node among the column values
        // the forward quantities at the node, in CF
        const CF phf = s_p[(j + 2) * PW + i + 2];
        CF uxf, uyf;
        vel_at(I, tabs, a, x, y, T, uxf, uyf);
        const CF gxf = op_mul(CF(1) / CF(12), s_wm[c + 1] - s_wm[c - 1]);  // grad mu
        const CF gyf = op_mul(CF(1) / CF(12), node_gy(s_dm[c - 1], s_dm[c], s_dm[c + 1]));
        const CF rhof = KF.a * phf + KF.b, rf = rcp<CF>(rhof);
        const CF dcoeff = phf * (KF.a * phf + CF(2) * KF.b) * (rf * rf);  // d coef / d phi, F1 = -coef grad mu
        const C ux = (C)uxf, uy = (C)uyf, gx = (C)gxf, gy = (C)gyf, dcoef = (C)dcoeff;
        // 36 times the moments of lambda'_q = lambda_q(x + c_q) (reverse streaming)
        C l0, M0, M1x, M1y, Mxx, Myy, Mxy;
        if constexpr (ONE) {
            l0 = s_l[(j + 1) * MW + i + 1];
            const C dE = s_d[c + 1], d = s_d[c], dW = s_d[c - 1], wE = s_w[c + 1], wW = s_w[c - 1];
            Mxx = wE + wW;
            M0 = fma(C(4), s_w[c], Mxx);
            M1x = wE - wW;
            M1y = fma(C(4), d, dE + dW);
            Myy = fma(C(4), s_v[c], s_v[c + 1] + s_v[c - 1]);
            Mxy = dE - dW;
        } else {
            C l[9];
#pragma unroll
            for (int q = 0; q < 9; q++)
                l[q] = lam_next[q * N + (long long)wp(y + cy(q), ny) * nx + wp(x + cx(q), nx)];
            // opposite pairs (1, 3) c = (1, 0); (2, 4) c = (0, 1); (5, 7) c = (1, 1); (6, 8) c = (-1, 1)
            const C E1 = l[1] + l[3], O1 = l[1] - l[3], E2 = l[2] + l[4], O2 = l[2] - l[4];
            const C E5 = l[5] + l[7], O5 = l[5] - l[7], E6 = l[6] + l[8], O6 = l[6] - l[8];
            const C s56 = E5 + E6;
            l0 = l[0];
            Mxx = fma(C(4), E1, s56);
            Myy = fma(C(4), E2, s56);
            Mxy = E5 - E6;
            M0 = fma(C(16), l0, fma(C(4), E2, Mxx));
            M1x = fma(C(4), O1, O5 - O6);
            M1y = fma(C(4), O2, O5 + O6);
        }
        const C r = C(3) * Mxy;
        const C Bx = fma(ux, fma(C(3), Mxx, -M0), fma(uy, r, M1x));
        const C By = fma(uy, fma(C(3), Myy, -M0), fma(ux, r, M1y));
        const C ub = fma(ux, Bx, uy * By), um = fma(ux, M1x, uy * M1y);
        const C pl = fma(C(1) / C(24), ub + um, l0);            // sum_q l_q d g_eq_q/d phi
        const C ml = fma(C(1) / C(36), M0, -l0);                // (1/eta) sum_q l_q d g_eq_q/d mu
        M1[k] = M1x;
        M1[N + k] = M1y;
        phib[k] = fma(K0.itau, pl, -(C(a.s12) * dcoef) * fma(M1x, gx, M1y * gy));
        mub[k] = C(a.ieta) * ml;
        uB[k] = K0.itau * ub;
    });
}

// mu_bar = local + G^T grad_mu_bar;  D_bar = 3 c_s^2 K G^T F_bar;
// phi_bar = local + f''(phi) mu_bar - kappa L^T mu_bar + u . G^T D_bar;
// lambda_q(x) = (1 - 1/tau) lambda_next_q(x + c_q) + phi_bar(x); dL/ds per node.  (G^T = -G, L^T = L.)
template <typename C, typename CF, typename TP, bool ONE>
__global__ void __launch_bounds__(NT, ONE ? 6 : 3) transpose_kernel(const InstDev* inst, const CF* tabs, AdjArgs a, CF T,
                                                          const TP* phi, const C* M1, const C* phib, const C* mub,
                                                          const C* uB, const C* lam_next, C* lam, double* ds)
{
    constexpr int VW = TX + 4, VH = TY + 4;  // M1 and coef M1 on tile + 2
    constexpr int ZW = TX + 4, ZH = TY + 2;  // the column values of their divergences
    constexpr int MW = TX + 2, MH = TY + 2;  // mu_bar, D_bar on tile + 1
    constexpr int GW = TX + 2, GH = TY;      // their column values
    constexpr int NV = VW * VH, NZ = ZW * ZH, NM = MW * MH, NG = GW * GH;
    // the vectors, later (their place taken over) mu_bar, D_bar and their column values; the shares of the divergences
    static_assert(4 * NV <= N_FIRST && 2 * NM + 4 * NG <= N_FIRST, "the first part holds either");
    extern __shared__ __align__(16) unsigned char smem_adj[];
    C *s_v = reinterpret_cast<C*>(smem_adj), *s_c = s_v + N_FIRST;
    const InstDev& I = inst[0];
    const Consts<C>& K0 = consts<C>(I);
    const Consts<CF>& KF = consts<CF>(I);
    const int nx = a.nx, ny = a.ny;
    const long long N = (long long)nx * ny;
    const int tiles_x = (nx + TX - 1) / TX;
    const int x0 = ((int)blockIdx.x % tiles_x) * TX, y0 = ((int)blockIdx.x / tiles_x) * TY;
    const bool model2 = a.model == 2;
    region<VW, VH>([&](int e, int i, int j) {
        const long long k = (long long)wrap_any(y0 - 2 + j, ny) * nx + wrap_any(x0 - 2 + i, nx);
        const CF phf = (CF)phi[k];
        const C coef = (C)(phf * phf * rcp<CF>(KF.a * phf + KF.b));  // F1 = -coef grad mu
        const C mx = M1[k], my = M1[N + k];
        s_v[e] = coef * mx;
        s_v[NV + e] = coef * my;
        s_v[2 * NV + e] = mx;
        s_v[3 * NV + e] = my;
    });
    __syncthreads();
    // the share of a column in the divergence (times 12) of the node to its west, to its east and of its own node (times 4)
    auto col = [&](const C* v, int e, C* o) {
        const C t = fma(C(4), v[e + VW], v[e + 2 * VW] + v[e]), d = v[NV + e + 2 * VW] - v[NV + e];
        o[e] = t + d;
        o[NZ + e] = d - t;
        o[2 * NZ + e] = d;
    };
    region<ZW, ZH>([&](int e, int i, int j) {
        col(s_v, e, s_c);
        if (model2) col(s_v + 2 * NV, e, s_c + 3 * NZ);
    });
    __syncthreads();
    C *s_mu = s_v, *s_D = s_v + NM, *s_z = s_v + 2 * NM;  // the vectors are read no more
    const C cm = C(a.s144), cD = C(a.sK144);
    region<MW, MH>([&](int e, int i, int j) {
        const int k = j * ZW + i + 1;
        const long long g = (long long)wrap_any(y0 - 1 + j, ny) * nx + wrap_any(x0 - 1 + i, nx);
        // grad_mu_bar = -coef src M1/12, and G^T is minus a twelfth of the sum of the shares
        s_mu[e] = fma(cm, fma(C(4), s_c[2 * NZ + k], s_c[k + 1] + s_c[NZ + k - 1]), mub[g]);
        if (model2) s_D[e] = cD * fma(C(4), s_c[5 * NZ + k], s_c[3 * NZ + k + 1] + s_c[4 * NZ + k - 1]);
    });
    __syncthreads();
    region<GW, GH>([&](int e, int i, int j) {
        const C S = s_mu[e], c = s_mu[e + MW], Nn = s_mu[e + 2 * MW];
        C dl;
        s_z[e] = node_z(S, c, Nn, dl);
        s_z[NG + e] = dl;
        if (model2) {
            const C dS = s_D[e], dN = s_D[e + 2 * MW];
            s_z[2 * NG + e] = node_w(dS, s_D[e + MW], dN);
            s_z[3 * NG + e] = dN - dS;
        }
    });
    __syncthreads();
    region<TX, TY>([&](int e, int i, int j) {
        const int x = x0 + i, y = y0 + j;
        if (x >= nx || y >= ny) return;
        const long long k = (long long)y * nx + x;
        const int c = j * GW + i + 1;
        // the forward quantities at the node, in CF
        const CF phf = (CF)phi[k];
        CF uxf, uyf;
        vel_at(I, tabs, a, x, y, T, uxf, uyf);
        const C ph = (C)phf, ux = (C)uxf, uy = (C)uyf;
        const C f2 = (C)d2f(phf, KF.beta, KF.phiA, KF.phiB);
        const C z = s_z[c], lap = s_z[NG + c] + fma(C(-2), z, s_z[c + 1] + s_z[c - 1]);
        C pb = fma(-K0.kappa, lap, fma(f2, s_mu[(j + 1) * MW + i + 1], phib[k]));
        C ub = uB[k];  // 12 u . (adjoint of phi u), to which 12 u . G^T D_bar adds
        if (model2) {
            const C* w = s_z + 2 * NG + c;
            const C* d = s_z + 3 * NG + c;
            const C uj = fma(ux, w[-1] - w[1], -(uy * fma(C(4), d[0], d[1] + d[-1])));
            pb = fma(C(1) / C(12), uj, pb);
            ub += uj;
        }
        // u = s u_ref: du/ds = u.  Accumulated per node over the adjoint steps and summed once at the end.
        ds[k] = fma(C(1) / C(12), ph * ub, ds[k]);
        if constexpr (ONE) {
            lam[k] = pb;  // (1 - 1/tau) = 0: the reverse streaming and collision leave phi_bar alone
        } else {
#pragma unroll
            for (int q = 0; q < 9; q++)  // reverse streaming and collision, plus phi = sum_q g_q
                lam[q * N + k] = K0.omt * lam_next[q * N + (long long)wp(y + cy(q), ny) * nx + wp(x + cx(q), nx)] + pb;
        }
    });
}

// adjoint of the initial equilibria: dL/dphi0 (two kernels: local, then the mu transpose)
template <typename C, bool ONE>
__global__ void init_local_kernel(const InstDev* inst, const double* tabs, AdjArgs a, double T, const double* phi0,
                                  int pitch0, const C* lam, C* mub, C* dphi0, double* ds)
{
    const InstDev& I = inst[0];
    const Consts<C>& K0 = consts<C>(I);
    const long long N = (long long)a.nx * a.ny;
    long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    int y = (int)k / a.nx, x = (int)k - y * a.nx;  // fewer than 2^31 nodes (lb_ch_adjoint_begin checks)
    C ph = (C)phi0[(long long)(I.row0 + y) * pitch0 + GC + x];
    C ux, uy;
    vel_at<C>(I, tabs, a, x, y, (C)T, ux, uy);
    C l[9];
#pragma unroll
    for (int q = 0; q < 9; q++) l[q] = lam[(ONE ? 0 : q * N) + k];
    C pl, ml, bx, by, m1x, m1y;
    geq_contract(l, ph, ux, uy, K0.eta, pl, ml, bx, by, m1x, m1y);
    dphi0[k] = pl;
    mub[k] = ml;
    ds[k] += (double)bx * (double)ux + (double)by * (double)uy;
}

template <typename C>
__global__ void init_transpose_kernel(const InstDev* inst, AdjArgs a, const double* phi0, int pitch0, const C* mub,
                                      C* dphi0)
{
    const InstDev& I = inst[0];
    const Consts<C>& K0 = consts<C>(I);
    long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)a.nx * a.ny) return;
    int y = (int)k / a.nx, x = (int)k - y * a.nx;  // fewer than 2^31 nodes (lb_ch_adjoint_begin checks)
    C ph = (C)phi0[(long long)(I.row0 + y) * pitch0 + GC + x];
    dphi0[k] += d2f(ph, K0.beta, K0.phiA, K0.phiB) * mub[k] - K0.kappa * lapT(mub, a.nx, a.ny, x, y);
}

// deterministic sum of ds[0..N) into *acc (one block, fixed order), executed once, at the end of the adjoint
// sweep (ds holds each node's contributions from every step)
__global__ void __launch_bounds__(256) sum_into_kernel(const double* ds, long long N, double* acc)
{
    __shared__ double sh[256];
    double s = 0.0;
    for (long long k = threadIdx.x; k < N; k += 256) s += ds[k];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *acc += sh[0];
}

// phi of the instance (padded storage, plus the low part on the float path) into a plain array
template <typename P, typename C>
__global__ void tape_kernel(const InstDev* inst, int pitch, const P* phi, const float* lo, C* out)
{
    const InstDev& I = inst[0];
    long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)I.nx * I.ny) return;
    int y = (int)k / I.nx, x = (int)k - y * I.nx;  // fewer than 2^31 nodes (lb_ch_tape_phi checks)
    long long gi = (long long)(I.row0 + y) * pitch + GC + x;
    out[k] = (C)((double)phi[gi] + (lo ? (double)lo[gi] : 0.0));
}

// lambda_T: dL/dg_q = dL/dphi(T) for every q (nq planes: 9, or 1 with ONE)
template <typename C>
__global__ void adj_begin_kernel(long long N, int nq, const C* dphiT, C* lam)
{
    long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    C v = dphiT[k];
    for (int q = 0; q < nq; q++) lam[q * N + k] = v;
}

}  // namespace adj
}  // namespace lbch
