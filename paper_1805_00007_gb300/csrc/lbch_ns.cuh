// lbch_ns.cuh -- the coupled Cahn-Hilliard / Navier-Stokes step (flows that are not prescribed).
//
// For the Rayleigh-Taylor problem (Sec. III.E) the velocity is not prescribed but solved by a second
// D2Q9 lattice Boltzmann equation for Eq. NS.  The paper calls that equation standard without writing
// it out; the library takes the incompressible, pressure-based single-relaxation-time form with forcing:
//   f_i(x + c_i, t + 1) = f_i - (f_i - f_i^eq)/tau_f + (1 - 1/(2 tau_f)) G_i,   tau_f = nu/c_s^2 + 1/2,
//   f_0^eq = (w_0 - 1) p/c_s^2 + rho s_0(u),  f_i^eq = w_i p/c_s^2 + rho s_i(u),
//   s_i(u) = w_i [c_i.u/c_s^2 + (c_i.u)^2/(2 c_s^4) - u^2/(2 c_s^2)],  Gamma_i = w_i + s_i(u),
//   G_i = (c_i - u) . [Gamma_i F + s_i(u) c_s^2 grad rho] / c_s^2,
//   rho u = sum_i c_i f_i + F/2,   p = c_s^2/(1 - w_0) [sum_{i>0} f_i + (1/2) u.grad rho + rho s_0(u)],
// with rho = a phi + b (Eq. rho) and F = -phi grad mu - (rho - (rhoA + rhoB)/2) g + (d rho/d phi) M lap(mu) u
// (Eq. NS, form c).  The Cahn-Hilliard lattice uses this u and F1 = (phi/rho)(-phi grad mu - grad p)
// (Eq. t0-phiu) plus the Eq. mark3 term.  Walls: halfway bounce-back for both lattices at rest; stencil
// operands at ghost rows take the mirror values.
//
// One step is two kernels on 32 x 8 tiles of nodes, one thread per node, with the stencil operands staged in shared
// memory, each launched as a programmatic dependent of the one before it.  fields_kernel sums phi = sum_q g_q on tile + 2,
// forms mu on tile + 1 and gives phi, mu, u and p at the tile's nodes.  collide_kernel stages these (and phi u) on tile + 2,
// forms D = div(phi u) on tile + 1 for Model II (kept there rather than stored), collides both lattices and pushes them to
// the neighbours (bounce-back at walls).  phi_kernel forms phi in the handle's array on demand before an observation.  A
// stencil operand at a ghost row beyond a wall takes the value of the mirror node: a staged operand is read at that node,
// and a derived one is formed at the mirror row of the tile's region.
//
// What bounds it: in float the instructions issued (387 and 662 per node) and, on small grids, the latency of two
// launches (3 us each); in double the FP64 pipe.  256 x 1024 in float: 14.3 us per step, against 17.9 with a plane per
// population, ordinary launches and the populations g read at tau_g = 1 too; 64 x 200: 5.9 against 11.1.  One thread per
// node against two nodes per thread in the collision: 5.9 and 7.1 us for 64 x 200, 11.8 and 14.4 for 200 x 760, 20.2 and
// 19.8 for 400 x 1000, and in double 101 and 155 for 160 x 640.
#pragma once
#include "lbch_kernels.cuh"

namespace lbch {
namespace ns {

template <typename C>
struct NsConsts {
    C tauf, gx, gy, M, rbar;
    C itauf, omtf, srcf;  // 1/tau_f, 1 - 1/tau_f and 1 - 1/(2 tau_f), formed once on the host
};

// Storage: the nodes of a row in groups of 32 (a tile's row, a warp), and the values of a group one after the other: the
// nine g and the nine f of a state, or the five fields between the kernels.  All of a node's values then lie at constant
// distances of multiples of 32 elements from one address (with a plane per population each access formed its own: 62 of the
// 463 instructions per node in the fields kernel, 300 integer ones of 896 in the collision), and an access of a warp is
// one aligned line.
constexpr int GW = 32, POPS = 18 * GW, AUXS = 5 * GW;
enum Aux { A_PHI = 0, A_UX = GW, A_UY = 2 * GW, A_MU = 3 * GW, A_P = 4 * GW };

template <typename C>
struct NsArgs {
    int nx, ny, walls, model, pitch, row0;
    int nb;            // groups per row
    Consts<C> k;       // the Cahn-Hilliard constants
    NsConsts<C> n;     // the flow's constants
    const C* in;       // [ny][nb][18][32]: g and f of the current state
    C* out;            // of the next one
    C* aux;            // [ny][nb][5][32]: phi, u, mu and p of the current state
    C* phi;            // the handle's padded phi array of the current state
    double* obs;       // [3][ny nx]: u and p for observation
    // constants of the form in double with the stencils' 1/12 and 1/6 folded in: kappa/6, a M/6, a/24, K/144, 3 src_f,
    // 3 src_f a/36, 3/tau_f, 3 src/9 and eta/tau_g
    C kappa6, aM6, a24, K144, s3, s3a36, itf3, src9, ieta;
};

template <typename C> inline void set_folded(NsArgs<C>& a)
{
    a.kappa6 = a.k.kappa / C(6);
    a.aM6 = a.k.a * a.n.M / C(6);
    a.a24 = a.k.a / C(24);
    a.K144 = a.k.K / C(144);
    a.s3 = C(3) * a.n.srcf;
    a.s3a36 = a.s3 * a.k.a / C(36);
    a.itf3 = C(3) * a.n.itauf;
    a.src9 = a.k.src / C(3);
    a.ieta = a.k.itau * a.k.eta;
}

// groups of a row, and elements of the coupled state: two of the populations and one of the fields
__host__ __device__ inline int groups_of(int nx) { return (nx + GW - 1) / GW; }
inline size_t state_elems(int nx, int ny) { return (size_t)groups_of(nx) * ny * POPS; }
inline size_t aux_elems(int nx, int ny) { return (size_t)groups_of(nx) * ny * AUXS; }

// element offset of node (x, y) in an array of STRIDE values per group
template <int STRIDE, typename C> __device__ __forceinline__ long long at(const NsArgs<C>& a, int x, int y)
{
    return (long long)(y * a.nb + (x >> 5)) * STRIDE + (x & 31);
}

// tiles, one node per thread, and the region staged around them
constexpr int TX = GW, TY = 8, NT = TX * TY;
constexpr int W = TX + 4, H = TY + 4, N2 = W * H;          // tile + 2
constexpr int W1 = TX + 2, H1 = TY + 2, N1 = W1 * H1;      // tile + 1, kept in the layout of tile + 2

__host__ __device__ inline int tiles_of(int nx, int ny) { return groups_of(nx) * ((ny + TY - 1) / TY); }

__device__ __forceinline__ int wrap_any(int v, int n)
{
    if (v < 0 || v >= n) {
        v %= n;
        if (v < 0) v += n;
    }
    return v;
}

// The node whose value a stencil operand at coordinate (x, y) takes: periodic in x; periodic in y or
// mirrored at walls.  (Coordinates more than one row beyond a wall occur only in the region of a ragged
// tile, where no node reads them; they are clamped into the domain.)
__device__ __forceinline__ int2 node_at(int nx, int ny, int walls, int x, int y)
{
    x = wrap_any(x, nx);
    if (walls) {
        y = y < 0 ? -1 - y : (y >= ny ? 2 * ny - 1 - y : y);
        y = min(max(y, 0), ny - 1);
    } else {
        y = wrap_any(y, ny);
    }
    return make_int2(x, y);
}

// The row of the staged region (its row 0 is y0 - 2) at which a derived field is formed for its row j: j itself, or the
// mirror row of a ghost row beyond a wall.
__device__ __forceinline__ int mirror_row(int walls, int ny, int y0, int j)
{
    if (!walls) return j;
    const int y = y0 - 2 + j;
    const int m = (y < 0 ? -1 - y : (y >= ny ? 2 * ny - 1 - y : y)) - (y0 - 2);
    return (m >= 1 && m <= H1) ? m : j;
}

// The isotropic stencils on a staged region around flat index c (x to the east, y to the
// north): grad psi = sum_k w_k c_k psi(x + c_k) / c_s^2 and lap psi = sum_k 2 w_k (psi(x + c_k) - psi) / c_s^2.
template <typename C> __device__ __forceinline__ C sgx(const C* s, int c)
{
    return op_fma(C(1) / C(3), s[c + 1] - s[c - 1],
                  op_mul(C(1) / C(12), (s[c + W + 1] - s[c + W - 1]) + (s[c - W + 1] - s[c - W - 1])));
}
template <typename C> __device__ __forceinline__ C sgy(const C* s, int c)
{
    return op_fma(C(1) / C(3), s[c + W] - s[c - W],
                  op_mul(C(1) / C(12), (s[c + W + 1] + s[c + W - 1]) - (s[c - W + 1] + s[c - W - 1])));
}
template <typename C> __device__ __forceinline__ C slap(const C* s, int c)
{
    const C ce = s[c];
    const C ax = (s[c + 1] + s[c - 1]) + (s[c + W] + s[c - W]);
    const C dg = (s[c + W + 1] + s[c + W - 1]) + (s[c - W + 1] + s[c - W - 1]);
    return op_fma(C(2) / C(3), op_fma(C(-4), ce, ax), op_mul(C(1) / C(6), op_fma(C(-4), ce, dg)));
}

// The same column first, for the form in double: with V = psi(N) + psi(S), A = V + 4 psi and D = psi(N) - psi(S) at every
// node, 12 d/dx = A(E) - A(W), 12 d/dy = D(E) + D(W) + 4 D and 6 lap = A(E) + A(W) + 4 A - 36 psi: nine operations per
// node for the three instead of 22.  columns() forms A and D for `rows` rows of the staged region from its row row0 on.
template <typename C> __device__ __forceinline__ void columns(const C* s, int row0, int rows, C* A, C* D)
{
    s += row0 * W;
    for (int e = threadIdx.x; e < rows * W; e += NT) {
        const C n = s[e + W], o = s[e - W];
        A[e] = fma(C(4), s[e], n + o);
        D[e] = n - o;
    }
}
template <typename C> __device__ __forceinline__ C cgx(const C* A, int e) { return A[e + 1] - A[e - 1]; }
template <typename C> __device__ __forceinline__ C cgy(const C* D, int e) { return fma(C(4), D[e], D[e + 1] + D[e - 1]); }
template <typename C> __device__ __forceinline__ C clap(const C* A, int e, C psi)
{
    return fma(C(-36), psi, fma(C(4), A[e], A[e + 1] + A[e - 1]));
}

// Forms of the two kernels: in double, which the FP64 pipe bounds, the stencils column first and the constants folded (255
// FP64 operations per node and step instead of 371: 256 x 1024 in 136 us instead of 191, the pipe 82 % busy in both
// kernels); in float, which integer work and latency bound, as the equations stand.
template <typename C> constexpr bool FOLDED = sizeof(C) == 8;

// The tile of this block: origin (x0, y0)
__device__ __forceinline__ void tile_origin(int nb, int& x0, int& y0)
{
    const unsigned t = blockIdx.x / (unsigned)nb;
    x0 = (int)(blockIdx.x - t * (unsigned)nb) * TX;
    y0 = (int)t * TY;
}

// phi = sum_q g_q (Eq. macroscopicg) of the populations at p, summed in the order of q
template <typename C> __device__ __forceinline__ C sum_g(const C* p)
{
    C s = C(0);
#pragma unroll
    for (int q = 0; q < 9; q++) s += p[q * GW];
    return s;
}

// f(e, x, y) for the region tile + 2, e counting it by row: (x, y) the node a stencil operand there takes its value from.
// A tile whose region lies inside the domain needs no wrapping.
template <typename C, typename F>
__device__ __forceinline__ void for_region(const NsArgs<C>& a, int x0, int y0, F&& f)
{
    const bool inside = x0 >= 2 && x0 + TX + 2 <= a.nx && y0 >= 2 && y0 + TY + 2 <= a.ny;
    for (int e = threadIdx.x; e < N2; e += NT) {
        const int j = e / W, i = e - j * W;
        int2 v = make_int2(x0 - 2 + i, y0 - 2 + j);
        if (!inside) v = node_at(a.nx, a.ny, a.walls, v.x, v.y);
        f(e, v.x, v.y);
    }
}

// f(e, c) for the region tile + 1: e the node's index in the staged region, c that of the node it is formed at
template <typename C, typename F>
__device__ __forceinline__ void for_inner(const NsArgs<C>& a, int y0, F&& f)
{
    for (int e = threadIdx.x; e < N1; e += NT) {
        const int j = e / W1 + 1, i = e - (j - 1) * W1 + 1;
        f(j * W + i, mirror_row(a.walls, a.ny, y0, j) * W + i);
    }
}

// phi = sum_q g_q of the current state, then mu and the flow's velocity and pressure at every node, for the collision
// kernel that follows; OBS: u and p into the contiguous planes of an observation instead
template <typename C, bool OBS>
__global__ void __launch_bounds__(NT) fields_kernel(NsArgs<C> a)
{
    constexpr bool F = FOLDED<C>;
    __shared__ C s2[N2], mu2[N2], phA[F ? H1 * W : 1], phD[F ? H1 * W : 1], muA[F ? TY * W : 1], muD[F ? TY * W : 1];
    int x0, y0;
    tile_origin(a.nb, x0, y0);
    grid_dependency_wait();
    grid_launch_dependents();
    for_region(a, x0, y0, [&](int e, int x, int y) { s2[e] = sum_g(a.in + at<POPS>(a, x, y)); });
    __syncthreads();
    if (F) {
        columns(s2, 1, H1, phA, phD);
        __syncthreads();
    }
    for_inner(a, y0, [&](int e, int c) {  // mu (Eq. mu)
        const C df = node_dfdphi(s2[c], a.k.beta, a.k.phiA, a.k.phiB);
        mu2[e] = F ? fma(-a.kappa6, clap(phA, c - W, s2[c]), df) : op_fma(-a.k.kappa, slap<C>(s2, c), df);
    });
    __syncthreads();
    if (F) {
        columns(mu2, 2, TY, muA, muD);
        __syncthreads();
    }
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX, x = x0 + tx, y = y0 + ty;
    if (x >= a.nx || y >= a.ny) return;
    const int c = (ty + 2) * W + tx + 2;
    const C* fk = a.in + at<POPS>(a, x, y) + 9 * GW;
    C f[9];
#pragma unroll
    for (int q = 0; q < 9; q++) f[q] = fk[q * GW];
    const C phi = s2[c], rho = op_fma(a.k.a, phi, a.k.b), db = rho - a.n.rbar;
    const C s1 = ((f[1] + f[2]) + (f[3] + f[4])) + ((f[5] + f[6]) + (f[7] + f[8]));
    C ux, uy, t;
    // rho u = m + F/2 with F = F0 + a M lap(mu) u, solved for u, and
    // p = c_s^2/(1 - w_0) [t + rho s_0(u)],  t = sum_{q>0} f_q + u.grad rho / 2,  s_0 = -(3/2) w_0 u^2
    if constexpr (F) {
        const int m = c - 2 * W, g = c - W;  // of the node in the columns of mu and phi
        const C ph = phi * (C(1) / C(12)), d57 = f[5] - f[7], d68 = f[6] - f[8];
        const C r = rcp<C>(fma(C(-0.5), a.aM6 * clap(muA, m, mu2[c]), rho));
        ux = fma(C(-0.5), fma(ph, cgx(muA, m), db * a.n.gx), ((f[1] - f[3]) + d57) - d68) * r;
        uy = fma(C(-0.5), fma(ph, cgy(muD, m), db * a.n.gy), ((f[2] - f[4]) + d57) + d68) * r;
        t = fma(a.a24, fma(ux, cgx(phA, g), uy * cgy(phD, g)), s1);
    } else {
        const C gmx = sgx<C>(mu2, c), gmy = sgy<C>(mu2, c), lap = slap<C>(mu2, c);
        const C grx = op_mul(a.k.a, sgx<C>(s2, c)), gry = op_mul(a.k.a, sgy<C>(s2, c));  // grad rho
        const C F0x = -op_fma(phi, gmx, op_mul(db, a.n.gx)), F0y = -op_fma(phi, gmy, op_mul(db, a.n.gy));
        const C mx = ((f[1] - f[3]) + (f[5] - f[7])) + (f[8] - f[6]);
        const C my = ((f[2] - f[4]) + (f[5] - f[7])) + (f[6] - f[8]);
        const C r = rcp<C>(op_fma(C(-0.5) * a.k.a, op_mul(a.n.M, lap), rho));
        ux = op_mul(op_fma(C(0.5), F0x, mx), r);
        uy = op_mul(op_fma(C(0.5), F0y, my), r);
        t = op_fma(C(0.5), op_fma(ux, grx, op_mul(uy, gry)), s1);
    }
    const C uu = op_fma(ux, ux, op_mul(uy, uy));
    const C pr = op_mul(C(3) / C(5), op_fma(-C(1.5) * wq<C>(0), op_mul(rho, uu), t));
    if (OBS) {
        const long long N = (long long)a.nx * a.ny, k = (long long)y * a.nx + x;
        a.obs[k] = (double)ux;
        a.obs[N + k] = (double)uy;
        a.obs[2 * N + k] = (double)pr;
    } else {
        C* w = a.aux + at<AUXS>(a, x, y);
        w[A_PHI] = phi;
        w[A_UX] = ux;
        w[A_UY] = uy;
        w[A_MU] = mu2[c];
        w[A_P] = pr;
    }
}

// both lattices: collide at x, push to x + c_q (bounce-back at walls).  ONE: tau_g = 1, where the populations g drop out
// of their own collision and are not read
template <typename C, bool ONE>
__global__ void __launch_bounds__(NT, sizeof(C) == 4 ? 4 : 3) collide_kernel(NsArgs<C> a)
{
    constexpr bool F = FOLDED<C>;
    constexpr int NA = F ? H1 * W : 1, NB = F ? TY * W : 1;
    __shared__ C s2[N2], jx2[N2], jy2[N2], mu2[N2], p2[N2], D2[N2];
    __shared__ C jA[NA], jD[NA], muA[NB], muD[NB], phA[NB], phD[NB], pA[NB], pD[NB];
    int x0, y0;
    tile_origin(a.nb, x0, y0);
    const bool model2 = a.model == 2;
    grid_dependency_wait();
    grid_launch_dependents();
    for_region(a, x0, y0, [&](int e, int x, int y) {
        const C* w = a.aux + at<AUXS>(a, x, y);
        const C ph = w[A_PHI];
        s2[e] = ph;
        mu2[e] = w[A_MU];
        p2[e] = w[A_P];
        if (model2) {
            jx2[e] = ph * w[A_UX];
            jy2[e] = ph * w[A_UY];
        }
    });
    __syncthreads();
    if (F) {
        columns(mu2, 2, TY, muA, muD);
        columns(s2, 2, TY, phA, phD);
        columns(p2, 2, TY, pA, pD);
        if (model2)  // of phi ux and phi uy only what their divergence takes
            for (int e = threadIdx.x; e < H1 * W; e += NT) {
                jA[e] = fma(C(4), jx2[e + W], jx2[e + 2 * W] + jx2[e]);
                jD[e] = jy2[e + 2 * W] - jy2[e];
            }
        __syncthreads();
    }
    if (model2)  // D = div(phi u) on tile + 1 (F: 12 D)
        for_inner(a, y0, [&](int e, int c) { D2[e] = F ? cgx(jA, c - W) + cgy(jD, c - W) : sgx<C>(jx2, c) + sgy<C>(jy2, c); });
    __syncthreads();
    if (F && model2) {
        columns(D2, 2, TY, jA, jD);
        __syncthreads();
    }
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX, x = x0 + tx, y = y0 + ty;
    if (x >= a.nx || y >= a.ny) return;
    const int c = (ty + 2) * W + tx + 2;
    const long long o = at<POPS>(a, x, y);
    const C *gk = a.in + o, *fk = gk + 9 * GW, *w = a.aux + at<AUXS>(a, x, y);

    // the node's fields
    const C phi = s2[c], mu = mu2[c], pr = p2[c], ux = w[A_UX], uy = w[A_UY];
    const C rho = op_fma(a.k.a, phi, a.k.b), db = rho - a.n.rbar;
    C pg[9], pf[9];
    // The collision (Eq. LB for g with Eq. geq and the source of Eq. liangFi; the flow's lattice with
    // f_eq and G as above) in pairs of opposite directions: with cu = c.u, s_q = e + o and
    // s_opp = e - o, e = w (9/2 cu^2 - 3/2 u^2), o = 3 w cu; and G = 3 (c - u).(A + o B) for q and
    // 3 (-c - u).(A - o B) for opp, A = (w + e) F + e c_s^2 grad rho, B = F + c_s^2 grad rho.
    // pairs (q, opp q): (1, 3) c = (1, 0); (2, 4) c = (0, 1); (5, 7) c = (1, 1); (6, 8) c = (-1, 1)
    if constexpr (F) {
        // With c.A = w c.F + e c.B and u.A = w u.F + e u.B, and S = 3 (1 - 1/(2 tau_f)), the even and odd parts of a
        // pair's f_eq/tau_f + source are
        //   e (rho/tau_f - S u.B) + o S c.B + w (3 p/tau_f - S u.F)  and  o (rho/tau_f - S u.B) + e S c.B + w S c.F
        const int m = c - 2 * W;
        const C gmx = cgx(muA, m), gmy = cgy(muD, m);
        const C ph = phi * (C(1) / C(12)), po = ph * rcp<C>(rho);
        // -F1 of the Cahn-Hilliard lattice (Eq. t0-phiu), with Eq. mark3 for Model II
        C Fx = po * fma(phi, gmx, cgx(pA, m)), Fy = po * fma(phi, gmy, cgy(pD, m));
        if (model2) {
            Fx = fma(-a.K144, cgx(jA, m), Fx);
            Fy = fma(-a.K144, cgy(jD, m), Fy);
        }
        const C aml = a.aM6 * clap(muA, m, mu);
        const C SFx = a.s3 * fma(aml, ux, -fma(ph, gmx, db * a.n.gx)), SFy = a.s3 * fma(aml, uy, -fma(ph, gmy, db * a.n.gy));
        const C SBx = fma(a.s3a36, cgx(phA, m), SFx), SBy = fma(a.s3a36, cgy(phD, m), SFy);
        const C uu = fma(ux, ux, uy * uy), SuF = fma(ux, SFx, uy * SFy);
        const C E1 = fma(a.n.itauf, rho, -fma(ux, SBx, uy * SBy)), itp = a.itf3 * pr;
        const C P1 = ONE ? phi : a.k.itau * phi, eta = a.ieta * mu;
        const C s0 = uu * C(-2.0 / 3.0);
        const C g0 = fma(P1, s0, fma(C(-5.0 / 9.0), eta, P1));
        pg[0] = ONE ? g0 : fma(a.k.omt, gk[0], g0);
        pf[0] = fma(a.n.omtf, fk[0], fma(s0, E1, fma(C(-5.0 / 9.0), itp, C(-4.0 / 9.0) * SuF)));
        const C W0 = itp - SuF;
        // the terms that a pair takes times its weight, for the axes (w = 1/9) and the diagonals (a quarter of it)
        const C wW = W0 * (C(1) / C(9)), wh = uu * (C(-1) / C(6)), we = eta * (C(1) / C(9));
        const C wSFx = SFx * (C(1) / C(9)), wSFy = SFy * (C(1) / C(9)), wFx = -a.src9 * Fx, wFy = -a.src9 * Fy;
        auto pair = [&](int q, int o_, C w3, C w45, C cu, C h, C we, C wF, C wW, C cB, C wSF) {
            const C o = w3 * cu, e = fma(w45 * cu, cu, h);
            const C Ge = fma(P1, e, we), Go = fma(P1, o, wF);
            pg[q] = ONE ? Ge + Go : fma(a.k.omt, gk[q * GW], Ge + Go);
            pg[o_] = ONE ? Ge - Go : fma(a.k.omt, gk[o_ * GW], Ge - Go);
            const C Fe = fma(e, E1, fma(o, cB, wW)), Fo = fma(o, E1, fma(e, cB, wSF));
            pf[q] = fma(a.n.omtf, fk[q * GW], Fe + Fo);
            pf[o_] = fma(a.n.omtf, fk[o_ * GW], Fe - Fo);
        };
        pair(1, 3, C(1) / C(3), C(0.5), ux, wh, we, wFx, wW, SBx, wSFx);
        pair(2, 4, C(1) / C(3), C(0.5), uy, wh, we, wFy, wW, SBy, wSFy);
        const C q4 = C(0.25), h4 = q4 * wh, e4 = q4 * we, W4 = q4 * wW;
        pair(5, 7, C(1) / C(12), C(0.125), ux + uy, h4, e4, q4 * (wFx + wFy), W4, SBx + SBy, q4 * (wSFx + wSFy));
        pair(6, 8, C(1) / C(12), C(0.125), uy - ux, h4, e4, q4 * (wFy - wFx), W4, SBy - SBx, q4 * (wSFy - wSFx));
    } else {
        const C gmx = sgx<C>(mu2, c), gmy = sgy<C>(mu2, c), lap = slap<C>(mu2, c);
        const C gpx = sgx<C>(p2, c), gpy = sgy<C>(p2, c);
        const C gr3x = op_mul(a.k.a * (C(1) / C(3)), sgx<C>(s2, c));  // c_s^2 grad rho
        const C gr3y = op_mul(a.k.a * (C(1) / C(3)), sgy<C>(s2, c));
        // Cahn-Hilliard force with the flow's pressure (Eq. t0-phiu), plus Eq. mark3 for Model II
        const C por = op_mul(phi, rcp<C>(rho));
        C Fx = op_mul(por, -op_fma(phi, gmx, gpx)), Fy = op_mul(por, -op_fma(phi, gmy, gpy));
        if (model2) {
            Fx = op_fma(a.k.K, sgx<C>(D2, c), Fx);
            Fy = op_fma(a.k.K, sgy<C>(D2, c), Fy);
        }
        // the flow's force F = -phi grad mu - (rho - rbar) g + a M lap(mu) u
        const C aml = op_mul(a.k.a, op_mul(a.n.M, lap));
        const C FFx = op_fma(aml, ux, -op_fma(phi, gmx, op_mul(db, a.n.gx)));
        const C FFy = op_fma(aml, uy, -op_fma(phi, gmy, op_mul(db, a.n.gy)));

        const C itau = a.k.itau, omt = a.k.omt, itauf = a.n.itauf, omtf = a.n.omtf;
        const C src3 = C(3) * a.k.src, srcf3 = C(3) * a.n.srcf;
        const C uu = op_fma(ux, ux, op_mul(uy, uy));
        const C P1 = op_mul(itau, phi), Pf = op_mul(itauf, rho);
        const C ietamu = op_mul(itau, op_mul(a.k.eta, mu)), itfp3 = op_mul(C(3) * itauf, pr);
        const C Bx = FFx + gr3x, By = FFy + gr3y;
        const C uB = op_fma(ux, Bx, op_mul(uy, By));
        const C uF = op_fma(ux, FFx, op_mul(uy, FFy)), ug = op_fma(ux, gr3x, op_mul(uy, gr3y));

        {   // q = 0: s_0 = -(3/2) w_0 u^2, S_0 = 0, G_0 = -3 (Gamma_0 u.F + s_0 u.c_s^2 grad rho)
            const C s0 = op_mul(C(-1.5) * wq<C>(0), uu);
            const C geq = op_fma(phi, s0, op_fma(wq<C>(0) - C(1), op_mul(a.k.eta, mu), phi));
            pg[0] = ONE ? geq : op_fma(omt, gk[0], op_mul(itau, geq));
            const C feq = op_fma(rho, s0, op_mul(C(3) * (wq<C>(0) - C(1)), pr));
            const C G = op_mul(C(-3), op_fma(wq<C>(0) + s0, uF, op_mul(s0, ug)));
            pf[0] = op_fma(omtf, fk[0], op_fma(itauf, feq, op_mul(a.n.srcf, G)));
        }
#pragma unroll
        for (int m = 0; m < 4; m++) {
            const int q = (m == 0) ? 1 : (m == 1) ? 2 : (m == 2) ? 5 : 6, o_ = opp(q);
            const C wt = wq<C>(q);
            const C cu = (m == 0) ? ux : (m == 1) ? uy : (m == 2) ? ux + uy : uy - ux;
            const C cF = (m == 0) ? Fx : (m == 1) ? Fy : (m == 2) ? Fx + Fy : Fy - Fx;
            const C cB = (m == 0) ? Bx : (m == 1) ? By : (m == 2) ? Bx + By : By - Bx;
            const C e = op_fma(op_mul(C(4.5) * wt, cu), cu, op_mul(C(-1.5) * wt, uu));
            const C o = op_mul(C(3) * wt, cu);
            // Cahn-Hilliard lattice: post = (1 - 1/tau) g + g_eq/tau + (1 - 1/(2 tau)) S
            const C Ge = op_fma(P1, e, op_mul(wt, ietamu));
            const C Go = op_fma(P1, o, op_mul(wt * src3, cF));
            pg[q] = ONE ? Ge + Go : op_fma(omt, gk[q * GW], Ge + Go);
            pg[o_] = ONE ? Ge - Go : op_fma(omt, gk[o_ * GW], Ge - Go);
            // the flow's lattice
            const C we = wt + e;
            const C Ax = op_fma(we, FFx, op_mul(e, gr3x)), Ay = op_fma(we, FFy, op_mul(e, gr3y));
            const C cA = (m == 0) ? Ax : (m == 1) ? Ay : (m == 2) ? Ax + Ay : Ay - Ax;
            const C uA = op_fma(ux, Ax, op_mul(uy, Ay));
            const C Fe = op_fma(srcf3, op_fma(o, cB, -uA), op_fma(Pf, e, op_mul(wt, itfp3)));
            const C Fo = op_fma(Pf, o, op_mul(srcf3, op_fma(-o, uB, cA)));
            pf[q] = op_fma(omtf, fk[q * GW], Fe + Fo);
            pf[o_] = op_fma(omtf, fk[o_ * GW], Fe - Fo);
        }
    }
    // element distances to the neighbours: the next node of the group or of the next group, periodic in x and y
    const int E = x == a.nx - 1 ? -((x >> 5) * POPS + (x & 31)) : (x & 31) == 31 ? POPS - 31 : 1;
    const int Wd = x == 0 ? ((a.nx - 1) >> 5) * POPS + ((a.nx - 1) & 31) : (x & 31) == 0 ? 31 - POPS : -1;
    const long long row = (long long)a.nb * POPS;
    C* ko = a.out + o;
    if (a.walls && (y == 0 || y == a.ny - 1)) {  // halfway bounce-back at a wall at rest
#pragma unroll
        for (int q = 0; q < 9; q++) {
            const bool out = y == 0 ? cy(q) < 0 : cy(q) > 0;
            C* d = out ? ko : ko + (cy(q) * row + (cx(q) > 0 ? E : cx(q) < 0 ? Wd : 0));
            const int qd = out ? opp(q) : q;
            d[qd * GW] = pg[q];
            d[(9 + qd) * GW] = pf[q];
        }
    } else {
        C* no = ko + (y == a.ny - 1 ? row - a.ny * row : row);
        C* so = ko + (y == 0 ? a.ny * row - row : -row);
#pragma unroll
        for (int q = 0; q < 9; q++) {
            C* d = (cy(q) > 0 ? no : cy(q) < 0 ? so : ko) + (cx(q) > 0 ? E : cx(q) < 0 ? Wd : 0);
            d[q * GW] = pg[q];
            d[(9 + q) * GW] = pf[q];
        }
    }
}

// phi = sum_q g_q of the current state into its padded phi array (before an observation); one thread per node
template <typename C>
__global__ void phi_kernel(NsArgs<C> a)
{
    const long long N = (long long)a.nx * a.ny;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    const int y = k / a.nx, x = k - y * a.nx;
    a.phi[(long long)(a.row0 + y) * a.pitch + GC + x] = sum_g(a.in + at<POPS>(a, x, y));
}

// initial state: g = g_eq(phi0, mu0, 0), f = f_eq(0, rho(phi0), 0) = 0; phi = phi0
template <typename C>
__global__ void init_kernel(NsArgs<C> a, const double* phi0)
{
    const long long N = (long long)a.nx * a.ny;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    const int y = k / a.nx, x = k - y * a.nx;
    auto phi_at = [&](int dx, int dy) -> double {
        const int2 v = node_at(a.nx, a.ny, a.walls, x + dx, y + dy);
        return phi0[(long long)(a.row0 + v.y) * a.pitch + GC + v.x];
    };
    double c0 = phi_at(0, 0), s = 0.0;
    for (int q = 1; q < 9; q++) s += 2.0 * wq<double>(q) * (phi_at(cx(q), cy(q)) - c0);
    double mu = dfdphi<double>(c0, (double)a.k.beta, (double)a.k.phiA, (double)a.k.phiB) - (double)a.k.kappa * 3.0 * s;
    C* o = a.out + at<POPS>(a, x, y);
    for (int q = 0; q < 9; q++) {
        double geq = (q == 0) ? c0 + (wq<double>(0) - 1.0) * (double)a.k.eta * mu : wq<double>(q) * (double)a.k.eta * mu;
        o[q * GW] = (C)geq;
        o[(9 + q) * GW] = C(0);
    }
    a.phi[(long long)(a.row0 + y) * a.pitch + GC + x] = (C)c0;
}

}  // namespace ns
}  // namespace lbch
