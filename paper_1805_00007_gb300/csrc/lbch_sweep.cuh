// lbch_sweep.cuh -- the step kernel as row sweeps in registers.
//
// Every quantity of the step at a node (mu, D = div(phi u), the gradients, the force, g*) depends only on phi
// within three rows and three columns, so one warp can produce a strip of output rows by sweeping upwards
// through it, one row per iteration, with everything the stencils need held in registers:
//
//   * a warp owns 64 consecutive columns, two per lane (a = 2 lane, b = 2 lane + 1); all but the outermost
//     three or four on each side are output (SweepShape);
//   * the stencils are taken column first (lbch_kernels.cuh): each lane forms the column values of its two
//     columns from the rows in its registers, and what the combination along the row needs of the left
//     neighbour of a and the right neighbour of b comes from the adjacent lanes by shuffles;
//   * the rows below stay in registers: iteration j takes phi of row yf = y0 - 3 + j, computes mu and D of row
//     yf - 1, collides row yf - 2 and completes phi(t+1) of row yf - 3.
//
// At tau_g = 1 (GEN = false), Eq. LB reduces to g* = g_eq + S / 2: the populations are multiplied by 1 - 1/tau = 0,
// so the step maps phi(t) to phi(t+1) = sum_i g*_i(x - c_i) and nothing else is carried between steps.  Streaming
// then needs only sums: the populations 1, 5, 8 that arrive from the column to the left are summed at their source
// node and cross one lane boundary as one number, as do 3, 6, 7 from the right (the grouping of the sum is the one
// the tile kernel uses too).
//
// GEN (any tau_g): the populations are read and written as well.  The warp copies what a step takes -- the populations of
// its collision row, its row of phi, the low part of its output row -- into a ring of slots in shared memory (cp.async), one
// step ahead in float, two in double and half storage (SweepShape::AHEAD; twice as many slots).  After the collision the
// nine g* of a node reach their destinations individually -- 1, 5, 8 from the lane to the left, 3, 6, 7 from the right,
// 2 and 4 from the rows below and above -- and g(t+1) is stored plane by plane.
//
// Division of work.  Every warp is on its own: it loads its rows of phi straight into registers, two rows ahead,
// and no block-wide wait joins it to others, so the length of its strip is free and the host cuts the grid to the
// device -- as many strips as the warps it wants resident, all of one length (sweep_rows).  A strip of R rows
// computes mu on R + 4 rows and collides R + 2: on a large grid R is near a hundred, where tiles of twelve rows per
// warp staged through shared memory computed a third of their mu and a seventh of their collisions twice.  Measured
// against that form (us per step, one GB300; now with the image stores below): 4096^2 tau_g = 0.8 in float 295 -> 248 (5.95
// TB/s of 88 B per update: bound by HBM), half storage 219 -> 136; tau_g = 1 in float 3001 x 1999 53 -> 32.7, 512^2
// 10.4 -> 6.1, 100^2 10.4 -> 3.5, an ensemble of 48 instances with walls 68 -> 26.6 (instruction issue, 77 % busy while an SM
// has work, at 159 instructions per update, of which 102 are the arithmetic).
#pragma once
#include <type_traits>

#include "lbch_kernels.cuh"

namespace lbch {

// One warp's strip: instance, first stored column of its 64, first output row and output rows.
struct SweepItem { int inst, col, y0, rows; };

template <typename C, typename S, typename P>
struct SweepArgs {
    InstDev inst0;          // the record of instance 0, for single-instance handles (read from the parameters)
    const InstDev* inst;
    const SweepItem* items; // several instances: every warp's strip
    const C* tabs;          // velocity tables in the arithmetic type
    int n_items;
    int strips, rows_per;   // a single instance: its strips side by side, and the rows each warp takes of one
    int pitch;
    const P* phi_in;
    const float* lo_in;     // low part of phi on the float-float path
    P* phi_out;
    float* lo_out;
    Ctl* ctl;
    int t_off;              // this launch's step is ctl->time + t_off
    int t_adv;              // when nonzero, the launch's last CTA advances ctl->time by t_adv
    int timed;              // some instance's flow has a time factor
    int read_n;             // the launch reads the step index: Model III, or a time factor without a table
    const double* Tf;       // the instances' time factors at this launch's step, or null (step_T)
    const S* g_in;          // populations (GEN): g[(row * nq + plane) * pitch + column]
    S* g_out;
    const C* H_in;          // M3 (Model III): H(t - 1) of Eq. F2-1's time derivatives, two planes (x, y) of
    C* H_out;               // rows x pitch values; H(t) is written for the warp's own nodes and their images
    long long H_plane;      // values per plane of H
};

// Shape of the sweep.  GEN: 56 output columns, box columns 4 .. 59, whole lanes (2 .. 29): the populations are stored
// in pairs.  Without the populations: 58, box columns 3 .. 60, where lanes 1 and 30 store one node each (3.5 % fewer
// strips for one more store per row; with nine planes the extra stores cost what the width gains).
template <typename S, typename P, bool FF, bool GEN, bool WIDE>
struct SweepShape {
    // warps per block, at most (lbch_sweep_launch.cuh), and resident blocks of that many: 16 warps per SM in float (128
    // registers a thread), 12 where the populations meet walls or several instances, 8 in double
    static constexpr int NW = sizeof(P) == 4 && !WIDE ? 16 : 4;
    static constexpr int BLOCKS = sizeof(P) == 8 ? 2 : WIDE ? 3 : 1;
    static constexpr int W = GEN ? 56 : 58;            // output columns of a strip
    static constexpr int BW = 64;                      // columns of a strip with its halo, two per lane
    static constexpr int FIRST = GEN ? 4 : 3;          // first output column among them
    static constexpr int LEAD = GEN ? 0 : 1;           // domain columns the first strip starts before column 0
    static constexpr int NQ = sizeof(S) == 2 ? 8 : 9;  // stored population planes
    // Rows under way per warp.  In float the step is bound by HBM, which serves 16 warps per SM best with one row each
    // under way (4096^2, us per step: 248 with one, 269 with two); the others hide latency with two (half storage: 153 with
    // one, 136 with two).
    static constexpr int AHEAD = FF ? 1 : 2;
    static constexpr int RING = 2 * AHEAD;             // ring slots per warp: a power of two above AHEAD
    static constexpr size_t SLOT = (size_t)NQ * BW * sizeof(S) + BW * sizeof(P) + (FF ? BW * 4 : 0);
    static constexpr size_t RING_BYTES = GEN ? RING * SLOT : 0;  // per warp
    __host__ __device__ static constexpr size_t bytes(int warps) { return GEN ? warps * RING_BYTES + 128 : 0; }
};

template <typename P> struct Pair;
template <> struct Pair<float> { using T = float2; };
template <> struct Pair<double> { using T = double2; };
template <> struct Pair<__half> { using T = __half2; };

template <typename C, typename S2> __device__ __forceinline__ void unpair(S2 v, C& x, C& y) { x = cvt<C>(v.x); y = cvt<C>(v.y); }
template <typename C> __device__ __forceinline__ void unpair(__half2 v, C& x, C& y)
{
    x = (C)__low2float(v);
    y = (C)__high2float(v);
}
template <typename S, typename C> __device__ __forceinline__ typename Pair<S>::T mkpair(C x, C y)
{
    typename Pair<S>::T v;
    v.x = (S)x;
    v.y = (S)y;
    return v;
}
template <> __device__ __forceinline__ __half2 mkpair<__half, float>(float x, float y) { return __floats2half2_rn(x, y); }

template <typename C> __device__ __forceinline__ C from_left(C v) { return __shfl_up_sync(0xffffffffu, v, 1); }
template <typename C> __device__ __forceinline__ C from_right(C v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// 16 bytes from global into shared memory (both aligned to 16), past the L1 cache: rows under way would need more of
// it than the rings leave (with copies of 8 bytes through L1 the step at 4096^2 took 334 us in float).
__device__ __forceinline__ void copy_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K> __device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory"); }

// One row of the sweep.  A slot is reused every third row, so each field lives at most three rows.
template <typename C>
struct SwRow {
    C pa, pb;                      // phi
    C ma, mb;                      // mu
    C da, db;                      // D = div(phi u)
    C y1, y2;                      // the Y velocity tables of the row
    C u5a, u5b, u2a, u2b, u6a, u6b;         // g*_5, a quarter of g*_2, g*_6 of the row: they stream to the row above
    C Ra, Rb, Ca, Cb, La, Lb, v0a, v0b;     // partial sums of the populations arriving at the row (C in a quarter)
    C n0a, n0b, n1a, n1b, n2a, n2b, n3a, n3b, n4a, n4b, n5a, n5b, n6a, n6b, n7a, n7b, n8a, n8b;  // GEN: g(t+1) of the row
};

// Writes phi(t+1) of domain node (x, y) into the ghost cells that stand for it (periodic images in x;
// periodic or mirror images in y, three deep).
template <typename P>
__device__ __forceinline__ void store_images(P* phi_out, long long row0, int pitch, int nx, int ny, int walls, int x,
                                             int y, P v)
{
    if (x >= 3 && x < nx - 3 && y >= 3 && y < ny - 3) return;
    for_images3(x, y, nx, ny, walls, [&](int xx, int yy) { phi_out[(row0 + yy) * pitch + GC + xx] = v; });
}

// Writes g(t+1) of domain node (x, y) into the ghost cells that stand for it, one deep: periodic images
// in x, and in y unless the instance has walls there.
template <typename S, typename C, int QOFF>
__device__ __forceinline__ void store_g_images(S* g_out, long long row0, int pitch, int nx, int ny, int walls, int x, int y,
                                               const C* v)
{
    constexpr int NQ = 9 - QOFF;
    for_images1(x, y, nx, ny, walls, [&](int xx, int yy) {
        S* o = g_out + ((row0 + yy) * NQ) * pitch + GC + xx;
#pragma unroll
        for (int q = QOFF; q < 9; q++) o[(long long)(q - QOFF) * pitch] = to_s<S>(v[q]);
    });
}

// SINGLE (a handle of one instance): the instance record stays in the launch parameters, and the arithmetic takes
// its constants as constant-bank operands; otherwise each warp reads those of its strip's instance from shared memory.
// WALLS: some instance has walls in y (bounce-back rows and the mirror substitution of mu and D next to them, a
// few warp-uniform tests per row).  M3: some instance uses Model III (the complete diffusive-scale force of Eq. F2-1):
// at every collision the force takes the backward difference of H over one step (reading R15), with H(t - 1) read at
// the collided node and H(t) stored for the warp's own nodes, as the tile kernel does.
// The warp's index is broadcast from its first lane, by which the compiler knows that everything derived from it --
// the strip, row pointers, the tests on rows -- is the same for the warp, and keeps and computes it once per warp rather
// than per lane.
template <typename C, typename S, typename P, bool FF, bool GEN, bool SINGLE, bool WALLS, bool M3>
__global__ void __launch_bounds__(SweepShape<S, P, FF, GEN, GEN && (WALLS || !SINGLE)>::NW * 32,
                                  SweepShape<S, P, FF, GEN, GEN && (WALLS || !SINGLE)>::BLOCKS)
    ch_sweep_kernel(const __grid_constant__ SweepArgs<C, S, P> a)
{
    using L = SweepShape<S, P, FF, GEN, GEN && (WALLS || !SINGLE)>;
    using P2 = typename Pair<P>::T;
    using S2 = typename Pair<S>::T;
    constexpr int BW = L::BW, NQ = L::NQ, RING = L::RING;
    constexpr bool kShift = sizeof(C) == 4;     // float arithmetic on g_0 - phi
    constexpr bool kHalf = sizeof(S) == 2;      // half storage: g_0 not stored (implied by phi)
    constexpr int QOFF = kHalf ? 1 : 0;         // stored plane of population q is q - QOFF

    extern __shared__ unsigned char smem_raw[];
    __shared__ InstDev s_I[SINGLE ? 1 : L::NW];  // each warp's instance (several instances)
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
    const int item = (int)(blockIdx.x * (blockDim.x >> 5)) + warp;
    const bool mine = item < a.n_items;

    // the strip, and this lane's velocity tables for it (constant data, read before the dependency wait): X by
    // stored column (clamped: the clamped columns feed halo lanes only), Y by row, one row per lane, 32 rows at a time
    int k_t = 0, col0 = 0, y0 = 0, R = 0;
    if (mine) {
        if constexpr (SINGLE) {
            const int chunk = item / a.strips;
            col0 = (item - chunk * a.strips) * L::W;
            y0 = chunk * a.rows_per;
            R = min(a.rows_per, a.inst0.ny - y0);
        } else {
            const SweepItem it = a.items[item];
            k_t = it.inst; col0 = it.col; y0 = it.y0; R = it.rows;
        }
    }
    if constexpr (!SINGLE) {
        const int* src = reinterpret_cast<const int*>(a.inst + k_t);
        int* dst = reinterpret_cast<int*>(&s_I[warp]);
        for (int w = lane; w < (int)(sizeof(InstDev) / 4); w += 32) dst[w] = src[w];
        __syncwarp();
    }
    const InstDev& I = SINGLE ? a.inst0 : s_I[warp];
    const Consts<C>& K0 = consts<C>(I);
    const int pitch = a.pitch;
    const C* tX1 = a.tabs + I.tab;
    const C* tY1 = tX1 + 2 * pitch;
    const int col = min(col0 + 2 * lane, pitch - 2);  // stored column of node a
    const C X1a = tX1[col], X1b = tX1[col + 1], X2a = tX1[pitch + col], X2b = tX1[pitch + col + 1];
    auto y_row = [&](int j) { return min(y0 + j + lane, I.ylen - 1); };  // domain row y0 - 3 + j + lane, GR = 3 rows up
    C ly1 = tY1[y_row(0)], ly2 = tY1[I.ylen + y_row(0)];

    // Launched as a programmatic dependent of the previous step: nothing that step writes (phi, the step
    // counter) is read before this wait.
    grid_dependency_wait();
    grid_launch_dependents();
    const long long n = a.read_n ? a.ctl->time + a.t_off : 0;
    const C T = a.timed ? (C)step_T(a.Tf, k_t, I, n) : C(1);

    if (mine) {
        const bool model2 = M3 ? I.model >= 2 : I.model == 2;  // D = div(phi u) is needed (Models II, III)
        [[maybe_unused]] const bool model3 = M3 && I.model == 3;
        [[maybe_unused]] const bool first = M3 && n == 0;  // no H(t - 1) at the first step
        const int xa = col0 - GC + 2 * lane, xb = xa + 1;  // domain columns
        // the lane's output nodes: box columns FIRST .. FIRST + W - 1 inside the domain
        const bool va = 2 * lane >= L::FIRST && 2 * lane < L::FIRST + L::W && xa >= 0 && xa < I.nx;
        const bool vb = 2 * lane + 1 >= L::FIRST && 2 * lane + 1 < L::FIRST + L::W && xb >= 0 && xb < I.nx;
        const bool both = va && vb, one = va != vb;
        // whether a node of the strip has ghost images in x (three columns from the domain's edge): the image stores
        // and their tests are skipped as a whole elsewhere.  A row that has no images in y takes its nodes' one image at
        // a distance the lane knows (iwa, iwb; GEN: gwa, gwb; 0: none); the other rows, and domains so narrow that a node
        // may have two images in x, take the general way.  (With the general way on every row of these strips, the SMs
        // that held them took 99 thousand cycles at 3001 x 1999 where the average took 75.)
        const bool ximg = col0 - GC + L::FIRST < 3 || col0 - GC + L::FIRST + L::W > I.nx - 3;
        const bool narrow = I.nx < 6;
        auto image = [&](bool v, int x, int deep) { return !v ? 0 : x < deep ? I.nx : x >= I.nx - deep ? -I.nx : 0; };
        const int iwa = image(va, xa, 3), iwb = image(vb, xb, 3);
        [[maybe_unused]] const int gwa = GEN ? image(va, xa, 1) : 0, gwb = GEN ? image(vb, xb, 1) : 0;
        const int wlo = WALLS && I.walls ? 0 : -1000000, whi = WALLS && I.walls ? I.ny - 1 : -1000000;  // wall rows
        const int row0 = I.row0, ylast = I.ny - 3;
        const C* tW = tY1 + 2 * I.ylen;  // Y1, Y2 at the walls y = -1/2, ny - 1/2

        // Every lane's own columns of the rows below, by pointers that advance a row at a time.  Past the strip's last
        // row they run on for up to three rows, which the arrays have to spare.  The output pointers of a lane with one output
        // node point at that node.
        const long long first_in = (long long)(row0 + y0 - 3) * pitch + col;
        const long long first_out = (long long)(row0 + y0) * pitch + col + (one && vb ? 1 : 0);
        const P* pin = a.phi_in + first_in;
        [[maybe_unused]] const float* lin = FF ? a.lo_in + first_in + 3 * pitch : nullptr;
        P* pout = a.phi_out + first_out;
        [[maybe_unused]] float* lout = FF ? a.lo_out + first_out : nullptr;
        [[maybe_unused]] S* gout = GEN ? a.g_out + ((long long)(row0 + y0) * NQ) * pitch + col + (one && vb ? 1 : 0) : nullptr;

        // Without the populations: phi comes straight into registers two rows ahead of its use and its low part one row
        // (a row takes about a microsecond with 16 warps on an SM, more than the latency of HBM), into registers that
        // the unrolled rows rename: a move of a value under way would wait for it.
        auto load_phi = [&]() {
            const P2 v = *reinterpret_cast<const P2*>(pin);
            pin += pitch;
            return v;
        };
        auto load_lo = [&]() {
            const float2 v = *reinterpret_cast<const float2*>(lin);
            lin += pitch;
            return v;
        };

        // GEN: a ring of rows in shared memory, a slot per row ([slot][plane][64 columns]: the populations, then phi, then
        // its low part).  Step j copies what step j + AHEAD takes: the populations of its collision row, its row of phi and
        // the low part of its output row, as one group in pieces of 16 bytes dealt out over the lanes.  At its head, step
        // j waits for the group it takes and the warp meets, which also says that every lane is done with the slot
        // about to be filled.
        constexpr int CH = BW * (int)sizeof(S) / 16, CP = BW * (int)sizeof(P) / 16;  // pieces of a plane's, phi's row
        constexpr int PIECES = NQ * CH;
        [[maybe_unused]] unsigned char* ring = smem_aligned128(smem_raw) + warp * L::RING_BYTES;
        [[maybe_unused]] const unsigned char *gsrc = nullptr, *psrc = nullptr;  // the lane's first piece of the next rows
        if constexpr (GEN) {
            const int gc = min(col0 + lane % CH * (16 / (int)sizeof(S)), pitch - 16 / (int)sizeof(S));
            gsrc = reinterpret_cast<const unsigned char*>(
                a.g_in + ((long long)(row0 + y0 - 1) * NQ + lane / CH) * pitch + gc);  // collision row of step 4
            const int pc = min(col0 + lane % CP * (16 / (int)sizeof(P)), pitch - 16 / (int)sizeof(P));
            // lanes past a row of phi bring its low part, whose rows are three behind
            if (FF && lane >= CP) psrc = reinterpret_cast<const unsigned char*>(a.lo_in + (long long)(row0 + y0 - 6) * pitch + pc);
            else psrc = reinterpret_cast<const unsigned char*>(a.phi_in + (long long)(row0 + y0 - 3) * pitch + pc);
        }
        auto fetch = [&](int j, bool g) {
            if constexpr (GEN) {
                unsigned char* dst = ring + (j & (RING - 1)) * L::SLOT + lane * 16;
                if (lane < CP || (FF && g && j >= 6 - L::AHEAD)) copy_async16(dst + PIECES * 16, psrc);
                psrc += (long long)pitch * sizeof(P);
                if (g) {
#pragma unroll
                    for (int i = 0; i < PIECES; i += 32)
                        if (i + 32 <= PIECES || lane < PIECES - i)
                            copy_async16(dst + i * 16, gsrc + (long long)(i / CH) * pitch * sizeof(S));
                    gsrc += (long long)NQ * pitch * sizeof(S);
                }
                copy_commit();
            }
        };
        if constexpr (GEN) {
#pragma unroll
            for (int j = -L::AHEAD; j < 0; j++) fetch(j, false);  // phi of the first steps
        }

        // One row: A is the slot of row yf (it held yf - 3), B of row yf - 1, Cs of row yf - 2: mu and D of row yf - 1,
        // the collision of row yf - 2, phi(t+1) of row yf - 3 (each once the pipeline has filled that far).
        // steady: the pipeline is full (j >= 6), known at compile time.
        // qc: phi of row yf, qn: takes that of row yf + 2; lc: the low part of phi of the output row, ln: takes the next.
        auto row_step = [&](auto steady, const int j, SwRow<C>& A, SwRow<C>& B, SwRow<C>& Cs, P2& qc, P2& qn, float2& lc,
                            float2& ln) {
            constexpr bool FULL = decltype(steady)::value;
            const int yf = y0 - 3 + j;
            if ((j & 31) == 0) {  // the Y tables (times T) of the next 32 rows
                if (j > 0) {
                    ly1 = tY1[y_row(j)];
                    ly2 = tY1[I.ylen + y_row(j)];
                }
                ly1 = op_mul(ly1, T);
                ly2 = op_mul(ly2, T);
            }
            [[maybe_unused]] const C ha = A.pa, hb = A.pb;  // phi(t) of the output row yf - 3
            if constexpr (GEN) {
                copy_wait<L::AHEAD - 1>();
                __syncwarp();
                const P* ps = reinterpret_cast<const P*>(ring + ((j - L::AHEAD) & (RING - 1)) * L::SLOT + PIECES * 16) + 2 * lane;
                qc = *reinterpret_cast<const P2*>(ps);
                if constexpr (FF) lc = *reinterpret_cast<const float2*>(ps + BW);
                fetch(j, j >= 4 - L::AHEAD && j <= R + 5 - L::AHEAD);
            } else {
                qn = load_phi();
                if (FF && (FULL || j >= 5)) ln = load_lo();
            }
            A.pa = cvt<C>(qc.x);
            A.pb = cvt<C>(qc.y);
            A.y1 = __shfl_sync(0xffffffffu, ly1, j & 31);
            A.y2 = __shfl_sync(0xffffffffu, ly2, j & 31);
            if (FULL || j >= 2) {
                C dla, dlb;
                const C za = node_z(Cs.pa, B.pa, A.pa, dla), zb = node_z(Cs.pb, B.pb, A.pb, dlb);
                const C zL = from_left(zb), zR = from_right(za);
                B.ma = node_mu(B.pa, dla, za, zb, zL, K0);
                B.mb = node_mu(B.pb, dlb, zb, zR, za, K0);
                if (model2) {
                    const C y14 = op_mul(C(4), B.y1);
                    C Ea, Wa, Eb, Wb;
                    const C fa = node_flux(Cs.pa, B.pa, A.pa, X1a, X2a, Cs.y1, y14, A.y1, Cs.y2, A.y2, Ea, Wa);
                    const C fb = node_flux(Cs.pb, B.pb, A.pb, X1b, X2b, Cs.y1, y14, A.y1, Cs.y2, A.y2, Eb, Wb);
                    B.da = node_div(fa, Eb, from_left(Wb));
                    B.db = node_div(fb, from_right(Ea), Wa);
                }
            }
            const int yc = yf - 2;
            [[maybe_unused]] C p8a = C(0), p8b = C(0), p7a = C(0), p7b = C(0), p4a = C(0), p4b = C(0);
            if (FULL || j >= 4) {
                // GEN: the populations g(t) of row yc (collision row j - 4 of the strip)
                C ga[9], gb[9];
                if constexpr (GEN) {
                    const S* rg = reinterpret_cast<const S*>(ring + ((j - L::AHEAD) & (RING - 1)) * L::SLOT) + 2 * lane;
                    if constexpr (kHalf) {
                        C resta = C(0), restb = C(0);
#pragma unroll
                        for (int q = 1; q < 9; q++) {
                            unpair(*reinterpret_cast<const S2*>(rg + (q - 1) * BW), ga[q], gb[q]);
                            resta += ga[q];
                            restb += gb[q];
                        }
                        ga[0] = -resta;  // g_0 - phi
                        gb[0] = -restb;
                    } else {
#pragma unroll
                        for (int q = 0; q < 9; q++) unpair(*reinterpret_cast<const S2*>(rg + q * BW), ga[q], gb[q]);
                    }
                }
                if constexpr (WALLS) {
                    // next to a wall, mu and D of the ghost row take the values of the mirror row (yc); the ghost
                    // row's own values are used by no other node.  (The ghost rows themselves are collided too, for
                    // nothing: what would stream from them is replaced below.)
                    if (yc == wlo) { A.ma = Cs.ma; A.mb = Cs.mb; A.da = Cs.da; A.db = Cs.db; }
                    if (yc == whi) { B.ma = Cs.ma; B.mb = Cs.mb; B.da = Cs.da; B.db = Cs.db; }
                }
                // 12 grad of the pair (a, b), from the column values w and d of both and of their neighbours
                auto grad_pair = [&](C sa_, C ca_, C na_, C sb_, C cb_, C nb_, C& gxa, C& gya, C& gxb, C& gyb) {
                    const C wa = node_w(sa_, ca_, na_), wb = node_w(sb_, cb_, nb_), da = na_ - sa_, db = nb_ - sb_;
                    gxa = wb - from_left(wb);
                    gxb = from_right(wa) - wa;
                    gya = node_gy(from_left(db), da, db);
                    gyb = node_gy(da, db, from_right(da));
                };
                C gmxa, gmya, gmxb, gmyb, gDxa = C(0), gDya = C(0), gDxb = C(0), gDyb = C(0);
                grad_pair(A.ma, Cs.ma, B.ma, A.mb, Cs.mb, B.mb, gmxa, gmya, gmxb, gmyb);
                if (model2) grad_pair(A.da, Cs.da, B.da, A.db, Cs.db, B.db, gDxa, gDya, gDxb, gDyb);
                const C uxa = node_u(X1a, Cs.y1), uya = node_u(X2a, Cs.y2);
                const C uxb = node_u(X1b, Cs.y1), uyb = node_u(X2b, Cs.y2);
                C Pxa, Pya, Pxb, Pyb, Jxa, Jya, Jxb, Jyb;
                node_flow(Cs.pa, uxa, uya, K0, Pxa, Pya);
                node_flow(Cs.pb, uxb, uyb, K0, Pxb, Pyb);
                if (M3 && model3) {
                    // H(t - 1) at the collided nodes: rows -1 .. ny hold it (images one deep); other rows
                    // and columns past the stored ones collide for no output and read nothing
                    const bool hrow = !first && yc >= -1 && yc <= I.ny;
                    const int sa = col0 + 2 * lane;
                    const long long hn = (long long)(row0 + yc) * pitch + sa;
                    const C Hpxa = hrow && sa < pitch ? a.H_in[hn] : C(0);
                    const C Hpya = hrow && sa < pitch ? a.H_in[a.H_plane + hn] : C(0);
                    const C Hpxb = hrow && sa + 1 < pitch ? a.H_in[hn + 1] : C(0);
                    const C Hpyb = hrow && sa + 1 < pitch ? a.H_in[a.H_plane + hn + 1] : C(0);
                    C Hxa, Hya, Hxb, Hyb;
                    node_force_full(Cs.pa, gmxa, gmya, gDxa, gDya, Hpxa, Hpya, first, Pxa, Pya, K0, Jxa, Jya, Hxa, Hya);
                    node_force_full(Cs.pb, gmxb, gmyb, gDxb, gDyb, Hpxb, Hpyb, first, Pxb, Pyb, K0, Jxb, Jyb, Hxb, Hyb);
                    if (yc >= y0 && yc < y0 + R) {  // the warp's own nodes
                        if (va) store_h(a.H_out, a.H_plane, row0, pitch, I.nx, I.ny, I.walls, xa, yc, Hxa, Hya);
                        if (vb) store_h(a.H_out, a.H_plane, row0, pitch, I.nx, I.ny, I.walls, xb, yc, Hxb, Hyb);
                    }
                } else {
                    node_force(Cs.pa, gmxa, gmya, gDxa, gDya, Pxa, Pya, model2, K0, Jxa, Jya);
                    node_force(Cs.pb, gmxb, gmyb, gDxb, gDyb, Pxb, Pyb, model2, K0, Jxb, Jyb);
                }
                C pa_[9], pb_[9];  // without the populations: 1..4 in a quarter
                collide9<C, !GEN>(Cs.ma, uxa, uya, Pxa, Pya, Jxa, Jya, ga, K0, pa_);
                collide9<C, !GEN>(Cs.mb, uxb, uyb, Pxb, Pyb, Jxb, Jyb, gb, K0, pb_);
                if constexpr (!kShift) {
                    pa_[0] = rest_add(pa_[0], Cs.pa, K0);
                    pb_[0] = rest_add(pb_[0], Cs.pb, K0);
                }
                if constexpr (GEN && kHalf) {
                    // the streamed populations are stored in half: they travel rounded.  g*_0 stays at the
                    // node, in float, and takes what the rounded ones leave of phi (g*_0 - phi = -sum of
                    // the rounded g*_q, q > 0), so that the rounding moves no phi between nodes: sum phi is
                    // kept exactly as in the other precisions (the same sum in the same order as the tile
                    // kernel forms)
                    C resta = C(0), restb = C(0);
#pragma unroll
                    for (int q = 1; q < 9; q++) {
                        const float2 v = __half22float2(__floats2half2_rn((float)pa_[q], (float)pb_[q]));
                        pa_[q] = (C)v.x;
                        pb_[q] = (C)v.y;
                        resta += pa_[q];
                        restb += pb_[q];
                    }
                    pa_[0] = -resta;
                    pb_[0] = -restb;
                }
                if constexpr (GEN) {
                    // g*_q reaches node x + c_q: the row above takes 2, 5, 6; this row 0, 1, 3; the row
                    // below 4, 7, 8 (1, 5, 8 from the lane to the left, 3, 6, 7 from the right)
                    B.n2a = pa_[2]; B.n2b = pb_[2];
                    B.n5a = from_left(pb_[5]); B.n5b = pa_[5];
                    B.n6a = pb_[6]; B.n6b = from_right(pa_[6]);
                    Cs.n0a = pa_[0]; Cs.n0b = pb_[0];
                    Cs.n1a = from_left(pb_[1]); Cs.n1b = pa_[1];
                    Cs.n3a = pb_[3]; Cs.n3b = from_right(pa_[3]);
                    A.n4a = pa_[4]; A.n4b = pb_[4];
                    A.n7a = pb_[7]; A.n7b = from_right(pa_[7]);
                    A.n8a = from_left(pb_[8]); A.n8b = pa_[8];
                    if constexpr (WALLS) {
                        // bottom wall: 2, 5, 6 of this row bounce back at the node.  Top wall: 4, 7, 8 likewise, kept
                        // in the row's slot until the ghost row above it has been collided, whose share they replace
                        if (yc == wlo) {
                            const C uwa = wall_u(X1a, tW[0], T), vwa = wall_u(X2a, tW[2], T);
                            const C uwb = wall_u(X1b, tW[0], T), vwb = wall_u(X2b, tW[2], T);
                            Cs.n2a = bounce<C, 2>(pa_[4], Cs.pa, uwa, vwa); Cs.n2b = bounce<C, 2>(pb_[4], Cs.pb, uwb, vwb);
                            Cs.n5a = bounce<C, 5>(pa_[7], Cs.pa, uwa, vwa); Cs.n5b = bounce<C, 5>(pb_[7], Cs.pb, uwb, vwb);
                            Cs.n6a = bounce<C, 6>(pa_[8], Cs.pa, uwa, vwa); Cs.n6b = bounce<C, 6>(pb_[8], Cs.pb, uwb, vwb);
                        }
                        if (yc == whi) {
                            const C uwa = wall_u(X1a, tW[1], T), vwa = wall_u(X2a, tW[3], T);
                            const C uwb = wall_u(X1b, tW[1], T), vwb = wall_u(X2b, tW[3], T);
                            Cs.Ca = bounce<C, 4>(pa_[2], Cs.pa, uwa, vwa); Cs.Cb = bounce<C, 4>(pb_[2], Cs.pb, uwb, vwb);
                            Cs.La = bounce<C, 7>(pa_[5], Cs.pa, uwa, vwa); Cs.Lb = bounce<C, 7>(pb_[5], Cs.pb, uwb, vwb);
                            Cs.Ra = bounce<C, 8>(pa_[6], Cs.pa, uwa, vwa); Cs.Rb = bounce<C, 8>(pb_[6], Cs.pb, uwb, vwb);
                        }
                        if (yf - 3 == whi) {
                            A.n4a = A.Ca; A.n4b = A.Cb; A.n7a = A.La; A.n7b = A.Lb; A.n8a = A.Ra; A.n8b = A.Rb;
                        }
                    }
                } else {
                    if constexpr (WALLS) {
                        if (yc == wlo) {
                            // bottom wall row: 2, 5, 6 bounce back at the node.  They take the place of what would
                            // stream in from the ghost row (slot A), at the column it would leave from
                            const C uwa = wall_u(X1a, tW[0], T), vwa = wall_u(X2a, tW[2], T);
                            const C uwb = wall_u(X1b, tW[0], T), vwb = wall_u(X2b, tW[2], T);
                            const C b5a = bounce<C, 5>(pa_[7], Cs.pa, uwa, vwa), b5b = bounce<C, 5>(pb_[7], Cs.pb, uwb, vwb);
                            const C b6a = bounce<C, 6>(pa_[8], Cs.pa, uwa, vwa), b6b = bounce<C, 6>(pb_[8], Cs.pb, uwb, vwb);
                            A.u5a = b5b; A.u5b = from_right(b5a);
                            A.u6b = b6a; A.u6a = from_left(b6b);
                            A.u2a = op_mul(C(0.25), bounce<C, 2>(op_mul(C(4), pa_[4]), Cs.pa, uwa, vwa));
                            A.u2b = op_mul(C(0.25), bounce<C, 2>(op_mul(C(4), pb_[4]), Cs.pb, uwb, vwb));
                        }
                    }
                    // (g_1 + g_5) and (g_3 + g_6) at their source nodes; g_2 (a quarter of it) from the row below
                    Cs.Ra = op_fma(C(4), pa_[1], A.u5a); Cs.Rb = op_fma(C(4), pb_[1], A.u5b);
                    Cs.La = op_fma(C(4), pa_[3], A.u6a); Cs.Lb = op_fma(C(4), pb_[3], A.u6b);
                    Cs.Ca = A.u2a; Cs.Cb = A.u2b;
                    Cs.v0a = pa_[0]; Cs.v0b = pb_[0];
                    p8a = pa_[8]; p8b = pb_[8];
                    p7a = pa_[7]; p7b = pb_[7];
                    p4a = pa_[4]; p4b = pb_[4];
                    if constexpr (WALLS) {
                        // top wall: what the ghost row (just collided) would stream into the output row (slot A) is
                        // replaced by that row's own 2, 5, 6 bounced back, at the column it would leave from
                        if (yf - 3 == whi) {
                            const C uwa = wall_u(X1a, tW[1], T), vwa = wall_u(X2a, tW[3], T);
                            const C uwb = wall_u(X1b, tW[1], T), vwb = wall_u(X2b, tW[3], T);
                            const C e7a = bounce<C, 7>(A.u5a, ha, uwa, vwa), e7b = bounce<C, 7>(A.u5b, hb, uwb, vwb);
                            const C e8a = bounce<C, 8>(A.u6a, ha, uwa, vwa), e8b = bounce<C, 8>(A.u6b, hb, uwb, vwb);
                            p8a = e8b; p8b = from_right(e8a);
                            p7b = e7a; p7a = from_left(e7b);
                            p4a = op_mul(C(0.25), bounce<C, 4>(op_mul(C(4), A.u2a), ha, uwa, vwa));
                            p4b = op_mul(C(0.25), bounce<C, 4>(op_mul(C(4), A.u2b), hb, uwb, vwb));
                        }
                    }
                    Cs.u5a = pa_[5]; Cs.u5b = pb_[5];
                    Cs.u2a = pa_[2]; Cs.u2b = pb_[2];
                    Cs.u6a = pa_[6]; Cs.u6b = pb_[6];
                }
            }
            if (!FULL && j < 6) return;
            // phi(t+1) -- GEN: and g(t+1) -- of row yo = yf - 3 (slot A): every population has arrived
            const int yo = yf - 3;
            C suma, sumb, v0a, v0b;
            if constexpr (GEN) {
                suma = stream_sum(A.n1a, A.n2a, A.n3a, A.n4a, A.n5a, A.n6a, A.n7a, A.n8a);
                sumb = stream_sum(A.n1b, A.n2b, A.n3b, A.n4b, A.n5b, A.n6b, A.n7b, A.n8b);
                v0a = A.n0a;
                v0b = A.n0b;
            } else {
                // the sums from the left and the right cross their lane boundary; the grouping of stream_sum
                const C Rsa = A.Ra + p8a, Rsb = A.Rb + p8b, Lsa = A.La + p7a, Lsb = A.Lb + p7b;
                suma = op_fma(C(4), A.Ca + p4a, from_left(Rsb)) + Lsb;
                sumb = op_fma(C(4), A.Cb + p4b, Rsa) + from_right(Lsa);
                v0a = A.v0a;
                v0b = A.v0b;
            }
            P hia, hib;
            float loa = 0.0f, lob = 0.0f;
            [[maybe_unused]] C g0a = v0a, g0b = v0b;  // the stored rest population
            if constexpr (FF) {
                // phi(t+1) = phi(t) + (g*_0 - phi(t)) + sum_{q>0}; hi + lo absorbs it exactly (TwoSum)
                {
                    const float h = (float)ha, tt = lc.x + (float)(v0a + suma);
                    const float sm = h + tt, bb = sm - h;
                    loa = (h - (sm - bb)) + (tt - bb);
                    hia = (P)sm;
                }
                {
                    const float h = (float)hb, tt = lc.y + (float)(v0b + sumb);
                    const float sm = h + tt, bb = sm - h;
                    lob = (h - (sm - bb)) + (tt - bb);
                    hib = (P)sm;
                }
                g0a = -suma;  // g_0 - phi(t+1) = -sum_{q>0} g_q(t+1)
                g0b = -sumb;
            } else if constexpr (kShift) {
                hia = (P)((float)ha + (float)(v0a + suma));
                hib = (P)((float)hb + (float)(v0b + sumb));
            } else {
                hia = (P)(v0a + suma);
                hib = (P)(v0b + sumb);
            }
            if (both) {
                P2 o;
                o.x = hia;
                o.y = hib;
                *reinterpret_cast<P2*>(pout) = o;
                if (FF) *reinterpret_cast<float2*>(lout) = make_float2(loa, lob);
            }
            if (one) {
                *pout = va ? hia : hib;
                if (FF) *lout = va ? loa : lob;
            }
            const bool images = yo < 3 || yo >= ylast || (ximg && narrow);  // the general way
            if (ximg && !images) {
                if (iwa) pout[iwa] = hia;
                if (iwb) pout[iwb + (both ? 1 : 0)] = hib;
            }
            pout += pitch;
            if (FF) lout += pitch;
            if constexpr (GEN) {
                const C va_[9] = {g0a, A.n1a, A.n2a, A.n3a, A.n4a, A.n5a, A.n6a, A.n7a, A.n8a};
                const C vb_[9] = {g0b, A.n1b, A.n2b, A.n3b, A.n4b, A.n5b, A.n6b, A.n7b, A.n8b};
                if (both) {
#pragma unroll
                    for (int q = QOFF; q < 9; q++)
                        *reinterpret_cast<S2*>(gout + (long long)(q - QOFF) * pitch) = mkpair<S>(va_[q], vb_[q]);
                }
                if (one) {  // the last column of an odd nx
#pragma unroll
                    for (int q = QOFF; q < 9; q++) gout[(long long)(q - QOFF) * pitch] = to_s<S>(va_[q]);
                }
                if (ximg && !images) {
                    if (gwa) {
                        S* o = gout + gwa;
#pragma unroll
                        for (int q = QOFF; q < 9; q++) o[(long long)(q - QOFF) * pitch] = to_s<S>(va_[q]);
                    }
                    if (gwb) {
                        S* o = gout + gwb + (both ? 1 : 0);
#pragma unroll
                        for (int q = QOFF; q < 9; q++) o[(long long)(q - QOFF) * pitch] = to_s<S>(vb_[q]);
                    }
                }
                gout += NQ * pitch;
                if (images) {
                    if (va) store_g_images<S, C, QOFF>(a.g_out, row0, pitch, I.nx, I.ny, I.walls, xa, yo, va_);
                    if (vb) store_g_images<S, C, QOFF>(a.g_out, row0, pitch, I.nx, I.ny, I.walls, xb, yo, vb_);
                }
            }
            if (images) {
                if (va) store_images(a.phi_out, row0, pitch, I.nx, I.ny, I.walls, xa, yo, hia);
                if (vb) store_images(a.phi_out, row0, pitch, I.nx, I.ny, I.walls, xb, yo, hib);
            }
        };

        SwRow<C> r0 = {}, r1 = {}, r2 = {};
        [[maybe_unused]] P2 q0 = {}, q1 = {}, q2 = {};
        [[maybe_unused]] float2 l0 = {}, l1 = {}, l2 = {};
        if constexpr (!GEN) {
            q0 = load_phi();
            q1 = load_phi();
        }
        const int rows = R + 6;
        using Fill = std::false_type;
        using Full = std::true_type;
        // the first six rows fill the pipeline (one body, its stages switched on by row; six turns of the slots
        // by register moves bring them back in place)
#pragma unroll 1
        for (int j = 0; j < 6; j++) {
            row_step(Fill(), j, r0, r1, r2, q0, q2, l0, l1);
            const SwRow<C> t_ = r0; r0 = r2; r2 = r1; r1 = t_;
            q0 = q1; q1 = q2;
            l0 = l1;
        }
        if constexpr (GEN) {
            // one row per iteration with the slots rotated by register moves: the body with the populations is large
            // enough that three copies of it cost more in instruction fetch than the moves do
#pragma unroll 1
            for (int j = 6; j < rows; j++) {
                row_step(Full(), j, r0, r1, r2, q0, q2, l0, l1);
                const SwRow<C> t_ = r0; r0 = r2; r2 = r1; r1 = t_;
            }
        } else {
            // three rows per iteration, so that the slots rotate by renaming
#pragma unroll 1
            for (int j = 6; j < rows; j += 3) {
                row_step(Full(), j, r0, r1, r2, q0, q2, l0, l1);
                if (j + 1 >= rows) break;
                row_step(Full(), j + 1, r2, r0, r1, q1, q0, l1, l2);
                if (j + 2 >= rows) break;
                row_step(Full(), j + 2, r1, r2, r0, q2, q1, l2, l0);
            }
        }
        if constexpr (GEN) copy_wait<0>();  // nothing may land in shared memory the block has left
    }

    // the last block of a batch's last launch advances the step counter read by the next launch (no fence:
    // the counter orders no other data, and the next launch reads it only after this grid has completed)
    // every warp has read it by then
    if (a.t_adv) __syncthreads();
    if (a.t_adv && threadIdx.x == 0) {
        const unsigned int prev = atomicAdd(&a.ctl->done, 1u);
        if (prev == gridDim.x - 1) {
            a.ctl->done = 0u;
            a.ctl->time = (a.read_n ? n - a.t_off : a.ctl->time) + a.t_adv;
        }
    }
}

}  // namespace lbch
