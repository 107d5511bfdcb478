// lbch_internal.h -- the handle of the C ABI and what the translation units of the library share.
#pragma once
#include <algorithm>
#include <vector>

#include "lbch.h"
#include "lbch_kernels.cuh"
#include "lbch_ns.cuh"

constexpr int kMaxShapes = 5;
struct Shape { int tx, ty, nt; };  // output nodes of a tile, threads per block

// Configurations of the row-sweep kernel: the warps per SM among which the grid is cut into strips (fewer where the
// kernel's registers allow fewer).  Many warps hide latency and give long runs of rows on large grids; a grid whose
// strips would get only a few rows each steps faster with fewer, longer ones (choose_default, lb_ch_tune).  A
// configuration is reported under a nominal tile of 56 columns.
constexpr int kSweepShapes = 4;
constexpr int kM3SweepShapes = 2;  // configurations used for handles with a Model III instance
constexpr int kSweepWarps[kSweepShapes] = {16, 8, 4, 12};
constexpr int kSweepTileRows[kSweepShapes] = {48, 24, 12, 24};
constexpr int kSweepW = 56;
inline Shape sweep_tile(int k) { return Shape{kSweepW, kSweepTileRows[k], 0}; }
// What a sweep kernel allows on the device: warps resident per SM, SMs, warps of one block at most, the output columns of a
// strip, and the domain columns that the first strip starts before column 0.
struct SweepFit { int warps, sms, nw, width, lead; };

// Tile shapes of the two-step kernel (periodic instances, tau_g = 1; f32 and f64 only).
constexpr int kPairShapes = 4;
constexpr Shape kPairF[kPairShapes] = {{32, 16, 512}, {32, 14, 512}, {16, 8, 256}, {32, 8, 512}};
constexpr Shape kPair64[kPairShapes] = {{32, 8, 512}, {16, 8, 256}, {16, 16, 512}, {32, 14, 1024}};
inline Shape pair_shape(int prec, int k) { return prec == LBCH_F64 ? kPair64[k] : kPairF[k]; }

struct lbch_handle {
    int device = 0;
    int prec = LBCH_F64;
    int n_inst = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    cudaMemPool_t pool = nullptr;  // the device's pool the handle's buffers come from (stream-ordered, on `stream`)
    std::vector<lbch::InstDev> inst;
    std::vector<long long> node_begin;  // first linear node index of each instance (+ total)
    lbch::InstDev* d_inst = nullptr;
    long long* d_node_begin = nullptr;
    double* d_tabs = nullptr;   // velocity tables in double (init kernel, FP64 step)
    float* d_tabs_f = nullptr;  // the same tables in float (float step kernels)
    int pitch = 0;              // elements per stored row
    int rows = 0;               // stored rows of all instances
    int nq = 9;                 // stored population planes
    size_t g_elem = 8, phi_elem = 8;
    long long nodes = 0;        // lattice nodes (all instances)
    int shape = 0;              // tile shape in use (index into the precision's shape list)
    bool tau1 = false;          // every instance has tau_g = 1: the populations drop out of the step
    bool force_general = false; // test hook: keep the populations even when tau1 holds
    bool force_tile = false;    // step with the tile kernel instead of the row sweep
    bool pair = false;          // step two at a time with the two-step kernel (when pair_ok holds); odd
    int pshape = 0;             // steps take the one-step kernel above; pshape indexes pair_shape()
    bool walls = false;         // an instance has walls
    bool slab = false;          // a slab of a larger periodic grid (lb_ch_init_slab): halos imported between steps
    bool tuning = false;        // lb_ch_tune is stepping the handle (a slab may then take several steps per call)
    bool model3 = false;        // an instance uses Model III (the row sweep's Model III build, or the tile kernel)
    bool need_time = false;     // an instance's step depends on the step index (time factor, Model III)
    void* H[2] = {nullptr, nullptr};  // Model III: H of Eq. F2-1's time derivatives, 2 planes, arithmetic type
    size_t c_elem() const { return prec == LBCH_F64 ? 8 : 4; }
    bool no_pdl = false;        // test hook: plain stream-ordered step launches
    struct PerShape {           // what depends on the tile shape
        int total_tiles = 0;
        int grid = 0;           // persistent CTAs per step launch
        int* d_tile_begin = nullptr;
        void* d_ttabs = nullptr;  // two-step shapes: each tile's velocity tables, contiguous (see lbch_pair.cuh)
        CUtensorMap tm_g[2], tm_phi[2], tm_lo[2];
    } ps[kMaxShapes], pr[kPairShapes];  // tile kernel shapes; two-step shapes (no maps)
    struct SweepCut {           // a row-sweep configuration's division of the handle's grids (see lbch_sweep.cuh)
        int n_items = 0;        // strips, one per warp
        int strips = 0;         // a single instance's strips side by side
        int rows_per = 0;       // rows of one strip (the most, over several instances)
        int nw = 2;             // warps per block
        void* d_items = nullptr;  // several instances: every strip (SweepItem)
    } sw[kSweepShapes][2];      // [..][0] without the populations (tau_g = 1), [..][1] with them
    void* g[2] = {nullptr, nullptr};
    void* phi[2] = {nullptr, nullptr};
    float* lo[2] = {nullptr, nullptr};  // low part of phi (float path)
    double* phi0 = nullptr;     // initial field, double, padded layout
    lbch::Ctl* ctl = nullptr;
    double* partials = nullptr; // reduction scratch: n_inst * chunks * RED_NV doubles
    int chunks = 0;
    long long n = 0;            // host mirror of the step index
    int flip = 0;               // the state of step n is in buffer (n & 1) ^ flip (two-step launches toggle it)
    int t_off = 0, t_adv = 1;   // the next launch's step offset and counter advance (see Ctl)
    bool timed = false;         // an instance's flow has a time factor
    double* d_T = nullptr;      // timed handles: the time factors of a batch of up to kTimeSteps steps
    int t_row = -1;             // the next launch's row of d_T, or -1: the launch forms its time factors itself
    int debug_skip = 0;
    cudaGraphExec_t graph[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};  // [chunk size][starting parity]
    struct TapeGraph {          // a captured taped replay (lb_ch_step_taped) for one starting parity
        cudaGraphExec_t exec = nullptr;
        void* tape = nullptr;
        long nsteps = 0;
    } tgraph[2];
    double* h_stage = nullptr;  // pinned host staging
    size_t h_stage_bytes = 0;
    // adjoint workspace (instance 0), allocated by the first lb_ch_adjoint_begin
    void* adj = nullptr;        // one block: lambda[2] (9N each, N at tau_g = 1), M1 (2N), phi_bar, mu_bar, u.B (AdjView);
                                // then ds (N) and dL/ds, double
    size_t adj_elem = 8;
    int adj_par = 0;            // which lambda holds the current adjoint
    // coupled Navier-Stokes state (LBCH_VEL_COUPLED): f[2], g[2] ([9][N]) and u, p, mu ([N]), one block
    bool coupled = false;
    void* ns = nullptr;
    lbch::ns::NsConsts<double> nsd;
    lbch::ns::NsConsts<float> nsf;
};

// The velocity tables in the arithmetic type of a step kernel.
template <typename C> inline const C* tables(lbch_handle* h);
template <> inline const double* tables<double>(lbch_handle* h) { return h->d_tabs; }
template <> inline const float* tables<float>(lbch_handle* h) { return h->d_tabs_f; }

// The buffer (0 or 1 of each ping-pong pair) holding the state of the current step.
inline int cur_buf(const lbch_handle* h) { return (int)(h->n & 1) ^ h->flip; }

constexpr int kTimeSteps = 512;  // steps per table of time factors (a big graph's; longer batches form several)
// The time factors of the next launch, and whether it reads the step index.
inline const double* launch_T(const lbch_handle* h)
{
    return h->timed && h->t_row >= 0 ? h->d_T + (size_t)h->t_row * h->n_inst : nullptr;
}
inline int launch_reads_n(const lbch_handle* h) { return h->model3 || (h->timed && h->t_row < 0); }

// The row sweep keeps the populations unless every instance has tau_g = 1 (and no test asks for them).
inline bool sweep_gen(const lbch_handle* h) { return !h->tau1 || h->force_general; }

// The two-step kernel serves handles whose instances are all periodic with tau_g = 1, in f32 or f64 (the
// half-storage path is left to the row sweep).
inline bool pair_ok(const lbch_handle* h)
{
    return h->tau1 && !h->force_general && !h->coupled && !h->model3 && !h->walls && !h->slab && h->prec != LBCH_F16S;
}

// Row-sweep launches and set-up, one translation unit per precision (lbch_sweep_*.cu).
#define LBCH_INTERNAL __attribute__((visibility("hidden")))
LBCH_INTERNAL cudaError_t lbch_launch_sweep_f64(lbch_handle* h, int parity);
LBCH_INTERNAL cudaError_t lbch_launch_sweep_f32(lbch_handle* h, int parity);
LBCH_INTERNAL cudaError_t lbch_launch_sweep_f16s(lbch_handle* h, int parity);
LBCH_INTERNAL cudaError_t lbch_prepare_sweep_f64(lbch_handle* h, bool gen, SweepFit* fit);
LBCH_INTERNAL cudaError_t lbch_prepare_sweep_f32(lbch_handle* h, bool gen, SweepFit* fit);
LBCH_INTERNAL cudaError_t lbch_prepare_sweep_f16s(lbch_handle* h, bool gen, SweepFit* fit);
// The same for handles with a Model III instance (lbch_sweep_*_m3.cu).
LBCH_INTERNAL cudaError_t lbch_launch_sweep_f64_m3(lbch_handle* h, int parity);
LBCH_INTERNAL cudaError_t lbch_launch_sweep_f32_m3(lbch_handle* h, int parity);
LBCH_INTERNAL cudaError_t lbch_launch_sweep_f16s_m3(lbch_handle* h, int parity);
LBCH_INTERNAL cudaError_t lbch_prepare_sweep_f64_m3(lbch_handle* h, bool gen, SweepFit* fit);
LBCH_INTERNAL cudaError_t lbch_prepare_sweep_f32_m3(lbch_handle* h, bool gen, SweepFit* fit);
LBCH_INTERNAL cudaError_t lbch_prepare_sweep_f16s_m3(lbch_handle* h, bool gen, SweepFit* fit);
// Two-step launches and set-up (lbch_pair.cu); pshape names a pair_shape().
LBCH_INTERNAL cudaError_t lbch_launch_pair(lbch_handle* h, int parity);
LBCH_INTERNAL cudaError_t lbch_prepare_pair(lbch_handle* h, int k);
// Shape k's velocity tables, every tile's own: their bytes, and the launch that forms them from the handle's.
LBCH_INTERNAL size_t lbch_pair_tables_bytes(const lbch_handle* h, int k);
LBCH_INTERNAL cudaError_t lbch_pair_tables(lbch_handle* h, int k);
// Launch limits of a kernel on a device, set and queried once per process (they depend on nothing else) and
// served from a table afterwards, so that making a handle does not repeat them for every kernel it may run:
// lbch_kernel_smem lets `kern` use `smem` bytes of dynamic shared memory; lbch_kernel_fit gives how many CTAs
// of `threads` threads with `smem` bytes one SM holds, and the device's SM count (lbch_api.cu).
LBCH_INTERNAL cudaError_t lbch_kernel_smem(const void* kern, int device, size_t smem);
LBCH_INTERNAL cudaError_t lbch_kernel_fit(const void* kern, int device, int threads, size_t smem, int* per_sm, int* sms);
