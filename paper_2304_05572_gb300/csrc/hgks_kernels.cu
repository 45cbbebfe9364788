// hgks_kernels.cu -- the S2O4 step of the hybrid WENO-AO gas-kinetic scheme as sm_103a
// FP64 kernels (arXiv 2304.05572, Sec. 2), and the host code that enqueues one step.
//
// Per stage: ghost fill -> for each sweep (x, then y in 2D):
//   raw normal flags -> normal reconstruction (linear inline, troubled sides appended to a
//   work list with warp-aggregated atomics) -> dense WENO-AO pass over that list ->
//   [2D: raw tangential flags -> spread flags and work list of the troubled passes -> dense
//   WENO-AO pass] -> gas-kinetic flux per Gauss point (which reconstructs the smooth passes itself)
// -> stage update.  Small sweeps (small_sweep in hgks_api.cu: below 49152 segments, in 1D below 16384 interfaces
// unless linear) take one launch per reconstruction direction instead (k_normal_small, k_tang_small) and the flux
// with one side of a Gauss point per warp (k_flux_small).  dt is reduced, clipped to t_end and applied on the
// device.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <cstdio>
#include <type_traits>

#include "hgks_internal.h"
#include "hgks_math.cuh"

namespace hgks {

const char* kclass_names[KC_COUNT] = {"ghost", "dt", "raw_normal_flags", "normal_recon", "normal_weno_ao",
                                      "raw_tangential_flags", "tangential_recon", "tangential_weno_ao",
                                      "gks_flux", "stage_update"};

namespace {

constexpr int TPB = 256;

// Global-memory access.  Every load and store of a kernel names the range its pointer must lie
// in (R.lo, R.hi: the solver's device buffers).  The debug build (HGKS_DEBUG_BOUNDS) checks each
// access against that range: an access outside it is skipped (a load returns 0), counted, and
// the address of the first one is kept for hgks_debug_bounds; nothing traps.  The normal build
// accesses memory directly.
#ifdef HGKS_DEBUG_BOUNDS
__device__ unsigned long long g_dbg_count;
__device__ unsigned long long g_dbg_first;
template <class T>
__device__ __forceinline__ bool in_range(const T* p, const char* lo, const char* hi)
{
    const char* c = (const char*)p;
    if (c >= lo && c + sizeof(T) <= hi) return true;
    atomicAdd(&g_dbg_count, 1ull);
    atomicCAS(&g_dbg_first, 0ull, (unsigned long long)(uintptr_t)c);
    return false;
}
template <class T, class R>
__device__ __forceinline__ T ldc(const T* p, const R& r) { return in_range(p, r.lo, r.hi) ? *p : T(0); }
template <class T, class R>
__device__ __forceinline__ T rdc(const T* p, const R& r) { return in_range(p, r.lo, r.hi) ? *p : T(0); }
template <class T, class V, class R>
__device__ __forceinline__ void stc(T* p, V v, const R& r) { if (in_range(p, r.lo, r.hi)) *p = (T)v; }
#else
template <class T, class R>
__device__ __forceinline__ T ldc(const T* p, const R&) { return *p; }
template <class T, class R>
__device__ __forceinline__ T rdc(const T* p, const R&) { return *p; }
template <class T, class V, class R>
__device__ __forceinline__ void stc(T* p, V v, const R&) { *p = (T)v; }
#endif

// Entry of every kernel of a step.  The step's launches carry the programmatic-serialisation attribute: a
// launch is set up while the one before it drains, and waits here until that one is complete and its
// memory visible, before anything is read (so loads are plain ones, not through the read-only path, whose
// data must not change while a kernel is resident).  About 2.5 us less per launch: a step of 200 cells in 1D 79 ->
// 60 us, of 48 x 48 four-quadrant 155 -> 131, of 1024^2 9.76 -> 9.71 ms.  The next launch is not let in early
// (launch_dependents at the start): its waiting blocks then crowd onto the multiprocessors that were free first (8191
// cells 84 -> 116 us, 48 x 48 155 -> 219).
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---------------------------------------------------------------- ghost cells
// x ghosts on interior rows, then y ghosts over the padded width (fills corners).
// Non-reflecting: zero-gradient copy; reflect / symmetry: mirror, normal momentum negated;
// no-slip adiabatic: mirror, both momenta negated.  Prescribed states (Sec. 3.5): inflow,
// the wall that starts at x = shock_x0, and the boundary that follows the oblique shock line
// x = shock_x0 + shock_cot (y + shock_speed t), all evaluated at the ghost cell's centre at the
// stage time (t^n, or t^n + dt/2 in the second stage).  The centre and line positions are
// computed in one fixed IEEE order (no contraction) so that the side of the line a ghost cell
// falls on is the same in every implementation that follows this order.
__device__ __forceinline__ double stage_time(const Ctrl* ctrl, int stage)
{
    return stage == 0 ? ctrl->t : (ex(ctrl->t) + ex(0.5) * ex(ctrl->dt)).v;
}

__device__ __forceinline__ double cell_centre(double origin, int i, double h)
{
    return (ex(origin) + (ex((double)i) + ex(0.5)) * ex(h)).v;
}

// Component k of cell (i, j) of an interior row j, i anywhere in the padded width: the interior cell, or
// the x ghost cell's value by its boundary.
__device__ __forceinline__ double x_value(const Params& P, const double* W, int k, int i, int j)
{
    const GridGeom& g = P.g;
    const double* base = W + g.origin + (long long)k * g.plane + (long long)j * g.pitch;
    if (i >= 0 && i < g.nx) return rdc(base + i, g);
    const int side = i < 0 ? 0 : 1, l = i < 0 ? -i : i - g.nx + 1;
    const int bc = P.bc[side];
    if (bc == HGKS_BC_INFLOW) return P.bc_state[side][k];
    const bool mirror = bc == HGKS_BC_REFLECT || bc == HGKS_BC_SYMMETRY || bc == HGKS_BC_NOSLIP;
    int src;
    if (bc == HGKS_BC_PERIODIC) src = side == 0 ? g.nx - l : l - 1;
    else if (bc == HGKS_BC_EXTRAP) src = side == 0 ? 0 : g.nx - 1;
    else src = side == 0 ? l - 1 : g.nx - l;
    double v = rdc(base + src, g);
    if (mirror) {
        if (k == 1) v = -v;
        if (bc == HGKS_BC_NOSLIP && g.dim == 2 && k == 2) v = -v;
    }
    return v;
}

// The ghost cells of a stage, one value per thread: the x sides on interior rows, then the y sides over the
// padded width.  A corner takes its y boundary's image of the x ghost cell beside it, formed from the
// interior cell behind both (x_value), so no ghost cell is read and one launch fills them all.
// The first thread also empties the stage's work lists (no kernel of the stage reads them before this launch
// is complete).
inline long long ghost_threads(const GridGeom& g)
{
    const long long x = (long long)g.nv * (g.dim == 2 ? g.ny : 1) * NG * 2;
    return g.dim == 2 ? x + (long long)g.nv * (g.nx + 2 * NG) * NG * 2 : x;
}

__device__ __forceinline__ void b_ghost(const Params& P, double* W, Ctrl* ctrl, int stage, long long id)
{
    if (id == 0) ctrl->cnt[0][0] = ctrl->cnt[0][1] = ctrl->cnt[1][0] = ctrl->cnt[1][1] = 0;
    const GridGeom& g = P.g;
    const int rowsI = g.dim == 2 ? g.ny : 1;
    const long long nxg = (long long)g.nv * rowsI * NG * 2;
    if (id < nxg) {
        const int side = (int)(id % 2); id /= 2;
        const int l = (int)(id % NG) + 1; id /= NG;
        const int j = (int)(id % rowsI);
        const int k = (int)(id / rowsI);
        const int dst = side == 0 ? -l : g.nx - 1 + l;
        stc(W + g.origin + (long long)k * g.plane + (long long)j * g.pitch + dst, x_value(P, W, k, dst, j), g);
        return;
    }
    id -= nxg;
    const int width = g.nx + 2 * NG;
    if (g.dim != 2 || id >= (long long)g.nv * width * NG * 2) return;
    const int i = (int)(id % width) - NG; id /= width;
    const int side = (int)(id % 2); id /= 2;
    const int l = (int)(id % NG) + 1;
    const int k = (int)(id / NG);
    const int bc = P.bc[2 + side];
    const int dst = side == 0 ? -l : g.ny - 1 + l;
    double* to = W + g.origin + (long long)k * g.plane + (long long)dst * g.pitch + i;
    if (bc == HGKS_BC_INFLOW) { stc(to, P.bc_state[2 + side][k], g); return; }
    if (bc == HGKS_BC_SHOCK_TRACK) {
        const double xc = cell_centre(P.x0, i, g.dx), yc = cell_centre(P.y0, dst, g.dy);
        const double t = stage_time(ctrl, stage);
        const double xs = (ex(P.shock_x0) + ex(P.shock_cot) * (ex(yc) + ex(P.shock_speed) * ex(t))).v;
        stc(to, xc < xs ? P.bc_state[2 + side][k] : P.shock_pre[k], g);
        return;
    }
    if (bc == HGKS_BC_SHOCK_WALL && cell_centre(P.x0, i, g.dx) < P.shock_x0) {
        stc(to, P.bc_state[2 + side][k], g);
        return;
    }
    const bool mirror = bc == HGKS_BC_REFLECT || bc == HGKS_BC_SYMMETRY || bc == HGKS_BC_NOSLIP || bc == HGKS_BC_SHOCK_WALL;
    int src;
    if (bc == HGKS_BC_PERIODIC) src = side == 0 ? g.ny - l : l - 1;
    else if (bc == HGKS_BC_EXTRAP) src = side == 0 ? 0 : g.ny - 1;
    else src = side == 0 ? l - 1 : g.ny - l;
    double v = x_value(P, W, k, i, src);
    if (mirror) {
        if (k == 2) v = -v;
        if (bc == HGKS_BC_NOSLIP && k == 1) v = -v;
    }
    stc(to, v, g);
}

// Second stage (W*)
__global__ void k_ghost(Params P, double* W, Ctrl* ctrl)
{
    pdl_enter();
    if (ctrl->done) return;
    b_ghost(P, W, ctrl, 1, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

// ---------------------------------------------------------------- time step
// Sec. 3 preamble: dt = CFL min(h/(|U|+a), h^2/(4 nu)), h = min(dx, dy), nu = mu/rho;
// same evaluation order as the CPU reference so that dt is reproduced exactly.
__device__ __forceinline__ void b_dt(const Params& P, const double* W, Ctrl* ctrl, double h, long long start, long long stride)
{
    const GridGeom& g = P.g;
    int rowsI = g.dim == 2 ? g.ny : 1;
    long long n = (long long)rowsI * g.nx;
    unsigned long long best = 0x7FF0000000000000ull;
    for (long long id = start; id < n; id += stride) {
        int i = (int)(id % g.nx), j = (int)(id / g.nx);
        const double* c = W + g.origin + (long long)j * g.pitch + i;
        ex rho(rdc(c, g));
        ex ri = ex(1.0) / rho;
        ex U = ex(rdc(c + g.plane, g)) * ri;
        ex V = g.dim == 2 ? ex(rdc(c + 2 * g.plane, g)) * ri : ex(0.0);
        ex q2 = U * U + V * V;
        ex p = (ex(P.gamma) - ex(1.0)) * (ex(rdc(c + (g.nv - 1) * g.plane, g)) - (ex(0.5) * rho) * q2);
        ex a = xsqrt((ex(P.gamma) * p) * ri);
        ex d = ex(h) / (xsqrt(q2) + a);
        if (P.viscous) {
            ex nu = ex(P.mu) * ri;
            ex dv = (ex(h) * ex(h)) / (ex(4.0) * nu);
            if (dv.v < d.v) d = dv;
        }
        unsigned long long bits = (unsigned long long)__double_as_longlong(d.v);
        if (!fixed::is_pos(d.v)) bits = 0x7FF8000000000000ull;   // non-physical cells are caught by the update
        best = bits < best ? bits : best;
    }
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
        best = other < best ? other : best;
    }
    if ((threadIdx.x & 31) == 0) atomicMin(&ctrl->dtmin_bits, best);
}

// Called by every thread of each of the `blocks` blocks that reduced a solver's dt: the last block to
// arrive applies the CFL number (or takes the fixed step), clips to t_end, decides whether the step
// runs, and leaves the reduction ready for the next step.
__device__ __forceinline__ void dt_finish(const Params& P, Ctrl* ctrl, double t_end, unsigned int blocks)
{
    __syncthreads();
    if (threadIdx.x != 0) return;
    __threadfence();
    if (atomicAdd(&ctrl->dt_blocks, 1u) != blocks - 1u) return;
    __threadfence();
    ctrl->dt_blocks = 0;
    const unsigned long long bits = atomicExch(&ctrl->dtmin_bits, 0x7FF0000000000000ull);
    const double tol = 1e-12 * (fabs(t_end) > 1.0 ? fabs(t_end) : 1.0);
    double dt = P.fixed_dt > 0.0 ? P.fixed_dt : P.cfl * __longlong_as_double((long long)bits);
    int done = ctrl->status != 0 || !(t_end - ctrl->t > tol);
    if (!done && ctrl->t + dt > t_end) dt = t_end - ctrl->t;
    if (!done && !(dt > 0.0 && dt < 1e300)) { ctrl->status = HGKS_ENONPHYSICAL; done = 1; }
    ctrl->dt = dt;
    ctrl->done = done;
}

// The first launch of a step: blocks [0, nb) reduce dt, the others fill the ghost cells of W^n (both only
// read interior cells; a step that turns out to be done has its ghost cells filled for nothing).  One launch
// for what took five (work-list reset, dt, its decision, two ghost fills).
__global__ void k_dt_ghost(Params P, double* W, Ctrl* ctrl, double h, double t_end, int nb)
{
    pdl_enter();
    const int b = (int)blockIdx.x;
    if (b >= nb) {
        b_ghost(P, W, ctrl, 0, (long long)(b - nb) * blockDim.x + threadIdx.x);
        return;
    }
    if (!(P.fixed_dt > 0.0)) b_dt(P, W, ctrl, h, (long long)b * blockDim.x + threadIdx.x, (long long)nb * blockDim.x);
    dt_finish(P, ctrl, t_end, (unsigned)nb);
}

__global__ void k_state_out(GridGeom g, const double* W, double* dst)
{
    pdl_enter();
    const long long n = (long long)g.nv * g.ny * g.nx;
    for (long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x; id < n; id += (long long)gridDim.x * blockDim.x) {
        const long long row = id / g.nx;
        const int i = (int)(id - row * g.nx), k = (int)(row / g.ny), j = (int)(row - (long long)k * g.ny);
        dst[id] = rdc(W + g.origin + (long long)k * g.plane + (long long)j * g.pitch + i, g);
    }
}

__device__ __forceinline__ void reset_ctrl(Ctrl* ctrl, double t0)
{
    ctrl->t = t0;
    ctrl->dtmin_bits = 0x7FF0000000000000ull;   // +inf
    ctrl->dt_blocks = 0;
    ctrl->dt = 0.0;
    ctrl->last_dt = 0.0;
    ctrl->steps = 0;
    ctrl->status = 0;
    ctrl->done = 0;
    for (int a = 0; a < 2; a++) for (int b = 0; b < 2; b++) for (int c = 0; c < 2; c++) {
        ctrl->troubled[a][b][c] = 0; ctrl->examined[a][b][c] = 0;
    }
}

__global__ void k_set_time(Ctrl* ctrl, double t0) { reset_ctrl(ctrl, t0); }

__device__ __forceinline__ void state_in(const GridGeom& g, const double* src, double* W, long long id, long long threads)
{
    const long long n = (long long)g.nv * g.ny * g.nx;
    for (; id < n; id += threads) {
        const long long row = id / g.nx;
        const int i = (int)(id - row * g.nx), k = (int)(row / g.ny), j = (int)(row - (long long)k * g.ny);
        stc(W + g.origin + (long long)k * g.plane + (long long)j * g.pitch + i, src[id], g);
    }
}

// The caller's [nv][ny][nx] state into and out of the padded layout, one launch for all components in place
// of a pitched copy each and a launch for the control block: 8 steps of a 200-cell tube with both
// transfers 714 -> 691 us, a 48 x 48 allocation-free step (which also copied its descriptor and cleared
// its 3.5 MB) 164 -> 131 us.
__global__ void k_state_in(GridGeom g, const double* src, double* W, Ctrl* ctrl, double t0)
{
    pdl_enter();
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id == 0) reset_ctrl(ctrl, t0);
    state_in(g, src, W, id, (long long)gridDim.x * blockDim.x);
}

// The same for the allocation-free step, whose descriptor travels as the launch's argument.
__global__ void k_noalloc_in(SolveDesc d, SolveDesc* self, const double* src)
{
    pdl_enter();
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id == 0) {
        *self = d;
        reset_ctrl(d.ctrl, 0.0);
    }
    state_in(d.P.g, src, d.W, id, (long long)gridDim.x * blockDim.x);
}

// warp-aggregated counter add
__device__ __forceinline__ void warp_count(unsigned long long* dst, unsigned int v)
{
    unsigned int tot = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0 && tot) atomicAdd(dst, (unsigned long long)tot);
}

// warp-aggregated append of one item per set predicate; returns nothing, writes list
template <class R>
__device__ __forceinline__ void warp_push(unsigned int* cnt, uint32_t* list, bool pred, uint32_t item, const R& rg)
{
    unsigned int mask = __ballot_sync(0xffffffffu, pred);
    if (!mask) return;
    int lane = threadIdx.x & 31;
    int leader = __ffs(mask) - 1;
    unsigned int base = 0;
    if (lane == leader) base = atomicAdd(cnt, (unsigned int)__popc(mask));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (pred) stc(list + base + __popc(mask & ((1u << lane) - 1u)), item, rg);
}

// The same for up to four items a lane, item | X for every set bit X of `bits`, with one atomic: the
// appends of all warps of a sweep meet on one counter.
template <class R>
__device__ __forceinline__ void warp_push4(unsigned int* cnt, uint32_t* list, unsigned int bits, uint32_t item, const R& rg)
{
    unsigned int mask[4];
    int total = 0;
#pragma unroll
    for (int X = 0; X < 4; X++) { mask[X] = __ballot_sync(0xffffffffu, (bits >> X) & 1u); total += __popc(mask[X]); }
    if (!total) return;
    const int lane = threadIdx.x & 31;
    unsigned int base = 0;
    if (lane == 0) base = atomicAdd(cnt, (unsigned int)total);
    base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
    for (int X = 0; X < 4; X++) {
        if ((bits >> X) & 1u) stc(list + base + __popc(mask[X] & ((1u << lane) - 1u)), item | (uint32_t)X, rg);
        base += __popc(mask[X]);
    }
}

// ---------------------------------------------------------------- normal pass
// local state access: component k of cell n on line t
__device__ __forceinline__ const double* cellp(const Params& P, const Sweep& S, const double* W, int t, int n)
{
    return W + P.g.origin + (long long)t * S.sT + (long long)n * S.sN;
}

template <int NV>
__device__ __forceinline__ void b_raw_nflags(const Params& P, const Sweep& S, const double* W, const Ctrl* ctrl, long long id)
{
    if (ctrl->done) return;
    int width = S.nn + 4;
    long long total = (long long)S.nlines * width;
    if (id >= total) return;
    int c = (int)(id % width), L = (int)(id / width);
    int t = L + S.tlo, n = c - 2;
    int tr = 0;
    if (P.recon_mode == HGKS_RECON_HYBRID) {
        const double* base = cellp(P, S, W, t, n - 2);
#pragma unroll
        for (int k = 0; k < NV; k++) {
            double q[5];
            float f[5];
            const double* b = base + (long long)S.perm[k] * P.g.plane;
#pragma unroll
            for (int s = 0; s < 5; s++) { q[s] = ldc(b + (long long)s * S.sN, S); f[s] = fixed::to_float(q[s]); }
            tr |= indicator_raw<false>(q, f, S.Z1n);
        }
    }
    stc(S.rawN + id, tr, S);
}

// A solver's own sweep kernels run the two sweeps of a 2D stage in one launch (they share no
// buffer and no result until the update): blocks [0, nb0) work on the x sweep, the others on the
// y sweep; 1D launches give every block to the x sweep.  `id` is the thread's index within its
// sweep's blocks, `lanes` the number of threads on that sweep.
struct SweepBlock { int dir; long long id, lanes; };

__device__ __forceinline__ SweepBlock sweep_block(int nb0)
{
    SweepBlock r;
    r.dir = (int)blockIdx.x >= nb0 ? 1 : 0;
    const long long first = r.dir ? nb0 : 0;
    const long long nb = r.dir ? (long long)gridDim.x - nb0 : (long long)nb0;
    r.id = ((long long)blockIdx.x - first) * blockDim.x + threadIdx.x;
    r.lanes = nb * blockDim.x;
    return r;
}

template <int NV>
__global__ void k_raw_nflags(const SolveDesc* D, int nb0, int stage)
{
    pdl_enter();
    const SweepBlock b = sweep_block(nb0);
    const SolveDesc& d = *D;
    b_raw_nflags<NV>(d.P, d.sw[b.dir], stage == 0 ? d.W : d.Ws, d.ctrl, b.id);
}


template <int NV>
__device__ __forceinline__ void store_line(const Params& P, const Sweep& S, int L, int m, int side, const double* val, const double* der)
{
    long long plane = (long long)S.nlines * S.nm;
    long long o = (long long)L * S.nm + m;
#pragma unroll
    for (int k = 0; k < NV; k++) {
        stc(S.line + (long long)(side * NV + k) * plane + o, val[k], S);
        stc(S.line + (long long)((2 + side) * NV + k) * plane + o, der[k], S);
    }
}

template <int NV>
__device__ __forceinline__ void b_normal(const Params& P, const Sweep& S, const double* W, Ctrl* ctrl, int stage, long long id)
{
    if (ctrl->done) return;
    long long total = (long long)S.nlines * S.nm;
    bool active = id < total;
    int L = 0, m = 0;
    if (active) { m = (int)(id % S.nm); L = (int)(id / S.nm); }
    int t = L + S.tlo;
    int fl[2] = {0, 0};
    if (active) {
        const uint8_t* raw = S.rawN + (long long)L * (S.nn + 4);
#pragma unroll
        for (int side = 0; side < 2; side++) {
            int c = m - 1 + side;     // cell index; raw index of cell c is c + 2
            int f;
            if (P.recon_mode == HGKS_RECON_LINEAR) f = 0;
            else if (P.recon_mode == HGKS_RECON_WENOAO) f = 1;
            else f = rdc(raw + c + 1, S) | rdc(raw + c + 2, S) | rdc(raw + c + 3, S);   // Step 4
            fl[side] = f;
        }
        uint8_t* fo = S.flagN + (long long)L * (S.nn + 2);
        stc(fo + m + 1, fl[1], S);
        if (m == 0) stc(fo, fl[0], S);
    }
    bool counted = active && t >= 0 && t < S.nt && m < S.nn;
    warp_count(&ctrl->troubled[stage][S.dir][0], counted && fl[1] ? 1u : 0u);
    if (id == 0) atomicAdd(&ctrl->examined[stage][S.dir][0], (unsigned long long)S.nt * S.nn);
#pragma unroll
    for (int side = 0; side < 2; side++) {
        bool push = active && fl[side];
        warp_push(&ctrl->cnt[S.dir][0], S.itemsN, push, (uint32_t)((((long long)L * S.nm + m) << 1) | side), S);
        if (!active || fl[side]) continue;
        int c = m - 1 + side;
        double val[NV], der[NV];
        const double* base = cellp(P, S, W, t, c - 2);
#pragma unroll
        for (int k = 0; k < NV; k++) {
            double q[5];
            const double* b = base + (long long)S.perm[k] * P.g.plane;
#pragma unroll
            for (int s = 0; s < 5; s++) q[s] = ldc(b + (long long)s * S.sN, S);
            if (side == 0) linear_left(q, S.inv12hn, val[k], der[k]);
            else linear_right(q, S.inv12hn, val[k], der[k]);
        }
        if (nonphysical<NV>(val)) {
            const double* cc = cellp(P, S, W, t, c);
#pragma unroll
            for (int k = 0; k < NV; k++) { val[k] = ldc(cc + (long long)S.perm[k] * P.g.plane, S); der[k] = 0.0; }
        }
        store_line<NV>(P, S, L, m, side, val, der);
    }
}

template <int NV>
__global__ void k_normal(const SolveDesc* D, int nb0, int stage)
{
    pdl_enter();
    const SweepBlock b = sweep_block(nb0);
    const SolveDesc& d = *D;
    b_normal<NV>(d.P, d.sw[b.dir], stage == 0 ? d.W : d.Ws, d.ctrl, stage, b.id);
}


// The window (cells i-2..i+2 across the face, all components) and the face average of the
// troubled side `it` of the normal pass.
template <int NV>
__device__ __forceinline__ void normal_ao_item(const Params& P, const Sweep& S, const double* W, uint32_t it,
                                               double (*Qw)[NV], double* Qs, int& side, int& L, int& m)
{
    side = it & 1;
    const long long lm = it >> 1;
    m = (int)(lm % S.nm); L = (int)(lm / S.nm);
    const int t = L + S.tlo;
    const int c = m - 1 + side;
    const double* base = cellp(P, S, W, t, c - 2);
#pragma unroll
    for (int s = 0; s < 5; s++)
#pragma unroll
        for (int k = 0; k < NV; k++) Qw[s][k] = ldc(base + (long long)s * S.sN + (long long)S.perm[k] * P.g.plane, S);
    const double* cl = cellp(P, S, W, t, m - 1);
    const double* cr = cellp(P, S, W, t, m);
#pragma unroll
    for (int k = 0; k < NV; k++) {
        long long o = (long long)S.perm[k] * P.g.plane;
        Qs[k] = ((ex(ldc(cl + o, S)) + ex(ldc(cr + o, S))) * ex(0.5)).v;
    }
}

// The troubled sides of the normal pass: one per lane (weno_ao_face) from kAoOneLaneMin items
// on, else one per aligned group of 4 lanes (weno_ao_face_x4: lane q carries characteristic
// field q and stores component q).  Both forms give the same bits.  `lane`, `lanes`: this
// thread's index among, and the number of, the lanes working on the pass.
template <int NV>
__device__ __forceinline__ void b_normal_ao(const Params& P, const Sweep& S, const double* W, const Ctrl* ctrl, long long lane, long long lanes)
{
    if (ctrl->done) return;
    unsigned int n = ctrl->cnt[S.dir][0];
    AOConst ak;
    for (int j = 0; j < 4; j++) ak.g[j] = P.g_ao[j];
    ak.g3inv = P.g3inv; ak.gr[0] = P.gr[0]; ak.gr[1] = P.gr[1]; ak.gr[2] = P.gr[2]; ak.eps = P.eps;
    const long long plane = (long long)S.nlines * S.nm;
    if (n >= kAoOneLaneMin) {
        for (unsigned int i = (unsigned int)lane; i < n; i += (unsigned int)lanes) {
            double Qw[5][NV], Qs[NV], val[NV], d[NV];
            int side, L, m;
            normal_ao_item<NV>(P, S, W, rdc(S.itemsN + i, S), Qw, Qs, side, L, m);
            weno_ao_face<NV>(P.gamma, ak, Qw, Qs, side == 0 ? +1 : -1, val, d);
            const bool bad = nonphysical<NV>(val);
            const long long o = (long long)L * S.nm + m;
#pragma unroll
            for (int k = 0; k < NV; k++) {
                stc(S.line + (long long)(side * NV + k) * plane + o, bad ? Qw[2][k] : val[k], S);
                stc(S.line + (long long)((2 + side) * NV + k) * plane + o, bad ? 0.0 : (ex(d[k]) * ex(S.inv_hn)).v, S);
            }
        }
        return;
    }
    const int q = threadIdx.x & 3;
    const unsigned gmask = 0xFu << (threadIdx.x & 28);
    for (unsigned int i = (unsigned int)(lane >> 2); i < n; i += (unsigned int)(lanes >> 2)) {
        double Qw[5][NV], Qs[NV], val[NV], dq;
        int side, L, m;
        normal_ao_item<NV>(P, S, W, rdc(S.itemsN + i, S), Qw, Qs, side, L, m);
        weno_ao_face_x4<NV>(P.gamma, ak, Qw, Qs, side == 0 ? +1 : -1, gmask, val, dq);
        double vq = 0.0;
        if (nonphysical<NV>(val)) {
            vq = Qw[2][q < NV ? q : 0];
            dq = 0.0;
        } else {
#pragma unroll
            for (int k = 0; k < NV; k++)
                if (k == q) vq = val[k];
            dq = (ex(dq) * ex(S.inv_hn)).v;
        }
        if (q < NV) {
            long long o = (long long)L * S.nm + m;
            stc(S.line + (long long)(side * NV + q) * plane + o, vq, S);
            stc(S.line + (long long)((2 + side) * NV + q) * plane + o, dq, S);
        }
    }
}

template <int NV>
__global__ void k_normal_ao(const SolveDesc* D, int nb0, int stage)
{
    pdl_enter();
    const SweepBlock b = sweep_block(nb0);
    const SolveDesc& d = *D;
    b_normal_ao<NV>(d.P, d.sw[b.dir], stage == 0 ? d.W : d.Ws, d.ctrl, b.id, b.lanes);
}


// Small sweeps: flags, linear reconstruction and WENO-AO of the normal pass in one launch.  A warp takes 8
// consecutive cells of a line, 4 lanes each (lane q carries component q), and one side: every group runs the
// raw indicator of its cell, the groups exchange the decisions for the Step-4 spread (OR over the components,
// then over the neighbouring groups), and the inner 6 reconstruct their face with the linear formulas or
// weno_ao_face_x4.  The arithmetic is b_normal's and b_normal_ao's, so every result is.  The warps of a
// block stand on neighbouring lines, which share the memory sectors of a y sweep.
// Such a sweep's time is made of launches (3 us each) and of each thread's chain of FP64 instructions (31 ns
// each): with one launch per direction in place of three (flags, linear pass, compacted WENO-AO) and the
// step's five control and ghost launches in two, a step of 200 cells in 1D went from 133 to 90 us, of
// 48 x 48 from 210 to 136.  Compaction and shared flags pay on larger sweeps.  The line of 49152 segments was placed
// when 200^2 (40200 segments) took 714 us a step in this form against 749 in the other, 250^2 990 against 941.
// With the present kernels (us per step, this form against the other; both forms' flux included) the two
// meet lower, and the line has not been moved since:
//   four-quadrant 64^2 173, 224; 100^2 257, 287; 141^2 377, 389; 180^2 523, 461; 200^2 626, 547; 221^2 744, 612;
//   viscous tube with the Prandtl fix 200 x 100 364, 418; 280 x 140 604, 616; 312 x 156 726, 718;
//   WENO-AO everywhere 64^2 280, 275; 100^2 563, 526; 200^2 2041, 1591.
constexpr int kSmallCells = 6;

template <int NV>
__device__ __forceinline__ void b_normal_small(const Params& P, const Sweep& S, const double* W, Ctrl* ctrl, int stage, long long id)
{
    if (ctrl->done) return;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, gi = lane >> 2, q = lane & 3, qc = q < NV ? q : NV - 1;
    const int lane0 = lane & 28;
    const unsigned gmask = 0xFu << lane0;
    const unsigned w = (unsigned)(id >> 5), nl = (unsigned)S.nlines;
    const unsigned rest = w / nl;
    const int L = (int)(w - rest * nl), side = (int)(rest & 1), c = (int)(rest >> 1) * kSmallCells + gi - 2;
    if ((int)(rest >> 1) * kSmallCells >= S.nn + 2) return;        // the same for the warp
    const int cc = c <= S.nn + 1 ? c : S.nn + 1;                   // (groups past the last halo cell repeat it)
    const int t = L + S.tlo;
    const double* b = cellp(P, S, W, t, cc - 2) + (long long)S.perm[qc] * P.g.plane;
    double v[5];
#pragma unroll
    for (int s = 0; s < 5; s++) v[s] = ldc(b + (long long)s * S.sN, S);
    int flag = 0;
    if (P.recon_mode == HGKS_RECON_WENOAO) flag = 1;
    else if (P.recon_mode == HGKS_RECON_HYBRID) {
        float f[5];
#pragma unroll
        for (int s = 0; s < 5; s++) f[s] = fixed::to_float(v[s]);
        flag = indicator_raw<true>(v, f, S.Z1n);
        flag |= __shfl_xor_sync(full, flag, 1);
        flag |= __shfl_xor_sync(full, flag, 2);
        flag |= __shfl_sync(full, flag, lane - 4) | __shfl_sync(full, flag, lane + 4);   // (used by the inner groups)
    }
    const bool out = gi >= 1 && gi <= kSmallCells && c <= S.nn;
    const bool first = out && side == 0 && q == 0;                 // one lane per cell -1..nn
    if (first) stc(S.flagN + (long long)L * (S.nn + 2) + c + 1, flag, S);
    const bool counted = first && t >= 0 && t < S.nt && c >= 0 && c < S.nn;
    warp_count(&ctrl->troubled[stage][S.dir][0], counted && flag ? 1u : 0u);
    warp_count(&ctrl->examined[stage][S.dir][0], counted ? 1u : 0u);
    // side 0: the left state of interface c + 1; side 1: the right state of interface c
    const int m = side == 0 ? c + 1 : c;
    if (!out || m < 0 || m >= S.nm) return;                        // the same for a group
    double val, der;
    if (!flag) {
        if (side == 0) linear_left(v, S.inv12hn, val, der);
        else linear_right(v, S.inv12hn, val, der);
        if (nonphysical_x4<NV>(val, lane0, gmask)) { val = v[2]; der = 0.0; }
    } else {
        AOConst ak;
        for (int j = 0; j < 4; j++) ak.g[j] = P.g_ao[j];
        ak.g3inv = P.g3inv; ak.gr[0] = P.gr[0]; ak.gr[1] = P.gr[1]; ak.gr[2] = P.gr[2]; ak.eps = P.eps;
        double Qw[5][NV], Qs[NV], vs[NV];
        const double avg = ((ex(side == 0 ? v[2] : v[1]) + ex(side == 0 ? v[3] : v[2])) * ex(0.5)).v;
#pragma unroll
        for (int k = 0; k < NV; k++) {
            Qs[k] = __shfl_sync(gmask, avg, lane0 + k);
#pragma unroll
            for (int s = 0; s < 5; s++) Qw[s][k] = __shfl_sync(gmask, v[s], lane0 + k);
        }
        weno_ao_face_x4<NV>(P.gamma, ak, Qw, Qs, side == 0 ? +1 : -1, gmask, vs, der);
        val = 0.0;
        if (nonphysical<NV>(vs)) {
            val = v[2];
            der = 0.0;
        } else {
#pragma unroll
            for (int k = 0; k < NV; k++)
                if (k == q) val = vs[k];
            der = (ex(der) * ex(S.inv_hn)).v;
        }
    }
    if (q < NV) {
        const long long plane = (long long)S.nlines * S.nm, o = (long long)L * S.nm + m;
        stc(S.line + (long long)(side * NV + q) * plane + o, val, S);
        stc(S.line + (long long)((2 + side) * NV + q) * plane + o, der, S);
    }
}

template <int NV>
__global__ void k_normal_small(const SolveDesc* D, int nb0, int stage)
{
    pdl_enter();
    const SweepBlock b = sweep_block(nb0);
    const SolveDesc& d = *D;
    b_normal_small<NV>(d.P, d.sw[b.dir], stage == 0 ? d.W : d.Ws, d.ctrl, stage, b.id);
}

// ---------------------------------------------------------------- tangential passes (2D)
__device__ __forceinline__ double lineval(const Sweep& S, int X, int k, int t, int m)
{
    long long plane = (long long)S.nlines * S.nm;
    return ldc(S.line + (long long)(X * 4 + k) * plane + (long long)(t - S.tlo) * S.nm + m, S);
}

// Large sweeps: each thread takes kTRows consecutive lines of one interface and one of the four passes, so
// that a line value is loaded and truncated once for up to 5 windows (8 rows instead of 20 for 4 segments);
// the four warps of a group take the four passes of the same 32 items and combine their bits through
// shared memory.  The launch lasts as long as its slowest warps, those on a shock, whose windows go
// through the exact chains one after the other: with all four passes in one thread (64 windows instead of 16)
// the four-quadrant step's launches took 64 us at 512^2 and 124 at 1024^2, so 36 and 106.
constexpr int kTRows = 4;
static_assert(kTRows == 4, "a warp of a group stores one row");

__device__ __forceinline__ void b_raw_tflags(const Params& P, const Sweep& S, const Ctrl* ctrl, long long id)
{
    if (ctrl->done) return;                                // the same for the block
    __shared__ unsigned int words[512];                    // the block's threads (at most 512, a multiple of 128)
    const int X = (int)(id >> 5) & 3, tid = threadIdx.x;
    const unsigned item = (unsigned)(id >> 7) * 32u + (unsigned)(tid & 31);
    const unsigned rg = item / (unsigned)S.nm;
    const int m = (int)(item - rg * (unsigned)S.nm);
    const int r0 = (int)rg * kTRows;                       // row of rawT: line r0 - 1
    const int rows = S.nt + 2 - r0 < kTRows ? S.nt + 2 - r0 : kTRows;
    unsigned word = 0;                                     // row r's bits in byte r
    if (rows > 0 && P.recon_mode == HGKS_RECON_HYBRID) {
#pragma unroll 1
        for (int k = 0; k < 4; k++) {
            double q[kTRows + 4];
            float f[kTRows + 4];
#pragma unroll
            for (int s = 0; s < kTRows + 4; s++) {
                // (lines past the last window repeat the last one: loaded, not used)
                q[s] = lineval(S, X, k, r0 - 3 + (s < rows + 4 ? s : rows + 3), m);
                f[s] = fixed::to_float(q[s]);
            }
#pragma unroll
            for (int r = 0; r < kTRows; r++)
                if (r < rows) word |= (unsigned)indicator_raw<false>(q + r, f + r, S.Z1t) << (8 * r + X);
        }
    }
    words[tid] = word;
    __syncthreads();
    if (X < rows) {                                        // (pass X's warp stores row X)
        const unsigned* w = words + (tid & ~127) + (tid & 31);
        stc(S.rawT + (long long)(r0 + X) * S.nm + m, ((w[0] | w[32] | w[64] | w[96]) >> (8 * X)) & 0xFFu, S);
    }
}

// Threads of the raw tangential flag kernel on sweep S.
inline long long raw_t_threads(const Sweep& S)
{
    return ((long long)((S.nt + 2 + kTRows - 1) / kTRows) * S.nm + 31) / 32 * 128;
}

__global__ void k_raw_tflags(const SolveDesc* D, int nb0)
{
    pdl_enter();
    const SweepBlock b = sweep_block(nb0);
    const SolveDesc& d = *D;
    b_raw_tflags(d.P, d.sw[b.dir], d.ctrl, b.id);
}


__device__ __forceinline__ void gp_positivity(const Params& P, const Sweep& S, int t, int m, int X, double (*v)[2], double (*d)[2])
{
    if (X > 1) return;
#pragma unroll
    for (int g = 0; g < 2; g++) {
        double Q[4] = {v[0][g], v[1][g], v[2][g], v[3][g]};
        if (nonphysical<4>(Q)) {
#pragma unroll
            for (int k = 0; k < 4; k++) { v[k][g] = lineval(S, X, k, t, m); d[k][g] = 0.0; }
        }
    }
}

// Large sweeps: the Step-4 spread flags of a segment (stored, counted, troubled passes appended
// to the WENO-AO work list); the smooth passes are reconstructed inside the flux kernel
// (b_flux, side_pair), so their Gauss-point states never go to memory.
__device__ __forceinline__ void b_tang(const Params& P, const Sweep& S, Ctrl* ctrl, int stage, long long id)
{
    if (ctrl->done) return;
    long long total = (long long)S.nt * S.nm;
    bool active = id < total;
    int m = 0, t = 0;
    unsigned int bits = 0;
    if (active) {
        m = (int)(id % S.nm); t = (int)(id / S.nm);
        if (P.recon_mode == HGKS_RECON_LINEAR) bits = 0;
        else if (P.recon_mode == HGKS_RECON_WENOAO) bits = 0xF;
        else bits = rdc(S.rawT + (long long)t * S.nm + m, S) | rdc(S.rawT + (long long)(t + 1) * S.nm + m, S)
                    | rdc(S.rawT + (long long)(t + 2) * S.nm + m, S);
        stc(S.flagT + id, bits, S);
    }
    warp_count(&ctrl->troubled[stage][S.dir][1], active ? (unsigned)__popc(bits) : 0u);
    // (a count known beforehand; with an atomic per warp for it and one per pass for the list the launch waited
    // on those few addresses: 54 us at 1024^2, now 16)
    if (id == 0) atomicAdd(&ctrl->examined[stage][S.dir][1], 4ull * (unsigned long long)total);
    warp_push4(&ctrl->cnt[S.dir][1], S.itemsT, bits, (uint32_t)(((long long)t * S.nm + m) << 2), S);
}

__global__ void k_tang(const SolveDesc* D, int nb0, int stage)
{
    pdl_enter();
    const SweepBlock b = sweep_block(nb0);
    const SolveDesc& d = *D;
    b_tang(d.P, d.sw[b.dir], d.ctrl, stage, b.id);
}


// The troubled tangential pass `it`: its pass X, segment (t, m), the eigenvectors at the face
// average (tangential direction) and the pass's 5 line values.
__device__ __forceinline__ void tang_ao_item(const Params& P, const Sweep& S, const double* W, uint32_t it,
                                             int& X, int& t, int& m, TangEig& e, double (*x)[4])
{
    X = it & 3;
    const uint32_t tm = it >> 2;
    t = (int)(tm / (uint32_t)S.nm); m = (int)(tm - (uint32_t)t * (uint32_t)S.nm);
    double qs[4];
    const double* cl = cellp(P, S, W, t, m - 1);
    const double* cr = cellp(P, S, W, t, m);
#pragma unroll
    for (int k = 0; k < 4; k++) {
        long long o = (long long)S.perm[k] * P.g.plane;
        qs[k] = scale2<-1>(ldc(cl + o, S) + ldc(cr + o, S));
    }
    tang_eig(P.gamma, qs, e);
#pragma unroll
    for (int s = 0; s < 5; s++)
#pragma unroll
        for (int k = 0; k < 4; k++) x[s][k] = lineval(S, X, k, t - 2 + s, m);
}

// The troubled tangential passes: one per lane (tang_ao) from kAoOneLaneMin items on, else one
// per aligned group of 4 lanes (tang_ao_x4, lane q computes and stores component q).  Free-order
// arithmetic (the outputs only feed the flux).  `lane`, `lanes`: this thread's index among, and
// the number of, the lanes working on the pass.
__device__ __forceinline__ void b_tang_ao(const Params& P, const Sweep& S, const double* W, const Ctrl* ctrl, long long lane, long long lanes)
{
    if (ctrl->done) return;
    unsigned int n = ctrl->cnt[S.dir][1];
    AOConst ak;
    for (int j = 0; j < 4; j++) ak.g[j] = P.g_ao[j];
    ak.g3inv = P.g3inv; ak.gr[0] = P.gr[0]; ak.gr[1] = P.gr[1]; ak.gr[2] = P.gr[2]; ak.eps = P.eps;
    // Gauss-point buffer: Q index 0 Wl, 1 Wlx, 2 Wly, 3 Wr, 4 Wrx, 5 Wry; pass X writes its values
    // to qv and (X = 0, 1) its tangential derivatives to qv + 2
    const long long plane = (long long)S.nt * S.nm;
    if (n >= kAoOneLaneMin) {
        for (unsigned int i = (unsigned int)lane; i < n; i += (unsigned int)lanes) {
            int X, t, m;
            TangEig e;
            double x[5][4], v[4][2], d[4][2];
            tang_ao_item(P, S, W, rdc(S.itemsT + i, S), X, t, m, e, x);
            tang_ao(e, x, ak, X <= 1, v, d);
            gp_positivity(P, S, t, m, X, v, d);
            const long long o = (long long)t * S.nm + m;
            const int qv = X == 0 ? 0 : (X == 1 ? 3 : (X == 2 ? 1 : 4));
#pragma unroll
            for (int k = 0; k < 4; k++)
#pragma unroll
                for (int g = 0; g < 2; g++) {
                    stc(S.gp + (long long)((g * 6 + qv) * 4 + k) * plane + o, v[k][g], S);
                    if (X <= 1) stc(S.gp + (long long)((g * 6 + qv + 2) * 4 + k) * plane + o, d[k][g] * S.inv_ht, S);
                }
        }
        return;
    }
    const int q = threadIdx.x & 3;
    const int lane0 = threadIdx.x & 28;
    const unsigned gmask = 0xFu << lane0;
    for (unsigned int i = (unsigned int)(lane >> 2); i < n; i += (unsigned int)(lanes >> 2)) {
        int X, t, m;
        TangEig e;
        double x[5][4], vq[2], dq[2];
        tang_ao_item(P, S, W, rdc(S.itemsT + i, S), X, t, m, e, x);
        tang_ao_x4(e, x, ak, X <= 1, gmask, vq, dq);
        if (X <= 1) {
            // positivity of the reconstructed Q^l, Q^r states (gp_positivity), on the gathered components
#pragma unroll
            for (int g = 0; g < 2; g++)
                if (nonphysical_x4<4>(vq[g], lane0, gmask)) { vq[g] = lineval(S, X, q, t, m); dq[g] = 0.0; }
        }
        const long long o = (long long)t * S.nm + m;
        const int qv = X == 0 ? 0 : (X == 1 ? 3 : (X == 2 ? 1 : 4));
#pragma unroll
        for (int g = 0; g < 2; g++) {
            stc(S.gp + (long long)((g * 6 + qv) * 4 + q) * plane + o, vq[g], S);
            if (X <= 1) stc(S.gp + (long long)((g * 6 + qv + 2) * 4 + q) * plane + o, dq[g] * S.inv_ht, S);
        }
    }
}

// The tangential WENO-AO pass and the flux contain products that the compiler may fuse into FMAs
// (free-order arithmetic).  They are compiled once, as non-inlined functions on a solver
// descriptor in device memory, and called by both a solver's own kernels and the batched
// kernels: the same machine code, so batched and solo results are bit-identical by construction.
__device__ __noinline__ void tang_ao_nl(const SolveDesc& d, int dir, int stage, long long lane, long long lanes)
{
    b_tang_ao(d.P, d.sw[dir], stage == 0 ? d.W : d.Ws, d.ctrl, lane, lanes);
}

__global__ void k_tang_ao(const SolveDesc* D, int nb0, int stage)
{
    pdl_enter();
    const SweepBlock b = sweep_block(nb0);
    tang_ao_nl(*D, b.dir, stage, b.id, b.lanes);
}


// Small sweeps: flags, quartics and WENO-AO of the four tangential passes in one launch.  A block of 4 warps
// takes 8 interfaces and `rows` consecutive lines, warp X pass X, 4 lanes an interface (lane q component q).  A
// warp walks along the lines with the window in registers: one load and one raw indicator per line, the
// decisions of the line before and the line after kept for the Step-4 spread.  Every pass ends in the
// Gauss-point buffer.  Free-order arithmetic: compiled once (tang_small_nl) like tang_ao_nl; it does not depend
// on `rows`, which is chosen for the number of blocks.
constexpr int kSmallCols = 8, kSmallRowsMax = 8, kSmallTangBlock = 128;

__device__ __forceinline__ void b_tang_small(const Params& P, const Sweep& S, const double* W, Ctrl* ctrl, int stage,
                                             unsigned block, int rows)
{
    __shared__ uint8_t s_flag[4][kSmallRowsMax][kSmallCols];
    if (ctrl->done) return;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, X = threadIdx.x >> 5, gi = lane >> 2, q = lane & 3;
    const int lane0 = lane & 28;
    const unsigned gmask = 0xFu << lane0;
    const unsigned nmb = (unsigned)(S.nm + kSmallCols - 1) / kSmallCols, tb = block / nmb;
    const int t0 = (int)tb * rows, m0 = (int)(block - tb * nmb) * kSmallCols;
    const int m = m0 + gi, mc = m < S.nm ? m : S.nm - 1;
    const bool inside = m < S.nm;
    const bool hybrid = P.recon_mode == HGKS_RECON_HYBRID;
    const long long total = (long long)S.nt * S.nm;
    const fixed::Scale inv = fixed::scale_of(S.inv_ht);
    AOConst ak;
    for (int j = 0; j < 4; j++) ak.g[j] = P.g_ao[j];
    ak.g3inv = P.g3inv; ak.gr[0] = P.gr[0]; ak.gr[1] = P.gr[1]; ak.gr[2] = P.gr[2]; ak.eps = P.eps;

    double v[6];                                 // lines t-2..t+3 (before the first line: t0-3..t0+2)
    float f[6];
    auto raw = [&](const double* vw, const float* fw) {
        unsigned r = (unsigned)indicator_raw<true>(vw, fw, S.Z1t);
        r |= __shfl_xor_sync(full, r, 1);
        return r | __shfl_xor_sync(full, r, 2);
    };
#pragma unroll
    for (int s = 0; s < 6; s++) { v[s] = lineval(S, X, q, t0 - 3 + s, mc); f[s] = fixed::to_float(v[s]); }
    unsigned before = 0, here = 0, troubled = 0, examined = 0;
    if (hybrid) { before = raw(v, f); here = raw(v + 1, f + 1); }
#pragma unroll 1
    for (int r = 0; r < rows; r++) {
        const int t = t0 + r;
        if (t >= S.nt) break;                    // the same for the block
#pragma unroll
        for (int s = 0; s < 5; s++) { v[s] = v[s + 1]; f[s] = f[s + 1]; }
        unsigned flag = P.recon_mode == HGKS_RECON_WENOAO ? 1u : 0u;
        if (hybrid) {
            v[5] = lineval(S, X, q, t + 3, mc);
            f[5] = fixed::to_float(v[5]);
            const unsigned after = raw(v + 1, f + 1);
            flag = before | here | after;
            before = here;
            here = after;
        } else if (r + 1 < rows && t + 1 < S.nt) {
            v[5] = lineval(S, X, q, t + 3, mc);
        }
        if (q == 0) {
            s_flag[X][r][gi] = (uint8_t)flag;
            troubled += inside ? flag : 0u;
            examined += inside ? 1u : 0u;
        }
        if (!inside) continue;                   // the same for a group
        double vq[2], dq[2] = {0.0, 0.0};
        if (!flag) {
            if (X <= 1) gauss_linear<true>(v, inv, S.inv_ht, vq, dq);
            else gauss_linear<false>(v, inv, S.inv_ht, vq, dq);
        } else {
            // the face average of the segment, one component a lane
            const long long oc = (long long)S.perm[q] * P.g.plane;
            const double avg = scale2<-1>(ldc(cellp(P, S, W, t, m - 1) + oc, S) + ldc(cellp(P, S, W, t, m) + oc, S));
            double qs[4], x[5][4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                qs[k] = __shfl_sync(gmask, avg, lane0 + k);
#pragma unroll
                for (int s = 0; s < 5; s++) x[s][k] = __shfl_sync(gmask, v[s], lane0 + k);
            }
            TangEig e;
            tang_eig(P.gamma, qs, e);
            tang_ao_x4(e, x, ak, X <= 1, gmask, vq, dq);
            dq[0] *= S.inv_ht;
            dq[1] *= S.inv_ht;
        }
        if (X <= 1) {
            // Reading: a reconstructed state with rho <= 0 or p <= 0 falls back to first order
#pragma unroll
            for (int g = 0; g < 2; g++)
                if (nonphysical_x4<4>(vq[g], lane0, gmask)) { vq[g] = v[2]; dq[g] = 0.0; }
        }
        // Q index: 0 Wl, 1 Wlx, 2 Wly, 3 Wr, 4 Wrx, 5 Wry
        const int qv = X == 0 ? 0 : (X == 1 ? 3 : (X == 2 ? 1 : 4));
        const long long o = (long long)t * S.nm + m;
#pragma unroll
        for (int g = 0; g < 2; g++) {
            stc(S.gp + (long long)((g * 6 + qv) * 4 + q) * total + o, vq[g], S);
            if (X <= 1) stc(S.gp + (long long)((g * 6 + qv + 2) * 4 + q) * total + o, dq[g], S);
        }
    }
    __syncwarp();
    warp_count(&ctrl->troubled[stage][S.dir][1], troubled);
    warp_count(&ctrl->examined[stage][S.dir][1], examined);
    __syncthreads();
    const int r = threadIdx.x / kSmallCols, j = threadIdx.x % kSmallCols;
    if (r < rows && t0 + r < S.nt && m0 + j < S.nm) {
        const unsigned bits = s_flag[0][r][j] | s_flag[1][r][j] << 1 | s_flag[2][r][j] << 2 | s_flag[3][r][j] << 3;
        stc(S.flagT + (long long)(t0 + r) * S.nm + m0 + j, bits, S);
    }
}

// Blocks of the small tangential launch on sweep S with `rows` lines a block; rows from the number of blocks
// that leaves: up to 8 while a launch still has 16 blocks for each SM.
inline long long tang_small_blocks(const Sweep& S, int rows)
{
    return (long long)((S.nm + kSmallCols - 1) / kSmallCols) * ((S.nt + rows - 1) / rows);
}
inline int tang_small_rows(long long blocks1, int sms)     // blocks1: blocks of the whole launch with one line a block
{
    const long long r = blocks1 / (16 * sms);
    return r < 1 ? 1 : r > kSmallRowsMax ? kSmallRowsMax : (int)r;
}

__device__ __noinline__ void tang_small_nl(const SolveDesc& d, int dir, int stage, unsigned block, int rows)
{
    b_tang_small(d.P, d.sw[dir], stage == 0 ? d.W : d.Ws, d.ctrl, stage, block, rows);
}

__global__ void __launch_bounds__(kSmallTangBlock) k_tang_small(const SolveDesc* D, int nb0, int stage, int rows)
{
    pdl_enter();
    const int dir = (int)blockIdx.x >= nb0 ? 1 : 0;
    tang_small_nl(*D, dir, stage, blockIdx.x - (dir ? (unsigned)nb0 : 0u), rows);
}

// ---------------------------------------------------------------- flux and update

// Shared memory of a 2D flux block of `threads`: the reconstructed side states (24 doubles a
// thread, see b_flux), then the segment fluxes of the Gauss point 1 warps (8 doubles a pair of threads).
constexpr int kFluxSideDoubles = 24;
inline size_t flux_smem(int dim, int threads)
{
    return dim == 2 ? (size_t)threads * (kFluxSideDoubles + 4) * sizeof(double) : 0;
}

// State, tangential and normal derivative of one side (0: left, 1: right) of segment (t, m) at both Gauss
// points (2D, large sweeps): the troubled passes from k_tang_ao, the smooth ones reconstructed
// here.  x[(12 g + j) stride]: j = 0..3 state, 4..7 normal, 8..11 tangential derivative at Gauss point g.
__device__ __forceinline__ void side_pair(const Params& P, const Sweep& S, int side, long long o, double* x, int stride)
{
    const long long per = (long long)S.nt * S.nm;
    const unsigned bits = rdc(S.flagT + o, S);
    const int t = (int)((unsigned)o / (unsigned)S.nm), m = (int)((unsigned)o - (unsigned)t * (unsigned)S.nm);   // o < 2^31
    // the Gauss-point buffer's quantities: 0 Wl, 1 Wlx, 2 Wly, 3 Wr, 4 Wrx, 5 Wry
    const double* gp = S.gp + (long long)(3 * side * 4) * per + o;
    const fixed::Scale inv = fixed::scale_of(S.inv_ht);
    if ((bits >> side) & 1) {
#pragma unroll 1
        for (int g = 0; g < 2; g++)
#pragma unroll
            for (int k = 0; k < 4; k++) {
                x[(12 * g + k) * stride] = ldc(gp + (long long)(24 * g + k) * per, S);
                x[(12 * g + 8 + k) * stride] = ldc(gp + (long long)(24 * g + 8 + k) * per, S);
            }
    } else {
        double v[4][2], d[2];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            double q[5];
#pragma unroll
            for (int j = 0; j < 5; j++) q[j] = lineval(S, side, k, t - 2 + j, m);
            gauss_linear<true>(q, inv, S.inv_ht, v[k], d);
            x[(8 + k) * stride] = d[0];
            x[(20 + k) * stride] = d[1];
        }
#pragma unroll
        for (int g = 0; g < 2; g++) {
            const double Q[4] = {v[0][g], v[1][g], v[2][g], v[3][g]};
            if (nonphysical<4>(Q)) {
                // Reading: a reconstructed state with rho <= 0 or p <= 0 falls back to first order
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    x[(12 * g + k) * stride] = lineval(S, side, k, t, m);
                    x[(12 * g + 8 + k) * stride] = 0.0;
                }
            } else {
#pragma unroll
                for (int k = 0; k < 4; k++) x[(12 * g + k) * stride] = Q[k];
            }
        }
    }
    if ((bits >> (2 + side)) & 1) {
#pragma unroll
        for (int g = 0; g < 2; g++)
#pragma unroll
            for (int k = 0; k < 4; k++) x[(12 * g + 4 + k) * stride] = ldc(gp + (long long)(24 * g + 4 + k) * per, S);
    } else {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            double q[5], v[2];
#pragma unroll
            for (int j = 0; j < 5; j++) q[j] = lineval(S, 2 + side, k, t - 2 + j, m);
            gauss_linear<false>(q, inv, S.inv_ht, v, nullptr);
            x[(4 + k) * stride] = v[0];
            x[(16 + k) * stride] = v[1];
        }
    }
}

// State Wv, normal derivative Wn and tangential derivative Wt (2D) of one side of segment o at Gauss point
// g: 1D from the line buffer; 2D from shared memory (large sweeps, side_pair) or, x = nullptr, from the
// Gauss-point buffer (small sweeps, where every pass was reconstructed before).
template <int DIM>
__device__ __forceinline__ void side_states(const Sweep& S, int side, int g, long long o, const double* x, int stride,
                                            double* Wv, double* Wn, double* Wt)
{
    constexpr int NV = DIM + 2;
    if constexpr (DIM == 2) {
        const long long per = (long long)S.nt * S.nm;
        if (!x) {
            const double* gp = S.gp + (long long)((g * 6 + 3 * side) * 4) * per + o;
#pragma unroll
            for (int k = 0; k < NV; k++) {
                Wv[k] = ldc(gp + (long long)k * per, S);
                Wn[k] = ldc(gp + (long long)(4 + k) * per, S);
                Wt[k] = ldc(gp + (long long)(8 + k) * per, S);
            }
        } else {
#pragma unroll
            for (int k = 0; k < NV; k++) {
                Wv[k] = x[(12 * g + k) * stride];
                Wn[k] = x[(12 * g + 4 + k) * stride];
                Wt[k] = x[(12 * g + 8 + k) * stride];
            }
        }
    } else {
        const long long plane = (long long)S.nlines * S.nm;
#pragma unroll
        for (int k = 0; k < NV; k++) {
            Wv[k] = ldc(S.line + (long long)(side * NV + k) * plane + o, S);
            Wn[k] = ldc(S.line + (long long)((2 + side) * NV + k) * plane + o, S);
            Wt[k] = 0.0;
        }
    }
}

// The segment's fluxes [output][component][segment].
template <int DIM, int STAGE>
__device__ __forceinline__ void store_flux(const Sweep& S, long long o, const double* o0, const double* o1)
{
    const long long per = (long long)S.nt * S.nm;
#pragma unroll
    for (int k = 0; k < DIM + 2; k++) {
        const int gk = S.perm[k];
        stc(S.flux + (long long)gk * per + o, o0[k], S);
        if (STAGE == 0) stc(S.flux + (long long)(DIM + 2 + gk) * per + o, o1[k], S);
    }
}

template <int DIM, int STAGE, bool PRFIX>
__device__ __forceinline__ void b_flux(const Params& P, const Sweep& S, Ctrl* ctrl, long long id)
{
    if (ctrl->done) return;                   // the same for every thread of a block
    constexpr int NV = DIM + 2;
    const long long per = (long long)S.nt * S.nm;
    // 2D: warps in pairs, warp 2w on Gauss point 0 and warp 2w + 1 on Gauss point 1 of the same
    // 32 segments, so that the pair shares its stencil reads in cache and sums the segment flux
    int g = 0;
    long long o = id;
    if constexpr (DIM == 2) {
        const long long warp = id >> 5;
        g = (int)(warp & 1);
        o = ((warp >> 1) << 5) + (id & 31);
    }
    const bool valid = o < per;
    double o0[NV], o1[NV];
    extern __shared__ double flux_sh[];
    const int stride = blockDim.x;
    const int pair0 = threadIdx.x & ~32;         // this thread's lane in the pair's first warp
    if constexpr (DIM == 2) {
        // warp 0 of the pair reconstructs the left side at both Gauss points, warp 1 the right side, and they
        // exchange through shared memory: every line value is loaded and converted once, and the two points
        // share their products (with the products in FP64 and each warp reconstructing both sides at its own
        // point the launch took 5.04 ms at 1024^2, so 4.18 ms)
        if (valid) side_pair(P, S, g, o, flux_sh + threadIdx.x, stride);
        __syncthreads();
    }
    if (valid) {
    // one side after the other: only the side at work holds its states and slopes in registers
    FluxSums<DIM> sums;
    double pl, pr;
    bool ok;
    {
        double Wv[NV], Wn[NV], Wt[NV];
        side_states<DIM>(S, 0, g, o, flux_sh + pair0, stride, Wv, Wn, Wt);
        ok = flux_side<DIM, PRFIX, true>(P.fc, Wv, Wn, Wt, true, sums, pl);
    }
    if (ok) {
        double Wv[NV], Wn[NV], Wt[NV];
        side_states<DIM>(S, 1, g, o, flux_sh + pair0 + 32, stride, Wv, Wn, Wt);
        ok = flux_side<DIM, PRFIX, false>(P.fc, Wv, Wn, Wt, false, sums, pr);
    }
    if (ok) ok = flux_finish<DIM, STAGE, PRFIX>(P.fc, sums, pl, pr, ctrl->dt, o0, o1);
    if (!ok) {
        // a non-physical state: the status is latched and the flux is a NaN, so that what the
        // failed step leaves behind does not depend on anything but the solve itself
        ctrl->status = HGKS_ENONPHYSICAL;
        const double nan = __longlong_as_double(0x7FF8000000000000LL);
#pragma unroll
        for (int k = 0; k < NV; k++) { o0[k] = nan; o1[k] = nan; }
    }
    }
    // the segment flux, the sum over the two Gauss points (their weight 1/2 is in the update's 1/dx, exactly):
    // the Gauss point 1 warp hands its fluxes to its partner
    // through shared memory
    if constexpr (DIM == 2) {
        // [output component][lane pair]
        double* pair = flux_sh + kFluxSideDoubles * stride + ((threadIdx.x >> 6) << 5) + (threadIdx.x & 31);
        const int ps = stride >> 1;
        if (g == 1 && valid) {
#pragma unroll
            for (int k = 0; k < NV; k++) {
                pair[k * ps] = o0[k];
                if (STAGE == 0) pair[(NV + k) * ps] = o1[k];
            }
        }
        __syncthreads();
        if (g == 1 || !valid) return;
#pragma unroll
        for (int k = 0; k < NV; k++) {
            o0[k] += pair[k * ps];
            if (STAGE == 0) o1[k] += pair[(NV + k) * ps];
        }
    } else {
        if (!valid) return;
    }
    store_flux<DIM, STAGE>(S, o, o0, o1);
}

// Small sweeps: the two sides of a Gauss point on two warps, so that a thread's chain is one side (about 160
// FP64 instructions) and, on the left side's warp, the sums' completion (about 150) instead of two sides and
// the completion.  2D: 4 warps on the same 32 segments (side = warp & 1, Gauss point = warp >> 1 of the 4);
// 1D: 2 warps.  The right side's sums and the second point's fluxes go through shared memory, one column
// per left thread.  Per launch: 200 cells in 1D 18 -> 15 us, 48 x 48 29 -> 21, 200 x 100 (Prandtl fix) 124 -> 111.
template <int DIM, bool PRFIX>
__host__ __device__ constexpr int flux_sums() { return (PRFIX ? 8 : 6) * (DIM + 2) + 1; }

inline size_t flux_small_smem(int dim, bool prfix, int threads)
{
    const int n = dim == 2 ? (prfix ? flux_sums<2, true>() : flux_sums<2, false>())
                           : (prfix ? flux_sums<1, true>() : flux_sums<1, false>());
    return (size_t)threads / 2 * n * sizeof(double);
}

template <int DIM, int STAGE, bool PRFIX>
__device__ __forceinline__ void b_flux_small(const Params& P, const Sweep& S, Ctrl* ctrl, long long id)
{
    if (ctrl->done) return;                   // the same for every thread of a block
    constexpr int NV = DIM + 2, NS = flux_sums<DIM, PRFIX>(), NVEC = PRFIX ? 8 : 6;
    const long long warp = id >> 5;
    const int side = (int)(warp & 1), g = DIM == 2 ? (int)(warp >> 1) & 1 : 0;
    const long long o = ((warp >> DIM) << 5) + (id & 31);
    const bool valid = o < (long long)S.nt * S.nm;
    const int cols = blockDim.x >> 1;
    extern __shared__ double flux_sh[];
    double* col = flux_sh + ((threadIdx.x >> 6) << 5) + (threadIdx.x & 31);
    FluxSums<DIM> q;
    double* vec[8] = {q.Wc, q.Wx, q.Wy, q.S4, q.S5, q.S6n, q.D5, q.D6n};
    const double nan = __longlong_as_double(0x7FF8000000000000LL);
    double p = 0.0;
    bool ok = false;
    if (valid) {
        double Wv[NV], Wn[NV], Wt[NV];
        side_states<DIM>(S, side, g, o, nullptr, 0, Wv, Wn, Wt);
        ok = flux_side<DIM, PRFIX, true>(P.fc, Wv, Wn, Wt, side == 0, q, p);
        if (side == 1) {
            if (!ok) q.Wc[0] = nan;             // the completion finds the state non-physical
#pragma unroll
            for (int j = 0; j < NVEC; j++) {
                if ((DIM == 1 && j == 2) || (j >= 3 && P.fc.tau_zero)) continue;
#pragma unroll
                for (int k = 0; k < NV; k++) col[(j * NV + k) * cols] = vec[j][k];
            }
            col[(NS - 1) * cols] = p;
        }
    }
    __syncthreads();
    double o0[NV], o1[NV];
    if (valid && side == 0) {
        const double pr = col[(NS - 1) * cols];
#pragma unroll
        for (int j = 0; j < NVEC; j++) {
            if ((DIM == 1 && j == 2) || (j >= 3 && P.fc.tau_zero)) continue;
#pragma unroll
            for (int k = 0; k < NV; k++) vec[j][k] += col[(j * NV + k) * cols];
        }
        if (ok) ok = flux_finish<DIM, STAGE, PRFIX>(P.fc, q, p, pr, ctrl->dt, o0, o1);
        if (!ok) {
            // the status is latched and the flux is a NaN (see b_flux)
            ctrl->status = HGKS_ENONPHYSICAL;
#pragma unroll
            for (int k = 0; k < NV; k++) { o0[k] = nan; o1[k] = nan; }
        }
        if (DIM == 2 && g == 1) {
#pragma unroll
            for (int k = 0; k < NV; k++) {
                col[k * cols] = o0[k];
                if (STAGE == 0) col[(NV + k) * cols] = o1[k];
            }
        }
    }
    if constexpr (DIM == 2) {
        __syncthreads();
        if (g == 0 && side == 0 && valid) {
            const double* c1 = col + 32;          // Gauss point 1 of the same segment
#pragma unroll
            for (int k = 0; k < NV; k++) {
                o0[k] += c1[k * cols];
                if (STAGE == 0) o1[k] += c1[(NV + k) * cols];
            }
        }
    }
    if (g == 0 && side == 0 && valid) store_flux<DIM, STAGE>(S, o, o0, o1);
}

inline long long flux_small_threads(int dim, long long per) { return (dim == 2 ? 4 : 2) * ((per + 31) / 32) * 32; }

// Threads of a 2D flux launch for a sweep of `per` segments: two Gauss points per segment, the
// segments padded to whole warps (see b_flux).
inline long long flux_threads(int dim, long long per) { return dim == 2 ? 2 * ((per + 31) / 32) * 32 : per; }


template <int DIM, int STAGE, bool PRFIX>
__device__ __noinline__ void flux_nl(const SolveDesc& d, int dir, long long id)
{
    b_flux<DIM, STAGE, PRFIX>(d.P, d.sw[dir], d.ctrl, id);
}

// 64-thread blocks, at least 4 per SM: the register budget this leaves (up to 256 per thread at
// 8 warps per SM) lets the flux keep its working set in registers (measured 3.5 % faster than
// under a 128-thread bound at the same occupancy, when the flux took all 255; it takes 138 now, 174 with
// the Prandtl fix)
template <int DIM, int STAGE, bool PRFIX>
__global__ void __launch_bounds__(64, 4) k_flux(const SolveDesc* D, int nb0)
{
    pdl_enter();
    const SweepBlock b = sweep_block(nb0);
    flux_nl<DIM, STAGE, PRFIX>(*D, b.dir, b.id);
}

template <int DIM, int STAGE, bool PRFIX>
__device__ __noinline__ void flux_small_nl(const SolveDesc& d, int dir, long long id)
{
    b_flux_small<DIM, STAGE, PRFIX>(d.P, d.sw[dir], d.ctrl, id);
}

constexpr int kFluxSmallBlock = 128;

template <int DIM, int STAGE, bool PRFIX>
__global__ void __launch_bounds__(kFluxSmallBlock) k_flux_small(const SolveDesc* D, int nb0)
{
    pdl_enter();
    const SweepBlock b = sweep_block(nb0);
    flux_small_nl<DIM, STAGE, PRFIX>(*D, b.dir, b.id);
}

// Stage 0: W* = W^n - dF(dt/2)/dx - dG(dt/2)/dy (Eq. (19)), Acc = W^n - d(dt F^n + dt^2/6 dF^n)/dx - ...
// Stage 1: W^{n+1} = Acc - d(dt^2/3 dF*)/dx - ... (Eqs. (20)-(22))
template <int DIM, int STAGE>
__device__ __forceinline__ void b_update(const Params& P, const Sweep& Sx, const Sweep& Sy, const double* Win, double* Wout, double* Acc, Ctrl* ctrl, long long id)
{
    if (ctrl->done) return;
    if (STAGE == 1 && id == 0) {              // the end of the step (no thread of this launch reads these)
        ctrl->t += ctrl->dt;
        ctrl->last_dt = ctrl->dt;
        ctrl->steps += 1;
    }
    constexpr int NV = DIM + 2;
    const GridGeom& g = P.g;
    int rowsI = DIM == 2 ? g.ny : 1;
    long long n = (long long)rowsI * g.nx;
    if (id >= n) return;
    int i = (int)(id % g.nx), j = (int)(id / g.nx);
    long long cell = g.origin + (long long)j * g.pitch + i;
    // 1/dx, 1/dy (host-divided), in 2D times the Gauss weight 1/2 of the segment fluxes
    const double inv_dx = DIM == 2 ? scale2<-1>(Sx.inv_hn) : Sx.inv_hn, inv_dy = DIM == 2 ? scale2<-1>(Sy.inv_hn) : 0.0;
    long long perx = (long long)Sx.nt * Sx.nm, pery = DIM == 2 ? (long long)Sy.nt * Sy.nm : 0;
    long long ox = (long long)j * Sx.nm + i, oy = (long long)i * (DIM == 2 ? Sy.nm : 0) + j;
    double out[NV], acc[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) {
        double fx0[2], fx1[2], fy0[2] = {0, 0}, fy1[2] = {0, 0};
        // segment fluxes [output][component][segment] of the interfaces on either side
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const double* fb = Sx.flux;
            fx0[s] = ldc(fb + (long long)(0 * NV + k) * perx + ox + s, g);
            fx1[s] = STAGE == 0 ? ldc(fb + (long long)(1 * NV + k) * perx + ox + s, g) : 0.0;
            if constexpr (DIM == 2) {
                const double* gb = Sy.flux;
                fy0[s] = ldc(gb + (long long)(0 * NV + k) * pery + oy + s, g);
                fy1[s] = STAGE == 0 ? ldc(gb + (long long)(1 * NV + k) * pery + oy + s, g) : 0.0;
            }
        }
        if (STAGE == 0) {
            double w = ldc(Win + cell + (long long)k * g.plane, g);
            double ws = fma(-(fx0[1] - fx0[0]), inv_dx, w);
            double wa = fma(-(fx1[1] - fx1[0]), inv_dx, w);
            if (DIM == 2) { ws = fma(-(fy0[1] - fy0[0]), inv_dy, ws); wa = fma(-(fy1[1] - fy1[0]), inv_dy, wa); }
            out[k] = ws; acc[k] = wa;
        } else {
            double a = ldc(Acc + cell + (long long)k * g.plane, g);
            double wn = fma(-(fx0[1] - fx0[0]), inv_dx, a);
            if (DIM == 2) wn = fma(-(fy0[1] - fy0[0]), inv_dy, wn);
            out[k] = wn;
        }
    }
#pragma unroll
    for (int k = 0; k < NV; k++) {
        stc(Wout + cell + (long long)k * g.plane, out[k], g);
        if (STAGE == 0) stc(Acc + cell + (long long)k * g.plane, acc[k], g);
    }
    // rho > 0 and p > 0, the latter as rho E - |m|^2/2 > 0 (no division; first in FP32, see fixed::surely_physical)
    if (fixed::surely_physical(fixed::to_float(out[0]), fixed::to_float(out[1]), DIM == 2 ? fixed::to_float(out[2]) : 0.0f,
                        fixed::to_float(out[NV - 1])))
        return;
    double ke = DIM == 2 ? 0.5 * fma(out[1], out[1], out[2] * out[2]) : 0.5 * out[1] * out[1];
    double pr = fma(out[NV - 1], out[0], -ke);
    if (!fixed::is_pos(out[0]) || !fixed::is_pos(pr) || !fixed::is_finite(out[0]) || !fixed::is_finite(pr)) ctrl->status = HGKS_ENONPHYSICAL;
}

template <int DIM, int STAGE>
__global__ void k_update(Params P, Sweep Sx, Sweep Sy, const double* Win, double* Wout,
                         double* Acc, Ctrl* ctrl)
{
    pdl_enter();
    b_update<DIM, STAGE>(P, Sx, Sy, Win, Wout, Acc, ctrl, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}


// ---------------------------------------------------------------- batched kernels
// One launch per kernel class covers the blocks of every solver of a batch: block b belongs
// to solver s with boff[s] <= b < boff[s+1] and runs that solver's kernel body on its local
// block index.  No block mixes solvers, so every result is bit-identical to stepping alone.
__device__ __forceinline__ int find_solve(const int* boff, int n, int b)
{
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (boff[mid] <= b) lo = mid; else hi = mid;
    }
    return lo;
}

#define HGKS_BATCH_BLOCK()                                                              \
    const int s_ = find_solve(boff, n, (int)blockIdx.x);                                 \
    const SolveDesc& d = D[s_];                                                          \
    const long long lblk_ = (long long)blockIdx.x - boff[s_];                            \
    const long long nblk_ = (long long)(boff[s_ + 1] - boff[s_]);                         \
    const long long id = lblk_ * blockDim.x + threadIdx.x;                               \
    (void)nblk_; (void)id;

// sweep classes: the units are (solver, sweep) pairs, unit u = 2 s + dir; n counts solvers
#define HGKS_BATCH_SWEEP_BLOCK()                                                        \
    const int u_ = find_solve(boff, 2 * n, (int)blockIdx.x);                             \
    const SolveDesc& d = D[u_ >> 1];                                                     \
    const int dir = u_ & 1;                                                              \
    const long long lblk_ = (long long)blockIdx.x - boff[u_];                            \
    const long long nblk_ = (long long)(boff[u_ + 1] - boff[u_]);                         \
    const long long id = lblk_ * blockDim.x + threadIdx.x;                               \
    (void)nblk_; (void)id;

__global__ void kb_dt(const SolveDesc* D, const int* boff, int n, const double* tend)
{
    pdl_enter();
    HGKS_BATCH_BLOCK();
    if (!(d.P.fixed_dt > 0.0)) b_dt(d.P, d.W, d.ctrl, d.h, id, nblk_ * blockDim.x);
    dt_finish(d.P, d.ctrl, tend[s_], (unsigned)nblk_);
}

__global__ void kb_ghost(const SolveDesc* D, const int* boff, int n, int stage)
{
    pdl_enter();
    HGKS_BATCH_BLOCK();
    if (d.ctrl->done) return;
    b_ghost(d.P, stage == 0 ? d.W : d.Ws, d.ctrl, stage, id);
}

template <int NV>
__global__ void kb_raw_nflags(const SolveDesc* D, const int* boff, int n, int stage)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    b_raw_nflags<NV>(d.P, d.sw[dir], stage == 0 ? d.W : d.Ws, d.ctrl, id);
}

template <int NV>
__global__ void kb_normal(const SolveDesc* D, const int* boff, int n, int stage)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    b_normal<NV>(d.P, d.sw[dir], stage == 0 ? d.W : d.Ws, d.ctrl, stage, id);
}

template <int NV>
__global__ void kb_normal_ao(const SolveDesc* D, const int* boff, int n, int stage)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    b_normal_ao<NV>(d.P, d.sw[dir], stage == 0 ? d.W : d.Ws, d.ctrl, id, nblk_ * blockDim.x);
}

template <int NV>
__global__ void kb_normal_small(const SolveDesc* D, const int* boff, int n, int stage)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    b_normal_small<NV>(d.P, d.sw[dir], stage == 0 ? d.W : d.Ws, d.ctrl, stage, id);
}

__global__ void __launch_bounds__(kSmallTangBlock) kb_tang_small(const SolveDesc* D, const int* boff, int n, int stage, int rows)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    tang_small_nl(d, dir, stage, (unsigned)lblk_, rows);
}

__global__ void kb_raw_tflags(const SolveDesc* D, const int* boff, int n)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    b_raw_tflags(d.P, d.sw[dir], d.ctrl, id);
}

__global__ void kb_tang(const SolveDesc* D, const int* boff, int n, int stage)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    b_tang(d.P, d.sw[dir], d.ctrl, stage, id);
}

__global__ void kb_tang_ao(const SolveDesc* D, const int* boff, int n, int stage)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    tang_ao_nl(d, dir, stage, id, nblk_ * blockDim.x);
}

template <int DIM, int STAGE, bool PRFIX>
__global__ void __launch_bounds__(64, 4) kb_flux(const SolveDesc* D, const int* boff, int n)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    flux_nl<DIM, STAGE, PRFIX>(d, dir, id);
}

template <int DIM, int STAGE, bool PRFIX>
__global__ void __launch_bounds__(kFluxSmallBlock) kb_flux_small(const SolveDesc* D, const int* boff, int n)
{
    pdl_enter();
    HGKS_BATCH_SWEEP_BLOCK();
    flux_small_nl<DIM, STAGE, PRFIX>(d, dir, id);
}

template <int DIM, int STAGE>
__global__ void kb_update(const SolveDesc* D, const int* boff, int n)
{
    pdl_enter();
    HGKS_BATCH_BLOCK();
    if (STAGE == 0) b_update<DIM, 0>(d.P, d.sw[0], d.sw[1], d.W, d.Ws, d.Acc, d.ctrl, id);
    else b_update<DIM, 1>(d.P, d.sw[0], d.sw[1], d.Ws, d.W, d.Acc, d.ctrl, id);
}

// Threads of the small-sweep normal launch: a warp per 6 cells of -1..nn, side and line.
inline long long normal_small_threads(const Sweep& S)
{
    return (long long)((S.nn + 2 + kSmallCells - 1) / kSmallCells) * 2 * S.nlines * 32;
}

inline unsigned int blocks_for(long long n, int tpb) { return (unsigned int)((n + tpb - 1) / tpb); }

// ---------------------------------------------------------------- FP64 rate probe
// Eight independent DFMA chains per thread: with 8 warps per SM scheduler slot the FP64 pipe
// never waits on a result, so the launch runs at the FMA issue rate of the device.  The sum is
// stored only under a condition the data never meet, which keeps the chains live.
__device__ double g_probe_sink;

__global__ void __launch_bounds__(256) k_dfma_probe(int iters, double seed)
{
    const double m = 0.9999999999, c = 1e-12;
    double a0 = seed + threadIdx.x * 1e-9, a1 = a0 + 1e-3, a2 = a0 + 2e-3, a3 = a0 + 3e-3;
    double a4 = a0 + 4e-3, a5 = a0 + 5e-3, a6 = a0 + 6e-3, a7 = a0 + 7e-3;
    for (int i = 0; i < iters; i++) {
        a0 = fma(a0, m, c); a1 = fma(a1, m, c); a2 = fma(a2, m, c); a3 = fma(a3, m, c);
        a4 = fma(a4, m, c); a5 = fma(a5, m, c); a6 = fma(a6, m, c); a7 = fma(a7, m, c);
    }
    const double s = ((a0 + a1) + (a2 + a3)) + ((a4 + a5) + (a6 + a7));
    if (s == -1.0) g_probe_sink = s;
}

}  // namespace

cudaError_t launch_dfma_probe(cudaStream_t st, int blocks, int iters)
{
    k_dfma_probe<<<blocks, 256, 0, st>>>(iters, 1.0);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- reciprocal check
// The flux's fixed-point reciprocal (rcp_nr) against IEEE division, and its reciprocal square
// root (rsqrt_nr) against IEEE division by the IEEE square root, on n arguments spread
// log-uniformly over 1e-8..1e8 (both signs for the reciprocal; splitmix64 hashes of the index);
// the largest differences in units in the last place go to g_rcp_max_ulp[0], [1].
__device__ unsigned long long g_rcp_max_ulp[2];

__global__ void k_rcp_check(long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long z = (unsigned long long)i + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const double u = (double)(z >> 11) * (1.0 / 9007199254740992.0);      // [0, 1)
    double x = exp10(16.0 * u - 8.0);
    if (z & 1) x = -x;
    auto ulps = [](double a, double b) {
        const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
        return (unsigned long long)(ia > ib ? ia - ib : ib - ia);
    };
    atomicMax(&g_rcp_max_ulp[0], ulps(rcp_nr(x), 1.0 / x));
    const double ax = fabs(x);
    atomicMax(&g_rcp_max_ulp[1], ulps(rsqrt_nr(ax), 1.0 / sqrt(ax)));
}

cudaError_t rcp_check(long long n, unsigned long long* max_ulp)
{
    const unsigned long long zero[2] = {0, 0};
    cudaError_t e = cudaMemcpyToSymbol(g_rcp_max_ulp, zero, sizeof(zero));
    if (e != cudaSuccess) return e;
    k_rcp_check<<<(unsigned)((n + 255) / 256), 256>>>(n);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return cudaMemcpyFromSymbol(max_ulp, g_rcp_max_ulp, 2 * sizeof(*max_ulp));
}

int debug_bounds_read(unsigned long long* count, unsigned long long* first)
{
#ifdef HGKS_DEBUG_BOUNDS
    cudaError_t e = cudaMemcpyFromSymbol(count, g_dbg_count, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(first, g_dbg_first, sizeof(unsigned long long));
    return e == cudaSuccess ? 1 : -1;
#else
    *count = 0;
    *first = 0;
    return 0;
#endif
}

int device_sm_count()
{
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

// ---------------------------------------------------------------- host: timing helpers
static cudaEvent_t take_event(hgks_solver* s)
{
    if (!s->event_pool.empty()) { cudaEvent_t e = s->event_pool.back(); s->event_pool.pop_back(); return e; }
    cudaEvent_t e;
    cudaEventCreate(&e);
    return e;
}

// NVTX range around the enqueue of one kernel class (named as in kclass_names), so that a
// timeline tool attributes the launches to their class; free when no tool is attached.
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
};

template <typename F>
static void timed(hgks_solver* s, int cls, int nkernels, F&& launch)
{
    NvtxRange range(kclass_names[cls]);
    s->launches += nkernels;
    if (!s->timing) { launch(); return; }
    cudaEvent_t a = take_event(s), b = take_event(s);
    cudaEventRecord(a, s->stream);
    launch();
    cudaEventRecord(b, s->stream);
    s->timers.push_back(TimerRec{cls, a, b});
}

template <class... K, class... A>
static void launch_chained(void (*kernel)(K...), unsigned int grid, int threads, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, (K)args...);
}

// The sweep kernels of one stage, each class one launch over both sweeps (2D): nb[0] blocks for
// the x sweep, then nb[1] for the y sweep.
template <int DIM>
static void enqueue_sweeps(hgks_solver* s, int stage)
{
    const Params& P = s->P;
    cudaStream_t st = s->stream;
    const SolveDesc* D = s->d_self;
    constexpr int NV = DIM + 2;
    const int sms = device_sm_count();
    // nb: the blocks of each sweep, none for a sweep of the other size class; returns their sum
    enum { LARGE = 0, SMALL = 1, ALL = 2 };
    unsigned int nb[2];
    auto pair = [&](int which, auto blocks) {
        for (int d = 0; d < 2; d++) nb[d] = d < DIM && (which == ALL || s->sw[d].small == which) ? blocks(s->sw[d]) : 0u;
        return nb[0] + nb[1];
    };
    // the compacted WENO-AO passes: a grid for 4 lanes per possible item, capped at 8 blocks per SM
    auto ao_blocks = [&](long long maxn) {
        unsigned int b = blocks_for(maxn, 128);
        return b > (unsigned)(sms * 8) ? (unsigned)(sms * 8) : b;
    };
    unsigned int g;
    if ((g = pair(LARGE, [](const Sweep& S) { return blocks_for((long long)S.nlines * (S.nn + 4), TPB); })))
        timed(s, KC_RAWN, 1, [&] { launch_chained(k_raw_nflags<NV>, g, TPB, 0, st, D, (int)nb[0], stage); });
    if ((g = pair(LARGE, [](const Sweep& S) { return blocks_for((long long)S.nlines * S.nm, TPB); })))
        timed(s, KC_NORMAL, 1, [&] { launch_chained(k_normal<NV>, g, TPB, 0, st, D, (int)nb[0], stage); });
    if ((g = pair(LARGE, [&](const Sweep& S) { return ao_blocks((long long)S.nlines * S.nm * 2 * 4); })))
        timed(s, KC_NORMAL_AO, 1, [&] { launch_chained(k_normal_ao<NV>, g, 128, 0, st, D, (int)nb[0], stage); });
    if ((g = pair(SMALL, [](const Sweep& S) { return blocks_for(normal_small_threads(S), 128); })))
        timed(s, KC_NORMAL, 1, [&] { launch_chained(k_normal_small<NV>, g, 128, 0, st, D, (int)nb[0], stage); });
    if constexpr (DIM == 2) {
        if ((g = pair(LARGE, [](const Sweep& S) { return blocks_for(raw_t_threads(S), TPB); })))
            timed(s, KC_RAWT, 1, [&] { launch_chained(k_raw_tflags, g, TPB, 0, st, D, (int)nb[0]); });
        if ((g = pair(LARGE, [](const Sweep& S) { return blocks_for((long long)S.nt * S.nm, TPB); })))
            timed(s, KC_TANG, 1, [&] { launch_chained(k_tang, g, TPB, 0, st, D, (int)nb[0], stage); });
        if ((g = pair(LARGE, [&](const Sweep& S) { return ao_blocks((long long)S.nt * S.nm * 4 * 4); })))
            timed(s, KC_TANG_AO, 1, [&] { launch_chained(k_tang_ao, g, 128, 0, st, D, (int)nb[0], stage); });
        const int rows = tang_small_rows(pair(SMALL, [](const Sweep& S) { return (unsigned)tang_small_blocks(S, 1); }), sms);
        if ((g = pair(SMALL, [&](const Sweep& S) { return (unsigned)tang_small_blocks(S, rows); })))
            timed(s, KC_TANG, 1, [&] { launch_chained(k_tang_small, g, kSmallTangBlock, 0, st, D, (int)nb[0], stage, rows); });
    }
    if (s->capture) {
        for (int d = 0; d < DIM; d++) {
            const Sweep& S = s->sw[d];
            size_t nbytes = (size_t)S.nlines * (S.nn + 2);
            cudaMemcpyAsync(s->cap[stage][d][0], S.flagN, nbytes, cudaMemcpyDeviceToDevice, st);
            if (DIM == 2) cudaMemcpyAsync(s->cap[stage][d][1], S.flagT, (size_t)S.nt * S.nm, cudaMemcpyDeviceToDevice, st);
        }
    }
    auto flux = [&](auto prfix) {
        constexpr bool PR = decltype(prfix)::value;
        if ((g = pair(LARGE, [](const Sweep& S) { return blocks_for(flux_threads(DIM, (long long)S.nt * S.nm), 64); })))
            timed(s, KC_FLUX, 1, [&] {
                if (stage == 0) launch_chained(k_flux<DIM, 0, PR>, g, 64, flux_smem(DIM, 64), st, D, (int)nb[0]);
                else launch_chained(k_flux<DIM, 1, PR>, g, 64, flux_smem(DIM, 64), st, D, (int)nb[0]);
            });
        constexpr int T = kFluxSmallBlock;
        if ((g = pair(SMALL, [](const Sweep& S) { return blocks_for(flux_small_threads(DIM, (long long)S.nt * S.nm), T); })))
            timed(s, KC_FLUX, 1, [&] {
                if (stage == 0) launch_chained(k_flux_small<DIM, 0, PR>, g, T, flux_small_smem(DIM, PR, T), st, D, (int)nb[0]);
                else launch_chained(k_flux_small<DIM, 1, PR>, g, T, flux_small_smem(DIM, PR, T), st, D, (int)nb[0]);
            });
    };
    if (P.fc.prfix != 0.0) flux(std::true_type{});
    else flux(std::false_type{});
}

template <int DIM>
static void enqueue_stage(hgks_solver* s, int stage)
{
    NvtxRange range(stage == 0 ? "S2O4 stage 1" : "S2O4 stage 2");
    const Params& P = s->P;
    cudaStream_t st = s->stream;
    if (stage == 1)
        timed(s, KC_GHOST, 1, [&] { launch_chained(k_ghost, blocks_for(ghost_threads(P.g), TPB), TPB, 0, st, P, s->Ws, s->ctrl); });
    enqueue_sweeps<DIM>(s, stage);
    timed(s, KC_UPDATE, 1, [&] {
        long long n = (long long)(DIM == 2 ? P.g.ny : 1) * P.g.nx;
        if (stage == 0) launch_chained(k_update<DIM, 0>, blocks_for(n, TPB), TPB, 0, st, P, s->sw[0], s->sw[1], s->W, s->Ws, s->Acc, s->ctrl);
        else launch_chained(k_update<DIM, 1>, blocks_for(n, TPB), TPB, 0, st, P, s->sw[0], s->sw[1], s->Ws, s->W, s->Acc, s->ctrl);
    });
}

cudaError_t launch_step(hgks_solver* s, double t_end)
{
    NvtxRange range("hgks_step");
    const Params& P = s->P;
    cudaStream_t st = s->stream;
    const double h = P.g.dim == 2 ? (P.g.dx < P.g.dy ? P.g.dx : P.g.dy) : P.g.dx;
    timed(s, KC_DT, 1, [&] {
        unsigned int nb = 1;
        if (!(P.fixed_dt > 0.0)) {
            nb = blocks_for((long long)(P.g.dim == 2 ? P.g.ny : 1) * P.g.nx, TPB);
            const unsigned int cap = (unsigned)device_sm_count() * 4;
            if (nb > cap) nb = cap;
        }
        launch_chained(k_dt_ghost, nb + blocks_for(ghost_threads(P.g), TPB), TPB, 0, st, P, s->W, s->ctrl, h, t_end, (int)nb);
    });
    if (P.g.dim == 2) { enqueue_stage<2>(s, 0); enqueue_stage<2>(s, 1); }
    else { enqueue_stage<1>(s, 0); enqueue_stage<1>(s, 1); }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- host: batched step
const int kBatchTpbDefault[BK_COUNT] = {
    256, 256,                 // dt, ghost cells
    256,                      // raw normal flags
    256,                      // normal reconstruction
    128,                      // normal WENO-AO
    128,                      // normal reconstruction of small sweeps
    256,                      // raw tangential flags
    256,                      // tangential flags
    128,                      // tangential WENO-AO
    128,                      // tangential reconstruction of small sweeps
    64, 64,                   // flux of large sweeps (Pr = 1, Prandtl fix)
    kFluxSmallBlock, kFluxSmallBlock,   // flux of small sweeps
    256                       // update
};

void batch_fill_desc(const hgks_solver* s, SolveDesc& d)
{
    d.P = s->P;
    d.sw[0] = s->sw[0];
    d.sw[1] = s->sw[1];
    d.W = s->W;
    d.Ws = s->Ws;
    d.Acc = s->Acc;
    d.ctrl = s->ctrl;
    d.h = s->P.g.dim == 2 ? (s->P.g.dx < s->P.g.dy ? s->P.g.dx : s->P.g.dy) : s->P.g.dx;
}

// Blocks of one unit of class c with t threads per block: solver d (sweep dir for the sweep classes).
static long long batch_unit_blocks(const SolveDesc& d, int dim, int c, int dir, int t, int rows)
{
    const GridGeom& g = d.P.g;
    const Sweep& S = d.sw[dir];
    const long long cells = (long long)(dim == 2 ? g.ny : 1) * g.nx;
    if (batch_sweep_class(c) && dir >= dim) return 0;          // 1D: no y sweep
    if (dim == 1 && c >= BK_RAWT && c <= BK_TSMALL) return 0;
    // the sweep classes of the other size, and the flux classes of the other Prandtl variant
    const bool small_class = c == BK_NSMALL || c == BK_TSMALL || c == BK_FSMALL || c == BK_FSMALL_PR;
    if (batch_sweep_class(c) && small_class != (S.small != 0)) return 0;
    const bool pr = d.P.fc.prfix != 0.0;
    if (((c == BK_FLUX || c == BK_FSMALL) && pr) || ((c == BK_FLUX_PR || c == BK_FSMALL_PR) && !pr)) return 0;
    long long b = 0;
    switch (c) {
        case BK_DT: b = (cells + (long long)t * 8 - 1) / ((long long)t * 8); break;
        case BK_GHOST: b = blocks_for(ghost_threads(g), t); break;
        case BK_RAWN: b = blocks_for((long long)S.nlines * (S.nn + 4), t); break;
        case BK_NORMAL: b = blocks_for((long long)S.nlines * S.nm, t); break;
        case BK_NAO: b = blocks_for((long long)S.nlines * S.nm * 2 * 4, t * 8); break;
        case BK_NSMALL: b = blocks_for(normal_small_threads(S), t); break;
        case BK_RAWT: b = blocks_for(raw_t_threads(S), t); break;
        case BK_TANG: b = blocks_for((long long)S.nt * S.nm, t); break;
        case BK_TAO: b = blocks_for((long long)S.nt * S.nm * 4 * 4, t * 8); break;
        case BK_TSMALL: b = tang_small_blocks(S, rows); break;
        case BK_FLUX: case BK_FLUX_PR: b = blocks_for(flux_threads(dim, (long long)S.nt * S.nm), t); break;
        case BK_FSMALL: case BK_FSMALL_PR: b = blocks_for(flux_small_threads(dim, (long long)S.nt * S.nm), t); break;
        case BK_UPD: b = blocks_for(cells, t); break;
    }
    return b < 1 ? 1 : b;
}

void batch_plan(const std::vector<const SolveDesc*>& descs, int dim, const int* tpb, BatchPlan& plan)
{
    const int n = (int)descs.size();
    const size_t stride = (size_t)2 * n + 1;
    plan.n = n;
    plan.dim = dim;
    for (int c = 0; c < BK_COUNT; c++) plan.tpb[c] = tpb[c];
    long long blocks1 = 0;
    for (int u = 0; u < 2 * n; u++) blocks1 += batch_unit_blocks(*descs[u >> 1], dim, BK_TSMALL, u & 1, tpb[BK_TSMALL], 1);
    plan.tang_rows = tang_small_rows(blocks1, device_sm_count());
    plan.boff.assign((size_t)BK_COUNT * stride, 0);
    for (int c = 0; c < BK_COUNT; c++) {
        int* bo = plan.boff.data() + (size_t)c * stride;
        const bool sw = batch_sweep_class(c);
        const int units = sw ? 2 * n : n;
        long long acc = 0;
        for (int u = 0; u < units; u++) {
            bo[u] = (int)acc;
            acc += sw ? batch_unit_blocks(*descs[u >> 1], dim, c, u & 1, tpb[c], plan.tang_rows)
                      : batch_unit_blocks(*descs[u], dim, c, 0, tpb[c], 1);
        }
        bo[units] = (int)acc;
        plan.nblk[c] = (int)acc;
    }
}

cudaError_t batch_enqueue_step(const BatchPlan& plan, const SolveDesc* dd, const int* dboff, const double* dtend,
                               cudaStream_t st, cudaEvent_t* ev)
{
    NvtxRange range("hgks_batch_step");
    const int n = plan.n;
    const int dim = plan.dim;
    auto bo = [&](int c) { return dboff + (size_t)c * (2 * n + 1); };
    auto mark = [&](int c, int which) { if (ev) cudaEventRecord(ev[2 * c + which], st); };
    auto grid = [&](int c) { return (unsigned int)plan.nblk[c]; };
    auto tp = [&](int c) { return plan.tpb[c]; };
    mark(BK_DT, 0);
    launch_chained(kb_dt, grid(BK_DT), tp(BK_DT), 0, st, dd, bo(BK_DT), n, dtend);
    mark(BK_DT, 1);
    for (int stage = 0; stage < 2; stage++) {
        mark(BK_GHOST, 0);
        launch_chained(kb_ghost, grid(BK_GHOST), tp(BK_GHOST), 0, st, dd, bo(BK_GHOST), n, stage);
        mark(BK_GHOST, 1);
        // every sweep class: one launch over both sweeps of every solver it applies to
        auto sweep = [&](int c, auto launch) {
            if (!grid(c)) return;
            mark(c, 0);
            launch();
            mark(c, 1);
        };
#define HGKS_BY_DIM(kernel, c) sweep(c, [&] {                                                          \
            if (dim == 2) launch_chained(kernel<4>, grid(c), tp(c), 0, st, dd, bo(c), n, stage);                      \
            else launch_chained(kernel<3>, grid(c), tp(c), 0, st, dd, bo(c), n, stage); })
        HGKS_BY_DIM(kb_raw_nflags, BK_RAWN);
        HGKS_BY_DIM(kb_normal, BK_NORMAL);
        HGKS_BY_DIM(kb_normal_ao, BK_NAO);
        HGKS_BY_DIM(kb_normal_small, BK_NSMALL);
#undef HGKS_BY_DIM
        sweep(BK_RAWT, [&] { launch_chained(kb_raw_tflags, grid(BK_RAWT), tp(BK_RAWT), 0, st, dd, bo(BK_RAWT), n); });
        sweep(BK_TANG, [&] { launch_chained(kb_tang, grid(BK_TANG), tp(BK_TANG), 0, st, dd, bo(BK_TANG), n, stage); });
        sweep(BK_TAO, [&] { launch_chained(kb_tang_ao, grid(BK_TAO), tp(BK_TAO), 0, st, dd, bo(BK_TAO), n, stage); });
        sweep(BK_TSMALL, [&] { launch_chained(kb_tang_small, grid(BK_TSMALL), kSmallTangBlock, 0, st, dd, bo(BK_TSMALL), n, stage, plan.tang_rows); });
        auto flux = [&](auto dimc, auto prfix) {
            constexpr int DIM = decltype(dimc)::value;
            constexpr bool PR = decltype(prfix)::value;
            const int cl = PR ? BK_FLUX_PR : BK_FLUX, cs = PR ? BK_FSMALL_PR : BK_FSMALL;
            sweep(cl, [&] {
                if (stage == 0) launch_chained(kb_flux<DIM, 0, PR>, grid(cl), tp(cl), flux_smem(DIM, tp(cl)), st, dd, bo(cl), n);
                else launch_chained(kb_flux<DIM, 1, PR>, grid(cl), tp(cl), flux_smem(DIM, tp(cl)), st, dd, bo(cl), n);
            });
            sweep(cs, [&] {
                if (stage == 0) launch_chained(kb_flux_small<DIM, 0, PR>, grid(cs), tp(cs), flux_small_smem(DIM, PR, tp(cs)), st, dd, bo(cs), n);
                else launch_chained(kb_flux_small<DIM, 1, PR>, grid(cs), tp(cs), flux_small_smem(DIM, PR, tp(cs)), st, dd, bo(cs), n);
            });
        };
        auto flux_dim = [&](auto dimc) { flux(dimc, std::false_type{}); flux(dimc, std::true_type{}); };
        if (dim == 2) flux_dim(std::integral_constant<int, 2>{});
        else flux_dim(std::integral_constant<int, 1>{});
        mark(BK_UPD, 0);
        const int tu = tp(BK_UPD);
        if (dim == 2) {
            if (stage == 0) launch_chained(kb_update<2, 0>, grid(BK_UPD), tu, 0, st, dd, bo(BK_UPD), n);
            else launch_chained(kb_update<2, 1>, grid(BK_UPD), tu, 0, st, dd, bo(BK_UPD), n);
        } else {
            if (stage == 0) launch_chained(kb_update<1, 0>, grid(BK_UPD), tu, 0, st, dd, bo(BK_UPD), n);
            else launch_chained(kb_update<1, 1>, grid(BK_UPD), tu, 0, st, dd, bo(BK_UPD), n);
        }
        mark(BK_UPD, 1);
    }
    return cudaGetLastError();
}

static unsigned int copy_blocks(const GridGeom& g)
{
    const unsigned int b = blocks_for((long long)g.nv * g.ny * g.nx, TPB), cap = (unsigned)device_sm_count() * 16;
    return b < cap ? b : cap;
}

cudaError_t launch_state_in(hgks_solver* s, const double* W, double t0)
{
    launch_chained(k_state_in, copy_blocks(s->P.g), TPB, 0, s->stream, s->P.g, W, s->W, s->ctrl, t0);
    return cudaGetLastError();
}

cudaError_t launch_noalloc_in(hgks_solver* s, const SolveDesc& self, const double* W)
{
    launch_chained(k_noalloc_in, copy_blocks(s->P.g), TPB, 0, s->stream, self, s->d_self, W);
    return cudaGetLastError();
}

cudaError_t launch_state_out(hgks_solver* s, double* W)
{
    launch_chained(k_state_out, copy_blocks(s->P.g), TPB, 0, s->stream, s->P.g, s->W, W);
    return cudaGetLastError();
}

cudaError_t launch_set_time(hgks_solver* s, double t0)
{
    k_set_time<<<1, 1, 0, s->stream>>>(s->ctrl, t0);
    return cudaGetLastError();
}

}  // namespace hgks
