// stage_short.cu -- the stage kernel for batches with too few cells to fill
// the chip with tall work items (one small domain, a few domains).
//
// The same Runge-Kutta stage as stage.cu on the same work list, for items of
// at most kShortRows rows.  There the chip is not short of issue slots but of
// items, and a stage takes as long as one item: a chain of loads, barriers and
// dependent arithmetic.  So this kernel shortens that chain:
//   - an item is one pass: its rows and their halo (at most 14 rows, which the
//     ring holds) are loaded and derived at once, with no prologue and no
//     sweep, and with what the cell update will need (W^n, dF_s/dt, the raw
//     stage input) put into shared memory in the same phase, so that no
//     later phase waits for global memory;
//   - 16 warps instead of 8, so that every face of an item of up to 7 rows
//     (h x-face rows and h + 1 y-face rows, one per warp) is computed at the
//     same time instead of x-faces, then y-faces;
//   - the last warp claims the CTA's next item and looks up its neighbours
//     while the current item's faces run; each warp of the cell update
//     releases its own rows; the wait for the neighbours polls without sleeping.
#include <mutex>

#include "stage_device.cuh"

namespace eulbfs {

namespace {

// FP32C: 16 warps.  FP64: 8, so that two CTAs share an SM and one's loads, waits
// and short phases pass under the other's arithmetic (the FP64 pipe takes 64
// clocks per warp instruction and sub-core: 8 warps keep it fed).
template <class R> struct Short;
template <> struct Short<float> { static constexpr int rows = kShortRows; };
template <> struct Short<double> { static constexpr int rows = kShortRows64; };
template <class R, int PER_SM>
constexpr int kThreads = sizeof(R) == 8 && PER_SM == 2 ? 256 : 512;
constexpr int kShortDeps = 64;       // neighbours kept in shared memory (9 one-row items of 3 or 4 strips fit)

template <class R>
struct ShortSmem : Core<R> {
    // the cell update's inputs: W^n and the stage input by plane, F_s^{n-1} or dF_s/dt
    R wn[Prec<R>::NP][Short<R>::rows][32];
    R ws[Prec<R>::NP][Short<R>::rows][32];
    R frac[Short<R>::rows][32];
    // the CTA's next work item, put here by the control warp while the
    // current one runs: its place in the launch, and what it waits for
    int4 item;
    int pos;                  // position in the launch's item sequence (>= its length: no more)
    int stage, index;         // stage of the launch, index in the work list
    int ndeps, dep0;          // neighbours, and their offset in dep_idx
    int dep[kShortDeps];      // the first kShortDeps of them
    int ready;                // the current item's inputs are done
};

// An item's done flag counts up to kDone: its updating warps add to it one by
// one, each after its own stores.
constexpr int kDone = kShortRows;

// Put item number g of the launch into S (one whole warp).
template <class R>
__device__ __forceinline__ void look_up(ShortSmem<R>& S, const StageLaunch& a, int g, int lane) {
    if (g < a.nitems * a.stages) {
        const int2 si = stage_item(a, g);
        const int4 item = a.items[si.y];
        int d0 = 0, n = 0;
        if (a.stages > 1 && si.x > 0) {   // one-stage launches are ordered by the kernel boundary
            d0 = a.dep_off[si.y];
            n = a.dep_off[si.y + 1] - d0;
            for (int j = lane; j < min(n, kShortDeps); j += 32) S.dep[j] = a.dep_idx[d0 + j];
        }
        if (lane == 0) {
            S.item = item;
            S.stage = si.x;
            S.index = si.y;
            S.ndeps = n;
            S.dep0 = d0;
        }
    }
    if (lane == 0) S.pos = g;
}

// Wait until every item that the current one reads has finished the previous
// stage (one warp; lanes take one neighbour each).  A bounded wait, as
// next_ready of stage.cu, but it polls without sleeping: the next stage
// starts when the slowest neighbour's flag is seen.
template <class R>
__device__ __forceinline__ bool wait_deps(const ShortSmem<R>& S, const StageLaunch& a, int st, int n, int lane) {
    const int* done = a.done + (size_t)(st - 1) * a.nitems;
    bool ok = true;
    for (int j = lane; j < n; j += 32) {
        const int* f = done + (j < kShortDeps ? S.dep[j] : a.dep_idx[S.dep0 + j]);
        if (ld_acquire(f) >= kDone) continue;
        const long long t0 = clock64();
        while (ld_acquire(f) < kDone)
            if (clock64() - t0 > (1LL << 31)) { ok = false; break; }
    }
    return __all_sync(0xffffffffu, ok);
}

__device__ __forceinline__ void add_release(int* p, int v) {
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void put_cell(float (*p)[Short<float>::rows][32], int r, int l, const SV<float>& w) {
    p[0][r][l] = w.Hh; p[1][r][l] = w.Hl; p[2][r][l] = w.p; p[3][r][l] = w.mx; p[4][r][l] = w.my;
    p[5][r][l] = w.Ch; p[6][r][l] = w.Cl;
}
__device__ __forceinline__ void put_cell(double (*p)[Short<double>::rows][32], int r, int l, const SV<double>& w) {
    p[0][r][l] = w.Hh; p[1][r][l] = w.p; p[2][r][l] = w.mx; p[3][r][l] = w.my; p[4][r][l] = w.Ch;
}
__device__ __forceinline__ SV<float> get_cell(const float (*p)[Short<float>::rows][32], int r, int l) {
    return SV<float>{p[0][r][l], p[1][r][l], p[2][r][l], p[3][r][l], p[4][r][l], p[5][r][l], p[6][r][l]};
}
__device__ __forceinline__ SV<double> get_cell(const double (*p)[Short<double>::rows][32], int r, int l) {
    return SV<double>{p[0][r][l], 0.0, p[1][r][l], p[2][r][l], p[3][r][l], p[4][r][l], 0.0};
}

// The cell update's inputs from shared memory.
template <class R>
struct SharedCell {
    const ShortSmem<R>& S;
    int row, lane;
    __device__ __forceinline__ R frac() const { return S.frac[row][lane]; }
    __device__ __forceinline__ SV<R> wn() const { return get_cell(S.wn, row, lane); }
    __device__ __forceinline__ SV<R> ws() const { return get_cell(S.ws, row, lane); }
};

// The halo of an item, narrowing away from its rows: what is read of the rows at
// distance 1 are ring columns 1 .. RW-2 (mu_c of the item's own end columns), at
// distance 2 columns 2 .. RW-3 and at distance 3 columns 3 .. RW-4 (C alone).  So
// an item of 8 rows has 37 x 8 + 198 = 494 cells, one for each of the 512 threads;
// the rectangle's 518 took one warp through a second round of loads.
// us per step: 400x200 22.8 -> 21.6, 333x251 22.4 -> 21.7, 256^2 20.1 (both).  Lower
// items and FP64 (bound by its arithmetic) keep the rectangle, whose indices are
// quicker: 1024x4 in one-row items 12.3, narrowing 12.6; FP64 256x4 44.7 (44.9).
template <class R, int PER_SM>
constexpr bool kNarrow = sizeof(R) == 4 && PER_SM == 2;
constexpr int kHalo1 = 2 * (RW - 2), kHalo2 = kHalo1 + 2 * (RW - 4), kHaloCells = kHalo2 + 2 * (RW - 6);

// Halo cell j of an item of `rows` rows: its row relative to the item's first, its
// ring column, and whether it lies at distance 3.
__device__ __forceinline__ bool halo_cell(int j, int rows, int& rr, int& cc) {
    int d = 1;
    if (j >= kHalo1) { d = 2; j -= kHalo1; }
    if (d == 2 && j >= kHalo2 - kHalo1) { d = 3; j -= kHalo2 - kHalo1; }
    const int w = RW - 2 * d;
    const bool above = j >= w;
    cc = d + (above ? j - w : j);
    rr = above ? rows - 1 + d : -d;
    return d == 3;
}

// Load and derive cell (gx, gy) into ring column cc; a halo cell outside the
// domain is mapped through the boundary rules (as load_rows).  Of the outer
// rows (the third halo row on both sides) only C is ever read, by mu_c.
template <class R>
__device__ __forceinline__ SV<R> ring_cell(ShortSmem<R>& S, const R* in, int gx, int gy, int cc, bool inside,
                                           bool outer) {
    const Consts<R>& K = S.K;
    int sx = gx, sy = gy, kx = 0, ky = 0, sdx = XLO, sdy = YLO;
    if (!inside) {
        map_axis(gx, K.nx, K.per_x, XLO, sx, kx, sdx);
        map_row(K, gy, sy, ky, sdy);
    }
    const SV<R> w = load_state(in, K.plane, (long long)sy * K.nx + sx + K.off);
    if (outer) {
        R C = pair_sum(w.Ch, w.Cl);
        if (kx) C = ghost_C(K, sdx, kx, wall_wetting(K, in, sdx, sy), C);
        if (ky) C = ghost_C(K, sdy, ky, wall_wetting(K, in, sdy, gx), C);
        S.P.rc[slot(gy)][cc].y = C;
        return w;
    }
    Prim<R> q = derive(K, w);
    if (!inside) {
        // x sides first, then y (corners)
        if (kx) apply_ghost(K, sdx, kx, true, wall_wetting(K, in, sdx, sy), q);
        if (ky) apply_ghost(K, sdy, ky, false, wall_wetting(K, in, sdy, gx), q);
    }
    store_prim(S, slot(gy), cc, q);
    return w;
}

// One work item: rows [y0, y1) (at most kShortRows) of the strip at x0.
// `claim`: the control warp's claimed next position, looked up in here.
template <class R, bool AXI, bool GEN, int NTS, bool NARROW>
__device__ __forceinline__ void short_item(ShortSmem<R>& S, const StageLaunch& a, const int stage, int x0, int y0,
                                           int y1, int claim) {
    constexpr int NWS = NTS / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Consts<R>& K = S.K;
    const R* in = reinterpret_cast<const R*>(K.st[stage]);
    const int rows = y1 - y0;

    column_radii<R, AXI>(S, x0);
    // all loads of the item in one go: the update's inputs of cell (ur, ul) ...
    const int ur = tid / kStripX, ul = tid - ur * kStripX;
    const bool upd = ur < rows && x0 + ul < K.nx;
    SV<R> wn = {};
    R fr = R(0);
    if (upd) {
        const long long c = (long long)(y0 + ur) * K.nx + x0 + ul + K.off;
        fr = ld_l2(reinterpret_cast<const R*>(stage == 0 ? K.Fsp : K.dFs) + c);
        if (stage != 0) wn = load_state(reinterpret_cast<const R*>(K.st[0]), K.plane, c);
    }
    // ... and the rows with their halo
    const bool inside = x0 >= kHalo && x0 + kStripX + kHalo <= K.nx && y0 - kHalo >= -K.hlo && y1 + kHalo <= K.ny + K.hhi;
    constexpr int low = NARROW ? 0 : -kHalo;   // the first row that comes whole
    const int own = (rows - 2 * low) * RW;
    for (int idx = tid; idx < own + (NARROW ? kHaloCells : 0); idx += NTS) {
        int rr = idx / RW, cc = idx - rr * RW;
        rr += low;
        bool outer = !NARROW && (rr == -kHalo || rr == rows + kHalo - 1);
        if (NARROW && idx >= own) outer = halo_cell(idx - own, rows, rr, cc);
        const SV<R> w = ring_cell(S, in, x0 + cc - kHalo, y0 + rr, cc, inside, outer);
        const int ic = cc - kHalo;
        if (rr >= 0 && rr < rows && ic >= 0 && ic < kStripX) put_cell(S.ws, rr, ic, w);
    }
    if (upd) {
        S.frac[ur][ul] = fr;
        if (stage != 0) put_cell(S.wn, ur, ul, wn);
    }
    const R ir_c = AXI ? wdiv(R(1), (R)(x0 + lane) + R(0.5)) : R(1);
    const R ir_f = (AXI && x0 + lane > 0) ? wdiv(R(1), (R)(x0 + lane)) : R(0);
    __syncthreads();
    // (of a halo that narrows, the end columns on either side take values of cells
    // that were not loaded; nothing reads those)
    muc_rows<R, AXI, NTS>(S, x0, y0 - 2, rows + 4);
    __syncthreads();
    if (warp == NWS - 1) look_up(S, a, __shfl_sync(0xffffffffu, claim, 0), lane);
    // face rows: x-faces of every row, then the y-faces below and above every row
#pragma unroll 1
    for (int t = warp; t < 2 * rows + 1; t += NWS) {
        if (t < rows) x_face<R, AXI, GEN>(S, x0, y0 + t, t, lane, ir_f);
        else if (lane < kStripX) y_face<R, AXI, GEN>(S, y0 + t - rows, lane, AXI ? ir_c : R(0));
    }
    __syncthreads();
    if (warp < rows && lane < kStripX && x0 + lane < K.nx) {
        const SharedCell<R> src{S, warp, lane};
        const long long c = (long long)(y0 + warp) * K.nx + x0 + lane + K.off;
        if (stage == 0) {   // W^n is the stage input
            struct First {
                const SharedCell<R>& s;
                __device__ __forceinline__ R frac() const { return s.frac(); }
                __device__ __forceinline__ SV<R> wn() const { return s.ws(); }
                __device__ __forceinline__ SV<R> ws() const { return s.ws(); }
            };
            cell_update<R, AXI>(S, First{src}, 0, c, y0 + warp, warp, lane, ir_c, a.flag);
        } else {
            cell_update<R, AXI>(S, src, stage, c, y0 + warp, warp, lane, ir_c, a.flag);
        }
    }
}

}  // namespace

// PER_SM: resident CTAs per SM.  1 is for batches of at most one item per SM:
// twice the registers, so nothing spills and more loads are in flight.
template <class R, int PER_SM>
__global__ void __launch_bounds__(kThreads<R, PER_SM>, PER_SM) short_kernel(StageLaunch a) {
    constexpr int NTS = kThreads<R, PER_SM>, NWS = NTS / 32;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    ShortSmem<R>& S = *reinterpret_cast<ShortSmem<R>*>(smem_raw);
    const int tid = threadIdx.x;
    const Consts<R>* consts = static_cast<const Consts<R>*>(a.consts);
    int* const counter = a.work + (a.stages == 1 ? a.stage : 0);
    const int lane = tid & 31, warp = tid >> 5;
    launch_dependents();
    wait_prior();
    // items are claimed in order, one ahead, as in stage.cu: every item waits
    // only for items claimed before it
    if (warp == NWS - 1) {
        int g = 0;
        if (lane == 0) g = atomicAdd(counter, 1);
        look_up(S, a, __shfl_sync(0xffffffffu, g, 0), lane);
    }
    __syncthreads();
    int domain = -1;
    // From here to the barrier below, warps may still be in the previous
    // item's cell update: only S.ready is written.  The look-up of the item
    // after this one comes behind two more barriers.
    while (S.pos < a.nitems * a.stages) {
        const int4 item = S.item;
        const int st = S.stage, index = S.index;
        if (item.x != domain) {
            if (domain >= 0) __syncthreads();   // the previous item is done with S.K
            domain = item.x;
            const unsigned* src = reinterpret_cast<const unsigned*>(consts + domain);
            unsigned* dst = reinterpret_cast<unsigned*>(&S.K);
            for (int k = tid; k < (int)(sizeof(Consts<R>) / 4); k += NTS) dst[k] = src[k];
        }
        if (warp == 0) {
            const bool ready = S.ndeps == 0 || wait_deps(S, a, st, S.ndeps, lane);
            if (lane == 0) S.ready = ready;
        }
        __syncthreads();                 // S.K, S.ready; the previous item is done with shared memory
        if (!S.ready) {                  // a bounded wait gave up: report it and stop
            if (tid == 0) atomicOr(a.flag, 2);
            return;
        }
        int claim = 0;
        if (tid == NTS - 32) claim = atomicAdd(counter, 1);
        const int x0 = item.y * kStripX;
        const int stage = st % 3;
        if (S.K.gen) {
            if (S.K.axi) short_item<R, true, true, NTS, kNarrow<R, PER_SM>>(S, a, stage, x0, item.z, item.w, claim);
            else short_item<R, false, true, NTS, kNarrow<R, PER_SM>>(S, a, stage, x0, item.z, item.w, claim);
        } else {
            if (S.K.axi) short_item<R, true, false, NTS, kNarrow<R, PER_SM>>(S, a, stage, x0, item.z, item.w, claim);
            else short_item<R, false, false, NTS, kNarrow<R, PER_SM>>(S, a, stage, x0, item.z, item.w, claim);
        }
        const int rows = item.w - item.z;
        if (a.stages > 1 && warp < rows && !a.dep_probe) {
            __syncwarp();                // every lane's stores of this row
            if (lane == 0) add_release(a.done + (size_t)st * a.nitems + index, warp == 0 ? kDone + 1 - rows : 1);
        }
    }
}

namespace {

constexpr int kMaxAttrDevices = 64;

// The dynamic shared-memory limit is a per-device attribute (see stage.cu).
template <class R, int PER_SM>
cudaError_t configure_t() {
    static std::mutex m;
    static bool done[kMaxAttrDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(m);
    if (!done[dev]) {
        e = cudaFuncSetAttribute(short_kernel<R, PER_SM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(ShortSmem<R>));
        if (e != cudaSuccess) return e;
        done[dev] = true;
    }
    return cudaSuccess;
}

template <class R, int PER_SM>
cudaError_t launch_t(const StageLaunch& a, int grid, cudaStream_t s) {
    cudaError_t e = configure_t<R, PER_SM>();
    if (e != cudaSuccess) return e;
    return launch_behind(a.behind, short_kernel<R, PER_SM>, dim3(grid), kThreads<R, PER_SM>, sizeof(ShortSmem<R>), s, a);
}

template <class R>
int blocks_per_sm_t() {
    if (configure_t<R, 2>() != cudaSuccess) return 1;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, short_kernel<R, 2>, kThreads<R, 2>, sizeof(ShortSmem<R>)) != cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

}  // namespace

cudaError_t launch_short(int precision, const StageLaunch& a, int grid, bool one_per_sm, cudaStream_t s) {
    if (one_per_sm) return precision == 0 ? launch_t<double, 1>(a, grid, s) : launch_t<float, 1>(a, grid, s);
    return precision == 0 ? launch_t<double, 2>(a, grid, s) : launch_t<float, 2>(a, grid, s);
}

int short_blocks_per_sm(int precision) { return precision == 0 ? blocks_per_sm_t<double>() : blocks_per_sm_t<float>(); }

}  // namespace eulbfs
