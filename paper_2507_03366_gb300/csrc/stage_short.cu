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
//   - the wait for the neighbouring items of the previous stage polls without
//     sleeping, and the CTA's next item is claimed while the current one runs.
#include <mutex>

#include "stage_device.cuh"

namespace eulbfs {

namespace {

constexpr int NTS = kShortThreads;   // 16 warps
constexpr int NWS = NTS / 32;

template <class R>
struct ShortSmem : Core<R> {
    // the cell update's inputs: W^n and the stage input by plane, F_s^{n-1} or dF_s/dt
    R wn[Prec<R>::NP][kShortRows][32];
    R ws[Prec<R>::NP][kShortRows][32];
    R frac[kShortRows][32];
    int cur_domain;
    int next;      // the CTA's next position in the launch's item sequence
    int ready;     // the current item's inputs are done
};

__device__ __forceinline__ void put_cell(float (*p)[kShortRows][32], int r, int l, const SV<float>& w) {
    p[0][r][l] = w.Hh; p[1][r][l] = w.Hl; p[2][r][l] = w.p; p[3][r][l] = w.mx; p[4][r][l] = w.my;
    p[5][r][l] = w.Ch; p[6][r][l] = w.Cl;
}
__device__ __forceinline__ void put_cell(double (*p)[kShortRows][32], int r, int l, const SV<double>& w) {
    p[0][r][l] = w.Hh; p[1][r][l] = w.p; p[2][r][l] = w.mx; p[3][r][l] = w.my; p[4][r][l] = w.Ch;
}
__device__ __forceinline__ SV<float> get_cell(const float (*p)[kShortRows][32], int r, int l) {
    return SV<float>{p[0][r][l], p[1][r][l], p[2][r][l], p[3][r][l], p[4][r][l], p[5][r][l], p[6][r][l]};
}
__device__ __forceinline__ SV<double> get_cell(const double (*p)[kShortRows][32], int r, int l) {
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

// Cell idx of the item's rows with halo: load its raw state.
template <class R>
struct HaloCell {
    int gx, gy, sx, sy, kx, ky, sdx, sdy;
};

template <class R>
__device__ __forceinline__ SV<R> fetch_cell(const Consts<R>& K, const R* in, int gx, int gy, HaloCell<R>& h) {
    h.gx = gx;
    h.gy = gy;
    map_axis(gx, K.nx, K.per_x, XLO, h.sx, h.kx, h.sdx);
    map_row(K, gy, h.sy, h.ky, h.sdy);
    return load_state(in, K.plane, (long long)h.sy * K.nx + h.sx + K.off);
}

template <class R>
__device__ __forceinline__ void derive_cell(ShortSmem<R>& S, const R* in, const HaloCell<R>& h, const SV<R>& w,
                                            int cc) {
    const Consts<R>& K = S.K;
    Prim<R> q = derive(K, w);
    // x sides first, then y (corners), as load_rows
    if (h.kx) apply_ghost(K, h.sdx, h.kx, true, wall_wetting(K, in, h.sdx, h.sy), q);
    if (h.ky) apply_ghost(K, h.sdy, h.ky, false, wall_wetting(K, in, h.sdy, h.gx), q);
    store_prim(S, slot(h.gy), cc, q);
}

// One work item: rows [y0, y1) (at most kShortRows) of the strip at x0.
template <class R, bool AXI, bool GEN>
__device__ __forceinline__ void short_item(ShortSmem<R>& S, const StageLaunch& a, const int stage, int x0, int y0,
                                           int y1) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Consts<R>& K = S.K;
    const R* in = reinterpret_cast<const R*>(K.st[stage]);
    const int rows = y1 - y0;

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
    const int total = (rows + 2 * kHalo) * RW;
    for (int idx = tid; idx < total; idx += NTS) {
        const int rr = idx / RW, cc = idx - rr * RW;
        HaloCell<R> h;
        const SV<R> w = fetch_cell(K, in, x0 + cc - kHalo, y0 + rr - kHalo, h);
        const int ir = rr - kHalo, ic = cc - kHalo;
        if (ir >= 0 && ir < rows && ic >= 0 && ic < kStripX) put_cell(S.ws, ir, ic, w);
        derive_cell(S, in, h, w, cc);
    }
    if (upd) {
        S.frac[ur][ul] = fr;
        if (stage != 0) put_cell(S.wn, ur, ul, wn);
    }
    const R ir_c = AXI ? wdiv(R(1), (R)(x0 + lane) + R(0.5)) : R(1);
    const R ir_f = (AXI && x0 + lane > 0) ? wdiv(R(1), (R)(x0 + lane)) : R(0);
    __syncthreads();
    muc_rows<R, AXI, NTS>(S, x0, y0 - 2, rows + 4);
    __syncthreads();
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

template <class R>
__global__ void __launch_bounds__(NTS, sizeof(R) == 4 ? 2 : 1) short_kernel(StageLaunch a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    ShortSmem<R>& S = *reinterpret_cast<ShortSmem<R>*>(smem_raw);
    const int tid = threadIdx.x;
    const Consts<R>* consts = static_cast<const Consts<R>*>(a.consts);
    int* const counter = a.work + (a.stages == 1 ? a.stage : 0);
    if (tid == 0) {
        S.cur_domain = -1;
        S.next = atomicAdd(counter, 1);
    }
    __syncthreads();
    // items are claimed in order, one ahead, as in stage.cu: every item waits
    // only for items claimed before it
    while (S.next < a.nitems * a.stages) {
        const int2 si = stage_item(a, S.next);
        const int4 item = a.items[si.y];
        const bool other = item.x != S.cur_domain;
        __syncthreads();                 // every thread has read S.next and S.cur_domain
        int claimed = 0;
        if (tid == 0) claimed = atomicAdd(counter, 1);
        if (other) {
            const unsigned* src = reinterpret_cast<const unsigned*>(consts + item.x);
            unsigned* dst = reinterpret_cast<unsigned*>(&S.K);
            for (int k = tid; k < (int)(sizeof(Consts<R>) / 4); k += NTS) dst[k] = src[k];
            if (tid == 0) S.cur_domain = item.x;
        }
        if (a.stages > 1 && si.x > 0 && tid < 32) {
            const bool ready = deps_ready(a, si.x, si.y, tid, true, 0);
            if (tid == 0) S.ready = ready;
        } else if (tid == 0) {
            S.ready = 1;
        }
        __syncthreads();                 // S.K, S.ready
        if (!S.ready) {                  // a bounded wait gave up: report it and stop
            if (tid == 0) atomicOr(a.flag, 2);
            return;
        }
        const int x0 = item.y * kStripX;
        const int stage = si.x % 3;
        if (S.K.gen) {
            if (S.K.axi) short_item<R, true, true>(S, a, stage, x0, item.z, item.w);
            else short_item<R, false, true>(S, a, stage, x0, item.z, item.w);
        } else {
            if (S.K.axi) short_item<R, true, false>(S, a, stage, x0, item.z, item.w);
            else short_item<R, false, false>(S, a, stage, x0, item.z, item.w);
        }
        if (tid == 0) S.next = claimed;
        __syncthreads();                 // every thread's stores of this item; S.next
        if (a.stages > 1 && tid == 0 && !a.dep_probe) {
            __threadfence();
            atomicExch(a.done + (size_t)si.x * a.nitems + si.y, 1);
        }
    }
}

namespace {

constexpr int kMaxAttrDevices = 64;

// The dynamic shared-memory limit is a per-device attribute (see stage.cu).
template <class R>
cudaError_t configure_t() {
    static std::mutex m;
    static bool done[kMaxAttrDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(m);
    if (!done[dev]) {
        e = cudaFuncSetAttribute(short_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(ShortSmem<R>));
        if (e != cudaSuccess) return e;
        done[dev] = true;
    }
    return cudaSuccess;
}

template <class R>
cudaError_t launch_t(const StageLaunch& a, int grid, cudaStream_t s) {
    cudaError_t e = configure_t<R>();
    if (e != cudaSuccess) return e;
    short_kernel<R><<<grid, NTS, sizeof(ShortSmem<R>), s>>>(a);
    return cudaGetLastError();
}

template <class R>
int blocks_per_sm_t() {
    if (configure_t<R>() != cudaSuccess) return 1;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, short_kernel<R>, NTS, sizeof(ShortSmem<R>)) != cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

}  // namespace

cudaError_t launch_short(int precision, const StageLaunch& a, int grid, cudaStream_t s) {
    return precision == 0 ? launch_t<double>(a, grid, s) : launch_t<float>(a, grid, s);
}

int short_blocks_per_sm(int precision) { return precision == 0 ? blocks_per_sm_t<double>() : blocks_per_sm_t<float>(); }

}  // namespace eulbfs
