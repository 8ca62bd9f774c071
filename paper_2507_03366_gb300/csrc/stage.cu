// stage.cu -- the hot path of libeulbfs (sm_103a): one SSP-RK3 stage (Eq. 58)
// of the EULBFS explicit step over every domain of a batch.
//
// Work decomposition.  A work item is a strip segment of one domain: 31
// interior columns wide and a run of rows high.  A CTA of 8 warps sweeps its segment
// upwards in chunks of 8 rows, keeping the derived fields of the rows it needs
// in a 16-row ring buffer in shared memory, so every cell of the segment is
// loaded and derived once per stage (plus a 3-column halo on each side and a
// 6-row prologue per segment).  Per chunk:
//   1. load and derive 8 new rows: stage state -> T, F_l, C_p, rho, lambda,
//      mu (Eq. 5-7), u = m / (rho cs^2), p, C; halo cells outside the domain
//      are mapped through the boundary rules (mirror + value rule, or wrap);
//   2. mu_c = 2 beta C (C-1)(2C-1) - kappa lap C (Sec. 2.3.1) for 8 rows;
//      a wall ghost takes the value at its mirror cell;
//   3. every face once: warp w computes the 32 x-faces of chunk row w (one
//      per lane: 31 cells have 32 x-faces) and the 31 y-faces below row w+1
//      (the face row below the chunk comes from the previous chunk);
//   4. per cell: R(W) = -div F + F_E (Eq. 51-52), the Runge-Kutta stage, the
//      optional solid projection, a non-finite check, and the store.
// Work items span all domains of the batch, so one launch advances every
// domain by one stage; the grid is persistent and strides over the items.
#include <mutex>

#include "stage_device.cuh"

namespace eulbfs {

namespace {

constexpr int NT = kStageThreads;         // 8 warps
constexpr int kTiledDeps = 32;            // neighbours kept in shared memory (further ones are read from dep_idx)

template <class R>
struct Smem : Core<R> {
    // the next rows' stage input, all planes, copied by TMA while the
    // current chunk computes (planes x rows x columns, as the tensor map's box)
    // (FP32C only: the FP64 step is bound by the FP64 pipe, not by its loads)
    alignas(128) R tile[sizeof(R) == 4 ? Prec<R>::NP : 1][kChunk][kTileX];
    unsigned long long tile_bar;      // mbarrier: the tile's copy has landed
    int cur_domain;
    int next;                         // the claimed position of the CTA's next work item
    int pre;                          // 1: the tile holds (or is receiving) the next item's prologue rows
    // the next work item, looked up while the current one runs
    int4 item;
    int pos;                          // its place in the launch's item sequence (>= its length: no more)
    int stage, index;                 // its stage of the launch and its place in the work list
    int ndeps, dep0;                  // the items it waits for: how many, and their offset in dep_idx
    int dep[kTiledDeps];              // the first kTiledDeps of them
    int ready;                        // they were all done when the current item's last chunk began
    int moves;                        // it lies in another domain than the current one
    int run_stage, run_index;         // the current item's (one thread's, for its done flag)
};

// ---------------------------------------------------------------------------
// Input tiles by TMA.  One thread issues a 3-D tensor copy (columns x rows x
// planes) into the shared tile with an mbarrier that counts its bytes; every
// thread waits on the barrier's phase.  A wait gives up after about 2^31 SM
// clocks (a second at 2 GHz): the kernel then sets bit 1 of the launch's
// flag, waits the same bound once more for the copy in flight, and returns.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_addr(const void* p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void bar_init(unsigned long long* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Per-CTA count of the tile copies waited for (the barrier's phase).
struct TileIO {
    unsigned phase;
};

// The first column of a tile: x0 - kHalo rounded down to 16 bytes.
template <class R>
__device__ __forceinline__ int tile_x(int x0) { return (x0 - kHalo) & ~(int)(16 / sizeof(R) - 1); }

// Rows [r0, r0 + nrows) of the strip at x0 come from a tile when the domain
// has tensor maps and every cell of those rows, with the column halo, is
// inside it (the chunks that need boundary rules load their cells directly).
template <class R>
__device__ __forceinline__ bool tile_rows(const Consts<R>& K, int x0, int r0, int nrows) {
    if constexpr (sizeof(R) != 4) return false;
    return K.tma && x0 >= kHalo && x0 + kStripX + kHalo <= K.nx && r0 >= -K.hlo && r0 + nrows <= K.ny + K.hhi;
}

// Thread 0 issues the copy of rows [r0, r0 + kChunk) of domain dom's stage
// buffer (its tensor map in the launch's map array; hlo: its halo rows below).
template <class R>
__device__ __forceinline__ void tile_fetch_from(Smem<R>& S, const StageLaunch& a, int stage, int dom, int hlo, int x0,
                                                int r0) {
    const unsigned bar = smem_addr(&S.tile_bar);
    const unsigned bytes = (unsigned)sizeof(S.tile) + a.tile_probe;
    const char* map = static_cast<const char*>(a.tmaps) + ((size_t)dom * 3 + stage) * kTmapBytes;
    // the tile's previous contents were read through the generic proxy
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_addr(&S.tile[0][0][0])), "l"(map), "r"(tile_x<R>(x0)), "r"(r0 + hlo), "r"(0), "r"(bar)
        : "memory");
}

// The same for the current domain.
template <class R>
__device__ __forceinline__ void tile_fetch(Smem<R>& S, const StageLaunch& a, int stage, int x0, int r0) {
    if (threadIdx.x == 0) tile_fetch_from(S, a, stage, S.cur_domain, S.K.hlo, x0, r0);
}

// Put item number g of the launch into S (one whole warp).
template <class R>
__device__ __forceinline__ void look_up(Smem<R>& S, const StageLaunch& a, int g, int lane) {
    if (g < a.nitems * a.stages) {
        const int2 si = stage_item(a, g);
        const int4 item = a.items[si.y];
        int d0 = 0, n = 0;
        if (a.stages > 1 && si.x > 0) {   // one-stage launches are ordered by the kernel boundary
            d0 = a.dep_off[si.y];
            n = a.dep_off[si.y + 1] - d0;
            if (lane < n) S.dep[lane] = a.dep_idx[d0 + lane];
        }
        if (lane == 0) {
            S.item = item;
            S.stage = si.x;
            S.index = si.y;
            S.ndeps = n;
            S.dep0 = d0;
            S.moves = item.x != S.cur_domain;
        }
    }
    if (lane == 0) S.pos = g;
}

// True once every item that the next one reads has finished the previous
// stage (one whole warp; lanes take one neighbour each).  With `wait` a bounded
// wait: after 2^31 clocks it gives up and returns false.
template <class R>
__device__ __forceinline__ bool next_ready(const Smem<R>& S, const StageLaunch& a, int lane, bool wait) {
    const int n = S.ndeps;
    const int* done = a.done + (size_t)(S.stage - 1) * a.nitems;
    bool ok = true;
    for (int j = lane; j < n; j += 32) {
        const int* f = done + (j < kTiledDeps ? S.dep[j] : a.dep_idx[S.dep0 + j]);
        if (ld_acquire(f)) continue;
        if (!wait) { ok = false; continue; }
        const long long t0 = clock64();
        while (!ld_acquire(f)) {
            if (clock64() - t0 > (1LL << 31)) { ok = false; break; }
            __nanosleep(256);
        }
    }
    return __all_sync(0xffffffffu, ok);
}

// During the last chunk of a work item (one whole warp; FP32C: the tile is
// free): records whether the CTA's next item can start, and if so thread 0
// copies its prologue rows, when they come from a tile (S.pre).
template <class R>
__device__ __forceinline__ void prepare_next(Smem<R>& S, const StageLaunch& a, int lane) {
    int pre = 0;
    bool ready = true;
    if (S.pos < a.nitems * a.stages) {
        ready = next_ready(S, a, lane, false);
        if constexpr (sizeof(R) == 4) {
            const int4 item = S.item;
            const Consts<R>& Kn = static_cast<const Consts<R>*>(a.consts)[item.x];
            const int x0 = item.y * kStripX, r0 = item.z - kHalo;
            if (ready && tile_rows(Kn, x0, r0, 2 * kHalo)) {
                __syncwarp();   // the lanes' acquire loads before lane 0's proxy fence
                if (lane == 0) {
                    // the rows were written by other CTAs through the generic proxy
                    asm volatile("fence.proxy.async.global;" ::: "memory");
                    tile_fetch_from(S, a, S.stage % 3, item.x, Kn.hlo, x0, r0);
                }
                pre = 1;
            }
        }
    }
    if (lane == 0) {
        S.pre = pre;
        S.ready = ready;
    }
}

// The cell update reads W^n and dF_s/dt (stages 2 and 3) or F_s^{n-1}
// (stage 1) straight from global memory, where nothing has touched them
// during the step.  One warp asks L2 for rows r0 .. r0+7 of those arrays
// a chunk before their update: lane l takes row r0 + l % 8 and arrays
// l / 8 and l / 8 + 4 (the 7 state planes, then dF_s/dt), both ends of the
// strip's segment of each row.  Prefetches are hints: they change no value.
__device__ __forceinline__ void l2_prefetch(const void* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(p)));
}

template <class R>
__device__ __forceinline__ void prefetch_update_rows(const Consts<R>& K, int stage, int x0, int r0, int y1, int lane) {
    const int r = r0 + (lane & 7);
    if (r >= y1) return;
    const long long c0 = (long long)r * K.nx + K.off + x0;
    const long long c1 = (long long)r * K.nx + K.off + min(x0 + kStripX, K.nx) - 1;
    const int k = lane >> 3;
    if (stage == 0) {
        if (k == 0) {
            const R* f = reinterpret_cast<const R*>(K.Fsp);
            l2_prefetch(f + c0);
            l2_prefetch(f + c1);
        }
        return;
    }
    const R* w = reinterpret_cast<const R*>(K.st[0]);
    l2_prefetch(w + k * K.plane + c0);
    l2_prefetch(w + k * K.plane + c1);
    const R* b = k + 4 < Prec<R>::NP ? w + (k + 4) * K.plane : reinterpret_cast<const R*>(K.dFs);
    if (k + 4 <= Prec<R>::NP) {
        l2_prefetch(b + c0);
        l2_prefetch(b + c1);
    }
}

__device__ __forceinline__ bool bar_try_wait(unsigned bar, unsigned parity) {
    unsigned done;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}

// The bounded retry loop (out of line: the tile has normally landed long
// before its chunk starts, and the first try succeeds).
__device__ __noinline__ bool bar_wait_bounded(unsigned bar, unsigned parity) {
    const long long t0 = clock64();
    while (!bar_try_wait(bar, parity))
        if (clock64() - t0 > (1LL << 31)) return false;
    return true;
}

// Wait for the copy issued last; false if the bound ran out.
template <class R>
__device__ __forceinline__ bool tile_wait(Smem<R>& S, TileIO& io) {
    const unsigned bar = smem_addr(&S.tile_bar), parity = io.phase & 1u;
    ++io.phase;
    return bar_try_wait(bar, parity) || bar_wait_bounded(bar, parity);
}

// The state of tile column cc (0 .. RW-1 of the strip) in row rr.
__device__ __forceinline__ SV<float> tile_state(const float* t) {
    constexpr int PS = kChunk * kTileX;
    SV<float> s;
    s.Hh = t[0]; s.Hl = t[PS]; s.p = t[2 * PS]; s.mx = t[3 * PS]; s.my = t[4 * PS]; s.Ch = t[5 * PS]; s.Cl = t[6 * PS];
    return s;
}
__device__ __forceinline__ SV<double> tile_state(const double* t) {
    constexpr int PS = kChunk * kTileX;
    SV<double> s;
    s.Hh = t[0]; s.Hl = 0.0; s.p = t[PS]; s.mx = t[2 * PS]; s.my = t[3 * PS]; s.Ch = t[4 * PS]; s.Cl = 0.0;
    return s;
}

// Step 1 from a tile: rows [r0, r0 + nrows) (all inside the domain, see
// tile_rows) read from shared memory instead of global memory.
template <class R>
__device__ __forceinline__ void load_rows_tile(Smem<R>& S, int x0, int r0, int nrows) {
    const Consts<R>& K = S.K;
    const int xoff = (x0 - kHalo) - tile_x<R>(x0);
    const int total = nrows * RW;
    for (int idx = threadIdx.x; idx < total; idx += NT) {
        const int rr = idx / RW, cc = idx - rr * RW;
        store_prim(S, slot(r0 + rr), cc, derive(K, tile_state(&S.tile[0][rr][cc + xoff])));
    }
}

// The barrier after a load phase; true (on every thread) if some thread's
// tile wait gave up.  Without tiles (FP64) a plain barrier.
template <class R>
__device__ __forceinline__ bool load_barrier_failed(Smem<R>& S, bool ok) {
    if constexpr (sizeof(R) == 4) {
        return __syncthreads_or(!ok) != 0;
    } else {
        __syncthreads();
        return false;
    }
}

// A wait for the items an item reads gave up (whole-step launches): report
// it as a bounded wait that gave up, wait for a prologue tile that may be in
// flight, and stop.
template <class R>
__device__ __noinline__ void dep_abort(Smem<R>& S, TileIO io, int* flag) {
    if (threadIdx.x == 0) atomicOr(flag, 2);
    if constexpr (sizeof(R) == 4)
        if (S.pre) tile_wait(S, io);
}

// A tile wait gave up: report it, wait (with the same bound) for the copy
// still in flight so that it cannot land in shared memory after the CTA has
// left, and stop.
template <class R>
__device__ __noinline__ bool tile_abort(Smem<R>& S, TileIO io, int* flag) {
    if (threadIdx.x == 0) atomicOr(flag, 2);
    --io.phase;
    tile_wait(S, io);
    return false;
}

// Steps 1 and 2 of an interior chunk from its tile (FP32C): rows
// [r0, r0 + kChunk) derived as in load_rows_tile and, by the same threads,
// mu_c of rows [r0 - 1, r0 + kChunk - 1) (muc_in_place must hold).  Their
// C comes from the tile (rows >= r0, C_hi + C_lo as derive forms it) or
// from the ring (rows r0 - 2, r0 - 1, derived by the previous chunk), so
// mu_c needs no barrier after the derive; the values are those muc_rows
// computes.
template <class R, bool AXI>
__device__ __forceinline__ void load_rows_tile_muc(Smem<R>& S, int x0, int r0, bool with_muc) {
    const Consts<R>& K = S.K;
    constexpr int PS = kChunk * kTileX;
    const int xoff = (x0 - kHalo) - tile_x<R>(x0);
    const R* t = &S.tile[0][0][0];
    for (int idx = threadIdx.x; idx < kChunk * RW; idx += NT) {
        const int rr = idx / RW, cc = idx - rr * RW;
        store_prim(S, slot(r0 + rr), cc, derive(K, tile_state(t + rr * kTileX + cc + xoff)));
    }
    if (!with_muc) return;
    // mu_c of ring row r0 + m, m = -1 .. kChunk-2, columns 1 .. RW-2
    const P2<R>* RC = &S.P.rc[0][0];
    constexpr int NC = RW - 2;
    for (int idx = threadIdx.x; idx < kChunk * NC; idx += NT) {
        const int m = idx / NC - 1, cc = 1 + idx - (m + 1) * NC;
        // C of row r0 + k at column cc + d: the tile for k >= 0, the ring below
        auto Cat = [&](int k, int d) -> R {
            const int ti = k * kTileX + cc + d + xoff;
            return k >= 0 ? t[5 * PS + ti] + t[6 * PS + ti] : RC[slot(r0 + k) * RW + cc + d].y;
        };
        S.P.pm[slot(r0 + m)][cc].y =
            chem_potential_of<R, AXI>(K, Cat(m, 0), Cat(m, 1), Cat(m, -1), Cat(m + 1, 0), Cat(m - 1, 0),
                                     AXI ? left_radius(S, cc, x0 + cc - kHalo) : R(0),
                                     AXI ? S.inv_rc[cc] : R(0));
    }
}

// One work item of Runge-Kutta stage `stage`: the strip segment
// [x0, x0 + 31) x [y0, y1) of the domain whose constants are in S.K (planar
// or axisymmetric, fixed per domain).  Returns false if a wait for an input
// tile gave up (the kernel then stops).
template <class R, bool AXI, bool GEN>
__device__ __forceinline__ bool sweep_item(Smem<R>& S, const StageLaunch& a, const int stage, TileIO& io, int x0,
                                           int y0, int y1) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const R* in = reinterpret_cast<const R*>(S.K.st[stage]);
    // a lane keeps its column through the item: in an axisymmetric domain
    // 1 / r of its cell centre (y-faces, cell volume) and of its x-face
    // (0 on the axis, where the face area is zero)
    const R ir_c = AXI ? wdiv(R(1), (R)(x0 + lane) + R(0.5)) : R(1);
    const R ir_f = (AXI && x0 + lane > 0) ? wdiv(R(1), (R)(x0 + lane)) : R(0);

    // prologue: rows y0-3 .. y0+2, mu_c of rows y0-2 .. y0+1, y-face row y0.
    // Its 6 x 37 cells leave the last warp idle: that one claims the next item,
    // and looks it up while the first warp computes the y-face row.
    column_radii<R, AXI>(S, x0);
    if (tid == NT - 32) S.next = atomicAdd(a.work + (a.stages == 1 ? a.stage : 0), 1);
    bool ok = true;
    if (tile_rows(S.K, x0, y0 - kHalo, 2 * kHalo)) {
        if (!S.pre) tile_fetch(S, a, stage, x0, y0 - kHalo);   // else copied during the previous item
        ok = tile_wait(S, io);
        load_rows_tile(S, x0, y0 - kHalo, 2 * kHalo);
    } else {
        load_rows<R, NT>(S, in, x0, y0 - kHalo, 2 * kHalo);
    }
    if (load_barrier_failed<R>(S, ok)) return tile_abort(S, io, a.flag);
    // the first chunk's rows arrive while the prologue computes
    if (tile_rows(S.K, x0, y0 + kHalo, kChunk)) tile_fetch(S, a, stage, x0, y0 + kHalo);
    if constexpr (sizeof(R) == 4)
        if (warp == NT / 32 - 1) prefetch_update_rows(S.K, stage, x0, y0, y1, lane);
    muc_rows<R, AXI, NT>(S, x0, y0 - 2, 4);
    __syncthreads();
    if (warp == NT / 32 - 1) look_up(S, a, S.next, lane);
    if (warp == 0 && lane < kStripX) y_face<R, AXI, GEN>(S, y0, lane, AXI ? ir_c : R(0));
    // (the first chunk writes other ring rows: no barrier needed here)

    for (int j0 = y0; j0 < y1; j0 += kChunk) {
        // rows j0+3 .. j0+10: from the tile copied during the previous chunk,
        // or directly where boundary rules apply
        bool muc_done = false;
        if (tile_rows(S.K, x0, j0 + kHalo, kChunk)) {
            ok = tile_wait(S, io);
            if constexpr (sizeof(R) == 4) muc_done = muc_in_place(S.K, x0, j0 + 2, kChunk);
            load_rows_tile_muc<R, AXI>(S, x0, j0 + kHalo, muc_done);
        } else {
            load_rows<R, NT>(S, in, x0, j0 + kHalo, kChunk);
        }
        if (load_barrier_failed<R>(S, ok)) return tile_abort(S, io, a.flag);
        // the tile is free again: copy the next chunk's rows behind this one,
        // or after the last chunk the next work item's prologue rows
        if (j0 + kChunk < y1) {
            if (tile_rows(S.K, x0, j0 + kChunk + kHalo, kChunk)) tile_fetch(S, a, stage, x0, j0 + kChunk + kHalo);
        } else if (warp == 0) {
            prepare_next(S, a, lane);
        }
        // the next chunk's update rows into L2 (FP32C: the FP64 step is
        // bound by its FP64 arithmetic)
        if constexpr (sizeof(R) == 4)
            if (warp == NT / 32 - 1 && j0 + kChunk < y1) prefetch_update_rows(S.K, stage, x0, j0 + kChunk, y1, lane);
        if (!muc_done) {   // rows j0+2 .. j0+9
            muc_rows<R, AXI, NT>(S, x0, j0 + 2, kChunk);
            __syncthreads();
        }
        // one face at a time per thread (x then y) keeps register use low
#pragma unroll 1
        for (int k = 0; k < 2; ++k) {
            if (j0 + warp >= y1) break;   // rows past the item's end (its last chunk)
            if (k == 0) x_face<R, AXI, GEN>(S, x0, j0 + warp, warp, lane, ir_f);
            else if (lane < kStripX) y_face<R, AXI, GEN>(S, j0 + 1 + warp, lane, AXI ? ir_c : R(0));
        }
        __syncthreads();
        const int r = j0 + warp;
        if (r < y1 && lane < kStripX && x0 + lane < S.K.nx) {
            const GlobalCell<R> src{S.K, stage, (long long)r * S.K.nx + x0 + lane + S.K.off};
            cell_update<R, AXI>(S, src, stage, src.c, r, warp, lane, ir_c, a.flag);
        }
        __syncthreads();
    }
    return true;
}

}  // namespace

template <class R>
__global__ void __launch_bounds__(NT, sizeof(R) == 4 ? 4 : 2) stage_kernel(StageLaunch a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem<R>& S = *reinterpret_cast<Smem<R>*>(smem_raw);
    const int tid = threadIdx.x;
    if (tid == 0) {
        S.cur_domain = -1;
        S.pre = 0;
        bar_init(&S.tile_bar);
    }
    __syncthreads();
    launch_dependents();
    wait_prior();
    const Consts<R>* consts = static_cast<const Consts<R>*>(a.consts);
    TileIO io{0u};

    // Every item is claimed from the launch's counter, one item ahead, and looked
    // up by the warp that the prologue leaves idle, so an item whose inputs are
    // done starts behind the barrier that ends the one before it (at the item's
    // start the look-up is an atomic and four dependent loads, with three more
    // barriers).  us per step, before and after: 512^2 58.9 -> 54.1, 640^2 74.9 -> 70.0,
    // 1024^2 164.3 -> 154.7, 16 domains 222 -> 214 (planar, streaming 244 -> 237),
    // 64 domains (7.23 M cells) 1041 -> 1022; FP64 unchanged (919 -> 917 at 512^2).
    // In a whole-step launch the items of stage 1 follow all of stage 0 and those
    // of stage 2 all of stage 1 (then stage 0 of the next step, when the
    // launch runs several), and an item waits for the items of the previous
    // stage it reads.  Only running CTAs hold items, and every item
    // waits only for items claimed before it, so the earliest unfinished
    // item can always proceed.
    if (tid < 32) {
        int g = 0;
        if (tid == 0) g = atomicAdd(a.work + (a.stages == 1 ? a.stage : 0), 1);
        look_up(S, a, __shfl_sync(0xffffffffu, g, 0), tid);
        if (tid == 0) S.ready = S.ndeps == 0;
    }
    __syncthreads();
    // An item starts behind the barrier that ends the one before it; S's next
    // item is replaced behind further barriers, in the sweep.
    while (S.pos < a.nitems * a.stages) {
        const int4 item = S.item;
        const int st = S.stage;
        if (S.moves || !S.ready) {
            __syncthreads();             // S.moves, S.ready read by every thread
            if (tid < 32 && !S.ready) {
                const bool ready = next_ready(S, a, tid, true);
                __syncwarp();
                if (tid == 0) S.ready = ready;
            }
            if (S.moves) {
                const unsigned* src = reinterpret_cast<const unsigned*>(consts + item.x);
                unsigned* dst = reinterpret_cast<unsigned*>(&S.K);
                for (int k = tid; k < (int)(sizeof(Consts<R>) / 4); k += NT) dst[k] = src[k];
                if (tid == 0) S.cur_domain = item.x;
            }
            __syncthreads();             // S.K, S.ready
            if (!S.ready) return dep_abort(S, io, a.flag);
        }
        if (a.stages > 1) {
            // the rows this item copies by TMA were written through the generic proxy
            if (tid == 0 && st > 0) asm volatile("fence.proxy.async.global;" ::: "memory");
            if (tid == NT - 32) {
                S.run_stage = st;
                S.run_index = S.index;
            }
        }
        const int x0 = item.y * kStripX;
        const int y0 = item.z, y1 = item.w;
        bool ok;
        if (S.K.gen) {   // some streaming step differs from 1/2 (reading R26)
            if (S.K.axi) ok = sweep_item<R, true, true>(S, a, st % 3, io, x0, y0, y1);
            else ok = sweep_item<R, false, true>(S, a, st % 3, io, x0, y0, y1);
        } else {
            if (S.K.axi) ok = sweep_item<R, true, false>(S, a, st % 3, io, x0, y0, y1);
            else ok = sweep_item<R, false, false>(S, a, st % 3, io, x0, y0, y1);
        }
        if (!ok) return;   // uniform: every thread saw the same __syncthreads_or
        if (a.stages > 1 && tid == NT - 32 && !a.dep_probe) {
            // publish: every thread's stores of this item (the sweep's last barrier), then its flag
            __threadfence();
            atomicExch(a.done + (size_t)S.run_stage * a.nitems + S.run_index, 1);
        }
    }
}

// The dynamic shared-memory limit of stage_kernel<R> is a per-device
// attribute: it is set once for every device the kernel is launched on, under
// a lock, so that solvers on several devices and several host threads can
// launch it.
constexpr int kMaxAttrDevices = 64;

template <class R>
static cudaError_t configure_t() {
    static std::mutex m;
    static bool done[kMaxAttrDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(m);
    if (!done[dev]) {
        e = cudaFuncSetAttribute(stage_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem<R>));
        if (e != cudaSuccess) return e;
        done[dev] = true;
    }
    return cudaSuccess;
}

template <class R>
static cudaError_t launch_t(const StageLaunch& a, int grid, cudaStream_t s) {
    cudaError_t e = configure_t<R>();
    if (e != cudaSuccess) return e;
    return launch_behind(a.behind, stage_kernel<R>, dim3(grid), NT, sizeof(Smem<R>), s, a);
}

template <class R>
static int blocks_per_sm_t() {
    const size_t smem = sizeof(Smem<R>);
    if (configure_t<R>() != cudaSuccess) return 1;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, stage_kernel<R>, NT, smem) != cudaSuccess) return 1;
    return nb > 0 ? nb : 1;
}

cudaError_t launch_stage(int precision, const StageLaunch& a, int grid, cudaStream_t s) {
    return precision == 0 ? launch_t<double>(a, grid, s) : launch_t<float>(a, grid, s);
}

int stage_blocks_per_sm(int precision) { return precision == 0 ? blocks_per_sm_t<double>() : blocks_per_sm_t<float>(); }

size_t stage_smem_bytes(int precision) { return precision == 0 ? sizeof(Smem<double>) : sizeof(Smem<float>); }

}  // namespace eulbfs
